// clot_eta_dct.cuh -- K2, direct form: the virtual-substance solve of App. A,
// Eq. eta, (I - (L_eta^2 / 4) lap_h) eta = theta_B with zero-flux walls, by
// separation of variables.  The second difference with zero-flux ends along y
// (and z) is diagonal in the orthonormal cosine modes
//     C_m(j) = s_m cos(pi m (2 j + 1) / (2 n)),   -lap -> 4 sin^2(pi m / (2 n)),
// so the solve is: cosine transform along y (and z), one tridiagonal solve
// along x per mode, and the transforms back.  It is applied to the residual:
// A d = theta_B - A eta0, eta = eta0 + d, so its FP32 rounding is relative to
// the correction, not to eta (and a second pass refines a cold start).
//
// Phases of the cooperative launch, a grid barrier between each two:
//   [residual of eta0 and its maxima, unless the fused step has written them]
//   y forward | z forward (3D) | x solves | z back (3D) | y back, added to eta.
//
//   transforms  dense matrix products on a folded axis: the sums and the
//       differences f_j +- f_{n-1-j} feed the even and the odd modes, half the
//       multiplications each.  Tiles of 64 (or 32) modes x 64 columns, operands
//       staged in shared memory 32 rows at a time with the next rows' loads in
//       flight, 8 x 4 (4 x 4) accumulators per thread.
//   x solves    a warp per mode line.  With rho the decaying root of the line's
//       constant stencil the free-space solution is a causal and an anticausal
//       first-order recursion, each lane running its 4 .. 32 cells and the lanes
//       joined by a weighted shuffle scan; the two ends add image terms
//       A rho^i + B rho^(w-1-i).  The recursions use u - (1 - rho) u, 1 - rho
//       being known to full relative accuracy where rho is close to 1.
//
// The predicted eta of the fused step is corrected on a slab of x only: the
// columns whose |r| exceeds stop / (2 (1 + c_x)), widened by
// ln(2 c_x max|r| / stop) / mu cells, cosh(mu) = 1 + 1 / (2 c_x), with d = 0
// outside (the x solves then end in a zero-value image).  exp(-mu |x|) times
// max|r| bounds the correction (A is an M-matrix and A exp(-mu |x|) >= 0), so
// the cells next to the slab keep a residual within the stopping rule.
//
// Where that is faster (direct_ns, box_cg_ns) the prediction is corrected by CG on
// a box instead.  Where no theta_B exceeds eta_t the kernel iterates too (clot_eta_cg.cuh):
// eta <= max theta_B, so the affinity g(eta) is zero in every cell whatever the
// solve returns, and what it returns is the iterate that first meets the
// stopping rule -- one or two iterations from a prediction.
//
// What bounds it: grid barriers and operand latency on small meshes, the FP32
// multiply-adds, 2 ncell (ny + nz) / 2 each way, on large ones.
#pragma once

#include "clot_eta_cg.cuh"

namespace clot {

constexpr int TN = 64, TK = 32;

struct DctSm {
  float a[2][2][TK][64];  // two stages of matrix rows (copied asynchronously), one operand per parity
  float b[2][TK][TN];
};
__device__ __forceinline__ void copy16(void* smem, const void* gmem) {
  const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(s), "l"(gmem) : "memory");
}
__device__ __forceinline__ void copies_landed() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }

struct Axis {
  int n, H;
  const float* F;  // [2][H][H] forward, F[par][j][m'] = C_{2 m' + par}(j)
  const float* I;  // [2][H][H] back, I[par][m'][j]
  const float* ev;
};
__device__ __forceinline__ Axis axis_of(int n, const float* mat) {
  const int H = dct_half(n);
  return Axis{n, H, mat, mat + 2 * (long long)H * H, mat + 4 * (long long)H * H};
}

template <int N>
__device__ __forceinline__ void load_rows(float (&v)[N], const float* p) {
#pragma unroll
  for (int u = 0; u < N; u += (N % 4 ? 2 : 4)) {
    if (N % 4) {
      const float2 a = *reinterpret_cast<const float2*>(p + u);
      v[u] = a.x;
      v[u + 1] = a.y;
    } else {
      const float4 a = *reinterpret_cast<const float4*>(p + u);
      v[u] = a.x;
      v[u + 1] = a.y;
      v[u + 2 < N ? u + 2 : u] = a.z;
      v[u + 3 < N ? u + 3 : u] = a.w;
    }
  }
}

// Forward modes 2 (m0 + .) + par of one tile of 16 column quads.  ld(j): the
// thread's quad (tid & 15) of row j; st(m, v): its quad of mode m.  sg: the
// stage of S.a that the next rows go to.  It alternates across the tiles of a
// block too: the first rows of a tile are copied without a block barrier since
// the last rows of the tile before were used, and those lie in the other stage.
template <int BS, int TM, class Ld, class St>
__device__ __forceinline__ void dct_forward(const Axis& X, int par, int m0, DctSm& S, int& sg, Ld ld, St st) {
  constexpr int GR = BS / 16, MT = TM / GR, NA = TK * TM / 4 / BS, NB = TK / GR;
  const int tid = threadIdx.x, q = tid & 15, g = tid >> 4, n = X.n, H = X.H;
  const int K = par ? n / 2 : (n + 1) / 2;
  if (K == 0) return;  // n = 1: no odd mode
  const float* Fm = X.F + (long long)par * H * H + m0;
  const float sgn = par ? -1.0f : 1.0f;
  float acc[MT][4];
#pragma unroll
  for (int u = 0; u < MT; ++u)
#pragma unroll
    for (int e = 0; e < 4; ++e) acc[u][e] = 0.0f;
  float4 pb[NB], ph[NB];  // rows j and n - 1 - j, folded when they are stored
  auto fetch = [&](int k0) {
#pragma unroll
    for (int u = 0; u < NA; ++u) {
      const int x = tid + u * BS, row = x / (TM / 4), col = 4 * (x % (TM / 4));
      copy16(&S.a[sg][0][row][col], Fm + (long long)(k0 + row) * H + col);
    }
#pragma unroll
    for (int u = 0; u < NB; ++u) {
      const int j = k0 + g + GR * u, jj = n - 1 - j;
      pb[u] = ph[u] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
      if (j < K) {
        pb[u] = ld(j);
        if (jj != j) ph[u] = ld(jj);
      }
    }
  };
  fetch(0);
  for (int k0 = 0; k0 < K; k0 += TK) {
    const int now = sg;
    sg ^= 1;
    __syncthreads();  // the last rows are used up
#pragma unroll
    for (int u = 0; u < NB; ++u)
      *reinterpret_cast<float4*>(&S.b[0][g + GR * u][4 * q]) =
          make_float4(fmaf(sgn, ph[u].x, pb[u].x), fmaf(sgn, ph[u].y, pb[u].y), fmaf(sgn, ph[u].z, pb[u].z),
                      fmaf(sgn, ph[u].w, pb[u].w));
    copies_landed();
    __syncthreads();
    if (k0 + TK < K) fetch(k0 + TK);
    const int kn = min(TK, K - k0);
#pragma unroll 4
    for (int k = 0; k < kn; ++k) {
      const float4 b = *reinterpret_cast<const float4*>(&S.b[0][k][4 * q]);
      float av[MT];
      load_rows<MT>(av, &S.a[now][0][k][g * MT]);
#pragma unroll
      for (int u = 0; u < MT; ++u) {
        acc[u][0] = fmaf(av[u], b.x, acc[u][0]);
        acc[u][1] = fmaf(av[u], b.y, acc[u][1]);
        acc[u][2] = fmaf(av[u], b.z, acc[u][2]);
        acc[u][3] = fmaf(av[u], b.w, acc[u][3]);
      }
    }
  }
#pragma unroll
  for (int u = 0; u < MT; ++u) {
    const int m = 2 * (m0 + g * MT + u) + par;
    if (m < n) st(m, make_float4(acc[u][0], acc[u][1], acc[u][2], acc[u][3]));
  }
}

// Back to rows j0 + . and their mirror rows of one tile of 16 column quads.
// ld(m): the thread's quad of mode m; st(j, v): its quad of row j; sg as in
// dct_forward.
template <int BS, int TM, class Ld, class St>
__device__ __forceinline__ void dct_back(const Axis& X, int j0, DctSm& S, int& sg, Ld ld, St st) {
  constexpr int GR = BS / 16, MT = TM / GR, NA = TK * TM / 4 / BS, NB = TK / GR;
  const int tid = threadIdx.x, q = tid & 15, g = tid >> 4, n = X.n, H = X.H;
  const int K = (n + 1) / 2;
  float acc[2][MT][4];
#pragma unroll
  for (int p = 0; p < 2; ++p)
#pragma unroll
    for (int u = 0; u < MT; ++u)
#pragma unroll
      for (int e = 0; e < 4; ++e) acc[p][u][e] = 0.0f;
  float4 pb[2][NB];
  auto fetch = [&](int k0) {
#pragma unroll
    for (int p = 0; p < 2; ++p) {
      const float* Im = X.I + (long long)p * H * H + j0;
#pragma unroll
      for (int u = 0; u < NA; ++u) {
        const int x = tid + u * BS, row = x / (TM / 4), col = 4 * (x % (TM / 4));
        copy16(&S.a[sg][p][row][col], Im + (long long)(k0 + row) * H + col);
      }
#pragma unroll
      for (int u = 0; u < NB; ++u) {
        const int m = 2 * (k0 + g + GR * u) + p;
        pb[p][u] = m < n ? ld(m) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
      }
    }
  };
  fetch(0);
  for (int k0 = 0; k0 < K; k0 += TK) {
    const int now = sg;
    sg ^= 1;
    __syncthreads();  // the last rows are used up
#pragma unroll
    for (int p = 0; p < 2; ++p)
#pragma unroll
      for (int u = 0; u < NB; ++u) *reinterpret_cast<float4*>(&S.b[p][g + GR * u][4 * q]) = pb[p][u];
    copies_landed();
    __syncthreads();
    if (k0 + TK < K) fetch(k0 + TK);
    const int kn = min(TK, K - k0);
#pragma unroll 2
    for (int k = 0; k < kn; ++k) {
#pragma unroll
      for (int p = 0; p < 2; ++p) {
        const float4 b = *reinterpret_cast<const float4*>(&S.b[p][k][4 * q]);
        float av[MT];
        load_rows<MT>(av, &S.a[now][p][k][g * MT]);
#pragma unroll
        for (int u = 0; u < MT; ++u) {
          acc[p][u][0] = fmaf(av[u], b.x, acc[p][u][0]);
          acc[p][u][1] = fmaf(av[u], b.y, acc[p][u][1]);
          acc[p][u][2] = fmaf(av[u], b.z, acc[p][u][2]);
          acc[p][u][3] = fmaf(av[u], b.w, acc[p][u][3]);
        }
      }
    }
  }
#pragma unroll
  for (int u = 0; u < MT; ++u) {
    const int j = j0 + g * MT + u;
    if (j >= K) continue;
    const float* e = acc[0][u];
    const float* o = acc[1][u];
    st(j, make_float4(e[0] + o[0], e[1] + o[1], e[2] + o[2], e[3] + o[3]));
    if (n - 1 - j != j) st(n - 1 - j, make_float4(e[0] - o[0], e[1] - o[1], e[2] - o[2], e[3] - o[3]));
  }
}

// One mode line: x <- the solution of (aa - c delta^2) x = line on w cells,
// in place, by one warp; lane l owns cells l L .. l L + L - 1.  End types: wall
// (zero flux) or cut (zero value beyond the slab).
template <int L>
__device__ __forceinline__ void x_line(float* line, int w, int W4, float aa, float c, bool wall0, bool wall1) {
  const int lane = threadIdx.x & 31, b0 = lane * L;
  float h[L], t[L];
#pragma unroll
  for (int u = 0; u < L; u += 4) {
    const float4 v = (b0 + u < W4) ? ld4(line + b0 + u) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    h[u] = v.x; h[u + 1] = v.y; h[u + 2] = v.z; h[u + 3] = v.w;
  }
  const float q = 0.5f * aa / c;
  const float s = q + sqrtf(q * (q + 2.0f));  // rho = 1 / (1 + s)
  const float mu = log1pf(s), del = s / (1.0f + s), rho = 1.0f - del;
  const float kap = (1.0f + s) / (c * s * (2.0f + s));
  // causal sums u_i = h_i + rho u_{i-1} and anticausal t_i = rho (h_{i+1} + t_{i+1}),
  // first inside the lane
  float u = 0.0f, v = 0.0f;
#pragma unroll
  for (int e = 0; e < L; ++e) u = fmaf(-del, u, u) + h[e];
#pragma unroll
  for (int e = L - 1; e >= 0; --e) v = fmaf(-del, v, v) + h[e];
  // joined across the lanes: cu the causal sum at the end of the lane's cells, cv the anticausal one at their start
  float cu = u, cv = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const float f = expf(-mu * (float)(L * o));
    const float xu = __shfl_up_sync(0xffffffffu, cu, o), xv = __shfl_down_sync(0xffffffffu, cv, o);
    if (lane >= o) cu = fmaf(f, xu, cu);
    if (lane < 32 - o) cv = fmaf(f, xv, cv);
  }
  float iu = __shfl_up_sync(0xffffffffu, cu, 1), iv = __shfl_down_sync(0xffffffffu, cv, 1);
  if (lane == 0) iu = 0.0f;
  if (lane == 31) iv = 0.0f;
  const float E0 = __shfl_sync(0xffffffffu, cv, 0);  // sum_j rho^j h_j
  v = iv;
#pragma unroll
  for (int e = L - 1; e >= 0; --e) {
    t[e] = fmaf(-del, v, v);  // rho v: what lies beyond cell e
    v = t[e] + h[e];
  }
  float E1 = 0.0f;  // sum_j rho^(w-1-j) h_j
  u = iu;
#pragma unroll
  for (int e = 0; e < L; ++e) {
    u = fmaf(-del, u, u) + h[e];
    if (b0 + e == w - 1) E1 = u;
    t[e] += u;
  }
  E1 = __shfl_sync(0xffffffffu, E1, (w - 1) / L);
  // image terms: A = sl (kap E0 + B R), B = sr (kap E1 + A R)
  const float sl = wall0 ? rho : -rho * rho, sr = wall1 ? rho : -rho * rho;
  const float R = expf(-mu * (float)(w - 1));
  const float ex = mu * (float)((wall0 ? 1 : 2) + (wall1 ? 1 : 2) + 2 * (w - 1));
  const float den = wall0 == wall1 ? -expm1f(-ex) : 1.0f + expf(-ex);
  const float A = sl * kap * (E0 + R * sr * E1) / den, B = sr * kap * (E1 + R * sl * E0) / den;
  float pA = A * expf(-mu * (float)b0), pB = 0.0f;
  // rho^(w-1-i) grows with i: start from the lane's last cell below w
  const int last = min(b0 + L, w) - 1;
  pB = last >= b0 ? B * expf(-mu * (float)(w - 1 - last)) : 0.0f;
#pragma unroll
  for (int e = L - 1; e >= 0; --e) {
    if (b0 + e <= last) {
      h[e] = pB;
      pB = fmaf(-del, pB, pB);
    } else {
      h[e] = 0.0f;
    }
  }
#pragma unroll
  for (int e = 0; e < L; ++e) {
    h[e] = fmaf(kap, t[e], pA + h[e]);
    pA = fmaf(-del, pA, pA);
  }
#pragma unroll
  for (int e = 0; e < L; e += 4)
    if (b0 + e < W4) st4(line + b0 + e, make_float4(h[e], h[e + 1], h[e + 2], h[e + 3]));
}

// One direct solve A d = a.r on the x slab [i0, i1], eta += d.  Every block of
// the grid calls it.  Returns false if a grid barrier gave up.
template <int BS>
__device__ __forceinline__ bool dct_solve(const EtaArgs& a, DctSm& S, int i0, int i1, Team& T) {
  const int nx = a.g.nx, ny = a.g.ny, nz = a.g.nz, tid = threadIdx.x, q = tid & 15;
  const int w = i1 - i0 + 1, W4 = (w + 3) & ~3, qpr = W4 >> 2;
  const bool d3 = a.g.dim == 3;
  const Axis Y = axis_of(ny, a.dct_y), Z = axis_of(d3 ? nz : 1, d3 ? a.dct_z : a.dct_y);
  const unsigned nb = T.nb;
  float* ga = a.dct_a;
  float* gb = a.dct_b;
  const bool vr = (nx & 3) == 0 && al16(a.r) && al16(a.eta);  // i0 is a multiple of 4
  const long long rowz = (long long)ny * W4;
  int sg = 0;  // stage of the shared matrix rows

  // ---- y forward: r -> ga
  {
    const int nq = nz * qpr, ct = (nq + 15) >> 4, mh = (ny + 1) >> 1;
    const bool big = 2u * ct * ((mh + 63) >> 6) >= nb;
    const int TM = big ? 64 : 32, mb = (mh + TM - 1) / TM, tiles = ct * mb * 2;
    for (int tile = blockIdx.x; tile < tiles; tile += nb) {
      const int c = tile % ct, rest = tile / ct, par = rest & 1, m0 = (rest >> 1) * TM;
      const int cq = c * 16 + q;
      const bool on = cq < nq;
      const int k = on ? cq / qpr : 0, i = on ? 4 * (cq - k * qpr) : 0;
      const float* src = a.r + (long long)k * ny * nx + i0 + i;
      float* dst = ga + (long long)k * rowz + i;
      auto ld = [&](int j) {
        float4 v = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        if (!on) return v;
        const float* p = src + (long long)j * nx;
        if (vr) return ld4(p);
        v.x = __ldcg(p);
        if (i + 1 < w) v.y = __ldcg(p + 1);
        if (i + 2 < w) v.z = __ldcg(p + 2);
        if (i + 3 < w) v.w = __ldcg(p + 3);
        return v;
      };
      auto st = [&](int m, float4 v) {
        if (on) st4(dst + (long long)m * W4, v);
      };
      if (big) dct_forward<BS, 64>(Y, par, m0, S, sg, ld, st);
      else dct_forward<BS, 32>(Y, par, m0, S, sg, ld, st);
    }
  }
  if (!team_sync(a, T)) return false;

  // ---- z forward: ga -> gb
  float* gx = ga;
  const int zq = ny * qpr, zct = (zq + 15) >> 4, zh = (nz + 1) >> 1;
  if (d3) {
    const bool big = 2u * zct * ((zh + 63) >> 6) >= nb;
    const int TM = big ? 64 : 32, mb = (zh + TM - 1) / TM, tiles = zct * mb * 2;
    for (int tile = blockIdx.x; tile < tiles; tile += nb) {
      const int c = tile % zct, rest = tile / zct, par = rest & 1, m0 = (rest >> 1) * TM;
      const int cq = c * 16 + q;
      const bool on = cq < zq;
      const float* src = ga + 4ll * cq;
      float* dst = gb + 4ll * cq;
      auto ld = [&](int k) { return on ? ld4(src + k * rowz) : make_float4(0.0f, 0.0f, 0.0f, 0.0f); };
      auto st = [&](int m, float4 v) {
        if (on) st4(dst + m * rowz, v);
      };
      if (big) dct_forward<BS, 64>(Z, par, m0, S, sg, ld, st);
      else dct_forward<BS, 32>(Z, par, m0, S, sg, ld, st);
    }
    if (!team_sync(a, T)) return false;
    gx = gb;
  }

  // ---- x solves, a warp per mode line
  {
    const int nl = ny * nz;
    const bool wall0 = i0 == 0, wall1 = i1 == nx - 1;
    for (int l = blockIdx.x * (BS / 32) + (tid >> 5); l < nl; l += nb * (BS / 32)) {
      const int p = l / ny, m = l - p * ny;
      const float aa = 1.0f + a.cy * __ldg(Y.ev + m) + (d3 ? a.cz * __ldg(Z.ev + p) : 0.0f);
      float* line = gx + (long long)l * W4;
      if (W4 <= 128) x_line<4>(line, w, W4, aa, a.cx, wall0, wall1);
      else if (W4 <= 256) x_line<8>(line, w, W4, aa, a.cx, wall0, wall1);
      else if (W4 <= 512) x_line<16>(line, w, W4, aa, a.cx, wall0, wall1);
      else x_line<32>(line, w, W4, aa, a.cx, wall0, wall1);
    }
  }
  if (!team_sync(a, T)) return false;

  // ---- z back: gb -> ga
  if (d3) {
    const bool big = (unsigned)zct * ((zh + 63) >> 6) >= nb;
    const int TM = big ? 64 : 32, mb = (zh + TM - 1) / TM, tiles = zct * mb;
    for (int tile = blockIdx.x; tile < tiles; tile += nb) {
      const int c = tile % zct, j0 = (tile / zct) * TM;
      const int cq = c * 16 + q;
      const bool on = cq < zq;
      const float* src = gb + 4ll * cq;
      float* dst = ga + 4ll * cq;
      auto ld = [&](int m) { return on ? ld4(src + m * rowz) : make_float4(0.0f, 0.0f, 0.0f, 0.0f); };
      auto st = [&](int k, float4 v) {
        if (on) st4(dst + k * rowz, v);
      };
      if (big) dct_back<BS, 64>(Z, j0, S, sg, ld, st);
      else dct_back<BS, 32>(Z, j0, S, sg, ld, st);
    }
    if (!team_sync(a, T)) return false;
  }

  // ---- y back: eta += d
  {
    const int nq = nz * qpr, ct = (nq + 15) >> 4, mh = (ny + 1) >> 1;
    const bool big = (unsigned)ct * ((mh + 63) >> 6) >= nb;
    const int TM = big ? 64 : 32, mb = (mh + TM - 1) / TM, tiles = ct * mb;
    for (int tile = blockIdx.x; tile < tiles; tile += nb) {
      const int c = tile % ct, j0 = (tile / ct) * TM;
      const int cq = c * 16 + q;
      const bool on = cq < nq;
      const int k = on ? cq / qpr : 0, i = on ? 4 * (cq - k * qpr) : 0;
      const float* src = ga + (long long)k * rowz + i;
      float* dst = a.eta + (long long)k * ny * nx + i0 + i;
      auto ld = [&](int m) { return on ? ld4(src + (long long)m * W4) : make_float4(0.0f, 0.0f, 0.0f, 0.0f); };
      auto st = [&](int j, float4 v) {
        if (!on) return;
        float* p = dst + (long long)j * nx;
        if (vr) {
          const float4 e = ld4(p);
          st4(p, make_float4(e.x + v.x, e.y + v.y, e.z + v.z, e.w + v.w));
          return;
        }
        p[0] = __ldcg(p) + v.x;
        if (i + 1 < w) p[1] = __ldcg(p + 1) + v.y;
        if (i + 2 < w) p[2] = __ldcg(p + 2) + v.z;
        if (i + 3 < w) p[3] = __ldcg(p + 3) + v.w;
      };
      if (big) dct_back<BS, 64>(Y, j0, S, sg, ld, st);
      else dct_back<BS, 32>(Y, j0, S, sg, ld, st);
    }
  }
  return true;
}

// Times, in ns, of correcting a 3D prediction by the direct solve on a slab of w
// columns, and by CG on a box of w columns and the given rows.  CG is faster on
// wide cross sections, whose dense transforms cost ny + nz multiply-adds for every
// cell of the slab, when cells couple weakly, so that few iterations are enough
// (in 2D the transforms never cost what CG's barriers do).  Fitted to (eta a step,
// direct / CG, us; h in um, 256 x n x n primed ducts):
//   h 1.5   n 128: 78 / 375   256: 258 / 375   320: 465 / 386   384: 667 / 421   (128 x 512 x 512: 1306 / 322)
//   h 3.0   n 128: 55 / 115   192:  94 / 104   256: 161 / 118   320: 276 / 116
//   h 0.75  n 128: 152 / 1342                  256: 573 / 5209  320: 1153 / 8312
// CG takes 0.6 of its bound, sqrt(condition) / 2 ln(2 max|r| / stop) iterations,
// each of two barriers and a pass over the box.
constexpr float CG_START_NS = 4.0e4f, CG_ITER_NS = 6.0e4f;
__device__ __forceinline__ float direct_ns(const EtaArgs& a, int w) {
  auto dense = [](int n) {  // multiply-adds a cell along an axis of n, whole tiles counted
    const int half = (n + 1) >> 1;
    return n > 1 ? 4.0f * (float)((half + 31) & ~31) * (float)((half + 63) & ~63) / (float)n : 0.0f;
  };
  return 3.0e4f + (float)w * (float)a.g.ny * (float)a.g.nz * (dense(a.g.ny) + dense(a.g.nz)) / 1.7e4f;
}
__device__ __forceinline__ float box_cg_ns(const EtaArgs& a, float rmax, float stop, int w, int rows) {
  const float its = fmaxf(0.3f * sqrtf(1.0f + 4.0f * (a.cx + a.cy + a.cz)) * logf(2.0f * rmax / stop), 1.0f);
  return CG_START_NS + its * (CG_ITER_NS + 0.018f * (float)w * (float)rows * (float)a.g.nz);
}

// Bound of a direct solve's error, relative to max |r|: 5e-7 measured on axes
// of 512 cells, 3e-7 up to 256.
constexpr float DCT_ERR = 1e-6f;

// One eta solve by every block of the team (of BS threads): from the fused
// step's prediction or from the eta passed in, direct or iterated.  The direct
// solve repeats until max |eta - eta_exact|, by its error bound, is within the
// stopping rule's max(tol max theta_B, atol), at most maxit times or until the
// residual stops falling (the rounding of eta itself).  solved:
// whether the prediction was not just accepted.  Returns false if a grid
// barrier gave up.  FLAT: for 2D meshes alone.
template <int BS, bool FLAT = false>
__device__ __forceinline__ bool eta_solve_team(const EtaArgs& a, DctSm& S, Team& T, EtaOut& o, bool& solved) {
  const int nx = a.g.nx;
  const bool v4 = (nx & 3) == 0 && (a.g.pitch & 3) == 0 && al16(a.c) && al16(a.eta) && al16(a.r) && al16(a.p) &&
                  al16(a.q) && al16(a.p2);
  solved = false;
  float rmax, bmax;
  double s_rr = 0.0;
  if (a.predicted && prediction_accepted(a, rmax, bmax)) return true;
  bool ok = true, iterate = false;
  float last = 0.0f;  // max |r| before the solve before
  for (int pass = 0;; ++pass) {
    if (pass || !a.predicted) ok = residual_reduce<BS>(a, T, v4, s_rr, bmax, rmax);
    const float stop = fmaxf(a.tol * bmax, a.atol);
    if (!ok || !(bmax > a.eta_t)) break;
    if (a.maxit <= pass || (pass == 0 && rmax <= stop)) break;
    if (pass && !(rmax < 0.5f * last)) break;  // down to the residual's own rounding
    last = rmax;
    int i0 = 0, i1 = nx - 1;
    if (a.predicted && pass == 0 && rmax < 3.0e38f) {
      const float thr = 0.5f * stop / (1.0f + a.cx);
      const int ntx = (nx + 31) >> 5;
      int lo = ntx, hi = -1;
      for (int t = threadIdx.x & 31; t < a.tiles; t += 32)
        if (__uint_as_float(__ldcg(a.maxw + 2 + t)) > thr) {
          lo = min(lo, t % ntx);
          hi = max(hi, t % ntx);
        }
      lo = __reduce_min_sync(0xffffffffu, lo);
      hi = __reduce_max_sync(0xffffffffu, hi);
      if (hi >= 0) {
        const int mx = box_margin(a.cx, rmax, stop);
        i0 = max(32 * lo - mx, 0) & ~3;
        i1 = min((32 * hi + 31 + mx) | 3, nx - 1);  // whole quads where nx has them
        const float direct = !FLAT && a.g.dim == 3 ? direct_ns(a, i1 - i0 + 1) : 0.0f;
        if (direct > CG_START_NS + CG_ITER_NS) {
          int ylo = a.g.ny, yhi = -1;
          for (int t = threadIdx.x & 31; t < a.tiles; t += 32)
            if (__uint_as_float(__ldcg(a.maxw + 2 + t)) > thr) {
              ylo = min(ylo, t / ntx);
              yhi = max(yhi, t / ntx);
            }
          const int my = box_margin(a.cy, rmax, stop);
          ylo = max(8 * __reduce_min_sync(0xffffffffu, ylo) - my, 0);
          yhi = min(8 * __reduce_max_sync(0xffffffffu, yhi) + 7 + my, a.g.ny - 1);
          if ((iterate = box_cg_ns(a, rmax, stop, i1 - i0 + 1, yhi - ylo + 1) < direct)) break;
        }
      }
    }
    ok = dct_solve<BS>(a, S, i0, i1, T);
    o.it = pass + 1;
    o.sync = true;
    if (pass == 0) o.box = (i0 > 0 || i1 < nx - 1) ? 1 : 0;
    // The solve leaves an error of its roundings, below DCT_ERR of max |d|, and
    // max |d| <= max |r|: another one on the new residual where that may exceed
    // the rule's bound (starts far from the solution, tight tolerances), and
    // for a whole-field start on long axes, where the roundings are largest.
    const bool fine = a.predicted || pass || max(a.g.ny, a.g.nz) <= 256;
    if (!ok || (fine && DCT_ERR * rmax <= stop)) break;
    if (!(ok = team_sync(a, T))) break;
  }
  if (ok && (iterate || !(bmax > a.eta_t))) ok = eta_iterate<BS>(a, T, v4, a.predicted != 0, s_rr, rmax, bmax, o);
  solved = true;
  return ok;
}

}  // namespace clot
