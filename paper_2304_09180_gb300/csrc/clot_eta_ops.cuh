// clot_eta_ops.cuh -- the operator of App. A, Eq. eta, and the cell loops its
// solvers share (clot_eta.cu: conjugate gradients, clot_eta_dct.cu: direct).
#pragma once

#include "clot_internal.cuh"

namespace clot {

__device__ __forceinline__ unsigned long long now_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// y = (I - cL lap) x at cell P = (i, j, k) with zero-flux boundaries (missing
// neighbours contribute nothing).  x is read through L2 (__ldcg): it changes
// between phases of the same launch, so the non-coherent path must not be used.
__device__ __forceinline__ float apply_op(const EtaArgs& a, const float* x, long long P, int i, int j, int k) {
  const int nx = a.g.nx, ny = a.g.ny, nz = a.g.nz;
  const float xp = __ldcg(x + P);
  float lx = 0.0f, ly = 0.0f, lz = 0.0f;
  if (i > 0) lx += __ldcg(x + P - 1) - xp;
  if (i < nx - 1) lx += __ldcg(x + P + 1) - xp;
  if (j > 0) ly += __ldcg(x + P - nx) - xp;
  if (j < ny - 1) ly += __ldcg(x + P + nx) - xp;
  if (a.g.dim == 3) {
    const long long sz = (long long)nx * ny;
    if (k > 0) lz += __ldcg(x + P - sz) - xp;
    if (k < nz - 1) lz += __ldcg(x + P + sz) - xp;
  }
  return xp - (a.cx * lx + a.cy * ly + a.cz * lz);
}

// The blocks of a launch that take part in a solve (blocks 0 .. nb - 1), the
// arrivals counted at their grid barrier and the half of the partials in use.
struct Team {
  int nb;
  unsigned target;
  int half;
  bool shrink;  // blocks that a solve does not need may leave the launch
};

// Grid barrier of the team: one arrival per block, whose first thread polls.
// Waits are bounded (wait_ns of globaltimer, by default that of the eta solves):
// a block that gives up sets ST_TIMEOUT and gets false in all its threads; it
// never arrives again, so every other block's next wait runs out in turn.
__device__ __forceinline__ bool team_sync(const EtaArgs& a, Team& T, unsigned long long wait_ns) {
  __shared__ int ok;
  T.target += (unsigned)T.nb;
  __syncthreads();
  if (threadIdx.x == 0) {
    ok = 1;
    asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(a.bar) : "memory");
    unsigned long long t0 = 0;
    for (;;) {
      unsigned v;
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(a.bar) : "memory");
      if ((int)(v - T.target) >= 0) break;
      const unsigned long long t = now_ns();
      if (t0 == 0) {
        t0 = t;
      } else if (t - t0 > wait_ns) {
        atomicOr(a.status, ST_TIMEOUT);
        ok = 0;
        break;
      }
    }
  }
  __syncthreads();
  return ok != 0;
}
__device__ __forceinline__ bool team_sync(const EtaArgs& a, Team& T) { return team_sync(a, T, a.wait_ns); }

// Barrier with a reduction over the team: NS sums s[] and one maximum m (of
// values >= 0).  Every block writes its partial values before it arrives; after
// the barrier every warp combines all blocks' by itself, lane l blocks l,
// l + 32, ..., then a fixed tree: all threads of all blocks get the same bits,
// on every run, without another block barrier.  The partials alternate between
// two halves, so that no block overwrites values another still reads.
// Per-thread values arrive in FP32; block and grid sums are FP64.
template <int BS, int NS>
__device__ __forceinline__ bool team_reduce(const EtaArgs& a, Team& T, const float (&x)[NS], float m, double (&s)[NS],
                                            float& smax) {
  __shared__ double sh[NS][BS / 32];
  __shared__ float shm[BS / 32];
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  double v[NS];
#pragma unroll
  for (int n = 0; n < NS; ++n) {
    v[n] = x[n];
    for (int o = 16; o > 0; o >>= 1) v[n] += __shfl_xor_sync(0xffffffffu, v[n], o);
  }
  m = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(m)));
  if (l == 0) {
#pragma unroll
    for (int n = 0; n < NS; ++n) sh[n][w] = v[n];
    shm[w] = m;
  }
  double* part = a.partials + 3ll * gridDim.x * T.half;
  T.half ^= 1;
  __syncthreads();
  if (threadIdx.x == 0) {
#pragma unroll
    for (int n = 0; n < NS; ++n) {
      for (int q = 1; q < BS / 32; ++q) v[n] += sh[n][q];
      part[n * gridDim.x + blockIdx.x] = v[n];
    }
    for (int q = 1; q < BS / 32; ++q) m = fmaxf(m, shm[q]);
    part[2 * gridDim.x + blockIdx.x] = (double)m;
  }
  if (!team_sync(a, T)) return false;
#pragma unroll
  for (int n = 0; n < NS; ++n) s[n] = 0.0;
  float g = 0.0f;
  for (int q = l; q < T.nb; q += 32) {
#pragma unroll
    for (int n = 0; n < NS; ++n) s[n] += __ldcg(part + n * gridDim.x + q);
    g = fmaxf(g, (float)__ldcg(part + 2 * gridDim.x + q));
  }
#pragma unroll
  for (int n = 0; n < NS; ++n)
    for (int o = 16; o > 0; o >>= 1) s[n] += __shfl_xor_sync(0xffffffffu, s[n], o);
  smax = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(g)));
  return true;
}

// Visit every cell once: each warp takes 32-cell chunks of x rows (one
// integer division per chunk, coalesced along x).
template <class Fn>
__device__ __forceinline__ void for_cells(const EtaArgs& a, int nb, Fn fn) {
  const int nx = a.g.nx, ny = a.g.ny;
  const int lane = threadIdx.x & 31;
  const int warp = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5);
  const int nwarps = (int)((nb * blockDim.x) >> 5);
  const int cprw = (nx + 31) >> 5;
  const int nch = ny * a.g.nz * cprw;
  for (int ch = warp; ch < nch; ch += nwarps) {
    const int xc = ch % cprw, r = ch / cprw;
    const int j = r % ny, k = r / ny;
    const int i = xc * 32 + lane;
    if (i < nx) fn((long long)i + (long long)nx * r, i, j, k);
  }
}

// Quads: four x-consecutive cells, moved as one float4 (needs nx % 4 == 0 and
// 16-byte aligned vectors).  Thread t takes quads t, t + T, ...: a warp reads
// 512 contiguous bytes per vector, and every thread has four cells' loads in
// flight at once -- the scalar passes are bound by memory latency, not by
// bandwidth.
__device__ __forceinline__ bool al16(const void* p) { return ((unsigned long long)p & 15u) == 0; }
__device__ __forceinline__ float4 ld4(const float* p) { return __ldcg(reinterpret_cast<const float4*>(p)); }
__device__ __forceinline__ void st4(float* p, float4 v) { *reinterpret_cast<float4*>(p) = v; }

template <class Fn>
__device__ __forceinline__ void for_quads(const EtaArgs& a, int nb, Fn fn) {
  const unsigned nqx = (unsigned)a.g.nx >> 2, ny = (unsigned)a.g.ny;
  const unsigned nq = (unsigned)(a.g.ncell >> 2);
  const unsigned T = nb * blockDim.x;
  for (unsigned qd = blockIdx.x * blockDim.x + threadIdx.x; qd < nq; qd += T) {
    const unsigned row = qd / nqx;
    fn(4ll * qd, (int)(4u * (qd - row * nqx)), (int)(row % ny), (int)(row / ny));
  }
}

// for_quads, two quads at a time: load(P, i, j, k) reads and computes, use(P,
// i, j, k, v) stores or accumulates.  Both quads' loads are in flight before
// either is used, which the blocks of the direct solver (384 threads an SM)
// need to keep a large mesh's passes off the memory latency.
template <class Load, class Use>
__device__ __forceinline__ void for_quads2(const EtaArgs& a, int nb, Load load, Use use) {
  const unsigned nqx = (unsigned)a.g.nx >> 2, ny = (unsigned)a.g.ny;
  const unsigned nq = (unsigned)(a.g.ncell >> 2);
  const unsigned T = nb * blockDim.x;
  for (unsigned qd = blockIdx.x * blockDim.x + threadIdx.x; qd < nq; qd += 2 * T) {
    const unsigned q2 = qd + T < nq ? qd + T : qd;
    const unsigned r1 = qd / nqx, r2 = q2 / nqx;
    const int i1 = (int)(4u * (qd - r1 * nqx)), j1 = (int)(r1 % ny), k1 = (int)(r1 / ny);
    const int i2 = (int)(4u * (q2 - r2 * nqx)), j2 = (int)(r2 % ny), k2 = (int)(r2 / ny);
    const auto v1 = load(4ll * qd, i1, j1, k1);
    const auto v2 = load(4ll * q2, i2, j2, k2);
    use(4ll * qd, i1, j1, k1, v1);
    if (q2 != qd) use(4ll * q2, i2, j2, k2, v2);
  }
}

// x - (cx lx + cy ly + cz lz) for the quad at P = (i..i+3, j, k), zero-flux
// walls, with the field given by a quad loader v4 and a single-cell loader v1;
// the same per-cell expression as apply_op.  Returns the quad's own values in x.
template <class V4, class V1>
__device__ __forceinline__ float4 quad_op(const EtaArgs& a, long long P, int i, int j, int k, V4 v4, V1 v1,
                                          float4& x) {
  const int nx = a.g.nx, ny = a.g.ny, nz = a.g.nz;
  x = v4(P);
  float lx[4], ly[4] = {0.0f, 0.0f, 0.0f, 0.0f}, lz[4] = {0.0f, 0.0f, 0.0f, 0.0f};
  const float c[4] = {x.x, x.y, x.z, x.w};
  lx[0] = (i > 0) ? (v1(P - 1) - c[0]) + (c[1] - c[0]) : (c[1] - c[0]);
  lx[1] = (c[0] - c[1]) + (c[2] - c[1]);
  lx[2] = (c[1] - c[2]) + (c[3] - c[2]);
  lx[3] = (i + 4 < nx) ? (c[2] - c[3]) + (v1(P + 4) - c[3]) : (c[2] - c[3]);
  if (j > 0) {
    const float4 d = v4(P - nx);
    ly[0] = d.x - c[0]; ly[1] = d.y - c[1]; ly[2] = d.z - c[2]; ly[3] = d.w - c[3];
  }
  if (j < ny - 1) {
    const float4 u = v4(P + nx);
    ly[0] += u.x - c[0]; ly[1] += u.y - c[1]; ly[2] += u.z - c[2]; ly[3] += u.w - c[3];
  }
  if (a.g.dim == 3) {
    const long long sz = (long long)nx * ny;
    if (k > 0) {
      const float4 d = v4(P - sz);
      lz[0] = d.x - c[0]; lz[1] = d.y - c[1]; lz[2] = d.z - c[2]; lz[3] = d.w - c[3];
    }
    if (k < nz - 1) {
      const float4 u = v4(P + sz);
      lz[0] += u.x - c[0]; lz[1] += u.y - c[1]; lz[2] += u.z - c[2]; lz[3] += u.w - c[3];
    }
  }
  float q[4];
#pragma unroll
  for (int m = 0; m < 4; ++m) q[m] = c[m] - (a.cx * lx[m] + a.cy * ly[m] + a.cz * lz[m]);
  return make_float4(q[0], q[1], q[2], q[3]);
}

// for_cells restricted to a box (32-cell chunks along x inside the box), four
// chunks at a time: load(P, i, j, k), then use(P, v), as in for_quads2.
template <class Load, class Use>
__device__ __forceinline__ void for_box_cells(const EtaArgs& a, int nb, const Box& b, Load load, Use use) {
  constexpr int U = 4;
  const int nx = a.g.nx, ny = a.g.ny;
  const int lane = threadIdx.x & 31;
  const int warp = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5);
  const int nwarps = (int)((nb * blockDim.x) >> 5);
  const int bnx = b.i1 - b.i0 + 1, bny = b.j1 - b.j0 + 1;
  const int cprw = (bnx + 31) >> 5;
  const int nch = cprw * bny * (b.k1 - b.k0 + 1);
  for (int ch = warp; ch < nch; ch += U * nwarps) {
    decltype(load(0ll, 0, 0, 0)) v[U];
    long long P[U];
    bool on[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int c = ch + u * nwarps, xc = c % cprw, r = c / cprw;
      const int j = b.j0 + r % bny, k = b.k0 + r / bny, i = b.i0 + xc * 32 + lane;
      on[u] = c < nch && i <= b.i1;
      P[u] = (long long)i + (long long)nx * (j + (long long)ny * k);
      if (on[u]) v[u] = load(P[u], i, j, k);
    }
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (on[u]) use(P[u], v[u]);
  }
}

}  // namespace clot
