// clot_step_zmarch.cu -- K1 on 3D meshes: the fused species step (Sec. 3.2)
// marching in z through planes staged in shared memory.
//
// A block owns a 32 x 8 tile column of the mesh and a run of planes (zm_run);
// its 256 threads hold one cell each per plane.  Data movement per plane:
//   - the nine species that neighbours read (P^{m,u}, P^{m,a}, P^{b,a},
//     P^{b,se}, ADP, S1, S2, E1, E2), with a halo of 4 cells in x (so that the
//     box starts on a 16-byte boundary) and 2 in y, arrive by one 4D TMA tile
//     load (40 x 12 x 1 x 9 floats; cells outside the mesh read as zero), eta
//     and eta of the previous step by 3D loads, into a ring of four
//     shared-memory planes completing on mbarriers (waits bounded by
//     %globaltimer).  Rows that are not 16-byte multiples are staged by
//     asynchronous copies of one or two floats instead.  The load of plane
//     k + 3 is issued while plane k computes, so planes k, k + 1, k + 2 are
//     resident;
//   - the six species only the cell itself reads and sigma are per-thread
//     loads issued before the wait for the plane's tile; the face fluxes, which
//     the plane needs first, are loaded a plane ahead (337 -> 332 us on the
//     duct; staging all of them a plane ahead by asynchronous copies: 349);
//   - results go out as coalesced stores (a warp writes 128 contiguous bytes
//     per species row).  Staging them in the ring slot of the plane just
//     computed and writing them by bulk tensor stores was measured slower
//     (the slot's refill must then wait for the store to read it).
// Compute per plane, with two block barriers (plane landed; faces published):
//   - the x and y face fluxes of every cell's low faces, exchanged through
//     shared memory; the high faces of the tile's last column and row are
//     spread over the warps, a species each (one warp taking all of them kept
//     the block waiting: 353 -> 338 us plasma, 494 -> 457 primed); the z
//     face above each cell from the own column (the face below is carried
//     from the plane underneath), so every face is computed once.  At the ends
//     of the mesh the staged tile holds copies one cell outwards, so that no
//     face tests its range;
//   - W(theta_T) of the staged tile of plane k + 1 (two cells per thread, no
//     bounds tests: cells outside the mesh are never read through W) for the
//     next plane, and whether plane k + 2 holds any of the four species plain
//     plasma lacks (P^{m,a}, ADP, E1, E2), OR-ing their bit patterns; both
//     ride on the barrier that publishes the faces;
//   - a plane transports those four species only if one of them is present in
//     planes k - 1 .. k + 1 (the fluxes of an absent species are then exactly
//     zero: van Leer returns the upwind value when the two cells of a face are
//     equal).  The species set is a template parameter, so the face code runs
//     without per-species branches;
//   - the shared epilogue (clot_cell.cuh: transport update, optional Heun
//     average and lagged wall, M_rxn RK4 reaction with the injury-wall
//     exchange) and the eta prediction for the next step.
// What bounds it: instruction issue and dependency latency at the 16 warps an
// SM holds (registers and the ring both allow two blocks), not HBM: 332 us on
// the 512 x 128 x 128 plasma duct where its 140 B a cell take 173.  Compiling
// the options out of the usual call (PLAIN) took 384 -> 353 us plasma and
// 546 -> 494 primed: the plane loop's code then fits the instruction cache better.
// Model: fractional step of Sec. 3.2; hindered platelet fluxes (Sec. 3.2),
// van Leer face values and Gauss-linear diffusion (App. D); boundary table of
// App. C; reaction terms of App. A and App. B.
#include <algorithm>

#include "clot_cell.cuh"
#include "clot_tma.cuh"

namespace clot {
namespace {

constexpr int TX = 32, TY = 8, TNT = TX * TY;
constexpr int HXT = 4, HYT = 2;
constexpr int SXT = TX + 2 * HXT;  // 40
constexpr int SYT = TY + 2 * HYT;  // 12
constexpr int SPT = SXT * SYT;     // 480 staged cells
constexpr int NSTG = 9;            // staged species rows 0 .. 8
constexpr int RING = 4;
constexpr int MAXRUN = 12;         // most planes per block

struct alignas(128) ZPlane {
  float c[NSTG][SPT];  // 17280 B
  float eta[SPT];
  float etp[SPT];
};
struct ZSm {
  ZPlane buf[RING];
  float W[2][SPT];  // hindrance of the staged tile of plane k and of plane k + 1
  float xf[NT][TY][TX + 1];
  float yf[NT][TY + 1][TX];
  float red[2][TNT / 32];
  unsigned long long bar[RING];
};
static_assert(sizeof(ZPlane) % 128 == 0, "ring planes must stay 128-byte aligned");
static_assert(SPT % 2 == 0 && SPT / 2 <= TNT, "the hindrance pass gives each thread at most one pair");

// Species sets of the face code: the three that plain plasma carries
// (P^{m,u}, S1, S2), or all seven mobile species.
constexpr int SET_PLASMA = 0, SET_ALL = 1;
__host__ __device__ constexpr bool in_set(int S, int t) { return S == SET_ALL || t == 0 || t == 3 || t == 4; }

struct ZGeo {
  int tx, ty, tid, x0, y0, gx, gy, lastx, lasty, sc;
  bool act;
};

// Bit patterns of the non-plasma species of staged pair `tid` of a plane
// (zero exactly when all of them are +0 there).
__device__ __forceinline__ unsigned nonplasma_bits(const ZPlane& B, int tid) {
  const int q = 2 * tid;
  const uint2 a = *reinterpret_cast<const uint2*>(&B.c[CLOT_PMA][q]);
  const uint2 b = *reinterpret_cast<const uint2*>(&B.c[CLOT_ADP][q]);
  const uint2 c = *reinterpret_cast<const uint2*>(&B.c[CLOT_E1][q]);
  const uint2 d = *reinterpret_cast<const uint2*>(&B.c[CLOT_E2][q]);
  return (a.x | a.y | b.x | b.y) | (c.x | c.y | d.x | d.y);
}

// Values beyond the mesh next to it, for tiles at its ends: the mobile species
// (and eta, eta of the previous step) of the first and last cells along x and y
// are copied one cell outwards, so that the face code and the eta prediction
// run without range tests (face_flux_in; a difference to a copy is zero).
__device__ __forceinline__ void zm_fill_ends(ZPlane& B, const ZGeo& G, int nx, int ny) {
  const int tid = G.tid;
  auto rowp = [&](int t) { return t < NT ? B.c[trow(t)] : t == NT ? B.eta : B.etp; };
  const int ex = nx - G.x0, ey = ny - G.y0;  // first column and row beyond the mesh, counted from the tile
  if (G.x0 == 0 || ex <= TX + 1)
    for (int q = tid; q < (NT + 2) * TY * 2; q += TNT) {
      const int hi = q & 1, y = (q >> 1) % TY;
      float* r = rowp((q >> 1) / TY) + (y + HYT) * SXT + HXT;
      if (hi && ex <= TX + 1) r[ex] = r[ex - 1];
      if (!hi && G.x0 == 0) r[-1] = r[0];
    }
  if (G.y0 == 0 || ey <= TY + 1)
    for (int q = tid; q < (NT + 2) * TX * 2; q += TNT) {
      const int x = q % TX, hi = (q / TX) & 1;
      float* r = rowp(q / (2 * TX)) + HYT * SXT + x + HXT;
      if (hi && ey <= TY + 1) r[ey * SXT] = r[(ey - 1) * SXT];
      if (!hi && G.y0 == 0) r[-SXT] = r[0];
    }
}

// x and y face fluxes of plane k for the species of set S, before the block
// barrier that publishes them: each thread's low x and y faces (kept in xlo,
// ylo and written to xf, yf), the high x face of every row's last cell and the
// high y face of the last row.  c0 receives the
// cell's mobile species (zero for species outside S, which are absent around
// this plane).  W: hindrance of the staged cells of plane k.
template <int S, bool PLAIN>
__device__ __forceinline__ void zm_xy_faces(const StepArgs& A, ZSm& Sm, const float* W, const ZPlane& B0,
                                            const ZGeo& G, int k, float WP, float fxlo, float fylo, float fend,
                                            float (&c0)[NT], float (&xlo)[NT], float (&ylo)[NT]) {
  const StepConst& K = A.K;
  const int nx = K.g.nx, ny = K.g.ny;
  const int tx = G.tx, ty = G.ty, sc = G.sc, gy = G.gy;
  const float* pl = &B0.c[0][0];
  // one face: its hindrance factors once, then the set's species
  auto face = [&](int q, int st, float F, float WL, float WH, int ax, auto put) {
    const bool adv = __any_sync(__activemask(), F != 0.0f), pos = F >= 0.0f;
    const float WaF = (pos ? WH : WL) * F, Wd = fminf(WL, WH);
#pragma unroll
    for (int t = 0; t < NT; ++t) {
      if (!in_set(S, t)) continue;
      const float* r = pl + trow(t) * SPT + q;
      const float D = K.dcoef[t][ax];
      put(t, face_flux_in(r[-2 * st], r[-st], r[0], r[st], F, pos, t < 2 ? WaF : F, t < 2 ? Wd * D : D, PLAIN || K.limiter, adv));
    }
  };
#pragma unroll
  for (int t = 0; t < NT; ++t) {
    c0[t] = in_set(S, t) ? B0.c[trow(t)][sc] : 0.0f;
    xlo[t] = ylo[t] = 0.0f;
  }
  if (!PLAIN && !K.do_transport) return;
  // the tile's end faces, a species a lane group or a warp so that no warp
  // keeps the block waiting: warp 0 the x high face of every row's last cell
  // (row lane % 8, species lane / 8), warps 1 .. the y high faces of the last row
  auto end_face = [&](int t, int q, int st, float F, float WL, float WH, int ax) {
    const bool adv = __any_sync(__activemask(), F != 0.0f), pos = F >= 0.0f;
    const float* r = pl + (t < 2 ? t : t + 2) * SPT + q;  // trow(t)
    const float D = K.dcoef[t][ax];
    return face_flux_in(r[-2 * st], r[-st], r[0], r[st], F, pos, t < 2 ? (pos ? WH : WL) * F : F,
                        t < 2 ? fminf(WL, WH) * D : D, PLAIN || K.limiter, adv);
  };
  if (ty == 0) {
    const int row = tx % TY, scl = (row + HYT) * SXT + (G.lastx + HXT);
    const float WPl = W[scl];
    if (G.y0 + row < ny) {
#pragma unroll
      for (int p = 0; p < (S == SET_ALL ? 2 : 1); ++p) {
        const int g = tx / TY + 4 * p, t = S == SET_ALL ? g : (g == 0 ? 0 : g + 2);
        if (g >= (S == SET_ALL ? NT : 3)) continue;
        float f;
        if (G.x0 + G.lastx < nx - 1)
          f = end_face(t, scl + 1, 1, fend, WPl, W[scl + 1], 0);
        else  // the outlet
          f = !PLAIN && K.closed_ends ? 0.0f : (t < 2 ? WPl : 1.0f) * fend * pl[(t < 2 ? t : t + 2) * SPT + scl];
        Sm.xf[t][row][G.lastx + 1] = f;
      }
    }
  } else if (ty <= (S == SET_ALL ? NT : 3) && G.gx < nx) {
    const int t = S == SET_ALL ? ty - 1 : (ty == 1 ? 0 : ty + 1);
    const int scl = (G.lasty + HYT) * SXT + (tx + HXT);
    float f = 0.0f;  // the top wall at y = ny
    if (G.y0 + G.lasty < ny - 1) f = end_face(t, scl + SXT, SXT, fend, W[scl], W[scl + SXT], 1);
    Sm.yf[t][G.lasty + 1][tx] = f;
  }
  if (!G.act) return;
  // x low face
  face(sc, 1, fxlo, W[sc - 1], WP, 0, [&](int t, float f) { xlo[t] = f; });
  if (G.x0 == 0 && tx == 0) {  // the inlet
#pragma unroll
    for (int t = 0; t < NT; ++t) xlo[t] = 0.0f;
    if (PLAIN || !K.closed_ends) {
      const int b = gy + ny * k;
      const float pin = __ldg(A.pmu_in + b);
      const float Wb =
          hindrance((pin + pl[CLOT_PMA * SPT + sc] + pl[CLOT_PBA * SPT + sc] + pl[CLOT_PBSE * SPT + sc]) * K.invPmax);
#pragma unroll
      for (int t = 0; t < NT; ++t) {
        if (!in_set(S, t)) continue;
        const bool hind = t < 2, dir = (t == 0 || t == 3 || t == 4);
        const float cP = c0[t];
        const float cb = !dir ? cP : (t == 0 ? pin : t == 3 ? __ldg(A.s1_in + b) : __ldg(A.s2_in + b));
        const float Fout = -fxlo;
        const float Wa = hind ? (Fout > 0.0f ? Wb : WP) : 1.0f;
        const float Wd = hind ? fminf(WP, Wb) : 1.0f;
        float out = Wa * Fout * cb;
        if (dir) out -= Wd * 2.0f * K.dcoef[t][0] * (cb - cP);
        xlo[t] = -out;
      }
    }
  }
#pragma unroll
  for (int t = 0; t < NT; ++t)
    if (in_set(S, t)) Sm.xf[t][ty][tx] = xlo[t];
  // y low face (the floor is a wall)
  if (gy > 0) face(sc, SXT, fylo, W[sc - SXT], WP, 1, [&](int t, float f) { ylo[t] = f; });
#pragma unroll
  for (int t = 0; t < NT; ++t)
    if (in_set(S, t)) Sm.yf[t][ty][tx] = ylo[t];
}

// After the block barrier: the z face above the cell (the one below is
// carried in fzlo from the plane underneath) and each cell's net outflow dv.
// Wp: W of the own column at k + 1.  B1, B2: the planes above, or the last
// plane of the mesh where there is none.
template <int S, bool PLAIN>
__device__ __forceinline__ void zm_z_faces(const StepArgs& A, const ZSm& Sm, const ZPlane& B1, const ZPlane& B2,
                                           const ZGeo& G, bool hp1, float WP, float Wp, float Fhi,
                                           const float (&cm1)[NT], const float (&c0)[NT], const float (&xlo)[NT],
                                           const float (&ylo)[NT], float (&fzlo)[NT], float (&dv)[NT]) {
  const StepConst& K = A.K;
  const int tx = G.tx, ty = G.ty, sc = G.sc;
  const bool adv = __any_sync(__activemask(), Fhi != 0.0f), pos = Fhi >= 0.0f;
  const float WaF = (pos ? Wp : WP) * Fhi, Wd = fminf(WP, Wp);
#pragma unroll
  for (int t = 0; t < NT; ++t) {
    if (!in_set(S, t)) {
      fzlo[t] = 0.0f;
      continue;
    }
    const float D = K.dcoef[t][2];
    float hi = 0.0f;
    if (hp1)
      hi = face_flux_in(cm1[t], c0[t], B1.c[trow(t)][sc], B2.c[trow(t)][sc], Fhi, pos, t < 2 ? WaF : Fhi,
                        t < 2 ? Wd * D : D, PLAIN || K.limiter, adv);
    dv[t] = (hi - fzlo[t]) + (Sm.xf[t][ty][tx + 1] - xlo[t]) + (Sm.yf[t][ty + 1][tx] - ylo[t]);
    fzlo[t] = hi;
  }
}

// W of the staged cells of a plane, two per thread (threads 0 .. SPT/2 - 1).
__device__ __forceinline__ void zm_w_pass(const ZPlane& B, float* W, int tid, float ip) {
  if (tid >= SPT / 2) return;
  const int q = 2 * tid;
  const float2 a = *reinterpret_cast<const float2*>(&B.c[CLOT_PMU][q]);
  const float2 b = *reinterpret_cast<const float2*>(&B.c[CLOT_PMA][q]);
  const float2 c = *reinterpret_cast<const float2*>(&B.c[CLOT_PBA][q]);
  const float2 d = *reinterpret_cast<const float2*>(&B.c[CLOT_PBSE][q]);
  float2 w;
  w.x = hindrance((a.x + b.x + c.x + d.x) * ip);
  w.y = hindrance((a.y + b.y + c.y + d.y) * ip);
  *reinterpret_cast<float2*>(&W[q]) = w;
}

// Block maxima of |r| and theta_B into eta_max (float bit patterns; both >= 0),
// and of |r| into the word of the block's tile column `tile` when tile >= 0.
__device__ __forceinline__ void block_max2(float rmax, float bmax, float (*red)[TNT / 32], unsigned* out, int tile, int tid) {
  for (int o = 16; o > 0; o >>= 1) {
    rmax = fmaxf(rmax, __shfl_xor_sync(0xffffffffu, rmax, o));
    bmax = fmaxf(bmax, __shfl_xor_sync(0xffffffffu, bmax, o));
  }
  if ((tid & 31) == 0) {
    red[0][tid >> 5] = rmax;
    red[1][tid >> 5] = bmax;
  }
  __syncthreads();
  if (tid == 0) {
    for (int q = 1; q < TNT / 32; ++q) {
      rmax = fmaxf(rmax, red[0][q]);
      bmax = fmaxf(bmax, red[1][q]);
    }
    if (rmax > 0.0f) {
      atomicMax(out, __float_as_uint(rmax));
      if (tile >= 0) atomicMax(out + 2 + tile, __float_as_uint(rmax));
    }
    if (bmax > 0.0f) atomicMax(out + 1, __float_as_uint(bmax));
  }
}

// Staging of a plane without the tensor memory accelerator (rows that are not
// 16-byte multiples): asynchronous copies of V floats, issued by every thread;
// cells outside the mesh read as zero.
template <int V>
__device__ __forceinline__ void zm_copy_plane(const StepArgs& A, ZPlane& B, const ZGeo& G, int k, bool eta, bool etp) {
  constexpr int CPR = (TX + 4) / V;  // the tile with two cells on either side
  const int nx = A.K.g.nx, ny = A.K.g.ny;
  const long long pitch = A.K.g.pitch;
  const unsigned dst0 = smem_u32(&B.c[0][0]);
  for (int q = G.tid; q < SYT * CPR; q += TNT) {
    const int y = q / CPR, x = (q - y * CPR) * V - 2;
    const int gx = G.x0 + x, gy = G.y0 - HYT + y;
    const bool in = gx >= 0 && gx < nx && gy >= 0 && gy < ny;  // nx and gx are multiples of V
    const long long go = in ? (long long)gx + (long long)nx * (gy + (long long)ny * k) : 0;
    const unsigned so = dst0 + 4u * (unsigned)(y * SXT + x + HXT);
    auto copy = [&](unsigned d, const float* s) {
      asm volatile("cp.async.ca.shared.global [%0], [%1], %2, %3;\n" ::"r"(d), "l"(s), "n"(4 * V), "r"(in ? 4 * V : 0)
                   : "memory");
    };
#pragma unroll
    for (int r = 0; r < NSTG; ++r) copy(so + 4u * r * SPT, A.cin + r * pitch + go);
    if (eta) copy(so + 4u * NSTG * SPT, A.eta + go);
    if (etp) copy(so + 4u * (NSTG + 1) * SPT, A.eta_prev + go);
  }
}

// LD: 0 stages planes by TMA, 1 and 2 by copies of that many floats.  IDX:
// unsigned (byte offsets, row_at) where the mesh has fewer than 2^30 cells.
template <int LD, bool EXT, typename IDX, bool PLAIN>
__global__ void __launch_bounds__(TNT, 2)
    zmarch_step_kernel(const StepArgs A, const __grid_constant__ CUtensorMap tm_c,
                       const __grid_constant__ CUtensorMap tm_eta, const __grid_constant__ CUtensorMap tm_etp, int run) {
  extern __shared__ unsigned char smraw[];
  ZSm& Sm = *reinterpret_cast<ZSm*>(smraw + ((128u - (smem_u32(smraw) & 127u)) & 127u));
  const StepConst& K = A.K;
  const int nx = K.g.nx, ny = K.g.ny, nz = K.g.nz;
  ZGeo G;
  G.tx = threadIdx.x;
  G.ty = threadIdx.y;
  G.tid = G.ty * TX + G.tx;
  G.x0 = blockIdx.x * TX;
  G.y0 = blockIdx.y * TY;
  G.gx = G.x0 + G.tx;
  G.gy = G.y0 + G.ty;
  G.act = G.gx < nx && G.gy < ny;
  G.lastx = min(TX - 1, nx - 1 - G.x0);
  G.lasty = min(TY - 1, ny - 1 - G.y0);
  G.sc = (G.ty + HYT) * SXT + (G.tx + HXT);
  const int tid = G.tid, sc = G.sc;
  const long long pitch = K.g.pitch, sxy = (long long)nx * ny;
  const float ip = K.invPmax;
  const int kb = blockIdx.z * run, ke = min(kb + run, nz);
  const bool predict = PLAIN || A.predict, transport = PLAIN || K.do_transport;
  const bool need_eta = PLAIN || K.do_reaction || predict;
  const bool ends = G.x0 == 0 || nx - G.x0 <= TX + 1 || G.y0 == 0 || ny - G.y0 <= TY + 1;
  const bool overx = G.gx >= K.g.i0 && G.gx <= K.g.i1;
  const long long P0 = (long long)G.gx + (long long)nx * G.gy;
  const unsigned bytes = (unsigned)(sizeof(float) * SPT * (NSTG + (need_eta ? 1 : 0) + (predict ? 1 : 0)));

  if (LD == 0) {
    if (tid == 0) {
      for (int b = 0; b < RING; ++b) mbar_init(&Sm.bar[b], 1);
      asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    }
  } else {  // the columns the copies leave out
    for (int q = tid; q < RING * (int)(sizeof(ZPlane) / 16); q += TNT)
      reinterpret_cast<float4*>(Sm.buf)[q] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
  }
  __syncthreads();

  auto planned = [&](int k) { return k < nz && k <= ke + 1; };
  auto issue = [&](int k) {  // thread 0: arm the plane's ring slot and start its tile loads
    if (LD != 0) {
      if (planned(k)) zm_copy_plane<LD == 0 ? 1 : LD>(A, Sm.buf[(k - kb) % RING], G, k, need_eta, predict);
      asm volatile("cp.async.commit_group;\n" ::: "memory");  // a group a plane, empty or not
      return;
    }
    if (tid != 0 || !planned(k)) return;
    const int b = (k - kb) % RING;
    ZPlane& B = Sm.buf[b];
    fence_proxy_async_smem();  // earlier reads of the slot before its refill
    mbar_expect_tx(&Sm.bar[b], bytes);
    const int x = G.x0 - HXT, y = G.y0 - HYT;
    tma_load_4d(&B.c[0][0], &tm_c, x, y, k, 0, &Sm.bar[b]);
    if (need_eta) tma_load_3d(B.eta, &tm_eta, x, y, k, &Sm.bar[b]);
    if (predict) tma_load_3d(B.etp, &tm_etp, x, y, k, &Sm.bar[b]);
  };
  // all threads wait for plane k's loads; the block leaves together on a
  // timeout.  `later`: planes issued after it
  auto landed = [&](int k, int later) -> bool {
    if (LD != 0) {
      if (later == 0) asm volatile("cp.async.wait_group 0;\n" ::: "memory");
      else asm volatile("cp.async.wait_group 1;\n" ::: "memory");
      __syncthreads();
      return true;
    }
    bool ok = true;
    if (planned(k)) ok = mbar_wait_bounded(&Sm.bar[(k - kb) % RING], (unsigned)(((k - kb) / RING) & 1));
    const bool all = __syncthreads_and(ok) != 0;
    if (!all && tid == 0 && A.status) atomicOr(A.status, ST_TIMEOUT);
    return all;
  };
  // after a timeout: thread 0 waits (bounded) for the loads still in flight
  // into the ring, so that none lands after the block has left
  auto drain = [&](int from, int to) {
    if (tid != 0) return;
    for (int q = from; q <= to; ++q)
      if (planned(q)) mbar_wait_bounded(&Sm.bar[(q - kb) % RING], (unsigned)(((q - kb) / RING) & 1));
  };
  issue(kb);
  issue(kb + 1);
  issue(kb + 2);
  int issued = kb + 2;

  // own column below the run: mobile species at kb - 1 (and kb - 2 for the
  // face below the first plane), W and the eta guess at kb - 1
  float cm1[NT], fzlo[NT];
  float Wm1 = 0.0f, gm1 = 0.0f;
  unsigned pre = 0u;
  float cm2[NT];
#pragma unroll
  for (int t = 0; t < NT; ++t) cm1[t] = cm2[t] = fzlo[t] = 0.0f;
  float Flo = 0.0f;
  if (G.act && kb >= 1) {
    const long long Q = P0 + (long long)(kb - 1) * sxy;
#pragma unroll
    for (int t = 0; t < NT; ++t) {
      cm1[t] = __ldg(A.cin + (long long)trow(t) * pitch + Q);
      if (kb >= 2) cm2[t] = __ldg(A.cin + (long long)trow(t) * pitch + Q - sxy);
      if (!in_set(SET_PLASMA, t)) pre |= __float_as_uint(cm1[t]);
    }
    Wm1 = hindrance((cm1[0] + cm1[1] + __ldg(A.cin + CLOT_PBA * pitch + Q) + __ldg(A.cin + CLOT_PBSE * pitch + Q)) *
                    ip);
    if (predict) gm1 = 2.0f * __ldg(A.eta + Q) - __ldg(A.eta_prev + Q);
    if (transport) Flo = __ldg(A.fz + Q + sxy);
  }
  // lastp: the highest plane (up to k + 1 at plane k) known to hold a
  // non-plasma species; plane k transports only the plasma species when
  // none of planes k - 1, k, k + 1 holds one (the fluxes of an absent species
  // through the faces of plane k are exactly zero when it is absent from the
  // staged tile and from the own column one plane down and up)
  int lastp = -(1 << 29);
  if (__syncthreads_or(pre != 0u)) lastp = kb - 1;
  if (!landed(kb, 2)) { drain(kb, issued); return; }
  if (!landed(kb + 1, 1)) { drain(kb + 1, issued); return; }
  zm_w_pass(Sm.buf[0], Sm.W[0], tid, ip);
  if (__syncthreads_or(tid < SPT / 2 && nonplasma_bits(Sm.buf[0], tid) != 0u)) lastp = kb;
  if (planned(kb + 1) && __syncthreads_or(tid < SPT / 2 && nonplasma_bits(Sm.buf[1], tid) != 0u)) lastp = kb + 1;
  if (ends) zm_fill_ends(Sm.buf[0], G, nx, ny);  // published by the first barrier of the plane loop
  // flux through the face below the first plane, for every mobile species
  if (G.act && transport && kb >= 1) {
    const ZPlane& B0 = Sm.buf[0];
    const ZPlane& B1 = Sm.buf[1];
    const bool hm2 = kb >= 2, hp1 = kb + 1 < nz;
    const bool advlo = __any_sync(__activemask(), Flo != 0.0f);
    const float WP0 = Sm.W[0][sc];
#pragma unroll
    for (int t = 0; t < NT; ++t) {
      const float c0 = B0.c[trow(t)][sc];
      const float cp1 = hp1 ? B1.c[trow(t)][sc] : c0;
      fzlo[t] = face_flux(hm2 ? cm2[t] : cm1[t], cm1[t], c0, cp1, hm2, hp1, Flo, Wm1, WP0, t < 2, K.dcoef[t][2],
                          K.limiter, advlo);
    }
  }
  float rmax = 0.0f, bmax = 0.0f;
  int wsel = 0;
  constexpr IDX E = sizeof(IDX) == 4 ? 4 : 1;  // offsets of row_at
  const IDX fx0 = E * ((IDX)G.gx + (IDX)(nx + 1) * G.gy), fy0 = E * (IDX)P0;
  const IDX fxe = E * ((IDX)(G.x0 + G.lastx + 1) + (IDX)(nx + 1) * (G.y0 + G.tx % TY));
  const IDX fye = E * ((IDX)G.gx + (IDX)nx * (G.y0 + G.lasty + 1));

  auto end_flux = [&](int k) {  // the flux of the end face this thread takes (zm_xy_faces)
    float f = 0.0f;
    if (!transport) return f;
    if (G.ty == 0) {
      if (G.y0 + G.tx % TY < ny) f = __ldg(&row_at(A.fx, k, (long long)(nx + 1) * ny, fxe));
    } else if (G.gx < nx && G.y0 + G.lasty < ny - 1) {
      f = __ldg(&row_at(A.fy, k, (long long)nx * (ny + 1), fye));
    }
    return f;
  };
  float fend1 = end_flux(kb), fx1 = 0.0f, fy1 = 0.0f, fz1 = 0.0f;
  auto own_flux = [&](int k) {
    if (!transport || !G.act) return;
    fx1 = __ldg(&row_at(A.fx, k, (long long)(nx + 1) * ny, fx0));
    if (G.gy > 0) fy1 = __ldg(&row_at(A.fy, k, (long long)nx * (ny + 1), fy0));
    fz1 = k + 1 < nz ? __ldg(&row_at(A.fz, 1, sxy, E * (IDX)(P0 + (long long)k * sxy))) : 0.0f;
  };
  own_flux(kb);

  for (int k = kb; k < ke; ++k) {
    const IDX P = E * (IDX)(P0 + (long long)k * sxy);
    const bool hp1 = k + 1 < nz;
    // per-thread values of plane k, issued before the wait for the plane's
    // tile and in flight through it and the hindrance pass
    float yb[CLOT_NS - NSTG];
    float sig = 0.0f;
    if (G.act) {
#pragma unroll
      for (int q = NSTG; q < CLOT_NS; ++q) yb[q - NSTG] = __ldg(&row_at(A.cin, q, pitch, P));
      if (transport && K.has_sigma) sig = __ldg(&row_at(A.sigma, 0, 0, P));
    }
    const float fxlo = fx1, fylo = fy1, Fhi = fz1;
    if (k + 1 < ke) own_flux(k + 1);
    const float fend = fend1;
    if (k + 1 < ke) fend1 = end_flux(k + 1);  // in flight through this plane

    if (!landed(k + 2, 0)) { drain(k + 2, issued); return; }
    // every thread is past plane k - 1: its ring slot takes plane k + 3
    issue(k + 3);
    if (planned(k + 3)) issued = k + 3;
    const ZPlane& B0 = Sm.buf[(k - kb) % RING];
    ZPlane& B1 = Sm.buf[(hp1 ? k + 1 - kb : k - kb) % RING];  // beyond the last plane: its own values
    const ZPlane& B2 = k + 2 < nz ? Sm.buf[(k + 2 - kb) % RING] : B1;
    const float* Wk = Sm.W[wsel];
    float* Wn = Sm.W[wsel ^ 1];

    // W of plane k + 1 for the next plane, and whether plane k + 2 holds a
    // non-plasma species; both published by the barrier after the faces
    if (hp1) zm_w_pass(B1, Wn, tid, ip);
    const unsigned np = (planned(k + 2) && tid < SPT / 2) ? nonplasma_bits(B2, tid) : 0u;

    const bool plasma = lastp < k - 1;
    const float WP = Wk[sc];
    float c0[NT], xlo[NT], ylo[NT], dv[NT];
    if (plasma)
      zm_xy_faces<SET_PLASMA, PLAIN>(A, Sm, Wk, B0, G, k, WP, fxlo, fylo, fend, c0, xlo, ylo);
    else
      zm_xy_faces<SET_ALL, PLAIN>(A, Sm, Wk, B0, G, k, WP, fxlo, fylo, fend, c0, xlo, ylo);
    const float yPba = B0.c[CLOT_PBA][sc], yPbse = B0.c[CLOT_PBSE][sc];
    if (__syncthreads_or(np != 0u)) lastp = k + 2;
    if (ends && k + 1 < ke) zm_fill_ends(B1, G, nx, ny);  // published by the next plane's first barrier

#pragma unroll
    for (int t = 0; t < NT; ++t) dv[t] = 0.0f;
    if (G.act && transport) {
      const float Wp = hp1 ? Wn[sc] : WP;
      if (k == 0) {
#pragma unroll
        for (int t = 0; t < NT; ++t) cm1[t] = c0[t];
      }
      if (plasma)
        zm_z_faces<SET_PLASMA, PLAIN>(A, Sm, B1, B2, G, hp1, WP, Wp, Fhi, cm1, c0, xlo, ylo, fzlo, dv);
      else
        zm_z_faces<SET_ALL, PLAIN>(A, Sm, B1, B2, G, hp1, WP, Wp, Fhi, cm1, c0, xlo, ylo, fzlo, dv);
    }

    if (G.act) {
      float y[CLOT_NS];
#pragma unroll
      for (int t = 0; t < NT; ++t) y[trow(t)] = c0[t];
      y[CLOT_PBA] = yPba;
      y[CLOT_PBSE] = yPbse;
#pragma unroll
      for (int q = NSTG; q < CLOT_NS; ++q) y[q] = yb[q - NSTG];
      cell_epilogue<IDX, EXT, PLAIN>(A, y, dv, sig, need_eta ? B0.eta[sc] : 0.0f, overx && k >= K.g.k0 && k <= K.g.k1, G.gx,
                              G.gy, k, P);
      if (predict) {
        // eta for the next step: 2 eta - eta_prev, and the exact residual of
        // that guess against the new theta_B (App. A, Eq. eta); the missing
        // neighbours of end cells hold the cell's own values
        const float thB = (y[CLOT_PBA] + y[CLOT_PBSE]) * ip;
        auto guess = [&](int q) { return 2.0f * B0.eta[q] - B0.etp[q]; };
        const float gP = guess(sc);
        if (k == 0) gm1 = gP;
        const float lx = (guess(sc - 1) - gP) + (guess(sc + 1) - gP);
        const float ly = (guess(sc - SXT) - gP) + (guess(sc + SXT) - gP);
        const float lz = (gm1 - gP) + ((2.0f * B1.eta[sc] - B1.etp[sc]) - gP);
        const float r = thB - (gP - (A.ecx * lx + A.ecy * ly + A.ecz * lz));
        row_at(A.eta_next, 0, 0, P) = gP;
        row_at(A.eta_res, 0, 0, P) = r;
        rmax = fmaxf(rmax, fabsf(r));
        bmax = fmaxf(bmax, fmaxf(thB, 0.0f));
        gm1 = gP;
      }
#pragma unroll
      for (int t = 0; t < NT; ++t) cm1[t] = c0[t];
    }
    wsel ^= 1;
  }
  if (predict) block_max2(rmax, bmax, Sm.red, A.eta_max, A.eta_tiles ? (int)(blockIdx.x + gridDim.x * blockIdx.y) : -1, tid);
}

}  // namespace

// Planes per block for `cols` tile columns of nz planes: about 4.6 blocks for
// each of the two slots of an SM, at most MAXRUN planes.  A run pays its
// prologue once (three planes' loads, the face below it), so long runs cost
// less; but blocks over the injury integrate the reaction at about 5 us a plane
// where others take 2.5, and a mesh with few blocks waits for them.  K1 in us,
// plasma / primed, by run:
//   512 x 128 x 128   4: 381 / 521   8: 346 / 493   12: 331 / 477   (16: 367 / 487,
//                     neighbouring columns drift apart in z and miss each other's halos in L2)
//   256 x 128 x 64    2: 127 / 189   6: 107 / 168   12: 111 / 188
//   203 x 67 x 45     1: 82 / 112    3: 63 / 95     12: 80 / 124
//   64 x 24 x 24      1: 13 / 14     4: 29 / 29     12: 70 / 70
static int zm_run(long long cols, int nz) {
  static int sms = 0;
  if (sms == 0) {
    int dev = 0, n = 0;
    if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
    sms = n > 0 ? n : 152;
  }
  const long long per = 92ll * sms / 10;  // 4.6 blocks x 2 slots an SM
  const long long run = (cols * nz + per - 1) / per;
  const long long least = (nz + 65534) / 65535;  // the grid's z extent
  return (int)std::max(least, std::min<long long>(MAXRUN, std::max<long long>(run, 1)));
}

cudaError_t launch_zmarch(const StepArgs& a, cudaStream_t s) {
  const Geom& g = a.K.g;
  const StepConst& K = a.K;
  const bool need_eta = K.do_reaction || a.predict, ext = a.xin != nullptr;
  CUtensorMap tc, te, tp;
  memset(&tc, 0, sizeof(tc));
  memset(&te, 0, sizeof(te));
  memset(&tp, 0, sizeof(tp));
  // TMA where rows and bases are 16-byte aligned and the driver offers tensor
  // maps, else copies of two floats or one
  auto al = [](const void* p, unsigned n) { return p == nullptr || ((uintptr_t)p & (n - 1u)) == 0; };
  auto all = [&](unsigned n) { return al(a.cin, n) && al(a.eta, n) && al(a.eta_prev, n); };
  const bool tma = g.nx % 4 == 0 && g.pitch % 4 == 0 && all(16) && tensor_map_encoder() != nullptr &&
                   encode_field(&tc, a.cin, g, g.pitch, CLOT_NS, SXT, SYT, NSTG) &&
                   (!need_eta || encode_field(&te, a.eta, g, 0, 0, SXT, SYT, 0)) &&
                   (!a.predict || encode_field(&tp, a.eta_prev, g, 0, 0, SXT, SYT, 0));
  const bool two = g.nx % 2 == 0 && g.pitch % 2 == 0 && all(8);
  if (ext && !tma) return cudaErrorNotSupported;  // checked by the caller: the extension takes the TMA z march
  const size_t smem = sizeof(ZSm) + 128;
  const int run = zm_run((long long)((g.nx + TX - 1) / TX) * ((g.ny + TY - 1) / TY), g.nz);
  const dim3 grid((g.nx + TX - 1) / TX, (g.ny + TY - 1) / TY, (g.nz + run - 1) / run);
  auto launch = [&](auto* kern) -> cudaError_t {
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    kern<<<grid, dim3(TX, TY, 1), smem, s>>>(a, tc, te, tp, run);
    return cudaGetLastError();
  };
  // PLAIN: the one-stage step with everything on, its switches known at compile
  // time (the usual call; no options' code in the plane loop)
  const bool small = g.ncell < (1ll << 30);
  const bool plain = !ext && small && K.do_transport && K.do_reaction && a.predict && K.limiter && !K.closed_ends &&
                     !K.wall_lagged && !a.cavg && !a.e0lo;
  if (tma) {
    if (plain) return launch(zmarch_step_kernel<0, false, unsigned, true>);
    if (ext) return small ? launch(zmarch_step_kernel<0, true, unsigned, false>)
                          : launch(zmarch_step_kernel<0, true, long long, false>);
    return small ? launch(zmarch_step_kernel<0, false, unsigned, false>)
                 : launch(zmarch_step_kernel<0, false, long long, false>);
  }
  if (plain) return two ? launch(zmarch_step_kernel<2, false, unsigned, true>)
                        : launch(zmarch_step_kernel<1, false, unsigned, true>);
  if (small) return two ? launch(zmarch_step_kernel<2, false, unsigned, false>)
                        : launch(zmarch_step_kernel<1, false, unsigned, false>);
  return two ? launch(zmarch_step_kernel<2, false, long long, false>)
             : launch(zmarch_step_kernel<1, false, long long, false>);
}

}  // namespace clot
