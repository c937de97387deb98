// clot_eta_cg.cuh -- the iterative solve of App. A, Eq. eta, by conjugate
// gradients, for a team of blocks (clot_eta_ops.cuh): the whole mesh in
// Chronopoulos and Gear's single-reduction form (or, for callers without its
// five extra vectors, the two-reduction form), and the correction of a
// predicted eta on a box.
#pragma once

#include "clot_eta_ops.cuh"

namespace clot {

// CG with one grid reduction per iteration (Chronopoulos and Gear's
// formulation: with s = A p carried by a recurrence, s_i = w_i + beta_i s_{i-1}
// and w = A r, the two inner products (r, r) and (w, r) of an iteration are
// taken together).  Per iteration one pass: at each cell and its neighbours
// s_i = w_i + beta_i s_{i-1} and r_{i+1} = r_i - alpha_i s_i are formed on the
// fly, the cell's p_i = r_i + beta_i p_{i-1} updates eta, and w_{i+1} = A r_{i+1}
// with (r_{i+1}, r_{i+1}), (w_{i+1}, r_{i+1}) and max |r_{i+1}| goes to the one
// reduction; then beta_{i+1} = gamma_{i+1} / gamma_i and
// alpha_{i+1} = gamma_{i+1} / (delta_{i+1} - beta_{i+1} gamma_{i+1} / alpha_i).
// Every vector is double-buffered (no block overwrites a value another block
// still reads), so the traffic per iteration is that of the two-pass form.
// On entry a.r holds r_0 (s_rr its squared norm, s_rmax its maximum, s_del0 its
// product with A r_0 where that is known, else 0).
// Returns false if a grid barrier gave up.
template <int BS>
__device__ bool cg_single_reduction(const EtaArgs& a, Team& T, bool v4, double s_rr, double s_del0, float& s_rmax,
                                    double stop, int& it) {
  const int nb = T.nb;
  const long long n = a.g.ncell;
  float* R[2] = {a.r, a.cg5};
  float* Sv[2] = {a.cg5 + n, a.cg5 + 2 * n};
  float* Wv[2] = {a.cg5 + 3 * n, a.cg5 + 4 * n};
  float* Pv[2] = {a.p, a.p2};
  double s_del = s_del0, gamma, alpha, beta;
  int cur;
  const float* r0 = R[0];
  if (s_del0 > 0.0) {
    // r_0 is unchanged since the launch, so these passes may read it through L1
    const auto r0v4 = [&](long long Q) { return *reinterpret_cast<const float4*>(r0 + Q); };
    const auto r0v1 = [&](long long Q) { return r0[Q]; };
    // (w_0, r_0) is known: the first iteration forms w_0 = A r_0 on the fly and
    // writes eta alone.  From a prediction it is most often the last one.
    if (it >= a.maxit) return true;
    alpha = s_rr / s_del;
    const float al = (float)alpha;
    float rm = 0.0f;
    if (v4) {
      struct V { float4 e, x, w; };
      for_quads2(
          a, nb,
          [&](long long P, int i, int j, int k) {
            V v;
            v.e = ld4(a.eta + P);
            v.w = quad_op(a, P, i, j, k, r0v4, r0v1, v.x);
            return v;
          },
          [&](long long P, int, int, int, const V& v) {
            const float4 e = v.e, x = v.x, w = v.w;
            st4(a.eta + P, make_float4(e.x + al * x.x, e.y + al * x.y, e.z + al * x.z, e.w + al * x.w));
            rm = fmaxf(fmaxf(rm, fmaxf(fabsf(x.x - al * w.x), fabsf(x.y - al * w.y))),
                       fmaxf(fabsf(x.z - al * w.z), fabsf(x.w - al * w.w)));
          });
    } else {
      for_cells(a, nb, [&](long long P, int i, int j, int k) {
        const float x = __ldcg(r0 + P), w = apply_op(a, r0, P, i, j, k);
        a.eta[P] = __ldcg(a.eta + P) + al * x;
        rm = fmaxf(rm, fabsf(x - al * w));
      });
    }
    float none;
    double sums[2], zero[1];
    if (!team_reduce<BS, 1>(a, T, {0.0f}, rm, zero, s_rmax)) return false;
    ++it;
    if (it >= a.maxit || !(s_rmax > stop)) return true;
    // more are needed: their vectors s_0 = w_0, p_0 = r_0, r_1 and w_1 = A r_1
    if (v4) {
      for_quads(a, nb, [&](long long P, int i, int j, int k) {
        float4 x;
        const float4 w = quad_op(a, P, i, j, k, r0v4, r0v1, x);
        st4(Sv[0] + P, w);
        st4(Pv[0] + P, x);
        st4(R[1] + P, make_float4(x.x - al * w.x, x.y - al * w.y, x.z - al * w.z, x.w - al * w.w));
      });
    } else {
      for_cells(a, nb, [&](long long P, int i, int j, int k) {
        const float x = __ldcg(r0 + P), w = apply_op(a, r0, P, i, j, k);
        Sv[0][P] = w;
        Pv[0][P] = x;
        R[1][P] = x - al * w;
      });
    }
    if (!team_sync(a, T)) return false;
    const float* r1 = R[1];
    float g = 0.0f, del = 0.0f;
    if (v4) {
      for_quads(a, nb, [&](long long P, int i, int j, int k) {
        float4 x;
        const float4 w = quad_op(a, P, i, j, k, [&](long long Q) { return ld4(r1 + Q); },
                                 [&](long long Q) { return __ldcg(r1 + Q); }, x);
        st4(Wv[1] + P, w);
        g += x.x * x.x + x.y * x.y + x.z * x.z + x.w * x.w;
        del += w.x * x.x + w.y * x.y + w.z * x.z + w.w * x.w;
      });
    } else {
      for_cells(a, nb, [&](long long P, int i, int j, int k) {
        const float x = __ldcg(r1 + P), w = apply_op(a, r1, P, i, j, k);
        Wv[1][P] = w;
        g += x * x;
        del += w * x;
      });
    }
    if (!team_reduce<BS, 2>(a, T, {g, del}, 0.0f, sums, none)) return false;
    beta = sums[0] / s_rr;
    const double den = sums[1] - beta * sums[0] / alpha;
    if (!(den > 0.0) || !(sums[0] > 0.0)) return true;
    alpha = sums[0] / den;
    gamma = sums[0];
    cur = 1;
  } else {
    // w_0 = A r_0 and delta_0 = (w_0, r_0)
    float del = 0.0f;
    if (v4) {
      for_quads(a, nb, [&](long long P, int i, int j, int k) {
        float4 x;
        const float4 w = quad_op(a, P, i, j, k, [&](long long Q) { return ld4(r0 + Q); },
                                 [&](long long Q) { return __ldcg(r0 + Q); }, x);
        st4(Wv[0] + P, w);
        del += w.x * x.x + w.y * x.y + w.z * x.z + w.w * x.w;
      });
    } else {
      for_cells(a, nb, [&](long long P, int i, int j, int k) {
        const float w = apply_op(a, r0, P, i, j, k);
        Wv[0][P] = w;
        del += w * __ldcg(r0 + P);
      });
    }
    float none;
    double sums[1];
    if (!team_reduce<BS, 1>(a, T, {del}, 0.0f, sums, none)) return false;
    s_del = sums[0];
    if (!(s_del > 0.0)) return true;
    gamma = s_rr;
    alpha = s_rr / s_del;
    beta = 0.0;
    cur = 0;
  }
  while (it < a.maxit && s_rmax > stop) {
    const float al = (float)alpha, bt = (float)beta;
    const float* r = R[cur];
    const float* w = Wv[cur];
    const float* sp = Sv[cur ^ 1];
    const float* pp = Pv[cur ^ 1];
    float* rn = R[cur ^ 1];
    float* wn = Wv[cur ^ 1];
    float* sc = Sv[cur];
    float* pc = Pv[cur];
    float g = 0.0f, del = 0.0f, rm = 0.0f;
    if (v4) {
      auto s4 = [&](long long Q) {
        float4 v = ld4(w + Q);
        if (bt != 0.0f) {
          const float4 o = ld4(sp + Q);
          v.x += bt * o.x; v.y += bt * o.y; v.z += bt * o.z; v.w += bt * o.w;
        }
        return v;
      };
      auto r4 = [&](long long Q) {
        const float4 sv = s4(Q), rv = ld4(r + Q);
        return make_float4(rv.x - al * sv.x, rv.y - al * sv.y, rv.z - al * sv.z, rv.w - al * sv.w);
      };
      auto r1 = [&](long long Q) {
        const float sv = __ldcg(w + Q) + (bt != 0.0f ? bt * __ldcg(sp + Q) : 0.0f);
        return __ldcg(r + Q) - al * sv;
      };
      for_quads(a, nb, [&](long long P, int i, int j, int k) {
        const float4 sv = s4(P), rv = ld4(r + P), e = ld4(a.eta + P);
        float4 pv = rv;
        if (bt != 0.0f) {
          const float4 o = ld4(pp + P);
          pv.x += bt * o.x; pv.y += bt * o.y; pv.z += bt * o.z; pv.w += bt * o.w;
        }
        st4(sc + P, sv);
        st4(pc + P, pv);
        st4(a.eta + P, make_float4(e.x + al * pv.x, e.y + al * pv.y, e.z + al * pv.z, e.w + al * pv.w));
        float4 x;
        const float4 wv = quad_op(a, P, i, j, k, r4, r1, x);  // x: r_{i+1} on the quad
        st4(rn + P, x);
        st4(wn + P, wv);
        g += x.x * x.x + x.y * x.y + x.z * x.z + x.w * x.w;
        del += wv.x * x.x + wv.y * x.y + wv.z * x.z + wv.w * x.w;
        rm = fmaxf(fmaxf(rm, fmaxf(fabsf(x.x), fabsf(x.y))), fmaxf(fabsf(x.z), fabsf(x.w)));
      });
    } else {
      for_cells(a, nb, [&](long long P, int i, int j, int k) {
        const int nx = a.g.nx, ny = a.g.ny, nz = a.g.nz;
        auto sv = [&](long long Q) { return __ldcg(w + Q) + (bt != 0.0f ? bt * __ldcg(sp + Q) : 0.0f); };
        auto rv = [&](long long Q) { return __ldcg(r + Q) - al * sv(Q); };
        const float sP = sv(P);
        const float pP = __ldcg(r + P) + (bt != 0.0f ? bt * __ldcg(pp + P) : 0.0f);
        sc[P] = sP;
        pc[P] = pP;
        a.eta[P] = __ldcg(a.eta + P) + al * pP;
        const float rP = __ldcg(r + P) - al * sP;
        float lx = 0.0f, ly = 0.0f, lz = 0.0f;
        if (i > 0) lx += rv(P - 1) - rP;
        if (i < nx - 1) lx += rv(P + 1) - rP;
        if (j > 0) ly += rv(P - nx) - rP;
        if (j < ny - 1) ly += rv(P + nx) - rP;
        if (a.g.dim == 3) {
          const long long sz = (long long)nx * ny;
          if (k > 0) lz += rv(P - sz) - rP;
          if (k < nz - 1) lz += rv(P + sz) - rP;
        }
        const float wP = rP - (a.cx * lx + a.cy * ly + a.cz * lz);
        rn[P] = rP;
        wn[P] = wP;
        g += rP * rP;
        del += wP * rP;
        rm = fmaxf(rm, fabsf(rP));
      });
    }
    double sums[2];
    if (!team_reduce<BS, 2>(a, T, {g, del}, rm, sums, s_rmax)) return false;
    const double s_g = sums[0];
    s_del = sums[1];
    ++it;
    beta = s_g / gamma;
    const double den = s_del - beta * s_g / alpha;
    if (!(den > 0.0) || !(s_g > 0.0)) break;
    alpha = s_g / den;
    gamma = s_g;
    cur ^= 1;
  }
  return true;
}

// The two-reduction form, on the vectors r, p, q, p2 alone.
template <int BS>
__device__ bool cg_two_reductions(const EtaArgs& a, Team& T, bool v4, double s_rr, float& s_rmax, double stop,
                                  int& it) {
  // CG with the search-direction update folded into the operator pass:
  // p_new = r + beta p_old is formed on the fly at each cell and its
  // neighbours (p_old and p_new live in two buffers, so no block overwrites
  // a value another block still reads).  Two grid reductions per iteration.
  float* pold = a.p;
  float* pnew = a.p2;
  float beta = 0.0f;  // first direction: p = r
  while (it < a.maxit && s_rmax > stop) {
    float pq = 0.0f;
    const float bt = beta;
    const float* po = pold;
    float* pn = pnew;
    if (v4) {
      auto pv4 = [&](long long Q) {
        float4 v = ld4(a.r + Q);
        if (bt != 0.0f) {
          const float4 o = ld4(po + Q);
          v.x += bt * o.x; v.y += bt * o.y; v.z += bt * o.z; v.w += bt * o.w;
        }
        return v;
      };
      auto pv1 = [&](long long Q) { return __ldcg(a.r + Q) + (bt != 0.0f ? bt * __ldcg(po + Q) : 0.0f); };
      for_quads(a, T.nb, [&](long long P, int i, int j, int k) {
        float4 pp;
        const float4 q = quad_op(a, P, i, j, k, pv4, pv1, pp);
        st4(pn + P, pp);
        st4(a.q + P, q);
        pq += pp.x * q.x + pp.y * q.y + pp.z * q.z + pp.w * q.w;
      });
    } else {
      for_cells(a, T.nb, [&](long long P, int i, int j, int k) {
        const int nx = a.g.nx, ny = a.g.ny, nz = a.g.nz;
        auto pv = [&](long long Q) { return __ldcg(a.r + Q) + (bt != 0.0f ? bt * __ldcg(po + Q) : 0.0f); };
        const float pp = pv(P);
        float lx = 0.0f, ly = 0.0f, lz = 0.0f;
        if (i > 0) lx += pv(P - 1) - pp;
        if (i < nx - 1) lx += pv(P + 1) - pp;
        if (j > 0) ly += pv(P - nx) - pp;
        if (j < ny - 1) ly += pv(P + nx) - pp;
        if (a.g.dim == 3) {
          const long long sz = (long long)nx * ny;
          if (k > 0) lz += pv(P - sz) - pp;
          if (k < nz - 1) lz += pv(P + sz) - pp;
        }
        const float q = pp - (a.cx * lx + a.cy * ly + a.cz * lz);
        pn[P] = pp;
        a.q[P] = q;
        pq += pp * q;
      });
    }
    float none;
    double sums[1];
    if (!team_reduce<BS, 1>(a, T, {pq}, 0.0f, sums, none)) return false;
    const double s_pq = sums[0];
    const float alpha = (float)(s_rr / s_pq);
    float rr2 = 0.0f, rm = 0.0f;
    if (v4) {
      for_quads(a, T.nb, [&](long long P, int, int, int) {
        const float4 pP = ld4(pn + P), e = ld4(a.eta + P), r0 = ld4(a.r + P), q = ld4(a.q + P);
        st4(a.eta + P, make_float4(e.x + alpha * pP.x, e.y + alpha * pP.y, e.z + alpha * pP.z, e.w + alpha * pP.w));
        const float4 r = make_float4(r0.x - alpha * q.x, r0.y - alpha * q.y, r0.z - alpha * q.z, r0.w - alpha * q.w);
        st4(a.r + P, r);
        rr2 += r.x * r.x + r.y * r.y + r.z * r.z + r.w * r.w;
        rm = fmaxf(fmaxf(rm, fmaxf(fabsf(r.x), fabsf(r.y))), fmaxf(fabsf(r.z), fabsf(r.w)));
      });
    } else {
      for_cells(a, T.nb, [&](long long P, int, int, int) {
        const float pP = __ldcg(pn + P);
        a.eta[P] = __ldcg(a.eta + P) + alpha * pP;
        const float r = __ldcg(a.r + P) - alpha * __ldcg(a.q + P);
        a.r[P] = r;
        rr2 += r * r;
        rm = fmaxf(rm, fabsf(r));
      });
    }
    if (!team_reduce<BS, 1>(a, T, {rr2}, rm, sums, s_rmax)) return false;
    const double s_rr2 = sums[0];
    beta = (float)(s_rr2 / s_rr);
    s_rr = s_rr2;
    float* t = pold;
    pold = pnew;
    pnew = t;
    ++it;
  }
  return true;
}

// theta_B - A eta into a.r, its squared norm, its maximum, and max |theta_B|.
template <int BS>
__device__ __forceinline__ bool residual_reduce(const EtaArgs& a, Team& T, bool v4, double& s_rr, float& s_bmax,
                                                float& s_rmax) {
  const long long pitch = a.g.pitch;
  float rr = 0.0f, rmax = 0.0f, bmax = 0.0f;
  if (v4) {
    const float* eta = a.eta;
    for_quads(a, T.nb, [&](long long P, int i, int j, int k) {
      const float4 b2 = ld4(a.c + 2 * pitch + P), b3 = ld4(a.c + 3 * pitch + P);
      float4 x;
      const float4 q = quad_op(a, P, i, j, k, [&](long long Q) { return ld4(eta + Q); },
                               [&](long long Q) { return __ldcg(eta + Q); }, x);
      const float b[4] = {(b2.x + b3.x) * a.invPmax, (b2.y + b3.y) * a.invPmax, (b2.z + b3.z) * a.invPmax,
                          (b2.w + b3.w) * a.invPmax};
      const float r[4] = {b[0] - q.x, b[1] - q.y, b[2] - q.z, b[3] - q.w};
      st4(a.r + P, make_float4(r[0], r[1], r[2], r[3]));
#pragma unroll
      for (int m = 0; m < 4; ++m) {
        rr += r[m] * r[m];
        rmax = fmaxf(rmax, fabsf(r[m]));
        bmax = fmaxf(bmax, fabsf(b[m]));
      }
    });
  } else {
    for_cells(a, T.nb, [&](long long P, int i, int j, int k) {
      const float b = (__ldcg(a.c + 2 * pitch + P) + __ldcg(a.c + 3 * pitch + P)) * a.invPmax;
      const float r = b - apply_op(a, a.eta, P, i, j, k);
      a.r[P] = r;
      rr += r * r;
      rmax = fmaxf(rmax, fabsf(r));
      bmax = fmaxf(bmax, fabsf(b));
    });
  }
  // one barrier for both maxima: |theta_B|'s rides on words of its own
  const unsigned b = __reduce_max_sync(0xffffffffu, __float_as_uint(bmax));
  if ((threadIdx.x & 31) == 0 && b != 0u) atomicMax(a.own + 6, b);
  double sums[1];
  if (!team_reduce<BS, 1>(a, T, {rr}, rmax, sums, s_rmax)) return false;
  s_rr = sums[0];
  s_bmax = __uint_as_float(__ldcg(a.own + 6));
  return true;
}

// What a solve did: iterations, whether a prediction was corrected on a box
// (1) or that was not enough (-1), whether this block left the team early, and
// whether eta was written after the last barrier (another must precede its use).
struct EtaOut {
  int it = 0, box = 0;
  bool gone = false, sync = false;
};

// CG until max |r| meets the stopping rule.  predicted: eta and r are the fused
// step's (s_rr is then not set): the cells with |r| > stop / (2 (1 + c)) are
// boxed and the box corrected first.  Returns false if a grid barrier gave up.
template <int BS>
__device__ __forceinline__ bool eta_iterate(const EtaArgs& a, Team& T, bool v4, bool predicted, double s_rr,
                                            float s_rmax, float s_bmax, EtaOut& o) {
  const long long pitch = a.g.pitch;
  const double stop = (double)a.inner * fmax((double)a.tol * s_bmax, (double)a.atol);
  if (s_bmax == 0.0f) {  // theta_B = 0 everywhere: eta = 0, whatever r holds
    o.sync = true;
    for_cells(a, T.nb, [&](long long P, int, int, int) { a.eta[P] = 0.0f; });
    return true;
  }
  double s_del = 0.0;
  if (predicted) {
    // Core threshold: a cell just inside the box edge with |r| <= thr gets a
    // correction of about thr, which the zero outside turns into a residual
    // of up to (1 + c) thr in the next cell out; with thr = stop / (2 (1 + c))
    // that and the decayed core correction each stay below stop / 2.
    const float pr = s_rmax;
    const float cmax = fmaxf(a.cx, fmaxf(a.cy, a.cz));
    const float thr = (float)(0.5 * stop) / (1.0f + cmax);
    // The bounding box of the cells with |r| > thr, kept as max(~lo) and
    // max(hi + 1) per axis in own[0..5].  Only tiles whose maximum the fused
    // step put above thr are swept; a small mesh is swept whole, together with
    // the two inner products that the whole-mesh iteration starts from.
    unsigned* bw = a.own;
    Box R{0, a.g.nx - 1, 0, a.g.ny - 1, 0, a.g.nz - 1};
    const bool all = a.tiles == 0 || a.g.ncell <= (1 << 17);
    if (!all) {
      const int ntx = (a.g.nx + 31) >> 5;
      int x0 = ntx, x1 = -1, y0 = 1 << 30, y1 = -1;
      for (int t = threadIdx.x & 31; t < a.tiles; t += 32)
        if (__uint_as_float(__ldcg(a.maxw + 2 + t)) > thr) {
          x0 = min(x0, t % ntx);
          x1 = max(x1, t % ntx);
          y0 = min(y0, t / ntx);
          y1 = max(y1, t / ntx);
        }
      R.i0 = 32 * __reduce_min_sync(0xffffffffu, x0);
      R.i1 = min(32 * __reduce_max_sync(0xffffffffu, x1) + 31, a.g.nx - 1);
      R.j0 = min(8 * __reduce_min_sync(0xffffffffu, min(y0, 1 << 24)), a.g.ny);
      R.j1 = min(8 * __reduce_max_sync(0xffffffffu, y1) + 7, a.g.ny - 1);
    }
    float rr = 0.0f, del = 0.0f;
    unsigned bl[3] = {0u, 0u, 0u}, bh[3] = {0u, 0u, 0u};
    auto mark = [&](float r, int i, int j, int k) {
      if (fabsf(r) > thr) {
        bl[0] = max(bl[0], ~(unsigned)i);
        bl[1] = max(bl[1], ~(unsigned)j);
        bl[2] = max(bl[2], ~(unsigned)k);
        bh[0] = max(bh[0], (unsigned)i + 1u);
        bh[1] = max(bh[1], (unsigned)j + 1u);
        bh[2] = max(bh[2], (unsigned)k + 1u);
      }
    };
    auto whole = [&](auto fn) {  // (r, r) and (A r, r) of the whole mesh (r read through L1: unchanged since the launch)
      if (v4) {
        const float* r0 = a.r;
        struct V { float4 r, w; };
        for_quads2(
            a, T.nb,
            [&](long long P, int i, int j, int k) {
              V v;
              v.w = quad_op(a, P, i, j, k, [&](long long Q) { return *reinterpret_cast<const float4*>(r0 + Q); },
                            [&](long long Q) { return r0[Q]; }, v.r);
              return v;
            },
            [&](long long, int i, int j, int k, const V& v) {
              const float4 r = v.r, w = v.w;
              rr += r.x * r.x + r.y * r.y + r.z * r.z + r.w * r.w;
              del += w.x * r.x + w.y * r.y + w.z * r.z + w.w * r.w;
              fn(r.x, i, j, k);
              fn(r.y, i + 1, j, k);
              fn(r.z, i + 2, j, k);
              fn(r.w, i + 3, j, k);
            });
      } else {
        for_cells(a, T.nb, [&](long long P, int i, int j, int k) {
          const float r = __ldcg(a.r + P);
          rr += r * r;
          del += apply_op(a, a.r, P, i, j, k) * r;
          fn(r, i, j, k);
        });
      }
    };
    if (all) {
      whole(mark);
    } else if (R.i1 >= R.i0 && R.j1 >= R.j0) {
      struct V { float r; int i, j, k; };
      for_box_cells(
          a, T.nb, R, [&](long long P, int i, int j, int k) { return V{__ldcg(a.r + P), i, j, k}; },
          [&](long long, const V& v) { mark(v.r, v.i, v.j, v.k); });
    }
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      bl[d] = __reduce_max_sync(0xffffffffu, bl[d]);
      bh[d] = __reduce_max_sync(0xffffffffu, bh[d]);
    }
    if ((threadIdx.x & 31) == 0 && bh[0] != 0u) {
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        atomicMax(bw + d, bl[d]);
        atomicMax(bw + 3 + d, bh[d]);
      }
    }
    double sums[2];
    float none;
    if (!team_reduce<BS, 2>(a, T, {rr, del}, 0.0f, sums, none)) return false;

    Box B;
    bool use_box = false;
    unsigned w[6];
#pragma unroll
    for (int d = 0; d < 6; ++d) w[d] = __ldcg(bw + d);
    const unsigned hx = w[3];
    if (pr < 3.0e38f && hx != 0u) {
      const int mx = box_margin(a.cx, pr, (float)stop), my = box_margin(a.cy, pr, (float)stop);
      const int mz = a.g.dim == 3 ? box_margin(a.cz, pr, (float)stop) : 0;
      B.i0 = max((int)~w[0] - mx, 0);
      B.j0 = max((int)~w[1] - my, 0);
      B.k0 = max((int)~w[2] - mz, 0);
      B.i1 = min((int)hx - 1 + mx, a.g.nx - 1);
      B.j1 = min((int)w[4] - 1 + my, a.g.ny - 1);
      B.k1 = min((int)w[5] - 1 + mz, a.g.nz - 1);
      use_box = 2 * B.cells() <= a.g.ncell;
    }
    if (use_box) {
      // about eight cells a thread: blocks beyond that would only add arrivals
      const int want = T.shrink ? (int)min((long long)T.nb, max(1ll, B.cells() / (8 * BS))) : T.nb;
      if ((int)blockIdx.x >= want) {
        o.gone = true;
        return true;
      }
      T.nb = want;
      // CG for the correction on the box, in place on eta and r, with the
      // search direction zero outside the box
      float* pold = a.p;
      float* pnew = a.p2;
      float beta = 0.0f;
      double s_rb = 0.0;
      float s_mb = pr;
      bool first = true;
      while (o.it < a.maxit && s_mb > stop) {
        float pq = 0.0f, r0 = 0.0f;
        const float bt = beta;
        const float* po = pold;
        float* pn = pnew;
        struct V { float p, q, r; };
        for_box_cells(
            a, T.nb, B,
            [&](long long P, int i, int j, int k) {
              const int nx = a.g.nx, ny = a.g.ny, nz = a.g.nz;
              auto pv = [&](long long Q) {  // the first iteration's r is unchanged since the launch: through L1
                return first ? a.r[Q] : __ldcg(a.r + Q) + bt * __ldcg(po + Q);
              };
              V v;
              v.p = pv(P);
              v.r = first ? __ldcg(a.r + P) : 0.0f;
              const float pp = v.p;
              float lx = 0.0f, ly = 0.0f, lz = 0.0f;
              if (i > 0) lx += (i - 1 >= B.i0 ? pv(P - 1) : 0.0f) - pp;
              if (i < nx - 1) lx += (i + 1 <= B.i1 ? pv(P + 1) : 0.0f) - pp;
              if (j > 0) ly += (j - 1 >= B.j0 ? pv(P - nx) : 0.0f) - pp;
              if (j < ny - 1) ly += (j + 1 <= B.j1 ? pv(P + nx) : 0.0f) - pp;
              if (a.g.dim == 3) {
                const long long sz = (long long)nx * ny;
                if (k > 0) lz += (k - 1 >= B.k0 ? pv(P - sz) : 0.0f) - pp;
                if (k < nz - 1) lz += (k + 1 <= B.k1 ? pv(P + sz) : 0.0f) - pp;
              }
              v.q = pp - (a.cx * lx + a.cy * ly + a.cz * lz);
              return v;
            },
            [&](long long P, const V& v) {
              pn[P] = v.p;
              a.q[P] = v.q;
              pq += v.p * v.q;
              r0 += v.r * v.r;
            });
        double sums[2], one[1];
        float none_;
        if (!team_reduce<BS, 2>(a, T, {pq, r0}, 0.0f, sums, none_)) return false;
        const double s_pq = sums[0], s_r0 = sums[1];
        if (first) s_rb = s_r0;
        first = false;
        if (!(s_pq > 0.0)) break;
        const float alpha = (float)(s_rb / s_pq);
        float rr2 = 0.0f, rm = 0.0f;
        struct U { float e, r; };
        for_box_cells(
            a, T.nb, B,
            [&](long long P, int, int, int) {
              return U{__ldcg(a.eta + P) + alpha * __ldcg(pn + P), __ldcg(a.r + P) - alpha * __ldcg(a.q + P)};
            },
            [&](long long P, const U& v) {
              a.eta[P] = v.e;
              a.r[P] = v.r;
              rr2 += v.r * v.r;
              rm = fmaxf(rm, fabsf(v.r));
            });
        if (!team_reduce<BS, 1>(a, T, {rr2}, rm, one, s_mb)) return false;
        const double s_rr2 = one[0];
        beta = (float)(s_rr2 / s_rb);
        s_rb = s_rr2;
        float* t = pold;
        pold = pnew;
        pnew = t;
        ++o.it;
      }
      // The box carries the CG residual (the recursive one, as in the global
      // iteration: recomputing theta_B - A eta in FP32 there would mostly show
      // eta's own rounding, amplified up to 1 + 12 c times).  The cells just
      // outside it get the true residual, which is where cutting the
      // correction off shows; every cell further out keeps its residual <= thr.
      Box L = B;
      L.i0 = max(B.i0 - 1, 0);
      L.j0 = max(B.j0 - 1, 0);
      L.k0 = max(B.k0 - 1, 0);
      L.i1 = min(B.i1 + 1, a.g.nx - 1);
      L.j1 = min(B.j1 + 1, a.g.ny - 1);
      L.k1 = min(B.k1 + 1, a.g.nz - 1);
      float vm = 0.0f;
      auto layer = [&](long long P, int i, int j, int k) {
        if (B.in(i, j, k)) return 0.0f;
        const float b = (__ldcg(a.c + 2 * pitch + P) + __ldcg(a.c + 3 * pitch + P)) * a.invPmax;
        const float r = b - apply_op(a, a.eta, P, i, j, k);
        a.r[P] = r;
        return r;
      };
      auto far = [&](long long, float r) { vm = fmaxf(vm, fabsf(r)); };
      // the six faces of the layer, edges with the x faces first
      const Box F[6] = {{L.i0, B.i0 - 1, L.j0, L.j1, L.k0, L.k1}, {B.i1 + 1, L.i1, L.j0, L.j1, L.k0, L.k1},
                        {B.i0, B.i1, L.j0, B.j0 - 1, L.k0, L.k1}, {B.i0, B.i1, B.j1 + 1, L.j1, L.k0, L.k1},
                        {B.i0, B.i1, B.j0, B.j1, L.k0, B.k0 - 1}, {B.i0, B.i1, B.j0, B.j1, B.k1 + 1, L.k1}};
#pragma unroll 1
      for (int f = 0; f < 6; ++f) for_box_cells(a, T.nb, F[f], layer, far);
      double zero[1];
      float s_vm;
      if (!team_reduce<BS, 1>(a, T, {0.0f}, vm, zero, s_vm)) return false;
      if (s_mb <= stop && s_vm <= stop) {
        o.box = 1;
        return true;
      }
      o.box = -1;  // continue on the whole mesh from the improved eta
      if (!residual_reduce<BS>(a, T, v4, s_rr, s_bmax, s_rmax)) return false;
    } else if (!all) {
      whole([](float, int, int, int) {});
      if (!team_reduce<BS, 2>(a, T, {rr, del}, 0.0f, sums, none)) return false;
    }
    if (o.box == 0) {
      s_rr = sums[0];
      s_del = sums[1];
    }
  }
  if (a.cg5)
    return cg_single_reduction<BS>(a, T, v4 && al16(a.cg5) && (a.g.ncell & 3) == 0, s_rr, s_del, s_rmax, stop, o.it);
  return cg_two_reductions<BS>(a, T, v4, s_rr, s_rmax, stop, o.it);
}

// The fused step's maxima of a prediction (in pr, pb) against the stopping
// rule; block 0 clears the words the next fused step adds to.
__device__ __forceinline__ bool prediction_accepted(const EtaArgs& a, float& pr, float& pb) {
  pr = __uint_as_float(__ldcg(a.maxw));
  pb = __uint_as_float(__ldcg(a.maxw + 1));
  if (blockIdx.x == 0) {
    for (int q = threadIdx.x; q < 2 + a.tiles; q += blockDim.x) a.maxw_clear[q] = 0u;
    if (threadIdx.x == 0) a.status[1] = 0;
  }
  const bool ok = pb > 0.0f && pr <= fmaxf(a.tol * pb, a.atol);
  if (ok && blockIdx.x == 0 && threadIdx.x == 0) atomicAdd(a.status + 3, 1);
  return ok;
}

// The status words of a solve.
__device__ __forceinline__ void eta_note(const EtaArgs& a, const EtaOut& o, bool ok) {
  if (threadIdx.x != 0 || blockIdx.x != 0 || !ok) return;
  a.status[1] = o.it;
  atomicAdd(a.status + 2, o.it);             // iterations summed over solves
  if (o.box > 0) atomicAdd(a.status + 4, 1);  // predictions corrected on a box
  if (o.box < 0) atomicAdd(a.status + 5, 1);  // box corrections not enough
}

// End of a launch, by every block: the last one to leave resets the barrier
// words for the next launch.
__device__ __forceinline__ void team_leave(const EtaArgs& a) {
  __syncthreads();
  if (threadIdx.x != 0) return;
  __threadfence();
  if (atomicAdd(a.bar + 1, 1u) == gridDim.x - 1)
    for (int q = 0; q < BAR_WORDS; ++q) a.bar[q] = 0u;
}

}  // namespace clot
