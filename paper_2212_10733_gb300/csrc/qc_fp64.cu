// Residual quantization and QoI correction with the per-point work in native
// FP64: one warp per histogram, the histogram staged in shared memory.  This
// is the plain form of Stages 4-5 and the GPU reference for the fast kernel.
//
//   targets   Q_k = sum vol phi_k x, phi = (1, v_par, v_perp^2, v_par^2),
//             the moments behind n, u_par, T_perp, T_par (Eq. (1)-(4));
//   quantizer Delta = 2^floor(log2(2 alpha tau max x)), exact round-half-even
//             codes with a zero level and escapes (Stage 4);
//   Newton    lambda <- lambda + s M^-1 g on the dual (Eq. (6)), the exponent
//             separated as exp(-lambda.phi) = a_i(lambda0, lambda1, lambda3)
//             b_j(lambda2), so each step takes n_par + n_perp exponentials;
//   fallback  round 2 (damped Newton from 0), end-to-end check, one retry with
//             alpha/4, verbatim (Stage 5 and the paper's parameter study).
#include "qc_common.cuh"

namespace aeqc {
namespace {

using namespace dev;

constexpr int WPC = 4;  // warps per CTA

struct WS {
  double xs[AEQC_MAX_P];  // x
  double xp[AEQC_MAX_P];  // x'
  double ta[AEQC_MAX_NPAR];
  double tb[AEQC_MAX_NPERP];
  int16_t codes[AEQC_MAX_P];
};

__device__ __forceinline__ double vol_of(const GridK& g, int p) {
  return g.has_vol ? __ldg(g.vol + p) : g.vol_uniform;
}

// One point's share of the sums, with every rounding written out: the cluster
// form further below forms the same sums from the same terms in the same order
// and has to get the same bits (left to contraction, the compiler decides per
// kernel which products it fuses).
struct Products {
  double v, w, vv, vvv;  // y v, y v_perp^2, y v^2, y v^3
};
__device__ __forceinline__ Products products_of(double y, double v, double v2) {
  Products t;
  t.v = __dmul_rn(y, v);
  t.w = __dmul_rn(y, v2);
  t.vv = __dmul_rn(t.v, v);
  t.vvv = __dmul_rn(t.vv, v);
  return t;
}
__device__ __forceinline__ void add_moments(double y, double v, double v2, double& a0, double& a1,
                                            double& a2, double& a3) {
  const double yv = __dmul_rn(y, v);
  a0 = __dadd_rn(a0, y);
  a1 = __dadd_rn(a1, yv);
  a2 = __fma_rn(y, v2, a2);
  a3 = __fma_rn(yv, v, a3);
}
__device__ __forceinline__ void add_abs_moments(double y, double v, double v2, double& s0,
                                                double& s1, double& s2, double& s3) {
  s0 = __dadd_rn(s0, y);
  s1 = __fma_rn(y, fabs(v), s1);
  s2 = __fma_rn(y, v2, s2);
  s3 = __fma_rn(__dmul_rn(y, v), v, s3);
}

// Q_k(x) and S_k(x) = sum vol |phi_k| |x| for the histogram in xs.
__device__ void moments_warp(const GridK& g, const double* xs, double Q[4], double S[4],
                             int lane) {
  double q0 = 0, q1 = 0, q2 = 0, q3 = 0, s0 = 0, s1 = 0, s2 = 0, s3 = 0;
  PointIter it(lane, g.n_par);
  for (; it.p < g.P; it.next()) {
    const double v = g.vpar[it.i], v2 = g.vperp2[it.j];
    const double w = __dmul_rn(vol_of(g, it.p), xs[it.p]);
    add_moments(w, v, v2, q0, q1, q2, q3);
    add_abs_moments(fabs(w), v, v2, s0, s1, s2, s3);
  }
  Q[0] = wsum(q0); Q[1] = wsum(q1); Q[2] = wsum(q2); Q[3] = wsum(q3);
  S[0] = wsum(s0); S[1] = wsum(s1); S[2] = wsum(s2); S[3] = wsum(s3);
}

struct Eval {
  double A[4];   // sum vol phi_k f
  double S[4];   // sum vol |phi_k| |f|
  double M[10];  // upper triangle of sum vol phi phi^T w (w = f for KL, 1 for L2)
  double res;    // max_k |A_k - Q_k| / S_k
};

// One pass over the histogram at lambda: f, A, S, (M).  For the KL loss the
// exponential tables ta, tb are left for lambda in shared memory.
__device__ void eval_warp(const GridK& g, WS& w, const double lam[4], const double Q[4],
                          int loss, bool want_M, Eval& r, int lane) {
  if (loss == 0) {
    for (int i = lane; i < g.n_par; i += 32) w.ta[i] = corr_a(lam, g.vpar[i]);
    for (int j = lane; j < g.n_perp; j += 32) w.tb[j] = corr_b(lam, g.vperp2[j]);
    __syncwarp();
  }
  double a0 = 0, a1 = 0, a2 = 0, a3 = 0, s0 = 0, s1 = 0, s2 = 0, s3 = 0;
  double m00 = 0, m01 = 0, m02 = 0, m03 = 0, m12 = 0, m13 = 0, m22 = 0, m23 = 0, m33 = 0;
  PointIter it(lane, g.n_par);
  for (; it.p < g.P; it.next()) {
    double v = g.vpar[it.i], v2 = g.vperp2[it.j];
    double vol = vol_of(g, it.p);
    double f, wm;
    if (loss == 0) {
      f = corr_kl(w.xp[it.p], w.ta[it.i], w.tb[it.j]);
      wm = __dmul_rn(f, vol);
    } else {
      f = corr_l2(w.xp[it.p], lam, v, v2);
      wm = vol;
    }
    const double fv = __dmul_rn(f, vol);
    add_moments(fv, v, v2, a0, a1, a2, a3);
    add_abs_moments(fabs(fv), v, v2, s0, s1, s2, s3);
    if (want_M) {
      const Products t = products_of(wm, v, v2);
      m00 = __dadd_rn(m00, wm);
      m01 = __dadd_rn(m01, t.v);
      m02 = __dadd_rn(m02, t.w);
      m03 = __dadd_rn(m03, t.vv);
      m12 = __fma_rn(t.v, v2, m12);
      m13 = __dadd_rn(m13, t.vvv);
      m22 = __fma_rn(t.w, v2, m22);
      m23 = __fma_rn(t.vv, v2, m23);
      m33 = __fma_rn(t.vvv, v, m33);
    }
  }
  r.A[0] = wsum(a0); r.A[1] = wsum(a1); r.A[2] = wsum(a2); r.A[3] = wsum(a3);
  r.S[0] = wsum(s0); r.S[1] = wsum(s1); r.S[2] = wsum(s2); r.S[3] = wsum(s3);
  if (want_M) {
    r.M[0] = wsum(m00); r.M[1] = wsum(m01); r.M[2] = wsum(m02); r.M[3] = wsum(m03);
    r.M[4] = r.M[3];  // sum w v^2 == m03
    r.M[5] = wsum(m12); r.M[6] = wsum(m13); r.M[7] = wsum(m22); r.M[8] = wsum(m23);
    r.M[9] = wsum(m33);
  }
  double gk[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) gk[k] = r.A[k] - Q[k];
  r.res = scaled_residual(gk, r.S);
}

// Round 1: plain steps of Eq. (6) from lam; returns 1 if converged.  r0 is the
// scaled residual at the starting point, e the last evaluation.
__device__ int round1_warp(const GridK& g, WS& w, const double Q[4], double lam[4],
                           int max_iter, double step, double tol, int loss, int* iters,
                           double* r0, Eval& e, int lane) {
  for (int it = 0;; ++it) {
    eval_warp(g, w, lam, Q, loss, true, e, lane);
    if (it == 0) *r0 = e.res;
    *iters = it;
    if (!isfinite(e.res)) return 0;
    if (e.res <= tol) return 1;
    if (it == max_iter) return 0;
    double gk[4], d[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) gk[k] = e.A[k] - Q[k];
    if (chol_solve4(e.M, gk, d) != 0) return 0;
#pragma unroll
    for (int k = 0; k < 4; ++k) lam[k] = __fma_rn(step, d[k], lam[k]);
  }
}

// Round 2: damped Newton from 0.  A step t in {1, 1/2, ...} is accepted when
// it lowers psi = sum vol f + lambda.Q by the Armijo amount, or, where that
// decrease is below psi's rounding (near the solution), when psi stays within
// 1e-12 of its scale sum vol |f| + sum |lambda_k Q_k| and the scaled residual
// falls by the factor (1 - t/2).  A step that raises psi beyond its rounding
// is never taken: one that blows f up also blows up S, the residual's scale.
__device__ int round2_warp(const GridK& g, WS& w, const double Q[4], double lam[4],
                           int max_iter, double tol, int loss, int* iters, Eval& e,
                           int lane) {
#pragma unroll
  for (int k = 0; k < 4; ++k) lam[k] = 0.0;
  for (int it = 0;; ++it) {
    eval_warp(g, w, lam, Q, loss, true, e, lane);
    *iters = it;
    if (!isfinite(e.res)) return 0;
    if (e.res <= tol) return 1;
    if (it == max_iter) return 0;
    double gk[4], d[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) gk[k] = e.A[k] - Q[k];
    if (chol_solve4(e.M, gk, d) != 0) return 0;
    double psi0 = e.A[0] + lam[0] * Q[0] + lam[1] * Q[1] + lam[2] * Q[2] + lam[3] * Q[3];
    double sc0 = e.S[0] + fabs(lam[0] * Q[0]) + fabs(lam[1] * Q[1]) + fabs(lam[2] * Q[2]) +
                 fabs(lam[3] * Q[3]);
    double slope = gk[0] * d[0] + gk[1] * d[1] + gk[2] * d[2] + gk[3] * d[3];
    double r = e.res, t = 1.0;
    int accepted = 0;
    for (int h = 0; h < 40; ++h, t *= 0.5) {
      double lt[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) lt[k] = lam[k] + t * d[k];
      Eval et;
      eval_warp(g, w, lt, Q, loss, false, et, lane);
      if (!isfinite(et.res)) continue;
      double psit = et.A[0] + lt[0] * Q[0] + lt[1] * Q[1] + lt[2] * Q[2] + lt[3] * Q[3];
      double flat = 1e-12 * (sc0 + et.S[0] + fabs(lt[0] * Q[0]) + fabs(lt[1] * Q[1]) +
                             fabs(lt[2] * Q[2]) + fabs(lt[3] * Q[3]));
      if (psit <= psi0 - 1e-4 * t * slope ||
          (psit <= psi0 + flat && et.res <= (1.0 - 0.5 * t) * r)) {
#pragma unroll
        for (int k = 0; k < 4; ++k) lam[k] = lt[k];
        accepted = 1;
        break;
      }
    }
    if (!accepted) return 0;
  }
}

constexpr unsigned NOT_CONVERGED = 0x8000u;

// Newton driver (rounds 1-2 and the warm-start probation).  Leaves the tables
// of the final lambda in shared memory and its evaluation in e.
__device__ unsigned newton_warp(const GridK& g, WS& w, const double Q[4], double lam[4],
                                int warm, const ParamsK& pr, int* iters, Eval& e,
                                int lane) {
  unsigned st = 0;
  int it1 = 0, it2 = 0, itw = 0, conv;
  double r0 = 0.0, rdummy;
  if (warm) {
    conv = round1_warp(g, w, Q, lam, pr.warm_iters, pr.step_s, pr.tol, pr.loss, &itw, &r0,
                       e, lane);
    if (conv) {
      *iters = itw;
      return AEQC_ST_CONVERGED;
    }
    double rw = e.res;
    if (!isfinite(rw) || !isfinite(r0) || rw > pr.warm_reject || rw > r0) {
      st |= AEQC_ST_WARM_REJECTED;
#pragma unroll
      for (int k = 0; k < 4; ++k) lam[k] = 0.0;
      conv = round1_warp(g, w, Q, lam, pr.max_iter, pr.step_s, pr.tol, pr.loss, &it1,
                         &rdummy, e, lane);
    } else {
      conv = round1_warp(g, w, Q, lam, pr.max_iter - pr.warm_iters, pr.step_s, pr.tol,
                         pr.loss, &it1, &rdummy, e, lane);
    }
  } else {
#pragma unroll
    for (int k = 0; k < 4; ++k) lam[k] = 0.0;
    conv = round1_warp(g, w, Q, lam, pr.max_iter, pr.step_s, pr.tol, pr.loss, &it1, &r0, e,
                       lane);
  }
  if (conv) {
    *iters = itw + it1;
    return st | AEQC_ST_CONVERGED;
  }
  conv = round2_warp(g, w, Q, lam, pr.r2_max_iter, pr.tol, pr.loss, &it2, e, lane);
  *iters = itw + it1 + it2;
  if (conv) return st | AEQC_ST_ROUND2;
  return st | AEQC_ST_ROUND2 | NOT_CONVERGED;
}

// Quantize the histogram in xs against xhat row xh into w.codes / w.xp.
// Returns status bits CODE_ESCAPE / AE_EXACT.
__device__ unsigned quantize_warp(const GridK& g, WS& w, const float* xh, double dl,
                                  int lane) {
  int esc = 0, nonzero = 0;
  for (int p = lane; p < g.P; p += 32) {
    double xp;
    int c = quant_point_fp64(w.xs[p], (double)__ldg(xh + p), dl, &xp);
    w.codes[p] = (int16_t)c;
    w.xp[p] = xp;
    esc |= c == AEQC_CODE_ESCAPE;
    nonzero |= c != 0;
  }
  __syncwarp();
  unsigned st = 0;
  if (__any_sync(FULL, esc)) st |= AEQC_ST_CODE_ESCAPE;
  if (!__any_sync(FULL, nonzero)) st |= AEQC_ST_AE_EXACT;
  return st;
}

__device__ void process_fp64(const FusedArgs& a, WS& w, long long b, int lane) {
  const GridK& g = a.grid;
  const ParamsK& pr = a.prm;
  const int P = g.P;
  const double* xb = a.x + b * (long long)P;
  double s = 0.0;
  int bad = 0;
  for (int p = lane; p < P; p += 32) {
    double v = __ldg(xb + p);
    w.xs[p] = v;
    if (!isfinite(v) || v < 0.0) bad = 1;
    else if (v > s) s = v;
  }
  s = wmax(s);
  bad = __any_sync(FULL, bad);
  __syncwarp();

  unsigned st = 0;
  double lam[4] = {0.0, 0.0, 0.0, 0.0};
  int total_it = 0;
  double dfeat[4] = {0.0, 0.0, 0.0, 0.0};
  bool verbatim = false, zero = false;
  if (bad) {
    st = AEQC_ST_NONFINITE_INPUT | AEQC_ST_VERBATIM;
    verbatim = true;
  } else if (s == 0.0) {
    st = AEQC_ST_ZERO_IMAGE;
    zero = true;
    for (int p = lane; p < P; p += 32) {
      w.codes[p] = 0;
      w.xp[p] = 0.0;
    }
  } else {
    double Q[4], Sx[4];
    moments_warp(g, w.xs, Q, Sx, lane);
    bool done = false;
    for (int level = 0; level < 2 && !done; ++level) {
      double alpha = level ? pr.alpha * 0.25 : pr.alpha;
      double dl = bin_width(pr.tau, s, alpha);
      unsigned qs = quantize_warp(g, w, a.xhat + b * a.ldx, dl, lane);
      st = qs | (level ? AEQC_ST_ALPHA_RETRY : 0u) | (st & AEQC_ST_WARM_REJECTED);
      Eval e;
      int warm = 0;
      if (level == 0 && (a.features || a.use_mlp)) {
        eval_warp(g, w, lam, Q, pr.loss, false, e, lane);  // lam == 0 here
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          double den = e.S[k] > 0.0 ? e.S[k] : 1e-300;
          dfeat[k] = (Q[k] - e.A[k]) / den;
        }
        if (a.use_mlp) {
          const int L = a.latent.L;
          mlp_eval_warp(
              a.mlp,
              [&](int k) { return k < L ? load_latent(a.latent, b, k) : (float)dfeat[k - L]; },
              lam, lane);
          warm = 1;
          bool ok = true;
#pragma unroll
          for (int k = 0; k < 4; ++k) ok = ok && isfinite(lam[k]);
          if (!ok) {
#pragma unroll
            for (int k = 0; k < 4; ++k) lam[k] = 1e300;  // rejected by the probation
          }
        }
      }
      int it = 0;
      unsigned ns = newton_warp(g, w, Q, lam, warm, pr, &it, e, lane);
      total_it += it;
      st |= ns & 0x7fffu;
      if (ns & NOT_CONVERGED) break;
      // end-to-end check: |f - x| <= e at every point, moments within qoi_check
      double ebound = __dmul_rn(pr.tau, s);
      int viol = 0;
      PointIter pi(lane, g.n_par);
      for (; pi.p < P; pi.next()) {
        double f = pr.loss == 0 ? corr_kl(w.xp[pi.p], w.ta[pi.i], w.tb[pi.j])
                                : corr_l2(w.xp[pi.p], lam, g.vpar[pi.i], g.vperp2[pi.j]);
        viol |= !(fabs(f - w.xs[pi.p]) <= ebound);
      }
      bool ok = !__any_sync(FULL, viol);
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        double den = Sx[k] > 0.0 ? Sx[k] : 1e-300;
        ok = ok && (fabs(e.A[k] - Q[k]) / den <= pr.qoi_check);
      }
      if (ok) done = true;
    }
    if (!done) {
      st = (st & AEQC_ST_WARM_REJECTED) | AEQC_ST_VERBATIM | (st & AEQC_ST_ALPHA_RETRY) |
           (st & AEQC_ST_ROUND2);
      verbatim = true;
    }
  }
  if (verbatim) {
    for (int p = lane; p < P; p += 32) {
      w.codes[p] = AEQC_CODE_ESCAPE;
      w.xp[p] = w.xs[p];
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) lam[k] = 0.0;
  }
  __syncwarp();
  // outputs
  int16_t* cb = a.codes + b * (long long)P;
  for (int p = lane; p < P; p += 32) cb[p] = w.codes[p];
  if (a.f_out) {
    double* fb = a.f_out + b * (long long)P;
    PointIter pi(lane, g.n_par);
    for (; pi.p < P; pi.next()) {
      double f;
      if (verbatim) f = w.xs[pi.p];
      else if (zero) f = 0.0;
      else if (pr.loss == 0) f = corr_kl(w.xp[pi.p], w.ta[pi.i], w.tb[pi.j]);
      else f = corr_l2(w.xp[pi.p], lam, g.vpar[pi.i], g.vperp2[pi.j]);
      fb[pi.p] = f;
    }
  }
  if (a.out.count && (verbatim || (st & AEQC_ST_CODE_ESCAPE))) {
    if (append_outliers(a.out, w.codes, w.xs, P, a.row0 + b, lane))
      st |= AEQC_ST_OUTLIER_OVERFLOW;
  }
  if (a.features) {
    float* fr = a.features + b * (long long)(a.latent.L + 4);
    for (int l = lane; l < a.latent.L; l += 32) fr[l] = load_latent(a.latent, b, l);
    if (lane < 4) fr[a.latent.L + lane] = (float)dfeat[lane];
  }
  if (lane == 0) {
    a.scale[b] = s;
    a.iters[b] = (uint8_t)(total_it > 255 ? 255 : total_it);
    a.status[b] = (uint16_t)st;
#pragma unroll
    for (int k = 0; k < 4; ++k) a.lambda[b * 4 + k] = lam[k];
  }
  __syncwarp();
}

__global__ void __launch_bounds__(WPC * 32) fused_fp64_kernel(const FusedArgs a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  WS& w = reinterpret_cast<WS*>(smem_raw)[threadIdx.x >> 5];
  const int lane = threadIdx.x & 31;
  const long long nw = (long long)gridDim.x * WPC;
  for (long long b = (long long)blockIdx.x * WPC + (threadIdx.x >> 5); b < a.n; b += nw)
    process_fp64(a, w, b, lane);
}

// The same per-histogram work for the histograms listed by the fast kernel
// (list[0 .. *count)); entries that the cluster kernel below has completed are
// negative.  A launch with nothing to do returns at once.
__global__ void __launch_bounds__(WPC * 32) fused_fp64_list_kernel(const FusedArgs a,
                                                                   const int* list,
                                                                   const int* count) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  WS& w = reinterpret_cast<WS*>(smem_raw)[threadIdx.x >> 5];
  const int lane = threadIdx.x & 31;
  const long long cnt = *count;
  const long long nw = (long long)gridDim.x * WPC;
  for (long long t = (long long)blockIdx.x * WPC + (threadIdx.x >> 5); t < cnt; t += nw) {
    const int b = list[t];
    if (b >= 0) process_fp64(a, w, b, lane);
  }
}

// ---- a few histograms at once: a cluster of SMs each ------------------------------
// One warp takes about 20,000 FP64 instructions for a histogram, and a quarter
// of an SM issues one in 64 cycles: 0.67 ms, whatever else the chip does.  The
// fast kernel defers a handful of histograms in a hundred thousand, and a
// small batch has fewer histograms than the chip has SMs, so here a cluster of
// CL blocks takes one histogram, a thread per point.  The sums are those of
// the warp form to the bit, so that a histogram's result does not depend on
// how many others its call has: each of the twelve different sums belongs to
// one warp, whose lane l adds the terms of the points l, l + 32, ... in that
// order; the terms come from the blocks of the points through the cluster's
// shared memory, every block summing one kind of term.  The last block solves
// for the step (chol_solve4's operations, a row of the matrix a lane) and
// sends it to the others.  Only the ordinary course is handled: a histogram
// with non-finite, negative or no input, one that round 1 does not solve, warm
// starts, features, volumes per cell and the L2 loss are left to the warp
// kernels.  What bounds it is the latency of a step: three cluster barriers,
// 48 dependent additions, and the solution's square roots and divisions.  FP64
// form of n histograms of 39 x 39 (tau = 1e-3), a cluster / a warp each: n = 1
// 66 / 348 us, 16 80 / 445, 64 145 / 731, 128 218 / 730, 320 497 / 731 us.
constexpr int CL = 8;
constexpr int CT = AEQC_MAX_P / CL;  // threads of a block: a point each
constexpr int CWARPS = CT / 32;
constexpr unsigned SOLVER = CL - 1;
static_assert(CT % 32 == 0 && CT >= AEQC_MAX_NPAR && CL * CWARPS <= 64, "block shape");

// A_k (= S_k but for k = 1), S_1 and the entries of M that are no A_k (M11 = M03)
enum Sum { A0, A1, A2, A3, S1, M02, M03, M12, M13, M22, M23, M33, SUMS };
enum Weight { ONE, V, ABSV, W };

struct ClusterShared {
  double val[AEQC_MAX_P];  // the terms that this block sums
  double v[AEQC_MAX_NPAR], av[AEQC_MAX_NPAR], w[AEQC_MAX_NPERP];  // v, |v|, v_perp^2
  double ta[AEQC_MAX_NPAR], tb[AEQC_MAX_NPERP];
  unsigned long long umax[CL * CWARPS];
  unsigned flags[CL * CWARPS];
  long long base;
  double lam[4];
  double tot[SUMS], Q[4], S1;  // block SOLVER only
  int verdict;
};

__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ unsigned cluster_rank() {
  unsigned r;
  asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
// address of *p in block r's shared memory
__device__ __forceinline__ unsigned remote(const void* p, unsigned r) {
  unsigned a;
  asm("mapa.shared::cluster.u32 %0, %1, %2;"
      : "=r"(a)
      : "r"((unsigned)__cvta_generic_to_shared(p)), "r"(r));
  return a;
}
__device__ __forceinline__ void put_u64(const void* p, unsigned r, unsigned long long v) {
  asm volatile("st.shared::cluster.u64 [%0], %1;" ::"r"(remote(p, r)), "l"(v) : "memory");
}
__device__ __forceinline__ void put_f64(const double* p, unsigned r, double v) {
  put_u64(p, r, (unsigned long long)__double_as_longlong(v));
}
__device__ __forceinline__ void put_u32(const void* p, unsigned r, unsigned v) {
  asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(remote(p, r)), "r"(v) : "memory");
}

__device__ __forceinline__ void load_weights(const GridK& g, ClusterShared& sh) {
  const int t = threadIdx.x;
  if (t < g.n_par) {
    sh.v[t] = g.vpar[t];
    sh.av[t] = fabs(g.vpar[t]);
  }
  if (t < g.n_perp) sh.w[t] = g.vperp2[t];
}

// The terms of point p (y = vol f) to the blocks that sum them
template <bool MATRIX>
__device__ __forceinline__ void send_terms(const ClusterShared& sh, int p, double y, double v,
                                           double v2) {
  const Products t = products_of(y, v, v2);
  put_f64(&sh.val[p], 0, y);
  put_f64(&sh.val[p], 1, y);
  put_f64(&sh.val[p], 2, t.v);
  if (MATRIX) {
    put_f64(&sh.val[p], 3, t.v);
    put_f64(&sh.val[p], 4, t.w);
    put_f64(&sh.val[p], 5, t.vv);
    put_f64(&sh.val[p], 6, t.vvv);
  }
}

// sums of blocks 0 .. 6 (a warp each) and the weights of their terms
__constant__ signed char SUM_OF[2][CL] = {{A0, S1, A1, M12, M02, M03, M13, -1},
                                          {A2, -1, A3, -1, M22, M23, M33, -1}};
__constant__ signed char WEIGHT_OF[2][CL] = {{ONE, ABSV, ONE, W, ONE, ONE, ONE, ONE},
                                             {W, ONE, V, ONE, W, W, V, ONE}};

// The sums (those up to `last`) of the terms sent before, to block SOLVER.  With the
// weight one the fused product is the plain sum.
__device__ __forceinline__ void sum_terms(const GridK& g, ClusterShared& sh, unsigned rank,
                                          int last) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  cluster_sync();
  const int sum = warp < 2 ? SUM_OF[warp][rank] : -1;
  if (sum >= 0 && sum <= last) {
    const int wt = WEIGHT_OF[warp][rank];
    const double* tab = wt == W ? sh.w : (wt == V ? sh.v : sh.av);
    double acc = 0.0;
    PointIter it(lane, g.n_par);
#pragma unroll 4
    for (; it.p < g.P; it.next())
      acc = __fma_rn(sh.val[it.p], wt == ONE ? 1.0 : tab[wt == W ? it.j : it.i], acc);
    acc = wsum(acc);
    if (lane == 0) put_f64(&sh.tot[sum], SOLVER, acc);
  }
  cluster_sync();
}

// chol_solve4 for the matrix of sh.tot with a row a lane: lanes 0 to 3 hold the
// rows of L, lane 4 the forward solution of the right-hand side (lane k's gk is
// its component k), which the same operations produce.  All lanes return d.
__device__ __forceinline__ int solve_rows(const ClusterShared& sh, double gk, double (&d)[4],
                                          int lane) {
  const int ix[4][4] = {{A0, A1, M02, M03}, {A1, M03, M12, M13}, {M02, M12, M22, M23},
                        {M03, M13, M23, M33}};
  double L[4], diag[4];
#pragma unroll
  for (int l = 0; l < 4; ++l) {
    const double rhs = __shfl_sync(FULL, gk, l);
    double t = sh.tot[lane == 0 ? ix[0][l] : (lane == 1 ? ix[1][l] : (lane == 2 ? ix[2][l]
                                                                                : ix[3][l]))];
    if (lane == 4) t = rhs;
#pragma unroll
    for (int q = 0; q < l; ++q) t = __fma_rn(-L[q], __shfl_sync(FULL, L[q], l), t);
    const double pivot = __shfl_sync(FULL, t, l);
    if (!(pivot > 0.0)) return -1;
    diag[l] = __dsqrt_rn(pivot);
    L[l] = __ddiv_rn(lane > l && lane <= 4 ? t : diag[l], diag[l]);
    if (lane == l) L[l] = diag[l];
  }
#pragma unroll
  for (int k = 3; k >= 0; --k) {
    double t = __shfl_sync(FULL, L[k], 4);
#pragma unroll
    for (int q = k + 1; q < 4; ++q) t = __fma_rn(-__shfl_sync(FULL, L[k], q), d[q], t);
    d[k] = __ddiv_rn(t, diag[k]);
  }
#pragma unroll
  for (int k = 0; k < 4; ++k)
    if (!isfinite(d[k])) return -1;
  return 0;
}

// CONVERGED: and the moments within qoi_check; MOMENTS_OFF: converged, but not that
enum { STEP = 0, CONVERGED = 1, MOMENTS_OFF = 2, GIVE_UP = 3 };

// One turn of round1_warp on the sums, by the first warp of block SOLVER: the
// verdict and the next multipliers to every block.
__device__ __forceinline__ void decide(const ParamsK& pr, ClusterShared& sh, int it, int lane) {
  const int k = lane & 3;
  const double A = sh.tot[k], Q = sh.Q[k], gk = __dsub_rn(A, Q);
  const double S = k == 1 ? sh.tot[S1] : A;
  int verdict = STEP;
  double next = 0.0;
  if (!__all_sync(FULL, isfinite(gk) && isfinite(S))) {
    verdict = GIVE_UP;
  } else {
    const double r = __ddiv_rn(fabs(gk), S > 0.0 ? S : 1e-300);
    if (!__all_sync(FULL, isfinite(r))) {
      verdict = GIVE_UP;
    } else if (__all_sync(FULL, r <= pr.tol)) {
      const double den = k == 1 ? sh.S1 : Q;
      verdict = __all_sync(FULL, __ddiv_rn(fabs(gk), den > 0.0 ? den : 1e-300) <= pr.qoi_check)
                    ? CONVERGED
                    : MOMENTS_OFF;
    } else if (it == pr.max_iter) {
      verdict = GIVE_UP;
    } else {
      double d[4];
      if (solve_rows(sh, gk, d, lane) != 0) verdict = GIVE_UP;
      else
        next = __fma_rn(pr.step_s, k == 0 ? d[0] : (k == 1 ? d[1] : (k == 2 ? d[2] : d[3])),
                        sh.lam[k]);
    }
  }
  __syncwarp();  // lam and tot have been read
  if (verdict == STEP) put_f64(&sh.lam[k], lane >> 2, next);
  if (lane < CL) put_u32(&sh.verdict, lane, (unsigned)verdict);
}

// One histogram by the cluster; false when it is left to the warp kernels.
__device__ bool process_cluster(const FusedArgs& a, ClusterShared& sh, long long b,
                                unsigned rank) {
  const GridK& g = a.grid;
  const ParamsK& pr = a.prm;
  const int P = g.P, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int cw = (int)rank * CWARPS + warp;  // the warp in the cluster
  const int p = (int)rank * CT + tid;
  const bool in = p < P;
  const int j = in ? p / g.n_par : 0, i = in ? p - j * g.n_par : 0;
  const int j0 = (int)rank * CT / g.n_par;  // first row of this block's points
  const double v = g.vpar[i], v2 = g.vperp2[j], vol = g.vol_uniform;
  const double x = in ? __ldg(a.x + b * (long long)P + p) : 0.0;
  const float xh = in ? __ldg(a.xhat + b * a.ldx + p) : 0.f;
  // maximum and validity on the bit patterns: finite values from +0 up; -0 is 0
  {
    const unsigned long long u = (unsigned long long)__double_as_longlong(x);
    const bool fine = u <= 0x7FEFFFFFFFFFFFFFull;
    unsigned long long um = fine ? u : 0ull;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const unsigned long long t = __shfl_xor_sync(FULL, um, o);
      um = t > um ? t : um;
    }
    // a value that is not valid shows as the largest pattern
    if (__any_sync(FULL, !fine && u != 0x8000000000000000ull)) um = ~0ull;
    if (lane < CL) put_u64(&sh.umax[cw], lane, um);
  }
  cluster_sync();
  unsigned long long us = 0;
  for (int w = 0; w < CL * CWARPS; ++w) us = sh.umax[w] > us ? sh.umax[w] : us;
  if (us == ~0ull || us == 0) return false;  // the same in every block
  const double s = __longlong_as_double((long long)us), ebound = __dmul_rn(pr.tau, s);
  // Q_k and S_1 of x (x >= 0: S_k = Q_k for the others)
  if (in) send_terms<false>(sh, p, __dmul_rn(vol, x), v, v2);
  sum_terms(g, sh, rank, S1);
  if (rank == SOLVER && warp == 0) {
    if (lane < 4) sh.Q[lane] = sh.tot[lane];
    if (lane == 4) sh.S1 = sh.tot[S1];
    __syncwarp();
  }
  unsigned st = 0;
  int total_it = 0, code = 0, escapes = 0, before = 0;
  double xp = 0.0, f = 0.0;
  bool done = false;
  for (int level = 0; level < 2 && !done; ++level) {
    const double dl = bin_width(pr.tau, s, level ? pr.alpha4 : pr.alpha);
    code = in ? quant_point_fp64(x, (double)xh, dl, &xp) : 0;
    if (tid < 4) sh.lam[tid] = 0.0;
    int verdict = STEP;
    for (int it = 0; verdict == STEP; ++it) {
      __syncthreads();
      // tables of this lambda: the columns, and the rows of this block's points
      const double lam[4] = {sh.lam[0], sh.lam[1], sh.lam[2], sh.lam[3]};
      if (tid < g.n_par) sh.ta[tid] = corr_a(lam, g.vpar[tid]);
      const int jt = j0 + CT - 1 - tid;  // from the block's last thread down
      if (jt >= j0 && jt < g.n_perp && jt <= (int)((rank + 1) * CT - 1) / g.n_par)
        sh.tb[jt] = corr_b(lam, g.vperp2[jt]);
      __syncthreads();
      f = in ? corr_kl(xp, sh.ta[i], sh.tb[j]) : 0.0;
      if (in) send_terms<true>(sh, p, __dmul_rn(f, vol), v, v2);
      sum_terms(g, sh, rank, M33);
      if (rank == SOLVER && warp == 0) decide(pr, sh, it, lane);
      cluster_sync();
      verdict = sh.verdict;
      if (verdict != STEP) total_it += it;
    }
    if (verdict == GIVE_UP) return false;
    // end-to-end check: what each warp of the cluster found
    const unsigned esc = __ballot_sync(FULL, in && code == AEQC_CODE_ESCAPE);
    const int viol = __any_sync(FULL, in && !(fabs(f - x) <= ebound));
    const int nonzero = __any_sync(FULL, in && code != 0);
    if (lane < CL)
      put_u32(&sh.flags[cw], lane,
              (unsigned)__popc(esc) | (viol ? 256u : 0u) | (nonzero ? 512u : 0u));
    cluster_sync();
    const unsigned f0 = sh.flags[lane], f1 = lane + 32 < CL * CWARPS ? sh.flags[lane + 32] : 0u;
    escapes = __reduce_add_sync(FULL, (int)(f0 & 255u) + (int)(f1 & 255u));
    before = __reduce_add_sync(FULL, (lane < cw ? (int)(f0 & 255u) : 0) +
                                         (lane + 32 < cw ? (int)(f1 & 255u) : 0));
    st = AEQC_ST_CONVERGED | (level ? AEQC_ST_ALPHA_RETRY : 0u) |
         (escapes > 0 ? AEQC_ST_CODE_ESCAPE : 0u) |
         (__any_sync(FULL, (f0 | f1) & 512u) ? 0u : AEQC_ST_AE_EXACT);
    done = verdict == CONVERGED && !__any_sync(FULL, (f0 | f1) & 256u);
  }
  if (!done) {
    st = AEQC_ST_VERBATIM | AEQC_ST_ALPHA_RETRY;
    code = AEQC_CODE_ESCAPE;
    f = x;
    escapes = P;
    before = (int)rank * CT + 32 * warp;
  }
  const long long o = b * (long long)P + p;
  if (in) a.codes[o] = (int16_t)code;
  if (in && a.f_out) a.f_out[o] = f;
  if (a.out.count && escapes > 0) {
    // positions in the outlier list: one range per histogram, in point order
    const unsigned m = __ballot_sync(FULL, in && code == AEQC_CODE_ESCAPE);
    if (rank == 0 && tid == 0) {
      const unsigned long long base =
          atomicAdd((unsigned long long*)a.out.count, (unsigned long long)escapes);
      for (unsigned r = 0; r < CL; ++r) put_u64(&sh.base, r, base);
    }
    cluster_sync();
    const long long pos = sh.base + before + __popc(m & ((1u << lane) - 1u));
    if (in && code == AEQC_CODE_ESCAPE && pos < a.out.capacity) {
      a.out.index[pos] = (a.row0 + b) * (long long)P + p;
      a.out.value[pos] = x;
    }
    if (sh.base + escapes > a.out.capacity) st |= AEQC_ST_OUTLIER_OVERFLOW;
  }
  if (rank == 0 && tid < 4) a.lambda[b * 4 + tid] = done ? sh.lam[tid] : 0.0;
  if (rank == 0 && tid == 0) {
    a.scale[b] = s;
    a.iters[b] = (uint8_t)(total_it > 255 ? 255 : total_it);
    a.status[b] = (uint16_t)st;
  }
  return true;
}

// The histograms list[0 .. *count) when there are at most `most` of them, one
// cluster each at a time; completed entries become negative.  all != 0: the
// list is written here, 0 .. all - 1, with its count.
__global__ void __cluster_dims__(CL, 1, 1) __launch_bounds__(CT, 3)
    fused_fp64_cluster_kernel(const __grid_constant__ FusedArgs a, int* list, int* count, int most,
                              int all) {
  __shared__ ClusterShared sh;
  const unsigned rank = cluster_rank();
  const int cnt = all ? all : *count;
  if (cnt > most) return;  // the same in every block
  // A block's shared memory may be written by another one only once it is known
  // to have started, which a barrier of the cluster shows and nothing else does
  // (process_cluster writes into all eight blocks before its first barrier).
  cluster_sync();
  load_weights(a.grid, sh);
  const int nc = gridDim.x / CL;
  if (all && blockIdx.x == 0 && threadIdx.x == 0) *count = all;
  for (int t = blockIdx.x / CL; t < cnt; t += nc) {
    const int b = all ? t : list[t];
    const bool done = process_cluster(a, sh, b, rank);
    // the blocks leave the histogram together: nobody writes into the shared
    // memory of one that still reads, or has ended; and every block has read
    // the entry before it changes
    cluster_sync();
    if (rank == 0 && threadIdx.x == 0) list[t] = done ? -1 : b;
  }
}

// what the cluster kernel handles
bool cluster_form(const FusedArgs& a) {
  return a.prm.loss == 0 && !a.grid.has_vol && !a.use_mlp && !a.features && a.fb_list &&
         a.fb_count;
}

// ---- single-stage kernels for the separate C-ABI calls ---------------------

__global__ void __launch_bounds__(128) moments_kernel(const GridK g, const double* x,
                                                      long long n, double* Q) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  double* xs = reinterpret_cast<double*>(smem_raw) + (threadIdx.x >> 5) * AEQC_MAX_P;
  const int lane = threadIdx.x & 31;
  const long long nw = (long long)gridDim.x * 4;
  for (long long b = (long long)blockIdx.x * 4 + (threadIdx.x >> 5); b < n; b += nw) {
    for (int p = lane; p < g.P; p += 32) xs[p] = __ldg(x + b * g.P + p);
    __syncwarp();
    double q[4], sabs[4];
    moments_warp(g, xs, q, sabs, lane);
    if (lane < 4) Q[b * 4 + lane] = q[lane];
    __syncwarp();
  }
}

struct QuantArgs {
  const double* x;
  const float* xhat;
  long long ld, n;
  int P;
  ParamsK prm;
  int16_t* codes;
  double* scale;
  uint16_t* status;
  OutliersK out;
  double* xrec;
};

__global__ void __launch_bounds__(128) quantize_kernel(const QuantArgs a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int lane = threadIdx.x & 31;
  int16_t* codes_s = reinterpret_cast<int16_t*>(smem_raw) + (threadIdx.x >> 5) * AEQC_MAX_P;
  double* raw = reinterpret_cast<double*>(smem_raw + 4 * AEQC_MAX_P * sizeof(int16_t)) +
                (threadIdx.x >> 5) * AEQC_MAX_P;
  const long long nw = (long long)gridDim.x * 4;
  for (long long b = (long long)blockIdx.x * 4 + (threadIdx.x >> 5); b < a.n; b += nw) {
    const double* xb = a.x + b * a.P;
    double s = 0.0;
    int bad = 0;
    for (int p = lane; p < a.P; p += 32) {
      double v = __ldg(xb + p);
      raw[p] = v;
      if (!isfinite(v) || v < 0.0) bad = 1;
      else if (v > s) s = v;
    }
    s = wmax(s);
    bad = __any_sync(FULL, bad);
    __syncwarp();
    unsigned st = 0;
    if (bad) {
      st = AEQC_ST_NONFINITE_INPUT | AEQC_ST_VERBATIM;
      for (int p = lane; p < a.P; p += 32) codes_s[p] = AEQC_CODE_ESCAPE;
      if (a.xrec)
        for (int p = lane; p < a.P; p += 32) a.xrec[b * a.P + p] = raw[p];
    } else if (s == 0.0) {
      st = AEQC_ST_ZERO_IMAGE;
      for (int p = lane; p < a.P; p += 32) {
        codes_s[p] = 0;
        if (a.xrec) a.xrec[b * a.P + p] = 0.0;
      }
    } else {
      double dl = bin_width(a.prm.tau, s, a.prm.alpha);
      int esc = 0, nonzero = 0;
      for (int p = lane; p < a.P; p += 32) {
        double xp;
        int c = quant_point_fp64(raw[p], (double)__ldg(a.xhat + b * a.ld + p), dl, &xp);
        codes_s[p] = (int16_t)c;
        if (a.xrec) a.xrec[b * a.P + p] = xp;
        esc |= c == AEQC_CODE_ESCAPE;
        nonzero |= c != 0;
      }
      if (__any_sync(FULL, esc)) st |= AEQC_ST_CODE_ESCAPE;
      if (!__any_sync(FULL, nonzero)) st |= AEQC_ST_AE_EXACT;
    }
    __syncwarp();
    for (int p = lane; p < a.P; p += 32) a.codes[b * a.P + p] = codes_s[p];
    if (a.out.count && (st & (AEQC_ST_CODE_ESCAPE | AEQC_ST_VERBATIM))) {
      if (append_outliers(a.out, codes_s, raw, a.P, b, lane)) st |= AEQC_ST_OUTLIER_OVERFLOW;
    }
    if (lane == 0) {
      a.scale[b] = s;
      a.status[b] = (uint16_t)st;
    }
    __syncwarp();
  }
}

// x' from codes (thread per value); escapes are filled by scatter_raw_kernel.
__global__ void dequantize_kernel(const float* xhat, long long ld, const int16_t* codes,
                                  const double* scale, const uint16_t* status, long long n,
                                  int P, ParamsK prm, double* xrec) {
  long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  long long total = n * (long long)P;
  for (; t < total; t += (long long)gridDim.x * blockDim.x) {
    long long b = t / P;
    int p = (int)(t - b * P);
    unsigned st = status[b];
    int c = codes[t];
    double v;
    if (st & AEQC_ST_ZERO_IMAGE) v = 0.0;
    else if (c == AEQC_CODE_ESCAPE) continue;
    else if (c == AEQC_CODE_ZERO) v = 0.0;
    else {
      double alpha = (st & AEQC_ST_ALPHA_RETRY) ? prm.alpha * 0.25 : prm.alpha;
      double dl = bin_width(prm.tau, scale[b], alpha);
      v = __dadd_rn((double)xhat[b * ld + p], __dmul_rn((double)c, dl));
    }
    xrec[t] = v;
  }
}

__global__ void scatter_raw_kernel(const OutliersK o, long long total, double* xrec) {
  long long cnt = *o.count;
  if (cnt > o.capacity) cnt = o.capacity;
  for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < cnt;
       t += (long long)gridDim.x * blockDim.x) {
    long long i = o.index[t];
    if (i >= 0 && i < total) xrec[i] = o.value[t];
  }
}

struct NewtonArgs {
  GridK g;
  const double* xrec;
  const double* Q;
  long long n;
  ParamsK prm;
  int use_warm;
  double* lambda;
  double* f_out;
  uint8_t* iters;
  uint16_t* status;
};

__global__ void __launch_bounds__(WPC * 32) newton_kernel(const NewtonArgs a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  WS& w = reinterpret_cast<WS*>(smem_raw)[threadIdx.x >> 5];
  const int lane = threadIdx.x & 31;
  const GridK& g = a.g;
  const long long nw = (long long)gridDim.x * WPC;
  for (long long b = (long long)blockIdx.x * WPC + (threadIdx.x >> 5); b < a.n; b += nw) {
    for (int p = lane; p < g.P; p += 32) w.xp[p] = __ldg(a.xrec + b * g.P + p);
    __syncwarp();
    double Q[4], lam[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      Q[k] = a.Q[b * 4 + k];
      lam[k] = a.use_warm ? a.lambda[b * 4 + k] : 0.0;
    }
    Eval e;
    int it = 0;
    unsigned st = newton_warp(g, w, Q, lam, a.use_warm, a.prm, &it, e, lane);
    if (a.f_out) {
      PointIter pi(lane, g.n_par);
      for (; pi.p < g.P; pi.next()) {
        double f = a.prm.loss == 0 ? corr_kl(w.xp[pi.p], w.ta[pi.i], w.tb[pi.j])
                                   : corr_l2(w.xp[pi.p], lam, g.vpar[pi.i], g.vperp2[pi.j]);
        a.f_out[b * g.P + pi.p] = f;
      }
    }
    if (lane == 0) {
#pragma unroll
      for (int k = 0; k < 4; ++k) a.lambda[b * 4 + k] = lam[k];
      a.iters[b] = (uint8_t)(it > 255 ? 255 : it);
      a.status[b] = (uint16_t)(st & 0x7fffu);
    }
    __syncwarp();
  }
}

// Decompression: f = x' exp(-lambda.phi) per value (warp per histogram for the
// exponential tables); escapes are written by scatter_corrected_kernel.
struct ApplyArgs {
  GridK g;
  const float* xhat;
  long long ld;
  const int16_t* codes;
  const double* scale;
  const double* lambda;
  const uint16_t* status;
  long long n;
  ParamsK prm;
  double* f;
};

// x' = fl(xhat + c dl) as a double without the FP64 pipe, dl = 2^k a normal
// float with room for c; false where the caller has to take the FP64 form.  The
// sum is the pair hi + lo exactly (Knuth's two-sum, |lo| <= half a last place of
// hi); lo in units of the double's last place, rounded half to even, is added to
// hi's bits.  That is the rounded sum as long as it stays in hi's binade, which
// it leaves only from a power of two downwards.
__device__ __forceinline__ bool level_value(int c, float xhat, float dl, double* out) {
  // float(c): 1.5 2^23 + c read off its bits
  const float cd = __fmul_rn(__fsub_rn(__int_as_float(0x4B400000 + c), 12582912.f), dl);
  const float hi = __fadd_rn(xhat, cd);
  const float bb = __fsub_rn(hi, xhat);
  const float lo = __fadd_rn(__fsub_rn(xhat, __fsub_rn(hi, bb)), __fsub_rn(cd, bb));
  const unsigned u = __float_as_uint(hi), E = u & 0x7f800000u;
  // 2^52 / 2^floor(log2 |hi|) with hi's sign
  const float sc = __uint_as_float((0x99000000u - E) ^ (u & 0x80000000u));
  const float t = __fmul_rn(lo, sc);  // |t| <= 2^28
  // round to nearest even in two steps of twelve and seventeen bits
  const float ma = fmaf(t, 1.f / 4096.f, 12582912.f);
  const float mb = __fadd_rn(fmaf(__fsub_rn(ma, 12582912.f), -4096.f, t), 12582912.f);
  const int n = (__float_as_int(ma) - 0x4B400000) * 4096 + (__float_as_int(mb) - 0x4B400000);
  const unsigned hw = (((u << 1) >> 4) + 0x38000000u) | (u & 0x80000000u);
  const unsigned long long r =
      (((unsigned long long)hw << 32) | (u << 29)) + (unsigned long long)(long long)n;
  *out = __longlong_as_double((long long)r);
  return E - (52u << 23) <= (202u << 23) && ((u << 9) != 0u || t >= 0.f);
}

// the same in FP64; a call, since inline it would be computed for every point
// and selected (the FP64 pipe then ran at 84 % and the kernel took 2.7 ms)
__device__ __noinline__ double level_value_fp64(int c, float xhat, double dl) {
  return __dadd_rn((double)xhat, __dmul_rn((double)c, dl));
}

// One column segment of a histogram: rows [j0, j1) of column i.  One point a
// turn, its operands loaded a row ahead.
__device__ __forceinline__ void apply_column(int i, int j0, int j1, int n_par, const int16_t* cb,
                                             const float* xb, double* fb, const double* ta,
                                             const double* tb, float dl_f, double dl) {
  if (j0 >= j1) return;
  const double ai = ta[i];
  int p = j0 * n_par + i;
  int cn = __ldg(cb + p);
  float hn = __ldg(xb + p);
#pragma unroll 1
  for (int j = j0; j < j1; ++j) {
    const int c = cn;
    const float xh = hn;
    const int q = p;
    p += n_par;
    if (j + 1 < j1) {
      cn = __ldg(cb + p);
      hn = __ldg(xb + p);
    }
    if (c == AEQC_CODE_ESCAPE) continue;  // scatter_corrected_kernel writes it
    double x;
    if (c == AEQC_CODE_ZERO) x = 0.0;
    else if (!level_value(c, xh, dl_f, &x)) x = level_value_fp64(c, xh, dl);
    fb[q] = corr_kl(x, ai, tb[j]);
  }
}

// One warp per histogram.  The FP64 form of a point is six instructions of the
// FP64 pipe (two conversions, the product with the bin width, the sum and the
// two factors), 4,600 cycles of an SM per histogram.  Here x' is put together on
// the FP32 and integer pipes with the same bits and the two factors are the FP64
// pipe's only work per point, 1,500 cycles, which bounds the kernel.  Each lane
// walks down columns, so that its factor in v_par stays in a register and the
// loop is short: a body that outgrows the instruction buffers costs more than
// its instructions (four points a turn with a 64-bit integer sum: 1,224 us for
// 150,001 histograms; this form 1,090 us, the FP64 pipe 78 % busy; the FP64
// form 4,060 us).
__global__ void __launch_bounds__(128, 10) apply_kernel(const __grid_constant__ ApplyArgs a) {
  __shared__ double ta[4][AEQC_MAX_NPAR], tb[4][AEQC_MAX_NPERP];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const GridK& g = a.g;
  const long long nw = (long long)gridDim.x * 4;
  // lane's columns: column `lane` of the first 32 (where there are as many), and
  // a chunk of rows of one of the rw others
  const int cw = g.n_par >= 32 ? 32 : 0, rw = g.n_par - cw;
  int c2 = 0, k0 = 0, k1 = 0;
  if (rw) {
    const int nchunk = 32 / rw, rpc = (g.n_perp + nchunk - 1) / nchunk;
    if (lane < rw * nchunk) {
      const int chunk = lane / rw;
      c2 = cw + lane - chunk * rw;
      k0 = chunk * rpc;
      k1 = min(g.n_perp, k0 + rpc);
    }
  }
  for (long long b = (long long)blockIdx.x * 4 + warp; b < a.n; b += nw) {
    const unsigned st = a.status[b];
    double lam[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) lam[k] = a.lambda[b * 4 + k];
    if (a.prm.loss == 0) {
      for (int i = lane; i < g.n_par; i += 32) ta[warp][i] = corr_a(lam, g.vpar[i]);
      for (int j = lane; j < g.n_perp; j += 32) tb[warp][j] = corr_b(lam, g.vperp2[j]);
    }
    __syncwarp();
    const bool zero = (st & AEQC_ST_ZERO_IMAGE) != 0;
    const double dl = (st & (AEQC_ST_ZERO_IMAGE | AEQC_ST_VERBATIM))
                          ? 0.0
                          : bin_width(a.prm.tau, a.scale[b],
                                      (st & AEQC_ST_ALPHA_RETRY) ? a.prm.alpha4 : a.prm.alpha);
    const int de = (int)((unsigned long long)__double_as_longlong(dl) >> 52);
    const int16_t* cb = a.codes + b * g.P;
    const float* xb = a.xhat + b * a.ld;
    double* fb = a.f + b * g.P;
    // the float form: dl = 2^k and c dl normal floats (a bin width is a power of
    // two or no normal number)
    if (a.prm.loss == 0 && de >= 1023 - 126 && de <= 1023 + 100) {
      const float dl_f = __int_as_float((de - 1023 + 127) << 23);
#pragma unroll 1
      for (int part = cw ? 0 : 1; part < 2; ++part)
        apply_column(part ? c2 : lane, part ? k0 : 0, part ? k1 : g.n_perp, g.n_par, cb, xb, fb,
                     ta[warp], tb[warp], dl_f, dl);
    } else {
      PointIter pi(lane, g.n_par);
#pragma unroll 1
      for (; pi.p < g.P; pi.next()) {
        const int c = __ldg(cb + pi.p);
        if (c == AEQC_CODE_ESCAPE && !zero) continue;
        const double xp = zero || c == AEQC_CODE_ZERO ? 0.0 : level_value_fp64(c, __ldg(xb + pi.p), dl);
        fb[pi.p] = a.prm.loss == 0 ? corr_kl(xp, ta[warp][pi.i], tb[warp][pi.j])
                                   : corr_l2(xp, lam, g.vpar[pi.i], g.vperp2[pi.j]);
      }
    }
    __syncwarp();
  }
}

struct ScatterArgs {
  GridK g;
  OutliersK o;
  const double* lambda;
  long long row0, n;
  int loss;
  double* f;
};

// raw values at escape points, with the histogram's correction applied
__global__ void scatter_corrected_kernel(const ScatterArgs a) {
  long long cnt = *a.o.count;
  if (cnt > a.o.capacity) cnt = a.o.capacity;
  const int P = a.g.P;
  for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < cnt;
       t += (long long)gridDim.x * blockDim.x) {
    long long idx = a.o.index[t] - a.row0 * P;
    if (idx < 0 || idx >= a.n * P) continue;
    long long b = idx / P;
    int p = (int)(idx - b * P);
    int j = p / a.g.n_par, i = p - j * a.g.n_par;
    double l[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) l[k] = a.lambda[b * 4 + k];
    a.f[idx] = a.loss == 0 ? corr_kl(a.o.value[t], corr_a(l, a.g.vpar[i]),
                                     corr_b(l, a.g.vperp2[j]))
                           : corr_l2(a.o.value[t], l, a.g.vpar[i], a.g.vperp2[j]);
  }
}

int grid_for(long long warps, int sm_mult = 8) {
  int dev = 0, sms = 148;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  long long blocks = (warps + 3) / 4;
  long long cap = (long long)sms * sm_mult;
  if (blocks > cap) blocks = cap;
  if (blocks < 1) blocks = 1;
  return (int)blocks;
}

}  // namespace

namespace {

// three blocks per SM (the launch bounds), at most one
// cluster per histogram
unsigned cluster_grid(long long most) {
  int dev = 0, sms = 148;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  long long c = (long long)sms * 3 / CL;
  if (c > most) c = most;
  return (unsigned)((c > 0 ? c : 1) * CL);
}

// Histograms of P points up to which the clusters take a call or a list for which
// there are as many warps as `warps`.  A cluster's time hardly depends on P (57 of
// them run at once, 1.1 to 2 us a histogram with the steps it takes); a warp's
// does, 104 to 158 us at P = 100, 172 to 270 at 400, 453 to 731 at 1,521, and is
// the call's time while there is a warp for each.  Over bounds from 1e-4 to 0.1
// the clusters were never slower up to 48 histograms at P = 64, 64 at 100, 96 at
// 225 and 400, 128 at 625, 160 at 900 and 200 at 1,221 and 1,521 (320 at 1,521:
// between 0.68 and 1.35 times a warp's time): the line runs below these.  A list
// in a small batch has few warps, whose work the clusters do faster at any number.
// Few points leave the system close to singular; what round 1 does not solve,
// the clusters try in vain and the warps do again (P = 20: 57 histograms 653
// instead of 411 us), so such grids go to the warps at once.
int cluster_most(int P, long long warps) {
  if (P < 64) return 0;
  const int line = 40 + P / 9;
  return warps < line ? 320 : line;
}

// the list kernel's blocks: sized for a few percent of the batch; the grid-stride
// loop covers any count
int list_blocks(long long n) { return grid_for(n / 16 + 1, 2); }

}  // namespace

static int launch_fused_fp64_rest(const FusedArgs& a, const int* list, const int* count,
                                  cudaStream_t s);

int launch_fused_fp64(const FusedArgs& a, cudaStream_t s) {
  if (a.n <= 0) return AEQC_OK;
  const int most = cluster_most(a.grid.P, a.n);
  if (a.n <= most && cluster_form(a)) {
    fused_fp64_cluster_kernel<<<cluster_grid(a.n), CT, 0, s>>>(a, a.fb_list, a.fb_count, most,
                                                               (int)a.n);
    int rc = check_launch("fused_fp64_cluster_kernel");
    return rc ? rc : launch_fused_fp64_rest(a, a.fb_list, a.fb_count, s);
  }
  size_t smem = sizeof(WS) * WPC;
  {
    const int rc_attr = raise_smem_limit((const void*)fused_fp64_kernel, (int)smem);
    if (rc_attr) return rc_attr;
  }
  fused_fp64_kernel<<<grid_for(a.n, 2), WPC * 32, smem, s>>>(a);
  return check_launch("fused_fp64_kernel");
}

int launch_fused_fp64_list(const FusedArgs& a, int* list, int* count, cudaStream_t s) {
  if (a.n <= 0) return AEQC_OK;
  const int most = cluster_most(a.grid.P, (long long)WPC * list_blocks(a.n));
  if (most > 0 && cluster_form(a)) {
    fused_fp64_cluster_kernel<<<cluster_grid(a.n), CT, 0, s>>>(a, list, count, most, 0);
    int rc = check_launch("fused_fp64_cluster_kernel");
    if (rc) return rc;
  }
  return launch_fused_fp64_rest(a, list, count, s);
}

static int launch_fused_fp64_rest(const FusedArgs& a, const int* list, const int* count,
                                  cudaStream_t s) {
  size_t smem = sizeof(WS) * WPC;
  {
    const int rc_attr = raise_smem_limit((const void*)fused_fp64_list_kernel, (int)smem);
    if (rc_attr) return rc_attr;
  }
  fused_fp64_list_kernel<<<list_blocks(a.n), WPC * 32, smem, s>>>(a, list, count);
  return check_launch("fused_fp64_list_kernel");
}

int launch_moments(const GridK& g, const double* x, long long n, double* Q, cudaStream_t s) {
  if (n <= 0) return AEQC_OK;
  size_t smem = 4 * AEQC_MAX_P * sizeof(double);
  {
    const int rc_attr = raise_smem_limit((const void*)moments_kernel, (int)smem);
    if (rc_attr) return rc_attr;
  }
  moments_kernel<<<grid_for(n, 4), 128, smem, s>>>(g, x, n, Q);
  return check_launch("moments_kernel");
}

int launch_quantize(const double* x, const float* xhat, long long ld, long long n, int P,
                    const ParamsK& prm, int16_t* codes, double* scale, uint16_t* status,
                    const OutliersK& out, double* xrec, cudaStream_t s) {
  if (n <= 0) return AEQC_OK;
  if (out.count) AEQC_CUDA_TRY(cudaMemsetAsync(out.count, 0, sizeof(long long), s));
  QuantArgs a{x, xhat, ld, n, P, prm, codes, scale, status, out, xrec};
  size_t smem = 4 * AEQC_MAX_P * (sizeof(int16_t) + sizeof(double));
  {
    const int rc_attr = raise_smem_limit((const void*)quantize_kernel, (int)smem);
    if (rc_attr) return rc_attr;
  }
  quantize_kernel<<<grid_for(n, 4), 128, smem, s>>>(a);
  return check_launch("quantize_kernel");
}

int launch_dequantize(const float* xhat, long long ld, const int16_t* codes,
                      const OutliersK* out, const double* scale, const uint16_t* status,
                      long long n, int P, const ParamsK& prm, double* xrec, cudaStream_t s) {
  if (n <= 0) return AEQC_OK;
  long long total = n * (long long)P;
  long long blocks = (total + 255) / 256;
  if (blocks > 65536) blocks = 65536;
  dequantize_kernel<<<(int)blocks, 256, 0, s>>>(xhat, ld, codes, scale, status, n, P, prm,
                                                xrec);
  int rc = check_launch("dequantize_kernel");
  if (rc != AEQC_OK) return rc;
  if (out && out->count) {
    scatter_raw_kernel<<<1024, 256, 0, s>>>(*out, total, xrec);
    rc = check_launch("scatter_raw_kernel");
  }
  return rc;
}

int launch_newton(const GridK& g, const double* xrec, const double* Q, long long n,
                  const ParamsK& prm, int use_warm, double* lambda, double* f_out,
                  uint8_t* iters, uint16_t* status, cudaStream_t s) {
  if (n <= 0) return AEQC_OK;
  NewtonArgs a{g, xrec, Q, n, prm, use_warm, lambda, f_out, iters, status};
  size_t smem = sizeof(WS) * WPC;
  {
    const int rc_attr = raise_smem_limit((const void*)newton_kernel, (int)smem);
    if (rc_attr) return rc_attr;
  }
  newton_kernel<<<grid_for(n, 2), WPC * 32, smem, s>>>(a);
  return check_launch("newton_kernel");
}

int launch_apply(const GridK& g, const float* xhat, long long ld, const int16_t* codes,
                 const OutliersK* out, const double* scale, const double* lambda,
                 const uint16_t* status, long long n, long long row0, const ParamsK& prm,
                 double* f, cudaStream_t s) {
  if (n <= 0) return AEQC_OK;
  ApplyArgs a{g, xhat, ld, codes, scale, lambda, status, n, prm, f};
  apply_kernel<<<grid_for(n, 10), 128, 0, s>>>(a);
  int rc = check_launch("apply_kernel");
  if (rc != AEQC_OK) return rc;
  if (out && out->count) {
    ScatterArgs sa{g, *out, lambda, row0, n, prm.loss, f};
    scatter_corrected_kernel<<<1024, 256, 0, s>>>(sa);
    rc = check_launch("scatter_corrected_kernel");
  }
  return rc;
}

}  // namespace aeqc
