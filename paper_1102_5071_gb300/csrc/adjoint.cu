// Backward (adjoint) sweep of the gradient of the fidelity loss
// L = 1 - |<phi|psi(T)>|^2 with respect to piecewise-constant drive amplitudes
// (FP64, sm_103a).  The paper has no gradients; the method is the chain rule
// through the CFET steps of Sec. 4 Eq. (Ucf) with the stage operators of
// Sec. 7 Eq. (OmGLeg):
//
//   d<phi|psi(T)>/dA_k = sum over stages (n, j) of segment k of
//       gamma_{n,j} <lambda_after| dE |psi_before>,
//   dE = d/dc exp(-i tau (c0 H0 + c V)) = -i tau int_0^1 e^{-i tau (1-s) H} V e^{-i tau s H} ds.
//
// With a(r) = e^{+i tau r H} psi_after (= e^{-i tau s H} psi_before, r = 1 - s)
// and b(r) = e^{+i tau r H} lambda_after the stage term is
//   -i tau int_0^1 <b(r)| V |a(r)> dr.
// Both families live in the Krylov spaces of psi_after and lambda_after
// (Sec. 8.1; a Krylov space does not depend on the time): a(r) =
// beta_a V_a exp(i tau r T_a) e_1 and likewise for b, so the integrand is
// y_b(r)^H W y_a(r) with W = V_b^H V V_a (k_b x k_a), integrated by
// Gauss-Legendre quadrature in r.  The same bases give psi_before = a(1) and
// lambda_before = b(1): the forward states are recovered by the inverse
// unitary step, and the driver replaces the recovered state by a stored
// checkpoint at every launch boundary (the drift is reported).
//
// One persistent cooperative launch undoes a range of stage exponentials, one CTA
// of 512 threads per SM.  The Lanczos processes of psi and lambda run jointly
// (one pass, one pair of reductions per iteration for both; warp 0 takes psi's
// scalars, warp 1 lambda's).  The quadrature needs only the two tridiagonal
// matrices, so its weights
//   C_ij = sum_q w_q conj(y_b,i(r_q)) y_a,j(r_q)
// are summed first (the nodes spread over the warps) and the stage integral is
// one pass over the elements,
//   sum_x sum_j (V q_j)(x) sum_i C_ij conj(l_i(x)),
// whose sum joins the reduction of the recovered states' norms: no Gram matrix,
// no reduction of its entries and no grid exchange for them.  Reductions are
// per-CTA trees, one record per CTA (ctl_exchange) and fixed-order sums, so every
// CTA holds identical scalars.
//
// Bound by the FP64 units (one warp instruction per 64 cycles and SM
// sub-partition): about 70 per element and Lanczos vector, 2 N + 4 k_l + 4 per
// element and column of the integral.  N = 16, 64 stage exponentials: see the
// time at k_adjoint.
#include <cuda_runtime.h>

#include <cmath>
#include <cstdint>

#include "cfet_internal.h"
#include "device_common.cuh"

namespace cfet {
namespace {

constexpr int kAdjWarps = kAdjThreads / 32;

struct SmemAdj {
  double red[kAdjWarps][8];
  double res[8];
  double alpha[2][kAdjMaxK + 2];
  double beta[2][kAdjMaxK + 2];
  double scale[2][kAdjMaxK + 3];
  double yr[2][kAdjMaxK], yi[2][kAdjMaxK];   // exp(+i tau T) e_1 (the inverse step)
  // per warp: y of a quadrature node (psi, lambda) and scratch of the small exponential
  double wyr[kAdjWarps][2][kAdjMaxK], wyi[kAdjWarps][2][kAdjMaxK];
  double wtr[kAdjWarps][kAdjMaxK], wti[kAdjWarps][kAdjMaxK];
  double2 C[kAdjMaxK][kAdjMaxK];             // [j][i]: weights of the stage integral
  double cre[2][kAdjMaxK], cim[2][kAdjMaxK];
  double bsite_raw[kMaxSites];
  double bsite[2][kMaxSites];
  double beta0[2];
  int k[2], active[2];
  int nq;   // Gauss-Legendre nodes of this stage integral (0: beyond the largest rule)
  int ok;
};

// Sums over the warp of P values per lane (P a power of two up to 8): lane l ends
// with the sum of value adj_value_of<P>(l), after P - 1 + (5 - log2 P) additions
// instead of 5 P (the FP64 pipe takes 64 cycles for each).
template <int P>
__device__ __forceinline__ double adj_warp_sum(double (&v)[P]) {
  const int lane = threadIdx.x & 31;
  int o = 16;
#pragma unroll
  for (int h = P / 2; h >= 1; h /= 2, o >>= 1) {
    const bool up = (lane & o) != 0;
#pragma unroll
    for (int i = 0; i < h; ++i) {
      const double keep = up ? v[i + h] : v[i], send = up ? v[i] : v[i + h];
      v[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
    }
  }
  double s = v[0];
  for (; o >= 1; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  return s;
}
// The value that lane l holds: its bits 4, 3, ... (log2 P of them), most significant first.
template <int P>
__device__ __forceinline__ int adj_value_of(int lane) {
  return P == 1 ? 0 : (P == 2 ? lane >> 4 : (P == 4 ? lane >> 3 : lane >> 2));
}

// Sum of two doubles per CTA record (fixed order per lane).
struct AdjAcc2 {
  double s[2];
  __device__ void reset() { s[0] = s[1] = 0.0; }
  __device__ void add(const unsigned (&v)[4]) {
    s[0] += __longlong_as_double((long long)(((unsigned long long)v[1] << 32) | v[0]));
    s[1] += __longlong_as_double((long long)(((unsigned long long)v[3] << 32) | v[2]));
  }
};

// Grid sums of P values per thread (P = 2, 4 or 8), two per exchange; results in
// S.res (all threads).  `fence`: vectors written before it are read by other CTAs after it.
template <int P>
__device__ bool adj_reduce(SmemAdj& S, double (&v)[P], bool fence, unsigned& tag, const AdjParams& p) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const double w = adj_warp_sum<P>(v);
  if ((lane & (32 / P - 1)) == 0) S.red[warp][adj_value_of<P>(lane)] = w;
  __syncthreads();
  if (warp == 0) {
    long long spin = 0;
    bool ok = true;
    for (int j = 0; j < P; j += 2) {
      // lanes 0..15 hold value j of the CTA's warps, lanes 16..31 value j + 1
      double c = S.red[lane & (kAdjWarps - 1)][j + (lane >> 4)];
#pragma unroll
      for (int o = 8; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
      const unsigned long long b0 = (unsigned long long)__double_as_longlong(__shfl_sync(0xffffffffu, c, 0));
      const unsigned long long b1 = (unsigned long long)__double_as_longlong(__shfl_sync(0xffffffffu, c, 16));
      const unsigned mine[4] = {(unsigned)b0, (unsigned)(b0 >> 32), (unsigned)b1, (unsigned)(b1 >> 32)};
      AdjAcc2 acc;
      ++tag;
      ok = ok && ctl_exchange<4>(reinterpret_cast<unsigned long long*>(p.partials), mine, tag, fence, &p.st->status,
                                 p.timeout_ns, spin, acc);
      const double t = adj_warp_sum<2>(acc.s);  // lanes 0..15: value j, lanes 16..31: value j + 1
      if ((lane & 15) == 0) S.res[j + (lane >> 4)] = t;
    }
    if (lane == 0) S.ok = ok;
  } else {
    tag += P / 2;
  }
  __syncthreads();
  return S.ok != 0;
}
static_assert(kAdjWarps == 16, "adj_reduce takes one value of 16 warps per half-warp");

// beta and the decision of Lanczos process pp at iteration it (one warp).
__device__ __noinline__ void adj_decide(SmemAdj& S, int pp, int it, double al, const AdjParams& p) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const double b = sqrt(S.res[pp]);
  const double prev_b = it > 1 ? S.beta[pp][it - 1] : 0.0;
  const bool breakdown = b <= 1e-13 * (fabs(al) + prev_b + 1.0);
  if (lane == 0) {
    S.alpha[pp][it] = al;
    S.beta[pp][it] = b;
    S.scale[pp][it + 1] = b > 0.0 ? div_call(1.0, b) : 0.0;
  }
  __syncwarp();
  int acc_flag = 0;
  if (p.tol <= 0.0) {
    acc_flag = (it == p.m_max) || breakdown;
  } else if (breakdown) {
    acc_flag = 1;
  } else if (it >= p.m_min && gersh_gate(it, S.alpha[pp] + 1, S.beta[pp] + 1, p.tau) &&
             !krylov_lead_rejects(it, S.alpha[pp] + 1, S.beta[pp] + 1, p.tau, S.beta0[pp] * b, p.tol)) {
    double *yr = S.wyr[warp][0], *yi = S.wyi[warp][0];
    small_expm_e1(it, S.alpha[pp] + 1, S.beta[pp] + 1, p.tau, yr, yi, S.wtr[warp], S.wti[warp]);
    acc_flag = S.beta0[pp] * b * hypot(yr[it - 1], yi[it - 1]) <= p.tol;
  }
  __syncwarp();
  if (lane == 0 && acc_flag) {
    S.active[pp] = 0;
    S.k[pp] = it;
  }
  __syncwarp();
}

// Nodes of the stage integral, the weights C and the coefficients of the inverse
// step, over the warps of the CTA (all threads).
__device__ __noinline__ void adj_weights(SmemAdj& S, int kp, int kl, const AdjParams& p) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  // the inverse step: warp 14 for psi, 15 for lambda; nodes on the others
  if (warp >= kAdjWarps - 2) {
    const int pp = warp - (kAdjWarps - 2), k = S.k[pp];
    if (k > 0)
      small_expm_e1(k, S.alpha[pp] + 1, S.beta[pp] + 1, -p.tau, S.yr[pp], S.yi[pp], S.wtr[warp], S.wti[warp]);
    __syncwarp();
    for (int i = lane; i < k; i += 32) {
      const double f = S.beta0[pp] * S.scale[pp][i + 1];
      S.cre[pp][i] = f * S.yr[pp][i];
      S.cim[pp][i] = f * S.yi[pp][i];
    }
  }
  const int nq = kp > 0 && kl > 0 ? S.nq : 0;
  const int q0 = nq == 6 ? p.nq6 : (nq == 12 ? p.nq12 : (nq == 24 ? p.nq24 : p.nq48));
  // entry (j, i) of C on thread 16 j + i (j, i < 16)
  const int ej = tid >> 4, ei = tid & 15;
  const bool mine = tid < kAdjMaxK * kAdjMaxK && ej < kp && ei < kl;
  double cr = 0.0, ci = 0.0;
  constexpr int kRound = kAdjWarps - 2;  // nodes per round
  for (int r0 = 0; r0 < nq; r0 += kRound) {
    const int q = r0 + warp;
    if (warp < kRound && q < nq) {  // y(r) = exp(+i tau r T) e_1
      const double r = p.glx[q0 + q];
      small_expm_e1(kp, S.alpha[0] + 1, S.beta[0] + 1, -p.tau * r, S.wyr[warp][0], S.wyi[warp][0], S.wtr[warp],
                    S.wti[warp]);
      small_expm_e1(kl, S.alpha[1] + 1, S.beta[1] + 1, -p.tau * r, S.wyr[warp][1], S.wyi[warp][1], S.wtr[warp],
                    S.wti[warp]);
    }
    __syncthreads();
    if (mine) {
      const int n = min(kRound, nq - r0);
#pragma unroll 1
      for (int w = 0; w < n; ++w) {
        const double wq = p.glw[q0 + r0 + w];
        const double ar = wq * S.wyr[w][0][ej], ai = wq * S.wyi[w][0][ej];
        const double br = S.wyr[w][1][ei], bi = S.wyi[w][1][ei];
        cr = fma(br, ar, fma(bi, ai, cr));   // conj(y_b) y_a
        ci = fma(br, ai, fma(-bi, ar, ci));
      }
    }
    __syncthreads();
  }
  if (mine) {  // with the normalisations of the stored vectors
    const double f = S.scale[1][ei + 1] * S.scale[0][ej + 1];
    S.C[ej][ei] = make_double2(cr * f, ci * f);
  }
  __syncthreads();
}

// One element's term of the stage integral: sum_j (V q_j)(x) sum_i C_ij conj(l_i(x)),
// KL >= kl basis vectors of lambda held in registers.
template <int KL, class Q>
__device__ __forceinline__ void adj_integral(const SmemAdj& S, const OpSpin& op, int x, int N, int kp, int kl,
                                             const Q& Qv, double& gr, double& gi) {
  double2 l[KL];
#pragma unroll
  for (int i = 0; i < KL; ++i) l[i] = i < kl ? Qv(1, i + 1)[x] : make_double2(0.0, 0.0);
#pragma unroll 1
  for (int j = 0; j < kp; ++j) {
    const double2* q = Qv(0, j + 1);
    double vr = 0.0, vi = 0.0;
#pragma unroll 4
    for (int s = 0; s < N; ++s) {
      const double2 w = q[x ^ (1 << s)];
      const double as = __ldg(op.xf + s);
      vr = fma(as, w.x, vr);
      vi = fma(as, w.y, vi);
    }
    double zr = 0.0, zi = 0.0;  // sum_i C_ij conj(l_i)
#pragma unroll
    for (int i = 0; i < KL; ++i)
      if (i < kl) {
        const double2 c = S.C[j][i];
        zr = fma(c.x, l[i].x, fma(c.y, l[i].y, zr));
        zi = fma(c.y, l[i].x, fma(-c.x, l[i].y, zi));
      }
    gr = fma(vr, zr, fma(-vi, zi, gr));
    gi = fma(vr, zi, fma(vi, zr, gi));
  }
}

// N = 16, 16 segments, 32 CF4:2 steps (64 stage exponentials of 7.8 joint Lanczos
// iterations): 21.9 ms, 342 us per stage exponential, of which the FP64 units
// need about 180.  With 256-thread CTAs behind a counter barrier, a Gram matrix
// reduced over the grid per column and every small exponential on one warp it
// took 42.1 ms.
__global__ void __launch_bounds__(kAdjThreads, 1) k_adjoint(AdjParams p, OpSpin op) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  SmemAdj& S = *reinterpret_cast<SmemAdj*>(smem_raw);
  const int tid = threadIdx.x;
  const int dim = p.dim, N = op.N;
  // contiguous chunks of whole warps
  const int chunk = ((dim + (int)gridDim.x - 1) / (int)gridDim.x + 31) & ~31;
  const int x0 = blockIdx.x * chunk + tid, xe = min(dim, ((int)blockIdx.x + 1) * chunk);
  constexpr int stride = kAdjThreads;
  const bool lead = blockIdx.x == 0 && tid == 0;
  const double tau = p.tau;
  unsigned tag = (unsigned)ld_volatile_i32((const int*)&p.st->tag_base);
  auto Qv = [&](int pp, int i) -> double2* {
    return i == 1 ? (pp == 0 ? p.psi : p.lam) : (pp == 0 ? p.Vp : p.Vl) + (size_t)(i - 2) * dim;
  };
  long long n_app = 0;

  // ---- entry: checkpoint, adjoint initial state, overlap, norms
  {
    double v[8] = {};
    for (int x = x0; x < xe; x += stride) {
      double2 a = p.psi[x];
      if (p.ckpt) {
        const double2 c = p.ckpt[x];
        const double dx = a.x - c.x, dy = a.y - c.y;
        v[0] = fma(dx, dx, fma(dy, dy, v[0]));
        a = c;
        p.psi[x] = a;
      }
      double2 l;
      if (p.phi) {
        l = p.phi[x];
        p.lam[x] = l;
        v[1] = fma(l.x, a.x, fma(l.y, a.y, v[1]));   // Re conj(phi) psi
        v[2] = fma(l.x, a.y, fma(-l.y, a.x, v[2]));  // Im conj(phi) psi
      } else {
        l = p.lam[x];
      }
      v[3] = fma(a.x, a.x, fma(a.y, a.y, v[3]));
      v[4] = fma(l.x, l.x, fma(l.y, l.y, v[4]));
    }
    if (!adj_reduce<8>(S, v, true, tag, p)) return;
    if (lead) {
      if (p.phi) {
        p.out[0] = S.res[1];
        p.out[1] = S.res[2];
      }
      p.out[2] = fmax(p.out[2], sqrt(S.res[0]));
    }
    if (tid == 0) {
      S.beta0[0] = sqrt(S.res[3]);
      S.beta0[1] = sqrt(S.res[4]);
    }
    __syncthreads();
  }

  for (long long e = p.e_hi - 1; e >= p.e_lo; --e) {
    const double c0 = p.c0[e], c1 = p.c1[e];
    if (tid < N) S.bsite_raw[tid] = c1 * __ldg(op.xf + tid);
    if (tid < 2) {
      const double b0 = S.beta0[tid];
      if (!(b0 < 1e300)) atomicCAS(&p.st->status, 0, (int)CFET_ENAN);
      S.scale[tid][1] = b0 > 0.0 ? 1.0 / b0 : 0.0;
      S.active[tid] = b0 > 0.0;
      S.k[tid] = 0;
    }
    __syncthreads();
    if (ld_volatile_i32(&p.st->status) != 0) return;
    // ---- joint Lanczos of psi_after (0) and lambda_after (1) under H_j
    for (int it = 1; it <= p.m_max; ++it) {
      const int act0 = S.active[0], act1 = S.active[1];
      if (!act0 && !act1) break;
      if (tid < 64 && (tid & 31) < N) S.bsite[tid >> 5][tid & 31] = S.bsite_raw[tid & 31] * S.scale[tid >> 5][it];
      __syncthreads();
      double v[2] = {0.0, 0.0};
#pragma unroll
      for (int pp = 0; pp < 2; ++pp) {
        if (!(pp == 0 ? act0 : act1)) continue;
        const double s_it = S.scale[pp][it];
        SpinScaled sc;
        sc.cz = c0 * s_it;
        sc.cxx = c0 * op.J2 * s_it;
        const double bm = it > 1 ? S.beta[pp][it - 1] * S.scale[pp][it - 1] : 0.0;
        const double2* q = Qv(pp, it);
        const double2* qm = it > 1 ? Qv(pp, it - 1) : q;
        double2* u = Qv(pp, it + 1);
        double acc = 0.0;
        for (int x = x0; x < xe; x += stride) {
          double2 hv = apply_spin_at(q, x, op, sc, S.bsite[pp]);
          if (it > 1) {
            const double2 w = qm[x];
            hv.x = fma(-bm, w.x, hv.x);
            hv.y = fma(-bm, w.y, hv.y);
          }
          u[x] = hv;
          const double2 a = q[x];
          acc = fma(a.x, hv.x, fma(a.y, hv.y, acc));
        }
        v[pp] = acc;
      }
      if (!adj_reduce<2>(S, v, false, tag, p)) return;
      const double al0 = S.res[0] * S.scale[0][it], al1 = S.res[1] * S.scale[1][it];
      v[0] = v[1] = 0.0;
#pragma unroll
      for (int pp = 0; pp < 2; ++pp) {
        if (!(pp == 0 ? act0 : act1)) continue;
        const double s_it = S.scale[pp][it];
        const double am = -(pp == 0 ? al0 : al1) * s_it;
        const double2* q = Qv(pp, it);
        double2* u = Qv(pp, it + 1);
        double acc = 0.0;
        for (int x = x0; x < xe; x += stride) {
          const double2 a = q[x];
          double2 w = u[x];
          w.x = fma(am, a.x, w.x);
          w.y = fma(am, a.y, w.y);
          u[x] = w;
          acc = fma(w.x, w.x, fma(w.y, w.y, acc));
        }
        v[pp] = acc;
      }
      if (!adj_reduce<2>(S, v, true, tag, p)) return;
      n_app += act0 + act1;
      if (tid < 32) {
        if (act0) adj_decide(S, 0, it, al0, p);
      } else if (tid < 64) {
        if (act1) adj_decide(S, 1, it, al1, p);
      }
      __syncthreads();
    }
    if (S.active[0] || S.active[1]) {  // the adjoint sweep takes no substeps
      if (lead) atomicCAS(&p.st->status, 0, (int)CFET_EKRYLOV);
      return;
    }
    const int kp = S.k[0], kl = S.k[1];
    // Rule of the stage integral: the integrand is a sum of e^{i om' r} with
    // |om'| <= om = |tau| (width_psi + width_lambda); the n-node rule on [0, 1]
    // integrates e^{i om r} to 1e-14 for om up to 1.25 (6), 10 (12), 39.5 (24)
    // and 114 (48 nodes).  Beyond that the sweep gives up (CFET_EKRYLOV);
    // every CTA takes the same decision (identical scalars).
    if (tid < 32) {
      int nq = 6;
      if (kp > 0 && kl > 0) {
        const double om = fabs(tau) * (gersh_width(kp, S.alpha[0] + 1, S.beta[0] + 1) +
                                       gersh_width(kl, S.alpha[1] + 1, S.beta[1] + 1));
        nq = om <= 1.25 ? 6 : (om <= 10.0 ? 12 : (om <= 39.5 ? 24 : (om <= 114.0 ? 48 : 0)));
      }
      if (tid == 0) S.nq = nq;
    }
    __syncthreads();
    if (S.nq == 0) {
      if (lead) atomicCAS(&p.st->status, 0, (int)CFET_EKRYLOV);
      return;
    }
    adj_weights(S, kp, kl, p);
    // ---- stage integral (V = sum_i a_i X_i)
    double v[4] = {0.0, 0.0, 0.0, 0.0};
    if (kp > 0 && kl > 0) {
      if (kl <= 8) {
        for (int x = x0; x < xe; x += stride) adj_integral<8>(S, op, x, N, kp, kl, Qv, v[2], v[3]);
      } else {
        for (int x = x0; x < xe; x += stride) adj_integral<kAdjMaxK>(S, op, x, N, kp, kl, Qv, v[2], v[3]);
      }
    }
    // every CTA has read the neighbours of q_1 before psi and lambda (q_1) are overwritten
    {
      double none[2] = {0.0, 0.0};
      if (!adj_reduce<2>(S, none, true, tag, p)) return;
    }
    // ---- psi_before = a(1), lambda_before = b(1)
    for (int x = x0; x < xe; x += stride) {
#pragma unroll
      for (int pp = 0; pp < 2; ++pp) {
        double re = 0.0, im = 0.0;
#pragma unroll 4
        for (int i = 0; i < S.k[pp]; ++i) {
          const double2 w = Qv(pp, i + 1)[x];
          const double cr = S.cre[pp][i], ci = S.cim[pp][i];
          re = fma(cr, w.x, fma(-ci, w.y, re));
          im = fma(cr, w.y, fma(ci, w.x, im));
        }
        Qv(pp, 1)[x] = make_double2(re, im);
        v[pp] = fma(re, re, fma(im, im, v[pp]));
      }
    }
    if (!adj_reduce<4>(S, v, true, tag, p)) return;
    if (lead) {
      // term = -i tau beta0_psi beta0_lambda I
      const double f = tau * S.beta0[0] * S.beta0[1] * p.gam[e];
      const int sg = p.seg[e];
      p.grad[2 * sg] += f * S.res[3];
      p.grad[2 * sg + 1] -= f * S.res[2];
    }
    __syncthreads();
    if (tid == 0) {
      S.beta0[0] = sqrt(S.res[0]);
      S.beta0[1] = sqrt(S.res[1]);
    }
    __syncthreads();
  }
  if (lead) {
    p.out[3] += (double)n_app;
    p.st->tag_base = tag;
  }
}

}  // namespace

int launch_adjoint_spin(const AdjParams& p, const OpSpin& op, int grid, void* stream) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(kAdjThreads);
  cfg.dynamicSmemBytes = sizeof(SmemAdj);
  cfg.stream = (cudaStream_t)stream;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeCooperative;
  at[0].val.cooperative = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return (int)cudaLaunchKernelEx(&cfg, k_adjoint, p, op);
}

int max_coresident_blocks_adjoint() {
  int dev = 0, nsm = 0, per = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_adjoint, kAdjThreads, sizeof(SmemAdj)) != cudaSuccess)
    return -1;
  return per * nsm;
}

}  // namespace cfet
