// Mixed-precision persistent Lanczos kernel (sm_103a): complex64 Krylov
// vectors, FP64-class reductions and FP64 scalar work.
//
// Same method and decisions as k_propagate (kernels.cu) and k_propagate_fx
// (kernels_fx.cu): the stage exponential exp(-i tau H_j) psi of a CFET step
// (Alvermann & Fehske, arXiv:1102.5071, Sec. 4 Eq. (Ucf), Sec. 7
// Eq. (OmGLeg)) by the Lanczos / Krylov method of Sec. 8.1 with the
// a-posteriori estimate, adaptive Krylov dimension and substepping.
//
// Number format.  The Krylov vectors q_i are complex64 (8 B per element, half
// the bytes of complex128) and the operator apply, the three-term recurrence
// and the reconstruction run in FP32 (the GB300 FP32 rate is 64x its FP64
// rate).  Everything that decides the method stays FP64-class:
//   * alpha_k, ||w||^2 and ||psi||^2 are compensated FP32 dot products per
//     thread (error-free product by FMA and error-free sum, i.e. the Dot2
//     scheme of Ogita, Rump and Oishi, "Accurate sum and dot product", 2005),
//     combined as float-float pairs over the warp and in FP64 over the CTA
//     and the grid, in one fixed order (every CTA holds bit-identical sums);
//   * the stage and Lanczos scalars, the tridiagonal exponential, the error
//     estimate and all decisions are FP64-class on the control warp (taken in
//     FP32 or integers only where scalar_bounds.cuh shows the FP64 decision
//     for certain);
//   * psi enters and leaves as complex128; in between it is held as q_1.
// The result differs from the FP64 method by FP32 rounding of the vectors
// (relative 2^-24 per element and operation), not by the Krylov decisions.
//
// Work split: NW worker warps do element work only; one control warp does
// the reductions, the bounded grid barrier, the per-pass scalars and the
// small exponential (the estimate of iteration k runs while the workers
// already apply H for iteration k+1, as in the fixed-point kernel).
//
// Chains of 17 to 21 sites: the staged form keeps the applied vector in the shared
// memory of 128 CTAs (clusters of four).  Long chains: the tiled form applies H in
// window passes over shared-memory tiles moved by TMA (tiled_common.cuh) instead
// of element by element; its window 0 also does the previous iteration's
// orthogonalisation step, so it has one grid exchange per iteration less.
#include <cuda_runtime.h>

#include <cmath>
#include <cstdint>

#include "cfet_internal.h"
#include "device_common.cuh"
#include "tiled_common.cuh"

namespace cfet {

// ------------------------------------------------------------------ compensated sums
// (s, c): running sum s and accumulated rounding errors c.  The _rn
// intrinsics keep the compiler from contracting the error-free steps.
__device__ __forceinline__ void ff_two_sum(float& s, float& c, float p) {
  const float t = __fadd_rn(s, p);
  const float z = __fsub_rn(t, s);
  const float e = __fadd_rn(__fsub_rn(s, __fsub_rn(t, z)), __fsub_rn(p, z));
  s = t;
  c = __fadd_rn(c, e);
}
__device__ __forceinline__ void ff_add_prod(float& s, float& c, float a, float b) {
  const float p = __fmul_rn(a, b);
  const float e = __fmaf_rn(a, b, -p);  // a b = p + e exactly
  ff_two_sum(s, c, p);
  c = __fadd_rn(c, e);
}
// Warp sum of (s, c) pairs (lane 0 result).
__device__ __forceinline__ void ff_warp_sum(float& s, float& c) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const float s2 = __shfl_down_sync(0xffffffffu, s, o);
    const float c2 = __shfl_down_sync(0xffffffffu, c, o);
    ff_two_sum(s, c, s2);
    c = __fadd_rn(c, c2);
  }
}

// ------------------------------------------------------------------ shared state
struct CConst {
  // phase A: u = s_k H_j q_k - beta_{k-1} s_{k-1} q_{k-1}
  union {                        // spin: c0 s_k, 2 J c0 s_k, uniform field s_k, -beta s_{k-1}
    struct { float cz, ch, cx, cp; };
    float c4[4];
  };
  float co[1 + kMaxDrives];      // dia: c_o s_k per operator
  int use_prev;
};

struct SmemC {
  float ws[3][32], wc[3][32];    // per-warp compensated partials of the workers (up to 3 sums)
  double alpha[kMaxKrylov + 2];
  double beta[kMaxKrylov + 2];
  double scale[kMaxKrylov + 3];  // 1 / ||q_i||
  double yr[kMaxKrylov], yi[kMaxKrylov];
  double tr[kMaxKrylov], ti[kMaxKrylov];
  float cr[kMaxKrylov], ci[kMaxKrylov];  // reconstruction coefficients
  double scal[1 + kMaxDrives];
  double cst[3];                 // spin: c_0, 2 J c_0, b_0 of the stage
  double bsite_raw[kMaxSites];
  float bx[kMaxSites];           // non-uniform fields: b_i s_k
  CConst ca;
  float am;                      // phase B: -alpha_k s_k
  double wnorm2;                 // ||w||^2 of the current iteration (from the phase-A sums)
  double qnorm2[kMaxKrylov + 3]; // ||q_i||^2 of the stored vectors (reduced after they are written)
  // commands to the workers
  int cmd, it;                   // CCmd; the iteration, or the number of basis vectors (kCRec)
  int final_rec;
  // control flow
  long long e, fpos;             // stage exponential of the launch; next forced decision
  double remaining;              // of the stage exponential
  double acc_err;                // estimate of the accepted substep
  int nsub_e;                    // substeps of the stage exponential
  int y_ready, acc_h;
  int tma_fail;                  // tiled apply: a tile wait gave up
  double beta0;
  // trace (cfet_stats.phase_ns; slots 0, 2, 4, 7 by thread 0, the others by the
  // control lane 0) and, by the control lane 0, the run's counters
  long long tacc[8];
  long long twe;                 // thread 0: end of its last element loop
  long long n_app, n_sub, rpos;
  int max_k;
  double max_err;
  LeadAcc lead;                  // running FP32 bounds of the current T_k for the estimate's screens
  GershAcc gfull;                // rows whose couplings are all known
};

// ------------------------------------------------------------------ applies
__device__ __forceinline__ float2 c_apply_spin(const float2* __restrict__ q, const float2* __restrict__ qm, int x,
                                               const OpSpinC& op, const CConst& c, const float* bx) {
  const int N = op.N, L = op.lo_bits;
  const float dz = __ldg(op.dz_lo + (x & ((1 << L) - 1))) + __ldg(op.dz_hi + (x >> (L - 1)));
  const float d = c.cz * dz;
  const float2 v = q[x];
  float ur = d * v.x, ui = d * v.y;
  float hr = 0.f, hi = 0.f;
  const unsigned anti = ((unsigned)x ^ ((unsigned)x >> 1)) & ((1u << (N - 1)) - 1u);
#pragma unroll 4
  for (int i = 0; i < N - 1; ++i) {  // antiparallel bonds only (predicated)
    if ((anti >> i) & 1u) {
      const float2 w = q[x ^ (3 << i)];
      hr += w.x;
      hi += w.y;
    }
  }
  ur = fmaf(c.ch, hr, ur);
  ui = fmaf(c.ch, hi, ui);
  if (op.uniform) {
    float xr = 0.f, xi = 0.f;
#pragma unroll 4
    for (int i = 0; i < N; ++i) {
      const float2 w = q[x ^ (1 << i)];
      xr += w.x;
      xi += w.y;
    }
    ur = fmaf(c.cx, xr, ur);
    ui = fmaf(c.cx, xi, ui);
  } else {
#pragma unroll 4
    for (int i = 0; i < N; ++i) {
      const float2 w = q[x ^ (1 << i)];
      ur = fmaf(bx[i], w.x, ur);
      ui = fmaf(bx[i], w.y, ui);
    }
  }
  if (c.use_prev) {
    const float2 w = qm[x];
    ur = fmaf(c.cp, w.x, ur);
    ui = fmaf(c.cp, w.y, ui);
  }
  return make_float2(ur, ui);
}

// Two elements x and x2 per call: the neighbour loads of both are issued in
// the same loop iterations (twice the independent requests per warp).
__device__ __forceinline__ void c_apply_spin2(const float2* __restrict__ q, const float2* __restrict__ qm, int x,
                                              int x2, const OpSpinC& op, const CConst& c, const float* bx,
                                              float2& r1, float2& r2) {
  const int N = op.N, L = op.lo_bits;
  const float d1 = c.cz * (__ldg(op.dz_lo + (x & ((1 << L) - 1))) + __ldg(op.dz_hi + (x >> (L - 1))));
  const float d2 = c.cz * (__ldg(op.dz_lo + (x2 & ((1 << L) - 1))) + __ldg(op.dz_hi + (x2 >> (L - 1))));
  const float2 v1 = q[x], v2 = q[x2];
  float ur1 = d1 * v1.x, ui1 = d1 * v1.y, ur2 = d2 * v2.x, ui2 = d2 * v2.y;
  float hr1 = 0.f, hi1 = 0.f, hr2 = 0.f, hi2 = 0.f;
  const unsigned mask = (1u << (N - 1)) - 1u;
  const unsigned anti1 = ((unsigned)x ^ ((unsigned)x >> 1)) & mask;
  const unsigned anti2 = ((unsigned)x2 ^ ((unsigned)x2 >> 1)) & mask;
#pragma unroll 4
  for (int i = 0; i < N - 1; ++i) {
    if ((anti1 >> i) & 1u) {
      const float2 w = q[x ^ (3 << i)];
      hr1 += w.x;
      hi1 += w.y;
    }
    if ((anti2 >> i) & 1u) {
      const float2 w = q[x2 ^ (3 << i)];
      hr2 += w.x;
      hi2 += w.y;
    }
  }
  ur1 = fmaf(c.ch, hr1, ur1);
  ui1 = fmaf(c.ch, hi1, ui1);
  ur2 = fmaf(c.ch, hr2, ur2);
  ui2 = fmaf(c.ch, hi2, ui2);
  if (op.uniform) {
    float xr1 = 0.f, xi1 = 0.f, xr2 = 0.f, xi2 = 0.f;
#pragma unroll 4
    for (int i = 0; i < N; ++i) {
      const float2 w1 = q[x ^ (1 << i)];
      const float2 w2 = q[x2 ^ (1 << i)];
      xr1 += w1.x;
      xi1 += w1.y;
      xr2 += w2.x;
      xi2 += w2.y;
    }
    ur1 = fmaf(c.cx, xr1, ur1);
    ui1 = fmaf(c.cx, xi1, ui1);
    ur2 = fmaf(c.cx, xr2, ur2);
    ui2 = fmaf(c.cx, xi2, ui2);
  } else {
#pragma unroll 4
    for (int i = 0; i < N; ++i) {
      const float2 w1 = q[x ^ (1 << i)];
      const float2 w2 = q[x2 ^ (1 << i)];
      ur1 = fmaf(bx[i], w1.x, ur1);
      ui1 = fmaf(bx[i], w1.y, ui1);
      ur2 = fmaf(bx[i], w2.x, ur2);
      ui2 = fmaf(bx[i], w2.y, ui2);
    }
  }
  if (c.use_prev) {
    const float2 w1 = qm[x], w2 = qm[x2];
    ur1 = fmaf(c.cp, w1.x, ur1);
    ui1 = fmaf(c.cp, w1.y, ui1);
    ur2 = fmaf(c.cp, w2.x, ur2);
    ui2 = fmaf(c.cp, w2.y, ui2);
  }
  r1 = make_float2(ur1, ui1);
  r2 = make_float2(ur2, ui2);
}

// Element pair (x, x + 1) of a chain whose applied vector is staged in the shared
// memory of 128 CTAs, 2^(N - 7) elements each, in clusters of four: flips and hops of
// bits below N - 7 from this CTA's shared memory, the next two from the cluster's,
// the five highest from global memory (issued ahead); any bit above bit 0 maps the
// pair onto a pair, one 16-byte access.  Every element's sum runs in the order of the
// element-wise form, so an apply gives the same bits (the compensated sums over the
// vector run over 128 parts instead of 152).  The far gathers bound it: 4.5 TB/s over
// the L2 fabric, where the element-wise form gathers twice as many bytes.  Lanczos
// iteration 12.1 us at 17 sites (element-wise 13.6), 15.2 at 18 (16.8), 30.8 at 20
// (32.4), 53.6 at 21 (58.0).  Near loops unrolled by 6 and 12 instead of 4: 3 and
// 8 % slower.  Fixed-point vectors (twice the bytes, on 128 of 152 SMs) were slower
// staged, 59.6 against 52.8 us at 20 sites.
constexpr int kCStagedBits = 7, kCStagedClusterBits = 2, kCStagedFar = kCStagedBits - kCStagedClusterBits;
__device__ __forceinline__ float4 c_ld_cluster(unsigned base, int j) {
  float4 v;
  asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];"
               : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
               : "r"(base + 8u * (unsigned)j));
  return v;
}
__device__ __forceinline__ void c_apply_spin_staged2(const float2* sq, const float2* __restrict__ q,
                                                     const float2* __restrict__ qm, int j, unsigned rank,
                                                     const OpSpinC& op, const CConst& c, const float* bx, float4& r,
                                                     float4& v) {
  const int N = op.N, L = op.lo_bits, lc = N - kCStagedBits, lg = N - kCStagedFar;
  const int x = (int)(blockIdx.x << lc) | j;
  const unsigned anti = ((unsigned)x ^ ((unsigned)x >> 1)) & ((1u << (N - 1)) - 1u);
  auto add = [](float4& s, const float4 w) {
    s.x += w.x;
    s.y += w.y;
    s.z += w.z;
    s.w += w.w;
  };
  auto near4 = [&](int jj) { return *reinterpret_cast<const float4*>(sq + jj); };
  auto far4 = [&](int xx) { return *reinterpret_cast<const float4*>(q + xx); };
  float4 f[kCStagedFar], pv = make_float4(0.f, 0.f, 0.f, 0.f);
  // far hops under way during the near ones (antiparallel bonds, uniform over the CTA)
#pragma unroll
  for (int k = 0; k < kCStagedFar; ++k) {
    f[k] = make_float4(0.f, 0.f, 0.f, 0.f);
    if ((anti >> (lg - 1 + k)) & 1u) f[k] = far4(x ^ (3 << (lg - 1 + k)));
  }
  if (c.use_prev) pv = *reinterpret_cast<const float4*>(qm + x);
  v = near4(j);
  const float2 dlo = __ldg(reinterpret_cast<const float2*>(op.dz_lo + (x & ((1 << L) - 1))));
  const float dhi = __ldg(op.dz_hi + (x >> (L - 1)));
  const float d0 = c.cz * (dlo.x + dhi), d1 = c.cz * (dlo.y + dhi);
  float4 u = make_float4(d0 * v.x, d0 * v.y, d1 * v.z, d1 * v.w);
  auto madd = [&](float a, const float4 w) {
    u.x = fmaf(a, w.x, u.x);
    u.y = fmaf(a, w.y, u.y);
    u.z = fmaf(a, w.z, u.z);
    u.w = fmaf(a, w.w, u.w);
  };
  float4 h = make_float4(0.f, 0.f, 0.f, 0.f);
  {  // bond (0, 1): one element of the pair j ^ 2
    const float4 w = near4(j ^ 2);
    if ((j >> 1) & 1) {
      h.x += w.z;
      h.y += w.w;
    } else {
      h.z += w.x;
      h.w += w.y;
    }
  }
#pragma unroll 4
  for (int i = 1; i < lc - 1; ++i)
    if ((anti >> i) & 1u) add(h, near4(j ^ (3 << i)));
  if ((anti >> (lc - 1)) & 1u) add(h, c_ld_cluster(cluster_addr(sq, rank ^ 1u), j ^ (1 << (lc - 1))));
  if ((anti >> lc) & 1u) add(h, c_ld_cluster(cluster_addr(sq, rank ^ 3u), j));
#pragma unroll
  for (int k = 0; k < kCStagedFar; ++k)
    if ((anti >> (lg - 1 + k)) & 1u) add(h, f[k]);
  // far flips under way during the near ones
#pragma unroll
  for (int k = 0; k < kCStagedFar; ++k) f[k] = far4(x ^ (1 << (lg + k)));
  madd(c.ch, h);
  float4 g[kCStagedClusterBits];
#pragma unroll
  for (int k = 0; k < kCStagedClusterBits; ++k) g[k] = c_ld_cluster(cluster_addr(sq, rank ^ (1u << k)), j);
  const float4 swap = make_float4(v.z, v.w, v.x, v.y);  // bit 0
  if (op.uniform) {
    float4 s = swap;
#pragma unroll 4
    for (int i = 1; i < lc; ++i) add(s, near4(j ^ (1 << i)));
#pragma unroll
    for (int k = 0; k < kCStagedClusterBits; ++k) add(s, g[k]);
#pragma unroll
    for (int k = 0; k < kCStagedFar; ++k) add(s, f[k]);
    madd(c.cx, s);
  } else {
    madd(bx[0], swap);
#pragma unroll 4
    for (int i = 1; i < lc; ++i) madd(bx[i], near4(j ^ (1 << i)));
#pragma unroll
    for (int k = 0; k < kCStagedClusterBits; ++k) madd(bx[lc + k], g[k]);
#pragma unroll
    for (int k = 0; k < kCStagedFar; ++k) madd(bx[lg + k], f[k]);
  }
  if (c.use_prev) madd(c.cp, pv);
  r = u;
}

__device__ __forceinline__ float2 c_apply_dia(const float2* __restrict__ q, const float2* __restrict__ qm, int r,
                                              int dim, const OpDiaC& op, const CConst& c) {
  float ur = 0.f, ui = 0.f;
  for (int o = 0; o < op.nops; ++o) {
    float ar = 0.f, ai = 0.f;
    const int d0 = op.dfirst[o], d1 = d0 + op.dcount[o];
    for (int d = d0; d < d1; ++d) {
      const long long cidx = (long long)r + __ldg(op.off + d);
      if (cidx >= 0 && cidx < dim) {
        const float a = __ldg(op.val + (size_t)d * dim + r);
        const float2 w = q[cidx];
        ar = fmaf(a, w.x, ar);
        ai = fmaf(a, w.y, ai);
      }
    }
    ur = fmaf(c.co[o], ar, ur);
    ui = fmaf(c.co[o], ai, ui);
  }
  if (c.use_prev) {
    const float2 w = qm[r];
    ur = fmaf(c.cp, w.x, ur);
    ui = fmaf(c.cp, w.y, ui);
  }
  return make_float2(ur, ui);
}

// CSR: per operator the row's sum of val * q in FP32 (complex values of
// Hermitian operators) in the order of the entries, then the operator's scalar.
__device__ __forceinline__ float2 c_apply_csr(const float2* __restrict__ q, const float2* __restrict__ qm, int r,
                                              int dim, const OpCsrC& op, const CConst& c) {
  float ur = 0.f, ui = 0.f;
  for (int o = 0; o < op.nops; ++o) {
    const int* rp = op.rp + (size_t)o * (dim + 1);
    const int e0 = __ldg(rp + r), e1 = __ldg(rp + r + 1);
    float ar = 0.f, ai = 0.f;
    if (op.vi) {
      for (int e = e0; e < e1; ++e) {
        const float a = __ldg(op.vr + e), b = __ldg(op.vi + e);
        const float2 w = q[__ldg(op.col + e)];
        ar = fmaf(a, w.x, fmaf(-b, w.y, ar));
        ai = fmaf(a, w.y, fmaf(b, w.x, ai));
      }
    } else {
      for (int e = e0; e < e1; ++e) {
        const float a = __ldg(op.vr + e);
        const float2 w = q[__ldg(op.col + e)];
        ar = fmaf(a, w.x, ar);
        ai = fmaf(a, w.y, ai);
      }
    }
    ur = fmaf(c.co[o], ar, ur);
    ui = fmaf(c.co[o], ai, ui);
  }
  if (c.use_prev) {
    const float2 w = qm[r];
    ur = fmaf(c.cp, w.x, ur);
    ui = fmaf(c.cp, w.y, ui);
  }
  return make_float2(ur, ui);
}

// ------------------------------------------------------------------ control warp
// Worker warps: compensated per-warp partial of sum j into shared memory.
__device__ __forceinline__ void c_worker_partial(SmemC& S, float s, float c, int j = 0) {
  ff_warp_sum(s, c);
  if ((threadIdx.x & 31) == 0) {
    S.ws[j][threadIdx.x >> 5] = s;
    S.wc[j][threadIdx.x >> 5] = c;
  }
}

// Float-float accumulation of the exchanged CTA partials (fixed order per lane).
template <int NS>
struct FFAcc {
  float s[NS], c[NS];
  __device__ void reset() {
    for (int j = 0; j < NS; ++j) s[j] = c[j] = 0.f;
  }
  __device__ void add(const unsigned (&v)[2 * NS]) {
    for (int j = 0; j < NS; ++j) {
      ff_two_sum(s[j], c[j], __uint_as_float(v[2 * j]));
      c[j] = __fadd_rn(c[j], __uint_as_float(v[2 * j + 1]));
    }
  }
};

// Control warp: publish the CTA's float-float partials of NS sums, exchange
// records with every CTA (the grid barrier), and return the global sums,
// accumulated in one fixed order and rounded to FP64 once, to all lanes.
// Keeping the chain in FP32 pairs avoids long dependent sequences on the
// 1/64-rate FP64 units.  NS = 0: a pure grid barrier.
template <int NS>
__device__ __forceinline__ bool c_ctl_reduce(SmemC& S, int NW, unsigned long long* part, unsigned tag, bool fence, int* status,
                             long long timeout_ns, double* sum, long long& spin) {
  const int lane = threadIdx.x & 31;
  constexpr int W = NS > 0 ? 2 * NS : 1;
  unsigned mine[W];
  mine[0] = 0u;
  for (int j = 0; j < NS; ++j) {
    float s = lane < NW ? S.ws[j][lane] : 0.f, c = lane < NW ? S.wc[j][lane] : 0.f;
    ff_warp_sum(s, c);
    mine[2 * j] = __float_as_uint(__shfl_sync(0xffffffffu, s, 0));
    mine[2 * j + 1] = __float_as_uint(__shfl_sync(0xffffffffu, c, 0));
  }
  if constexpr (NS > 0) {
    FFAcc<NS> acc;
    if (!ctl_exchange<W>(part, mine, tag, fence, status, timeout_ns, spin, acc)) return false;
    for (int j = 0; j < NS; ++j) {
      float s = acc.s[j], c = acc.c[j];
      ff_warp_sum(s, c);
      sum[j] = (double)__shfl_sync(0xffffffffu, s, 0) + (double)__shfl_sync(0xffffffffu, c, 0);
    }
  } else {
    struct NoAcc {
      __device__ void reset() {}
      __device__ void add(const unsigned (&)[1]) {}
    } acc;
    if (!ctl_exchange<1>(part, mine, tag, fence, status, timeout_ns, spin, acc)) return false;
  }
  return true;
}

// One sum out of line, for the passes that run once per launch or substep: the
// norm of the new q_1.
__device__ __noinline__ bool c_ctl_reduce_cold(SmemC& S, int NW, unsigned long long* part, unsigned tag, int* status,
                                               long long timeout_ns) {
  double sum[1];
  const bool ok = c_ctl_reduce<1>(S, NW, part, tag, true, status, timeout_ns, sum, S.tacc[5]);
  if (ok && (threadIdx.x & 31) == 0) {
    S.beta0 = sqrt(sum[0]);
    S.qnorm2[1] = sum[0];
  }
  __syncwarp();
  return ok;
}

// Phase-A constants for iteration `it`, one scalar per lane: a product and a
// conversion of the FP64 units (64 and 190 cycles) for all of them at once.
// spin: the stage scalars c_0, 2 J c_0 and b_0 times s_k, and -beta s_{k-1};
// DIA, CSR: one operator scalar per lane, then -beta s_{k-1}.
template <int FAMILY, class Op>
__device__ __forceinline__ void c_const_a(SmemC& S, const Op& op, int it) {
  const int lane = threadIdx.x & 31;
  CConst& c = S.ca;
  const double sk = S.scale[it];
  const int np = FAMILY == kFamilySpin ? 3 : 1 + kMaxDrives;  // lane of the q_{k-1} coefficient
  double a = 0.0, f = sk;
  if constexpr (FAMILY == kFamilySpin) {
    if (lane < 3) a = S.cst[lane];
  } else {
    if (lane < op.nops) a = S.scal[lane];
  }
  if (lane == np && it > 1) {
    a = -S.beta[it - 1];
    f = S.scale[it - 1];
  }
  const float v = (float)(a * f);
  if constexpr (FAMILY == kFamilySpin) {
    if (lane < 4) c.c4[lane] = v;
    if (!op.uniform)
      for (int i = lane; i < op.N; i += 32) S.bx[i] = (float)(S.bsite_raw[i] * sk);
  } else {
    if (lane < op.nops) c.co[lane] = v;
    if (lane == np) c.cp = v;
  }
  if (lane == 0) c.use_prev = it > 1;
}

// Error estimate of iteration k (control warp), with the FP32 screen of
// fx_estimate: above thr without the FP64 small exponential when it can.
__device__ __noinline__ double c_estimate(SmemC& S, int k, double ts, double thr) {
  const int dec = krylov_lead_decide(S.lead, k, ts, S.beta0, S.beta[k], thr);
  if (dec == 0) return 2.0 * thr + 1e-300;
  const double scale = S.beta0 * S.beta[k];
  if (dec < 0 && small_expm_rejects32(k, S.alpha + 1, S.beta + 1, ts, scale, thr)) return 2.0 * thr + 1e-300;
  small_expm_e1(k, S.alpha + 1, S.beta + 1, ts, S.yr, S.yi, S.tr, S.ti);
  const double yr = S.yr[k - 1], yi = S.yi[k - 1];
  return scale * sqrt(fma(yr, yr, yi * yi));
}

// ------------------------------------------------------------------ tiled apply (large chains)
// Window tiling of tiled_common.cuh with tiles of 2^12 complex64 elements
// moved by TMA.  Each of kTmaStages stages holds the q tile and the tile of
// the vector each element reads for itself (q_{k-1} in window 0, the partial
// u after it): 64 KB per stage.  One worker (the producer) keeps two tiles in
// flight ahead of the others: it arms the stage's mbarrier with the bytes of
// both loads and issues them, and once the workers have written a tile's
// results (in place over its own-element buffer) it stores that buffer with a
// bulk tensor store.  The loop touches global memory only for the diagonal
// tables; the last window also takes <q, u> and ||u||^2.
constexpr int kTileBits = kC64TileBits;
constexpr int kTileElems = 1 << kTileBits;
constexpr unsigned kTileBytes = kTileElems * sizeof(float2);

struct TmaPass {
  const unsigned char* maps;  // kTmaMapBytes per window
  unsigned long long* bar;    // [kTmaStages] in shared memory
  float2* stage;              // [kTmaStages][2][kTileElems] in shared memory
  int* fail;                  // shared flag: a wait gave up
  unsigned* phase;            // parity bits of the stages (per thread, identical in all workers)
  int* status;
  long long timeout_ns;
};

// Bounded wait for a stage's tile; false (status CFET_ETIMEOUT) when it gave up.
__device__ bool tile_wait(unsigned long long* bar, unsigned parity, int* status, long long timeout_ns) {
  if (mbar_try_wait(bar, parity)) return true;
  const long long t0 = global_timer_ns();
  unsigned spins = 0;
  while (!mbar_try_wait(bar, parity)) {
    if ((++spins & 255u) == 0u) {
      if (ld_volatile_i32(status) != 0) return false;
      if (global_timer_ns() - t0 > timeout_ns) {
        atomicCAS(status, 0, (int)CFET_ETIMEOUT);
        return false;
      }
    }
  }
  return true;
}

// One window pass of this CTA's worker threads over its tiles (vectors are
// basis indices: iq the applied q, ia the own-element input, iu the output).
// ORTH (window 0 from the second iteration on): the q tile holds u_{k-1} and
// the aux tile q_{k-1}; the pass first forms q_k = w_{k-1} = u_{k-1} + am q_{k-1}
// in place (the orthogonalisation step of iteration k-1, with ||w||^2 into
// s2/c2), applies H to it and stores both w (over u_{k-1}) and the result.
template <bool FIRST, bool LAST, bool ORTH = false>
__device__ void c_tiled_pass(const TmaPass& T, const OpSpinC& op, const CConst& c, const float* bx, int iq, int ia,
                             int iu, const TileWin& W, int w, int nworkers, float& s0, float& c0, float& s1,
                             float& c1, float am = 0.f, float* s2 = nullptr, float* c2 = nullptr) {
  static_assert(!ORTH || FIRST, "the orthogonalisation step runs in window 0");
  const int tid = threadIdx.x;
  const int G = gridDim.x;
  const int ntiles = 1 << (op.N - kTileBits);
  const bool aux = !FIRST || c.use_prev;
  const unsigned bytes = aux ? 2 * kTileBytes : kTileBytes;
  const void* map = T.maps + (size_t)w * kTmaMapBytes;
  const bool prod = tid == 0;
  auto issue = [&](int k, int t) {  // producer: tile t into stage k % kTmaStages
    const int st = k % kTmaStages;
    float2* qb = T.stage + (size_t)st * 2 * kTileElems;
    mbar_arrive_expect_tx(T.bar + st, bytes);
    tile_load(qb, map, FIRST, W, op.N, t, iq, T.bar + st);
    if (aux) tile_load(qb + kTileElems, map, FIRST, W, op.N, t, ia, T.bar + st);
  };
  if (prod) {
    fence_proxy_async_all();  // vectors written by generic stores before the exchange, read by TMA now
    for (int k = 0; k < kTmaStages - 1; ++k)
      if (blockIdx.x + k * G < ntiles) issue(k, blockIdx.x + k * G);
  }
  int k = 0;
  for (int t = blockIdx.x; t < ntiles; ++k, t += G) {
    const int st = k % kTmaStages;
    float2* cur = T.stage + (size_t)st * 2 * kTileElems;
    float2* acur = T.stage + (size_t)st * 2 * kTileElems + kTileElems;
    const unsigned par = (*T.phase >> st) & 1u;
    *T.phase ^= 1u << st;
    if (!tile_wait(T.bar + st, par, T.status, T.timeout_ns)) *T.fail = 1;
    if constexpr (ORTH) {
      if (!*T.fail) {
        float4* w4 = reinterpret_cast<float4*>(cur);
        const float4* p4 = reinterpret_cast<const float4*>(acur);
        for (int jp = tid; jp < kTileElems / 2; jp += nworkers) {
          const float4 uu = w4[jp], qq = p4[jp];
          const float4 wv = make_float4(fmaf(am, qq.x, uu.x), fmaf(am, qq.y, uu.y), fmaf(am, qq.z, uu.z),
                                        fmaf(am, qq.w, uu.w));
          w4[jp] = wv;
          ff_add_prod(*s2, *c2, wv.x, wv.x);
          ff_add_prod(*s2, *c2, wv.y, wv.y);
          ff_add_prod(*s2, *c2, wv.z, wv.z);
          ff_add_prod(*s2, *c2, wv.w, wv.w);
        }
      }
      workers_sync(nworkers);  // every w of the tile written before its neighbours are read
    }
    if (!*T.fail) {
      // Element pairs (2 jp, 2 jp + 1) of the tile: a flip or hop of any bit
      // above bit 0 moves both elements of a pair to the two elements of
      // another pair, so each such neighbour pair is one 16-byte load; the
      // flip of bit 0 swaps the pair, and the hop of bond (0, 1) takes one
      // element of pair jp ^ 1.
      const float4* cur4 = reinterpret_cast<const float4*>(cur);
      float4* acur4 = reinterpret_cast<float4*>(acur);
      for (int jp = tid; jp < kTileElems / 2; jp += nworkers) {
        const int j = 2 * jp;
        const float4 v = cur4[jp];
        float ur0, ui0, ur1, ui1;
        float hr0 = 0.f, hi0 = 0.f, hr1 = 0.f, hi1 = 0.f, fr0 = 0.f, fi0 = 0.f, fr1 = 0.f, fi1 = 0.f;
        if (FIRST) {
          const int x = (t << kTileBits) | j;  // even
          const int L = op.lo_bits;
          const float2 dlo = *reinterpret_cast<const float2*>(op.dz_lo + (x & ((1 << L) - 1)));
          const float dhi = __ldg(op.dz_hi + (x >> (L - 1)));
          const float d0 = c.cz * (dlo.x + dhi), d1 = c.cz * (dlo.y + dhi);
          ur0 = d0 * v.x;
          ui0 = d0 * v.y;
          ur1 = d1 * v.z;
          ui1 = d1 * v.w;
          const unsigned anti = ((unsigned)j ^ ((unsigned)j >> 1)) & ((1u << (kTileBits - 1)) - 1u);
          {  // bond (0, 1): element 0 hops when bit 1 is set, element 1 when it is clear
            const float4 w = cur4[jp ^ 1];
            if ((j >> 1) & 1) {
              hr0 += w.z;
              hi0 += w.w;
            } else {
              hr1 += w.x;
              hi1 += w.y;
            }
          }
#pragma unroll
          for (int i = 1; i < kTileBits - 1; ++i)
            if ((anti >> i) & 1u) {
              const float4 w = cur4[jp ^ (3 << (i - 1))];
              hr0 += w.x;
              hi0 += w.y;
              hr1 += w.z;
              hi1 += w.w;
            }
          if (op.uniform) {
            fr0 = v.z;  // flip of bit 0
            fi0 = v.w;
            fr1 = v.x;
            fi1 = v.y;
#pragma unroll
            for (int i = 1; i < kTileBits; ++i) {
              const float4 w = cur4[jp ^ (1 << (i - 1))];
              fr0 += w.x;
              fi0 += w.y;
              fr1 += w.z;
              fi1 += w.w;
            }
          } else {
            ur0 = fmaf(bx[0], v.z, ur0);
            ui0 = fmaf(bx[0], v.w, ui0);
            ur1 = fmaf(bx[0], v.x, ur1);
            ui1 = fmaf(bx[0], v.y, ui1);
#pragma unroll
            for (int i = 1; i < kTileBits; ++i) {
              const float4 w = cur4[jp ^ (1 << (i - 1))];
              ur0 = fmaf(bx[i], w.x, ur0);
              ui0 = fmaf(bx[i], w.y, ui0);
              ur1 = fmaf(bx[i], w.z, ur1);
              ui1 = fmaf(bx[i], w.w, ui1);
            }
          }
          if (c.use_prev) {
            const float4 w = acur4[jp];
            ur0 = fmaf(c.cp, w.x, ur0);
            ui0 = fmaf(c.cp, w.y, ui0);
            ur1 = fmaf(c.cp, w.z, ur1);
            ui1 = fmaf(c.cp, w.w, ui1);
          }
        } else {
          // the window's bits are slot bits c .. c + width - 1, pair bits c - 1 ..
          const float4 a = acur4[jp];
          ur0 = a.x;
          ui0 = a.y;
          ur1 = a.z;
          ui1 = a.w;
          const unsigned jh = (unsigned)j >> W.c;  // bits b0 .. b0+width-1 of x
          const unsigned anti = (jh ^ (jh >> 1)) & ((1u << (W.width - 1)) - 1u);
          for (int i = 0; i < W.width - 1; ++i)
            if ((anti >> i) & 1u) {
              const float4 w = cur4[jp ^ (3 << (W.c - 1 + i))];
              hr0 += w.x;
              hi0 += w.y;
              hr1 += w.z;
              hi1 += w.w;
            }
          if (op.uniform) {
            for (int i = 1; i < W.width; ++i) {
              const float4 w = cur4[jp ^ (1 << (W.c - 1 + i))];
              fr0 += w.x;
              fi0 += w.y;
              fr1 += w.z;
              fi1 += w.w;
            }
          } else {
            for (int i = 1; i < W.width; ++i) {
              const float4 w = cur4[jp ^ (1 << (W.c - 1 + i))];
              const float b = bx[W.b0 + i];
              ur0 = fmaf(b, w.x, ur0);
              ui0 = fmaf(b, w.y, ui0);
              ur1 = fmaf(b, w.z, ur1);
              ui1 = fmaf(b, w.w, ui1);
            }
          }
        }
        ur0 = fmaf(c.ch, hr0, ur0);
        ui0 = fmaf(c.ch, hi0, ui0);
        ur1 = fmaf(c.ch, hr1, ur1);
        ui1 = fmaf(c.ch, hi1, ui1);
        if (op.uniform) {
          ur0 = fmaf(c.cx, fr0, ur0);
          ui0 = fmaf(c.cx, fi0, ui0);
          ur1 = fmaf(c.cx, fr1, ur1);
          ui1 = fmaf(c.cx, fi1, ui1);
        }
        acur4[jp] = make_float4(ur0, ui0, ur1, ui1);  // the own pair only: read above by this thread
        if (LAST) {
          ff_add_prod(s0, c0, v.x, ur0);
          ff_add_prod(s0, c0, v.y, ui0);
          ff_add_prod(s0, c0, v.z, ur1);
          ff_add_prod(s0, c0, v.w, ui1);
          ff_add_prod(s1, c1, ur0, ur0);
          ff_add_prod(s1, c1, ui0, ui0);
          ff_add_prod(s1, c1, ur1, ur1);
          ff_add_prod(s1, c1, ui1, ui1);
        }
      }
    }
    fence_proxy_async_smem();  // the results, written by generic stores, are read by the TMA store
    workers_sync(nworkers);
    if (*T.fail) break;
    if (prod) {
      tile_store(map, FIRST, W, op.N, t, iu, acur);
      if constexpr (ORTH) tile_store(map, FIRST, W, op.N, t, iq, cur);
      bulk_commit();
      const int tn = t + (kTmaStages - 1) * G;
      if (tn < ntiles) {
        bulk_wait_read_1();  // the stage to refill was stored from at tile k - 1
        issue(k + kTmaStages - 1, tn);
      }
    }
  }
  if (prod) {
    bulk_wait_all();         // u written before the exchange that follows
    fence_proxy_async_all();
    if (*T.fail) {           // tiles still in flight: wait for them, again with a limit
      for (int s2 = 0; s2 < kTmaStages; ++s2) {
        const unsigned par = (*T.phase >> s2) & 1u;
        tile_wait(T.bar + s2, par, T.status, T.timeout_ns);
      }
    }
  }
  workers_sync(nworkers);
}

// Halves the step on the basis of iteration it until the estimate meets the
// proportional tolerance (control warp): S.acc_h, 0 when no step does.
__device__ __noinline__ void c_halve(SmemC& S, int it, double tol, double tau) {
  const double remaining = S.remaining;
  int hh = 0;
  double err = 0.0;
  const double width = gersh_width(it, S.alpha + 1, S.beta + 1);
#pragma unroll 1
  for (int h = 1; h <= 40; ++h) {
    const double ts = ldexp(remaining, -h);
    if (!(fabs(ts) * width <= 2.0 * it)) continue;
    err = c_estimate(S, it, ts, tol * ts / tau);
    if (err <= tol * ts / tau) { hh = h; break; }
  }
  if ((threadIdx.x & 31) == 0) { S.acc_h = hh; S.acc_err = err; S.y_ready = hh > 0; }
  __syncwarp();
}

// Estimate of iteration it against the proportional tolerance (control warp):
// 1 (accepted, S.yr / S.yi hold y) or 0; the estimate in S.acc_err.
__device__ __noinline__ int c_check(SmemC& S, int it, double tol, double tau) {
  const double thr = tol * S.remaining / tau;
  const double err = c_estimate(S, it, S.remaining, thr);
  const int acc = err <= thr;
  __syncwarp();
  if ((threadIdx.x & 31) == 0) {
    S.acc_err = err;
    S.y_ready = acc;
  }
  __syncwarp();
  return acc;
}

// Reconstruction coefficients of the accepted (k, ts) into S (control warp).
__device__ __noinline__ void c_rec_consts(SmemC& S, int acc_k, double ts) {
  const int lane = threadIdx.x & 31;
  if (!S.y_ready) small_expm_e1(acc_k, S.alpha + 1, S.beta + 1, ts, S.yr, S.yi, S.tr, S.ti);
  __syncwarp();
#pragma unroll 1
  for (int i = lane; i < acc_k; i += 32) {
    const double f = S.beta0 * S.scale[i + 1];
    S.cr[i] = (float)(f * S.yr[i]);
    S.ci[i] = (float)(f * S.yi[i]);
  }
}

// ------------------------------------------------------------------ the kernel
// Worker and control warps run separate loops, as in kernels_fx.cu (fx_worker,
// fx_control): the control warp publishes one element pass at a time.
enum CCmd { kCExit = 0, kCConvert, kCApply, kCOrth, kCRec };

// Forms of the kernel, separate instantiations: element-wise; the window-tiled
// apply of long spin chains; spin chains staged in the shared memory of all CTAs.
enum CMode { kCGrid = 0, kCTiled, kCStaged };

template <int FAMILY, class Op, int MODE>
__device__ __forceinline__ void c_worker(const PropParams& p, const Op& op, SmemC& S, unsigned char* tiles_base,
                                         int wstep) {
  constexpr bool TILED = MODE == kCTiled, STAGED = MODE == kCStaged;
  const int tid = threadIdx.x, lane = tid & 31;
  const int dim = p.dim;
  int wx0, wxe;  // one contiguous chunk per CTA
  if constexpr (FAMILY == kFamilyCsr) {  // rows split by their work, not their number (csr_row_split)
    wx0 = __ldg(op.rb + blockIdx.x) + tid;
    wxe = __ldg(op.rb + blockIdx.x + 1);
  } else {
    const int chunk = (dim + gridDim.x - 1) / gridDim.x;
    wx0 = blockIdx.x * chunk + tid;
    wxe = min(dim, ((int)blockIdx.x + 1) * chunk);
  }
  auto Q = [&](int i) -> float2* { return p.qbasis32 + (size_t)(i - 1) * dim; };
  // staged: this CTA's part of the applied vector
  float2* const sq = reinterpret_cast<float2*>(tiles_base);
  const int xb = wx0 - tid;
  TileWin win[kTiledMaxWindows] = {};
  int nwin = 1;
  if constexpr (TILED) nwin = tiled_windows<kTileBits>(op.N, win);
  unsigned tph = 0;  // parities of the stages' mbarriers (the same in every worker)
  if (tid == 0) S.twe = 0;
  while (true) {
    __syncthreads();  // the command and its constants are set
    const int cmd = S.cmd;
    if (tid == 0 && S.twe) S.tacc[7] += sm_clock() - S.twe;
    if (cmd == kCExit) break;
    const long long tw0 = sm_clock();
    if (cmd == kCApply) {
      // -------- phase A: u = s H q_it - beta s q_{it-1}.  <q,u> and ||u||^2: with
      // ||q||^2 (reduced when q was written) they give alpha and
      // ||u - alpha s q||^2, so the decisions need not wait for the
      // orthogonalisation pass
      const int it = S.it;
      const CConst& c = S.ca;
      const float2* q = Q(it);
      const float2* qm = it > 1 ? Q(it - 1) : q;
      float2* u = Q(it + 1);
      float s0 = 0.f, c0 = 0.f, s1 = 0.f, c1 = 0.f, s2 = 0.f, c2 = 0.f;
      int x = wx0;
      if constexpr (TILED) {  // window passes, grid exchanges between them (control warp)
        const TmaPass TP{p.tmaps, reinterpret_cast<unsigned long long*>(tiles_base),
                         reinterpret_cast<float2*>(tiles_base + 128), &S.tma_fail, &tph, &p.st->status, p.timeout_ns};
        for (int w = 0; w < nwin; ++w) {
          // basis indices: q_it is vector it - 1, q_{it-1} vector it - 2, u vector it
          // (from it = 2 on, window 0 first turns u_{it-1} in vector
          // it - 1 into q_it = u_{it-1} - alpha s q_{it-1}: ORTH)
          const int iq = it - 1, ia = w == 0 ? (it > 1 ? it - 2 : 0) : it, iu = it;
          if (w == 0) {
            const float am = S.am;
            if (nwin == 1) {
              if (it > 1)
                c_tiled_pass<true, true, true>(TP, op, c, S.bx, iq, ia, iu, win[0], 0, wstep, s0, c0, s1, c1, am, &s2,
                                               &c2);
              else
                c_tiled_pass<true, true>(TP, op, c, S.bx, iq, ia, iu, win[0], 0, wstep, s0, c0, s1, c1);
            } else {
              if (it > 1)
                c_tiled_pass<true, false, true>(TP, op, c, S.bx, iq, ia, iu, win[0], 0, wstep, s0, c0, s1, c1, am, &s2,
                                                &c2);
              else
                c_tiled_pass<true, false>(TP, op, c, S.bx, iq, ia, iu, win[0], 0, wstep, s0, c0, s1, c1);
            }
          } else if (w == nwin - 1) {
            c_tiled_pass<false, true>(TP, op, c, S.bx, iq, ia, iu, win[w], w, wstep, s0, c0, s1, c1);
          } else {
            c_tiled_pass<false, false>(TP, op, c, S.bx, iq, ia, iu, win[w], w, wstep, s0, c0, s1, c1);
          }
          if (w + 1 < nwin) {
            window_written_sync();    // all threads: window w written
            window_exchanged_sync();  // all threads: the grid exchange passed
          }
        }
      } else if constexpr (STAGED) {
        const unsigned rank = cluster_rank();
        for (int j = 2 * tid; j < wxe - xb; j += 2 * wstep) {
          float4 h, v;
          c_apply_spin_staged2(sq, q, qm, j, rank, op, c, S.bx, h, v);
          *reinterpret_cast<float4*>(u + xb + j) = h;
          ff_add_prod(s0, c0, v.x, h.x);
          ff_add_prod(s0, c0, v.y, h.y);
          ff_add_prod(s0, c0, v.z, h.z);
          ff_add_prod(s0, c0, v.w, h.w);
          ff_add_prod(s1, c1, h.x, h.x);
          ff_add_prod(s1, c1, h.y, h.y);
          ff_add_prod(s1, c1, h.z, h.z);
          ff_add_prod(s1, c1, h.w, h.w);
        }
      } else {
        // spin apply on two elements per thread and loop iteration (twice the
        // independent neighbour loads per warp)
        if constexpr (FAMILY == kFamilySpin) {
          for (; x + wstep < wxe; x += 2 * wstep) {
            float2 h1, h2;
            c_apply_spin2(q, qm, x, x + wstep, op, c, S.bx, h1, h2);
            u[x] = h1;
            u[x + wstep] = h2;
            const float2 v1 = q[x], v2 = q[x + wstep];
            ff_add_prod(s0, c0, v1.x, h1.x);
            ff_add_prod(s0, c0, v1.y, h1.y);
            ff_add_prod(s0, c0, v2.x, h2.x);
            ff_add_prod(s0, c0, v2.y, h2.y);
            ff_add_prod(s1, c1, h1.x, h1.x);
            ff_add_prod(s1, c1, h1.y, h1.y);
            ff_add_prod(s1, c1, h2.x, h2.x);
            ff_add_prod(s1, c1, h2.y, h2.y);
          }
        }
        for (; x < wxe; x += wstep) {
          float2 hv;
          if constexpr (FAMILY == kFamilySpin) hv = c_apply_spin(q, qm, x, op, c, S.bx);
          else if constexpr (FAMILY == kFamilyDia) hv = c_apply_dia(q, qm, x, dim, op, c);
          else hv = c_apply_csr(q, qm, x, dim, op, c);
          u[x] = hv;
          const float2 v = q[x];
          ff_add_prod(s0, c0, v.x, hv.x);
          ff_add_prod(s0, c0, v.y, hv.y);
          ff_add_prod(s1, c1, hv.x, hv.x);
          ff_add_prod(s1, c1, hv.y, hv.y);
        }
      }
      c_worker_partial(S, s0, c0, 0);
      c_worker_partial(S, s1, c1, 1);
      if constexpr (TILED) c_worker_partial(S, s2, c2, 2);  // ||q_it||^2 of the w stored in window 0
      if (tid == 0) S.tacc[0] += (S.twe = sm_clock()) - tw0;
    } else if (cmd == kCOrth) {
      // -------- phase B: w = u - alpha s q_it, ||w||^2 of the stored w for the
      // next iteration (the tiled form does it in the next window 0)
      const int it = S.it;
      const float am = S.am;
      const float2* q = Q(it);
      float2* u = Q(it + 1);
      float s0 = 0.f, c0 = 0.f;
      int x = wx0;
      // four elements per step with every load issued first (more bytes
      // in flight per thread); the sums keep the order of the plain loop
      for (; x + 3 * wstep < wxe; x += 4 * wstep) {
        float2 v[4], uu[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          v[j] = q[x + j * wstep];
          uu[j] = u[x + j * wstep];
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const float2 w = make_float2(fmaf(am, v[j].x, uu[j].x), fmaf(am, v[j].y, uu[j].y));
          u[x + j * wstep] = w;
          if constexpr (STAGED) sq[x + j * wstep - xb] = w;
          ff_add_prod(s0, c0, w.x, w.x);
          ff_add_prod(s0, c0, w.y, w.y);
        }
      }
      for (; x < wxe; x += wstep) {
        const float2 v = q[x];
        const float2 uu = u[x];
        const float2 w = make_float2(fmaf(am, v.x, uu.x), fmaf(am, v.y, uu.y));
        u[x] = w;
        if constexpr (STAGED) sq[x - xb] = w;
        ff_add_prod(s0, c0, w.x, w.x);
        ff_add_prod(s0, c0, w.y, w.y);
      }
      c_worker_partial(S, s0, c0, 0);
      if (tid == 0) S.tacc[2] += (S.twe = sm_clock()) - tw0;
    } else if (cmd == kCRec) {
      // -------- reconstruct q_1 <- beta0 sum_i y_i s_i q_i
      const int acc_k = S.it;
      const bool final_rec = S.final_rec;
      float s = 0.f, cc = 0.f;
      for (int x = wx0; x < wxe; x += wstep) {
        float re = 0.f, im = 0.f;
        int i = 0;
        for (; i + 3 < acc_k; i += 4) {  // four basis loads in flight before their use (same order)
          float2 v[4];
#pragma unroll
          for (int j = 0; j < 4; ++j) v[j] = Q(i + j + 1)[x];
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const float cr = S.cr[i + j], ci = S.ci[i + j];
            re = fmaf(cr, v[j].x, fmaf(-ci, v[j].y, re));
            im = fmaf(cr, v[j].y, fmaf(ci, v[j].x, im));
          }
        }
        for (; i < acc_k; ++i) {
          const float2 v = Q(i + 1)[x];
          const float cr = S.cr[i], ci = S.ci[i];
          re = fmaf(cr, v.x, fmaf(-ci, v.y, re));
          im = fmaf(cr, v.y, fmaf(ci, v.x, im));
        }
        Q(1)[x] = make_float2(re, im);
        if constexpr (STAGED) sq[x - xb] = make_float2(re, im);
        if (final_rec) p.psi[x] = make_double2((double)re, (double)im);
        ff_add_prod(s, cc, re, re);
        ff_add_prod(s, cc, im, im);
      }
      c_worker_partial(S, s, cc);
      if (tid == 0) S.tacc[4] += (S.twe = sm_clock()) - tw0;
    } else {
      // -------- psi (complex128) -> q_1 (complex64), ||q_1||^2, finiteness
      float s = 0.f, c = 0.f;
      int bad = 0;
      for (int x = wx0; x < wxe; x += wstep) {
        const double2 v = p.psi[x];
        bad |= !(isfinite(v.x) && isfinite(v.y));
        const float2 f = make_float2((float)v.x, (float)v.y);
        Q(1)[x] = f;
        if constexpr (STAGED) sq[x - xb] = f;
        ff_add_prod(s, c, f.x, f.x);
        ff_add_prod(s, c, f.y, f.y);
      }
      if (__any_sync(0xffffffffu, bad) && lane == 0) atomicCAS(&p.st->status, 0, (int)CFET_ENAN);
      c_worker_partial(S, s, c);
    }
    __syncthreads();  // the pass is done
  }
}

template <int FAMILY, class Op, int MODE>
__device__ __forceinline__ void c_control(const PropParams& p, const Op& op, SmemC& S, int NW) {
  constexpr bool TILED = MODE == kCTiled;
  const int lane = threadIdx.x & 31;
  const int G = gridDim.x;
  const int ncoef = 1 + p.nV;
  DevStatus* const st = p.st;
  // record exchange (ctl_exchange): tags continue across launches
  unsigned tag = (unsigned)ld_volatile_i32((const int*)&st->tag_base);
  unsigned long long* const rec = reinterpret_cast<unsigned long long*>(p.partials);
  const bool glead = blockIdx.x == 0 && lane == 0;
  const bool fixed_k = p.tol <= 0.0;
  const bool forced = p.f_nsub != nullptr;
  if (lane == 0) {
    for (int i = 0; i < 8; ++i) S.tacc[i] = 0;
    S.n_app = S.n_sub = 0;
    S.rpos = st->rec_pos;
    S.fpos = st->forced_pos;
    S.max_k = 0;
    S.max_err = 0.0;
    S.e = 0;
  }
  auto start = [&](int cmd, int it) {  // one element pass of the workers
    if (lane == 0) {
      S.cmd = cmd;
      S.it = it;
    }
    __syncwarp();
    __syncthreads();
  };

  // ---------------- psi (complex128) -> q_1 (complex64)
  start(kCConvert, 0);
  __syncthreads();
  if (!c_ctl_reduce_cold(S, NW, rec, ++tag, &st->status, p.timeout_ns)) return;
  if (ld_volatile_i32(&st->status) != 0) return;

  while (S.e < p.nexp) {
    if (lane < ncoef) S.scal[lane] = p.scal[S.e * ncoef + lane];
    if (lane == 0) {
      S.remaining = p.tau;
      S.nsub_e = 0;
    }
    __syncwarp();
    if constexpr (FAMILY == kFamilySpin) {
      if (lane < op.N) {
        double bi = 0.0;
        for (int k = 0; k < p.nV; ++k) bi = fma(S.scal[1 + k], __ldg(op.xf + k * op.N + lane), bi);
        S.bsite_raw[lane] = bi;
        if (lane == 0) {
          S.cst[0] = S.scal[0];
          S.cst[1] = S.scal[0] * op.J2;
          S.cst[2] = bi;
        }
      }
      __syncwarp();
    }
    while (true) {
      if (S.nsub_e >= p.max_substeps || (forced && S.nsub_e >= p.f_nsub[p.exp_base + S.e])) {
        if (glead) atomicCAS(&st->status, 0, (int)CFET_EKRYLOV);
        return;
      }
      const int klimit = forced ? p.f_k[S.fpos] : p.m_max;
      int acc_k = 0, acc_h = 0;
      if (lane == 0) S.acc_err = 0.0;
      if (S.beta0 != 0.0) {
        if (lane == 0) {
          S.scale[1] = div_call(1.0, S.beta0);
          S.y_ready = 0;
        }
        __syncwarp();
        c_const_a<FAMILY>(S, op, 1);
        bool accepted = false, pend = false;
        int it = 1;
        for (;; ++it) {
          // -------- phase A(it) on the workers; deferred estimate of it-1 here
          start(kCApply, it);
          bool stop_prev = false;
          if (pend) {
            const long long te0 = sm_clock();
            stop_prev = c_check(S, it - 1, p.tol, p.tau) != 0;
            if (lane == 0) S.tacc[6] += sm_clock() - te0;
          }
          if constexpr (TILED) {  // grid exchanges between the window passes of the workers
            TileWin win[kTiledMaxWindows] = {};
            const int nwin = tiled_windows<kTileBits>(op.N, win);
            bool ok = true;
            for (int w = 0; w + 1 < nwin; ++w) {
              window_written_sync();
              double none[1];
              ok = ok && c_ctl_reduce<0>(S, NW, rec, ++tag, true, &st->status, p.timeout_ns, none, S.tacc[5]);
              window_exchanged_sync();
            }
            if (!ok) {
              __syncthreads();
              return;
            }
          }
          __syncthreads();
          {
            const long long sp0 = S.tacc[5];
            double sum[3];
            // (the tiled apply leaves u written by other CTAs: fence; it also
            // carries ||q_it||^2 of the w that its window 0 stored)
            if (!c_ctl_reduce<TILED ? 3 : 2>(S, NW, rec, ++tag, TILED, &st->status, p.timeout_ns, sum, S.tacc[5]))
              return;
            if (stop_prev) {  // the deferred estimate accepted it-1
              it -= 1;
              accepted = true;
              break;
            }
            if (lane == 0) {
              if (TILED && it > 1) S.qnorm2[it] = sum[2];
              // q_it holds the Lanczos vector v_it times 1/scale[it]:
              // alpha = <v, u>,  ||w||^2 = ||u - alpha v||^2
              //       = ||u||^2 - alpha^2 (2 - s^2 ||q||^2)
              // (the stored q is a unit vector only to FP32 rounding, which the
              // last factor keeps out of the cancellation)
              const double s_it = S.scale[it];
              const double alpha = sum[0] * s_it;
              S.alpha[it] = alpha;
              S.am = (float)(-alpha * s_it);
              S.wnorm2 = sum[1] - alpha * alpha * (2.0 - s_it * s_it * S.qnorm2[it]);
              S.tacc[1] += sm_clock() - S.twe - (S.tacc[5] - sp0);
            }
          }
          // -------- phase B(it): w = u - alpha s_it q_it on the workers (the
          // tiled form does it in the next iteration's window 0); beta (known
          // from the phase-A sums), the decisions and the next iteration's
          // constants here at the same time
          if constexpr (!TILED) start(kCOrth, it);
          else __syncwarp();
          bool acc = false;
          {
            const long long tc0 = sm_clock();
            // beta and 1/beta from one reciprocal square root (a rounding-level
            // negative ||w||^2 is an exact breakdown)
            const double wn = S.wnorm2;
            const double rb = wn > 0.0 ? rsqrt(wn) : 0.0;
            const double b = wn > 0.0 ? wn * rb : 0.0;
            const double prev_b = it > 1 ? S.beta[it - 1] : 0.0;
            const bool breakdown =
                sb_no_breakdown(b, S.alpha[it], prev_b) != 1 && b <= 1e-13 * (fabs(S.alpha[it]) + prev_b + 1.0);
            int gate = -1;
            __syncwarp();
            if (lane == 0) {
              S.beta[it] = b;
              S.scale[it + 1] = rb;
              gate = krylov_bounds_update(S, it, S.remaining);
              S.acc_err = 0.0;
            }
            gate = __shfl_sync(0xffffffffu, gate, 0);
            __syncwarp();
            pend = false;
            if (forced) {
              acc = it == klimit;
            } else if (fixed_k) {
              acc = it == p.m_max || breakdown;
            } else if (breakdown) {
              acc = true;
            } else if (it >= p.m_min &&
                       (gate >= 0 ? gate == 1
                                  : fabs(S.remaining) * gersh_width(it, S.alpha + 1, S.beta + 1) <= 2.0 * it)) {
              if (it < klimit) pend = true;  // the estimate runs during the next apply
              else acc = c_check(S, it, p.tol, p.tau) != 0;
            }
            if (!acc && it < klimit) c_const_a<FAMILY>(S, op, it + 1);
            if (lane == 0) S.tacc[3] += sm_clock() - tc0;
          }
          if constexpr (!TILED) {
            __syncthreads();
            if (!acc && it < klimit) {
              // every CTA's w must be visible before the next apply reads it; the
              // exchange also carries ||w||^2 of the stored w
              double wsum[1];
              if (!c_ctl_reduce<1>(S, NW, rec, ++tag, true, &st->status, p.timeout_ns, wsum, S.tacc[5])) return;
              if (lane == 0) S.qnorm2[it + 1] = wsum[0];
            }
          }
          __syncwarp();
          if (acc) {
            accepted = true;
            break;
          }
          if (it >= klimit) break;
        }
        acc_k = it;
        if (forced) {
          acc_h = p.f_h[S.fpos];
        } else if (!accepted) {
          // halve the substep on the same basis until the estimate meets the
          // proportional tolerance
          c_halve(S, it, p.tol, p.tau);
          acc_h = S.acc_h;
          if (acc_h == 0) {
            if (glead) atomicCAS(&st->status, 0, (int)CFET_EKRYLOV);
            return;
          }
        }
        // -------- reconstruct q_1 <- beta0 sum_i y_i s_i q_i
        {
          const long long tr0 = sm_clock();
          c_rec_consts(S, acc_k, ldexp(S.remaining, -acc_h));
          if (lane == 0) {
            S.final_rec = S.e == p.nexp - 1 && acc_h == 0;
            S.tacc[6] += sm_clock() - tr0;
          }
        }
        start(kCRec, acc_k);
        __syncthreads();
        if (!c_ctl_reduce_cold(S, NW, rec, ++tag, &st->status, p.timeout_ns)) return;
      }
      if (lane == 0) {
        if (glead && p.r_k != nullptr) {
          if (S.rpos < p.r_cap) {
            p.r_k[S.rpos] = acc_k;
            p.r_h[S.rpos] = acc_h;
          } else {
            st->rec_overflow = 1;
          }
        }
        S.rpos += 1;
        S.n_sub += 1;
        S.n_app += acc_k;
        if (acc_k > S.max_k) S.max_k = acc_k;
        if (S.acc_err > S.max_err) S.max_err = S.acc_err;
        if (forced) S.fpos += 1;
        S.nsub_e += 1;
        S.remaining -= ldexp(S.remaining, -acc_h);
      }
      __syncwarp();
      if (acc_h == 0) break;
    }
    if (glead && p.r_nsub != nullptr) p.r_nsub[p.exp_base + S.e] = S.nsub_e;
    if (lane == 0) S.e += 1;
    __syncwarp();
  }
  if (glead) {
    st->tag_base = tag;
    st->forced_pos = S.fpos;
    st->rec_pos = S.rpos;
    st->n_exp += p.nexp;
    st->n_sub += S.n_sub;
    st->n_app += S.n_app;
    if (S.max_k > st->max_k) st->max_k = S.max_k;
    if (S.max_err > st->max_err) st->max_err = S.max_err;
  }
  if (lane < 8) {  // every CTA: mean and max of its phase times (see cfet_stats.phase_ns), SM clock cycles
    const long long t = S.tacc[lane];
    atomicAdd((unsigned long long*)&st->phase_ns[lane], (unsigned long long)(t / G));
    atomicMax(&st->phase_max_ns[lane], t);
  }
}

template <int FAMILY, class Op, int MODE>
__global__ void __launch_bounds__(CFET_CTL_MAX_THREADS, 1) k_propagate_c64(PropParams p, Op op) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  SmemC& S = *reinterpret_cast<SmemC*>(smem_raw);
  const int NW = (int)(blockDim.x >> 5) - 1;
  if constexpr (MODE == kCStaged) {
    if (!cluster_is(kStagedCluster, &p.st->status)) return;
  }
  // tiled apply: the stages' mbarriers and tile buffers behind SmemC
  unsigned char* const tiles_base = smem_raw + ((sizeof(SmemC) + 127) & ~size_t(127));
  if constexpr (MODE == kCTiled) {
    if (threadIdx.x == 0) {  // ordered before any use by the CTA barriers of the conversion pass
      for (int s2 = 0; s2 < kTmaStages; ++s2) mbar_init(reinterpret_cast<unsigned long long*>(tiles_base) + s2, 1);
      S.tma_fail = 0;
      mbar_init_fence();
    }
  }
  if ((int)(threadIdx.x >> 5) < NW) {
    c_worker<FAMILY, Op, MODE>(p, op, S, tiles_base, NW * 32);
  } else {
    c_control<FAMILY, Op, MODE>(p, op, S, NW);
    __syncwarp();
    if ((threadIdx.x & 31) == 0) S.cmd = kCExit;  // also after an error
    __syncwarp();
    __syncthreads();
  }
  if constexpr (MODE == kCStaged) {
    __syncwarp();
    cluster_sync_all();  // no CTA leaves while another may read its shared memory
  }
}

// ------------------------------------------------------------------ launchers
size_t c64_tiled_smem_bytes() {
  return ((sizeof(SmemC) + 127) & ~size_t(127)) + 128 + (size_t)kTmaStages * 2 * kTileBytes;
}

static size_t c64_staged_smem_bytes(int part) {
  return ((sizeof(SmemC) + 127) & ~size_t(127)) + (size_t)part * sizeof(float2);
}

template <int FAMILY, class Op>
static int launch_prop_c64(const PropParams& p, const Op& op, int grid, int block, void* stream) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(block);
  cfg.dynamicSmemBytes = p.tiled     ? c64_tiled_smem_bytes()
                         : p.cluster ? c64_staged_smem_bytes(p.dim / grid)
                                     : sizeof(SmemC);
  cfg.stream = (cudaStream_t)stream;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeCooperative;
  at[0].val.cooperative = 1;
  at[1].id = cudaLaunchAttributeClusterDimension;
  at[1].val.clusterDim.x = p.cluster;
  at[1].val.clusterDim.y = 1;
  at[1].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = p.cluster ? 2 : 1;
  if constexpr (FAMILY == kFamilySpin) {
    if (p.tiled) return (int)cudaLaunchKernelEx(&cfg, k_propagate_c64<FAMILY, Op, kCTiled>, p, op);
    if (p.cluster) return (int)cudaLaunchKernelEx(&cfg, k_propagate_c64<FAMILY, Op, kCStaged>, p, op);
  }
  return (int)cudaLaunchKernelEx(&cfg, k_propagate_c64<FAMILY, Op, kCGrid>, p, op);
}

bool c64_staged_prepare(int dim, int block) {
  return staged_fits((const void*)k_propagate_c64<kFamilySpin, OpSpinC, kCStaged>, kStagedGrid, kStagedCluster, block,
                     c64_staged_smem_bytes(dim / kStagedGrid));
}

int launch_propagate_spin_c64(const PropParams& p, const OpSpinC& op, int grid, int block, void* stream) {
  return launch_prop_c64<kFamilySpin>(p, op, grid, block, stream);
}
int launch_propagate_dia_c64(const PropParams& p, const OpDiaC& op, int grid, int block, void* stream) {
  return launch_prop_c64<kFamilyDia>(p, op, grid, block, stream);
}
int launch_propagate_csr_c64(const PropParams& p, const OpCsrC& op, int grid, int block, void* stream) {
  return launch_prop_c64<kFamilyCsr>(p, op, grid, block, stream);
}

int max_coresident_blocks_c64(int family, int block, bool tiled) {
  int dev = 0, nsm = 0, per = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  // a few KB of shared memory: leave the unified storage to L1 (a tiled launch
  // asks for its tile buffers and gets the shared-memory split it needs)
  cudaFuncSetAttribute(k_propagate_c64<kFamilySpin, OpSpinC, kCGrid>, cudaFuncAttributePreferredSharedMemoryCarveout, 0);
  cudaFuncSetAttribute(k_propagate_c64<kFamilyDia, OpDiaC, kCGrid>, cudaFuncAttributePreferredSharedMemoryCarveout, 0);
  cudaFuncSetAttribute(k_propagate_c64<kFamilyCsr, OpCsrC, kCGrid>, cudaFuncAttributePreferredSharedMemoryCarveout, 0);
  cudaFuncSetAttribute(k_propagate_c64<kFamilySpin, OpSpinC, kCTiled>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                       (int)c64_tiled_smem_bytes());
  cudaError_t e;
  if (family == kFamilySpin)
    e = tiled ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_propagate_c64<kFamilySpin, OpSpinC, kCTiled>, block,
                                                              c64_tiled_smem_bytes())
              : cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_propagate_c64<kFamilySpin, OpSpinC, kCGrid>, block, sizeof(SmemC));
  else if (family == kFamilyCsr)
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_propagate_c64<kFamilyCsr, OpCsrC, kCGrid>, block,
                                                      sizeof(SmemC));
  else
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_propagate_c64<kFamilyDia, OpDiaC, kCGrid>, block,
                                                      sizeof(SmemC));
  if (e != cudaSuccess) return -1;
  return per * nsm;
}

}  // namespace cfet
