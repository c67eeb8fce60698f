// Fixed-point number format of the Krylov and Chebyshev kernels (sm_103a):
// int64 (re, im) mantissas with one exponent per vector, exact integer
// neighbour sums, products of a scalar mantissa with a stored value by the
// high half of a 64 x 64 product, exact 128-bit reductions; and the stage
// operator applies in that format (XXZ chain, DIA, CSR).  See kernels_fx.cu for
// the number format's bounds and rounding.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

#include "cfet_internal.h"
#include "device_common.cuh"
#include "scalar_bounds.cuh"

namespace cfet {

// ------------------------------------------------------------------ fixed-point helpers
constexpr int kFxBits = 57;  // stored |M| < 2^57
// Per-thread exact 128-bit sums of products (< 2^115 each, at most 4096 per
// thread) are shifted right by kRedShift before the CTA and grid reductions,
// so that up to 2^17 threads cannot overflow 127 bits; the dropped bits are
// below 2^-68 of any non-zero sum of squares.
constexpr int kRedShift = 24;

// The scalar bookkeeping below uses integer operations on the bit patterns of
// positive normal doubles (the FP64 units run at 1/64 rate).
__device__ __forceinline__ int fx_ilog2(double v) {  // floor(log2 v), v > 0 normal
  return (int)((__double_as_longlong(v) >> 52) & 0x7ff) - 1023;
}
// floor(log2(v (1 + eps))) for a tiny eps > 0: values within 2^-40 below a power
// of two count as that power (a safety margin for bounds computed in FP64).
__device__ __forceinline__ int fx_ilog2_up(double v) {
  const long long b = __double_as_longlong(v);
  const int e = (int)((b >> 52) & 0x7ff) - 1023;
  return ((b & 0xFFFFFFFFFFFFFLL) >= 0xFFFFFFFFFF000LL) ? e + 1 : e;
}
// Exponent E with bound < 2^(bits + E); a zero, negative, tiny (< 2^-963)
// or huge bound gives a very small E.  (Range checks on the bit pattern.)
__device__ __forceinline__ int fx_exp_for(double bound, int bits) {
  const long long b = __double_as_longlong(bound);
  const int ex = (int)((b >> 52) & 0x7ff);
  if (b <= 0 || ex < 1023 - 963 || ex > 1023 + 963) return -960;
  return fx_ilog2_up(bound) - (bits - 1);
}
// x * 2^e exactly, by exponent arithmetic when the result stays normal.
__device__ __forceinline__ double fx_scale2(double x, int e) {
  const long long b = __double_as_longlong(x);
  const int ex = (int)((b >> 52) & 0x7ff);
  if (ex == 0 || ex + e <= 0 || ex + e >= 2047) return ldexp(x, e);
  return __longlong_as_double(b + ((long long)e << 52));
}

// Exact decomposition v = m * 2^e with |m| in [2^61, 2^62) (m = 0 for 0).
struct Mant {
  long long m;
  int e;
};
__device__ __forceinline__ Mant fx_mant(double v) {
  Mant r;
  const long long b = __double_as_longlong(v);
  const int ex = (int)((b >> 52) & 0x7ff);
  if (ex == 0) { r.m = 0; r.e = 0; return r; }  // zero (subnormals treated as zero)
  const long long frac = (b & 0xFFFFFFFFFFFFFLL) | (1LL << 52);
  r.m = frac << 9;
  r.e = ex - 1075 - 9;
  if (b < 0) r.m = -r.m;
  return r;
}

// h * 2^-s rounded (half up); s is uniform across the warp.
__device__ __forceinline__ long long fx_rshr(long long h, int s) {
  if (s <= 0) return s <= -62 ? 0LL : (h << (-s));
  if (s >= 63) return 0LL;
  return (h + (1LL << (s - 1))) >> s;
}
// round(m * x * 2^-(64 + s)); |m|, |x| < 2^62.
// High 64 bits of m * x from three 32x32 partial products (the dropped low
// partial product changes the result by at most 2 units).
__device__ __forceinline__ long long fx_mulhi(long long m, long long x) {
  const int mh = (int)(m >> 32), xh = (int)(x >> 32);
  const unsigned ml = (unsigned)m, xl = (unsigned)x;
  // 32 x 32 -> 64-bit partial products; |mid| < 2^63 for |m|, |x| < 2^62
  const long long mid = (long long)mh * (long long)xl + (long long)xh * (long long)ml;
  return (long long)mh * (long long)xh + (mid >> 32);
}
__device__ __forceinline__ long long fx_mul(long long m, long long x, int s) {
  return fx_rshr(fx_mulhi(m, x), s);
}
// Scalar mantissa with the product shift folded in: fx_mulhi(fx_fold(m, s), x)
// ~= fx_mul(m, x, s).  For s <= 9 the fold is exact (the mantissa of a double
// uses 53 of its 62 bits); for larger s the term is at most 2^-s of the result
// bound and the dropped bits stay below 2^-62 of it.  s < 0 does not occur for
// non-zero terms (the result bound covers every term); it is clamped.
__device__ __forceinline__ long long fx_fold(long long m, int s) {
  if (s <= 0) return m;
  if (s >= 63) return 0;
  return (m + (1LL << (s - 1))) >> s;
}
// p * 2^-sh as int64 (truncated); callers guarantee the result fits.
__device__ __forceinline__ long long fx_shr128(__int128 p, int sh) {
  if (sh >= 127) return p < 0 ? -1LL : 0LL;
  if (sh >= 0) return (long long)(p >> sh);
  if (sh <= -63) return 0LL;
  return (long long)(p << (-sh));
}
__device__ __forceinline__ long long fx_absmax(long long a, long long b) {
  const long long x = a < 0 ? -a : a, y = b < 0 ? -b : b;
  return x > y ? x : y;
}

// ------------------------------------------------------------------ exact reductions
// Sum over a warp of (lo, hi) 128-bit values and max of a non-negative int64,
// results in every lane.  The sum goes through five 26-bit limbs (the top one
// signed, |value| < 2^122), each one warp reduction instruction: shorter than
// five levels of six shuffles with carries.
__device__ __forceinline__ void fx_warp_reduce(unsigned long long& lo, long long& hi, long long& mx) {
  constexpr unsigned kM26 = (1u << 26) - 1u, kAll = 0xffffffffu;
  const unsigned r0 = __reduce_add_sync(kAll, (unsigned)lo & kM26);
  const unsigned r1 = __reduce_add_sync(kAll, (unsigned)(lo >> 26) & kM26);
  const unsigned r2 = __reduce_add_sync(kAll, ((unsigned)(lo >> 52) | ((unsigned)hi << 12)) & kM26);
  const unsigned r3 = __reduce_add_sync(kAll, (unsigned)(hi >> 14) & kM26);
  const int r4 = __reduce_add_sync(kAll, (int)(hi >> 40));
  const unsigned mh = (unsigned)((unsigned long long)mx >> 32);
  const unsigned xh = __reduce_max_sync(kAll, mh);
  const unsigned xl = __reduce_max_sync(kAll, mh == xh ? (unsigned)mx : 0u);
  const unsigned long long t = (unsigned long long)r0 + ((unsigned long long)r1 << 26);
  lo = t + ((unsigned long long)r2 << 52);
  hi = (long long)(r2 >> 12) + (lo < t ? 1 : 0) + ((long long)r3 << 14) + ((long long)r4 << 40);
  mx = (long long)(((unsigned long long)xh << 32) | xl);
}
// (hi 2^64 + lo) 2^kRedShift rounded to the nearest double, by integer operations.
__device__ __forceinline__ double fx_i128_to_double(unsigned long long lo, long long hi) {
  return sb_i128_to_double(lo, hi, kRedShift);
}


// ------------------------------------------------------------------ apply constants
struct FxConstA {
  // spin: mantissas of the diagonal, hop, uniform field and q_{k-1} terms with
  // their product shifts folded in, and the normalising shifts of their inputs
  // (by name, or by term number)
  union {
    struct { long long m_cz, m_hop, m_x, m_p; };
    long long m4[4];
  };
  union {
    struct { int pk, ph, px, pp; };
    int p4[4];
  };
  int use_prev;
  int Eu;
  // dia: per operator P_o = shr128(sum VAL q, sh_pre[o]); term = fx_mul(m_op[o], P_o, s_op[o])
  long long m_op[1 + kMaxDrives];
  int sh_pre[1 + kMaxDrives];
};

// ------------------------------------------------------------------ applies
// WIDE (chains of at most kWideSites sites, vectors in shared memory): the
// neighbour loops are unrolled whole, so that all loads of an element are in
// flight at once; one warp per scheduler has nothing else to hide them behind.
constexpr int kWideSites = 10;
template <bool WIDE>
__device__ __forceinline__ longlong2 fx_apply_spin(const longlong2* q, const longlong2* qm, int x,
                                                   const OpSpinFx& op, const FxConstA& c, const long long* mb) {
  const int N = op.N, L = op.lo_bits;
  const long long dz = __ldg(op.DZ_lo + (x & ((1 << L) - 1))) + __ldg(op.DZ_hi + (x >> (L - 1)));
  // D = c0 s_k dz(x) (m_cz carries the shift), then D * q_k[x]
  const long long Dp = fx_mulhi(c.m_cz, dz << 1) << 3;
  const longlong2 v = q[x];
  long long ur = fx_mulhi(Dp, v.x << c.pk);
  long long ui = fx_mulhi(Dp, v.y << c.pk);
  long long hr = 0, hi = 0;
  const unsigned anti = ((unsigned)x ^ ((unsigned)x >> 1)) & ((1u << (N - 1)) - 1u);
  constexpr int kUnroll = WIDE ? kWideSites : 4;
#pragma unroll kUnroll
  for (int i = 0; i < (WIDE ? kWideSites : N - 1); ++i) {  // antiparallel bonds only (predicated)
    if ((anti >> i) & 1u) {
      const longlong2 w = q[x ^ (3 << i)];
      hr += w.x;
      hi += w.y;
    }
  }
  ur += fx_mulhi(c.m_hop, hr << c.ph);
  ui += fx_mulhi(c.m_hop, hi << c.ph);
  if (op.uniform) {
    long long xr = 0, xi = 0;
#pragma unroll kUnroll
    for (int i = 0; i < (WIDE ? kWideSites : N); ++i) {
      if (WIDE && i >= N) break;
      const longlong2 w = q[x ^ (1 << i)];
      xr += w.x;
      xi += w.y;
    }
    ur += fx_mulhi(c.m_x, xr << c.px);
    ui += fx_mulhi(c.m_x, xi << c.px);
  } else {
#pragma unroll kUnroll
    for (int i = 0; i < (WIDE ? kWideSites : N); ++i) {
      if (WIDE && i >= N) break;
      const longlong2 w = q[x ^ (1 << i)];
      ur += fx_mulhi(mb[i], w.x << c.pk);
      ui += fx_mulhi(mb[i], w.y << c.pk);
    }
  }
  if (c.use_prev) {
    const longlong2 w = qm[x];
    ur += fx_mulhi(c.m_p, w.x << c.pp);
    ui += fx_mulhi(c.m_p, w.y << c.pp);
  }
  return make_longlong2(ur, ui);
}

// One element of a chain whose applied vector is staged in the shared memory of
// the cluster's CTAs, 2^lc elements each (x = rank 2^lc + j): flips and hops of
// bits below lc read this CTA's part, those of the rank's bits the same (or, for
// the bond across, a neighbouring) element of another CTA's part.
__device__ __forceinline__ longlong2 fx_ld_cluster(unsigned base, int j) {
  longlong2 v;
  asm volatile("ld.shared::cluster.v2.s64 {%0, %1}, [%2];" : "=l"(v.x), "=l"(v.y) : "r"(base + 16u * (unsigned)j));
  return v;
}
__device__ __forceinline__ longlong2 fx_apply_spin_cluster(const longlong2* sq, const longlong2* qm, int j, int rank,
                                                           int lc, const OpSpinFx& op, const FxConstA& c,
                                                           const long long* mb, longlong2& v) {
  const int N = op.N, L = op.lo_bits;
  const int x = (rank << lc) | j;
  longlong2 wp = make_longlong2(0, 0);
  if (c.use_prev) wp = qm[x];  // global memory: issued ahead of the neighbour sums
  const long long dz = __ldg(op.DZ_lo + (x & ((1 << L) - 1))) + __ldg(op.DZ_hi + (x >> (L - 1)));
  v = sq[j];
  long long hr = 0, hi = 0;
  const unsigned anti = ((unsigned)x ^ ((unsigned)x >> 1)) & ((1u << (N - 1)) - 1u);
  for (int i = lc - 1; i < N - 1; ++i)
    if ((anti >> i) & 1u) {  // bond across (i = lc - 1) and bonds of the rank's bits
      const unsigned other = i == lc - 1 ? 1u : 3u << (i - lc);
      const longlong2 w = fx_ld_cluster(cluster_addr(sq, (unsigned)rank ^ other), i == lc - 1 ? j ^ (1 << i) : j);
      hr += w.x;
      hi += w.y;
    }
#pragma unroll 4
  for (int i = 0; i < lc - 1; ++i)
    if ((anti >> i) & 1u) {
      const longlong2 w = sq[j ^ (3 << i)];
      hr += w.x;
      hi += w.y;
    }
  const long long Dp = fx_mulhi(c.m_cz, dz << 1) << 3;
  long long ur = fx_mulhi(Dp, v.x << c.pk) + fx_mulhi(c.m_hop, hr << c.ph);
  long long ui = fx_mulhi(Dp, v.y << c.pk) + fx_mulhi(c.m_hop, hi << c.ph);
  if (op.uniform) {
    long long xr = 0, xi = 0;
    for (int i = lc; i < N; ++i) {
      const longlong2 w = fx_ld_cluster(cluster_addr(sq, (unsigned)rank ^ (1u << (i - lc))), j);
      xr += w.x;
      xi += w.y;
    }
#pragma unroll 4
    for (int i = 0; i < lc; ++i) {
      const longlong2 w = sq[j ^ (1 << i)];
      xr += w.x;
      xi += w.y;
    }
    ur += fx_mulhi(c.m_x, xr << c.px);
    ui += fx_mulhi(c.m_x, xi << c.px);
  } else {
    for (int i = lc; i < N; ++i) {
      const longlong2 w = fx_ld_cluster(cluster_addr(sq, (unsigned)rank ^ (1u << (i - lc))), j);
      ur += fx_mulhi(mb[i], w.x << c.pk);
      ui += fx_mulhi(mb[i], w.y << c.pk);
    }
#pragma unroll 4
    for (int i = 0; i < lc; ++i) {
      const longlong2 w = sq[j ^ (1 << i)];
      ur += fx_mulhi(mb[i], w.x << c.pk);
      ui += fx_mulhi(mb[i], w.y << c.pk);
    }
  }
  if (c.use_prev) {
    ur += fx_mulhi(c.m_p, wp.x << c.pp);
    ui += fx_mulhi(c.m_p, wp.y << c.pp);
  }
  return make_longlong2(ur, ui);
}

// Two elements x and x2 per call: the neighbour loads of both are issued in
// the same loop iterations (twice the independent requests per warp).
__device__ __forceinline__ void fx_apply_spin2(const longlong2* q, const longlong2* qm, int x, int x2,
                                               const OpSpinFx& op, const FxConstA& c, const long long* mb,
                                               longlong2& r1, longlong2& r2) {
  const int N = op.N, L = op.lo_bits;
  const long long dz1 = __ldg(op.DZ_lo + (x & ((1 << L) - 1))) + __ldg(op.DZ_hi + (x >> (L - 1)));
  const long long dz2 = __ldg(op.DZ_lo + (x2 & ((1 << L) - 1))) + __ldg(op.DZ_hi + (x2 >> (L - 1)));
  const long long Dp1 = fx_mulhi(c.m_cz, dz1 << 1) << 3;
  const long long Dp2 = fx_mulhi(c.m_cz, dz2 << 1) << 3;
  const longlong2 v1 = q[x], v2 = q[x2];
  long long ur1 = fx_mulhi(Dp1, v1.x << c.pk), ui1 = fx_mulhi(Dp1, v1.y << c.pk);
  long long ur2 = fx_mulhi(Dp2, v2.x << c.pk), ui2 = fx_mulhi(Dp2, v2.y << c.pk);
  long long hr1 = 0, hi1 = 0, hr2 = 0, hi2 = 0;
  const unsigned mask = (1u << (N - 1)) - 1u;
  const unsigned anti1 = ((unsigned)x ^ ((unsigned)x >> 1)) & mask;
  const unsigned anti2 = ((unsigned)x2 ^ ((unsigned)x2 >> 1)) & mask;
#pragma unroll 4
  for (int i = 0; i < N - 1; ++i) {
    if ((anti1 >> i) & 1u) {
      const longlong2 w = q[x ^ (3 << i)];
      hr1 += w.x;
      hi1 += w.y;
    }
    if ((anti2 >> i) & 1u) {
      const longlong2 w = q[x2 ^ (3 << i)];
      hr2 += w.x;
      hi2 += w.y;
    }
  }
  ur1 += fx_mulhi(c.m_hop, hr1 << c.ph);
  ui1 += fx_mulhi(c.m_hop, hi1 << c.ph);
  ur2 += fx_mulhi(c.m_hop, hr2 << c.ph);
  ui2 += fx_mulhi(c.m_hop, hi2 << c.ph);
  if (op.uniform) {
    long long xr1 = 0, xi1 = 0, xr2 = 0, xi2 = 0;
#pragma unroll 4
    for (int i = 0; i < N; ++i) {
      const longlong2 w1 = q[x ^ (1 << i)];
      const longlong2 w2 = q[x2 ^ (1 << i)];
      xr1 += w1.x;
      xi1 += w1.y;
      xr2 += w2.x;
      xi2 += w2.y;
    }
    ur1 += fx_mulhi(c.m_x, xr1 << c.px);
    ui1 += fx_mulhi(c.m_x, xi1 << c.px);
    ur2 += fx_mulhi(c.m_x, xr2 << c.px);
    ui2 += fx_mulhi(c.m_x, xi2 << c.px);
  } else {
#pragma unroll 4
    for (int i = 0; i < N; ++i) {
      const longlong2 w1 = q[x ^ (1 << i)];
      const longlong2 w2 = q[x2 ^ (1 << i)];
      ur1 += fx_mulhi(mb[i], w1.x << c.pk);
      ui1 += fx_mulhi(mb[i], w1.y << c.pk);
      ur2 += fx_mulhi(mb[i], w2.x << c.pk);
      ui2 += fx_mulhi(mb[i], w2.y << c.pk);
    }
  }
  if (c.use_prev) {
    const longlong2 w1 = qm[x], w2 = qm[x2];
    ur1 += fx_mulhi(c.m_p, w1.x << c.pp);
    ui1 += fx_mulhi(c.m_p, w1.y << c.pp);
    ur2 += fx_mulhi(c.m_p, w2.x << c.pp);
    ui2 += fx_mulhi(c.m_p, w2.y << c.pp);
  }
  r1 = make_longlong2(ur1, ui1);
  r2 = make_longlong2(ur2, ui2);
}

__device__ __forceinline__ longlong2 fx_apply_dia(const longlong2* q, const longlong2* qm, int r, int dim,
                                                  const OpDiaFx& op, const FxConstA& c) {
  long long ur = 0, ui = 0;
  for (int o = 0; o < op.nops; ++o) {
    __int128 ar = 0, ai = 0;
    const int d0 = op.dfirst[o], d1 = d0 + op.dcount[o];
    for (int d = d0; d < d1; ++d) {
      const long long cidx = (long long)r + __ldg(op.off + d);
      if (cidx >= 0 && cidx < dim) {
        const long long a = __ldg(op.VAL + (size_t)d * dim + r);
        const longlong2 w = q[cidx];
        ar += (__int128)a * w.x;
        ai += (__int128)a * w.y;
      }
    }
    ur += fx_mulhi(c.m_op[o], fx_shr128(ar, c.sh_pre[o]));
    ui += fx_mulhi(c.m_op[o], fx_shr128(ai, c.sh_pre[o]));
  }
  if (c.use_prev) {
    const longlong2 w = qm[r];
    ur += fx_mulhi(c.m_p, w.x << c.pp);
    ui += fx_mulhi(c.m_p, w.y << c.pp);
  }
  return make_longlong2(ur, ui);
}

// CSR: per operator the exact 128-bit sums of VAL * q over the row's entries
// (complex values: re = sum VR w.x - VI w.y, im = sum VR w.y + VI w.x; the row
// sums of |VR| + |VI| stay below 2^62 and |q| < 2^57, so no sum overflows),
// then one rounded product with the operator's scalar mantissa as for DIA.
// 2^op.lane_bits neighbouring threads (all of them in the call, `on` false past
// the CTA's rows) share the row r: each takes every 2^lane_bits-th entry and the
// exact partial sums are added by shuffles, so the result does not depend on
// the split; the first of them returns it.
// Bound by the gathers: every entry fetches a 32-byte sector of q at random from
// L2 besides its 20 B of matrix data.  60 001 rows of 20 entries (random complex
// H0, banded real V) take 15.5 us per apply on 152 CTAs, 3.9 TB/s of those
// bytes; more loads in flight per thread (unrolled by 4, or batches of 4 and 6
// entries loaded before their use) measured 18-21 us.  One thread per row over
// equal row counts, as before, took 22.5 us in the mean CTA and 48 in the last.
__device__ __forceinline__ void fx_lane_sum128(__int128& a, int lane_bits) {
  for (int b = 0; b < lane_bits; ++b) {
    const unsigned long long lo = __shfl_xor_sync(0xffffffffu, (unsigned long long)a, 1 << b);
    const long long hi = __shfl_xor_sync(0xffffffffu, (long long)(a >> 64), 1 << b);
    a += ((__int128)hi << 64) | lo;
  }
}
__device__ __forceinline__ longlong2 fx_apply_csr(const longlong2* q, const longlong2* qm, int r, bool on, int dim,
                                                  const OpCsrFx& op, const FxConstA& c) {
  const int T = 1 << op.lane_bits, sub = threadIdx.x & (T - 1);
  long long ur = 0, ui = 0;
  for (int o = 0; o < op.nops; ++o) {
    const int* rp = op.rp + (size_t)o * (dim + 1);
    const int e0 = on ? __ldg(rp + r) + sub : 0, e1 = on ? __ldg(rp + r + 1) : 0;
    __int128 ar = 0, ai = 0;
    if ((op.cplx >> o) & 1u) {
#pragma unroll 2
      for (int e = e0; e < e1; e += T) {
        const long long a = __ldg(op.VR + e), b = __ldg(op.VI + e);
        const longlong2 w = q[__ldg(op.col + e)];
        ar += (__int128)a * w.x - (__int128)b * w.y;
        ai += (__int128)a * w.y + (__int128)b * w.x;
      }
    } else {
#pragma unroll 2
      for (int e = e0; e < e1; e += T) {
        const long long a = __ldg(op.VR + e);
        const longlong2 w = q[__ldg(op.col + e)];
        ar += (__int128)a * w.x;
        ai += (__int128)a * w.y;
      }
    }
    fx_lane_sum128(ar, op.lane_bits);
    fx_lane_sum128(ai, op.lane_bits);
    ur += fx_mulhi(c.m_op[o], fx_shr128(ar, c.sh_pre[o]));
    ui += fx_mulhi(c.m_op[o], fx_shr128(ai, c.sh_pre[o]));
  }
  if (c.use_prev && on && sub == 0) {
    const longlong2 w = qm[r];
    ur += fx_mulhi(c.m_p, w.x << c.pp);
    ui += fx_mulhi(c.m_p, w.y << c.pp);
  }
  return make_longlong2(ur, ui);
}

}  // namespace cfet
