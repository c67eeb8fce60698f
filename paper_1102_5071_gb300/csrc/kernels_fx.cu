// Fixed-point persistent Lanczos kernel (sm_103a).
//
// Same method and decisions as k_propagate (kernels.cu): the stage
// exponential exp(-i tau H_j) psi of a CFET step (Alvermann & Fehske,
// arXiv:1102.5071, Sec. 4 Eq. (Ucf), Sec. 7 Eq. (OmGLeg)) by the Lanczos /
// Krylov method of Sec. 8.1 with the a-posteriori estimate, adaptive Krylov
// dimension and substepping.  Two things differ.
//
// Number format.  On GB300 FP64 runs at 1/64 of the FP32 rate while 32-bit
// integer add/logic/multiply-add run at full or half rate, so every Krylov
// vector q_i is stored as int64 (re, im) mantissas with one exponent per
// vector (value = M * 2^E_i, |M| < 2^57):
//   * neighbour sums of the apply are exact integer additions (up to 32
//     terms stay below 2^62);
//   * a product of a real scalar (or a per-element table value) with a stored
//     value or sum takes the high 64 bits of a 64x64 product of operands
//     normalised to 62 bits, shifted (rounding) once to the result exponent;
//   * the result exponent of each new vector comes from a rigorous bound
//     built from the scalars and the measured maxima of the inputs, so no
//     value overflows; the resolution is 2^-57 of that bound;
//   * alpha, ||w||^2 and ||psi||^2 are exact 128-bit sums, reduced exactly
//     over the CTA and the grid (order-independent, deterministic) and
//     rounded to FP64 once.
//
// Work split.  Each CTA has NW worker warps doing only integer element work
// and one control warp doing all scalar work: the global reductions, the grid
// barrier, the per-pass constants, and the small tridiagonal exponential of
// the error estimate (FP64 where the result must be exact; bounds and certain
// decisions in integer and FP32 arithmetic, scalar_bounds.cuh, because one
// FP64 warp instruction costs 64 cycles here).  The error estimate of iteration k runs
// on the control warp while the workers already compute the apply of
// iteration k+1; if it accepts k, that apply is discarded.  The accepted
// estimate's y = exp(-i tau T_k) e_1 is reused for the reconstruction.
//
// Long chains.  The kFxTiled instantiation replaces the element-wise spin apply
// by window passes over shared-memory tiles moved by TMA (tiled_common.cuh)
// separated by grid exchanges, for chains whose vectors leave L2.  Small
// problems.  kFxSmall runs one CTA with the whole Krylov basis in shared memory,
// kFxCluster one thread-block cluster with the applied vector staged in it.
#include <cuda_runtime.h>

#include <cmath>
#include <cstdint>

#include "cfet_internal.h"
#include "device_common.cuh"
#include "fx_common.cuh"
#include "tiled_common.cuh"

namespace cfet {

// Forms of the kernel (separate instantiations, so that none carries the code of
// the others and the vectors keep their address space).
enum FxMode {
  kFxGrid = 0,     // element-wise, vectors in global memory, exchange through L2
  kFxTiled = 1,    // long spin chains: window-tiled apply
  kFxSmall = 2,    // one CTA with the Krylov basis in shared memory
  kFxCluster = 3,  // spin chains on one thread-block cluster, applied vector in its shared memory
};

// ------------------------------------------------------------------ shared state
struct SmemFx {
  // per-warp partials of the workers
  unsigned long long wlo[32];
  long long whi[32];
  long long wmx[32];
  // Lanczos scalars (FP64) and vector metadata
  double alpha[kMaxKrylov + 2];
  double beta[kMaxKrylov + 2];
  double nq[kMaxKrylov + 3];     // ||q_i||^2, in [1, 4) (or 0)
  double scale[kMaxKrylov + 3];  // 1 / ||q_i||
  double rn[kMaxKrylov + 3];     // 1 / ||q_i||^2
  double cprev[kMaxKrylov + 3];  // coefficient of q_{i-1} in the recurrence of q_{i+1}
  long long A[kMaxKrylov + 3];   // max stored |M| of q_i
  int E[kMaxKrylov + 3];         // exponent of q_i
  int pw[kMaxKrylov + 3];        // q_{i+1} = w_i 2^-pw[i]
  double yr[kMaxKrylov], yi[kMaxKrylov];
  double tr[kMaxKrylov], ti[kMaxKrylov];
  // reconstruction constants
  long long crm[kMaxKrylov], cim[kMaxKrylov];
  int cp[kMaxKrylov];
  // stage data: the scalars' mantissas, fixed for the exponential
  double scal[1 + kMaxDrives];
  Mant mcz, mh, mx;           // c_0, 2 J c_0, the uniform field
  Mant mop[1 + kMaxDrives];   // DIA, CSR: operator scalars
  UpB hbound;                 // bound of |H q| / max|q|
  UpB rowb[1 + kMaxDrives];   // DIA, CSR: maxrow of each operator
  int eb;                     // exponent of the per-site table mbraw
  long long mbraw[kMaxSites]; // per-site fields, fixed for the exponential
  long long mb[kMaxSites];    // the same with the iteration's product shift
  FxConstA ca;
  // phase B constants
  long long m_a;
  int sh_u, pk_b;
  int Eu, Ew, Epsi;
  // commands to the workers
  int cmd, it;                // FxCmd; the iteration, or the number of basis vectors (kFxRec)
  int final_rec;
  // control flow
  long long e, fpos;  // stage exponential of the launch; next forced decision
  double remaining;   // of the stage exponential
  double acc_err;     // estimate of the accepted substep
  int nsub_e;         // substeps of the stage exponential
  int y_ready;        // yr/yi hold exp(-i ts T_k) e_1 for the accepted (k, ts)
  int acc_h;
  double beta0;
  double rsum;  // fx_ctl_reduce_cold
  long long rmx;
  double nsum;  // ||q_1||^2 in units of 2^(2 E[1])
  // running FP32 bounds of the current T_k for the estimate's screens
  LeadAcc lead;
  GershAcc gfull;  // rows whose couplings are all known
  int gate_it;     // FP32 gate of the current iteration (1, 0, -1: FP64 needed)
  int tma_fail;    // tiled apply: a tile wait gave up
  // kept here, not in registers (the element loops need those): the trace
  // (cfet_stats.phase_ns; slots 0, 2, 4, 7 by thread 0, the others by the
  // control lane 0) and, by the control lane 0, the run's counters
  long long tacc[8];
  long long twe;      // thread 0: end of its last element loop
  long long n_app, n_sub, rpos;
  int max_k;
  double max_err;
};

// ------------------------------------------------------------------ control-warp helpers
// Exact accumulation of exchanged CTA records: 128-bit sum (words 0-3) and
// int64 max (words 4-5).
struct FxAcc {
  unsigned long long lo;
  long long hi, m;
  __device__ void reset() { lo = 0; hi = 0; m = 0; }
  __device__ void add(const unsigned (&v)[6]) {
    const unsigned long long l2 = ((unsigned long long)v[1] << 32) | v[0];
    const long long h2 = (long long)(((unsigned long long)v[3] << 32) | v[2]);
    const long long m2 = (long long)(((unsigned long long)v[5] << 32) | v[4]);
    const unsigned long long t = lo + l2;
    hi = hi + h2 + (t < lo ? 1 : 0);
    lo = t;
    m = m > m2 ? m : m2;
  }
};

// Control warp: combine the workers' per-warp partials into this CTA's record,
// exchange records with every CTA (the grid barrier), and return the exact
// global sum (as FP64) and the global max to all lanes (FxMode; kFxCluster: part
// is the cluster's exchange slots in shared memory).
template <int MODE>
__device__ __forceinline__ bool fx_ctl_reduce(SmemFx& S, int NW, unsigned long long* part, unsigned tag, bool fence, int* status,
                              long long timeout_ns, double& sum, long long& mxi, long long& spin) {
  const int lane = threadIdx.x & 31;
  unsigned long long lo = 0;
  long long hi = 0, m = 0;
  if (lane < NW) { lo = S.wlo[lane]; hi = S.whi[lane]; m = S.wmx[lane]; }
  fx_warp_reduce(lo, hi, m);
  if constexpr (MODE == kFxSmall) {
    sum = fx_i128_to_double(lo, hi);
    mxi = m;
    return true;
  }
  const unsigned mine[6] = {(unsigned)lo, (unsigned)(lo >> 32), (unsigned)hi,
                            (unsigned)((unsigned long long)hi >> 32), (unsigned)m,
                            (unsigned)((unsigned long long)m >> 32)};
  FxAcc acc;
  if constexpr (MODE == kFxCluster) {
    if (!cluster_exchange<6>(part, mine, tag, status, timeout_ns, spin, acc)) return false;
  } else {
    if (!ctl_exchange<6>(part, mine, tag, fence, status, timeout_ns, spin, acc)) return false;
  }
  lo = acc.lo;
  hi = acc.hi;
  m = acc.m;
  fx_warp_reduce(lo, hi, m);
  sum = fx_i128_to_double(lo, hi);
  mxi = m;
  return true;
}

// The same out of line, for the passes that run once per launch or substep:
// results in S.rsum and S.rmx.
template <int MODE>
__device__ __noinline__ bool fx_ctl_reduce_cold(SmemFx& S, int NW, unsigned long long* part, unsigned tag, int* status,
                                                long long timeout_ns) {
  double sum;
  long long mxi;
  const bool ok = fx_ctl_reduce<MODE>(S, NW, part, tag, true, status, timeout_ns, sum, mxi, S.tacc[5]);
  if (ok && (threadIdx.x & 31) == 0) {
    S.rsum = sum;
    S.rmx = mxi;
  }
  __syncwarp();
  return ok;
}

// Worker warps: per-warp reduction of (int128 sum, int64 max) into shared memory.
__device__ __forceinline__ void fx_worker_partial(SmemFx& S, __int128 acc, long long mx) {
  acc >>= kRedShift;
  unsigned long long lo = (unsigned long long)acc;
  long long hi = (long long)(acc >> 64);
  fx_warp_reduce(lo, hi, mx);
  if ((threadIdx.x & 31) == 0) {
    const int w = threadIdx.x >> 5;
    S.wlo[w] = lo;
    S.whi[w] = hi;
    S.wmx[w] = mx;
  }
}

// Control warp: a grid-wide exchange of one tagged word per CTA (a barrier),
// with the fences that make the vectors written before it visible after it.
__device__ bool fx_ctl_barrier(unsigned long long* part, unsigned tag, int* status, long long timeout_ns,
                               long long& spin) {
  struct NoAcc {
    __device__ void reset() {}
    __device__ void add(const unsigned (&)[1]) {}
  } acc;
  const unsigned mine[1] = {0u};
  return ctl_exchange<1>(part, mine, tag, true, status, timeout_ns, spin, acc);
}

// ------------------------------------------------------------------ tiled apply (long chains)
// Window tiling of tiled_common.cuh with tiles of 2^11 elements (32 KB of
// int64 pairs), moved by TMA: one tensor map per window over the whole Krylov
// basis (two 8-byte words per element), three pipeline stages of a q tile and
// a tile of the vector each element reads for itself (q_{k-1} in window 0, the
// partial u after it), 192 KB, one mbarrier per stage.  Worker thread 0 issues
// the loads two tiles ahead; once the workers have written a tile's results
// (in place over its own-element tile) it stores that tile with a bulk tensor
// store.  Every window adds its terms in the format of the apply above (exact
// integer neighbour sums, one rounded product per sum and window), so the
// result differs from the element-wise apply by the rounding of the extra
// products (units of the last place of u).  The last window takes <q, u>
// exactly and max |u|.
constexpr int kFxTileElems = 1 << kFxTileBits;
constexpr unsigned kFxTileBytes = kFxTileElems * sizeof(longlong2);

size_t fx_tiled_smem_bytes();

struct FxTma {
  const unsigned char* maps;  // kTmaMapBytes per window
  unsigned long long* bar;    // [kTmaStages] in shared memory
  longlong2* stage;           // [kTmaStages][2][kFxTileElems] in shared memory
  int* fail;                  // shared flag: a wait gave up
  unsigned* phase;            // parity bits of the stages (per thread, identical in all workers)
  int* status;
  long long timeout_ns;
};

// Bounded wait for a stage's tile; false (status CFET_ETIMEOUT) when it gave up.
__device__ bool fx_tile_wait(unsigned long long* bar, unsigned parity, int* status, long long timeout_ns) {
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

// One window pass of this CTA's worker threads over its tiles (basis indices:
// iq the applied q, ia the own-element input, iu the output).
template <bool FIRST, bool LAST>
__device__ void fx_tiled_pass(const FxTma& T, const OpSpinFx& op, const FxConstA& c, const long long* mb, int iq,
                              int ia, int iu, const TileWin& W, int w, int nworkers, __int128& a2, long long& mx) {
  const int tid = threadIdx.x;
  const int G = gridDim.x;
  const int ntiles = 1 << (op.N - kFxTileBits);
  const bool aux = !FIRST || c.use_prev;
  const unsigned bytes = aux ? 2 * kFxTileBytes : kFxTileBytes;
  const void* map = T.maps + (size_t)w * kTmaMapBytes;
  const bool prod = tid == 0;
  auto issue = [&](int k, int t) {  // producer: tile t into stage k % kTmaStages
    const int st = k % kTmaStages;
    longlong2* qb = T.stage + (size_t)st * 2 * kFxTileElems;
    mbar_arrive_expect_tx(T.bar + st, bytes);
    tile_load_t<kFxTileBits, 2>(qb, map, FIRST, W, op.N, t, iq, T.bar + st);
    if (aux) tile_load_t<kFxTileBits, 2>(qb + kFxTileElems, map, FIRST, W, op.N, t, ia, T.bar + st);
  };
  if (prod) {
    fence_proxy_async_all();  // vectors written by generic stores before the exchange, read by TMA now
    for (int k = 0; k < kTmaStages - 1; ++k)
      if (blockIdx.x + k * G < ntiles) issue(k, blockIdx.x + k * G);
  }
  int k = 0;
  for (int t = blockIdx.x; t < ntiles; ++k, t += G) {
    const int st = k % kTmaStages;
    const longlong2* cur = T.stage + (size_t)st * 2 * kFxTileElems;
    longlong2* acur = T.stage + (size_t)st * 2 * kFxTileElems + kFxTileElems;
    const unsigned par = (*T.phase >> st) & 1u;
    *T.phase ^= 1u << st;
    if (!fx_tile_wait(T.bar + st, par, T.status, T.timeout_ns)) *T.fail = 1;
    if (!*T.fail) {
      for (int j = tid; j < kFxTileElems; j += nworkers) {
        long long ur, ui, hr = 0, hi = 0;
        const longlong2 v = cur[j];
        if (FIRST) {
          const int x = (t << kFxTileBits) | j;
          const int L = op.lo_bits;
          const long long dz = __ldg(op.DZ_lo + (x & ((1 << L) - 1))) + __ldg(op.DZ_hi + (x >> (L - 1)));
          const long long Dp = fx_mulhi(c.m_cz, dz << 1) << 3;
          ur = fx_mulhi(Dp, v.x << c.pk);
          ui = fx_mulhi(Dp, v.y << c.pk);
          const unsigned anti = ((unsigned)j ^ ((unsigned)j >> 1)) & ((1u << (kFxTileBits - 1)) - 1u);
#pragma unroll
          for (int i = 0; i < kFxTileBits - 1; ++i)
            if ((anti >> i) & 1u) {
              const longlong2 wv = cur[j ^ (3 << i)];
              hr += wv.x;
              hi += wv.y;
            }
          if (op.uniform) {
            long long xr = 0, xi = 0;
#pragma unroll
            for (int i = 0; i < kFxTileBits; ++i) {
              const longlong2 wv = cur[j ^ (1 << i)];
              xr += wv.x;
              xi += wv.y;
            }
            ur += fx_mulhi(c.m_x, xr << c.px);
            ui += fx_mulhi(c.m_x, xi << c.px);
          } else {
#pragma unroll
            for (int i = 0; i < kFxTileBits; ++i) {
              const longlong2 wv = cur[j ^ (1 << i)];
              ur += fx_mulhi(mb[i], wv.x << c.pk);
              ui += fx_mulhi(mb[i], wv.y << c.pk);
            }
          }
          if (c.use_prev) {
            const longlong2 wv = acur[j];
            ur += fx_mulhi(c.m_p, wv.x << c.pp);
            ui += fx_mulhi(c.m_p, wv.y << c.pp);
          }
        } else {
          const longlong2 a = acur[j];
          ur = a.x;
          ui = a.y;
          const unsigned jh = (unsigned)j >> W.c;  // bits b0 .. b0+width-1 of x
          const unsigned anti = (jh ^ (jh >> 1)) & ((1u << (W.width - 1)) - 1u);
          for (int i = 0; i < W.width - 1; ++i)
            if ((anti >> i) & 1u) {
              const longlong2 wv = cur[j ^ (3 << (W.c + i))];
              hr += wv.x;
              hi += wv.y;
            }
          if (op.uniform) {
            long long xr = 0, xi = 0;
            for (int i = 1; i < W.width; ++i) {
              const longlong2 wv = cur[j ^ (1 << (W.c + i))];
              xr += wv.x;
              xi += wv.y;
            }
            ur += fx_mulhi(c.m_x, xr << c.px);
            ui += fx_mulhi(c.m_x, xi << c.px);
          } else {
            for (int i = 1; i < W.width; ++i) {
              const longlong2 wv = cur[j ^ (1 << (W.c + i))];
              ur += fx_mulhi(mb[W.b0 + i], wv.x << c.pk);
              ui += fx_mulhi(mb[W.b0 + i], wv.y << c.pk);
            }
          }
        }
        ur += fx_mulhi(c.m_hop, hr << c.ph);
        ui += fx_mulhi(c.m_hop, hi << c.ph);
        acur[j] = make_longlong2(ur, ui);  // the own element only: read above by this thread
        if (LAST) {
          a2 += (__int128)v.x * ur + (__int128)v.y * ui;
          mx = max(mx, fx_absmax(ur, ui));
        }
      }
    }
    fence_proxy_async_smem();  // the results, written by generic stores, are read by the TMA store
    workers_sync(nworkers);
    if (*T.fail) break;
    if (prod) {
      tile_store_t<kFxTileBits, 2>(map, FIRST, W, op.N, t, iu, acur);
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
        fx_tile_wait(T.bar + s2, par, T.status, T.timeout_ns);
      }
    }
  }
  workers_sync(nworkers);
}

// The Krylov basis is built by the unnormalised three-term recurrence
//   u_k = H q_k - c_k q_{k-1},  w_k = u_k - alpha_k q_k,  q_{k+1} = w_k 2^-p_k,
//   alpha_k = <q_k, u_k> / ||q_k||^2,  c_k = beta_{k-1}^2 2^-p_{k-1}
//           = 2^p_{k-1} ||q_k||^2 / ||q_{k-1}||^2,
// v_k = q_k / ||q_k|| being the Lanczos vectors of Sec. 8.1 and p_k the power
// of two that brings ||q_{k+1}||^2 into [1, 4) (only the exponent of the stored
// vector changes).  The stage scalars then enter every apply with the same
// mantissas and only shifts depend on the iteration, and between the reduction
// of ||w_k||^2 and the next apply stands one FP64 product: on this GPU a
// dependent FP64 instruction of the control warp costs 64 cycles, a reciprocal
// square root 370.  beta_k, 1 / ||q_{k+1}|| and the tests that need them are
// taken while the workers already apply H (fx_close_iteration and the deferred
// estimate).  With the normalised recurrence (scalars times 1 / beta in every
// iteration) the control warp held the workers 2.5 us after every phase B and
// 1.05 us after every phase A.

// Per-exponential constants (whole control warp; S.scal is set).
template <int FAMILY, class Op>
__device__ __noinline__ void fx_stage_consts(SmemFx& S, const Op& op, int nV) {
  const int lane = threadIdx.x & 31;
  if constexpr (FAMILY == kFamilySpin) {
    double bi = 0.0;  // per-site transverse fields of this stage (N <= 30 lanes)
    if (lane < op.N)
      for (int k = 0; k < nV; ++k) bi = fma(S.scal[1 + k], __ldg(op.xf + k * op.N + lane), bi);
    double bs = fabs(bi), bm = fabs(bi);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      bs += __shfl_xor_sync(0xffffffffu, bs, o);
      bm = fmax(bm, __shfl_xor_sync(0xffffffffu, bm, o));
    }
    if (!op.uniform) {
      const int eb = fx_exp_for(bm, 62);
      if (lane < op.N) S.mbraw[lane] = __double2ll_rn(fx_scale2(bi, -eb));
      if (lane == 0) S.eb = eb;
    }
    if (lane == 0) {
      const double cz = S.scal[0], ch = cz * op.J2, db = fabs(cz) * op.maxdz;
      S.mcz = fx_mant(cz);
      S.mh = fx_mant(ch);
      S.mx = fx_mant(bi);
      S.hbound = sb_upb(db + fabs(ch) * op.nbond + bs);
    }
  } else {
    if (lane == 0) {
      double hb = 0.0;
      for (int o = 0; o < op.nops; ++o) {
        S.mop[o] = fx_mant(S.scal[o]);
        S.rowb[o] = sb_upb(op.maxrow[o]);
        hb += fabs(S.scal[o]) * op.maxrow[o];
      }
      S.hbound = sb_upb(hb);
    }
  }
  if (lane == 0) S.hbound = sb_upb_mul(S.hbound, UpB{1.0f + 0x1p-20f, 0});  // FP64 rounding of the sums above
  __syncwarp();
}

// Phase-A constants of iteration it (called by the whole control warp): result
// exponent of u = H q_it - c q_{it-1} from the bound of every term (in every
// lane), then one lane per term: value m 2^e times a sum of cnt entries of a
// vector with maximum A at exponent E takes the normalising shift p and the
// product shift Eu - e - (E - p) - 64.
template <int FAMILY, class Op>
__device__ __forceinline__ void fx_const_a(SmemFx& S, const Op& op, int it) {
  const int lane = threadIdx.x & 31;
  FxConstA& c = S.ca;
  const long long Ak = S.A[it], Ap = it > 1 ? S.A[it - 1] : 0;
  const int Ek = S.E[it], Ep = it > 1 ? S.E[it - 1] : 0;
  const double cp = it > 1 ? S.cprev[it] : 0.0;
  const UpB Akr = sb_upb_scale2(sb_upb_ll(Ak), Ek);
  const UpB B = sb_upb_add(sb_upb_mul(S.hbound, Akr), sb_upb_mul(sb_upb(cp), sb_upb_scale2(sb_upb_ll(Ap), Ep)));
  const int Eu = sb_upb_exp_for(B, kFxBits);
  if (lane == 0) {
    c.use_prev = it > 1;
    c.Eu = Eu;
    S.Eu = Eu;
  }
  if constexpr (FAMILY == kFamilySpin) {
    // terms: diagonal (c_0 times the table at 2^E_dz), hops, uniform field, q_{it-1}
    if (lane < 4) {
      const Mant m = lane == 0 ? S.mcz : (lane == 1 ? S.mh : (lane == 2 ? S.mx : fx_mant(-cp)));
      const int e = lane == 0 ? m.e + op.E_dz + 60 : m.e;
      const int cnt = lane == 1 ? (op.N > 1 ? op.N - 1 : 1) : (lane == 2 ? op.N : 1);
      const int ps = sb_norm_shift_ll(cnt * (lane == 3 ? Ap : Ak));
      c.p4[lane] = ps;
      c.m4[lane] = fx_fold(m.m, Eu - e - ((lane == 3 ? Ep : Ek) - ps) - 64);
    }
    if (!op.uniform) {
      const int s_nu = Eu - S.eb - (Ek - sb_norm_shift_ll(Ak)) - 64;
      for (int i = lane; i < op.N; i += 32) S.mb[i] = fx_fold(S.mbraw[i], s_nu);
    }
  } else {
    if (lane < op.nops) {
      const int Epre = sb_upb_exp_for(sb_upb_mul(S.rowb[lane], Akr), 62);  // |P_o| < 2^62
      const Mant m = S.mop[lane];
      c.sh_pre[lane] = Epre - op.E_op[lane] - Ek;
      c.m_op[lane] = fx_fold(m.m, Eu - m.e - Epre - 64);
    } else if (lane == op.nops) {
      const Mant m = fx_mant(-cp);
      c.pp = sb_norm_shift_ll(Ap);
      c.m_p = fx_fold(m.m, Eu - m.e - (Ep - c.pp) - 64);
    }
  }
}

template <int FAMILY, class Op>
__device__ __noinline__ void fx_const_a_cold(SmemFx& S, const Op& op, int it) {  // once per substep
  fx_const_a<FAMILY>(S, op, it);
}

// Squared norm `sum` 2^(2E) of a vector stored at exponent E: the power of two
// p that brings it into [1, 4), and the scaled value (0 and 0 for sum = 0).
__device__ __forceinline__ double fx_norm_pow(double sum, int E, int& p) {
  if (!(__double_as_longlong(sum) > 0)) {
    p = 0;
    return 0.0;
  }
  p = (fx_ilog2(sum) + 2 * E) >> 1;
  return fx_scale2(sum, 2 * (E - p));
}

// What iteration it leaves for later (one lane): 1 / ||q_{it+1}||, its square
// and beta_it = ||q_{it+1}|| 2^p / ||q_it||.
__device__ void fx_close_iteration(SmemFx& S, int it) {
  const double n = S.nq[it + 1];
  const double rs = __double_as_longlong(n) > 0 ? rsqrt(n) : 0.0;
  S.scale[it + 1] = rs;
  S.rn[it + 1] = rs * rs;
  S.beta[it] = fx_scale2(n * rs * S.scale[it], S.pw[it]);
}
// Lanczos breakdown at iteration it (closed).
__device__ __forceinline__ bool fx_breakdown(const SmemFx& S, int it) {
  const double b = S.beta[it], prev_b = it > 1 ? S.beta[it - 1] : 0.0;
  return sb_no_breakdown(b, S.alpha[it], prev_b) != 1 && b <= 1e-13 * (fabs(S.alpha[it]) + prev_b + 1.0);
}

// Error estimate of iteration k (control warp): err = beta0 beta_k |y_k| with
// y = exp(-i ts T_k) e_1 left in S.yr/S.yi.  When the FP32 screen shows that
// err exceeds the threshold thr, the FP64 evaluation is skipped and a value
// above thr is returned (S.yr/S.yi then stay untouched).
__device__ __noinline__ double fx_estimate(SmemFx& S, int k, double ts, double thr) {
  const int dec = krylov_lead_decide(S.lead, k, ts, S.beta0, S.beta[k], thr);
  if (dec == 0) return 2.0 * thr + 1e-300;
  const double scale = S.beta0 * S.beta[k];
  if (dec < 0 && small_expm_rejects32(k, S.alpha + 1, S.beta + 1, ts, scale, thr)) return 2.0 * thr + 1e-300;
  small_expm_e1(k, S.alpha + 1, S.beta + 1, ts, S.yr, S.yi, S.tr, S.ti);
  const double yr = S.yr[k - 1], yi = S.yi[k - 1];
  return scale * sqrt(fma(yr, yr, yi * yi));
}

// Halves the step on the basis of iteration it until the estimate meets the
// proportional tolerance (control warp): S.acc_h, 0 when no step does.
__device__ __noinline__ void fx_halve(SmemFx& S, int it, double tol, double tau) {
  const double remaining = S.remaining;
  int hh = 0;
  double err = 0.0;
  const double width = gersh_width(it, S.alpha + 1, S.beta + 1);
#pragma unroll 1
  for (int h = 1; h <= 40; ++h) {
    const double ts = fx_scale2(remaining, -h);
    if (!(fabs(ts) * width <= 2.0 * it)) continue;
    err = fx_estimate(S, it, ts, tol * ts / tau);
    if (err <= tol * ts / tau) { hh = h; break; }
  }
  if ((threadIdx.x & 31) == 0) { S.acc_h = hh; S.acc_err = err; S.y_ready = hh > 0; }
}

// ------------------------------------------------------------------ the kernel
// Worker and control warps run separate loops: the control warp publishes one
// command (an element pass) at a time with its constants in shared memory, a CTA
// barrier starts the pass, a second one ends it.  Both have the 72 registers of an
// 800-thread CTA; the control flow, the counters and the trace are kept in shared
// memory instead.  What the separate loops give by themselves was not measured: they
// came with the unnormalised recurrence, the warp reductions, the packed records and
// the functions out of line, 8 sites 6.1 us per iteration together (7.6 before).
enum FxCmd { kFxExit = 0, kFxMax, kFxConvert, kFxApply, kFxOrth, kFxRec };

__device__ __forceinline__ void fx_cta_sync() { __syncthreads(); }  // by workers and control warp, each from its loop

template <int FAMILY, class Op, int MODE>
__device__ __forceinline__ void fx_worker(const PropParams& p, const Op& op, SmemFx& S, unsigned char* tiles_base,
                                          int wstep) {
  constexpr bool TILED = MODE == kFxTiled, SMALL = MODE == kFxSmall, CLUSTER = MODE == kFxCluster;
  const int tid = threadIdx.x;
  const int dim = p.dim;
  // each CTA walks one contiguous chunk of the vectors, so that the
  // neighbours of low-bit flips (and short band offsets) are found in L1
  int wx0, wxe;
  if constexpr (FAMILY == kFamilyCsr) {  // rows split by their work, not their number (csr_row_split)
    wx0 = __ldg(op.rb + blockIdx.x) + tid;
    wxe = __ldg(op.rb + blockIdx.x + 1);
  } else {
    const int chunk = (dim + gridDim.x - 1) / gridDim.x;
    wx0 = blockIdx.x * chunk + tid;
    wxe = min(dim, ((int)blockIdx.x + 1) * chunk);
  }
  // one-CTA launches of small problems keep the basis in shared memory
  longlong2* const qb = SMALL ? reinterpret_cast<longlong2*>(tiles_base) : p.qbasis;
  auto Q = [&](int i) -> longlong2* { return qb + (size_t)(i - 1) * dim; };
  // kFxCluster: this CTA's part of the applied vector, behind the exchange slots
  longlong2* const sq = reinterpret_cast<longlong2*>(tiles_base + kClusterSlotWords * 8);
  const int xb = wx0 - tid;
  TileWin win[kTiledMaxWindows] = {};
  int nwin = 1;
  if constexpr (TILED) nwin = tiled_windows<kFxTileBits>(op.N, win);
  unsigned tph = 0;  // parities of the stages' mbarriers (the same in every worker)
  if (tid == 0) S.twe = 0;
  while (true) {
    fx_cta_sync();  // the command and its constants are set
    const int cmd = S.cmd;
    if (tid == 0 && S.twe) S.tacc[7] += sm_clock() - S.twe;
    if (cmd == kFxExit) break;
    const long long tw0 = sm_clock();
    if (cmd == kFxApply) {
      // -------- phase A: u = H q_it - c q_{it-1}, <q, u>
      const int it = S.it;
      const FxConstA& c = S.ca;
      const longlong2* q = Q(it);
      const longlong2* qm = it > 1 ? Q(it - 1) : q;
      longlong2* u = Q(it + 1);
      __int128 a2 = 0;
      long long mx = 0;
      int x = wx0;
      if constexpr (TILED) {  // window passes, grid exchanges between them (control warp)
        const FxTma TP{p.tmaps, reinterpret_cast<unsigned long long*>(tiles_base),
                       reinterpret_cast<longlong2*>(tiles_base + 128), &S.tma_fail, &tph, &p.st->status,
                       p.timeout_ns};
        for (int w = 0; w < nwin; ++w) {
          // basis indices: q_it is vector it - 1, q_{it-1} vector it - 2, u vector it
          const int iq = it - 1, ia = w == 0 ? (it > 1 ? it - 2 : 0) : it, iu = it;
          if (w == 0) {
            if (nwin == 1)
              fx_tiled_pass<true, true>(TP, op, c, S.mb, iq, ia, iu, win[0], 0, wstep, a2, mx);
            else
              fx_tiled_pass<true, false>(TP, op, c, S.mb, iq, ia, iu, win[0], 0, wstep, a2, mx);
          } else if (w == nwin - 1) {
            fx_tiled_pass<false, true>(TP, op, c, S.mb, iq, ia, iu, win[w], w, wstep, a2, mx);
          } else {
            fx_tiled_pass<false, false>(TP, op, c, S.mb, iq, ia, iu, win[w], w, wstep, a2, mx);
          }
          if (w + 1 < nwin) {
            window_written_sync();    // all threads: window w written
            window_exchanged_sync();  // all threads: the grid exchange passed
          }
        }
      } else if constexpr (CLUSTER) {
        const int lc = 31 - __clz(wxe - xb), rank = blockIdx.x;
        for (; x < wxe; x += wstep) {
          longlong2 v;
          const longlong2 hv = fx_apply_spin_cluster(sq, qm, x - xb, rank, lc, op, c, S.mb, v);
          u[x] = hv;
          a2 += (__int128)v.x * hv.x + (__int128)v.y * hv.y;
          mx = max(mx, fx_absmax(hv.x, hv.y));
        }
      } else {
        if constexpr (FAMILY == kFamilySpin) {
          for (; x + wstep < wxe; x += 2 * wstep) {
            longlong2 h1, h2;
            fx_apply_spin2(q, qm, x, x + wstep, op, c, S.mb, h1, h2);
            u[x] = h1;
            u[x + wstep] = h2;
            const longlong2 v1 = q[x], v2 = q[x + wstep];
            a2 += (__int128)v1.x * h1.x + (__int128)v1.y * h1.y;
            a2 += (__int128)v2.x * h2.x + (__int128)v2.y * h2.y;
            mx = max(mx, max(fx_absmax(h1.x, h1.y), fx_absmax(h2.x, h2.y)));
          }
        }
        if constexpr (FAMILY == kFamilyCsr) {
          const int lb = op.lane_bits;
          for (int r0 = wx0 - tid; r0 < wxe; r0 += wstep >> lb) {
            const int r = r0 + (tid >> lb);
            const bool on = r < wxe;
            const longlong2 hv = fx_apply_csr(q, qm, r, on, dim, op, c);
            if (on && (tid & ((1 << lb) - 1)) == 0) {
              u[r] = hv;
              const longlong2 v = q[r];
              a2 += (__int128)v.x * hv.x + (__int128)v.y * hv.y;
              mx = max(mx, fx_absmax(hv.x, hv.y));
            }
          }
        } else {
          for (; x < wxe; x += wstep) {
            longlong2 hv;
            if constexpr (FAMILY == kFamilySpin)
              hv = SMALL && op.N <= kWideSites ? fx_apply_spin<true>(q, qm, x, op, c, S.mb)
                                               : fx_apply_spin<false>(q, qm, x, op, c, S.mb);
            else
              hv = fx_apply_dia(q, qm, x, dim, op, c);
            u[x] = hv;
            const longlong2 v = q[x];
            a2 += (__int128)v.x * hv.x + (__int128)v.y * hv.y;
            mx = max(mx, fx_absmax(hv.x, hv.y));
          }
        }
      }
      fx_worker_partial(S, a2, mx);
      if (tid == 0) S.tacc[0] += (S.twe = sm_clock()) - tw0;
    } else if (cmd == kFxOrth) {
      // -------- phase B: w = u - alpha q_it, ||w||^2
      const int sh_u = S.sh_u, pk = S.pk_b, it = S.it;
      const long long m_a = S.m_a;
      const longlong2* q = Q(it);
      longlong2* u = Q(it + 1);
      __int128 b2 = 0;
      long long mx = 0;
      int x = wx0;
      // two elements per step with every load issued first (exact sums:
      // the order does not matter)
      for (; x + wstep < wxe; x += 2 * wstep) {
        const longlong2 v0 = q[x], v1 = q[x + wstep];
        const longlong2 u0 = u[x], u1 = u[x + wstep];
        const long long wr0 = fx_rshr(u0.x, sh_u) + fx_mulhi(m_a, v0.x << pk);
        const long long wi0 = fx_rshr(u0.y, sh_u) + fx_mulhi(m_a, v0.y << pk);
        const long long wr1 = fx_rshr(u1.x, sh_u) + fx_mulhi(m_a, v1.x << pk);
        const long long wi1 = fx_rshr(u1.y, sh_u) + fx_mulhi(m_a, v1.y << pk);
        u[x] = make_longlong2(wr0, wi0);
        u[x + wstep] = make_longlong2(wr1, wi1);
        if constexpr (CLUSTER) {
          sq[x - xb] = make_longlong2(wr0, wi0);
          sq[x + wstep - xb] = make_longlong2(wr1, wi1);
        }
        b2 += (__int128)wr0 * wr0 + (__int128)wi0 * wi0;
        b2 += (__int128)wr1 * wr1 + (__int128)wi1 * wi1;
        mx = max(mx, max(fx_absmax(wr0, wi0), fx_absmax(wr1, wi1)));
      }
      for (; x < wxe; x += wstep) {
        const longlong2 v = q[x];
        const longlong2 uu = u[x];
        const long long wr = fx_rshr(uu.x, sh_u) + fx_mulhi(m_a, v.x << pk);
        const long long wi = fx_rshr(uu.y, sh_u) + fx_mulhi(m_a, v.y << pk);
        u[x] = make_longlong2(wr, wi);
        if constexpr (CLUSTER) sq[x - xb] = make_longlong2(wr, wi);
        b2 += (__int128)wr * wr + (__int128)wi * wi;
        mx = max(mx, fx_absmax(wr, wi));
      }
      fx_worker_partial(S, b2, mx);
      if (tid == 0) S.tacc[2] += (S.twe = sm_clock()) - tw0;
    } else if (cmd == kFxRec) {
      // -------- reconstruct q_1 <- beta0 sum_i y_i s_i q_i
      const int acc_k = S.it;
      const bool final_rec = S.final_rec;
      const double outscale = fx_scale2(1.0, S.Epsi);
      __int128 a2 = 0;
      long long mx = 0;
      // (cr + i ci)(vr + i vi) with three products; the sums (< 2^63) are
      // halved to stay in fx_mulhi's operand range
      auto term = [&](int i, const longlong2 v, long long& re, long long& im) {
        const int pi = S.cp[i];
        const long long cr = S.crm[i], ci = S.cim[i];
        const long long vr = v.x << pi, vi = v.y << pi;
        const long long p1 = fx_mulhi(cr, vr), p2 = fx_mulhi(ci, vi);
        const long long p3 = fx_mulhi((cr + ci) >> 1, (vr + vi) >> 1) << 2;
        re += p1 - p2;
        im += p3 - p1 - p2;
      };
      for (int x = wx0; x < wxe; x += wstep) {
        long long re = 0, im = 0;
        int i = 0;
        for (; i + 3 < acc_k; i += 4) {  // four basis loads in flight before their use
          longlong2 v[4];
#pragma unroll
          for (int j = 0; j < 4; ++j) v[j] = Q(i + j + 1)[x];
#pragma unroll
          for (int j = 0; j < 4; ++j) term(i + j, v[j], re, im);
        }
        for (; i < acc_k; ++i) term(i, Q(i + 1)[x], re, im);
        Q(1)[x] = make_longlong2(re, im);
        if constexpr (CLUSTER) sq[x - xb] = make_longlong2(re, im);
        if (final_rec) p.psi[x] = make_double2(__ll2double_rn(re) * outscale, __ll2double_rn(im) * outscale);
        a2 += (__int128)re * re + (__int128)im * im;
        mx = max(mx, fx_absmax(re, im));
      }
      fx_worker_partial(S, a2, mx);
      if (tid == 0) S.tacc[4] += (S.twe = sm_clock()) - tw0;
    } else if (cmd == kFxMax) {
      // -------- max |component| of psi (as ordered bit patterns of |v|; finds NaN and Inf too)
      long long mx = 0;
      for (int x = wx0; x < wxe; x += wstep) {
        const double2 v = p.psi[x];
        const long long a = __double_as_longlong(v.x) & 0x7FFFFFFFFFFFFFFFLL;
        const long long b = __double_as_longlong(v.y) & 0x7FFFFFFFFFFFFFFFLL;
        mx = max(mx, max(a, b));
      }
      fx_worker_partial(S, 0, mx);
    } else {
      // -------- psi (complex128) -> q_1, ||q_1||^2, max |M|
      const double sc = fx_scale2(1.0, -S.E[1]);
      __int128 a2 = 0;
      long long mx = 0;
      for (int x = wx0; x < wxe; x += wstep) {
        const double2 v = p.psi[x];
        const longlong2 qv = make_longlong2(__double2ll_rn(v.x * sc), __double2ll_rn(v.y * sc));
        Q(1)[x] = qv;
        if constexpr (CLUSTER) sq[x - xb] = qv;
        a2 += (__int128)qv.x * qv.x + (__int128)qv.y * qv.y;
        mx = max(mx, fx_absmax(qv.x, qv.y));
      }
      fx_worker_partial(S, a2, mx);
    }
    fx_cta_sync();  // the pass is done
  }
}

// Reconstruction coefficients of the accepted (k, ts) into S (control warp).
__device__ __noinline__ void fx_rec_consts(SmemFx& S, int acc_k, double ts) {
  const int lane = threadIdx.x & 31;
  if (!S.y_ready) small_expm_e1(acc_k, S.alpha + 1, S.beta + 1, ts, S.yr, S.yi, S.tr, S.ti);
  __syncwarp();
  double bnd = 0.0;
#pragma unroll 1
  for (int i = lane; i < acc_k; i += 32) {
    const double f = S.beta0 * S.scale[i + 1];
    const double cr = f * S.yr[i], ci = f * S.yi[i];
    S.yr[i] = cr;
    S.yi[i] = ci;
    bnd += (fabs(cr) + fabs(ci)) * fx_scale2(sb_ll_to_double_up(S.A[i + 1]), S.E[i + 1]);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) bnd += __shfl_xor_sync(0xffffffffu, bnd, o);
  const int Ep = fx_exp_for(bnd, kFxBits);
#pragma unroll 1
  for (int i = lane; i < acc_k; i += 32) {
    const Mant mr = fx_mant(S.yr[i]), mi = fx_mant(S.yi[i]);
    const int pi = sb_norm_shift_ll(S.A[i + 1]);
    S.cp[i] = pi;
    S.crm[i] = fx_fold(mr.m, Ep - mr.e - (S.E[i + 1] - pi) - 64);
    S.cim[i] = fx_fold(mi.m, Ep - mi.e - (S.E[i + 1] - pi) - 64);
  }
  if (lane == 0) S.Epsi = Ep;
}

// Full check of iteration it on the control warp: breakdown, then the gate and
// the estimate (err, into S.acc_err).  Returns 1 (accepted) or 0; y_ready is set
// when S.yr / S.yi hold y for the accepted (it, remaining).
__device__ __noinline__ int fx_check(SmemFx& S, int it, double tol, double tau, int m_min, bool estimate) {
  const int lane = threadIdx.x & 31;
  const double remaining = S.remaining, thr = tol * remaining / tau;
  int acc = 0, have_y = 0;
  double err = 0.0;
  if (fx_breakdown(S, it)) {
    acc = 1;
  } else if (estimate && it >= m_min) {
    const int gate = S.gate_it;
    if (gate >= 0 ? gate == 1 : fabs(remaining) * gersh_width(it, S.alpha + 1, S.beta + 1) <= 2.0 * it) {
      err = fx_estimate(S, it, remaining, thr);
      acc = have_y = err <= thr;
    }
  }
  __syncwarp();
  if (lane == 0) {
    S.acc_err = err;
    S.y_ready = have_y;
  }
  __syncwarp();
  return acc;
}

template <int FAMILY, class Op, int MODE>
__device__ __forceinline__ void fx_control(const PropParams& p, const Op& op, SmemFx& S, unsigned char* tiles_base,
                                           int NW) {
  constexpr bool TILED = MODE == kFxTiled;
  const int lane = threadIdx.x & 31;
  const int G = gridDim.x;
  const int ncoef = 1 + p.nV;
  // record exchange (ctl_exchange): tags continue across launches
  DevStatus* const st = p.st;
  // (kFxCluster: the launch's own slots in shared memory, tags from 1)
  unsigned tag = MODE == kFxCluster ? 0u : (unsigned)ld_volatile_i32((const int*)&st->tag_base);
  unsigned long long* const rec =
      reinterpret_cast<unsigned long long*>(MODE == kFxCluster ? (void*)tiles_base : (void*)p.partials);
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
  }
  // one element pass of the workers: start (command and constants set by lane
  // 0 or the warp) and end
  auto start = [&](int cmd, int it) {
    if (lane == 0) {
      S.cmd = cmd;
      S.it = it;
    }
    __syncwarp();
    fx_cta_sync();
  };
  double sum;
  long long mxi;

  // ---------------- psi (complex128) -> q_1
  start(kFxMax, 0);
  fx_cta_sync();
  if (!fx_ctl_reduce_cold<MODE>(S, NW, rec, ++tag, &st->status, p.timeout_ns)) return;
  if (S.rmx >= 0x7FF0000000000000LL) {
    if (lane == 0) atomicCAS(&st->status, 0, (int)CFET_ENAN);
    return;
  }
  if (lane == 0) S.E[1] = fx_exp_for(__longlong_as_double(S.rmx), kFxBits);
  start(kFxConvert, 0);
  fx_cta_sync();
  if (!fx_ctl_reduce_cold<MODE>(S, NW, rec, ++tag, &st->status, p.timeout_ns)) return;
  if (lane == 0) {
    S.nsum = S.rsum;
    S.A[1] = S.rmx;
  }
  __syncwarp();

  if (lane == 0) S.e = 0;
  __syncwarp();
  while (S.e < p.nexp) {
    if (lane < ncoef) S.scal[lane] = p.scal[S.e * ncoef + lane];
    if (lane == 0) {
      S.remaining = p.tau;
      S.nsub_e = 0;
    }
    __syncwarp();
    fx_stage_consts<FAMILY>(S, op, p.nV);
    while (true) {
      if (S.nsub_e >= p.max_substeps || (forced && S.nsub_e >= p.f_nsub[p.exp_base + S.e])) {
        if (glead) atomicCAS(&st->status, 0, (int)CFET_EKRYLOV);
        return;
      }
      const int klimit = forced ? p.f_k[S.fpos] : p.m_max;
      int acc_k = 0, acc_h = 0;
      if (lane == 0) S.acc_err = 0.0;
      if (__double_as_longlong(S.nsum) != 0) {  // (a zero state stays zero)
        if (lane == 0) {
          int p0;
          const double n = fx_norm_pow(S.nsum, S.E[1], p0), rs = rsqrt(n);
          S.E[1] -= p0;
          S.nq[1] = n;
          S.scale[1] = rs;
          S.rn[1] = rs * rs;
          S.beta0 = fx_scale2(n * rs, p0);
          S.y_ready = 0;
        }
        __syncwarp();
        fx_const_a_cold<FAMILY>(S, op, 1);
        bool accepted = false, pend = false;
        int it = 1;
        for (;; ++it) {
          // -------- phase A(it) on the workers; what iteration it-1 left here
          start(kFxApply, it);
          bool stop_prev = false;
          if (it > 1) {
            const long long te0 = sm_clock();
            if (lane == 0) fx_close_iteration(S, it - 1);
            __syncwarp();
            if (pend) {
              stop_prev = fx_check(S, it - 1, p.tol, p.tau, p.m_min, !fixed_k) != 0;
            }
            if (lane == 0) S.tacc[6] += sm_clock() - te0;
          }
          if constexpr (TILED) {  // grid exchanges between the window passes of the workers
            TileWin win[kTiledMaxWindows] = {};
            const int nwin = tiled_windows<kFxTileBits>(op.N, win);
            bool ok = true;
            for (int w = 0; w + 1 < nwin; ++w) {
              window_written_sync();
              ok = ok && fx_ctl_barrier(rec, ++tag, &st->status, p.timeout_ns, S.tacc[5]);
              window_exchanged_sync();
            }
            if (!ok) {
              fx_cta_sync();
              return;
            }
          }
          fx_cta_sync();
          {
            const long long sp0 = S.tacc[5];
            // (the tiled apply leaves u written by other CTAs: fence)
            if (!fx_ctl_reduce<MODE>(S, NW, rec, ++tag, TILED, &st->status, p.timeout_ns, sum, mxi, S.tacc[5]))
              return;
            if (stop_prev) {  // the deferred check accepted it-1
              it -= 1;
              accepted = true;
              break;
            }
            if (mxi >= (1LL << 60)) {  // fixed-point range exceeded (not expected)
              if (lane == 0) atomicCAS(&st->status, 0, (int)CFET_ENAN);
              return;
            }
            if (lane == 0) {
              const int Eu = S.Eu, Ek = S.E[it];
              const double alpha = fx_scale2(sum, Ek + Eu) * S.rn[it];
              S.alpha[it] = alpha;
              // phase-B constants: w = u - alpha q_it
              const long long Ak = S.A[it];
              const UpB Bw = sb_upb_add(sb_upb_scale2(sb_upb_ll(mxi), Eu),
                                        sb_upb_mul(sb_upb(alpha), sb_upb_scale2(sb_upb_ll(Ak), Ek)));
              const int Ew = sb_upb_exp_for(Bw, kFxBits);
              const Mant ma = fx_mant(-alpha);
              const int pk = sb_norm_shift_ll(Ak);
              S.Ew = Ew;
              S.sh_u = Ew - Eu;
              S.pk_b = pk;
              S.m_a = fx_fold(ma.m, Ew - ma.e - (Ek - pk) - 64);
              S.tacc[1] += sm_clock() - S.twe - (S.tacc[5] - sp0);
            }
          }
          // -------- phase B(it) on the workers; running bounds of T_it (alpha_it
          // and beta_{it-1} are known) and the FP32 gate of its estimate here
          start(kFxOrth, it);
          if (lane == 0) S.gate_it = krylov_bounds_update(S, it, S.remaining);
          __syncwarp();
          fx_cta_sync();
          {
            const long long sp0 = S.tacc[5];
            if (!fx_ctl_reduce<MODE>(S, NW, rec, ++tag, true, &st->status, p.timeout_ns, sum, mxi,
                                      S.tacc[5]))
              return;
            if (lane == 0) {
              int pw;
              const double n = fx_norm_pow(sum, S.Ew, pw);
              S.nq[it + 1] = n;
              S.pw[it] = pw;
              S.E[it + 1] = S.Ew - pw;
              S.A[it + 1] = mxi;
              S.cprev[it + 1] = fx_scale2(n * S.rn[it], pw);
            }
            __syncwarp();
            // the tests of this iteration run during the next apply (deferred
            // check) unless it is the last one or w vanished
            const bool zero = !(__double_as_longlong(sum) > 0);
            bool acc = false;
            pend = false;
            if (forced) {
              acc = it == klimit;
            } else if (fixed_k && it == klimit) {
              acc = true;
            } else if (zero || it == klimit) {
              if (lane == 0) fx_close_iteration(S, it);
              __syncwarp();
              acc = fx_check(S, it, p.tol, p.tau, p.m_min, !zero) != 0 || zero;
            } else {
              pend = true;
            }
            if (acc) {
              accepted = true;
              break;
            }
            if (it >= klimit) break;
            fx_const_a<FAMILY>(S, op, it + 1);
            if (lane == 0) S.tacc[3] += sm_clock() - S.twe - (S.tacc[5] - sp0);
          }
        }
        acc_k = it;
        if (forced) {
          acc_h = p.f_h[S.fpos];
        } else if (!accepted) {
          fx_halve(S, it, p.tol, p.tau);
          __syncwarp();
          acc_h = S.acc_h;
          if (acc_h == 0) {
            if (glead) atomicCAS(&st->status, 0, (int)CFET_EKRYLOV);
            return;
          }
        }
        // -------- reconstruct q_1 <- beta0 sum_i y_i s_i q_i
        {
          const long long tr0 = sm_clock();
          fx_rec_consts(S, acc_k, fx_scale2(S.remaining, -acc_h));
          if (lane == 0) {
            S.final_rec = S.e == p.nexp - 1 && acc_h == 0;
            S.tacc[6] += sm_clock() - tr0;
          }
        }
        start(kFxRec, acc_k);
        fx_cta_sync();
        if (!fx_ctl_reduce_cold<MODE>(S, NW, rec, ++tag, &st->status, p.timeout_ns)) return;
        if (lane == 0) {
          S.nsum = S.rsum;
          S.E[1] = S.Epsi;
          S.A[1] = S.rmx;
        }
        __syncwarp();
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
        S.remaining -= fx_scale2(S.remaining, -acc_h);
      }
      __syncwarp();
      if (acc_h == 0) break;
    }
    if (glead && p.r_nsub != nullptr) p.r_nsub[p.exp_base + S.e] = S.nsub_e;
    if (lane == 0) S.e += 1;
    __syncwarp();
  }
  if (glead) {
    if (MODE != kFxCluster) st->tag_base = tag;
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
__global__ void __launch_bounds__(CFET_CTL_MAX_THREADS, 1) k_propagate_fx(PropParams p, Op op) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  SmemFx& S = *reinterpret_cast<SmemFx*>(smem_raw);
  const int NW = (int)(blockDim.x >> 5) - 1;  // worker warps
  // behind SmemFx: the shared-memory basis of one-CTA launches, the tiled
  // apply's stage mbarriers (128 bytes) and tile buffers, or a cluster's
  // exchange slots and part of the applied vector
  unsigned char* const tiles_base = smem_raw + ((sizeof(SmemFx) + 127) & ~size_t(127));
  if constexpr (MODE == kFxTiled) {
    if (threadIdx.x == 0) {  // ordered before any use by the CTA barriers of the conversion pass
      for (int s2 = 0; s2 < kTmaStages; ++s2) mbar_init(reinterpret_cast<unsigned long long*>(tiles_base) + s2, 1);
      S.tma_fail = 0;
      mbar_init_fence();
    }
  }
  if constexpr (MODE == kFxCluster) {
    if (!cluster_is(gridDim.x, &p.st->status)) return;
    for (int i = threadIdx.x; i < kClusterSlotWords; i += blockDim.x)
      reinterpret_cast<unsigned long long*>(tiles_base)[i] = 0;
    __syncwarp();
    cluster_sync_all();  // every CTA runs, with its slots cleared
  }
  if ((int)(threadIdx.x >> 5) < NW) {
    fx_worker<FAMILY, Op, MODE>(p, op, S, tiles_base, NW * 32);
  } else {
    fx_control<FAMILY, Op, MODE>(p, op, S, tiles_base, NW);
    __syncwarp();
    if ((threadIdx.x & 31) == 0) S.cmd = kFxExit;  // also after an error
    __syncwarp();
    fx_cta_sync();
  }
  if constexpr (MODE == kFxCluster) {
    __syncwarp();
    cluster_sync_all();  // no CTA leaves while another may access its shared memory
  }
}

// ------------------------------------------------------------------ launchers
size_t fx_cluster_smem_bytes(int part) {
  return ((sizeof(SmemFx) + 127) & ~size_t(127)) + kClusterSlotWords * 8 + (size_t)part * sizeof(longlong2);
}

template <int FAMILY, class Op>
static int launch_prop_fx(const PropParams& p, const Op& op, int grid, int block, void* stream) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(block);
  cfg.dynamicSmemBytes = p.tiled     ? fx_tiled_smem_bytes()
                         : p.small   ? fx_small_smem_bytes(p.dim, p.m_max)
                         : p.cluster ? fx_cluster_smem_bytes(p.dim / grid)
                                     : sizeof(SmemFx);
  cfg.stream = (cudaStream_t)stream;
  cudaLaunchAttribute at[1];
  if (p.cluster) {
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = grid;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
  } else {
    at[0].id = cudaLaunchAttributeCooperative;
    at[0].val.cooperative = 1;
  }
  cfg.attrs = at;
  cfg.numAttrs = 1;
  if constexpr (FAMILY == kFamilySpin) {
    if (p.tiled) return (int)cudaLaunchKernelEx(&cfg, k_propagate_fx<FAMILY, Op, kFxTiled>, p, op);
    if (p.cluster) return (int)cudaLaunchKernelEx(&cfg, k_propagate_fx<FAMILY, Op, kFxCluster>, p, op);
  }
  if (p.small) return (int)cudaLaunchKernelEx(&cfg, k_propagate_fx<FAMILY, Op, kFxSmall>, p, op);
  return (int)cudaLaunchKernelEx(&cfg, k_propagate_fx<FAMILY, Op, kFxGrid>, p, op);
}

int launch_propagate_spin_fx(const PropParams& p, const OpSpinFx& op, int grid, int block, void* stream) {
  return launch_prop_fx<kFamilySpin>(p, op, grid, block, stream);
}
int launch_propagate_dia_fx(const PropParams& p, const OpDiaFx& op, int grid, int block, void* stream) {
  return launch_prop_fx<kFamilyDia>(p, op, grid, block, stream);
}
int launch_propagate_csr_fx(const PropParams& p, const OpCsrFx& op, int grid, int block, void* stream) {
  return launch_prop_fx<kFamilyCsr>(p, op, grid, block, stream);
}

size_t fx_tiled_smem_bytes() {
  return ((sizeof(SmemFx) + 127) & ~size_t(127)) + 128 + (size_t)kTmaStages * 2 * kFxTileBytes;
}

// Shared memory of a one-CTA launch that holds q_1 .. q_{m_max+1} (0 when it
// does not fit in an SM's shared memory).
size_t fx_small_smem_bytes(int dim, int m_max) {
  const size_t b = ((sizeof(SmemFx) + 127) & ~size_t(127)) + (size_t)(m_max + 1) * dim * sizeof(longlong2);
  return b <= kStagedSmemMax ? b : 0;
}

int fx_small_prepare() {
  cudaError_t e = cudaFuncSetAttribute(k_propagate_fx<kFamilySpin, OpSpinFx, kFxSmall>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kStagedSmemMax);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_propagate_fx<kFamilyDia, OpDiaFx, kFxSmall>,
                             cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kStagedSmemMax);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_propagate_fx<kFamilyCsr, OpCsrFx, kFxSmall>,
                             cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kStagedSmemMax);
  return (int)e;
}

// Largest cluster of at most `most` CTAs (a power of two) of `block` threads that
// holds a vector of dim elements in its shared memory; 0 when there is none.
int fx_cluster_prepare(int dim, int most, int block) {
  const void* k = (const void*)k_propagate_fx<kFamilySpin, OpSpinFx, kFxCluster>;
  if (cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) cudaGetLastError();
  if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kStagedSmemMax) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  for (int cs = most; cs >= 2; cs /= 2) {
    const size_t bytes = fx_cluster_smem_bytes(dim / cs);
    if (bytes > kStagedSmemMax) return 0;  // smaller clusters need more
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(cs);
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = bytes;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = cs;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, k, &cfg) == cudaSuccess && n >= 1) return cs;
    cudaGetLastError();
  }
  return 0;
}

int max_coresident_blocks_fx(int family, int block, bool tiled) {
  int dev = 0, nsm = 0, per = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  // the element-wise kernel needs only a few KB of shared memory: leave the
  // rest of the unified L1/shared storage to L1, which holds each CTA's chunk
  // (a tiled launch asks for its tile buffers and gets the split it needs)
  cudaFuncSetAttribute(k_propagate_fx<kFamilySpin, OpSpinFx, kFxGrid>, cudaFuncAttributePreferredSharedMemoryCarveout, 0);
  cudaFuncSetAttribute(k_propagate_fx<kFamilyDia, OpDiaFx, kFxGrid>, cudaFuncAttributePreferredSharedMemoryCarveout, 0);
  cudaFuncSetAttribute(k_propagate_fx<kFamilyCsr, OpCsrFx, kFxGrid>, cudaFuncAttributePreferredSharedMemoryCarveout, 0);
  cudaFuncSetAttribute(k_propagate_fx<kFamilySpin, OpSpinFx, kFxTiled>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                       (int)fx_tiled_smem_bytes());
  cudaError_t e;
  if (family == kFamilySpin)
    e = tiled ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_propagate_fx<kFamilySpin, OpSpinFx, kFxTiled>, block,
                                                              fx_tiled_smem_bytes())
              : cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_propagate_fx<kFamilySpin, OpSpinFx, kFxGrid>, block, sizeof(SmemFx));
  else if (family == kFamilyCsr)
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_propagate_fx<kFamilyCsr, OpCsrFx, kFxGrid>, block,
                                                      sizeof(SmemFx));
  else
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_propagate_fx<kFamilyDia, OpDiaFx, kFxGrid>, block,
                                                      sizeof(SmemFx));
  if (e != cudaSuccess) return -1;
  return per * nsm;
}

}  // namespace cfet
