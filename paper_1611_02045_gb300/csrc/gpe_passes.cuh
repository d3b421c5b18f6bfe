// gpe_passes.cuh -- the per-axis pass kernels of one PCG_C iteration
// (arXiv:1611.02045, Algorithm 2 with the operators of Sections 2, 3, 5.5).
//
// Each pass streams every point of a field once along one axis: it loads a
// line (x) or a tile of TX adjacent lines (y, z) into registers, applies a
// pointwise prologue, a line DFT (gpe_fft.cuh), a Fourier-space multiplier,
// optionally the inverse DFT, and a pointwise epilogue, then writes the
// result.  Reductions are accumulated per thread, combined per block in FP64
// and summed over blocks in a fixed order by the last block to finish, which
// then runs the scalar step that belongs after that pass (chemical potential,
// convergence test, Polak-Ribiere coefficient, step size).
//
// Pass roles (Pass enum in gpe_internal.h), 2D order per iteration:
//   HX   : [phi <- (c phi + s p/|p|)/nrm] ; t = (1/2 xi^2 + omega y xi) f + (V + eta|phi|^2) f
//   HMID : t += (1/2 mu^2 - omega x mu) f   (y)      or  (1/2 zeta^2) f  (z)
//   C1   : s = FFT_x[ P_V^{1/2} (t - lambda phi) ]
//   CCORE: s = IFFT_y[ FFT_y(s) / (alpha + |k|^2/2) ] / N
//   C3   : Pr = P_V^{1/2} IFFT_x[s]; r_prev <- r
//   AX   : p = -Pr + beta p_prev - gamma phi;  moments of p and of FFT_x p
//   AMID : moments of FFT_y p
// (3D inserts HMID for z, CFWD/CINV for y around CCORE on z, AMID for z.)
#pragma once
#include <cuda_runtime.h>
#include <math.h>

#include <type_traits>

#include "gpe_fft.cuh"
#include "gpe_internal.h"

namespace gpe {

enum StatusCode { ST_OK = 0, ST_ARG = 1, ST_CUDA = 2, ST_NOT_CONVERGED = 3, ST_NONFINITE = 4, ST_PRECOND = 5 };

// A line of M points is held by Tl = M / E threads, E values each (E = 8 by
// default; E = 4 doubles the threads per line for latency-bound passes).
template <int M, int EV = 8> struct LineCfg {
  static constexpr int E = EV;      // values per thread
  static constexpr int Tl = M / E;  // threads per line
  static_assert(M >= 8 && (M & (M - 1)) == 0, "M must be a power of two >= 8");
  static_assert((EV == 4 || EV == 8) && M >= EV, "E must be 4 or 8");
};

// ---------------------------------------------------------------------------
// Reductions.
//
// Sums are accumulated in double-single arithmetic: an unevaluated pair of
// FP32 numbers (hi, lo), added with Knuth's TwoSum error-free transformation
// (D. E. Knuth, TAOCP vol. 2, 4.2.2) followed by a fast renormalisation
// (T. J. Dekker, "A floating-point technique for extending the available
// precision", Numer. Math. 18, 1971).  The pair carries ~48 significant bits
// (relative error ~2^-47 per addition), so sums of FP32 terms lose nothing
// and sums of FP64 terms lose ~1e-14 relative.  On GB300 an FP64 warp
// instruction occupies the FP64 pipe ~64x longer than an FP32 one, so the
// pair arithmetic keeps the many-level block and grid reductions off that
// pipe; totals are converted to FP64 once, for the scalar steps.
// Slots flagged in MAXMASK take the maximum instead (of non-negative values).
// ---------------------------------------------------------------------------
struct Acc {
  float hi, lo;
};

__device__ __forceinline__ Acc acc_from(float x) { return Acc{x, 0.0f}; }
__device__ __forceinline__ Acc acc_from(double x) {
  const float h = (float)x;
  return Acc{h, (float)(x - (double)h)};
}
__device__ __forceinline__ Acc acc_from(dsf x) { return Acc{x.hi, x.lo}; }
__device__ __forceinline__ double acc_to_double(Acc a) { return (double)a.hi + (double)a.lo; }

__device__ __forceinline__ Acc acc_add(Acc a, Acc b) {
  const float s = a.hi + b.hi;
  const float bp = s - a.hi;
  float e = (a.hi - (s - bp)) + (b.hi - bp);  // TwoSum: s + e = a.hi + b.hi exactly
  e += a.lo + b.lo;
  const float h = s + e;                      // renormalise (|e| <= ulp(s))
  return Acc{h, e - (h - s)};
}
__device__ __forceinline__ Acc acc_max(Acc a, Acc b) {
  return (b.hi > a.hi || (b.hi == a.hi && b.lo > a.lo)) ? b : a;
}

// Slot k's reduction (k may differ between lanes).
template <unsigned MAXMASK>
__device__ __forceinline__ Acc red_op(Acc a, Acc b, int k) {
  const Acc s = acc_add(a, b);
  if constexpr (MAXMASK == 0u) return s;
  return ((MAXMASK >> k) & 1u) ? acc_max(a, b) : s;
}

// Two double-single additions at once on the packed two-wide FP32 pipe: lane by
// lane the same operations in the same order as acc_add (each lane rounds like
// the scalar .rn operation), so the sums are bit-identical with half the
// floating-point instructions.
__device__ __forceinline__ unsigned long long f2add(unsigned long long a, unsigned long long b) {
  unsigned long long d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ unsigned long long f2sub(unsigned long long a, unsigned long long b) {
  unsigned long long d;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ void acc_add2(Acc& a0, Acc& a1, Acc b0, Acc b1) {
  const unsigned long long ah = f2_pack(a0.hi, a1.hi), al = f2_pack(a0.lo, a1.lo);
  const unsigned long long bh = f2_pack(b0.hi, b1.hi), bl = f2_pack(b0.lo, b1.lo);
  const unsigned long long sm = f2add(ah, bh);
  const unsigned long long bp = f2sub(sm, ah);
  unsigned long long e = f2add(f2sub(ah, f2sub(sm, bp)), f2sub(bh, bp));
  e = f2add(e, f2add(al, bl));
  const unsigned long long h = f2add(sm, e);
  const unsigned long long lo = f2sub(e, f2sub(h, sm));
  const float2 H = f2_unpack(h), Lo = f2_unpack(lo);
  a0 = Acc{H.x, Lo.x};
  a1 = Acc{H.y, Lo.y};
}

__device__ __forceinline__ Acc shfl_acc(unsigned mask, Acc v, int o) {
  return Acc{__shfl_xor_sync(mask, v.hi, o), __shfl_xor_sync(mask, v.lo, o)};
}

// Slots padded to a power of two.
template <int K> struct Slots {
  static constexpr int lg = K <= 1 ? 0 : K <= 2 ? 1 : K <= 4 ? 2 : K <= 8 ? 3 : 4;
  static constexpr int P = 1 << lg;
};

// The K slots reduced over a full warp in a fixed order: lane l returns the total
// of slot l >> (5 - lg).  Each of the first lg steps halves the slots a lane keeps
// along with the lanes, so K = 9 takes 16 additions, not 45.  These sums are short
// on purpose: in the last block of a pass, and in every pass of a resident solve,
// they run once through, and their time is that of fetching the instructions (a
// fully unrolled tree over all slots, in several copies, was most of the code:
// cluster solve 39 -> 26 us per iteration at 64^2, 60 -> 48 at 256^2; graph loop
// 487 -> 458 us per refinement iteration at 128^3, 85 -> 75 at 256^2).
template <int K, unsigned MAXMASK>
__device__ __forceinline__ Acc warp_slots(const Acc (&v)[K]) {
  constexpr int lg = Slots<K>::lg, P = Slots<K>::P;
  const int lane = threadIdx.x & 31;
  Acc w[P];
#pragma unroll
  for (int k = 0; k < P; ++k) w[k] = (k < K && !((MAXMASK >> k) & 1u)) ? v[k < K ? k : 0] : Acc{0.0f, 0.0f};
#pragma unroll
  for (int st = 0; st < lg; ++st) {
    const int o = 16 >> st, h = P >> (st + 1);
    const bool up = lane & o;
#pragma unroll
    for (int j = 0; j < h; j += 2) {
      const Acc k0 = up ? w[j + h] : w[j], s0 = up ? w[j] : w[j + h];
      const Acc r0 = shfl_acc(0xffffffffu, s0, o);
      if (j + 1 < h) {
        const Acc k1 = up ? w[j + 1 + h] : w[j + 1], s1 = up ? w[j + 1] : w[j + 1 + h];
        const Acc r1 = shfl_acc(0xffffffffu, s1, o);
        w[j] = k0;
        w[j + 1] = k1;
        acc_add2(w[j], w[j + 1], r0, r1);
      } else {
        w[j] = acc_add(k0, r0);
      }
    }
  }
#pragma unroll
  for (int o = 16 >> lg; o > 0; o >>= 1) w[0] = acc_add(w[0], shfl_acc(0xffffffffu, w[0], o));
  if constexpr (MAXMASK != 0u) {
#pragma unroll
    for (int k = 0; k < K; ++k)
      if ((MAXMASK >> k) & 1u) {
        Acc x = v[k];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) x = acc_max(x, shfl_acc(0xffffffffu, x, o));
        if ((lane >> (5 - lg)) == k) w[0] = x;
      }
  }
  return w[0];
}

// Block totals: sink(k, total of slot k) is called once per slot by a thread of
// warp 0 (thread k where the block has a full warp).  red_sm: kRedSlots elements.
// LEAD = false skips the barrier that protects red_sm from the previous call's
// readers: for callers that alternate between two red_sm buffers, whose other
// barriers already order a buffer's readers before its next writers.
constexpr int kRedSlots = 256;
template <int K, unsigned MAXMASK, bool LEAD = true, typename Sink>
__device__ __forceinline__ void block_reduce(const Acc (&v)[K], Acc* red_sm, Sink sink) {
  constexpr int lg = Slots<K>::lg, P = Slots<K>::P;
  // blockDim.x is a power of two: either a multiple of 32 or one partial warp
  if (blockDim.x >= 32) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    Acc t = warp_slots<K, MAXMASK>(v);
    if (nw == 1) {
      const int src = (lane & (P - 1)) << (5 - lg);
      t = Acc{__shfl_sync(0xffffffffu, t.hi, src), __shfl_sync(0xffffffffu, t.lo, src)};
    } else {
      if constexpr (LEAD) __syncthreads();
      if ((lane & ((32 >> lg) - 1)) == 0) red_sm[warp * P + (lane >> (5 - lg))] = t;
      __syncthreads();
      if (warp != 0) return;
      const int k = lane & (P - 1);
      t = Acc{0.0f, 0.0f};  // also the identity of the maxima, which are >= 0
#pragma unroll 2
      for (int w = lane >> lg; w < nw; w += 32 >> lg) t = red_op<MAXMASK>(t, red_sm[w * P + k], k);
#pragma unroll
      for (int o = P; o < 32; o <<= 1) t = red_op<MAXMASK>(t, shfl_acc(0xffffffffu, t, o), k);
    }
    if (lane < K) sink(lane, t);
  } else {
    if constexpr (LEAD) __syncthreads();
#pragma unroll
    for (int k = 0; k < K; ++k) red_sm[threadIdx.x * K + k] = v[k];
    __syncthreads();
    for (int k = threadIdx.x; k < K; k += blockDim.x) {
      Acc t = red_sm[k];
      for (int j = 1; j < (int)blockDim.x; ++j) t = red_op<MAXMASK>(t, red_sm[j * K + k], k);
      sink(k, t);
    }
  }
}

// Partials live in a double-sized slot each (an Acc is 8 bytes).
__device__ __forceinline__ Acc* acc_slots(double* p) { return reinterpret_cast<Acc*>(p); }

// Reduction slots per pass, which of them are maxima, and which carry the
// quadrature weight h^d in their total.
template <int ROLE> struct Moments { static constexpr int K = 0; static constexpr unsigned MAX = 0u, W = 0u; };
template <> struct Moments<P_HX> { static constexpr int K = 6; static constexpr unsigned MAX = 32u, W = 31u; };
template <> struct Moments<P_HMID> { static constexpr int K = 2; static constexpr unsigned MAX = 0u, W = 3u; };
template <> struct Moments<P_C1> { static constexpr int K = 3; static constexpr unsigned MAX = 1u, W = 2u; };
template <> struct Moments<P_C3> { static constexpr int K = 6; static constexpr unsigned MAX = 0u, W = 63u; };
template <> struct Moments<P_AX> { static constexpr int K = 9; static constexpr unsigned MAX = 0u, W = 511u; };
template <> struct Moments<P_AMID> { static constexpr int K = 1; static constexpr unsigned MAX = 0u, W = 1u; };

// A total in FP64, times the weight where W says so.  Each thread converts its own
// slot: an FP64 instruction occupies its sub-partition's pipe for 64 cycles
// whatever the number of active lanes, so one thread converting K slots in turn
// would take K times as long.
template <unsigned W>
__device__ __forceinline__ double total(Acc x, double weight, int k) {
  return acc_to_double(x) * (((W >> k) & 1u) ? weight : 1.0);
}

// Sums of block partials in a fixed order, K slots at once: slot k adds elements
// src(k)[b * kMaxMoments], b < nb(k); sink as for block_reduce.  A thread sums one
// slot over a subset of the blocks, 16 L2-coherent loads in flight: a few hundred
// instructions where one thread per block and all slots in registers takes
// thousands.
template <int K, unsigned MAXMASK, typename Src, typename Nb, typename Sink>
__device__ __forceinline__ void sum_partials(Src src, Nb nb, Acc* red_sm, Sink sink) {
  constexpr int lg = Slots<K>::lg, P = Slots<K>::P, U = 16;
  static_assert(16 * K <= kRedSlots, "one row of slots per thread of a block below a warp");
  if (blockDim.x < 32) {
    // a thread takes every blockDim-th block, all slots' loads in flight at once: one
    // slot per thread, one load at a time, took 360 us over the 1024 blocks of 16 threads
    // of a z pass of 128 x 128 x 8
    Acc t[K];
    int n[K], most = 0;
#pragma unroll
    for (int k = 0; k < K; ++k) {
      t[k] = Acc{0.0f, 0.0f};
      n[k] = nb(k);
      most = n[k] > most ? n[k] : most;
    }
#pragma unroll 2
    for (int b = threadIdx.x; b < most; b += blockDim.x) {
      float2 x[K];
#pragma unroll
      for (int k = 0; k < K; ++k)
        x[k] = b < n[k] ? __ldcg(reinterpret_cast<const float2*>(src(k)) + (size_t)b * kMaxMoments) : make_float2(0.0f, 0.0f);
#pragma unroll
      for (int k = 0; k < K; ++k) t[k] = red_op<MAXMASK>(t[k], Acc{x[k].x, x[k].y}, k);
    }
    __syncthreads();  // earlier readers of red_sm
#pragma unroll
    for (int k = 0; k < K; ++k) red_sm[threadIdx.x * K + k] = t[k];
    __syncthreads();
    for (int k = threadIdx.x; k < K; k += blockDim.x) {
      Acc r = red_sm[k];
      for (int j = 1; j < (int)blockDim.x; ++j) r = red_op<MAXMASK>(r, red_sm[j * K + k], k);
      sink(k, r);
    }
    return;
  }
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const int k = lane & (P - 1), J = (int)blockDim.x >> lg;
  const int n = k < K ? nb(k) : 0;
  const float2* p = reinterpret_cast<const float2*>(src(k < K ? k : 0));
  Acc t{0.0f, 0.0f};
  for (int b0 = threadIdx.x >> lg; b0 < n; b0 += U * J) {
    float2 x[U];
#pragma unroll
    for (int i = 0; i < U; ++i)
      x[i] = b0 + i * J < n ? __ldcg(p + (size_t)(b0 + i * J) * kMaxMoments) : make_float2(0.0f, 0.0f);
#pragma unroll
    for (int i = 0; i < U; ++i) t = red_op<MAXMASK>(t, Acc{x[i].x, x[i].y}, k);
  }
  __syncwarp();
#pragma unroll
  for (int o = P; o < 32; o <<= 1) t = red_op<MAXMASK>(t, shfl_acc(0xffffffffu, t, o), k);
  if (nw > 1) {
    __syncthreads();  // earlier readers of red_sm
    if (lane < P) red_sm[warp * P + lane] = t;
    __syncthreads();
    if (warp != 0) return;
    t = Acc{0.0f, 0.0f};
#pragma unroll 2
    for (int w = lane >> lg; w < nw; w += 32 >> lg) t = red_op<MAXMASK>(t, red_sm[w * P + k], k);
#pragma unroll
    for (int o = P; o < 32; o <<= 1) t = red_op<MAXMASK>(t, shfl_acc(0xffffffffu, t, o), k);
  }
  if (lane < K) sink(lane, t);
}

// ---------------------------------------------------------------------------
// Scalar steps.  Run by warp 0 of the last block (all its lanes hold the same
// values; lane 0 writes), or by every CTA of a resident solve, on a control
// block in shared memory.  They are chains of FP64 instructions of 64 cycles
// each, on the critical path of every iteration, so they are written for few
// of them: moments arrive weighted (totals), reciprocal square roots take the
// place of square root and division, and what is independent (square roots,
// sine and cosine, the splits of a Num) is spread over the lanes, which cost
// nothing extra.
// ---------------------------------------------------------------------------
// Constants the scalar steps need (from the pass arguments).
struct Fin {
  double eta, omega;
  int dim, solver;
};

__device__ __forceinline__ Fin fin_of(const PassArgs& a) { return Fin{a.eta, a.omega, a.dim, a.solver}; }

// par: the caller is a full warp (blocks of fewer than 32 threads run the
// scalar steps on thread 0 alone).
__device__ __forceinline__ bool full_warp() { return blockDim.x >= 32; }
__device__ __forceinline__ double lane_value(double v, int src) { return __shfl_sync(0xffffffffu, v, src); }

// The square roots of three values.
__device__ __forceinline__ void sqrt3(double& a, double& b, double& c) {
  if (full_warp()) {
    const int l = threadIdx.x & 31;
    const double r = sqrt(l == 0 ? a : (l == 1 ? b : c));
    a = lane_value(r, 0); b = lane_value(r, 1); c = lane_value(r, 2);
  } else {
    a = sqrt(a); b = sqrt(b); c = sqrt(c);
  }
}

// *na = num(a), *nb = num(b).
__device__ __forceinline__ void put_nums(double a, Num* na, double b, Num* nb) {
  if (full_warp()) {
    const int l = threadIdx.x & 31;
    const Num n = num(l == 0 ? a : b);
    if (l < 2) *(l == 0 ? na : nb) = n;
  } else {
    *na = num(a);
    *nb = num(b);
  }
}

__device__ __forceinline__ bool finite_d(double x) { return (__double2hiint(x) & 0x7ff00000) != 0x7ff00000; }

// Row n of the iteration log, or null (no log, full, or not the writing block).
__device__ __forceinline__ double* log_row(Ctl* c, bool writer) {
  return (writer && c->log && c->iter < c->log_cap) ? c->log + (size_t)c->iter * kLogFields : nullptr;
}

// After the last H pass: energy terms, lambda_n, lambda~_n, E_n (Section 2, eq. Opt_Alpha).
// h0: the x pass's totals; h1, h2: those of the y and z passes (kinetic, rotation).
static __device__ void finalize_H(Ctl* c, const Fin& a, const double* h0, const double* h1, const double* h2,
                                  bool writer) {
  double kin = h0[0] + h1[0], lz = h0[1] + h1[1];
  if (a.dim == 3) { kin += h2[0]; lz += h2[1]; }
  const double pot = h0[2], U0 = h0[3];
  const double rot = a.omega * lz;  // -omega <phi, L_z phi>: the passes sum the symbol without omega
  const double kp = kin + pot, eU = a.eta * U0;
  const double quad = kp + rot;
  const double lam = quad + eU;    // <phi, H phi>
  const double alpha = kp + eU;    // lambda~ (no rotation term)
  const double E = quad + 0.5 * eU;
  put_nums(lam, &c->lam_n, alpha, &c->alpha_n);
  if ((threadIdx.x & 31) != 0) return;
  c->kin = kin; c->Lz = -lz; c->rot = rot; c->pot = pot; c->U0 = U0;
  c->norm2 = h0[4];
  c->umax = h0[5];
  c->lam = lam; c->alpha = alpha; c->E = E;
  if (a.solver && c->log) {
    double* row = log_row(c, writer);
    if (row) {
      row[0] = c->iter; row[1] = c->phase; row[2] = E; row[3] = lam;
      row[6] = alpha;
      row[4] = row[5] = row[7] = row[8] = row[9] = row[10] = row[11] = 0.0;
    }
    if (c->iter + 1 > c->log_len) c->log_len = (c->iter + 1 < c->log_cap) ? c->iter + 1 : c->log_cap;
  }
}

// After C1: residual norms and the stopping rule (eq. Stop_Residual), the
// iteration cap, the optional energy rule, and (mixed phase) stall detection.
// tot: max |r|^2, ||r||_2^2, count of alpha + V + eta|phi|^2 <= 0
static __device__ void finalize_C1(Ctl* c, const double* tot, bool writer) {
  double res_inf = tot[0], res_l2 = tot[1], phimax = c->umax;
  sqrt3(res_inf, res_l2, phimax);
  if ((threadIdx.x & 31) != 0) return;
  c->res_inf = res_inf;
  c->res_l2 = res_l2;
  double* row = log_row(c, writer);
  if (row) { row[4] = res_inf; row[5] = res_l2; }
  const int nphase = c->iter - c->iter_phase0;
  if (!finite_d(c->E) || !finite_d(res_inf) || !finite_d(c->lam)) {
    c->status = ST_NONFINITE; c->done = 1;
  } else if (tot[2] > 0.0) {
    c->status = ST_PRECOND; c->done = 1;
  } else if (res_inf < c->tol_res_inf || c->stop_dE) {
    c->status = ST_OK; c->done = 1;
  } else if (c->iter >= c->max_iter) {
    c->status = ST_NOT_CONVERGED; c->done = 1;
  } else if (c->lo_phase) {
    // complex64 phase: stop at the single-precision residual floor, estimated
    // as eps32 (max |k|^2/2 + max V + |lambda|) max|phi|, or on a stall near it
    const double floor_est = (c->floor_coef + 5.96e-8 * fabs(c->lam)) * phimax;
    const double thr = c->switch_res > 0.0 ? c->switch_res : c->switch_fac * floor_est;
    if (res_inf <= 0.5 * c->anchor_res) { c->anchor_res = res_inf; c->anchor_iter = c->iter; }
    const bool stalled = c->iter - c->anchor_iter >= c->stall_window && res_inf < 3.0 * thr;
    if (res_inf < thr || stalled || nphase >= c->max_iter_phase) {
      c->switch_req = 1; c->status = ST_NOT_CONVERGED; c->done = 1;
    }
  } else if (c->stall_switch) {
    // refinement phase: its step moments are single precision; if ||r||_inf
    // has not halved for 4 stall_window iterations, finish in FP64 (after the
    // beta restart ||r||_inf first grows ~10x; on the 256^2 and 128^3 bench
    // problems the longest gap between halvings is ~1500 iterations)
    if (res_inf <= 0.5 * c->anchor_res) { c->anchor_res = res_inf; c->anchor_iter = c->iter; }
    if (c->iter - c->anchor_iter >= 4 * c->stall_window) {
      c->switch_req = 1; c->status = ST_NOT_CONVERGED; c->done = 1;
    }
  }
}

// After C3: Polak-Ribiere beta+ (eq. CG:PR), gamma = Re<d, phi>, and the
// descent check of Section 5.2 (Re<grad E, p> >= 0 -> gradient step).
// tot: 0 <r,Pr>, 1 Re<r - r_prev, Pr>, 2 Re<Pr,phi>, 3 Re<p_prev,phi>,
//      4 Re<r,p_prev>, 5 Re<r,phi>
static __device__ void finalize_C3(Ctl* c, const double* tot, bool writer) {
  const double rPr = tot[0], Prphi = tot[2], pphi = tot[3], rp = tot[4], rphi = tot[5];
  double beta = 0.0;
  if (!c->restart && c->cg)
    beta = c->beta_rule == 1 ? rPr / c->rPr_prev               // Fletcher-Reeves (eq. CG:FR)
                             : fmax(tot[1] / c->rPr_prev, 0.0);  // Polak-Ribiere beta+
  double gamma = beta * pphi - Prphi;
  // Re<H phi, p> = Re<r, d> - gamma Re<r, phi> + lambda gamma (1 - ||phi||^2)
  const double desc = beta * rp - rPr + gamma * (c->lam * (1.0 - c->norm2) - rphi);
  const bool fallback = desc >= 0.0;
  if (fallback) {
    beta = 0.0;
    gamma = -Prphi;
  }
  if (full_warp()) __syncwarp();  // every lane has read the previous scalars
  put_nums(beta, &c->beta_n, gamma, &c->gamma_n);
  if ((threadIdx.x & 31) != 0) return;
  c->fallback = fallback ? 1 : 0;
  c->fallbacks += fallback ? 1 : 0;
  c->rPr_prev = rPr;
  double* row = log_row(c, writer);
  if (row) { row[7] = beta; row[10] = c->fallback; }
}

// sin and cos of a step angle.  Steps are usually tiny, so for |t| < 0.05
// the Maclaurin series (truncation below 1e-18 there: t^9/9! and t^10/10!)
// replaces the general FP64 sincos, which is long on GB300's FP64 pipe; even
// lanes sum the sine's, odd lanes the cosine's.
__device__ __forceinline__ void step_sincos(double t, double* s, double* c) {
  if (fabs(t) < 0.05) {
    const double t2 = t * t;
    if (full_warp()) {
      const bool odd = threadIdx.x & 1;
      double v = odd ? -1.0 / 3628800 : 1.0 / 362880;
      v = fma(t2, v, odd ? 1.0 / 40320 : -1.0 / 5040);
      v = fma(t2, v, odd ? -1.0 / 720 : 1.0 / 120);
      v = fma(t2, v, odd ? 1.0 / 24 : -1.0 / 6);
      v = fma(t2, v, odd ? -0.5 : 1.0);
      v = fma(odd ? t2 : t, v, odd ? 1.0 : 0.0);
      *s = lane_value(v, 0);
      *c = lane_value(v, 1);
      return;
    }
    *s = t * (1.0 + t2 * (-1.0 / 6 + t2 * (1.0 / 120 + t2 * (-1.0 / 5040 + t2 * (1.0 / 362880)))));
    *c = 1.0 + t2 * (-0.5 + t2 * (1.0 / 24 + t2 * (-1.0 / 720 + t2 * (1.0 / 40320 + t2 * (-1.0 / 3628800)))));
  } else {
    sincos(t, s, c);
  }
}

// Energy change along the geodesic (reading R6), an exact trigonometric
// polynomial in s = sin(theta), c = cos(theta):
//   2 R cs + A s^2 + B s^4 + C c^2 s^2 + D c s^3,
// A = aqq - lam, B = eta/2 (U0 + W2), C = eta/2 (4 V2 + 2 UW), D = 2 eta (VW - U1).
struct StepPoly {
  double R, A, B, C, D;
};
__device__ __forceinline__ double delta_E(const StepPoly& P, double s, double c) {
  const double s2 = s * s, cs = c * s;
  return 2.0 * P.R * cs + s2 * (P.A + P.B * s2 + P.C * (c * c) + P.D * cs);
}

// Newton's method on d/dt of the step polynomial delta_E (closed-form first
// and second derivatives) from the model step t0; t0 is kept when the
// curvature is not positive or the iterate leaves (0, pi/2].
static __device__ __noinline__ double exact_step(double t0, const StepPoly& P) {
  const double R = P.R, A = P.A, B = P.B, C = P.C, D = P.D;
  double t = t0;
  for (int it = 0; it < 30; ++it) {
    double s, c, s2, c2, s4, c4;
    sincos(t, &s, &c);
    sincos(2.0 * t, &s2, &c2);
    sincos(4.0 * t, &s4, &c4);
    const double d1 = 2.0 * R * c2 + A * s2 + 4.0 * B * s * s * s * c + 0.5 * C * s4 + D * (3.0 * c * c * s * s - s * s * s * s);
    const double d2 = -4.0 * R * s2 + 2.0 * A * c2 + 4.0 * B * (3.0 * s * s * c * c - s * s * s * s) + 2.0 * C * c4 +
                      D * (6.0 * c * s * (c * c - s * s) - 4.0 * s * s * s * c);
    if (!(d2 > 0.0)) return t0;
    const double dt = d1 / d2;
    t -= dt;
    if (!(t > 0.0 && t <= 1.5707963267948966)) return t0;
    if (fabs(dt) <= 1e-15 * fabs(t)) break;
  }
  return t;
}

// After the last A pass: step size by the model minimiser (eq. theta_opt,
// reading R4) with energy-decrease backtracking (Section 5.1), then the
// retraction scalars for the next H pass.
// m: the x pass's totals: 0 Re<H phi,p>, 1 <p,A_x p>+<p,V p>, 2 |p|^2, 3 u v,
//    4 v^2, 5 u w, 6 v w, 7 w^2, 8 v (u = |phi|^2, v = Re(conj(phi) p), w = |p|^2);
// ay, az: <p, A_axis p> of the y and z passes.
static __device__ void finalize_A(Ctl* c, const Fin& a, const double* m, double ay, double az, bool writer) {
  const double inv = rsqrt(m[2]);  // 1 / ||p||
  const double inv2 = inv * inv;
  double app = m[1] + ay;
  if (a.dim == 3) app += az;
  const double lam = c->lam, U0 = c->U0, norm2 = c->norm2;
  const double eta2 = a.eta * inv2;
  // moments of q = p / ||p||
  StepPoly P;
  P.R = m[0] * inv;
  P.A = app * inv2 - lam;
  P.B = 0.5 * (eta2 * (inv2 * m[7]) + a.eta * U0);
  P.C = eta2 * (2.0 * m[4] + m[5]);
  P.D = 2.0 * a.eta * inv * (inv2 * m[6] - m[3]);
  const double rho = m[8] * inv;
  const double curv = P.A + P.C;  // T2(q) - lambda = aqq + eta UW + 2 eta V2 - lambda
  double th = (curv > 0.0) ? -P.R / curv : c->theta_default;
  if (c->line_search == 1) th = exact_step(th, P);
  double sn, cs;
  step_sincos(th, &sn, &cs);
  double dE = delta_E(P, sn, cs);
  int bt = 0;
  while (!(dE < 0.0) && bt < c->max_backtracks) {
    th *= 0.5; ++bt;
    step_sincos(th, &sn, &cs);
    dE = delta_E(P, sn, cs);
  }
  const double inv_nrm = rsqrt(cs * (cs * norm2 + 2.0 * sn * rho) + sn * sn);
  put_nums(cs * inv_nrm, &c->cc, sn * inv * inv_nrm, &c->ss);
  if (full_warp()) __syncwarp();  // every lane has read c
  if ((threadIdx.x & 31) != 0) return;
  c->theta = th;
  c->dE = dE; c->backtracks = bt; c->backtracks_total += bt;
  double* row = log_row(c, writer);
  if (row) { row[8] = th; row[9] = dE; row[11] = bt; }
  c->retract = 1;
  c->restart = 0;
  c->iter += 1;
  if (c->tol_dE > 0.0 && fabs(dE) <= c->tol_dE) c->stop_dE = 1;
  if (!finite_d(dE) || !finite_d(th)) { c->status = ST_NONFINITE; c->done = 1; }
}

__device__ __forceinline__ void set_loop_condition(const PassArgs& a, int keep_going) {
  if (a.cond) cudaGraphSetConditional((cudaGraphConditionalHandle)a.cond, keep_going ? 1u : 0u);
}

// A Num in a kernel's precision.
template <typename T> __device__ __forceinline__ T num_as(const Num& n);
template <> __device__ __forceinline__ float num_as<float>(const Num& n) { return n.hi; }
template <> __device__ __forceinline__ double num_as<double>(const Num& n) { return n.d; }
template <> __device__ __forceinline__ dsf num_as<dsf>(const Num& n) { return dsf(n.hi, n.lo); }

// Scalars a pass body reads (from the control block).  In a solve, done is
// only looked at once a pass has its operands in flight: nothing is written
// after that, so the control block's latency hides behind the fields'.
struct Scal {
  int retract, done;
  int pc;  // preconditioner kind (Ctl::pc_kind; API calls: 0, P_C)
  Num cc, ss, lam, alpha, beta, gamma;
};

// The preconditioners of Section 5.4 as P_V^a P_Delta^b P_V^c around the
// Fourier core: exponents of P_V before (pre) and after (post) the core,
// coded 0 (none), 1 (P_V^{1/2}), 2 (P_V), and whether the core divides by
// alpha + |k|^2/2 (P_Delta, eq. PDelta) or is the identity.
//   P_C  = P_V^{1/2} P_Delta P_V^{1/2} (eq. combinedP_12): 1, Delta, 1
//   P_Delta (eq. PDelta): 0, Delta, 0      P_V (eq. PV): 2, identity, 0
//   P_C1 = P_V P_Delta (eq. combinedP): 0, Delta, 2  (P_Delta first)
//   P_C2 = P_Delta P_V (eq. combinedP): 2, Delta, 0  (P_V first)
//   none: 0, identity, 0
__device__ __forceinline__ int pc_pre(int k) { return k == 0 ? 1 : (k == 2 || k == 4) ? 2 : 0; }
__device__ __forceinline__ int pc_post(int k) { return k == 0 ? 1 : k == 3 ? 2 : 0; }
__device__ __forceinline__ bool pc_core(int k) { return !(k == 2 || k == 5); }
template <typename T> __device__ __forceinline__ T pv_factor(T den, int code) {
  return code == 0 ? T(1) : (code == 2 ? T(1) / den : T(1) / sqrt(den));
}
// FP64: one reciprocal square root instead of a square root and a division.
template <> __device__ __forceinline__ double pv_factor<double>(double den, int code) {
  return code == 0 ? 1.0 : (code == 2 ? __drcp_rn(den) : rsqrt(den));
}
// Double-single: the FP32 reciprocal square root with a second-order correction from
// its residual e = 1 - den y^2 ((1 - e)^{-1/2} = 1 + e/2 + 3 e^2/8 + ..., e ~ 2^-22, so
// e^3 is below the last bit), about 20 operations where a square root and a division
// take some 110; relative error against FP64 1.6e-14 at most, 1.9e-15 rms (1.6e-14 and
// 2.4e-15 with root and division).
template <> __device__ __forceinline__ dsf pv_factor<dsf>(dsf den, int code) {
  if (code == 0) return dsf(1.0f);
  if (code == 2) return dsf(1.0f) / den;
  const float y = rsqrtf(den.hi);
  const float th = den.hi * y, tl = fmaf(den.lo, y, fmaf(den.hi, y, -th));  // den y
  const float p = th * y;
  const float e = (1.0f - p) - fmaf(tl, y, fmaf(th, y, -p));
  return ds_fast_two_sum(y, y * e * fmaf(0.375f, e, 0.5f));
}
// p / den for a power of two p: FP64 takes the (correctly rounded) reciprocal,
// whose scaling is exact, in place of the longer division.
template <typename T> __device__ __forceinline__ T over(T p, T den) { return p / den; }
template <> __device__ __forceinline__ double over<double>(double p, double den) { return p * __drcp_rn(den); }

__device__ __forceinline__ Scal scal_of(const Ctl* c, const PassArgs& a) {
  Scal S;
  S.retract = a.solver ? c->retract : 0;
  S.done = a.solver ? c->done : 0;
  S.pc = a.solver ? c->pc_kind : 0;
  S.cc = c->cc; S.ss = c->ss;
  S.lam = c->lam_n;
  S.alpha = (a.solver || __double_as_longlong(a.api_alpha.d) <= 0) ? c->alpha_n : a.api_alpha;  // <= 0: adaptive
  S.beta = c->beta_n; S.gamma = c->gamma_n;
  return S;
}

// ---------------------------------------------------------------------------
// Multipliers
// ---------------------------------------------------------------------------
template <typename T>
__device__ __forceinline__ const T* tab(const void* p) { return static_cast<const T*>(p); }

// Products of a state value with a direction value, and of two direction values, in
// the state's type.
template <typename S, typename D> __device__ __forceinline__ S mul_sd(S a, D b) { return a * S(b); }
template <> __device__ __forceinline__ dsf mul_sd<dsf, float>(dsf a, float b) { return ds_mul(a, b); }
template <typename S, typename D> __device__ __forceinline__ S mul_dd(D a, D b) { return S(a) * S(b); }
template <> __device__ __forceinline__ dsf mul_dd<dsf, float>(float a, float b) { return ds_mul(a, b); }
// Re(conj(a) b)
template <typename S, typename CS, typename CD> __device__ __forceinline__ S dot_sd(CS a, CD b) {
  return mul_sd<S>(a.x, b.x) + mul_sd<S>(a.y, b.y);
}

// Parseval's sums over this thread's modes (k = xi[t + q Tl]): kinetic akin = sum k^2 / 2
// |v|^2 and rotation arot = r sum k |v|^2.  FP64 and double-single take the factors out
// of the loop (4 of 8 operations a mode); in single precision, where the operations are
// cheap, each mode's symbol is rounded by itself: a field of few modes shows the rounding
// in the sum (2.7e-7 of an energy between the two forms).
template <int E, typename T, typename C>
__device__ __forceinline__ void symbol_sums(const C (&v)[E], const T* __restrict__ xi, int t, int Tl, T r, T& akin, T& arot) {
  akin = T(0);
  arot = T(0);
  if constexpr (std::is_same<T, float>::value) {
#pragma unroll
    for (int q = 0; q < E; ++q) {
      const T k = xi[t + q * Tl];
      const T mk = T(0.5) * k * k, kr = r * k;
      const T a2 = v[q].x * v[q].x + v[q].y * v[q].y;
      akin += mk * a2; arot += kr * a2;
    }
  } else {
#pragma unroll
    for (int q = 0; q < E; ++q) {
      const T k = xi[t + q * Tl], ka = k * (v[q].x * v[q].x + v[q].y * v[q].y);
      arot += ka;
      akin += k * ka;
    }
    akin = T(0.5) * akin;
    arot = r * arot;
  }
}
// v *= k (h k + c): the symbol (1/2 k^2 + r k) / M with h = 1/(2M), c = r / M.
template <int E, typename T, typename C>
__device__ __forceinline__ void apply_symbol(C (&v)[E], const T* __restrict__ xi, int t, int Tl, T h, T c) {
#pragma unroll
  for (int q = 0; q < E; ++q) {
    const T k = xi[t + q * Tl];
    v[q] = cscale(v[q], k * (h * k + c));
  }
}

// ---------------------------------------------------------------------------
// Contiguous (x) passes.  Block = lpb lines x Tl threads; tid = t + Tl*l.
//
// Three element types: TF for the line transform, TS for the state fields
// (phi, H phi, r_{n-1}, V) and TD for the direction fields (P_C workspace s,
// P r, p).  TF = TS = TD gives the plain complex64 or complex128 passes; the
// refinement passes use TS = double with TF = TD = float for the direction
// (P_C r and the moments of A p), and TF = TS = double, TD = float for H phi.
// ---------------------------------------------------------------------------
// Max threads per block: 512 with single-precision transforms, 256 with double.
template <typename T> struct MaxThreads { static constexpr int value = sizeof(T) == 8 ? 256 : 512; };
// Roles whose passes take part in programmatic dependent launch: those of the combined
// preconditioner.  In the H passes the two instructions cost registers (FP64 x pass at
// M = 128 from 128 to 158, one block per SM where two fit: H phi on 128^3 complex128 545
// us instead of 522, energy and gradient on 512^2 469 instead of 452), so they stay out.
template <int ROLE> constexpr bool kEarlyRole = ROLE == P_C1 || ROLE == P_C3 || ROLE == P_CFWD || ROLE == P_CCORE || ROLE == P_CINV;

// Blocks per SM that the compiler must leave room for (0: as it likes; 1 would already
// change what it takes): two in the FP64 H passes of 8 values per thread (256 threads).
// Left alone it takes up to 158 registers, one block per SM, where two blocks with 64 to
// 100 bytes of spills are faster: H phi on 256 x 256 x 32 complex128 570 -> 539 us, on
// 64 x 256 x 128 567 -> 534, on 32 x 256 x 256 574 -> 539; on 128^3 531 both ways.
template <typename TF, typename TS, int ROLE, int E> constexpr int kMinBlocks =
    (std::is_same<TF, double>::value && std::is_same<TS, double>::value && (ROLE == P_HX || ROLE == P_HMID) && E == 8) ? 2 : 0;

__device__ __forceinline__ void prefetch_l2(const void* p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); }

template <typename To, typename From>
__device__ __forceinline__ cplx<To> cconv(From v) { return cmk<cplx<To>>((To)v.x, (To)v.y); }

// One unit of a contiguous pass: lines unit*lpb .. unit*lpb + lpb - 1 (the
// block has lpb * M/8 threads).  Adds this thread's reduction terms to acc[]
// (Moments<ROLE>: sums, or maxima for the slots flagged in MAX).
// RES: a resident solve (fields in shared memory): operands are taken as they are
// used, since nothing is gained by having them in flight early.
template <typename TF, typename TS, typename TD, int M, int ROLE, int EV = 8, bool RES = false>
__device__ __forceinline__ void xunit(const PassArgs& a, const Scal& S, long long unit, unsigned char* smraw,
                                      Acc* acc) {
  using CF = cplx<TF>;
  using CS = cplx<TS>;
  using CD = cplx<TD>;
  constexpr int E = LineCfg<M, EV>::E, Tl = LineCfg<M, EV>::Tl;
  constexpr int LS = M + M / 16;  // padded line stride in shared memory
  // lines of at most 32 threads lie inside one warp (tid = t + Tl l) and own
  // their shared-memory rows: their transforms need only warp barriers
  constexpr bool W = Tl <= 32;
  CF* sm = reinterpret_cast<CF*>(smraw);

  const int t = threadIdx.x % Tl, l = threadIdx.x / Tl;
  const long long line = unit * a.lpb + l;
  const long long base = line * M;
  const int iy = (int)((a.row0 + line) % a.ny);  // row0: global row of local line 0 (cluster slices)
  const CF* __restrict__ tw = static_cast<const CF*>(a.tw);
  const TF* __restrict__ xi = tab<TF>(a.xi[0]);
  const TS* __restrict__ V = tab<TS>(a.V);
  auto si = [l](int pos) { return l * LS + pos + (pos >> 4); };
  const TF invM = TF(1) / TF(M);

  CF v[E];
  if constexpr (ROLE == P_HX) {
    // ---- H_phi f, x part, plus the real-space terms (TF == TS) --------------------
    static_assert(sizeof(TF) == sizeof(TS), "H passes transform the state precision");
    const CS* __restrict__ phi = static_cast<const CS*>(a.phi);
    const CS* __restrict__ f = static_cast<const CS*>(a.f ? a.f : a.phi);
    if (a.pf > 0 && unit + a.pf < a.nblocks) {
      // fields larger than L2: the block about one wave later reads the rows of
      // unit + pf; start bringing them (phi, f, V) into L2 now, 128-byte lines
      const long long e0 = (unit + a.pf) * a.lpb * M;
      const int nb = a.lpb * M * (int)sizeof(CS);
      for (int off = threadIdx.x * 128; off < nb; off += blockDim.x * 128) {
        prefetch_l2(reinterpret_cast<const char*>(phi + e0) + off);
        if (a.f && a.f != a.phi) prefetch_l2(reinterpret_cast<const char*>(f + e0) + off);
      }
      const int nv = a.lpb * M * (int)sizeof(TS);
      for (int off = threadIdx.x * 128; off < nv; off += blockDim.x * 128)
        prefetch_l2(reinterpret_cast<const char*>(V + e0) + off);
    }
    CS ph[E];
    TS vv[E];
    const bool retract = S.retract;
    const CD* __restrict__ p = static_cast<const CD*>(a.p);
    CS* __restrict__ phi_out = static_cast<CS*>(a.phi_out);
    // ONE: the second field -- p in a solve, the operand f of an API call -- has the state's
    // type and comes through one pointer into v, all loads of the block in flight together.
    // A choice per element put f behind phi: 0.5 to 1 us of L2 latency in H phi with f != phi
    // (device time on 512^2 complex64 10.4 -> 8.9 us, 64 x 128 6.8 -> 4.8).  Complex64 passes
    // keep the operand over the transforms (512^2: 9.3 with f read again behind them); FP64
    // passes, short of registers, read it again.
    constexpr bool ONE = std::is_same<TS, TD>::value && !RES, KEEP = ONE && std::is_same<TS, float>::value;
    CD pq[ONE && !KEEP ? 1 : E];  // p of a refinement; the operand kept
    if constexpr (RES) {
      const TS cc = num_as<TS>(S.cc), ss = num_as<TS>(S.ss);
#pragma unroll
      for (int q = 0; q < E; ++q) {
        const long long g = base + t + q * Tl;
        CS x = phi[g];
        if (retract) {
          const CS d = cconv<TS>(p[g]);
          x = cmk<CS>(cc * x.x + ss * d.x, cc * x.y + ss * d.y);
          phi_out[g] = x;
        }
        ph[q] = x;
        vv[q] = V[g];
        v[q] = cconv<TF>(x);
      }
    } else if constexpr (ONE) {
      const CS* __restrict__ second = a.solver ? p : f;
#pragma unroll
      for (int q = 0; q < E; ++q) {
        const long long g = base + t + q * Tl;
        v[q] = second[g];
        ph[q] = phi[g];
        vv[q] = V[g];
        if constexpr (KEEP) pq[q] = v[q];
      }
    } else {  // the refinement's state: inside a solve only
#pragma unroll
      for (int q = 0; q < E; ++q) {
        const long long g = base + t + q * Tl;
        ph[q] = phi[g];
        vv[q] = V[g];
        pq[q] = p[g];
      }
    }
    if (!RES && a.solver) {
      if (S.done) return;
      const TS cc = num_as<TS>(S.cc), ss = num_as<TS>(S.ss);
#pragma unroll
      for (int q = 0; q < E; ++q) {
        if (retract) {
          CD d;
          if constexpr (ONE) d = v[q];
          else d = pq[q];
          ph[q] = cmk<CS>(cc * ph[q].x + mul_sd<TS>(ss, d.x), cc * ph[q].y + mul_sd<TS>(ss, d.y));
          phi_out[base + t + q * Tl] = ph[q];
        }
        v[q] = cconv<TF>(ph[q]);
      }
    }
    line_dft<M, E, -1, W>(v, sm, si, t, tw);
    const TF y = tab<TF>(a.xc[1])[iy];
    if (!a.nomoments) {  // uniform; the rotation symbol without omega (applied in finalize_H)
      TF akin, arot;
      symbol_sums<E>(v, xi, t, Tl, y, akin, arot);
      acc[0] = acc_add(acc[0], acc_from(akin * invM));
      acc[1] = acc_add(acc[1], acc_from(arot * invM));
    }
    if (!a.eonly) {  // uniform
      apply_symbol<E>(v, xi, t, Tl, TF(0.5) * invM, num_as<TF>(a.omega_n) * y * invM);
      line_dft<M, E, +1, W>(v, sm, si, t, tw);
      CS* __restrict__ tout = static_cast<CS*>(a.t);
      const TS eta = num_as<TS>(a.eta_n);
#pragma unroll
      for (int q = 0; q < E; ++q) {
        const long long g = base + t + q * Tl;
        const TS u = ph[q].x * ph[q].x + ph[q].y * ph[q].y;
        const TS m = vv[q] + eta * u;
        CS fq = ph[q];
        if (!a.solver) {
          if constexpr (KEEP) fq = pq[q];
          else if (a.f) fq = f[g];
        }
        tout[g] = cmk<CS>(TS(v[q].x) + m * fq.x, TS(v[q].y) + m * fq.y);
      }
    }
    if (!a.nomoments) {
      TS apot = 0, au2 = 0, an2 = 0, umax = 0;
#pragma unroll
      for (int q = 0; q < E; ++q) {
        const TS u = ph[q].x * ph[q].x + ph[q].y * ph[q].y;
        apot += vv[q] * u; au2 += u * u; an2 += u;
        if constexpr (sizeof(TS) == 4) umax = fmax(umax, u);  // read by the complex64 phase's switch rule only
      }
      acc[2] = acc_add(acc[2], acc_from(apot));
      acc[3] = acc_add(acc[3], acc_from(au2));
      acc[4] = acc_add(acc[4], acc_from(an2));
      acc[5] = acc_max(acc[5], acc_from(umax));
    }
  } else if constexpr (ROLE == P_C1) {
    // ---- s = FFT_x[P_V^{1/2} r], r = H phi - lambda phi (solver) or r_in (API) ----
    const CS* __restrict__ phi = after_wait(static_cast<const CS*>(a.phi));
    const CS* __restrict__ rin = after_wait(static_cast<const CS*>(a.solver ? a.t : a.r_in));
    const TS lam = num_as<TS>(S.lam);
    const TS alpha = num_as<TS>(S.alpha);
    const TS eta = num_as<TS>(a.eta_n);
    TS rmax = 0, r2 = 0;
    float bad = 0.0f;
    const int pre = pc_pre(S.pc);
    const bool uses_pv = pre != 0 || pc_post(S.pc) != 0;
#pragma unroll
    for (int q = 0; q < E; ++q) {
      const long long g = base + t + q * Tl;
      const CS ph = phi[g];
      CS r = rin[g];
      if (a.solver) r = cmk<CS>(r.x - lam * ph.x, r.y - lam * ph.y);
      const TS den = alpha + V[g] + eta * (ph.x * ph.x + ph.y * ph.y);
      bad += (den > TS(0) || !uses_pv) ? 0.0f : 1.0f;
      const TS a2 = r.x * r.x + r.y * r.y;
      rmax = fmax(rmax, a2); r2 += a2;
      v[q] = cconv<TF>(cscale(r, pv_factor(den, pre)));
    }
    if (S.done) return;
    line_dft<M, E, -1, W>(v, sm, si, t, tw);
    CD* __restrict__ sout = static_cast<CD*>(a.s);
#pragma unroll
    for (int q = 0; q < E; ++q) sout[base + t + q * Tl] = cconv<TD>(v[q]);
    acc[0] = acc_max(acc[0], acc_from(rmax));
    acc[1] = acc_add(acc[1], acc_from(r2));
    acc[2] = acc_add(acc[2], acc_from(bad));
  } else if constexpr (ROLE == P_C3) {
    // ---- Pr = P_V^{1/2} IFFT_x[s] (the 1/N is applied in the core pass) ----
    const CS* __restrict__ phi = after_wait(static_cast<const CS*>(a.phi));
    CD* __restrict__ sbuf = after_wait(static_cast<CD*>(a.s));
#pragma unroll
    for (int q = 0; q < E; ++q) v[q] = cconv<TF>(sbuf[base + t + q * Tl]);
    const TS alpha = num_as<TS>(S.alpha);
    const TS eta = num_as<TS>(a.eta_n);
    if (!a.solver) {
      TS den[E];  // loaded before the transform, which hides the latency
#pragma unroll
      for (int q = 0; q < E; ++q) {
        const long long g = base + t + q * Tl;
        const CS ph = phi[g];
        den[q] = alpha + V[g] + eta * (ph.x * ph.x + ph.y * ph.y);
      }
      line_dft<M, E, +1, W>(v, sm, si, t, tw);
      CD* __restrict__ out = static_cast<CD*>(a.out);
#pragma unroll
      for (int q = 0; q < E; ++q)
        out[base + t + q * Tl] = cconv<TD>(cscale(cconv<TS>(v[q]), pv_factor(den[q], pc_post(S.pc))));
      return;
    }
    // every operand of the epilogue is loaded before the transform, so the
    // loads overlap it instead of waiting behind its barriers
    const CS* __restrict__ Hphi = static_cast<const CS*>(a.t);
    CS* __restrict__ rprev = static_cast<CS*>(a.r_prev);
    const CD* __restrict__ pprev = static_cast<const CD*>(a.p);
    CS ph[E], hq[E], ro[E];
    CD pp[E];
    TS vv[E];
#pragma unroll
    for (int q = 0; q < E; ++q) {
      const long long g = base + t + q * Tl;
      ph[q] = phi[g];
      hq[q] = Hphi[g];
      ro[q] = rprev[g];
      pp[q] = pprev[g];
      vv[q] = V[g];
    }
    if (S.done) return;
    line_dft<M, E, +1, W>(v, sm, si, t, tw);
    const TS lam = num_as<TS>(S.lam);
    const int post = pc_post(S.pc);
    TS a0 = 0, a1 = 0, a2 = 0, a3 = 0, a4 = 0, a5 = 0;
#pragma unroll
    for (int q = 0; q < E; ++q) {
      const long long g = base + t + q * Tl;
      const TS den = alpha + vv[q] + eta * (ph[q].x * ph[q].x + ph[q].y * ph[q].y);
      const CD Prd = cconv<TD>(cscale(cconv<TS>(v[q]), pv_factor(den, post)));
      sbuf[g] = Prd;
      // the moments take the stored direction, as later passes see it
      const CS r = cmk<CS>(hq[q].x - lam * ph[q].x, hq[q].y - lam * ph[q].y);
      a0 += dot_sd<TS>(r, Prd);
      a1 += dot_sd<TS>(cmk<CS>(r.x - ro[q].x, r.y - ro[q].y), Prd);
      a2 += dot_sd<TS>(ph[q], Prd);
      a3 += dot_sd<TS>(ph[q], pp[q]);
      a4 += dot_sd<TS>(r, pp[q]);
      a5 += r.x * ph[q].x + r.y * ph[q].y;
      rprev[g] = r;
    }
    acc[0] = acc_add(acc[0], acc_from(a0)); acc[1] = acc_add(acc[1], acc_from(a1));
    acc[2] = acc_add(acc[2], acc_from(a2)); acc[3] = acc_add(acc[3], acc_from(a3));
    acc[4] = acc_add(acc[4], acc_from(a4)); acc[5] = acc_add(acc[5], acc_from(a5));
  } else if constexpr (ROLE == P_AX) {
    // ---- p = -Pr + beta p_prev - gamma phi ; moments for the step size ----
    const CS* __restrict__ phi = static_cast<const CS*>(a.phi);
    const CD* __restrict__ Pr = static_cast<const CD*>(a.s);
    const CS* __restrict__ Hphi = static_cast<const CS*>(a.t);
    CD* __restrict__ pbuf = static_cast<CD*>(a.p);
    const TS beta = num_as<TS>(S.beta), gamma = num_as<TS>(S.gamma);
    TS aR = 0, aV = 0, aW1 = 0, aUV = 0, aV2 = 0, aUW = 0, aVW = 0, aW2 = 0, aRho = 0;
#pragma unroll
    for (int q = 0; q < E; ++q) {
      const long long g = base + t + q * Tl;
      const CS ph = phi[g], h = Hphi[g];
      const CS pr = cconv<TS>(Pr[g]);
      const CD pp = pbuf[g];
      const CD pnd = cconv<TD>(cmk<CS>(-pr.x + mul_sd<TS>(beta, pp.x) - gamma * ph.x,
                                       -pr.y + mul_sd<TS>(beta, pp.y) - gamma * ph.y));
      v[q] = cconv<TF>(pnd);
      const TS u = ph.x * ph.x + ph.y * ph.y;
      const TS vr = dot_sd<TS>(ph, pnd);  // moments of the stored p
      const TS wq = mul_dd<TS>(pnd.x, pnd.x) + mul_dd<TS>(pnd.y, pnd.y);
      aR += dot_sd<TS>(h, pnd);
      aV += V[g] * wq;
      aW1 += wq; aUV += u * vr; aV2 += vr * vr; aUW += u * wq; aVW += vr * wq; aW2 += wq * wq; aRho += vr;
    }
    if (S.done) return;
#pragma unroll
    for (int q = 0; q < E; ++q) pbuf[base + t + q * Tl] = cconv<TD>(v[q]);
    line_dft<M, E, -1, W>(v, sm, si, t, tw);
    const TF y = tab<TF>(a.xc[1])[iy];
    const TF oy = num_as<TF>(a.omega_n) * y;
    TF akr = 0;
#pragma unroll
    for (int q = 0; q < E; ++q) {
      const TF k = xi[t + q * Tl];
      akr += k * (TF(0.5) * k + oy) * (v[q].x * v[q].x + v[q].y * v[q].y);
    }
    acc[0] = acc_add(acc[0], acc_from(aR));
    acc[1] = acc_add(acc_add(acc[1], acc_from(aV)), acc_from(akr * invM));
    acc[2] = acc_add(acc[2], acc_from(aW1)); acc[3] = acc_add(acc[3], acc_from(aUV));
    acc[4] = acc_add(acc[4], acc_from(aV2)); acc[5] = acc_add(acc[5], acc_from(aUW));
    acc[6] = acc_add(acc[6], acc_from(aVW)); acc[7] = acc_add(acc[7], acc_from(aW2));
    acc[8] = acc_add(acc[8], acc_from(aRho));
  }
}

// ---------------------------------------------------------------------------
// Strided (y, z) passes.  Block = tx columns x Tl threads; tid = c + tx*t.
// ---------------------------------------------------------------------------
// One unit of a strided pass: the tile of tx adjacent x-columns number unit
// (block = tx * M/8 threads).  Reduction terms are added to acc[].
template <typename T, int M, int ROLE, int EV = 8>
__device__ __forceinline__ void sunit(const PassArgs& a, const Scal& S, long long unit, unsigned char* smraw,
                                      Acc* acc) {
  using C = cplx<T>;
  constexpr int E = LineCfg<M, EV>::E, Tl = LineCfg<M, EV>::Tl;
  C* sm = reinterpret_cast<C*>(smraw);
  const int tx = a.tx;
  const int c = threadIdx.x % tx, t = threadIdx.x / tx;
  const int xt = (int)(unit % a.ntx);
  const long long outer = unit / a.ntx;
  const int ix = xt * tx + c;
  const long long base = outer * a.outer_stride + ix;
  const long long st = a.stride;
  const C* __restrict__ tw = static_cast<const C*>(a.tw);
  auto si = [tx, c](int pos) { return pos * tx + c; };
  const T* __restrict__ xia = tab<T>(a.xi[a.axis]);
  const T invM = T(1) / T(M);

  C v[E];
  if constexpr (ROLE == P_HMID) {
    const C* __restrict__ f = static_cast<const C*>((a.f && !a.solver) ? a.f : a.phi);
    const C* tb = static_cast<const C*>(a.t);
    C tv[E];  // the accumulated t, loaded before the transforms so the loads overlap them
#pragma unroll
    for (int q = 0; q < E; ++q) {
      v[q] = f[base + (t + q * Tl) * st];
      if (!a.eonly) tv[q] = tb[base + (t + q * Tl) * st];
    }
    if (S.done) return;
    line_dft<M, E, -1>(v, sm, si, t, tw);
    const T rx = (a.axis == 1) ? -tab<T>(a.xc[0])[ix] : T(0);  // rotation symbol -omega x mu (y); none for z
    if (!a.nomoments) {
      T akin, arot;
      symbol_sums<E>(v, xia, t, Tl, rx, akin, arot);
      acc[0] = acc_add(acc[0], acc_from(akin * invM));
      acc[1] = acc_add(acc[1], acc_from(arot * invM));
    }
    if (a.eonly) return;  // uniform
    apply_symbol<E>(v, xia, t, Tl, T(0.5) * invM, num_as<T>(a.omega_n) * rx * invM);
    line_dft<M, E, +1>(v, sm, si, t, tw);
    C* __restrict__ dst = static_cast<C*>(a.out ? a.out : a.t);  // API: final pass writes the caller's buffer
#pragma unroll
    for (int q = 0; q < E; ++q) dst[base + (t + q * Tl) * st] = cadd(tv[q], v[q]);
  } else if constexpr (ROLE == P_CFWD || ROLE == P_CINV || ROLE == P_CCORE) {
    C* __restrict__ sb = after_wait(static_cast<C*>(a.s));
#pragma unroll
    for (int q = 0; q < E; ++q) v[q] = sb[base + (t + q * Tl) * st];
    if (S.done) return;
    if constexpr (ROLE == P_CINV) {
      line_dft<M, E, +1>(v, sm, si, t, tw);
    } else {
      line_dft<M, E, -1>(v, sm, si, t, tw);
    }
    if constexpr (ROLE == P_CCORE) {
      // (alpha + |k|^2 / 2)^{-1} / N on the full frequency grid (eq. PDelta)
      const T alpha = num_as<T>(S.alpha);
      const T invN = num_as<T>(a.invN);
      const T kx = tab<T>(a.xi[0])[ix];
      T kother = 0;
      if (a.dim == 3) {
        // axis == 2 (z) here; y index is the outer index
        const T ky = tab<T>(a.xi[1])[outer];
        kother = ky * ky;
      }
      const bool core = pc_core(S.pc);
#pragma unroll
      for (int q = 0; q < E; ++q) {
        const T k = xia[t + q * Tl];
        const T den = alpha + T(0.5) * (kx * kx + kother + k * k);
        v[q] = cscale(v[q], core ? over(invN, den) : invN);
      }
      line_dft<M, E, +1>(v, sm, si, t, tw);
    }
#pragma unroll
    for (int q = 0; q < E; ++q) sb[base + (t + q * Tl) * st] = v[q];
  } else if constexpr (ROLE == P_AMID) {
    const C* __restrict__ pb = static_cast<const C*>(a.p);
#pragma unroll
    for (int q = 0; q < E; ++q) v[q] = pb[base + (t + q * Tl) * st];
    if (S.done) return;
    line_dft<M, E, -1>(v, sm, si, t, tw);
    const T om = num_as<T>(a.omega_n);
    const T x = (a.axis == 1) ? tab<T>(a.xc[0])[ix] : T(0);
    const T rs = (a.axis == 1) ? -om * x : T(0);
    T akr = 0;
#pragma unroll
    for (int q = 0; q < E; ++q) {
      const T k = xia[t + q * Tl];
      akr += k * (T(0.5) * k + rs) * (v[q].x * v[q].x + v[q].y * v[q].y);
    }
    acc[0] = acc_add(acc[0], acc_from(akr * invM));
  }
}


// ---------------------------------------------------------------------------
// Standalone pass kernels (one unit per block): used by the API entry points,
// the graph-captured solve and the host-loop solve.
//
// Reductions: every block stores its partials in the region of its pass.  The
// x and y passes of H phi and A p stop there (kernel order makes the partials
// visible to the operator's last pass); the passes that end an operator, and
// C1 and C3, count their blocks with a ticket, and the last block to arrive
// sums every region of the operator in a fixed order and runs the scalar step
// on a copy of the control block in shared memory: read once, written back
// once, instead of a memory round trip per scalar.  Passes look at `done` only
// once their operands are in flight.  With the shorter scalar steps, the scalars
// split once (Num), the short sums above and four values per thread, an iteration of
// the graph loop went from 121 to 74 us (256^2, refinement) and from 585 to 445 us
// (128^3, refinement).
// ---------------------------------------------------------------------------
// All the sums of ROLE's operator, in the order its scalar step reads them: those of
// the x pass, then of each further axis (KM per axis).
template <int ROLE> struct OpSums { static constexpr int KX = Moments<ROLE>::K, KM = 0; };
template <> struct OpSums<P_HMID> { static constexpr int KX = Moments<P_HX>::K, KM = Moments<P_HMID>::K; };
template <> struct OpSums<P_AMID> { static constexpr int KX = Moments<P_AX>::K, KM = Moments<P_AMID>::K; };
template <int ROLE> struct OpMasks {
  static constexpr int KX = OpSums<ROLE>::KX, KM = OpSums<ROLE>::KM, K = KX + 2 * KM;
  static constexpr unsigned WX = ROLE == P_HMID ? Moments<P_HX>::W : ROLE == P_AMID ? Moments<P_AX>::W : Moments<ROLE>::W;
  static constexpr unsigned MAX =
      ROLE == P_HMID ? Moments<P_HX>::MAX : ROLE == P_AMID ? Moments<P_AX>::MAX : Moments<ROLE>::MAX;
  static constexpr unsigned W = WX | (((1u << (2 * KM)) - 1u) << KX);
};

// The scalar step of ROLE's operator, by warp 0 of the last block.
template <int ROLE>
__device__ __forceinline__ void run_scalar_step(const PassArgs& a, Ctl* c, const double* tot) {
  const Fin F = fin_of(a);
  constexpr int KX = OpSums<ROLE>::KX, KM = OpSums<ROLE>::KM;
  if constexpr (ROLE == P_HMID) finalize_H(c, F, tot, tot + KX, tot + KX + KM, true);
  else if constexpr (ROLE == P_C1) finalize_C1(c, tot, true);
  else if constexpr (ROLE == P_C3) finalize_C3(c, tot, true);
  else if constexpr (ROLE == P_AMID) finalize_A(c, F, tot, tot[KX], tot[KX + KM], true);
}

template <int ROLE>
__device__ __forceinline__ void reduce_and_finish(const PassArgs& a, const Acc* acc) {
  constexpr int K = Moments<ROLE>::K;
  if (a.nomoments) return;  // uniform over the launch
  if constexpr (K > 0) {
    constexpr bool xpart = ROLE == P_HX || ROLE == P_AX, mid = ROLE == P_HMID || ROLE == P_AMID;
    // the P_C passes reduce only inside a solve
    if ((ROLE == P_C1 || ROLE == P_C3) && !a.solver) return;
    __shared__ Acc red_sm[kRedSlots];
    Acc v[K];
#pragma unroll
    for (int k = 0; k < K; ++k) v[k] = acc[k];
    const int reg = (xpart || mid) ? a.axis : 0;
    Acc* part = acc_slots(a.partials);
    Acc* mine = part + reg * a.region + (size_t)blockIdx.x * kMaxMoments;
    block_reduce<K, Moments<ROLE>::MAX>(v, red_sm, [&](int k, Acc t) { mine[k] = t; });
    if ((xpart || mid) && blockIdx.x == 0 && threadIdx.x == 0) a.nparts[reg] = (int)gridDim.x;
    if (xpart || (mid && !a.last_axis)) return;
    if constexpr (!xpart) {
      using OM = OpMasks<ROLE>;
      __shared__ double tot[OM::K];
      __shared__ int s_last;
      __shared__ Ctl sctl;
      if (threadIdx.x < 32) {  // the warp that stored the partials
        __threadfence();
        if (full_warp()) __syncwarp();
        else __syncwarp((1u << blockDim.x) - 1u);
        if (threadIdx.x == 0) s_last = (atomicAdd(a.ticket, 1u) == gridDim.x - 1) ? 1 : 0;
      }
      __syncthreads();
      if (!s_last) return;
      __threadfence();
      constexpr int words = sizeof(Ctl) / 8;
      static_assert(sizeof(Ctl) % 8 == 0, "the control block is copied in 8-byte words");
      const unsigned long long* from = reinterpret_cast<const unsigned long long*>(a.ctl);
      unsigned long long* cp = reinterpret_cast<unsigned long long*>(&sctl);
      for (int i = threadIdx.x; i < words; i += blockDim.x) cp[i] = __ldcg(from + i);
      auto region_of = [&](int k) { return k < OM::KX ? 0 : (k < OM::KX + OM::KM ? 1 : 2); };
      auto src = [&](int k) {
        const int r = region_of(k);
        return part + r * a.region + (r == 0 ? k : (k - OM::KX) % (OM::KM ? OM::KM : 1));
      };
      auto nb = [&](int k) {
        const int r = region_of(k);
        if (mid && r != a.axis) return r < a.dim ? __ldcg(a.nparts + r) : 0;
        return (int)gridDim.x;
      };
      sum_partials<OM::K, OM::MAX>(src, nb, red_sm, [&](int k, Acc t) { tot[k] = total<OM::W>(t, a.weight, k); });
      __syncthreads();  // totals and the control block copy
      if (threadIdx.x < (full_warp() ? 32 : 1)) {
        run_scalar_step<ROLE>(a, &sctl, tot);
        if (threadIdx.x == 0) {
          *a.ticket = 0u;  // ready for the next pass
          if (ROLE == P_AMID) set_loop_condition(a, sctl.done ? 0 : 1);
        }
      }
      __syncthreads();
      unsigned long long* to = reinterpret_cast<unsigned long long*>(a.ctl);
      for (int i = threadIdx.x; i < words; i += blockDim.x) to[i] = cp[i];
    }
  }
}

template <typename TF, typename TS, typename TD, int M, int ROLE, int EV>
__global__ void __launch_bounds__(MaxThreads<TF>::value < MaxThreads<TS>::value ? MaxThreads<TF>::value : MaxThreads<TS>::value,
                                  kMinBlocks<TF, TS, ROLE, EV>) pass_x(PassArgs a) {
  extern __shared__ __align__(16) unsigned char smraw[];
  if constexpr (kEarlyRole<ROLE>) pdl_wait();
  const Scal S = scal_of(a.ctl, a);
  Acc acc[kMaxMoments];
#pragma unroll
  for (int k = 0; k < kMaxMoments; ++k) acc[k] = Acc{0.0f, 0.0f};
  xunit<TF, TS, TD, M, ROLE, EV>(a, S, blockIdx.x, smraw, acc);
  if constexpr (kEarlyRole<ROLE>) pdl_trigger();
  if (S.done) return;
  reduce_and_finish<ROLE>(a, acc);
}

template <typename T, int M, int ROLE, int EV>
__global__ void __launch_bounds__(MaxThreads<T>::value, kMinBlocks<T, T, ROLE, EV>) pass_s(PassArgs a) {
  extern __shared__ __align__(16) unsigned char smraw[];
  if constexpr (kEarlyRole<ROLE>) pdl_wait();
  const Scal S = scal_of(a.ctl, a);
  Acc acc[kMaxMoments];
#pragma unroll
  for (int k = 0; k < kMaxMoments; ++k) acc[k] = Acc{0.0f, 0.0f};
  sunit<T, M, ROLE, EV>(a, S, blockIdx.x, smraw, acc);
  if constexpr (kEarlyRole<ROLE>) pdl_trigger();
  if (S.done) {
    if (ROLE == P_AMID && a.last_axis && blockIdx.x == 0 && threadIdx.x == 0) set_loop_condition(a, 0);
    return;
  }
  reduce_and_finish<ROLE>(a, acc);
}

// ---------------------------------------------------------------------------
// Host-side dispatch over M
// ---------------------------------------------------------------------------
// Precision modes of a launch: 0 complex64, 1 complex128, 2 refinement split:
// the state (phi, H phi, r_{n-1}, V) and the H phi transforms in double-single
// (dsf, ~48 bits on the FP32 pipe), the direction (P_C workspace, p) in FP32.
template <int MODE, int ROLE> struct ModeTypes;
template <int ROLE> struct ModeTypes<0, ROLE> { using TF = float; using TS = float; using TD = float; };
template <int ROLE> struct ModeTypes<1, ROLE> { using TF = double; using TS = double; using TD = double; };
template <int ROLE> struct ModeTypes<2, ROLE> {
  static constexpr bool h = (ROLE == P_HX || ROLE == P_HMID);
  static constexpr bool state = (ROLE == P_C1 || ROLE == P_C3 || ROLE == P_AX);
  using TF = typename std::conditional<h, dsf, float>::type;
  using TS = typename std::conditional<h || state, dsf, float>::type;
  using TD = float;
};

template <int MODE, int M, int ROLE, int EV>
cudaError_t launch_one(const PassArgs& a, cudaStream_t st) {
  using MT = ModeTypes<MODE, ROLE>;
  using TF = typename MT::TF;
  using C = cplx<TF>;
  constexpr int Tl = LineCfg<M, EV>::Tl;
  constexpr bool contig = (ROLE == P_HX || ROLE == P_C1 || ROLE == P_C3 || ROLE == P_AX);
  int threads, smem;
  if constexpr (contig) {
    threads = Tl * a.lpb;
    smem = a.lpb * (M + M / 16) * (int)sizeof(C);
  } else {
    threads = Tl * a.tx;
    smem = M * a.tx * (int)sizeof(C);
  }
  void (*kern)(PassArgs);
  if constexpr (contig) kern = pass_x<TF, typename MT::TS, typename MT::TD, M, ROLE, EV>;
  else kern = pass_s<TF, M, ROLE, EV>;
  static DeviceOnce attr;
  const int dev = DeviceOnce::device();
  if (!attr.done(dev)) {
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
    if (e != cudaSuccess) return e;
    attr.set(dev);
  }
  return launch_early(kEarlyRole<ROLE> && a.early && !a.solver, kern, a.nblocks, threads, smem, st, a);
}

// E = 8 for every M; E = 4 (plans chosen by the tuner) for M >= 32, in
// their own translation units (gpe_k_e4_*.cu).
template <int MODE, int ROLE, int EV = 8>
cudaError_t launch_role(const PassArgs& a, cudaStream_t st) {
  if constexpr (EV == 8) {
    switch (a.M) {
      case 8: return launch_one<MODE, 8, ROLE, 8>(a, st);
      case 16: return launch_one<MODE, 16, ROLE, 8>(a, st);
      case 32: return launch_one<MODE, 32, ROLE, 8>(a, st);
      case 64: return launch_one<MODE, 64, ROLE, 8>(a, st);
      case 128: return launch_one<MODE, 128, ROLE, 8>(a, st);
      case 256: return launch_one<MODE, 256, ROLE, 8>(a, st);
      case 512: return launch_one<MODE, 512, ROLE, 8>(a, st);
      default: return cudaErrorInvalidValue;
    }
  } else {
    switch (a.M) {
      case 32: return launch_one<MODE, 32, ROLE, EV>(a, st);
      case 64: return launch_one<MODE, 64, ROLE, EV>(a, st);
      case 128: return launch_one<MODE, 128, ROLE, EV>(a, st);
      case 256: return launch_one<MODE, 256, ROLE, EV>(a, st);
      case 512: return launch_one<MODE, 512, ROLE, EV>(a, st);
      default: return cudaErrorInvalidValue;
    }
  }
}

}  // namespace gpe
