// gpe_misc.cu -- pass dispatch and the small elementwise kernels around a
// solve (precision conversion, initial normalisation).
#include "gpe_internal.h"
#include "gpe_ds.cuh"

namespace gpe {

static cudaError_t launch_pass_f32(Pass pass, const PassArgs& a, cudaStream_t st) {
  switch (pass) {
    case P_HX: case P_HMID: return launch_group_f32_h(pass, a, st);
    case P_AX: case P_AMID: return launch_group_f32_a(pass, a, st);
    default: return launch_group_f32_c(pass, a, st);
  }
}

static cudaError_t launch_pass_f64(Pass pass, const PassArgs& a, cudaStream_t st) {
  switch (pass) {
    case P_HX: case P_HMID: return launch_group_f64_h(pass, a, st);
    case P_AX: case P_AMID: return launch_group_f64_a(pass, a, st);
    default: return launch_group_f64_c(pass, a, st);
  }
}

static cudaError_t launch_pass_f32_e4(Pass pass, const PassArgs& a, cudaStream_t st) {
  switch (pass) {
    case P_HX: case P_HMID: return launch_group_f32_h_e4(pass, a, st);
    case P_AX: case P_AMID: return launch_group_f32_a_e4(pass, a, st);
    default: return launch_group_f32_c_e4(pass, a, st);
  }
}

static cudaError_t launch_pass_e4(int mode, Pass pass, const PassArgs& a, cudaStream_t st) {
  if (mode == 0) return launch_pass_f32_e4(pass, a, st);
  if (mode == 1) {
    switch (pass) {
      case P_HX: case P_HMID: return launch_group_f64_h_e4(pass, a, st);
      case P_AX: case P_AMID: return launch_group_f64_a_e4(pass, a, st);
      default: return launch_group_f64_c_e4(pass, a, st);
    }
  }
  switch (pass) {
    case P_HX: case P_HMID: case P_C1: case P_C3: case P_AX: return launch_group_split_e4(pass, a, st);
    default: return launch_pass_f32_e4(pass, a, st);
  }
}

cudaError_t launch_pass(int mode, Pass pass, const PassArgs& a, cudaStream_t st) {
  if (a.E == 4) return launch_pass_e4(mode, pass, a, st);
  // complex64 passes through the TMA pipelines where the plan and the fields allow:
  // the x passes (H phi; in a solve also C1, C3 and AX) and every strided pass (also
  // the single-precision strided passes of the refinement phase, mode 2)
  const bool strided = pass == P_HMID || pass == P_CFWD || pass == P_CCORE || pass == P_CINV || pass == P_AMID;
  const bool xc = pass == P_C1 || pass == P_C3 || pass == P_AX;
  if ((mode == 0 && (strided || pass == P_HX || xc)) || (mode == 2 && strided && pass != P_HMID)) {
    bool used = false;
    const cudaError_t e = pass == P_HX ? launch_hx_bulk(a, st, &used)
                          : xc        ? launch_xc_bulk(pass, a, st, &used)
                                      : launch_strided_tma(pass, a, st, &used);
    if (e != cudaSuccess || used) return e;
  }
  if (mode == 0) return launch_pass_f32(pass, a, st);
  if (mode == 1) return launch_pass_f64(pass, a, st);
  // refinement split: H phi and the state in double-single, the strided
  // direction passes are plain complex64.
  switch (pass) {
    case P_HX: case P_HMID: case P_C1: case P_C3: case P_AX: return launch_group_split(pass, a, st);
    default: return launch_pass_f32(pass, a, st);
  }
}

__global__ void k_c128_to_c64(const double2* __restrict__ s, float2* __restrict__ d, long long n) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const double2 v = s[i];
    d[i] = make_float2((float)v.x, (float)v.y);
  }
}
__global__ void k_c64_to_c128(const float2* __restrict__ s, double2* __restrict__ d, long long n) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const float2 v = s[i];
    d[i] = make_double2((double)v.x, (double)v.y);
  }
}
// double-single <-> complex64 / complex128 (the refinement state)
__global__ void k_c64_to_ds(const float2* __restrict__ s, dsc* __restrict__ d, long long n) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const float2 v = s[i];
    dsc o;
    o.x = dsf(v.x);
    o.y = dsf(v.y);
    d[i] = o;
  }
}
__global__ void k_ds_to_c128(const dsc* __restrict__ s, double2* __restrict__ d, long long n) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const dsc v = s[i];
    d[i] = make_double2((double)v.x, (double)v.y);
  }
}

static int grid_for(long long n) {
  long long g = (n + 255) / 256;
  return (int)(g < 4096 ? (g > 0 ? g : 1) : 4096);
}

cudaError_t launch_convert_c128_to_c64(const void* src, void* dst, long long n, cudaStream_t st) {
  k_c128_to_c64<<<grid_for(n), 256, 0, st>>>((const double2*)src, (float2*)dst, n);
  return cudaGetLastError();
}
cudaError_t launch_convert_c64_to_c128(const void* src, void* dst, long long n, cudaStream_t st) {
  k_c64_to_c128<<<grid_for(n), 256, 0, st>>>((const float2*)src, (double2*)dst, n);
  return cudaGetLastError();
}
cudaError_t launch_convert_c64_to_ds(const void* src, void* dst, long long n, cudaStream_t st) {
  k_c64_to_ds<<<grid_for(n), 256, 0, st>>>((const float2*)src, (dsc*)dst, n);
  return cudaGetLastError();
}
cudaError_t launch_convert_ds_to_c128(const void* src, void* dst, long long n, cudaStream_t st) {
  k_ds_to_c128<<<grid_for(n), 256, 0, st>>>((const dsc*)src, (double2*)dst, n);
  return cudaGetLastError();
}
// Extremes and finiteness of V on the integer pipe: the bits of a double, negative
// ones with the magnitude inverted, order like the values.
__device__ __forceinline__ long long order_key(long long b) { return b ^ ((b >> 63) & 0x7fffffffffffffffll); }
__global__ void k_check_init(VCheck* out) {
  out->lo = 0x7fffffffffffffffll;
  out->hi = -0x7fffffffffffffffll - 1;
  out->bad = 0;
}
__global__ void __launch_bounds__(256) k_check_V(const double* __restrict__ V, long long n, VCheck* out) {
  long long lo = 0x7fffffffffffffffll, hi = -lo - 1;
  int bad = 0;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const long long b = __double_as_longlong(V[i]), k = order_key(b);
    bad |= (b & 0x7ff0000000000000ll) == 0x7ff0000000000000ll;
    lo = k < lo ? k : lo;
    hi = k > hi ? k : hi;
  }
  for (int o = 16; o > 0; o >>= 1) {
    const long long l2 = __shfl_xor_sync(0xffffffffu, lo, o), h2 = __shfl_xor_sync(0xffffffffu, hi, o);
    lo = l2 < lo ? l2 : lo;
    hi = h2 > hi ? h2 : hi;
  }
  bad = __any_sync(0xffffffffu, bad);
  if ((threadIdx.x & 31) == 0) {
    atomicMin(&out->lo, lo);
    atomicMax(&out->hi, hi);
    if (bad) atomicOr(&out->bad, 1);
  }
}
cudaError_t launch_check_V(const double* V, long long n, VCheck* out, cudaStream_t st) {
  k_check_init<<<1, 1, 0, st>>>(out);
  const int g = grid_for(n);
  k_check_V<<<g < 608 ? g : 608, 256, 0, st>>>(V, n, out);
  return cudaGetLastError();
}
__global__ void k_take_V(const double* __restrict__ V, long long n, const VCheck* __restrict__ check,
                         double* __restrict__ v64, float* __restrict__ v32, dsf* __restrict__ vds) {
  if (check->bad) return;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const double v = V[i];
    if (v64) v64[i] = v;
    if (v32) v32[i] = (float)v;
    if (vds) vds[i] = dsf(v);
  }
}
cudaError_t launch_take_V(const double* V, long long n, const VCheck* check, double* v64, float* v32, void* vds,
                          cudaStream_t st) {
  k_take_V<<<grid_for(n), 256, 0, st>>>(V, n, check, v64, v32, (dsf*)vds);
  return cudaGetLastError();
}

// One step towards the Thomas-Fermi chemical potential (eq. TF_App with mu
// fixed by the normalisation ||phi^TF|| = 1): the root of S(mu) = 1 with
// S(mu) = h^d sum max(mu - V, 0) / eta, which is convex, increasing and
// piecewise linear with slope h^d #{V < mu} / eta.  One sweep over V evaluates
// S and the slope at x; the last block to finish shrinks the bracket [lo, hi]
// (S(lo) < 1 <= S(hi)) and takes the next Newton iterate.  From the right of the
// root those iterates fall monotonically onto it (convexity): about 8 sweeps
// for a harmonic trap instead of the ~55 halvings that a bracket of doubles
// needs.  An iterate outside the bracket, or a step more than 3/4 of the one
// before it, is replaced by the bracket's midpoint, so the search also halves.
//
// A sweep is bound by latency: the launch, two reductions, and FP64
// instructions, each of which holds its SM sub-partition's FP64 pipe for 64
// cycles per warp.  Hence blocks of one warp per sub-partition, two FP64
// operations per value (difference and sum; the sign test and the count are
// integer) and one division in the scalar step.  At 256^2 a sweep takes 5.4 us
// (7.4 us with the sums over blocks in one thread); the state on 256^2 and its
// interpolation onto 512^2 went from 1316 (120 halvings) to 161 us per call.
constexpr int kTfThreads = 128;
__device__ __forceinline__ double tf_warp_sum(double v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__global__ void __launch_bounds__(kTfThreads) k_tf_step(const double* __restrict__ V, long long n, double w_eta,
                                                       TfState* st, TfState init, int first,
                                                       double* __restrict__ partials, unsigned* ticket) {
  constexpr int NW = kTfThreads / 32;
  __shared__ double sm[NW];
  __shared__ unsigned long long smc[NW];
  __shared__ int s_last;
  pdl_wait();
  V = after_wait(V);
  const TfState S = first ? init : *st;  // *st: written by the previous launch
  if (S.done) return;
  const double x = S.x;
  double acc = 0.0;
  unsigned long long cnt = 0;
  const long long step = (long long)gridDim.x * blockDim.x;
#pragma unroll 4
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += step) {
    const double d = x - V[i];
    if (__double2hiint(d) >= 0) { acc += d; ++cnt; }  // d >= 0 (V is finite)
  }
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  auto warp_count = [](unsigned long long c) {
    for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
    return c;
  };
  auto block_sum = [&]() {  // totals in thread 0, fixed order
    acc = tf_warp_sum(acc);
    cnt = warp_count(cnt);
    if (lane == 0) { sm[warp] = acc; smc[warp] = cnt; }
    __syncthreads();
    if (threadIdx.x == 0)
      for (int w = 1; w < NW; ++w) { acc += sm[w]; cnt += smc[w]; }
  };
  pdl_trigger();
  block_sum();
  unsigned long long* pc = reinterpret_cast<unsigned long long*>(partials) + 1024;
  if (threadIdx.x == 0) {
    partials[blockIdx.x] = acc;
    pc[blockIdx.x] = cnt;
    __threadfence();
    s_last = (atomicAdd(ticket, 1u) == gridDim.x - 1) ? 1 : 0;
  }
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  acc = 0.0;
  cnt = 0;
  for (unsigned b = threadIdx.x; b < gridDim.x; b += blockDim.x) {
    acc += __ldcg(partials + b);
    cnt += __ldcg(pc + b);
  }
  __syncthreads();  // sm: the first sum's readers are done
  block_sum();
  if (threadIdx.x != 0) return;
  const double f = w_eta * acc - 1.0;  // S(x) - 1
  TfState N = S;
  if (f < 0.0) N.lo = x;
  else N.hi = x;
  double nx = cnt ? x - f / (w_eta * (double)cnt) : N.lo;
  const double mid = 0.5 * (N.lo + N.hi);
  const double dx = fabs(nx - x);
  // the root: a step that no longer moves x, or neighbouring bracket ends
  N.done = nx == x || !(mid > N.lo && mid < N.hi);
  N.dx = dx;
  if (!(nx >= N.lo && nx <= N.hi) || (!N.done && dx > 0.75 * S.dx)) {
    nx = mid;
    N.dx = 1.7976931348623157e308;  // the next Newton step starts afresh
  }
  N.x = nx;
  *st = N;
  *ticket = 0u;
}
cudaError_t launch_tf_step(const double* V, long long n, double w_eta, TfState* state, const TfState& init, bool first,
                           double* partials, unsigned* ticket, cudaStream_t st) {
  long long g = (n + 4LL * kTfThreads - 1) / (4LL * kTfThreads);
  if (g < 1) g = 1;
  if (g > 1024) g = 1024;
  return launch_early(true, k_tf_step, g, kTfThreads, 0, st, V, n, w_eta, state, init, first ? 1 : 0, partials, ticket);
}

__global__ void k_tf_fill(const double* __restrict__ V, long long n, double eta, const TfState* state,
                          double2* __restrict__ phi) {
  pdl_wait();
  V = after_wait(V);
  const double mu = state->x;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    phi[i] = make_double2(sqrt(fmax(mu - V[i], 0.0) / eta), 0.0);
}
cudaError_t launch_tf_fill(const double* V, long long n, double eta, const TfState* state, void* phi128,
                           cudaStream_t st) {
  return launch_early(true, k_tf_fill, grid_for(n), 256, 0, st, V, n, eta, state, (double2*)phi128);
}

// Epilogue of gpe_energy_grad: grad_phi <- 2 h^d H_phi phi in place (Section 2,
// nabla E = 2 H_phi phi, h^d converting to the coefficient vector) and
// grad_V = h^d |phi|^2.  Either output may be null.
template <typename C>
__global__ void k_grad_epilogue(const C* __restrict__ phi, C* __restrict__ gphi, double* __restrict__ gV, long long n,
                                double weight) {
  using R = decltype(C::x);
  const R two_w = R(2.0 * weight);
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    if (gphi) {
      const C h = gphi[i];
      C g;
      g.x = two_w * h.x;
      g.y = two_w * h.y;
      gphi[i] = g;
    }
    if (gV) {
      const C v = phi[i];
      const double re = (double)v.x, im = (double)v.y;
      gV[i] = weight * (re * re + im * im);
    }
  }
}
cudaError_t launch_grad_epilogue(int prec, const void* phi, void* gphi, double* gV, long long n, double weight,
                                 cudaStream_t st) {
  if (prec == 1)
    k_grad_epilogue<double2><<<grid_for(n), 256, 0, st>>>((const double2*)phi, (double2*)gphi, gV, n, weight);
  else
    k_grad_epilogue<float2><<<grid_for(n), 256, 0, st>>>((const float2*)phi, (float2*)gphi, gV, n, weight);
  return cudaGetLastError();
}

__device__ __forceinline__ bool phase_failed(int status) { return status == 4 || status == 5; }  // non-finite, P_V

__global__ void k_batch_between(const float2* __restrict__ s, double2* __restrict__ d128, dsc* __restrict__ dds,
                                long long n, const Ctl* __restrict__ ctl) {
  if (phase_failed(ctl->status)) return;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const float2 v = s[i];
    d128[i] = make_double2((double)v.x, (double)v.y);
    dsc w;
    w.x = dsf(v.x);
    w.y = dsf(v.y);
    dds[i] = w;
  }
}
cudaError_t launch_batch_between(const void* phi64, void* phi128, void* phids, long long n, const Ctl* ctl,
                                 cudaStream_t st) {
  k_batch_between<<<grid_for(n), 256, 0, st>>>((const float2*)phi64, (double2*)phi128, (dsc*)phids, n, ctl);
  return cudaGetLastError();
}

__global__ void k_batch_gate(Ctl* ctl, cudaGraphConditionalHandle cond) {
  Ctl& c = *ctl;
  c.iters_lo = c.iter;
  const bool go_on = (c.switch_req || c.status == 0) && !phase_failed(c.status);
  unsigned refine = 0;
  if (go_on && c.iter < c.max_iter) {
    c.done = 0; c.status = 0; c.switch_req = 0; c.lo_phase = 0; c.phase = 1; c.restart = 1; c.stop_dE = 0;
    c.iter_phase0 = c.iter; c.max_iter_phase = c.max_iter;
    c.stall_switch = 1; c.anchor_res = 1e300; c.anchor_iter = c.iter;
    refine = 1;
  }
  cudaGraphSetConditional(cond, refine);
}

__global__ void k_batch_gate64(Ctl* ctl, cudaGraphConditionalHandle cond) {
  Ctl& c = *ctl;
  unsigned run = 0;
  if (c.phase == 1 && c.lo_phase == 0 && c.stall_switch && c.switch_req && c.iter < c.max_iter) {
    c.iters_hi = c.iter;
    c.done = 0; c.status = 0; c.switch_req = 0; c.phase = 2; c.restart = 1; c.stop_dE = 0;
    c.iter_phase0 = c.iter; c.max_iter_phase = c.max_iter; c.stall_switch = 0;
    run = 1;
  }
  cudaGraphSetConditional(cond, run);
}
cudaError_t launch_batch_gate64(Ctl* ctl, unsigned long long cond, cudaStream_t st) {
  k_batch_gate64<<<1, 1, 0, st>>>(ctl, (cudaGraphConditionalHandle)cond);
  return cudaGetLastError();
}
cudaError_t launch_batch_gate(Ctl* ctl, unsigned long long cond, cudaStream_t st) {
  k_batch_gate<<<1, 1, 0, st>>>(ctl, (cudaGraphConditionalHandle)cond);
  return cudaGetLastError();
}

__global__ void k_batch_final(const dsc* __restrict__ s, double2* __restrict__ d, long long n, const Ctl* __restrict__ ctl) {
  if (ctl->phase != 1 || ctl->lo_phase != 0 || phase_failed(ctl->status)) return;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const dsc v = s[i];
    d[i] = make_double2((double)v.x, (double)v.y);
  }
}
cudaError_t launch_batch_final(const void* phids, void* phi128, long long n, const Ctl* ctl, cudaStream_t st) {
  k_batch_final<<<grid_for(n), 256, 0, st>>>((const dsc*)phids, (double2*)phi128, n, ctl);
  return cudaGetLastError();
}

// Fixed-order FP64 sum of |phi|^2 over all blocks (runs once per solve
// phase): per-block partials, the last block to finish sums them in block
// order and arms the control block: cc = 1 / ||phi||, ss = 0, retract = 1, so that the next H pass normalises phi in place.
constexpr int kNormThreads = 256;
template <typename C>
__global__ void __launch_bounds__(kNormThreads) k_init_norm(const C* __restrict__ phi, long long n, double weight,
                                                            Ctl* ctl, double* __restrict__ partials,
                                                            unsigned* ticket) {
  __shared__ double sm[kNormThreads / 32];
  __shared__ int s_last;
  double acc = 0.0;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const C v = phi[i];
    const double re = (double)v.x, im = (double)v.y;
    acc += re * re + im * im;
  }
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if ((threadIdx.x & 31) == 0) sm[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    double b = 0.0;
    for (int w = 0; w < kNormThreads / 32; ++w) b += sm[w];
    partials[blockIdx.x] = b;
    __threadfence();
    s_last = (atomicAdd(ticket, 1u) == gridDim.x - 1) ? 1 : 0;
  }
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  // FP64 additions are 64 cycles apart in one thread: the block shares them
  acc = 0.0;
  for (unsigned b = threadIdx.x; b < gridDim.x; b += blockDim.x) acc += __ldcg(partials + b);
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if ((threadIdx.x & 31) == 0) sm[threadIdx.x >> 5] = acc;  // read by thread 0 before s_last's barrier
  __syncthreads();
  if (threadIdx.x != 0) return;
  double tot = 0.0;
  for (int w = 0; w < kNormThreads / 32; ++w) tot += sm[w];
  ctl->cc = num(1.0 / sqrt(weight * tot));
  ctl->ss = num(0.0);
  ctl->retract = 1;
  *ticket = 0u;  // ready for the next reduction
}

cudaError_t launch_init_norm(int prec, const void* phi, long long n, double weight, Ctl* ctl, double* partials,
                             unsigned* ticket, cudaStream_t st) {
  long long g = (n + 8LL * kNormThreads - 1) / (8LL * kNormThreads);
  if (g < 1) g = 1;
  if (g > 1024) g = 1024;
  const int grid = (int)g;
  if (prec == 1) k_init_norm<double2><<<grid, kNormThreads, 0, st>>>((const double2*)phi, n, weight, ctl, partials, ticket);
  else if (prec == 2) k_init_norm<dsc><<<grid, kNormThreads, 0, st>>>((const dsc*)phi, n, weight, ctl, partials, ticket);
  else k_init_norm<float2><<<grid, kNormThreads, 0, st>>>((const float2*)phi, n, weight, ctl, partials, ticket);
  return cudaGetLastError();
}

}  // namespace gpe
