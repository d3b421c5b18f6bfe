// gpe_adjoint.cu -- pointwise and reduction kernels of the tangent-space
// adjoint solve (gpe_tangent_solve): the projected conjugate gradient method
// for K z = P g on {z : <phi, z> = 0}, with
//   K f = H_phi f + eta |phi|^2 f + eta phi^2 conj(f) - lambda f
// (the operator of 1/2 grad^2 E(phi)[f, f] - lambda ||f||^2, Section 2) and
// P h = h - <phi, h> phi (the tangent projector M_phi of Section 2 with the
// phase direction i phi removed too).  H_phi f and the preconditioner P_C are
// the pass kernels of the solver; this file adds the fused epilogues, the
// inner products (FP64 sums, fixed order) and the scalar steps, which run on
// the device so that the host reads scalars only at convergence checks.
//
// Every kernel here may be launched early (launch_early), so fields are read by coherent
// loads (__ldcg): the kernel in front may still be writing r, y or q, and the caller's
// phi and g_rho, when this one starts.
#include "gpe_internal.h"

namespace gpe {

namespace {

// Blocks of one warp per SM sub-partition: an FP64 instruction holds its
// sub-partition's pipe for 64 cycles per warp, so these kernels last as long as
// the warps' FP64 chains on the busiest sub-partition (256^2: 512 warps of four
// points on 608 sub-partitions).
constexpr int kDotThreads = 128;

template <typename C> struct Real;
template <> struct Real<float2> { using type = float; };
template <> struct Real<double2> { using type = double; };

__device__ __forceinline__ double2 dconj_mul(double ax, double ay, double bx, double by) {
  // conj(a) * b
  return make_double2(ax * bx + ay * by, ax * by - ay * bx);
}

// Sums over a warp of up to eight values at once: each of the first three steps
// halves the values a lane keeps as well as the lanes, 9 additions instead of 5
// per value.  Lane l returns the total of value 4 (l/16 & 1) + 2 (l/8 & 1) + (l/4 & 1).
__device__ __forceinline__ double warp_sum8(const double (&v)[8]) {
  const int l = threadIdx.x & 31;
  const bool b4 = l & 16, b3 = l & 8, b2 = l & 4;
  double w[4], u[2];
#pragma unroll
  for (int j = 0; j < 4; ++j)
    w[j] = (b4 ? v[4 + j] : v[j]) + __shfl_xor_sync(0xffffffffu, b4 ? v[j] : v[4 + j], 16);
#pragma unroll
  for (int j = 0; j < 2; ++j) u[j] = (b3 ? w[2 + j] : w[j]) + __shfl_xor_sync(0xffffffffu, b3 ? w[j] : w[2 + j], 8);
  double x = (b2 ? u[1] : u[0]) + __shfl_xor_sync(0xffffffffu, b2 ? u[0] : u[1], 4);
  x += __shfl_xor_sync(0xffffffffu, x, 2);
  x += __shfl_xor_sync(0xffffffffu, x, 1);
  return x;
}

// Block totals (fixed order): in warp 0, lane l returns the total of value l mod 8.
__device__ __forceinline__ double block_sum8(const double (&v)[8], double (*sm)[8]) {
  constexpr int NW = kDotThreads / 32;
  static_assert(NW == 4, "four warps: the last two steps sum over lane bits 3 and 4");
  const int l = threadIdx.x & 31;
  const double x = warp_sum8(v);
  if ((l & 3) == 0) sm[threadIdx.x >> 5][4 * (l >> 4) + 2 * ((l >> 3) & 1) + ((l >> 2) & 1)] = x;
  __syncthreads();
  double t = 0.0;
  if (threadIdx.x < 32) {
    t = sm[l >> 3][l & 7];
    t += __shfl_xor_sync(0xffffffffu, t, 8);
    t += __shfl_xor_sync(0xffffffffu, t, 16);
  }
  return t;
}

// The scalar step `stage` from the weighted totals t (all lanes of warp 0 hold
// them; lane 0 writes).
__device__ __forceinline__ void adj_scalar_step(int stage, const double (&t)[6], AdjScalars* __restrict__ S) {
  if (threadIdx.x != 0 || S->stop) return;  // stop: the solve has ended; later kernels of the last round change nothing
  switch (stage) {
    case ADJ_PROJ:  // t = <phi, h>
      S->c_re = t[0]; S->c_im = t[1];
      break;
    case ADJ_BB:  // t = ||r0||^2
      S->bb = t[0]; S->rr = t[0];
      if (!isfinite(t[0])) { S->bad = 3; S->stop = 1; }
      else if (t[0] == 0.0) S->stop = 1;  // P g = 0: z = 0
      break;
    case ADJ_PQ: {  // t = <phi, q>, <p, q>, <p, phi>;  Re<p, q - c phi>
      S->c_re = t[0]; S->c_im = t[1];
      // <p, c phi> = c <p, phi>
      const double pq = t[2] - (t[0] * t[4] - t[1] * t[5]);
      S->pq = pq;
      if (!(pq > 0.0) || !isfinite(pq)) { S->bad = 1; S->stop = 1; }  // K not positive on the tangent space
      else S->a = S->ry / pq;
      break;
    }
    case ADJ_RR:  // t = ||r||^2
      S->rr = t[0];
      S->iters += 1;
      if (!isfinite(t[0])) { S->bad = 3; S->stop = 1; }
      else if (t[0] <= S->tol2 * S->bb) S->stop = 1;  // ||r|| <= tol ||P g||
      break;
    case ADJ_RY:        // t = <phi, y>, <r, y>, <r, phi>;  Re<r, y - c phi>
    case ADJ_RY_FIRST: {
      S->c_re = t[0]; S->c_im = t[1];
      const double ry = t[2] - (t[0] * t[4] - t[1] * t[5]);
      S->beta = (stage == ADJ_RY_FIRST) ? 0.0 : ry / S->ry;
      if (!(ry > 0.0) || !isfinite(ry)) { S->bad = 2; S->stop = 1; }  // preconditioner not positive
      S->ry = ry;
      break;
    }
    default:
      break;
  }
}

// Sum over the grid in a fixed order: block totals to red.partials, and the last
// block to arrive sums them and runs the scalar step, so that a reduction needs
// no kernel of its own (one that summed 1024 slots on one SM took 17.6 us).
struct AdjRed {
  double* partials;  // [blocks][8]
  unsigned* ticket;  // zero on entry, zero on return
  double weight;
  int stage;
  AdjScalars* S;
};
__device__ __forceinline__ void adj_reduce(const double (&v)[8], const AdjRed& red) {
  __shared__ double sm[kDotThreads / 32][8];
  __shared__ int s_last;
  double t = block_sum8(v, sm);
  if (threadIdx.x < 8) red.partials[(size_t)blockIdx.x * 8 + threadIdx.x] = t;
  if (threadIdx.x < 32) {
    __threadfence();
    __syncwarp();
    if (threadIdx.x == 0) s_last = (atomicAdd(red.ticket, 1u) == gridDim.x - 1) ? 1 : 0;
  }
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  double w[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) w[j] = 0.0;
  for (unsigned b = threadIdx.x; b < gridDim.x; b += kDotThreads) {
    const double2* pb = reinterpret_cast<const double2*>(red.partials + (size_t)b * 8);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const double2 x = __ldcg(pb + j);
      w[2 * j] += x.x;
      w[2 * j + 1] += x.y;
    }
  }
  t = block_sum8(w, sm) * red.weight;
  if (threadIdx.x >= 32) return;
  double tot[6];
#pragma unroll
  for (int j = 0; j < 6; ++j) tot[j] = __shfl_sync(0xffffffffu, t, j);
  adj_scalar_step(red.stage, tot, red.S);
  if (threadIdx.x == 0) *red.ticket = 0u;
}

// Up to three inner products sum conj(x_j) y_j (x_j null: skipped; the real part of the second).
template <typename C>
__global__ void __launch_bounds__(kDotThreads) k_dots(const C* x0, const C* y0,
                                                      const C* x1, const C* y1,
                                                      const C* x2, const C* y2, long long n,
                                                      AdjRed red) {
  pdl_wait();
  x0 = after_wait(x0);
  y0 = after_wait(y0);
  x1 = after_wait(x1);
  y1 = after_wait(y1);
  x2 = after_wait(x2);
  y2 = after_wait(y2);
  double v[8] = {0, 0, 0, 0, 0, 0, 0, 0};
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    if (x0) { const C a = __ldcg(x0 + i), b = __ldcg(y0 + i); const double2 d = dconj_mul(a.x, a.y, b.x, b.y); v[0] += d.x; v[1] += d.y; }
    if (x1) { const C a = __ldcg(x1 + i), b = __ldcg(y1 + i); v[2] += (double)a.x * b.x + (double)a.y * b.y; }  // real part
    if (x2) { const C a = __ldcg(x2 + i), b = __ldcg(y2 + i); const double2 d = dconj_mul(a.x, a.y, b.x, b.y); v[4] += d.x; v[5] += d.y; }
  }
  pdl_trigger();
  adj_reduce(v, red);
}

// q <- q + eta |phi|^2 p + eta phi^2 conj(p) - lam p  (q holds H_phi p on entry),
// then the sums <phi, q>, Re<p, q>, <p, phi>.
template <typename C>
__global__ void __launch_bounds__(kDotThreads) k_hess_epi(const C* phi, const C* p,
                                                          C* __restrict__ q, long long n, double eta, double lam,
                                                          AdjRed red) {
  using R = typename Real<C>::type;
  const R e = R(eta), l = R(lam);
  pdl_wait();
  phi = after_wait(phi);
  p = after_wait(p);
  q = after_wait(q);
  double v[8] = {0, 0, 0, 0, 0, 0, 0, 0};
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const C f = __ldcg(phi + i), d = __ldcg(p + i);
    C h = q[i];
    const R u = f.x * f.x + f.y * f.y;
    const R s2x = f.x * f.x - f.y * f.y, s2y = R(2) * f.x * f.y;  // phi^2
    // phi^2 conj(p) = (s2x + i s2y)(d.x - i d.y)
    const R cx = s2x * d.x + s2y * d.y, cy = s2y * d.x - s2x * d.y;
    h.x += e * (u * d.x + cx) - l * d.x;
    h.y += e * (u * d.y + cy) - l * d.y;
    q[i] = h;
    double2 t = dconj_mul(f.x, f.y, h.x, h.y); v[0] += t.x; v[1] += t.y;
    v[2] += (double)d.x * h.x + (double)d.y * h.y;
    t = dconj_mul(d.x, d.y, f.x, f.y); v[4] += t.x; v[5] += t.y;
  }
  pdl_trigger();
  adj_reduce(v, red);
}

// z += a p; r -= a (q - c phi); and the sum |r|^2.
template <typename C>
__global__ void __launch_bounds__(kDotThreads) k_step(C* __restrict__ z, C* __restrict__ r, const C* p,
                                                      const C* q, const C* phi, long long n,
                                                      AdjRed red) {
  using R = typename Real<C>::type;
  const AdjScalars* S = red.S;
  pdl_wait();
  p = after_wait(p);
  q = after_wait(q);
  phi = after_wait(phi);
  z = after_wait(z);
  r = after_wait(r);
  if (S->stop) return;  // converged or broken down: leave z and r as they are
  const R a = R(S->a), cr = R(S->c_re), ci = R(S->c_im);
  double v[8] = {0, 0, 0, 0, 0, 0, 0, 0};
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const C d = __ldcg(p + i), h = __ldcg(q + i), f = __ldcg(phi + i);
    C zz = z[i], rr = r[i];
    const R qx = h.x - (cr * f.x - ci * f.y), qy = h.y - (cr * f.y + ci * f.x);
    zz.x += a * d.x; zz.y += a * d.y;
    rr.x -= a * qx; rr.y -= a * qy;
    z[i] = zz; r[i] = rr;
    v[0] += (double)rr.x * rr.x + (double)rr.y * rr.y;
  }
  pdl_trigger();
  adj_reduce(v, red);
}

// h_out = h_in - c phi (c complex from S), h_out may alias h_in.
template <typename C>
__global__ void k_proj(const C* h_in, C* __restrict__ h_out, const C* phi, long long n,
                       const AdjScalars* S) {
  using R = typename Real<C>::type;
  pdl_wait();
  phi = after_wait(phi);
  const R cr = R(S->c_re), ci = R(S->c_im);
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const C h = h_in[i], f = __ldcg(phi + i);
    C o;
    o.x = h.x - (cr * f.x - ci * f.y);
    o.y = h.y - (cr * f.y + ci * f.x);
    h_out[i] = o;
  }
}

// p = (y - c phi) + beta p (beta = 0: p is not read).
template <typename C>
__global__ void k_dir(C* __restrict__ p, const C* y, const C* phi, long long n,
                      const AdjScalars* S) {
  using R = typename Real<C>::type;
  pdl_wait();
  y = after_wait(y);
  phi = after_wait(phi);
  p = after_wait(p);
  if (S->stop) return;
  const R cr = R(S->c_re), ci = R(S->c_im), b = R(S->beta);
  const bool keep = S->beta != 0.0;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const C h = __ldcg(y + i), f = __ldcg(phi + i);
    C o;
    o.x = h.x - (cr * f.x - ci * f.y);
    o.y = h.y - (cr * f.y + ci * f.x);
    if (keep) { const C q = p[i]; o.x += b * q.x; o.y += b * q.y; }
    p[i] = o;
  }
}

// rhs = s g_rho phi (s = 2 / h^d: the weighted gradient of a loss of the
// density |phi|^2 whose coefficient gradient is g_rho).
template <typename C>
__global__ void k_density_rhs(const C* phi, const double* g_rho, C* __restrict__ rhs,
                              long long n, double s) {
  using R = typename Real<C>::type;
  pdl_wait();
  phi = after_wait(phi);
  g_rho = after_wait(g_rho);
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const C f = __ldcg(phi + i);
    const R k = R(s * __ldcg(g_rho + i));
    C o;
    o.x = k * f.x;
    o.y = k * f.y;
    rhs[i] = o;
  }
}

// grad_V = -h^d Re(conj(z) phi)
template <typename C>
__global__ void k_dV_from_z(const C* phi, const C* z, double* __restrict__ gV, long long n,
                            double weight) {
  pdl_wait();
  phi = after_wait(phi);
  z = after_wait(z);
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const C f = __ldcg(phi + i), q = __ldcg(z + i);
    gV[i] = -weight * ((double)q.x * f.x + (double)q.y * f.y);
  }
}

int grid_of(long long n, int max_blocks) {
  long long g = (n + 4LL * kDotThreads - 1) / (4LL * kDotThreads);
  if (g < 1) g = 1;
  if (g > max_blocks) g = max_blocks;
  return (int)g;
}

}  // namespace

cudaError_t adj_dots(int prec, const void* x0, const void* y0, const void* x1, const void* y1, const void* x2,
                     const void* y2, long long n, double weight, int stage, const AdjWork& w, cudaStream_t st) {
  const int g = grid_of(n, kAdjMaxBlocks);
  cudaError_t e;
  const AdjRed red = {w.partials, w.ticket, weight, stage, w.S};
  if (prec == 1)
    e = launch_early(true, k_dots<double2>, g, kDotThreads, 0, st, (const double2*)x0, (const double2*)y0, (const double2*)x1, (const double2*)y1, (const double2*)x2, (const double2*)y2, n, red);
  else
    e = launch_early(true, k_dots<float2>, g, kDotThreads, 0, st, (const float2*)x0, (const float2*)y0, (const float2*)x1, (const float2*)y1, (const float2*)x2, (const float2*)y2, n, red);
  return e;
}

cudaError_t adj_hess_epi(int prec, const void* phi, const void* p, void* q, long long n, double eta, double lam,
                         double weight, const AdjWork& w, cudaStream_t st) {
  const int g = grid_of(n, kAdjMaxBlocks);
  cudaError_t e;
  const AdjRed red = {w.partials, w.ticket, weight, ADJ_PQ, w.S};
  if (prec == 1)
    e = launch_early(true, k_hess_epi<double2>, g, kDotThreads, 0, st, (const double2*)phi, (const double2*)p, (double2*)q, n, eta, lam, red);
  else
    e = launch_early(true, k_hess_epi<float2>, g, kDotThreads, 0, st, (const float2*)phi, (const float2*)p, (float2*)q, n, eta, lam, red);
  return e;
}

cudaError_t adj_step(int prec, void* z, void* r, const void* p, const void* q, const void* phi, long long n,
                     double weight, const AdjWork& w, cudaStream_t st) {
  const int g = grid_of(n, kAdjMaxBlocks);
  cudaError_t e;
  const AdjRed red = {w.partials, w.ticket, weight, ADJ_RR, w.S};
  if (prec == 1)
    e = launch_early(true, k_step<double2>, g, kDotThreads, 0, st, (double2*)z, (double2*)r, (const double2*)p, (const double2*)q, (const double2*)phi, n, red);
  else
    e = launch_early(true, k_step<float2>, g, kDotThreads, 0, st, (float2*)z, (float2*)r, (const float2*)p, (const float2*)q, (const float2*)phi, n, red);
  return e;
}

cudaError_t adj_proj(int prec, const void* h_in, void* h_out, const void* phi, long long n, const AdjScalars* S,
                     cudaStream_t st) {
  const int g = grid_of(n, 4096);
  cudaError_t e;
  if (prec == 1) e = launch_early(true, k_proj<double2>, g, kDotThreads, 0, st, (const double2*)h_in, (double2*)h_out, (const double2*)phi, n, S);
  else e = launch_early(true, k_proj<float2>, g, kDotThreads, 0, st, (const float2*)h_in, (float2*)h_out, (const float2*)phi, n, S);
  return e;
}

cudaError_t adj_dir(int prec, void* p, const void* y, const void* phi, long long n, const AdjScalars* S, cudaStream_t st) {
  const int g = grid_of(n, 4096);
  cudaError_t e;
  if (prec == 1) e = launch_early(true, k_dir<double2>, g, kDotThreads, 0, st, (double2*)p, (const double2*)y, (const double2*)phi, n, S);
  else e = launch_early(true, k_dir<float2>, g, kDotThreads, 0, st, (float2*)p, (const float2*)y, (const float2*)phi, n, S);
  return e;
}

cudaError_t adj_density_rhs(int prec, const void* phi, const double* g_rho, void* rhs, long long n, double s,
                            cudaStream_t st) {
  const int g = grid_of(n, 4096);
  cudaError_t e;
  if (prec == 1) e = launch_early(true, k_density_rhs<double2>, g, kDotThreads, 0, st, (const double2*)phi, g_rho, (double2*)rhs, n, s);
  else e = launch_early(true, k_density_rhs<float2>, g, kDotThreads, 0, st, (const float2*)phi, g_rho, (float2*)rhs, n, s);
  return e;
}

cudaError_t adj_dV_from_z(int prec, const void* phi, const void* z, double* gV, long long n, double weight,
                          cudaStream_t st) {
  const int g = grid_of(n, 4096);
  cudaError_t e;
  if (prec == 1) e = launch_early(true, k_dV_from_z<double2>, g, kDotThreads, 0, st, (const double2*)phi, (const double2*)z, gV, n, weight);
  else e = launch_early(true, k_dV_from_z<float2>, g, kDotThreads, 0, st, (const float2*)phi, (const float2*)z, gV, n, weight);
  return e;
}

}  // namespace gpe
