// gpe_hflow.cu -- H_phi f on a batch of complex64 planes (the fields of a 2D batch,
// or the x and y parts on the z planes of a 3D field; arXiv:1611.02045, Section 2
// operator with the discretisation of eq. FFTdiscret, Section 3) as a dataflow of
// independent work units.
//
// H_phi f = A_x f + A_y f + (V + eta|phi|^2) f with the per-axis spectral parts
//   A_x f = IFFT_x[ (1/2 xi^2 + omega y xi) FFT_x f ]   (row lines)
//   A_y f = IFFT_y[ (1/2 mu^2 - omega x mu) FFT_y f ]   (column lines).
// Planes are MX x MY points, each 64, 128 or 256.  A plane is split into MX MY / 4096
// x units (4096 / MX rows) and as many y units (4096 / MY columns): every unit is
// 4096 points, 256 threads of 16 values.  An x unit stores t = A_x f + (V +
// eta|phi|^2) f to its rows of out; a y unit adds A_y f into its columns of out,
// which is only allowed once the plane's x units have stored their rows.  Units
// come from one ticket counter in an order that puts every x unit of a plane `lag`
// planes ahead of the plane's y units; a y unit that finds its plane incomplete
// waits (bounded) on the plane's x-unit counter.  Persistent blocks (two per SM,
// all SMs) walk the tickets with two shared-memory stages: while one unit is
// transformed, the TMA copies the next unit's input into the other stage
//   x unit: contiguous rows of f (32 KB) and of V (16 KB), 1D bulk copies; phi,
//           where it is not f, comes by plain loads issued before the wait;
//   y unit: column tiles of f (32 KB), 3D tensor-map boxes of 16 columns with
//           the 128-byte swizzle (conflict-free column access);
// and a y unit's result tiles are added into out by TMA reduce-adds.  A line of M
// points is transformed by M/16 threads of one warp (radix 16, then M/16), with
// shared-memory exchanges inside the warp, so the only block barrier is the one at
// the end of each unit.
//
// Global traffic per point: read f (x unit) and write out once (16 bytes); the y
// unit's re-read of f and the read-modify-write of out hit L2 while the plane is in
// flight (lag planes hold 2^21 points, 32 MB of f and out).  The same arithmetic in
// 16-CTA clusters (gpe_cluster.cuh) leaves SM slots empty: clusters of 16 pack into
// 14 x 16 = 224 of the 304 CTA slots of the GPU, and every field waits for its
// slowest CTA; here all slots are busy and no unit waits for another block except
// through the x-unit counters.
//
// Measured (us): 512 x 256^2, f = phi 227 -> 200 with the half-warp layout of the column
// lines (their 8-byte accesses hit each bank twice before); 333 x 128^2, f != phi 62.6
// (clusters) -> 49.4; 256 x 256 x 512 field, whole H phi with the z pass 521 (three
// passes) -> 391.  2048 x 128^2 and 8192 x 64^2, f = phi: 207 and 228 (332 and 329 in
// clusters).
//
// Counters (ctr, owned by the context, zero between launches): ctr[0] ticket,
// ctr[1] blocks finished, ctr[2 + b] x units of plane b done.  The last block to
// finish zeroes them, so no separate reset runs before the next launch.
//
// A wait that gives up marks *status, leaves its unit's sum out and its block takes no
// further unit: the launch ends (later waits on what the block dropped give up as well),
// out is not valid and the next launch starts from zero counters again.
#include <cuda_runtime.h>

#include <atomic>

#include "gpe_cluster.cuh"
#include "gpe_fft.cuh"
#include "gpe_internal.h"
#include "gpe_tma.cuh"

namespace gpe {

namespace {

constexpr int kUnit = 4096;                                 // points per unit
constexpr size_t kFlowStage = 48 * 1024;                    // bytes per stage
constexpr long long kFlowLagPoints = 32ll * 256 * 256;      // points between a plane's x and y units

// Lines of M points: TL threads per line, PW lines per warp, LU lines per unit.
template <int M> struct FlowLine {
  static constexpr int TL = M / 16, PW = 32 / TL, LU = kUnit / M;
  static constexpr int NBOX = LU / 16;  // 16-column boxes per y unit
};
template <int MX, int MY> struct FlowSmem {
  static constexpr size_t tws = (MX == MY ? 1 : 2) * 16 * kTw256Stride * sizeof(float4);
  static constexpr size_t kt = (MX + MY) * sizeof(float2);  // multiplier tables (x, y)
  static constexpr size_t bytes = 2 * kFlowStage + tws + kt + 32;  // + 2 mbarriers, 2 unit ids, flag
};

struct FlowArgs {
  int nbatch, lag;
  long long stride;   // elements between consecutive planes
  long long vstride;  // elements between the planes of V (0: one V for all)
  float eta, omega;
  const float *xi, *xiy, *xc, *yc, *V;
  const float2 *twx, *twy;  // e^{-2 pi i m/MX}, e^{-2 pi i m/MY}
  const float2* phi;        // density field
  const float2* f;          // operand (may equal phi)
  float2* out;
  int* ctr;     // [0] ticket, [1] blocks finished, [2 + b] x units done of plane b
  int* status;  // set to GPE_ERR_TIMEOUT (6) when a bounded wait gives up (may be null)
  long long polls;  // of a y unit's wait for its plane's x units before it gives up
};

// Ticket u -> (type 0 = x unit / 1 = y unit, plane, unit of the plane), NU units of
// each type per plane.  Order: the x units of planes 0 .. D-1; then, for j = 0, 1,
// ...: the y units of plane j followed by the x units of plane D + j; then the
// remaining y units.  Every x unit of a plane comes before its y units.
template <int NU>
__host__ __device__ inline void flow_unit(long long u, int B, int D, int* type, int* fld, int* blk) {
  const long long head = (long long)NU * D;
  if (u < head) { *type = 0; *fld = (int)(u / NU); *blk = (int)(u % NU); return; }
  long long k = u - head;
  const long long P = (long long)B - D;
  if (k < 2 * NU * P) {
    const long long pair = k / (2 * NU), w = k % (2 * NU);
    if (w < NU) { *type = 1; *fld = (int)pair; *blk = (int)w; }
    else { *type = 0; *fld = (int)(D + pair); *blk = (int)(w - NU); }
    return;
  }
  k -= 2 * NU * P;
  *type = 1; *fld = (int)(P + k / NU); *blk = (int)(k % NU);
}

// Stage-2 twiddles e^{-2 pi i j r / M}, j = 0 .. 15 (row of 9 float4), r < M/16, two per float4.
template <int M>
__device__ __forceinline__ void flow_twiddles(float4* tws, const float2* __restrict__ tw) {
  constexpr int R2 = M / 16;
  for (int i = threadIdx.x; i < 16 * (R2 / 2); i += blockDim.x) {
    const int j = i / (R2 / 2), h = i % (R2 / 2);
    const float2 a = tw[j * 2 * h], b = tw[j * (2 * h + 1)];
    tws[j * kTw256Stride + h] = make_float4(a.x, a.y, b.x, b.y);
  }
}

// Stage 2 of a line of M: values v[q] at positions t + q M/16, radix M/16.
template <int M, int DIR>
__device__ __forceinline__ void flow_stage2(float2 (&v)[16], int t, const float4* tws) {
  constexpr int R2 = M / 16, NB = 16 / R2, TL = M / 16;
#pragma unroll
  for (int b = 0; b < NB; ++b) {
    const float4* w = tws + (t + b * TL) * kTw256Stride;
    float2 x[R2];
#pragma unroll
    for (int r = 0; r < R2; r += 2) {
      const float4 p = w[r / 2];
      x[r] = r ? ctw<DIR>(v[b + r * NB], make_float2(p.x, p.y)) : v[b];
      x[r + 1] = ctw<DIR>(v[b + (r + 1) * NB], make_float2(p.z, p.w));
    }
    dft_small<R2, DIR>(x);
#pragma unroll
    for (int r = 0; r < R2; ++r) v[b + r * NB] = x[r];
  }
}

// A row line of M points held by M/16 threads (v[q] = position t + q M/16),
// transformed in place in the line's own M slots: the stage-1 results of thread t
// (positions 16t .. 16t+15) go out as eight 16-byte chunks, chunk index XOR (t mod
// 8) XOR s, so the vector stores and the stage-2 loads are free of bank conflicts
// without padding; s separates the lines of a warp that share banks (row_swz).
template <int M> __device__ __forceinline__ int row_swz(int l) {
  return M == 256 ? 0 : (M == 128 ? 4 * (l & 1) : 4 * (l & 1) + (l & 2));
}
template <int M, int DIR>
__device__ __forceinline__ void dft_row(float2 (&v)[16], float2* row, int t, int s, const float4* tws) {
  constexpr int TL = M / 16;
  dft16<DIR>(v);
  __syncwarp();
  {
    float4* d = reinterpret_cast<float4*>(row + 16 * t);
    const int sw = (t & 7) ^ s;
#pragma unroll
    for (int i = 0; i < 8; ++i) d[i ^ sw] = make_float4(v[2 * i].x, v[2 * i].y, v[2 * i + 1].x, v[2 * i + 1].y);
  }
  __syncwarp();
#pragma unroll
  for (int q = 0; q < 16; ++q) {
    const int p = t + TL * q, g = p >> 4;
    v[q] = row[16 * g + 2 * (((p >> 1) & 7) ^ (g & 7) ^ s) + (p & 1)];
  }
  flow_stage2<M, DIR>(v, t, tws);
}

// Element (row y, column 2 c + j) of a [M][16] complex64 tile written by the TMA
// with the 128-byte swizzle: 16-byte chunk c of row y sits at chunk c ^ (y mod 8)
// of that 128-byte row.  Index in float2 units.
__device__ __forceinline__ int tile_cell(int y, int c, int j) { return y * 16 + 2 * (c ^ (y & 7)) + j; }

// A column line of the swizzled tile (column 2 c + j) held by M/16 threads of a
// warp; the exchange stores position p in row pi(p) = p ^ ((p >> 4) & 7) (a
// permutation), which keeps the stage-1 stores and stage-2 loads conflict-free and
// inside the warp's own cells of the tile.
template <int M, int DIR>
__device__ __forceinline__ void dft_col(float2 (&v)[16], float2* tile, int t, int c, int j, const float4* tws) {
  constexpr int TL = M / 16;
  dft16<DIR>(v);
  __syncwarp();
#pragma unroll
  for (int r = 0; r < 16; ++r) {
    const int p = 16 * t + r;
    tile[tile_cell(p ^ ((p >> 4) & 7), c, j)] = v[r];
  }
  __syncwarp();
#pragma unroll
  for (int q = 0; q < 16; ++q) {
    const int p = t + TL * q;
    v[q] = tile[tile_cell(p ^ ((p >> 4) & 7), c, j)];
  }
  flow_stage2<M, DIR>(v, t, tws);
}

template <int MX, int MY, bool SAME>
__global__ void __launch_bounds__(256, 2)
    h_batch_flow(const __grid_constant__ FlowArgs a, const __grid_constant__ CUtensorMap tmF, const __grid_constant__ CUtensorMap tmO) {
  using C = float2;
  using LX = FlowLine<MX>;
  using LY = FlowLine<MY>;
  using SM = FlowSmem<MX, MY>;
  constexpr int NU = MX * MY / kUnit;  // units of each type per plane
  extern __shared__ __align__(1024) unsigned char flow_sm[];
  float4* twsx = reinterpret_cast<float4*>(flow_sm + 2 * kFlowStage);
  float4* twsy = MX == MY ? twsx : twsx + 16 * kTw256Stride;
  // kt[p] = (k_p, k_p^2 / (2M)): the Fourier multiplier of a line is (k^2/2 + c k)/M
  // = fma(c/M, k, k^2/(2M)) with c = omega y (x lines) or -omega x (y lines); 1/M is exact
  float2* ktx = reinterpret_cast<float2*>(flow_sm + 2 * kFlowStage + SM::tws);
  float2* kty = ktx + MX;
  unsigned char* ctl_sm = flow_sm + 2 * kFlowStage + SM::tws + SM::kt;
  unsigned long long* full = reinterpret_cast<unsigned long long*>(ctl_sm);
  volatile int* uid = reinterpret_cast<volatile int*>(ctl_sm + 16);
  volatile int* last_block = reinterpret_cast<volatile int*>(ctl_sm + 24);
  const int tid = threadIdx.x, lane = tid & 31, wp = tid >> 5;
  const long long total = 2ll * NU * a.nbatch;
  const float om = a.omega, eta = a.eta;
  auto stage = [&](int s) { return reinterpret_cast<C*>(flow_sm + s * kFlowStage); };
  bool ok = (smem_u32(flow_sm) & 1023u) == 0;  // the swizzled tiles need 1024-byte alignment

  // thread 0: the ticket taken one refill ahead, and the x-unit count of the
  // next unit's plane read one unit ahead (when that unit is a y unit)
  int tk_next = 0, early = 0;
  // thread 0: start the copies of the next ticket's unit into stage s
  auto grab_issue = [&](int s) {
    const long long u = tk_next;
    tk_next = atomicAdd(a.ctr, 1);
    if (u >= total || !ok) { uid[s] = -1; return; }
    uid[s] = (int)u;
    int type, fld, blk;
    flow_unit<NU>(u, a.nbatch, a.lag, &type, &fld, &blk);
    C* d = stage(s);
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // earlier generic accesses of the stage
    if (type == 0) {
      mbar_expect_tx(&full[s], 48 * 1024);
      bulk_load(d, a.f + fld * a.stride + (long long)blk * kUnit, 32 * 1024, &full[s]);
      bulk_load(reinterpret_cast<unsigned char*>(d) + 32 * 1024, a.V + fld * a.vstride + (long long)blk * kUnit,
                16 * 1024, &full[s]);
    } else {
      mbar_expect_tx(&full[s], 32 * 1024);
#pragma unroll
      for (int b = 0; b < LY::NBOX; ++b)
        tma_load_3d(d + b * 16 * MY, &tmF, 32 * (blk * LY::NBOX + b), 0, fld, &full[s]);
    }
  };
  if (tid == 0) {
    mbar_init(&full[0], 1);
    mbar_init(&full[1], 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  flow_twiddles<MX>(twsx, a.twx);
  if (MX != MY) flow_twiddles<MY>(twsy, a.twy);
  for (int i = tid; i < MX + MY; i += blockDim.x) {
    const float k = i < MX ? a.xi[i] : a.xiy[i - MX];
    ktx[i] = make_float2(k, 0.5f * k * k * (i < MX ? 1.0f / MX : 1.0f / MY));
  }
  __syncthreads();
  if (tid == 0) {
    tk_next = atomicAdd(a.ctr, 1);
    grab_issue(0);
    grab_issue(1);
  }
  __syncthreads();

  unsigned par = 0u;  // bit s: phase parity of stage s
  int s = 0;
  for (;;) {
    const int u = uid[s];
    if (u < 0) break;
    int type, fld, blk;
    flow_unit<NU>(u, a.nbatch, a.lag, &type, &fld, &blk);
    C* st = stage(s);
    if (type == 0) {
      // ---- x unit: row LU blk + l ----
      constexpr int TL = LX::TL;
      const int t = lane % TL, l = LX::PW * wp + lane / TL;
      const long long rowg = fld * a.stride + (long long)(LX::LU * blk + l) * MX + t;
      C ph[SAME ? 1 : 16];
      if constexpr (!SAME) {
#pragma unroll
        for (int q = 0; q < 16; ++q) ph[q] = __ldg(a.phi + rowg + TL * q);
      }
      if (!mbar_wait(&full[s], (par >> s) & 1u)) ok = false;
      C* row = st + l * MX;
      const float* Vr = reinterpret_cast<const float*>(st + kUnit) + l * MX;
      C w[16], sr[16];
#pragma unroll
      for (int q = 0; q < 16; ++q) {
        w[q] = row[t + TL * q];
        const C d = SAME ? w[q] : ph[SAME ? 0 : q];
        const float m = Vr[t + TL * q] + eta * (d.x * d.x + d.y * d.y);
        sr[q] = make_float2(m * w[q].x, m * w[q].y);
      }
      const int sw = row_swz<MX>(l);
      dft_row<MX, -1>(w, row, t, sw, twsx);
      const float cy = om * a.yc[LX::LU * blk + l] * (1.0f / MX);
#pragma unroll
      for (int q = 0; q < 16; ++q) {
        const float2 k = ktx[t + TL * q];
        w[q] = cscale(w[q], fmaf(cy, k.x, k.y));
      }
      dft_row<MX, +1>(w, row, t, sw, twsx);
      C* orow = a.out + rowg;
#pragma unroll
      for (int q = 0; q < 16; ++q) orow[TL * q] = cadd(w[q], sr[q]);
    } else {
      // ---- y unit: column LU blk + 16 box + 2 c + j; A_y f written back into the tile ----
      constexpr int TL = LY::TL;
      // M = 256: a half-warp takes eight threads of both columns of its chunk, so that its
      // 8-byte accesses (rows t mod 8, both halves of a chunk) cover all banks once
      const int t = MY == 256 ? ((lane & 7) | ((lane >> 1) & 8)) : lane % TL;
      const int ci = MY == 256 ? (lane >> 3) & 1 : lane / TL;
      const int j = ci & 1, h = ci >> 1;
      // chunks of a warp: 1 (M = 256), a neighbouring pair (128), two pairs c, c ^ 4 (64: the
      // four rows of a half-warp's lines then use different halves of the 128-byte rows)
      constexpr int CW = LY::PW / 2;  // chunks per warp
      const int box = wp * CW / 8;
      const int c = MY == 64 ? ((((wp & 1) << 1) + (h >> 1)) ^ ((h & 1) << 2)) : (wp * CW + h) % 8;
      C* tile = st + box * 16 * MY;
      if (!mbar_wait(&full[s], (par >> s) & 1u)) ok = false;
      C w[16];
#pragma unroll
      for (int q = 0; q < 16; ++q) w[q] = tile[tile_cell(t + TL * q, c, j)];
      dft_col<MY, -1>(w, tile, t, c, j, twsy);
      const float cx = -om * a.xc[LY::LU * blk + 16 * box + 2 * c + j] * (1.0f / MY);
#pragma unroll
      for (int q = 0; q < 16; ++q) {
        const float2 k = kty[t + TL * q];
        w[q] = cscale(w[q], fmaf(cx, k.x, k.y));
      }
      dft_col<MY, +1>(w, tile, t, c, j, twsy);
      __syncwarp();
#pragma unroll
      for (int q = 0; q < 16; ++q) tile[tile_cell(t + TL * q, c, j)] = w[q];
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // tile stores -> the TMA's reads
    }
    par ^= 1u << s;
    __syncthreads();  // the stage is consumed (y: rewritten); this unit's stores are issued
    if (type == 0 && tid == 32) {
      // the x unit's rows are stored: count it (the fence waits in warp 1, off thread 0's path)
      __threadfence();
      atomicAdd(a.ctr + 2 + fld, 1);
    }
    if (tid == 0) {
      if (type == 1) {
        // the plane's x units must have stored t before the TMA adds A_y f to it
        long long n = 0;
        if (early < NU)
          while (ld_acquire_gpu(a.ctr + 2 + fld) < NU && n < a.polls) ++n;
        if (n >= a.polls) ok = false;
        asm volatile("fence.proxy.async;" ::: "memory");  // generic stores of out -> the TMA's adds
        if (ok) {
#pragma unroll
          for (int b = 0; b < LY::NBOX; ++b)
            tma_reduce_add_3d(&tmO, st + b * 16 * MY, 32 * (blk * LY::NBOX + b), 0, fld);
        }
        asm volatile("cp.async.bulk.commit_group;" ::: "memory");
        asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");  // tiles read before the refill
      }
      grab_issue(s);
      early = 0;
      const int un = uid[s ^ 1];
      if (un >= 0) {
        int ty, fl, bl;
        flow_unit<NU>(un, a.nbatch, a.lag, &ty, &fl, &bl);
        if (ty == 1) early = ld_acquire_gpu(a.ctr + 2 + fl);
      }
    }
    s ^= 1;
  }
  if (tid == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
  if (!ok && a.status) atomicExch(a.status, 6);  // GPE_ERR_TIMEOUT
  // the last block to finish returns the counters to zero for the next launch
  __syncthreads();
  if (tid == 0) {
    __threadfence();
    *last_block = atomicAdd(a.ctr + 1, 1) == (int)gridDim.x - 1;
  }
  __syncthreads();
  if (*last_block) {
    __threadfence();
    for (int i = tid; i < a.nbatch; i += blockDim.x) a.ctr[2 + i] = 0;
    if (tid == 0) { a.ctr[0] = 0; a.ctr[1] = 0; }
  }
}

// FP32 view [B][my][2 mx] of complex64 planes, boxes of 16 complex columns x my rows, 128-byte swizzle.
bool encode_flow_map(CUtensorMap* m, const void* base, int mx, int my, int nbatch, long long stride) {
  PFN_cuTensorMapEncodeTiled_v12000 fn = encode_fn();
  if (!fn) return false;
  const cuuint64_t dims[3] = {2 * (cuuint64_t)mx, (cuuint64_t)my, (cuuint64_t)nbatch};
  const cuuint64_t strides[2] = {(cuuint64_t)mx * 8, (cuuint64_t)stride * 8};
  const cuuint32_t box[3] = {32, (cuuint32_t)my, 1};
  const cuuint32_t es[3] = {1, 1, 1};
  return fn(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, const_cast<void*>(base), dims, strides, box, es,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

template <int MX, int MY, bool SAME>
cudaError_t launch_flow_one(const FlowArgs& fa, const CUtensorMap& tmF, const CUtensorMap& tmO, cudaStream_t st,
                            bool* used) {
  auto kern = h_batch_flow<MX, MY, SAME>;
  constexpr size_t smem = FlowSmem<MX, MY>::bytes;
  static std::atomic<int> grid_dev[64];  // resident blocks per device; 0 = not yet queried
  const int dev = DeviceOnce::device();
  int grid = (dev >= 0 && dev < 64) ? grid_dev[dev].load() : 0;
  if (grid <= 0) {
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    int per_sm = 0, nsm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, 256, smem);
    if (e != cudaSuccess) return e;
    e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev < 0 ? 0 : dev);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) return cudaSuccess;
    grid = per_sm * nsm;
    if (dev >= 0 && dev < 64) grid_dev[dev].store(grid);
  }
  const long long units = 2ll * (MX * MY / kUnit) * fa.nbatch;
  if (units < grid) grid = (int)units;
  kern<<<grid, 256, smem, st>>>(fa, tmF, tmO);
  *used = true;
  return cudaGetLastError();
}

template <int MX, int MY>
cudaError_t launch_flow_same(const FlowArgs& fa, const CUtensorMap& tmF, const CUtensorMap& tmO, cudaStream_t st,
                             bool* used) {
  return fa.phi == fa.f ? launch_flow_one<MX, MY, true>(fa, tmF, tmO, st, used)
                        : launch_flow_one<MX, MY, false>(fa, tmF, tmO, st, used);
}

template <int MX>
cudaError_t launch_flow_y(int my, const FlowArgs& fa, const CUtensorMap& tmF, const CUtensorMap& tmO, cudaStream_t st,
                          bool* used) {
  switch (my) {
    case 64: return launch_flow_same<MX, 64>(fa, tmF, tmO, st, used);
    case 128: return launch_flow_same<MX, 128>(fa, tmF, tmO, st, used);
    case 256: return launch_flow_same<MX, 256>(fa, tmF, tmO, st, used);
    default: return cudaSuccess;
  }
}

}  // namespace

size_t h_batch_flow_counters(int nbatch) { return (size_t)nbatch + 2; }

cudaError_t launch_h_batch_flow(const FlowHArgs& a, cudaStream_t st, bool* used) {
  *used = false;
  const auto al = [](const void* p, unsigned n) { return (reinterpret_cast<uintptr_t>(p) & (n - 1u)) == 0; };
  if (a.nbatch < 1 || !a.ctr || (size_t)a.ctr_cap < h_batch_flow_counters(a.nbatch) || !al(a.f, 16) || !al(a.out, 16) ||
      !al(a.V, 16) || !al(a.phi, 8) || (a.stride & 1) || (a.vstride & 3))
    return cudaSuccess;
  const auto side = [](int m) { return m == 64 || m == 128 || m == 256; };
  if (!side(a.mx) || !side(a.my)) return cudaSuccess;
  if (2ll * (a.mx * a.my / kUnit) * a.nbatch > 0x3fffffff) return cudaSuccess;  // tickets are ints
  CUtensorMap tmF, tmO;
  if (!encode_flow_map(&tmF, a.f, a.mx, a.my, a.nbatch, a.stride) ||
      !encode_flow_map(&tmO, a.out, a.mx, a.my, a.nbatch, a.stride)) {
    cudaGetLastError();
    return cudaSuccess;
  }
  FlowArgs fa;
  fa.nbatch = a.nbatch;
  const long long lag = kFlowLagPoints / ((long long)a.mx * a.my);
  fa.lag = a.nbatch < lag ? a.nbatch : (int)lag;
  fa.stride = a.stride;
  fa.vstride = a.vstride;
  fa.eta = (float)a.eta;
  fa.omega = (float)a.omega;
  fa.xi = static_cast<const float*>(a.xi);
  fa.xiy = static_cast<const float*>(a.xiy);
  fa.xc = static_cast<const float*>(a.xc);
  fa.yc = static_cast<const float*>(a.yc);
  fa.V = static_cast<const float*>(a.V);
  fa.twx = static_cast<const float2*>(a.twx);
  fa.twy = static_cast<const float2*>(a.twy);
  fa.phi = static_cast<const float2*>(a.phi);
  fa.f = static_cast<const float2*>(a.f);
  fa.out = static_cast<float2*>(a.out);
  fa.ctr = a.ctr;
  fa.status = a.status;
  fa.polls = a.polls == 0 ? kTmaWaitLimit : (a.polls < 0 ? 0 : a.polls);
  switch (a.mx) {
    case 64: return launch_flow_y<64>(a.my, fa, tmF, tmO, st, used);
    case 128: return launch_flow_y<128>(a.my, fa, tmF, tmO, st, used);
    default: return launch_flow_y<256>(a.my, fa, tmF, tmO, st, used);
  }
}

}  // namespace gpe
