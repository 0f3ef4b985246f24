// kernels_jtj.cu -- the contraction [J r]^T [J r] of materialised FP32 rows (Eqs. JTJ, JTr), as a
// standalone operation on caller device buffers.
//
// Each CTA takes a contiguous range of rows and adds them in order: every output entry is one chain of
// multiply-adds per CTA, and the per-CTA partials are then added in CTA order in FP64 (deterministic for a
// given grid).
#include <algorithm>
#include <cstdio>
#include <mutex>
#include <string>

#include "../../include/trk.h"
#include "trk_internal.cuh"

namespace trk {

constexpr int kJBlock = 256;      // rows that make a CTA worth having (the grid's rule)
constexpr int kJStages = 4;       // pipeline stages
constexpr int kJLoaders = 128;    // threads that only load
constexpr int kJMaxBlocks = 296;

// The product is symmetric (a b and b a round alike), so only tiles that hold entries on or right of the
// diagonal are formed: TA x TB entries per thread, tile (i, j) with TB j + TB > TA i.  An entry's chain over
// the CTA's rows cannot be split (its rounding is part of the result), so what there is to fill the SM is
// the tiles.  Per SM and row that is bound by the FMAs' operand reads (fma.rn.f32x2: about 3 cycles per
// warp and sub-partition, measured) and by shared memory returning 32 floats per cycle: 8 x 4 tiles take
// 96 and 96 cycles at 73 columns (8 x 8 tiles: 113, and only half of the sub-partitions get one of the
// CTA's two warps of them, 206 in all; 4 x 4 ones: 84 and 112).  Fewer columns leave a CTA one to three warps
// whose rows are a chain that nothing else overlaps; there 4 x 4 tiles have the shorter one.  The row loop is
// unrolled by 16 so that its loads run ahead (62 cycles a row unrolled by 4).
//
// Four further warps copy the rows ahead with cp.async (16-byte pieces where base and ld allow, else 4-byte
// ones) through four stages, one barrier per STAGE rows; missing rows of the last stage are zeros.  Rows lie
// W floats apart, so that narrow ones share the memory among more of them: with 16 rows a stage whatever
// their width, up to 16 columns a stage was little but its barrier and a quarter of the loaders' lanes
// had a piece.  A row's pieces are spread over kLanes lanes.
// A call on one million rows, microseconds (64 rows staged between two barriers and the whole square formed; 16 rows
// a stage at any width; this): 8 columns 105, 115, 64; 32: 165, 112, 90; 48: 477, 155, 120; 73: 838, 221,
// 217.  20,000 rows of 8 columns: 15.6, 17.6, 15.5.
template <int TA, int TB>
struct JTiles {
  static __host__ __device__ int cols(int nc) { return (nc + TB - 1) / TB; }
  static __host__ __device__ int count(int nc) {
    int t = 0;
    for (int i = 0; TA * i < nc; ++i) t += cols(nc) - TA * i / TB;
    return t;
  }
  static __host__ __device__ int compute_threads(int nc) { return (count(nc) + 31) / 32 * 32; }
};

__device__ __forceinline__ void cp_async4(void* s, const void* g) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"((uint32_t)__cvta_generic_to_shared(s)),
               "l"(__cvta_generic_to_global(g))
               : "memory");
}
// 16 bytes of shared memory from `bytes` (<= 16) of global memory, the rest zeros
__device__ __forceinline__ void cp_async16_part(void* s, const void* g, int bytes) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"((uint32_t)__cvta_generic_to_shared(s)),
               "l"(__cvta_generic_to_global(g)), "r"(bytes)
               : "memory");
}

template <int N>
__device__ __forceinline__ void load_floats(const float* p, float (&v)[N]) {
#pragma unroll
  for (int k = 0; k < N; k += 4) {
    const float4 q = *reinterpret_cast<const float4*>(p + k);
    v[k] = q.x, v[k + 1] = q.y, v[k + 2] = q.z, v[k + 3] = q.w;
  }
}

template <int TA, int TB, int W, int STAGE>
__global__ void __launch_bounds__(kJLoaders + 128) k_jtj_rows(const float* __restrict__ rows, int n, int nc, int ld,
                                                            int rows_per_block, bool vec, float* __restrict__ partial) {
  // (W >= nc, a multiple of 16; tiles past nc read a row's leftovers, which count nowhere)
  constexpr int kLanes = W <= 16 ? 4 : W <= 32 ? 8 : W <= 64 ? 16 : 32;
  constexpr int kRowsAtOnce = kJLoaders / kLanes, kRowsEach = STAGE / kRowsAtOnce;
  static_assert(STAGE % kRowsAtOnce == 0 && STAGE % 16 == 0, "whole rounds of the loaders and of the row loop");
  __shared__ __align__(16) float st[kJStages][STAGE][W];
  const int tid = threadIdx.x, nthr = blockDim.x, ncomp = nthr - kJLoaders;
  const int r0 = blockIdx.x * rows_per_block, r1 = min(n, r0 + rows_per_block);
  const int nst = r1 > r0 ? (r1 - r0 + STAGE - 1) / STAGE : 0;
  // this thread's tile
  int ti = 0, tj = tid;
  const int ncols = JTiles<TA, TB>::cols(nc);
  while (TA * ti < nc && tj >= ncols - TA * ti / TB) {
    tj -= ncols - TA * ti / TB;
    ++ti;
  }
  tj += TA * ti / TB;
  const bool comp = tid < ncomp && TA * ti < nc;
  const int pieces = vec ? (nc + 3) / 4 : nc, lt = tid - ncomp;
  auto load = [&](int q) {  // stage q, by the loader threads
    const int base = r0 + q * STAGE, cnt = min(STAGE, r1 - base), row = lt / kLanes;
    for (int piece = lt % kLanes; piece < pieces; piece += kLanes) {
      const int col = vec ? 4 * piece : piece, bytes = vec ? 4 * min(4, nc - col) : 4;
      const float* src = rows + (size_t)(base + row) * ld + col;
      float* dst = &st[q % kJStages][row][col];
      const size_t step = (size_t)kRowsAtOnce * ld;
      if (cnt == STAGE) {
#pragma unroll
        for (int i = 0; i < kRowsEach; ++i) {
          if (vec) cp_async16_part(dst + i * kRowsAtOnce * W, src + i * step, bytes);
          else cp_async4(dst + i * kRowsAtOnce * W, src + i * step);
        }
      } else {
        for (int i = 0; row + i * kRowsAtOnce < cnt; ++i) {
          if (vec) cp_async16_part(dst + i * kRowsAtOnce * W, src + i * step, bytes);
          else cp_async4(dst + i * kRowsAtOnce * W, src + i * step);
        }
      }
    }
    for (int e = cnt * W + lt; e < STAGE * W; e += kJLoaders) st[q % kJStages][0][e] = 0.f;
  };
  unsigned long long acc[TA][TB / 2];
#pragma unroll
  for (int a = 0; a < TA; ++a)
#pragma unroll
    for (int b = 0; b < TB / 2; ++b) acc[a][b] = 0ull;
  if (tid >= ncomp) {
    for (int q = 0; q < kJStages - 1; ++q) {
      if (q < nst) load(q);
      asm volatile("cp.async.commit_group;\n" ::: "memory");
    }
  }
  for (int q = 0; q < nst; ++q) {
    if (tid >= ncomp) asm volatile("cp.async.wait_group %0;\n" ::"n"(kJStages - 2) : "memory");
    __syncthreads();  // stage q has arrived; every thread is done with stage q - 1, which is loaded next
    if (tid >= ncomp) {
      if (q + kJStages - 1 < nst) load(q + kJStages - 1);
      asm volatile("cp.async.commit_group;\n" ::: "memory");
    } else if (comp) {
      const float* pa = &st[q % kJStages][0][TA * ti];
      const float* pb = &st[q % kJStages][0][TB * tj];
#pragma unroll 16
      for (int s = 0; s < STAGE; ++s) {
        float ra[TA], rb[TB];
        load_floats(pa + s * W, ra);
        load_floats(pb + s * W, rb);
        unsigned long long B2[TB / 2];
#pragma unroll
        for (int b = 0; b < TB / 2; ++b)
          asm("mov.b64 %0, {%1, %2};" : "=l"(B2[b]) : "f"(rb[2 * b]), "f"(rb[2 * b + 1]));
#pragma unroll
        for (int a = 0; a < TA; ++a) {
          unsigned long long A2;
          asm("mov.b64 %0, {%1, %1};" : "=l"(A2) : "f"(ra[a]));
#pragma unroll
          for (int b = 0; b < TB / 2; ++b)
            asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc[a][b]) : "l"(A2), "l"(B2[b]));
        }
      }
    }
  }
  if (!comp) return;
  float* out = partial + (size_t)blockIdx.x * nc * nc;
#pragma unroll
  for (int a = 0; a < TA; ++a)
#pragma unroll
    for (int b = 0; b < TB; ++b) {
      const int r = TA * ti + a, c = TB * tj + b;
      float lo, hi;
      asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(acc[a][b / 2]));
      if (c < nc && r <= c) out[r * nc + c] = b & 1 ? hi : lo;  // the upper triangle (the reduction mirrors)
    }
}

// FP64 sum of the nblk partials in a fixed order: warp w of the block's S adds partials w, w + S, ... (all
// its loads of a round in flight), warp 0 the warps' sums.  kUpper: the partials hold the upper triangle,
// whose entries are written to both places.
template <bool kUpper>
__global__ void __launch_bounds__(1024) k_jtj_reduce(const float* __restrict__ partial, int nblk, int nc,
                                                     double* __restrict__ out) {
  __shared__ double sm[32][33];
  constexpr int kBatch = 8;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, S = blockDim.x >> 5;
  const int n2 = nc * nc, total = kUpper ? nc * (nc + 1) / 2 : n2, u = blockIdx.x * 32 + lane;
  int r = 0, c = 0;
  if (kUpper && u < total) {  // counted from the end, row nc - 1 - m holds m + 1 entries
    const int v = total - 1 - u;
    int m = (int)((sqrtf(8.f * (float)v + 1.f) - 1.f) * 0.5f);
    if ((m + 1) * (m + 2) / 2 <= v) ++m;
    if (m * (m + 1) / 2 > v) --m;
    r = nc - 1 - m;
    c = nc - 1 - (v - m * (m + 1) / 2);
  }
  const int e = kUpper ? r * nc + c : u;
  double s = 0.0;
  for (int b0 = w; b0 < nblk; b0 += kBatch * S) {
    float q[kBatch];
    bool other = false;
#pragma unroll
    for (int k = 0; k < kBatch; ++k) q[k] = b0 + k * S < nblk && u < total ? partial[(size_t)(b0 + k * S) * n2 + e] : 0.f;
    double d[kBatch];
#pragma unroll
    for (int k = 0; k < kBatch; ++k) d[k] = widen(q[k], other);
    if (__any_sync(0xffffffffu, other)) {
#pragma unroll
      for (int k = 0; k < kBatch; ++k) d[k] = (double)q[k];
    }
#pragma unroll
    for (int k = 0; k < kBatch; ++k)
      if (b0 + k * S < nblk) s += d[k];
  }
  sm[w][lane] = s;
  __syncthreads();
  if (w != 0 || u >= total) return;
  double t = 0.0;
#pragma unroll 8
  for (int k = 0; k < S; ++k) t += sm[k][lane];
  out[e] = t;
  if (kUpper) out[c * nc + r] = t;
}

template <bool kUpper>
static void launch_reduce(const float* partial, int nblk, int nc, double* out, cudaStream_t st) {
  const int total = kUpper ? nc * (nc + 1) / 2 : nc * nc;
  k_jtj_reduce<kUpper><<<(total + 31) / 32, 32 * std::min(32, std::max(1, (nblk + 1) / 2)), 0, st>>>(partial, nblk, nc, out);
}

template <int TA, int TB, int W, int STAGE>
static void launch_rows(const float* rows, int n, int nc, int ld, int nblk, int rpb, bool vec, float* partial,
                        cudaStream_t st) {
  k_jtj_rows<TA, TB, W, STAGE><<<nblk, JTiles<TA, TB>::compute_threads(nc) + kJLoaders, 0, st>>>(rows, n, nc, ld, rpb, vec, partial);
}

// Launches the two kernels with nblk CTAs and the given partial buffer (nblk * nc * nc floats).
cudaError_t jtj_rows_launch(const float* rows, int n, int nc, int ld, double* out, int nblk, float* partial,
                            cudaStream_t st) {
  const int rpb = (n + nblk - 1) / nblk;
  const bool vec = ld % 4 == 0 && reinterpret_cast<uintptr_t>(rows) % 16 == 0;
  // 4 x 4 tiles up to 48 columns: there 3,001, 50,010 and a million rows take 13, 18.6 and 120 us, with 8 x 4 ones
  // 16.6, 22.7 and 155; at 56 columns 15, 22.7 and 159 against 16.6, 22.8 and 156
  if (nc <= 16) launch_rows<4, 4, 16, 64>(rows, n, nc, ld, nblk, rpb, vec, partial, st);
  else if (nc <= 32) launch_rows<4, 4, 32, 32>(rows, n, nc, ld, nblk, rpb, vec, partial, st);
  else if (nc <= 48) launch_rows<4, 4, 48, 32>(rows, n, nc, ld, nblk, rpb, vec, partial, st);
  else launch_rows<8, 4, kMaxNP, 16>(rows, n, nc, ld, nblk, rpb, vec, partial, st);
  launch_reduce<true>(partial, nblk, nc, out, st);
  return cudaGetLastError();
}

// Fixed-order FP64 sum of nslots partials of nc x nc floats into out.
cudaError_t jtj_reduce_launch(const float* partial, int nslots, int nc, double* out, cudaStream_t st) {
  launch_reduce<false>(partial, nslots, nc, out, st);
  return cudaGetLastError();
}

int jtj_rows_blocks(int n) { return std::max(1, std::min(kJMaxBlocks, (n + kJBlock - 1) / kJBlock)); }

// ---------------------------------------------------------------------------------------------
// Allocation-free variant: the per-CTA partials live in a fixed file-scope device array (at most
// kNoAllocBlocks CTAs x 80 x 80 floats, 3.9 MB held by every device that loads the library).  Each CTA
// overwrites its whole partial on every call, so nothing has to be cleared between calls.
// ---------------------------------------------------------------------------------------------
constexpr int kNoAllocBlocks = 152;
static __device__ __align__(256) float g_noalloc_partial[kNoAllocBlocks * kMaxNP * kMaxNP];

constexpr int kMaxDevices = 64;
static float* g_noalloc_ptr[kMaxDevices];
static std::mutex g_noalloc_mutex;

// Device address of g_noalloc_partial on the current device (looked up once per device).  In host code
// the symbol itself is only a host-side stand-in, never a device address.
static cudaError_t noalloc_scratch(float** out) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> lock(g_noalloc_mutex);
  if (!g_noalloc_ptr[dev]) {
    float* p = nullptr;
    e = cudaGetSymbolAddress(reinterpret_cast<void**>(&p), g_noalloc_partial);
    if (e != cudaSuccess) return e;
    g_noalloc_ptr[dev] = p;
  }
  *out = g_noalloc_ptr[dev];
  return cudaSuccess;
}

}  // namespace trk

extern "C" {

trk_status trk_jtj_rows(const float* d_rows, int32_t n_rows, int32_t n_cols, int32_t ld, double* d_out,
                        void* cuda_stream) {
  if (!d_rows || !d_out || n_rows < 0 || n_cols <= 0 || n_cols > trk::kMaxNP || ld < n_cols)
    return trk::set_error(TRK_ERR_INVALID_ARG, "trk_jtj_rows: bad arguments");
  cudaStream_t st = (cudaStream_t)cuda_stream;
  const int nblk = trk::jtj_rows_blocks(n_rows);
  float* partial = nullptr;
  cudaError_t e = cudaMallocAsync(&partial, sizeof(float) * (size_t)nblk * n_cols * n_cols, st);
  if (e != cudaSuccess)
    return trk::set_error(e == cudaErrorMemoryAllocation ? TRK_ERR_OOM : TRK_ERR_CUDA, cudaGetErrorString(e));
  e = trk::jtj_rows_launch(d_rows, n_rows, n_cols, ld, d_out, nblk, partial, st);
  const cudaError_t f = cudaFreeAsync(partial, st);
  if (e != cudaSuccess) return trk::set_error(TRK_ERR_CUDA, cudaGetErrorString(e));
  if (f != cudaSuccess) return trk::set_error(TRK_ERR_CUDA, cudaGetErrorString(f));
  return TRK_OK;
}

trk_status trk_jtj_rows_noalloc(const float* d_rows, int32_t n_rows, int32_t n_cols, int32_t ld, double* d_out,
                                void* cuda_stream) {
  if (!d_rows || !d_out || n_rows < 0 || ld < n_cols)
    return trk::set_error(TRK_ERR_INVALID_ARG, "trk_jtj_rows_noalloc: bad arguments");
  if (n_cols <= 0 || n_cols > trk::kMaxNP)
    return trk::set_error(TRK_ERR_INVALID_ARG, "trk_jtj_rows_noalloc: n_cols must be in [1, 80] (fixed scratch size)");
  float* partial = nullptr;
  cudaError_t e = trk::noalloc_scratch(&partial);
  if (e != cudaSuccess) return trk::set_error(TRK_ERR_CUDA, cudaGetErrorString(e));
  const int nblk = std::min(trk::kNoAllocBlocks, trk::jtj_rows_blocks(n_rows));
  e = trk::jtj_rows_launch(d_rows, n_rows, n_cols, ld, d_out, nblk, partial, (cudaStream_t)cuda_stream);
  if (e != cudaSuccess) return trk::set_error(TRK_ERR_CUDA, cudaGetErrorString(e));
  return TRK_OK;
}

}  // extern "C"
