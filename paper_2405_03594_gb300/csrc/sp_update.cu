// sp_update.cu -- sp_masked_update: the masked weight step of Algorithm 1 (Sec. 2.1)
// applied directly to the compressed form.
//
// Sparse pretraining and fine-tuning keep the pruning mask fixed: a step computes
// theta <- theta - lr * (grad o Mask), so masked-out weights stay zero and only the kept
// weights change.  In the bitmask format the kept weights are exactly the stored values,
// so the step rewrites the packed values in place and leaves masks, offsets, padding and
// the quarter index untouched; the matrix never has to be decompressed.
//
// Arithmetic per kept (n, k): w <- bf16_rne(fma(-lr, grad[n, k], w)) in float32, one
// fused multiply-add and one rounding.  The dense float32 gradient is the large stream
// (4 bytes per weight against ~0.7 bytes of compressed weight at 70 % sparsity), so the
// kernel is laid out for it: one CTA of 8 warps per 128 x 64 chunk, a thread owning eight
// columns of four rows, whose gradients (one 32-byte load each) are all requested before
// anything else.  The chunk comes to shared memory by one bulk copy; a thread walks the
// kept columns of its eight (sp_expand.cuh's scheme), so a dropped column costs no shared
// memory access, updates the values in place there, and the CTA writes the value area back
// with 16-byte stores.  The walk is what the instruction budget goes to: a gradient tile
// costs ~0.3 us of the SM's issue slots against 0.75 us of its share of the HBM rate.
// Measured, 4096 x 11008 at 70 %, the step and the weight read back dense: 105.5 us with the
// gradient in two-column pieces and the values read and written in global memory, 64.3 us so.
// Five CTAs per SM (48 registers, 12 bytes of spills) against four: 22016 x 4096 78.5 -> 74.2 us;
// 512 threads per CTA with half the rows each 87.  That moves 480 MB, the whole gradient among
// them (6.5 TB/s); 460 MB would do, since 6 % of its 32-byte sectors hold no kept weight (6.2).
#include "sp_internal.cuh"

namespace sp {
namespace {

constexpr int kUpdThreads = 256;  // 8 warps per chunk, 16 rows each, 4 rows at a time
constexpr int kUpdIters = kRows / (kUpdThreads / 8);

// Eight consecutive gradients: one 32-byte load, or two of 16 bytes where the caller's
// pointer is only 16-byte aligned (rows are a multiple of 32 bytes apart: K % 8 == 0).
template <bool WIDE>
__device__ __forceinline__ void load_grad8(const float* p, float (&g)[8]) {
  if constexpr (WIDE) {
    asm volatile("ld.global.nc.L1::no_allocate.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=f"(g[0]), "=f"(g[1]), "=f"(g[2]), "=f"(g[3]), "=f"(g[4]), "=f"(g[5]), "=f"(g[6]), "=f"(g[7])
                 : "l"(p));
  } else {
    const float4 a = __ldcs(reinterpret_cast<const float4*>(p)), b = __ldcs(reinterpret_cast<const float4*>(p) + 1);
    g[0] = a.x, g[1] = a.y, g[2] = a.z, g[3] = a.w, g[4] = b.x, g[5] = b.y, g[6] = b.z, g[7] = b.w;
  }
}

// Column I of the walk: a kept column's value (bf16 bits) from shared address pa, which
// advances.
template <int I>
__device__ __forceinline__ void walk_load(uint32_t m, uint32_t& pa, uint16_t (&v)[8]) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t.reg .b32 t;\n\t"
      "and.b32 t, %2, %3;\n\t"
      "setp.ne.b32 p, t, 0;\n\t"
      "mov.b16 %0, 0;\n\t"
      "@p ld.shared.b16 %0, [%1];\n\t"
      "@p add.u32 %1, %1, 2;\n\t}"
      : "=h"(v[I]), "+r"(pa)
      : "r"(m), "n"(1u << I)
      : "memory");
  if constexpr (I + 1 < 8) walk_load<I + 1>(m, pa, v);
}
template <int I>
__device__ __forceinline__ void walk_store(uint32_t m, uint32_t& pa, const uint16_t (&v)[8]) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t.reg .b32 t;\n\t"
      "and.b32 t, %1, %2;\n\t"
      "setp.ne.b32 p, t, 0;\n\t"
      "@p st.shared.b16 [%0], %3;\n\t"
      "@p add.u32 %0, %0, 2;\n\t}"
      : "+r"(pa)
      : "r"(m), "n"(1u << I), "h"(v[I])
      : "memory");
  if constexpr (I + 1 < 8) walk_store<I + 1>(m, pa, v);
}

template <bool WIDE>
__global__ void __launch_bounds__(kUpdThreads, 5)
    masked_update_kernel(uint8_t* __restrict__ buf, const uint64_t* __restrict__ off,
                         const uint64_t* __restrict__ qidx, const float* __restrict__ grad, float neg_lr, int64_t N,
                         int64_t K, int T, uint64_t timeout_ns, int* status) {
  extern __shared__ __align__(128) uint8_t chunk[];
  __shared__ uint64_t bar;
  __shared__ uint32_t s_start[2 * kRows];  // byte offset of each 32-column half row's first value
  const int64_t c = blockIdx.x;
  const int64_t rb = c / T, t = c % T;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int seg = lane & 7;  // the thread's columns: 8 * seg .. 8 * seg + 7 of the tile
  const int64_t col = (int64_t)kTileK * t + 8 * seg;
  const int row0 = 16 * warp + (lane >> 3);  // rows row0, row0 + 4, row0 + 8, row0 + 12

  const uint64_t o0 = off[c], o1 = off[c + 1];
  if (tid == 0) {
    mbar_init(&bar, 1);
    fence_barrier_init();
    mbar_arrive_expect_tx(&bar, (uint32_t)(o1 - o0));
    bulk_g2s(chunk, buf + o0, (uint32_t)(o1 - o0), &bar);
  }
  float g[kUpdIters][8];
#pragma unroll
  for (int i = 0; i < kUpdIters; ++i) {
    const int64_t n = rb * kRows + row0 + 4 * i;
#pragma unroll
    for (int j = 0; j < 8; ++j) g[i][j] = 0.f;
    if (n < N && col < K) load_grad8<WIDE>(grad + n * K + col, g[i]);
  }
  const uint64_t qi = qidx[c];
  __syncthreads();
  const bool ok = __all_sync(0xffffffffu, mbar_wait(&bar, 0, timeout_ns));
  if (!ok) set_status(status, kStatusTimeout);
  if (tid < kRows && ok) {  // start of every half row: warp scan, quarter index before it
    const uint2 m = reinterpret_cast<const uint2*>(chunk)[tid];
    const int plo = __popc(m.x), pc = plo + __popc(m.y);
    int incl = pc;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const int u = __shfl_up_sync(0xffffffffu, incl, d);
      if (lane >= d) incl += u;
    }
    const int before = warp == 0 ? 0 : (int)((qi >> (16 * (warp - 1))) & 0xffffu);
    const uint32_t e0 = (uint32_t)(before + incl - pc);
    reinterpret_cast<uint2*>(s_start)[tid] = make_uint2(2 * e0, 2 * (e0 + (uint32_t)plo));
  }
  // a chunk that did not arrive in time is left as it is
  if (!__syncthreads_and(ok)) return;

  const uint32_t* words = reinterpret_cast<const uint32_t*>(chunk);
  const uint32_t vbase = smem_u32(chunk) + kMaskBytes;
  const int sh = 8 * (seg & 3);
  const uint32_t below = (1u << sh) - 1u;
#pragma unroll
  for (int i = 0; i < kUpdIters; ++i) {
    const int r = row0 + 4 * i;
    const uint32_t w = words[2 * r + (seg >> 2)];
    const uint32_t p0 = vbase + s_start[2 * r + (seg >> 2)] + 2u * (uint32_t)__popc(w & below);
    uint32_t m = w >> sh;
    // A well-formed chunk has no bits in rows >= N or columns >= K; skip any such bit
    // rather than use a gradient entry that was not read.
    if (!(rb * kRows + r < N && col < K)) m = 0;
    uint16_t v[8];
    uint32_t pa = p0;
    walk_load<0>(m, pa, v);
#pragma unroll
    for (int j = 0; j < 8; ++j)
      v[j] = float_to_bf16_bits_rn(__fmaf_rn(neg_lr, g[i][j], bf16_bits_to_float(v[j])));
    pa = p0;
    walk_store<0>(m, pa, v);
  }
  __syncthreads();
  uint4* dst = reinterpret_cast<uint4*>(buf + o0 + kMaskBytes);
  const uint4* src = reinterpret_cast<const uint4*>(chunk + kMaskBytes);
  const int n16 = (int)((o1 - o0 - kMaskBytes) / 16);
  for (int i = tid; i < n16; i += kUpdThreads) dst[i] = src[i];
}

bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

}  // namespace
}  // namespace sp

using namespace sp;

extern "C" sp_status sp_masked_update(sp_matrix* h, const float* grad_dev, float lr, void* stream) {
  if (!h || h->magic != SP_MAGIC) return SP_ERR_BAD_HANDLE;
  if (!grad_dev || !isfinite(lr)) return SP_ERR_INVALID_ARG;
  if (h->dtype != SP_BF16) return SP_ERR_UNSUPPORTED;
  if (!aligned16(grad_dev)) return SP_ERR_ALIGNMENT;
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess) {
    cudaGetLastError();
    return SP_ERR_CUDA;
  }
  if (dev != h->device) return SP_ERR_INVALID_ARG;
  const int64_t C = (int64_t)h->RB * h->T;  // < 2^31, checked by sp_compress
  if (h->nnz == 0) return SP_OK;
  auto kern = (reinterpret_cast<uintptr_t>(grad_dev) & 31u) == 0 ? masked_update_kernel<true>
                                                                : masked_update_kernel<false>;
  kern<<<(unsigned)C, kUpdThreads, (size_t)h->max_chunk, (cudaStream_t)stream>>>(
      h->d_buf, h->d_off, h->d_qidx, grad_dev, -lr, h->N, h->K, h->T, wait_timeout_ns(), device_status_ptr());
  if (cudaGetLastError() != cudaSuccess) return SP_ERR_CUDA;
  h->weights_written = 1;
  return SP_OK;
}
