// sp_format.cu -- building and expanding the bitmask-compressed weight.
//
// sp_compress turns a dense weight plus keep-mask into the chunked format of
// include/sp.h (the submatrix storage of Sec. 2.4.2: dense nonzeros plus a
// bitmask per submatrix, with the per-block bitmask encoding of Sec. 2.4.1):
//   1. count:   one CTA per chunk reads its mask bytes (8 per lane, whole row segments per
//               warp), packs them into the 64-bit row masks and counts the kept entries of
//               the chunk and of its four 32-row quarters;
//   2. scan:    one CTA: exclusive scan of padded chunk sizes -> byte offsets;
//   3. (host)   read the total size, allocate the buffer;
//   4. scatter: one CTA per chunk: a popcount scan gives each row's first value slot, the
//               kept values are packed in shared memory in ascending column order behind the
//               masks, and the finished chunk (padding zeroed) leaves in 16-byte stores.
// All of them are bound by memory: dense weight and mask in, compressed form out.  (With one
// thread reading or writing a row's 64 columns one at a time, compressing 4096 x 4096 bf16 at
// 70 % and reading it back dense took 149 us, against 110 us this way; most of the rest is the
// call's two synchronisations and its allocations.)
// sp_decompress is the inverse (described at its kernel).
#include <algorithm>

#include "sp_expand.cuh"

namespace sp {
namespace {

// Bit i of the result: byte i of v is nonzero.
__device__ __forceinline__ uint32_t nonzero_bytes(uint32_t v) {
  const uint32_t x = (((v & 0x7f7f7f7fu) + 0x7f7f7f7fu) | v) & 0x80808080u;  // bit 7 of each nonzero byte
  // bits 0, 8, 16, 24 of x >> 7 land in bits 24 .. 27 of the product; no two terms meet
  return ((x >> 7) * 0x01020408u) >> 24 & 0xfu;
}

// Also writes the chunk's quarter index (kept entries before rows 32, 64 and 96, and in the
// whole chunk; 16 bits each).  Warp q takes rows 32q .. 32q+31, four at a time; a lane packs
// eight columns of one row.
__global__ void __launch_bounds__(kRows) count_kernel(const uint8_t* __restrict__ mask, int64_t N, int64_t K, int T,
                                                      uint8_t* __restrict__ masks_out,
                                                      uint64_t* __restrict__ qidx) {
  __shared__ int s_q[kRows / 32];
  const int64_t c = blockIdx.x;
  const int64_t rb = c / T, t = c % T;
  const int lane = threadIdx.x & 31, q = threadIdx.x >> 5;
  const int64_t col = (int64_t)kTileK * t + 8 * (lane & 7);
  const int r0 = 32 * q + (lane >> 3);
  uint2 v[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int64_t n = rb * kRows + r0 + 4 * i;
    v[i] = make_uint2(0u, 0u);
    if (n < N && col < K) v[i] = __ldcs(reinterpret_cast<const uint2*>(mask + n * K + col));
  }
  int kept = 0;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const uint32_t m = nonzero_bytes(v[i].x) | nonzero_bytes(v[i].y) << 4;
    masks_out[c * kMaskBytes + 8 * (r0 + 4 * i) + (lane & 7)] = (uint8_t)m;
    kept += __popc(m);
  }
  kept = (int)__reduce_add_sync(0xffffffffu, (unsigned)kept);
  if (lane == 0) s_q[q] = kept;
  __syncthreads();
  if (threadIdx.x == 0) {
    const int a = s_q[0], b = a + s_q[1], d = b + s_q[2], total = d + s_q[3];
    qidx[c] = (uint64_t)a | ((uint64_t)b << 16) | ((uint64_t)d << 32) | ((uint64_t)total << 48);
  }
}

// meta[0] = total bytes, meta[1] = largest chunk, meta[2] = kept entries, meta[3] = most kept
// entries in a quarter, all from the chunks' quarter indices.  Thread i owns the
// run of ceil(C / 1024) chunks from i * ceil(C / 1024): one pass sums the runs, one block scan
// gives their starts, a second pass writes the offsets.
__global__ void __launch_bounds__(1024) scan_kernel(const uint64_t* __restrict__ qidx, int64_t C, int esize,
                                                    uint64_t* __restrict__ off, uint64_t* __restrict__ meta) {
  __shared__ uint64_t s_warp[32];
  __shared__ uint64_t s_max[32], s_nnz[32];
  __shared__ uint32_t s_quarter[32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t run = (C + 1023) / 1024;
  const int64_t c0 = imin64(run * threadIdx.x, C), c1 = imin64(c0 + run, C);
  uint64_t sum = 0, mx = 0, nnz = 0;
  uint32_t quarter = 0;
  for (int64_t i = c0; i < c1; ++i) {
    const uint64_t qi = qidx[i], kept = qi >> 48;
    const uint32_t a = (uint32_t)(qi & 0xffffu), b = (uint32_t)(qi >> 16) & 0xffffu, d = (uint32_t)(qi >> 32) & 0xffffu;
    quarter = max(quarter, max(max(a, b - a), max(d - b, (uint32_t)kept - d)));
    const uint64_t sz = (kMaskBytes + kept * esize + 15) / 16 * 16;
    mx = max(mx, sz);
    nnz += kept;
    sum += sz;
  }
  uint64_t incl = sum;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const uint64_t u = __shfl_up_sync(0xffffffffu, incl, d);
    if (lane >= d) incl += u;
  }
  if (lane == 31) s_warp[warp] = incl;
  for (int d = 16; d > 0; d >>= 1) {
    mx = max(mx, __shfl_down_sync(0xffffffffu, mx, d));
    nnz += __shfl_down_sync(0xffffffffu, nnz, d);
  }
  quarter = __reduce_max_sync(0xffffffffu, quarter);
  if (lane == 0) {
    s_quarter[warp] = quarter;
    s_max[warp] = mx;
    s_nnz[warp] = nnz;
  }
  __syncthreads();
  uint64_t o = incl - sum;
  for (int w = 0; w < warp; ++w) o += s_warp[w];
  for (int64_t i = c0; i < c1; ++i) {
    off[i] = o;
    o += (kMaskBytes + (qidx[i] >> 48) * esize + 15) / 16 * 16;
  }
  if (threadIdx.x == 0) {
    uint64_t all = 0, a = 0, b = 0;
    uint32_t most = 0;
    for (int w = 0; w < 32; ++w) {
      most = max(most, s_quarter[w]);
      all += s_warp[w];
      a = max(a, s_max[w]);
      b += s_nnz[w];
    }
    off[C] = all;
    meta[0] = all;
    meta[1] = a;
    meta[2] = b;
    meta[3] = most;
  }
}

// One kept column (bit I of m) of a lane's segment: its value goes to shared address pa,
// which advances.
template <int ES, int I>
__device__ __forceinline__ void pack_column(uint32_t m, uint32_t& pa, uint32_t word) {
  if constexpr (ES == 2) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t.reg .b32 t;\n\t.reg .b16 l, h;\n\t"
        "mov.b32 {l, h}, %2;\n\t"
        "and.b32 t, %1, %3;\n\t"
        "setp.ne.b32 p, t, 0;\n\t"
        "@p st.shared.b16 [%0], l;\n\t"
        "@p add.u32 %0, %0, 2;\n\t"
        "and.b32 t, %1, %4;\n\t"
        "setp.ne.b32 p, t, 0;\n\t"
        "@p st.shared.b16 [%0], h;\n\t"
        "@p add.u32 %0, %0, 2;\n\t}"
        : "+r"(pa)
        : "r"(m), "r"(word), "n"(1u << (2 * I)), "n"(2u << (2 * I))
        : "memory");
  } else {
#pragma unroll
    for (int b = 0; b < 4; ++b) {
      if ((m >> (4 * I + b)) & 1u) {
        asm volatile("st.shared.u8 [%0], %1;" ::"r"(pa), "r"(word >> (8 * b)) : "memory");
        ++pa;
      }
    }
  }
}

// Warp q packs rows 32q .. 32q+31; a lane takes 16 bytes (16 / ES columns) of one row at a
// time, so the dense weight is read in whole row segments.
template <int ES>
__global__ void __launch_bounds__(kRows) scatter_kernel(const uint8_t* __restrict__ w, int64_t N, int64_t K, int T,
                                                        const uint64_t* __restrict__ masks,
                                                        const uint64_t* __restrict__ off,
                                                        const uint64_t* __restrict__ qidx, uint8_t* __restrict__ buf) {
  extern __shared__ __align__(128) uint8_t chunk[];
  __shared__ uint32_t s_start[2 * kRows];  // byte offset of each 32-column half row's first value
  constexpr int kCols = 16 / ES;
  constexpr int kSegs = kTileK / kCols;  // lanes per row; also the warp's passes over its rows
  const int64_t c = blockIdx.x;
  const int64_t rb = c / T, t = c % T;
  const int tid = threadIdx.x, lane = tid & 31, q = tid >> 5;
  const int seg = lane % kSegs;
  const int64_t col = (int64_t)kTileK * t + kCols * seg;
  uint4 v[kSegs];
#pragma unroll
  for (int i = 0; i < kSegs; ++i) {
    const int64_t n = rb * kRows + 32 * q + i * (32 / kSegs) + lane / kSegs;
    v[i] = make_uint4(0u, 0u, 0u, 0u);
    if (n < N && col < K) {
      const uint8_t* src = w + (n * K + col) * ES;
      // an int8 row starts on an 8-byte boundary only, and its last segment may be half
      if (ES == 2 || K % 16 == 0) {
        v[i] = __ldcs(reinterpret_cast<const uint4*>(src));
      } else {
        const uint2 a = *reinterpret_cast<const uint2*>(src);
        v[i].x = a.x, v[i].y = a.y;
        if (col + 8 < K) {
          const uint2 b = *reinterpret_cast<const uint2*>(src + 8);
          v[i].z = b.x, v[i].w = b.y;
        }
      }
    }
  }
  const uint64_t o0 = off[c], o1 = off[c + 1], qi = qidx[c];
  {
    const uint64_t m = masks[c * kRows + tid];
    reinterpret_cast<uint64_t*>(chunk)[tid] = m;
    const int plo = __popc((uint32_t)m), pc = __popcll(m);
    int incl = pc;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const int u = __shfl_up_sync(0xffffffffu, incl, d);
      if (lane >= d) incl += u;
    }
    const int before = q == 0 ? 0 : (int)((qi >> (16 * (q - 1))) & 0xffffu);
    const uint32_t e0 = (uint32_t)(before + incl - pc);
    reinterpret_cast<uint2*>(s_start)[tid] = make_uint2(e0 * ES, (e0 + (uint32_t)plo) * ES);
  }
  // the chunk ends in up to 15 bytes of zero padding
  const uint32_t size = (uint32_t)(o1 - o0), used = kMaskBytes + (uint32_t)(qi >> 48) * ES;
  if (used + tid < size) chunk[used + tid] = 0;
  __syncwarp();
  const uint32_t* words = reinterpret_cast<const uint32_t*>(chunk);
  const int half = seg / (kSegs / 2), sh = kCols * (seg % (kSegs / 2));
  const uint32_t below = (1u << sh) - 1u;
  const uint32_t vbase = smem_u32(chunk) + kMaskBytes;
#pragma unroll
  for (int i = 0; i < kSegs; ++i) {
    const int r = 32 * q + i * (32 / kSegs) + lane / kSegs;
    const uint32_t mw = words[2 * r + half];
    uint32_t pa = vbase + s_start[2 * r + half] + (uint32_t)(ES * __popc(mw & below));
    const uint32_t m = mw >> sh;
    pack_column<ES, 0>(m, pa, v[i].x);
    pack_column<ES, 1>(m, pa, v[i].y);
    pack_column<ES, 2>(m, pa, v[i].z);
    pack_column<ES, 3>(m, pa, v[i].w);
  }
  __syncthreads();
  uint4* dst = reinterpret_cast<uint4*>(buf + o0);
  const uint4* src = reinterpret_cast<const uint4*>(chunk);
  for (int i = tid; i < (int)(size / 16); i += kRows) dst[i] = src[i];
}

// Dense masked weight from the compressed form.  Bound by memory: the compressed bytes in,
// N * K * ES bytes out, so the kernel is laid out for the dense stores.  One CTA of four
// warps per chunk: one bulk copy brings the chunk to shared memory, warp q expands rows
// 32q .. 32q+31 on its own (the quarter index gives its first value, one warp scan the start
// of each 32-column half row), and a lane expands 16 bytes of one row, so a warp stores
// whole 64 * ES byte row segments, 16 bytes per lane.  One thread per row storing its 64
// columns two bytes at a time touched 32 rows per store.  Measured, 22016 x 4096 bf16 at 70 %:
// 654 -> 39.1 us (245 MB in and out, 6.3 TB/s).
template <int ES>
__global__ void __launch_bounds__(kRows) decompress_kernel(const uint8_t* __restrict__ buf,
                                                           const uint64_t* __restrict__ off,
                                                           const uint64_t* __restrict__ qidx, int64_t N, int64_t K,
                                                           int T, uint8_t* __restrict__ out, uint64_t timeout_ns,
                                                           int* status) {
  extern __shared__ __align__(128) uint8_t chunk[];
  __shared__ uint64_t bar;
  __shared__ uint32_t s_start[2 * kRows];  // byte offset of each 32-column half row's first value
  constexpr int kCols = 16 / ES;           // columns per lane
  constexpr int kSegs = kTileK / kCols;    // lanes per row
  const int64_t c = blockIdx.x;
  const int64_t rb = c / T, t = c % T;
  const int tid = threadIdx.x, lane = tid & 31, q = tid >> 5;
  if (tid == 0) {
    mbar_init(&bar, 1);
    fence_barrier_init();
    const uint64_t o0 = off[c];
    const uint32_t bytes = (uint32_t)(off[c + 1] - o0);
    mbar_arrive_expect_tx(&bar, bytes);
    bulk_g2s(chunk, buf + o0, bytes, &bar);
  }
  const uint64_t qi = qidx[c];
  __syncthreads();
  if (!__all_sync(0xffffffffu, mbar_wait(&bar, 0, timeout_ns))) {
    set_status(status, kStatusTimeout);
    return;
  }
  const uint32_t* words = reinterpret_cast<const uint32_t*>(chunk);  // word 2r, 2r + 1: row r's mask
  {
    const uint2 m = reinterpret_cast<const uint2*>(chunk)[tid];
    const int plo = __popc(m.x), pc = plo + __popc(m.y);
    int incl = pc;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const int u = __shfl_up_sync(0xffffffffu, incl, d);
      if (lane >= d) incl += u;
    }
    const int before = q == 0 ? 0 : (int)((qi >> (16 * (q - 1))) & 0xffffu);
    const uint32_t e0 = (uint32_t)(before + incl - pc);
    reinterpret_cast<uint2*>(s_start)[tid] = make_uint2(e0 * ES, (e0 + (uint32_t)plo) * ES);
  }
  __syncwarp();
  const int seg = lane % kSegs;
  const int half = seg / (kSegs / 2);                 // which mask word holds the lane's columns
  const int sh = kCols * (seg % (kSegs / 2));         // and where they start in it
  const uint32_t below = (1u << sh) - 1u;
  const uint32_t vbase = smem_u32(chunk) + kMaskBytes;
  const int64_t col = (int64_t)kTileK * t + kCols * seg;
  const int64_t pitch = K * ES;
  uint8_t* dst = out + (rb * kRows + 32 * q + lane / kSegs) * pitch + col * ES;
#pragma unroll 2
  for (int i = 0; i < kSegs; ++i) {  // 32 / kSegs rows at a time
    const int r = 32 * q + i * (32 / kSegs) + lane / kSegs;
    const uint32_t w = words[2 * r + half];
    uint32_t pa = vbase + s_start[2 * r + half] + (uint32_t)(ES * __popc(w & below));
    const uint32_t m = w >> sh;
    uint4 o;
    if constexpr (ES == 2) {
      o.x = expand_word_bf16<1u, 2u>(m, pa);
      o.y = expand_word_bf16<4u, 8u>(m, pa);
      o.z = expand_word_bf16<16u, 32u>(m, pa);
      o.w = expand_word_bf16<64u, 128u>(m, pa);
    } else {
      uint32_t a[8];
      a[0] = expand_word_u8<1u << 0, 1u << 1>(m, pa);
      a[1] = expand_word_u8<1u << 2, 1u << 3>(m, pa);
      a[2] = expand_word_u8<1u << 4, 1u << 5>(m, pa);
      a[3] = expand_word_u8<1u << 6, 1u << 7>(m, pa);
      a[4] = expand_word_u8<1u << 8, 1u << 9>(m, pa);
      a[5] = expand_word_u8<1u << 10, 1u << 11>(m, pa);
      a[6] = expand_word_u8<1u << 12, 1u << 13>(m, pa);
      a[7] = expand_word_u8<1u << 14, 1u << 15>(m, pa);
      o = make_uint4(__byte_perm(a[0], a[1], 0x6420), __byte_perm(a[2], a[3], 0x6420),
                     __byte_perm(a[4], a[5], 0x6420), __byte_perm(a[6], a[7], 0x6420));
    }
    if (rb * kRows + r < N && col < K) {
      // K % 8 == 0: a bf16 row's segments are whole and 16-byte aligned; an int8 row starts
      // on an 8-byte boundary and its last segment may hold 8 columns
      if (ES == 2 || K % 16 == 0) {
        __stcs(reinterpret_cast<uint4*>(dst), o);
      } else {
        __stcs(reinterpret_cast<uint2*>(dst), make_uint2(o.x, o.y));
        if (col + 8 < K) __stcs(reinterpret_cast<uint2*>(dst + 8), make_uint2(o.z, o.w));
      }
    }
    dst += (int64_t)(32 / kSegs) * pitch;
  }
}

}  // namespace

namespace {
size_t round256(size_t b) { return (b + 255) / 256 * 256; }
}  // namespace

void* dev_alloc(const sp_matrix* h, size_t bytes) {
  if (bytes == 0) bytes = 16;
  if (h->alloc) return h->alloc(bytes, h->ctx);
  void* p = nullptr;
  if (cudaMalloc(&p, bytes) != cudaSuccess) {
    cudaGetLastError();
    return nullptr;
  }
  return p;
}

void dev_free(const sp_matrix* h, void* p) {
  if (!p) return;
  if (h->free_fn)
    h->free_fn(p, h->ctx);
  else
    cudaFree(p);
}

size_t index_bytes(const sp_matrix* h) {
  const size_t C = (size_t)h->RB * h->T;
  return round256((C + 1) * sizeof(uint64_t)) + round256(C * sizeof(uint64_t)) +
         (h->dtype == SP_INT8 ? (size_t)h->N * sizeof(float) : 0);
}

bool alloc_index(sp_matrix* h) {
  const size_t C = (size_t)h->RB * h->T;
  uint8_t* p = (uint8_t*)dev_alloc(h, index_bytes(h));
  h->d_off = (uint64_t*)p;
  h->d_qidx = p ? (uint64_t*)(p + round256((C + 1) * sizeof(uint64_t))) : nullptr;
  h->d_scale = p && h->dtype == SP_INT8 ? (float*)((uint8_t*)h->d_qidx + round256(C * sizeof(uint64_t))) : nullptr;
  return p != nullptr;
}

sp_status launch_compress(const void* w, const uint8_t* mask, int64_t N, int64_t K, sp_dtype dt, const float* scale,
                          sp_alloc_fn alloc, sp_free_fn free_fn, void* ctx, cudaStream_t stream, sp_matrix** out) {
  sp_matrix* h = new sp_matrix();
  h->magic = 0;
  h->N = N;
  h->K = K;
  h->T = (int32_t)((K + kTileK - 1) / kTileK);
  h->RB = (int32_t)((N + kRows - 1) / kRows);
  h->dtype = dt;
  h->esize = dt == SP_BF16 ? 2 : 1;
  h->alloc = alloc;
  h->free_fn = free_fn;
  h->ctx = ctx;
  cudaGetDevice(&h->device);
  cudaDeviceGetAttribute(&h->num_sms, cudaDevAttrMultiProcessorCount, h->device);
  const int64_t C = (int64_t)h->RB * h->T;

  sp_status st = SP_OK;
  // scratch for the call: the masks, then the totals
  uint64_t* d_masks = (uint64_t*)dev_alloc(h, (size_t)C * kMaskBytes + 4 * sizeof(uint64_t));
  uint64_t* d_meta = d_masks ? d_masks + (size_t)C * kRows : nullptr;
  uint64_t meta[4] = {0, 0, 0, 0};
  if (!d_masks || !alloc_index(h)) {
    st = SP_ERR_OUT_OF_MEMORY;
    goto fail;
  }
  count_kernel<<<(unsigned)C, kRows, 0, stream>>>(mask, N, K, h->T, reinterpret_cast<uint8_t*>(d_masks), h->d_qidx);
  scan_kernel<<<1, 1024, 0, stream>>>(h->d_qidx, C, h->esize, h->d_off, d_meta);
  if (cudaGetLastError() != cudaSuccess) {
    st = SP_ERR_CUDA;
    goto fail;
  }
  if (cudaMemcpyAsync(meta, d_meta, sizeof(meta), cudaMemcpyDeviceToHost, stream) != cudaSuccess ||
      cudaStreamSynchronize(stream) != cudaSuccess) {
    st = SP_ERR_CUDA;
    goto fail;
  }
  h->bytes = meta[0];
  h->max_chunk = meta[1];
  h->nnz = (int64_t)meta[2];
  h->max_quarter = (uint32_t)(meta[3] & 0xffffffffu);
  h->d_buf = (uint8_t*)dev_alloc(h, (size_t)std::max<uint64_t>(h->bytes, 16));
  if (!h->d_buf) {
    st = SP_ERR_OUT_OF_MEMORY;
    goto fail;
  }
  if (dt == SP_INT8) {
    if (cudaMemcpyAsync(h->d_scale, scale, (size_t)N * sizeof(float), cudaMemcpyDeviceToDevice, stream) !=
        cudaSuccess) {
      st = SP_ERR_CUDA;
      goto fail;
    }
  }
  if (h->esize == 2)
    scatter_kernel<2><<<(unsigned)C, kRows, (size_t)h->max_chunk, stream>>>((const uint8_t*)w, N, K, h->T, d_masks,
                                                                            h->d_off, h->d_qidx, h->d_buf);
  else
    scatter_kernel<1><<<(unsigned)C, kRows, (size_t)h->max_chunk, stream>>>((const uint8_t*)w, N, K, h->T, d_masks,
                                                                            h->d_off, h->d_qidx, h->d_buf);
  if (cudaGetLastError() != cudaSuccess || cudaStreamSynchronize(stream) != cudaSuccess) {
    st = SP_ERR_CUDA;
    goto fail;
  }
  dev_free(h, d_masks);
  h->magic = SP_MAGIC;
  *out = h;
  return SP_OK;

fail:
  cudaStreamSynchronize(stream);
  cudaGetLastError();
  dev_free(h, d_masks);
  dev_free(h, h->d_off);
  dev_free(h, h->d_buf);
  delete h;
  return st;
}

sp_status launch_decompress(const sp_matrix* h, void* w_out, cudaStream_t stream) {
  const int64_t C = (int64_t)h->RB * h->T;
  const size_t smem = (size_t)h->max_chunk;  // at most 1024 + 128 * 64 * 2 bytes
  auto kern = h->esize == 2 ? decompress_kernel<2> : decompress_kernel<1>;
  kern<<<(unsigned)C, kRows, smem, stream>>>(h->d_buf, h->d_off, h->d_qidx, h->N, h->K, h->T, (uint8_t*)w_out,
                                             wait_timeout_ns(), device_status_ptr());
  return cudaGetLastError() == cudaSuccess ? SP_OK : SP_ERR_CUDA;
}

}  // namespace sp
