// sp_linear_dense.cu -- prefill-sized sparse linear: every chunk expanded once, then a dense
// tcgen05 product.
//
// linear_tc_kernel expands a chunk again for every tile of up to 256 tokens, and one SM cannot
// expand as fast as its tensor core multiplies (a 128 x 64 chunk costs ~0.4 us of shared-memory
// and issue slots, its product with 256 tokens 0.33 us).  Past a few hundred tokens it is
// cheaper to expand the matrix once, to a bf16 scratch in the workspace (2 bytes written per
// weight, at the HBM rate, and largely read back from L2), and to run the product as a dense
// GEMM at the tensor cores' rate:
//
//   1. expand_kernel   one CTA per chunk, as sp_decompress's kernel: the chunk's 128 x 64 bf16
//                      tile, 16 KB, goes to its place in panel t of the scratch
//                      ([T][128 RB rows][64 columns]) in one contiguous piece; rows past N and
//                      columns past K are zero because their mask bits are.
//   2. dense_kernel    y = x . W^T on pairs of SMs (cta_group::2): a pair's tile is 256 rows of
//                      W by up to 256 tokens, D (fp32) in tensor memory, double-buffered, so
//                      that the epilogue of one tile runs under the main loop of the next.
//                      INT8 values are exact in bf16; their row scales are applied here.
#include <cuda.h>
#include <cudaTypedefs.h>

#include <algorithm>
#include <atomic>
#include <cstring>

#include "sp_expand.cuh"
#include "sp_tcgen05.cuh"

namespace sp {
namespace {

constexpr int kMaxDevices = 64;

// ------------------------------------------------------------------ 1. expansion
// Lane: eight columns (16 bytes of bf16) of one row; a warp, four rows at a time.
template <int ES>
__global__ void __launch_bounds__(kRows) expand_kernel(const uint8_t* __restrict__ buf,
                                                       const uint64_t* __restrict__ off,
                                                       const uint64_t* __restrict__ qidx, int T, int64_t rows,
                                                       uint4* __restrict__ out, uint64_t timeout_ns, int* status) {
  extern __shared__ __align__(128) uint8_t chunk[];
  __shared__ uint64_t bar;
  __shared__ uint32_t s_start[2 * kRows];  // byte offset of each 32-column half row's first value
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
  const uint32_t* words = reinterpret_cast<const uint32_t*>(chunk);
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
  const int seg = lane & 7, half = seg >> 2, sh = 8 * (seg & 3);
  const uint32_t below = (1u << sh) - 1u;
  const uint32_t vbase = smem_u32(chunk) + kMaskBytes;
  uint4* dst = out + ((t * rows + rb * kRows + 32 * q) * 8 + lane);
#pragma unroll 2
  for (int i = 0; i < 8; ++i) {
    const int r = 32 * q + 4 * i + (lane >> 3);
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
      o.x = i8x2_to_bf16x2(expand_word_u8<1u, 2u>(m, pa));
      o.y = i8x2_to_bf16x2(expand_word_u8<4u, 8u>(m, pa));
      o.z = i8x2_to_bf16x2(expand_word_u8<16u, 32u>(m, pa));
      o.w = i8x2_to_bf16x2(expand_word_u8<64u, 128u>(m, pa));
    }
    dst[32 * i] = o;
  }
}

// ------------------------------------------------------------------ 2. dense product
constexpr int kTileRows = 256;    // rows of W per CTA pair (128 per CTA)
constexpr int kMaxTok = 256;      // tokens per tile (MMA N), a multiple of 32
constexpr int kMaxStages = 10;    // of W and x tiles; as many as fit beside the y staging
constexpr uint32_t kABytes = kRows * 128;  // 128 rows x 64 columns of W
constexpr int kStgTokens = 32, kStgBox = 16;     // y staging block; tokens per TMA store
constexpr uint32_t kStgBytes = kStgTokens * kRows * 2;
constexpr uint32_t kCtlBytes = 256;
constexpr uint32_t kStgOff = kCtlBytes + 768;  // 1024-byte aligned
constexpr uint32_t kRingOff = kStgOff + 2 * kStgBytes;
constexpr uint32_t kRingBytes = 6 * 32 * 1024;
constexpr size_t kDenseSmem = 1024 + kRingOff + kRingBytes;  // + base alignment
constexpr int kDenseThreads = 256;
constexpr int kEpiWarp0 = 4;

struct DenseParams {
  uint16_t* y;
  const float* scale;  // INT8 only
  int* status;
  int64_t N, M;
  int64_t rows;        // rows of a panel (128 RB)
  int32_t T;
  int32_t tok;         // tokens per full tile
  int32_t tok_tiles;   // token tiles per 256 rows
  int64_t full;        // full tiles, tok tokens each
  int64_t tiles;       // full tiles and the pieces of the rest
  int32_t split;       // pieces per remaining tile, tok_piece tokens each
  int32_t tok_piece;
  int32_t y_tma;
  int32_t stages;      // ring stages of stage_bytes: W's 16 KB, then a CTA's half of tok tokens of x
  uint32_t stage_bytes;
  uint64_t timeout_ns;
};

// Tile i of the work list: first row / 256, first token, tokens.  The first `full` tiles fill
// whole waves of CTA pairs; the rest, less than a wave, is cut into narrower pieces so that
// all pairs share it.
__device__ __forceinline__ void tile_at(const DenseParams& p, int64_t i, int64_t* rt, int64_t* tok0, int* ntok) {
  int64_t k = i, sub = 0;
  *ntok = p.tok;
  if (i >= p.full) {
    k = p.full + (i - p.full) / p.split;
    sub = (i - p.full) % p.split;
    *ntok = min(p.tok_piece, p.tok - (int)sub * p.tok_piece);
  }
  *rt = k / p.tok_tiles;
  *tok0 = (k % p.tok_tiles) * p.tok + sub * p.tok_piece;
}

__global__ void __launch_bounds__(kDenseThreads, 1) __cluster_dims__(2, 1, 1)
    dense_kernel(const __grid_constant__ DenseParams p, const __grid_constant__ CUtensorMap tmap_w,
                 const __grid_constant__ CUtensorMap tmap_x, const __grid_constant__ CUtensorMap tmap_y) {
  extern __shared__ uint8_t smem_raw[];
  // the same offset in both CTAs of the pair: dynamic shared memory starts at one address
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  uint64_t* full = reinterpret_cast<uint64_t*>(smem);  // leader's: both CTAs' copies of a stage landed
  uint64_t* empty = full + kMaxStages;    // each CTA's: the MMAs that read the stage are done
  uint64_t* d_full = empty + kMaxStages;  // each CTA's: a tile's accumulators are complete
  uint64_t* d_empty = d_full + 2;      // leader's: both CTAs' epilogues have read the buffer
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(d_empty + 2);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const uint32_t rank = cluster_rank();
  const int64_t pair = blockIdx.x >> 1, pairs = gridDim.x >> 1;
  const int T = p.T;

  if (tid == 0) {
    for (int s = 0; s < p.stages; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&d_full[b], 1);
      mbar_init(&d_empty[b], 8);  // four epilogue warps of each CTA
    }
    fence_barrier_init();
  }
  if (warp == 2) {
    tmem_alloc2(tmem_slot, 512);
    tmem_relinquish2();
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();  // the peer's barriers are initialised
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;

  if (warp == 0) {
    if (lane == 0) {
      // ---------------------------------------------------------- producer (both CTAs)
      prefetch_tmap(&tmap_w);
      prefetch_tmap(&tmap_x);
      pdl_wait();
      int s = 0;
      uint32_t ph = 0;
      bool dead = false;
      const uint32_t full0 = cluster_map(smem_u32(full), 0);
      for (int64_t i = pair; i < p.tiles && !dead; i += pairs) {
        int64_t rt, tok0;
        int ntok;
        tile_at(p, i, &rt, &tok0, &ntok);
        const int wrow = (int)(rt * kTileRows + rank * kRows);  // (rows past the panel: clamped below)
        const int xrow = (int)(tok0 + (int64_t)rank * (ntok / 2));
        for (int t = 0; t < T; ++t) {
          if (!mbar_wait(&empty[s], ph ^ 1u, p.timeout_ns)) {
            set_status(p.status, kStatusTimeout);
            dead = true;
            break;
          }
          uint8_t* st = smem + kRingOff + (size_t)s * p.stage_bytes;
          if (rank == 0) mbar_arrive_expect_tx(&full[s], 2 * (kABytes + (uint32_t)p.tok / 2 * 128));
          // an odd number of row blocks leaves the last pair's second half without rows: it
          // repeats the first half's, and its results are not stored
          const int64_t row = (int64_t)t * p.rows + (wrow < p.rows ? wrow : wrow - kRows);
          tma_load_2d_pair(st, &tmap_w, 0, (int)row, full0 + 8u * s);
          tma_load_2d_pair(st + kABytes, &tmap_x, kTileK * t, xrow, full0 + 8u * s);
          if (++s == p.stages) {
            s = 0;
            ph ^= 1u;
          }
        }
      }
      // the MMAs' last arrivals on this CTA's barriers, before it may exit
      for (int j = 0; j < p.stages && !dead; ++j) {
        if (!mbar_wait(&empty[s], ph ^ 1u, p.timeout_ns)) {
          set_status(p.status, kStatusTimeout);
          dead = true;
        }
        if (++s == p.stages) {
          s = 0;
          ph ^= 1u;
        }
      }
    }
  } else if (warp == 1) {
    if (rank == 0) {
      // ---------------------------------------------------------- MMA issuer (leader)
      int s = 0;
      uint32_t ph = 0;
      int64_t k = 0;  // tile number of this pair
      bool dead = false;
      for (int64_t i = pair; i < p.tiles && !dead; i += pairs, ++k) {
        int64_t rt, tok0;
        int ntok;
        tile_at(p, i, &rt, &tok0, &ntok);
        const uint32_t idesc = idesc_bf16(kTileRows, ntok);
        const int db = (int)(k & 1);
        const uint32_t d = tmem + (uint32_t)db * kMaxTok;
        if (k >= 2 && !__all_sync(0xffffffffu, mbar_wait(&d_empty[db], (uint32_t)((k / 2 - 1) & 1), p.timeout_ns))) {
          set_status(p.status, kStatusTimeout);
          dead = true;
          break;
        }
        tc_fence_after();
        for (int t = 0; t < T; ++t) {
          if (!__all_sync(0xffffffffu, mbar_wait(&full[s], ph, p.timeout_ns))) {
            set_status(p.status, kStatusTimeout);
            dead = true;
            break;
          }
          tc_fence_after();
          const uint32_t a = smem_u32(smem + kRingOff + (size_t)s * p.stage_bytes);
          if (elect_one()) {
#pragma unroll
            for (int kk = 0; kk < 4; ++kk)
              mma_ss2(d, smem_desc_sw128(a + kk * 32u), smem_desc_sw128(a + kABytes + kk * 32u), idesc,
                      (t > 0 || kk > 0) ? 1u : 0u);
            mma_commit2(&empty[s]);
            if (t == T - 1) mma_commit2(&d_full[db]);
          }
          __syncwarp();
          if (++s == p.stages) {
            s = 0;
            ph ^= 1u;
          }
        }
      }
    }
  } else if (warp >= kEpiWarp0) {
    // ------------------------------------------------------------ epilogue: thread = row of W
    const int q = warp & 3;
    const int r = q * 32 + lane;
    const uint32_t lane_base = (uint32_t)(q * 32) << 16;
    uint16_t* stg = reinterpret_cast<uint16_t*>(smem + kStgOff);
    const uint32_t d_empty0 = cluster_map(smem_u32(d_empty), 0);
    int step = 0;
    int64_t k = 0;
    bool dead = false;
    pdl_wait();  // y belongs to the stream order
    for (int64_t i = pair; i < p.tiles; i += pairs, ++k) {
      int64_t rt, tok0;
      int ntok;
      tile_at(p, i, &rt, &tok0, &ntok);
      const int db = (int)(k & 1);
      if (!dead && !__all_sync(0xffffffffu, mbar_wait(&d_full[db], (uint32_t)((k / 2) & 1), p.timeout_ns))) {
        set_status(p.status, kStatusTimeout);
        dead = true;
      }
      // every epilogue warp takes the same branch: a warp that timed out keeps the barriers
      tc_fence_after();
      const int64_t row0 = rt * kTileRows + rank * kRows;
      const int64_t n = row0 + r;
      const float sc = (p.scale && n < p.N) ? p.scale[n] : 1.f;
      for (int c0 = 0; c0 < ntok; c0 += 32) {
        uint32_t v[32];
        if (!dead) {
          tmem_load32(tmem + (uint32_t)db * kMaxTok + lane_base + (uint32_t)c0, v);
          tmem_load_wait();
        }
        if (c0 + 32 >= ntok) {  // the buffer is read: the issuer may start the tile after next
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive_remote(d_empty0 + 8u * db);
        }
        if (row0 >= p.N) continue;  // the same for the whole CTA
        if (p.y_tma) {
          uint16_t* buf = stg + (size_t)(step & 1) * (kStgBytes / 2);
          if (warp == kEpiWarp0 && lane == 0) bulk_wait_read<1>();  // the store that last read it is done
          named_bar_sync(1, 128);
#pragma unroll
          for (int j = 0; j < 32; ++j) buf[j * kRows + r] = float_to_bf16_bits_rn(__uint_as_float(v[j]) * sc);
          fence_proxy_async_smem();
          named_bar_sync(1, 128);
          if (warp == kEpiWarp0 && lane == 0) {
            for (int b = 0; b < 32; b += kStgBox)
              if (tok0 + c0 + b < p.M) tma_store_2d(&tmap_y, buf + b * kRows, (int)row0, (int)(tok0 + c0 + b));
            bulk_commit();
          }
          ++step;
        } else if (n < p.N) {
          uint16_t* yp = p.y + (tok0 + c0) * p.N + n;
          const int nv = (int)imin64(32, p.M - (tok0 + c0));
#pragma unroll
          for (int j = 0; j < 32; ++j) {
            if (j < nv) *yp = float_to_bf16_bits_rn(__uint_as_float(v[j]) * sc);
            yp += p.N;
          }
        }
      }
    }
    if (p.y_tma && warp == kEpiWarp0 && lane == 0) bulk_wait_all();
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();  // no arrive or copy of the peer is still to come
  if (warp == 2) {
    tc_fence_after();
    tmem_dealloc2(tmem, 512);
  }
}

// ------------------------------------------------------------------ host side
// Work list for M tokens on `pairs` CTA pairs: the tile width (a multiple of 32 tokens) with
// the least estimated time.  A tile costs per K-tile the larger of its tensor time, 2 clocks
// per token, and its shared-memory traffic, 256 clocks for W's side (written and read) and one
// per token for x's, and a fixed share for its start and end.
void plan_tiles(const sp_matrix* h, int64_t M, int pairs, DenseParams* p) {
  const int64_t rt = (h->RB + 1) / 2;
  auto tile_cost = [&](int t) { return (double)h->T * std::max(2 * t, 256 + t) + 1500.0; };
  double best = 0;
  for (int t = 32; t <= kMaxTok; t += 32) {
    const int64_t tt = (M + t - 1) / t;
    const int64_t total = rt * tt, waves = total / pairs, rest = total - waves * pairs;
    double cost = (double)waves * tile_cost(t);
    int split = 1, piece = t;
    if (rest > 0) {
      const int units = t / 32;
      const int want = (int)std::min<int64_t>(pairs / rest, units);
      piece = (units + want - 1) / want * 32;
      split = (t + piece - 1) / piece;
      cost += tile_cost(piece);
    }
    if (best == 0 || cost < best) {
      best = cost;
      p->tok = t;
      p->tok_tiles = (int32_t)tt;
      p->full = waves * pairs;
      p->split = split;
      p->tok_piece = piece;
      p->tiles = p->full + rest * split;
    }
  }
}

// CTA pairs that the device holds at once (0: the kernel cannot run); looked up once per device.
int resident_pairs(int dev) {
  static std::atomic<int> pairs[kMaxDevices] = {};  // + 1; 0 = not looked up
  if (dev < 0 || dev >= kMaxDevices) return 0;
  int n = pairs[dev].load(std::memory_order_acquire);
  if (n == 0) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(2);
    cfg.blockDim = dim3(kDenseThreads);
    cfg.dynamicSmemBytes = kDenseSmem;
    int c = 0;
    if (cudaFuncSetAttribute(dense_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kDenseSmem) !=
            cudaSuccess ||
        cudaOccupancyMaxActiveClusters(&c, dense_kernel, &cfg) != cudaSuccess) {
      cudaGetLastError();
      c = 0;
    }
    n = c + 1;
    pairs[dev].store(n, std::memory_order_release);
  }
  return n - 1;
}

size_t round256(size_t b) { return (b + 255) / 256 * 256; }

}  // namespace

// Against linear_tc_kernel, measured at 70 %: from 33 tokens on where the matrix is small (4096 x
// 4096 30.8 us against 34.6 at M = 64, 31.6 / 102 at 256; 1003 x 1096 11.7 / 65), later where the
// scratch is much traffic for few tokens (q/k/v INT8 45 / 43 at 33, 50 / 83 at 256; down 71 / 67 at
// 128, 72 / 90 at 192; gate/up 90 / 82 at 256, 102 / 121 at 384, 233 / 377 at 2048).  A matrix of
// fewer chunks than SMs keeps the one launch.
bool uses_dense(const sp_matrix* h, int64_t M) {
  const int64_t C = (int64_t)h->RB * h->T, rows = (int64_t)h->RB * kRows;
  if (C < h->num_sms || M > (int64_t)1 << 24 || (int64_t)h->T * rows >= (int64_t)1 << 31) return false;
  return M > kMmaMaxRows && M >= (C <= 2500 ? 0 : C / 40);
}

size_t workspace_bytes_dense(const sp_matrix* h) {
  return ws_counter_bytes(h->num_sms) + round256((size_t)h->T * h->RB * kRows * 128);
}

sp_status launch_linear_dense(const sp_matrix* h, const uint16_t* x, int64_t M, uint16_t* y, void* ws, size_t ws_bytes,
                              cudaStream_t stream) {
  if (!ws || ws_bytes < workspace_bytes_dense(h)) return SP_ERR_WORKSPACE;
  const int64_t rows = (int64_t)h->RB * kRows;
  PFN_cuTensorMapEncodeTiled_v12000 encode = nullptr;
  sp_status st = tensor_map_encoder(&encode);
  if (st != SP_OK) return st;
  const int pairs = resident_pairs(h->device);
  if (pairs < 1) return SP_ERR_CUDA;

  // the scratch follows the arrival counters, which stay zero for the other kernels
  uint8_t* scratch = static_cast<uint8_t*>(ws) + ws_counter_bytes(h->num_sms);
  DenseParams p{};
  p.y = y;
  p.scale = h->d_scale;
  p.status = device_status_ptr();
  p.N = h->N;
  p.M = M;
  p.rows = rows;
  p.T = h->T;
  p.y_tma = h->N % 8 == 0 ? 1 : 0;
  p.timeout_ns = wait_timeout_ns();
  plan_tiles(h, M, pairs, &p);
  p.stage_bytes = (uint32_t)(kABytes + p.tok / 2 * 128);  // a multiple of 2 KB
  p.stages = (int32_t)std::min<uint32_t>(kMaxStages, kRingBytes / p.stage_bytes);

  CUtensorMap map_w, map_x, map_y;
  const cuuint32_t estride[2] = {1, 1};
  {
    const cuuint64_t dim[2] = {(cuuint64_t)kTileK, (cuuint64_t)(h->T * rows)}, stride[1] = {128};
    const cuuint32_t box[2] = {(cuuint32_t)kTileK, (cuuint32_t)kRows};
    if (encode(&map_w, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, scratch, dim, stride, box, estride,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
      return SP_ERR_CUDA;
  }
  {  // rows past M and columns past K read as zero
    const cuuint64_t dim[2] = {(cuuint64_t)h->K, (cuuint64_t)M}, stride[1] = {(cuuint64_t)h->K * 2};
    const cuuint32_t box[2] = {(cuuint32_t)kTileK, (cuuint32_t)(p.tok / 2)};
    if (encode(&map_x, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<uint16_t*>(x), dim, stride, box, estride,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
      return SP_ERR_CUDA;
  }
  memset(&map_y, 0, sizeof(map_y));
  if (p.y_tma) {
    const cuuint64_t dim[2] = {(cuuint64_t)h->N, (cuuint64_t)M}, stride[1] = {(cuuint64_t)h->N * 2};
    const cuuint32_t box[2] = {(cuuint32_t)kRows, (cuuint32_t)kStgBox};
    if (encode(&map_y, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, y, dim, stride, box, estride,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_NONE,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
      return SP_ERR_CUDA;
  }

  const int64_t C = (int64_t)h->RB * h->T;
  auto ek = h->esize == 2 ? expand_kernel<2> : expand_kernel<1>;
  ek<<<(unsigned)C, kRows, (size_t)h->max_chunk, stream>>>(h->d_buf, h->d_off, h->d_qidx, h->T, rows,
                                                           reinterpret_cast<uint4*>(scratch), p.timeout_ns, p.status);
  if (cudaGetLastError() != cudaSuccess) return SP_ERR_CUDA;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(2 * std::min<int64_t>(pairs, p.tiles)));
  cfg.blockDim = dim3(kDenseThreads);
  cfg.dynamicSmemBytes = kDenseSmem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  if (cudaLaunchKernelEx(&cfg, dense_kernel, p, map_w, map_x, map_y) != cudaSuccess) {
    cudaGetLastError();
    return SP_ERR_CUDA;
  }
  h->weights_written = 0;
  return SP_OK;
}

}  // namespace sp
