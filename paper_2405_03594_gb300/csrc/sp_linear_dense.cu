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
#include "sp_lookup.h"
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
  pdl_launch_dependents();  // the product's CTAs may set up while the last chunks are expanded
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
  pdl_wait();  // the scratch belongs to the stream order, the weights do not
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
  int64_t items;       // full tiles and the pieces of the rest, or tiles * split_k
  int32_t split;       // pieces per remaining tile, tok_piece tokens each
  int32_t tok_piece;
  int32_t split_k;     // items that share a tile's K-tiles (1: none)
  float* ws;           // split_k: partials [items][2 CTAs][tok][kRows]
  int* cnt;            // split_k: arrival counters [tiles][2 CTAs]
  int32_t y_tma;
  int32_t stages;      // ring stages of stage_bytes: W's 16 KB, then a CTA's half of tok tokens of x
  uint32_t stage_bytes;
  uint64_t timeout_ns;
};

// Item i of the work list: first row / 256, first token, tokens, K-tiles [t0, t1).  Without
// split_k the first `full` items fill whole waves of CTA pairs with full tiles, and the rest,
// less than a wave, is cut into narrower pieces so that all pairs share it.  With split_k (fewer
// tiles than pairs, so one item per pair) a tile's K-tiles are shared by split_k items.
struct Item {
  int64_t rt, tok0;
  int ntok, t0, t1;
};
__device__ __forceinline__ Item item_at(const DenseParams& p, int64_t i) {
  Item it;
  it.ntok = p.tok;
  it.t0 = 0;
  it.t1 = p.T;
  int64_t k = i, sub = 0;
  if (p.split_k > 1) {
    k = i / p.split_k;
    const int part = (int)(i % p.split_k);
    it.t0 = (int)((int64_t)part * p.T / p.split_k);
    it.t1 = (int)((int64_t)(part + 1) * p.T / p.split_k);
  } else if (i >= p.full) {
    k = p.full + (i - p.full) / p.split;
    sub = (i - p.full) % p.split;
    it.ntok = min(p.tok_piece, p.tok - (int)sub * p.tok_piece);
  }
  it.rt = k / p.tok_tiles;
  it.tok0 = (k % p.tok_tiles) * p.tok + sub * p.tok_piece;
  return it;
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
  volatile int* s_last = reinterpret_cast<volatile int*>(tmem_slot + 1);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const uint32_t rank = cluster_rank();
  const int64_t pair = blockIdx.x >> 1, pairs = gridDim.x >> 1;
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
      for (int64_t i = pair; i < p.items && !dead; i += pairs) {
        const Item it = item_at(p, i);
        const int wrow = (int)(it.rt * kTileRows + rank * kRows);  // (rows past the panel: clamped below)
        const int xrow = (int)(it.tok0 + (int64_t)rank * (it.ntok / 2));
        for (int t = it.t0; t < it.t1; ++t) {
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
      for (int64_t i = pair; i < p.items && !dead; i += pairs, ++k) {
        const Item it = item_at(p, i);
        const uint32_t idesc = idesc_bf16(kTileRows, it.ntok);
        const int db = (int)(k & 1);
        const uint32_t d = tmem + (uint32_t)db * kMaxTok;
        if (k >= 2 && !__all_sync(0xffffffffu, mbar_wait(&d_empty[db], (uint32_t)((k / 2 - 1) & 1), p.timeout_ns))) {
          set_status(p.status, kStatusTimeout);
          dead = true;
          break;
        }
        tc_fence_after();
        for (int t = it.t0; t < it.t1; ++t) {
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
                      (t > it.t0 || kk > 0) ? 1u : 0u);
            mma_commit2(&empty[s]);
            if (t == it.t1 - 1) mma_commit2(&d_full[db]);
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
    const int etid = tid - kEpiWarp0 * 32;
    // tokens tok .. tok + 31 of the CTA's rows from their sums v
    auto store = [&](const float (&v)[32], int64_t tok, int64_t row0, float sc) {
      const int64_t n = row0 + r;
      if (p.y_tma) {
        uint16_t* buf = stg + (size_t)(step & 1) * (kStgBytes / 2);
        if (etid == 0) bulk_wait_read<1>();  // the store that last read it is done
        named_bar_sync(1, 128);
#pragma unroll
        for (int j = 0; j < 32; ++j) buf[j * kRows + r] = float_to_bf16_bits_rn(v[j] * sc);
        fence_proxy_async_smem();
        named_bar_sync(1, 128);
        if (etid == 0) {
          for (int b = 0; b < 32; b += kStgBox)
            if (tok + b < p.M) tma_store_2d(&tmap_y, buf + b * kRows, (int)row0, (int)(tok + b));
          bulk_commit();
        }
        ++step;
      } else if (n < p.N) {
        uint16_t* yp = p.y + tok * p.N + n;
        const int nv = (int)imin64(32, p.M - tok);
#pragma unroll
        for (int j = 0; j < 32; ++j) {
          if (j < nv) *yp = float_to_bf16_bits_rn(v[j] * sc);
          yp += p.N;
        }
      }
    };
    for (int64_t i = pair; i < p.items; i += pairs, ++k) {
      const Item it = item_at(p, i);
      const int db = (int)(k & 1);
      if (!dead && !__all_sync(0xffffffffu, mbar_wait(&d_full[db], (uint32_t)((k / 2) & 1), p.timeout_ns))) {
        set_status(p.status, kStatusTimeout);
        dead = true;
      }
      // every epilogue warp takes the same branch: a warp that timed out keeps the barriers
      tc_fence_after();
      const int64_t row0 = it.rt * kTileRows + rank * kRows;
      const bool rows = row0 < p.N;  // the same for the whole CTA
      const float sc = (p.scale && row0 + r < p.N) ? p.scale[row0 + r] : 1.f;
      const int64_t part = (int64_t)kRows * p.tok;
      float* wsp = p.ws + (i * 2 + rank) * part + r;
      for (int c0 = 0; c0 < it.ntok; c0 += 32) {
        float v[32];
        if (!dead) {
          uint32_t u[32];
          tmem_load32(tmem + (uint32_t)db * kMaxTok + lane_base + (uint32_t)c0, u);
          tmem_load_wait();
#pragma unroll
          for (int j = 0; j < 32; ++j) v[j] = __uint_as_float(u[j]);
        } else {
#pragma unroll
          for (int j = 0; j < 32; ++j) v[j] = 0.f;
        }
        if (c0 + 32 >= it.ntok) {  // the buffer is read: the issuer may start the tile after next
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive_remote(d_empty0 + 8u * db);
        }
        if (!rows) continue;
        if (p.split_k == 1) {
          store(v, it.tok0 + c0, row0, sc);
        } else {
#pragma unroll
          for (int j = 0; j < 32; ++j) __stcg(wsp + (int64_t)(c0 + j) * kRows, v[j]);
        }
      }
      if (p.split_k == 1 || !rows) continue;
      // the last of the tile's items to arrive adds up their partials in order
      __threadfence();
      named_bar_sync(1, 128);
      const int64_t tile = i / p.split_k;
      int* ctr = p.cnt + tile * 2 + rank;
      if (etid == 0) *s_last = atomicAdd(ctr, 1) == p.split_k - 1 ? 1 : 0;
      named_bar_sync(1, 128);
      if (*s_last) {
        __threadfence();
        // a warp takes a token's 128 rows (four per lane), eight tokens at a time, so that 8
        // or more 16-byte loads per lane are in flight: one CTA reads all of a tile's partials
        const float4* src = reinterpret_cast<const float4*>(p.ws + (tile * p.split_k * 2 + rank) * part) + lane;
        const int64_t n = row0 + 4 * lane;
        float s4[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) s4[j] = (p.scale && n + j < p.N) ? p.scale[n + j] : 1.f;
        for (int tk = (warp & 3) * 8; tk < it.ntok; tk += 32) {
          float4 v[8];
#pragma unroll
          for (int j = 0; j < 8; ++j) v[j] = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 2
          for (int q = 0; q < p.split_k; ++q) {
#pragma unroll
            for (int j = 0; j < 8; ++j) {
              const float4 u = __ldcg(src + (2 * q * part + (int64_t)(tk + j) * kRows) / 4);
              v[j].x += u.x, v[j].y += u.y, v[j].z += u.z, v[j].w += u.w;
            }
          }
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            const int64_t tok = it.tok0 + tk + j;
            if (tok >= p.M) continue;
            const uint32_t lo = (uint32_t)float_to_bf16_bits_rn(v[j].x * s4[0]) |
                                ((uint32_t)float_to_bf16_bits_rn(v[j].y * s4[1]) << 16);
            const uint32_t hi = (uint32_t)float_to_bf16_bits_rn(v[j].z * s4[2]) |
                                ((uint32_t)float_to_bf16_bits_rn(v[j].w * s4[3]) << 16);
            uint16_t* yp = p.y + tok * p.N + n;
            if (p.N % 4 == 0) {
              if (n < p.N) *reinterpret_cast<uint2*>(yp) = make_uint2(lo, hi);
            } else {
              if (n < p.N) yp[0] = (uint16_t)lo;
              if (n + 1 < p.N) yp[1] = (uint16_t)(lo >> 16);
              if (n + 2 < p.N) yp[2] = (uint16_t)hi;
              if (n + 3 < p.N) yp[3] = (uint16_t)(hi >> 16);
            }
          }
        }
        if (etid == 0) atomicExch(ctr, 0);
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
// Work list for M tokens on `pairs` CTA pairs: the tile width (a multiple of 32 tokens) and K
// split with the least estimated time.  A tile costs per K-tile the largest of its tensor time,
// 2 clocks per token, its shared-memory traffic, 256 clocks for W's side (written and read) and
// one per token for x's, and ~430 clocks of issue and barriers, and a fixed share for its start
// and end.  Splitting K (at least 8 K-tiles per item) pays where the tiles would leave pairs
// idle; its partial sums are written once and read by one CTA per tile (~600 clocks per 32
// tokens and part).  Measured at 70 %, unsplit / split: 4096 x 4096 24.6 / 20.4 us at 64 tokens,
// 4096 x 11008 55.4 / 37.1 at 64, 55.6 / 41.8 at 128.
void plan_items(const sp_matrix* h, int64_t M, int pairs, DenseParams* p) {
  const int64_t rt = (h->RB + 1) / 2, T = h->T;
  auto cost = [&](int64_t kt, int t) { return (double)kt * std::max({2 * t, 256 + t, 430}) + 1500.0; };
  double best = 0;
  auto take = [&](double c) {
    if (best != 0 && c >= best) return false;
    best = c;
    return true;
  };
  for (int t = 32; t <= kMaxTok; t += 32) {
    const int64_t tt = (M + t - 1) / t;
    const int64_t total = rt * tt, waves = total / pairs, rest = total - waves * pairs;
    double c = (double)waves * cost(T, t);
    int split = 1, piece = t;
    if (rest > 0) {
      const int units = t / 32;
      const int want = (int)std::min<int64_t>(pairs / rest, units);
      piece = (units + want - 1) / want * 32;
      split = (t + piece - 1) / piece;
      c += cost(T, piece);
    }
    if (take(c)) {
      p->tok = t;
      p->tok_tiles = (int32_t)tt;
      p->full = waves * pairs;
      p->split = split;
      p->tok_piece = piece;
      p->items = p->full + rest * split;
      p->split_k = 1;
    }
    const int64_t sk = std::min<int64_t>(pairs / total, T / 8);
    if (sk >= 2 && take(cost((T + sk - 1) / sk, t) + 3000.0 + 600.0 * (double)(sk * (t / 32)))) {
      p->tok = p->tok_piece = t;
      p->tok_tiles = (int32_t)tt;
      p->full = 0;
      p->split = 1;
      p->items = total * sk;
      p->split_k = (int32_t)sk;
    }
  }
}

// CTA pairs that the device, which is current, holds at once; 0: none, or the lookup failed.
int resident_pairs(int dev) {
  static std::atomic<int> pairs[kMaxDevices] = {};
  if (dev < 0 || dev >= kMaxDevices) return 0;
  return kept_or_looked_up(pairs[dev], [] {
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
    return c;
  });
}

size_t round256(size_t b) { return (b + 255) / 256 * 256; }

}  // namespace

// Against linear_tc_kernel (one token tile up to 256 rows), measured at 70 %, this way / that, us.
// bf16: small matrices from 33 tokens on (o, 2048 chunks, 19.5 / 24.7 at 33, 25.0 / 51.9 at 256);
// middling ones from ~110 (8192 x 4096, 28.8 / 28.1 at 80, 32.4 / 36.7 at 160; down, 5504 chunks,
// 39.7 / 36.1 and 45.0 / 47.2); where the scratch is much traffic for few tokens only beyond one
// token tile (q/k/v, 6144 chunks, 41.3 / 31.8 at 64, 49.8 / 48.5 at 256; gate/up, 11008, 76.5 / 42.0
// and 82.4 / 61.9; two tiles 94 / 120 at 384).  INT8, which linear_tc_kernel expands slower: down
// 37.5 / 39.7 at 64, q/k/v 41.9 / 41.7 at 128, 14336 x 4096 (7168 chunks) 51.4 / 50.8 at 192, gate/up
// 82.9 / 67.5 at 256.  A matrix of a few chunks keeps the one launch.  The lines go by the chunk
// count alone and hold for 50 to 80 %; on unpruned rows, where linear_tc_kernel's value loads
// meet in one bank, this way would win far earlier (gate/up at 256: 104 / 368).
bool uses_dense(const sp_matrix* h, int64_t M) {
  const int64_t C = (int64_t)h->RB * h->T, rows = (int64_t)h->RB * kRows;
  if (C < 16 || M > (int64_t)1 << 24 || (int64_t)h->T * rows >= (int64_t)1 << 31) return false;
  const int64_t from = h->esize == 2 ? (C < 4000 ? 33 : C < 6000 ? 110 : 257) : std::min<int64_t>(257, (C - 5400) / 10 + 33);
  return M > kMmaMaxRows && M >= from;
}

namespace {
size_t scratch_bytes(const sp_matrix* h) { return round256((size_t)h->T * h->RB * kRows * 128); }
}  // namespace

// [arrival counters][expanded matrix][split-K partials: two CTAs of at most num_sms / 2 items]
size_t workspace_bytes_dense(const sp_matrix* h, int64_t M) {
  const size_t tok = (size_t)std::min<int64_t>(kMaxTok, (M + 31) / 32 * 32);
  return ws_counter_bytes(h->num_sms) + scratch_bytes(h) + (size_t)(h->num_sms / 2) * 2 * kRows * tok * sizeof(float);
}

sp_status launch_linear_dense(const sp_matrix* h, const uint16_t* x, int64_t M, uint16_t* y, void* ws, size_t ws_bytes,
                              cudaStream_t stream) {
  if (!ws || ws_bytes < workspace_bytes_dense(h, M)) return SP_ERR_WORKSPACE;
  const int64_t rows = (int64_t)h->RB * kRows;
  PFN_cuTensorMapEncodeTiled_v12000 encode = nullptr;
  sp_status st = tensor_map_encoder(&encode);
  if (st != SP_OK) return st;
  const int pairs = std::min(resident_pairs(h->device), h->num_sms / 2);
  if (pairs < 1) return SP_ERR_UNSUPPORTED;  // nothing launched; linear_tc_kernel takes the batch

  // the scratch follows the arrival counters, which stay zero for the other kernels
  uint8_t* scratch = static_cast<uint8_t*>(ws) + ws_counter_bytes(h->num_sms);
  DenseParams p{};
  p.cnt = static_cast<int*>(ws);
  p.ws = reinterpret_cast<float*>(scratch + scratch_bytes(h));
  p.y = y;
  p.scale = h->d_scale;
  p.status = device_status_ptr();
  p.N = h->N;
  p.M = M;
  p.rows = rows;
  p.T = h->T;
  p.y_tma = h->N % 8 == 0 ? 1 : 0;
  p.timeout_ns = wait_timeout_ns();
  plan_items(h, M, pairs, &p);
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
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  // after an in-place weight update the expansion waits for the whole previous grid
  attr[0].val.programmaticStreamSerializationAllowed = h->weights_written ? 0 : 1;
  cfg.gridDim = dim3((unsigned)C);
  cfg.blockDim = dim3(kRows);
  cfg.dynamicSmemBytes = (size_t)h->max_chunk;
  cfg.stream = stream;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  if (cudaLaunchKernelEx(&cfg, ek, h->d_buf, h->d_off, h->d_qidx, h->T, rows, reinterpret_cast<uint4*>(scratch),
                         p.timeout_ns, p.status) != cudaSuccess) {
    cudaGetLastError();
    return SP_ERR_CUDA;
  }
  h->weights_written = 0;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.gridDim = dim3((unsigned)(2 * std::min<int64_t>(pairs, p.items)));
  cfg.blockDim = dim3(kDenseThreads);
  cfg.dynamicSmemBytes = kDenseSmem;
  if (cudaLaunchKernelEx(&cfg, dense_kernel, p, map_w, map_x, map_y) != cudaSuccess) {
    cudaGetLastError();
    return SP_ERR_CUDA;
  }
  return SP_OK;
}

}  // namespace sp
