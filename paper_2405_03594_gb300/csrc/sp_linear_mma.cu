// sp_linear_mma.cu -- sparse linear for batches of 2 .. 32 rows, and for one row of an INT8
// matrix that keeps many weights: chunks expanded in registers straight into the operands of
// warp-level matrix instructions.
//
// Between one row (linear_ccw_kernel walks the kept weights only) and a few dozen rows the
// product is bound by neither HBM nor the tensor pipe but by the work of turning a chunk's
// mask and packed values into operands.  A walk over kept weights on the CUDA cores pays M
// multiply-adds and M / 2 shuffles per weight; the tcgen05 kernel pays the trip through tensor
// memory on one CTA per SM, whatever the tokens.  Here a warp expands 16 columns of two rows per lane
// directly into the A registers of mma.sync m16n8k16 (bf16, FP32 accumulation), so the cost
// of a chunk hardly depends on M: four matrix instructions per 16 rows and 8 tokens beside
// ~290 instructions of expansion.  What takes most of its time is shared memory: ~520 wavefronts
// per chunk (predicated two-byte value loads at 1.6 each), 62 % of the peak rate over a gate/up
// launch (ncu), the rest being launch latency and tail.  Measured at 70 %, bf16, graphs of launches on
// matrices beyond L2, before / here: gate/up 32.2 / 28.1 us at M = 3, 48.7 / 28.4 at M = 5,
// 61.6 / 31.5 at M = 10, 46.4 / 32.1 at M = 16, 47.2 / 40.9 at M = 32; o 15.3 / 8.8, 18.2 / 9.6,
// 20.9 / 9.8, 23.4 / 12.8 at M = 5, 10, 16, 32; INT8 gate/up 54 / 30.8 at M = 5, 55.5 / 35.0 at
// M = 16.
//
// The product is free to permute K: in k-step s, lane (g, t) of a warp (g = lane / 4,
// t = lane % 4) supplies columns 16t + 4s .. 16t + 4s + 3 of its two rows, and of token g of
// x, so its 16 columns are one contiguous run of a row's values and of x's 128-byte tile row.
//
// CTA: one row block's share of K-tiles (a thread-block cluster of S CTAs covers the row
// block, as in linear_ccw_kernel).
//   warp CW, lane 0  producer: one cp.async.bulk per chunk and one TMA box of x (8 NT tokens
//                    x 64 columns, 128-byte swizzle; tokens past M and columns past K read as
//                    zero) into a ring of `slots` slots, full/empty mbarriers.
//   warps 0..CW-1    consumers.  128 / RW warps share a chunk, each taking RW of its rows; the
//                    CTA has CW * RW / 128 chunks in work.  A warp scans the popcounts of its
//                    16-column mask pieces into a table (mask piece, first value) of its own,
//                    and expands and multiplies 16 rows at a time.
// At the end of its K-tiles a CTA adds its warps' sums in warp order in shared memory (on the
// ring, which is idle by then); the cluster's CTAs then each sum a share of the tokens over
// all ranks in rank order (distributed shared memory: pushed to the owner by the eight-warp form
// up to 8 tokens, read by it otherwise) and write y through the launch's output epilogue.  All
// orders are fixed: results are bitwise repeatable.
#include <cuda.h>
#include <cudaTypedefs.h>

#include <algorithm>

#include "../../include/sp_stack.h"
#include "sp_expand.cuh"
#include "sp_mma_plan.h"

namespace sp {
namespace {

using namespace mma;

constexpr int kMaxDevices = 64;

struct MmaParams {
  const uint8_t* buf;
  const uint64_t* off;
  const uint64_t* qidx;
  const float* scale;  // INT8 only
  const uint16_t* x;
  uint16_t* y;
  const uint16_t* r;   // SP_EPI_RESIDUAL
  int* status;
  int64_t N, K, C;     // output rows; columns; chunks
  int32_t T, M;
  int32_t cluster;     // CTAs per row block
  int32_t slots;
  uint32_t chunk_region, ring_off, tab_off, bar_off, lut_off, rx_off;
  int32_t epi;
  int32_t early;       // release the next launch as soon as this one's inputs are ready
  int32_t kept_only;   // x of a dropped column takes no part, infinite or NaN either
  uint64_t timeout_ns;
};

// volatile: keeps its place among the (volatile) expansion steps, so that the table entries
// are not all loaded, and held in registers, at once
__device__ __forceinline__ uint32_t lds32(uint32_t saddr) {
  uint32_t v;
  asm volatile("ld.shared.b32 %0, [%1];" : "=r"(v) : "r"(saddr) : "memory");
  return v;
}
__device__ __forceinline__ void mma_bf16(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                         uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, "
      "%2, %3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// Four columns (bits 4S .. 4S + 3 of the mask piece m) as two bf16x2 from a row's value stream
// at shared address pa, which advances.
//
// bf16: a predicated load per column (sp_expand.cuh).  INT8: four values are one word, so the
// four columns' bytes are placed by a single byte permutation of the next four stream bytes (two
// aligned words and a funnel shift), its selector and the kept count looked up by the four mask
// bits in a 16-word table that no two lanes' different words share a bank of.  That takes 19
// instructions where four byte loads, their tests and increments took 24: gate/up 34.1 -> 30.5 us
// at M = 4, 70 %.
template <int ES, int S>
__device__ __forceinline__ void expand4(uint32_t m, uint32_t& pa, uint32_t lut, uint32_t& c01, uint32_t& c23) {
  if constexpr (ES == 2) {
    c01 = expand_word_bf16<1u << (4 * S), 2u << (4 * S)>(m, pa);
    c23 = expand_word_bf16<4u << (4 * S), 8u << (4 * S)>(m, pa);
  } else {
    const uint32_t e = lds32(lut + ((S == 0 ? m << 2 : m >> (4 * S - 2)) & 0x3cu));
    const uint32_t a = pa & ~3u;
    const uint32_t win = __funnelshift_r(lds32(a), lds32(a + 4), pa << 3);
    const uint32_t x = __byte_perm(win, 0u, e);
    pa += e >> 16;
    // byte q -> 0x43qq: 128 + its low seven bits, minus 128 or (sign bit) 256, as i8x2_to_bf16x2
    const uint32_t y0 = __byte_perm(x, 0x43434343u, 0x4140u), y1 = __byte_perm(x, 0x43434343u, 0x4342u);
    c01 = sub_bf16x2(y0 & 0xff7fff7fu, y0 & 0xff80ff80u);
    c23 = sub_bf16x2(y1 & 0xff7fff7fu, y1 & 0xff80ff80u);
  }
}
// Entry v of the table: the byte selector (a dropped column takes a zero byte) and, above it,
// the kept count.
__device__ __forceinline__ uint32_t lut_entry(uint32_t v) {
  uint32_t sel = 0, k = 0;
  for (int j = 0; j < 4; ++j) sel |= ((v >> j & 1u) ? k++ : 4u) << (4 * j);
  return sel | k << 16;
}

// 16 rows (two per lane) x 64 columns against NT token tiles.
template <int ES, int NT, int S>
__device__ __forceinline__ void tile_mma(uint32_t m0, uint32_t& pa0, uint32_t m1, uint32_t& pa1, uint32_t lut,
                                         const uint32_t (&xb)[NT][8], float (&acc)[NT][4]) {
  uint32_t a0, a1, a2, a3;
  expand4<ES, S>(m0, pa0, lut, a0, a2);
  expand4<ES, S>(m1, pa1, lut, a1, a3);
#pragma unroll
  for (int nt = 0; nt < NT; ++nt) mma_bf16(acc[nt], a0, a1, a2, a3, xb[nt][2 * S], xb[nt][2 * S + 1]);
  if constexpr (S + 1 < 4) tile_mma<ES, NT, S + 1>(m0, pa0, m1, pa1, lut, xb, acc);
}

// y[m, n] from its FP32 sum v (INT8: times the row's scale sc) through the launch's epilogue
// (sp_chain_epilogue).  All lanes of a warp call it together with consecutive rows n and one
// token m; rows past N write nothing.
__device__ __forceinline__ void write_one(const MmaParams& p, int64_t n, int m, float v, float sc) {
  const bool in = n < p.N;
  const uint32_t b = in ? float_to_bf16_bits_rn(v * sc) : 0u;
  if (p.epi == SP_EPI_PAIR_PRODUCT) {
    const uint32_t u = __shfl_xor_sync(0xffffffffu, b, 1);
    if (in && (n & 1) == 0)
      p.y[(int64_t)m * (p.N >> 1) + (n >> 1)] = float_to_bf16_bits_rn(bf16_bits_to_float(b) * bf16_bits_to_float(u));
  } else if (in) {
    uint16_t* yp = p.y + (int64_t)m * p.N + n;
    if (p.epi == SP_EPI_RESIDUAL)
      *yp = float_to_bf16_bits_rn(
          (bf16_bits_to_float(__ldcg(reinterpret_cast<const unsigned short*>(yp))) + bf16_bits_to_float(b)) +
          bf16_bits_to_float(p.r[n]));
    else
      *yp = (uint16_t)b;
  }
}

// Row rr of row block seg times tokens m, m + step, .. (four, those past M repeat m) over the kept
// columns of K-tiles [t0, t1), from global memory: the kept-weight walk's sums.  All lanes of a warp
// call it together with consecutive rows.  Bound by the latency of its loads.
template <int ES>
__device__ __forceinline__ float4 kept_sums(const MmaParams& p, int64_t seg, int t0, int t1, int rr, int m, int step) {
  const int lane = rr & 31;
  const uint16_t* x[4];
  float sum[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    x[j] = p.x + (int64_t)(m + j * step < p.M ? m + j * step : m) * p.K;
    sum[j] = 0.f;
  }
  for (int t = t0; t < t1; ++t) {
    const int64_t c = seg * p.T + t;
    const uint8_t* chunk = p.buf + p.off[c];
    uint64_t mk = reinterpret_cast<const uint64_t*>(chunk)[rr];
    const int pc = __popcll(mk);
    int e = pc;  // kept entries of the warp's rows up to this one
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const int u = __shfl_up_sync(0xffffffffu, e, d);
      if (lane >= d) e += u;
    }
    e -= pc;
    if (rr >= 32) e += (int)((p.qidx[c] >> (16 * (rr / 32 - 1))) & 0xffffu);
    const uint8_t* val = chunk + kMaskBytes + (int64_t)e * ES;
    while (mk) {
      float w[4], v[4][4];
      bool on[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        on[i] = mk != 0;
        if (on[i]) {
          const int64_t k = (int64_t)kTileK * t + __ffsll((long long)mk) - 1;
          w[i] = ES == 2 ? bf16_bits_to_float(*reinterpret_cast<const uint16_t*>(val))
                         : (float)*reinterpret_cast<const int8_t*>(val);
#pragma unroll
          for (int j = 0; j < 4; ++j)
            v[i][j] = bf16_bits_to_float(__ldcg(reinterpret_cast<const unsigned short*>(x[j] + k)));
          val += ES;
          mk &= mk - 1;
        }
      }
#pragma unroll
      for (int i = 0; i < 4; ++i)
        if (on[i]) {
#pragma unroll
          for (int j = 0; j < 4; ++j) sum[j] = fmaf(w[i], v[i][j], sum[j]);
        }
    }
    __syncwarp();
  }
  return make_float4(sum[0], sum[1], sum[2], sum[3]);
}

// The matrix product multiplies a dropped column's +0 with x, which for an infinite or NaN x makes
// every row of the token NaN; the walk, which runs the CUDA-core family's other batches, never
// touches a dropped column.  For that family the CTA's sums ([groups][M][kRows] in comb) that are
// not finite are therefore taken again over the kept columns, by the thread that reads them next:
// row rr of tokens m0, m0 + step, ..  Finite inputs pay a multiply-add per sum and a vote, where the
// sums are read anyway: gate/up at M = 4 27.64 -> 27.69 us, a captured step of four layers at
// M = 4 304.9 -> 307.3.  In line, and only in the forms that need it: a call, taken or not, costs
// every launch ~0.2 us (the step 309.6; at 16 rows, which never take it, 375.2 -> 379); tested in the
// registers, before the sums meet in shared memory, gate/up took 27.95.  With a NaN in one of 3 to
// 10 tokens o takes 100 us, gate/up 110 to 136.
template <int ES>
__device__ __forceinline__ void redo_sums(const MmaParams& p, float* comb, int64_t seg, int t0, int t1, int rr, int m0,
                                       int step, int groups) {
  const int M = p.M;
  for (int m = m0; m < M; m += 4 * step) {
    bool redo[4];
    bool any = false;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int mj = m + j * step;
      float z = 0.f;
      for (int q = 0; mj < M && q < groups; ++q) z = fmaf(comb[(q * M + mj) * kRows + rr], 0.f, z);
      any |= redo[j] = z != z;
    }
    if (!__any_sync(0xffffffffu, any)) continue;
    const float4 k = kept_sums<ES>(p, seg, t0, t1, rr, m, step);
    const float kj[4] = {k.x, k.y, k.z, k.w};
#pragma unroll
    for (int j = 0; j < 4; ++j)
      if (redo[j]) {
        for (int q = 0; q < groups; ++q) comb[(q * M + m + j * step) * kRows + rr] = q == 0 ? kj[j] : 0.f;
      }
  }
}

// KO: the batch may be the CUDA-core family's (p.kept_only says), whose sums that are not finite are
// taken again.
template <int NT, int ES, int RW, int CW, int OCC, bool KO>
__global__ void __launch_bounds__((CW + 1) * 32, OCC)
    linear_mma_kernel(const __grid_constant__ MmaParams p, const __grid_constant__ CUtensorMap tmap_x) {
  extern __shared__ __align__(1024) uint8_t smem[];
  constexpr int kParts = kRows / RW;       // warps that share a chunk
  constexpr int kGroups = CW / kParts;     // chunks in work at once
  constexpr int R = RW / 32;               // rows per lane in the scan
  constexpr int kTiles = RW / 16;          // 16-row tiles of a warp
  constexpr uint32_t kXBytes = NT * 1024u;
  constexpr bool kPush = NT == 1 && CW == 8;  // how the cluster's sums meet (at the end)
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int slots = p.slots;
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + p.bar_off);
  uint64_t* empty = full + kMaxSlots;
  uint64_t* qx = empty + kMaxSlots;                                   // quarter index of each slot's chunk
  volatile int* tag = reinterpret_cast<volatile int*>(qx + kMaxSlots);  // item each slot was claimed for
  const int T = p.T;
  const int64_t seg = blockIdx.x / p.cluster;  // row block
  const int rank = blockIdx.x % p.cluster;
  const int t0 = (int)((int64_t)rank * T / p.cluster), t1 = (int)((int64_t)(rank + 1) * T / p.cluster);
  const int n_items = t1 - t0;

  if (tid == 0) {
    for (int s = 0; s < slots; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], kParts);
      tag[s] = -1;
    }
    fence_barrier_init();
  }
  if (ES == 1 && warp == 1 && lane < 16) reinterpret_cast<uint32_t*>(smem + p.lut_off)[lane] = lut_entry(lane);
  __syncthreads();
  if (kPush && p.cluster > 1) cluster_arrive_relaxed();  // this CTA runs: its shared memory may be written

  if (warp == CW) {
    // ------------------------------------------------------------ producer
    const uint64_t pol = policy_evict_first();
    const int64_t c0 = seg * T + t0;
    int64_t base = -64;  // offsets (and quarter indices) of chunks base .. base + 31, one per lane
    uint64_t vo = 0, vq = 0;
    auto chunk_at = [&](int i, uint64_t* o0, uint64_t* o1, uint64_t* qi) {
      const int64_t c = c0 + i;
      if (c - base >= 31 || c < base) {
        base = c;
        vo = c + lane <= p.C ? __ldg(p.off + c + lane) : 0ull;
        if (kParts > 1) vq = c + lane < p.C ? __ldg(p.qidx + c + lane) : 0ull;
      }
      *o0 = __shfl_sync(0xffffffffu, vo, (int)(c - base));
      *o1 = __shfl_sync(0xffffffffu, vo, (int)(c - base) + 1);
      if (kParts > 1) *qi = __shfl_sync(0xffffffffu, vq, (int)(c - base));
    };
    auto issue_chunk = [&](int i, int s, uint64_t o0, uint64_t o1, uint64_t qi) {
      const uint32_t bytes = (uint32_t)(o1 - o0);
      if (kGroups > 1) tag[s] = i;
      if (kParts > 1) qx[s] = qi;
      mbar_arrive_expect_tx(&full[s], bytes + kXBytes);
      bulk_g2s_hint(smem + p.ring_off + (size_t)s * p.chunk_region, p.buf + o0, bytes, &full[s], pol);
    };
    if (lane == 0) prefetch_tmap(&tmap_x);
    const int n_pre = n_items < slots ? n_items : slots;
    for (int i = 0; i < n_pre; ++i) {  // weight bytes do not depend on the previous grid
      uint64_t o0, o1, qi = 0;
      chunk_at(i, &o0, &o1, &qi);
      if (lane == 0) issue_chunk(i, i, o0, o1, qi);
    }
    pdl_wait();
    if (p.early) pdl_launch_dependents();
    int s = 0;
    uint32_t ph = 0;
    bool failed = false;
    for (int i = 0; i < n_items; ++i) {
      if (i >= n_pre) {
        uint64_t o0, o1, qi = 0;
        chunk_at(i, &o0, &o1, &qi);
        if (lane == 0) {
          if (!mbar_wait(&empty[s], ph ^ 1u, p.timeout_ns)) {
            set_status(p.status, kStatusTimeout);
            failed = true;
          } else {
            issue_chunk(i, s, o0, o1, qi);
          }
        }
        failed = __shfl_sync(0xffffffffu, failed, 0);
        if (failed) break;
      }
      if (lane == 0) tma_load_2d(smem + (size_t)s * kXBytes, &tmap_x, kTileK * (t0 + i), 0, &full[s]);
      if (++s == slots) {
        s = 0;
        ph ^= 1u;
      }
    }
    return;
  }

  // -------------------------------------------------------------- consumers
  pdl_wait();
  if (p.early) pdl_launch_dependents();
  const int grp = warp / kParts, part = warp % kParts;
  const int g = lane >> 2, t = lane & 3;
  // The table entry of piece t of row 8q + g of the warp's rows is word 4 * (8q + (g ^ (q % R))) + t:
  // a tile's loads are one 128-byte line, and the turn by q keeps the 16-byte stores of the scan,
  // in which lane l writes rows R l .. R l + R - 1, off each other's banks.
  uint32_t* tab = reinterpret_cast<uint32_t*>(smem + p.tab_off) + warp * RW * 4;
  const uint32_t lut = smem_u32(smem + p.lut_off);
  const uint32_t tab_lane = smem_u32(tab) + 16u * g + 4u * t;
  const int turn = R == 4 ? (lane >> 1) & 3 : R == 2 ? (lane >> 2) & 1 : 0;
  float acc[kTiles][NT][4];
#pragma unroll
  for (int i = 0; i < kTiles; ++i)
#pragma unroll
    for (int nt = 0; nt < NT; ++nt)
#pragma unroll
      for (int c = 0; c < 4; ++c) acc[i][nt][c] = 0.f;
  bool dead = false;
  int s = grp;
  uint32_t ph = 0;
  for (int n = grp; n < n_items; n += kGroups) {
    // one vote, in front of which every lane comes: the slot is claimed for this item (where
    // other warps' items pass through it too) and its copies have landed
    if (!dead && !__all_sync(0xffffffffu, (kGroups == 1 || wait_claimed(tag + s, n, p.timeout_ns)) &&
                                              mbar_wait(&full[s], ph, p.timeout_ns))) {
      dead = true;
      set_status(p.status, kStatusTimeout);
    }
    if (!dead) {
      const uint8_t* chunk = smem + p.ring_off + (size_t)s * p.chunk_region;
      // ---- table: lane l scans rows R l .. R l + R - 1 of the warp's part
      {
        uint32_t w[2 * R];  // mask words, 32 columns each
        if constexpr (R == 1) {
          const uint2 a = reinterpret_cast<const uint2*>(chunk)[part * RW + lane];
          w[0] = a.x, w[1] = a.y;
        } else {
#pragma unroll
          for (int i = 0; i < R / 2; ++i) {
            const uint4 a = reinterpret_cast<const uint4*>(chunk)[part * (RW / 2) + lane * (R / 2) + i];
            w[4 * i] = a.x, w[4 * i + 1] = a.y, w[4 * i + 2] = a.z, w[4 * i + 3] = a.w;
          }
        }
        int before[4 * R], run = 0;
#pragma unroll
        for (int i = 0; i < 2 * R; ++i) {
          before[2 * i] = run;
          before[2 * i + 1] = run + __popc(w[i] & 0xffffu);
          run += __popc(w[i]);
        }
        int incl = run;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
          const int u = __shfl_up_sync(0xffffffffu, incl, d);
          if (lane >= d) incl += u;
        }
        int e0 = incl - run;
        if constexpr (kParts > 1) {  // kept entries before rows 32, 64, 96: the chunk's quarter index
          const uint64_t qi = qx[s];
          if (part > 0) e0 += (int)((qi >> (16 * (part * (RW / 32) - 1))) & 0xffffu);
        }
        __syncwarp();  // the last chunk's reads of the table
#pragma unroll
        for (int e = 0; e < R; ++e) {
          uint32_t v[4];
#pragma unroll
          for (int k = 0; k < 4; ++k)
            v[k] = __byte_perm(w[2 * e + (k >> 1)], (uint32_t)(e0 + before[4 * e + k]), (k & 1) ? 0x5432 : 0x5410);
          reinterpret_cast<uint4*>(tab)[R * lane + (e ^ turn)] = make_uint4(v[0], v[1], v[2], v[3]);
        }
        __syncwarp();
      }
      // ---- x: token 8 nt + g, columns 16t .. 16t + 15 (two 16-byte pieces of its swizzled row)
      uint32_t xb[NT][8];
      const uint8_t* xs = smem + (size_t)s * kXBytes + g * 128;
#pragma unroll
      for (int nt = 0; nt < NT; ++nt) {
        const uint4 a = *reinterpret_cast<const uint4*>(xs + nt * 1024 + (((2 * t) ^ g) << 4));
        const uint4 b = *reinterpret_cast<const uint4*>(xs + nt * 1024 + (((2 * t + 1) ^ g) << 4));
        xb[nt][0] = a.x, xb[nt][1] = a.y, xb[nt][2] = a.z, xb[nt][3] = a.w;
        xb[nt][4] = b.x, xb[nt][5] = b.y, xb[nt][6] = b.z, xb[nt][7] = b.w;
      }
      const uint32_t vbase = smem_u32(chunk) + kMaskBytes;
#pragma unroll
      for (int i = 0; i < kTiles; ++i) {
        // rows 16 i + g and 16 i + 8 + g of the warp's part
        const uint32_t en0 = lds32((tab_lane ^ (16u * ((2 * i) % R))) + 256u * i);
        const uint32_t en1 = lds32((tab_lane ^ (16u * ((2 * i + 1) % R))) + 256u * i + 128u);
        uint32_t pa0 = vbase + (en0 >> 16) * ES, pa1 = vbase + (en1 >> 16) * ES;
        tile_mma<ES, NT, 0>(en0, pa0, en1, pa1, lut, xb, acc[i]);
      }
    }
    __syncwarp();
    if (lane == 0) mbar_arrive(&empty[s]);
    if ((s += kGroups) >= slots) {
      s -= slots;
      ph ^= 1u;
    }
  }

  // ---------------------------------------------------------------- the CTA's sums
  // Every copy into the ring has landed (its item was waited for), so the ring's memory now
  // holds the partials: [kGroups][M][kRows] floats, group 0's part becoming the CTA's sum.
  named_bar_sync(1, CW * 32);
  const int M = p.M;
  float* comb = reinterpret_cast<float*>(smem);
#pragma unroll
  for (int i = 0; i < kTiles; ++i)
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const int row = part * RW + 16 * i + 8 * (c >> 1) + g;
#pragma unroll
      for (int nt = 0; nt < NT; ++nt) {
        const int tok = 8 * nt + 2 * t + (c & 1);
        if (tok < M) comb[(grp * M + tok) * kRows + row] = acc[i][nt][c];
      }
    }
  named_bar_sync(1, CW * 32);
  // warps 4h .. 4h + 3 take tokens h, h + CW / 4, ...; a thread takes one row
  constexpr int kStep = CW / 4;
  const int rr = tid % kRows, m0 = tid / kRows;
  const int64_t row = seg * kRows + rr;
  const float sc = (ES == 1 && row < p.N) ? p.scale[row] : 1.f;
  auto cta_sum = [&](int m) {
    float v = comb[m * kRows + rr];
#pragma unroll
    for (int q = 1; q < kGroups; ++q) v += comb[(q * M + m) * kRows + rr];
    return v;
  };
  // z: 0 times each of the warp's sums, added up; not 0 if one of them is not finite.  The CUDA-core
  // family's batches (at most 16 rows a launch) then take those sums again.
  auto redo = [&](float z, int groups) {
    if (!KO || !__any_sync(0xffffffffu, p.kept_only && z != 0.f)) return false;
    redo_sums<ES>(p, comb, seg, t0, t1, rr, m0, kStep, groups);
    return true;
  };
  float z = 0.f;
  if (p.cluster == 1) {
    if (KO && p.kept_only) {
      for (int m = m0; m < M; m += kStep) z = fmaf(cta_sum(m), 0.f, z);
      redo(z, kGroups);
    }
    for (int m = m0; m < M; m += kStep) write_one(p, row, m, cta_sum(m), sc);
    return;
  }
  if constexpr (kPush) {
    // Few tokens: rank m % S owns token m, and every CTA stores its sum of it straight into the
    // owner's receive area ([tokens owned][S][kRows] floats, apart from the ring, which the
    // owner may still be using): one cluster barrier at the end.  Reading the sums from the
    // other CTAs' memory takes one before, so that they are there, and one after, so that they
    // stay.  Measured, read / pushed: 512 x 11008 7.6 / 7.2 us, down at 80 % 17.4 / 16.9, q/k/v
    // at 50 % 21.6 / 21.0 (M = 4).  The four-warp form reads: its grids fill every CTA slot, and
    // how the CTAs leave decides how evenly the next launch's come in (gate/up 28.1 us read at
    // M = 3 and 4, pushed 30.0 and 26.9).
    const int S = p.cluster;
    const uint32_t rx = smem_u32(smem + p.rx_off) + 4u * (uint32_t)(rank * kRows + rr);
    cluster_wait();
    auto push = [&](int m, float v) {
      st_cluster_f32(cluster_map(rx + 4u * (uint32_t)(m / S * S * kRows), (uint32_t)(m % S)), v);
    };
    for (int m = m0; m < M; m += kStep) {
      const float v = cta_sum(m);
      push(m, v);
      z = fmaf(v, 0.f, z);
    }
    if (redo(z, kGroups))
      for (int m = m0; m < M; m += kStep) push(m, cta_sum(m));
    cluster_arrive_release();
    cluster_wait();
    const float* got = reinterpret_cast<const float*>(smem + p.rx_off) + rr;
    for (int m = rank + m0 * S; m < M; m += kStep * S) {
      float v = 0.f;
#pragma unroll 4
      for (int q = 0; q < S; ++q) v += got[(m / S * S + q) * kRows];
      write_one(p, row, m, v, sc);
    }
    return;
  }
  if (kGroups > 1 || (KO && p.kept_only)) {
    for (int m = m0; m < M; m += kStep) {
      const float v = cta_sum(m);
      if (kGroups > 1) comb[m * kRows + rr] = v;
      z = fmaf(v, 0.f, z);
    }
    redo(z, 1);
  }
  cluster_sync_all();
  const uint32_t mine = smem_u32(comb) + 4u * (uint32_t)rr;
  for (int m = rank + m0 * p.cluster; m < M; m += kStep * p.cluster) {
    float v = 0.f;
#pragma unroll 4
    for (int q = 0; q < p.cluster; ++q) v += ld_cluster_f32(cluster_map(mine + 4u * (uint32_t)(m * kRows), (uint32_t)q));
    write_one(p, row, m, v, sc);
  }
  cluster_sync_all();  // every CTA's sums stay until the others have read them
}

// ------------------------------------------------------------------ host side
template <int NT, int ES, int RW, int CW, int OCC, bool KO>
sp_status launch(const sp_matrix* h, const MmaParams& p, const CUtensorMap& map, const MmaPlan& pl,
                 cudaStream_t stream, bool pdl) {
  auto kern = linear_mma_kernel<NT, ES, RW, CW, OCC, KO>;
  static bool configured[kMaxDevices] = {};
  const int dev = h->device;
  if (dev < 0 || dev >= kMaxDevices) return SP_ERR_UNSUPPORTED;
  if (!configured[dev]) {
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024) != cudaSuccess ||
        cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) {
      cudaGetLastError();
      return SP_ERR_CUDA;
    }
    configured[dev] = true;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(h->RB * pl.cluster));
  cfg.blockDim = dim3((CW + 1) * 32);
  cfg.dynamicSmemBytes = pl.smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = pdl ? 1 : 0;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = (unsigned)pl.cluster;
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = pl.cluster > 1 ? 2 : 1;
  if (cudaLaunchKernelEx(&cfg, kern, p, map) != cudaSuccess) {
    cudaGetLastError();
    return SP_ERR_CUDA;
  }
  return SP_OK;
}

template <int ES>
sp_status dispatch(const sp_matrix* h, const MmaParams& p, const CUtensorMap& map, const MmaPlan& pl,
                   const MmaChoice& c, cudaStream_t stream, bool pdl) {
  if (c.nt == 1)
    return c.cw == 4 ? launch<1, ES, 64, 4, 6, true>(h, p, map, pl, stream, pdl)
                     : launch<1, ES, 64, 8, 3, true>(h, p, map, pl, stream, pdl);
  if (c.nt == 2 && p.kept_only)
    return c.cw == 4 ? launch<2, ES, 32, 4, 5, true>(h, p, map, pl, stream, pdl)
                     : launch<2, ES, 64, 8, 2, true>(h, p, map, pl, stream, pdl);
  if (c.nt == 2)
    return c.cw == 4 ? launch<2, ES, 32, 4, 5, false>(h, p, map, pl, stream, pdl)
                     : launch<2, ES, 64, 8, 2, false>(h, p, map, pl, stream, pdl);
  return c.cw == 4 ? launch<4, ES, 32, 4, 4, false>(h, p, map, pl, stream, pdl)
                   : launch<4, ES, 32, 8, 2, false>(h, p, map, pl, stream, pdl);
}

}  // namespace

// One row, and two of a large matrix, stay with the kept-weight walk, whose time follows the
// weights kept, except where an INT8 matrix keeps many: its walk takes an instruction more per
// weight, the expansion here the same time at any sparsity.  Four layers of the Llama-2 7B stack,
// INT8, walk / here: M = 2 at 50 % 592 / 334 us, 60 % 396 / 334, 70 % 350 / 332, 80 % 299 / 331;
// M = 1 (the o linear, 14 chunks per SM, on the walk) at 50 % 383 / 321, at 60 % 341 / 321, at 70 %
// 299 / 321.  bf16 at M = 2: 364 / 370, 327 / 350, 295 / 319, 260 / 294; at M = 1 357 / 389,
// 307 / 359, 263 / 321, 224 / 298.  The lines on the kept share come from that stack alone.
bool uses_mma(const sp_matrix* h, int64_t M) {
  if (M < 1 || M > kMmaMaxRows || (M == 1 && !large(h))) return false;
  if (M == 1 || (M == 2 && large(h))) {
    const double kept = (double)h->nnz / ((double)h->N * (double)h->K);
    if (h->esize == 2 || kept < (M == 1 ? 0.36 : 0.26)) return false;
  }
  MmaChoice c;
  MmaPlan pl;
  return choose(h, (int)M, &c, &pl);
}

sp_status launch_linear_mma(const sp_matrix* h, const uint16_t* x, int64_t M, uint16_t* y, cudaStream_t stream,
                            int32_t epi, const uint16_t* r, bool kept_only) {
  if (M < 1 || M > kMmaMaxRows) return SP_ERR_UNSUPPORTED;
  MmaChoice c;
  MmaPlan pl;
  if (!choose(h, (int)M, &c, &pl)) return SP_ERR_UNSUPPORTED;
  PFN_cuTensorMapEncodeTiled_v12000 encode = nullptr;
  sp_status st = tensor_map_encoder(&encode);
  if (st != SP_OK) return st;
  MmaParams p{};
  p.buf = h->d_buf;
  p.off = h->d_off;
  p.qidx = h->d_qidx;
  p.scale = h->d_scale;
  p.x = x;
  p.y = y;
  p.r = r;
  p.status = device_status_ptr();
  p.N = h->N;
  p.K = h->K;
  p.C = (int64_t)h->RB * h->T;
  p.T = h->T;
  p.M = (int32_t)M;
  p.cluster = pl.cluster;
  p.slots = pl.slots;
  p.chunk_region = pl.chunk_region;
  p.ring_off = pl.ring_off;
  p.tab_off = pl.tab_off;
  p.bar_off = pl.bar_off;
  p.lut_off = pl.lut_off;
  p.rx_off = pl.rx_off;
  p.epi = epi;
  p.kept_only = kept_only ? 1 : 0;
  p.early = overlaps((int64_t)h->RB * pl.cluster, (int64_t)c.occ * h->num_sms) ? 1 : 0;
  p.timeout_ns = wait_timeout_ns();
  // x [M, K] bf16, box = 64 columns x 8 NT tokens, 128-byte swizzle; rows past M and columns
  // past K read as zero
  CUtensorMap map;
  const cuuint64_t gdim[2] = {(cuuint64_t)h->K, (cuuint64_t)M};
  const cuuint64_t gstride[1] = {(cuuint64_t)h->K * 2};
  const cuuint32_t box[2] = {(cuuint32_t)kTileK, (cuuint32_t)(8 * c.nt)};
  const cuuint32_t estride[2] = {1, 1};
  if (encode(&map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<uint16_t*>(x), gdim, gstride, box, estride,
             CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
    return SP_ERR_CUDA;
  // after an in-place weight update the launch waits for the whole previous grid (no weight
  // copy may start before its writes are visible)
  const bool pdl = !h->weights_written;
  st = h->esize == 2 ? dispatch<2>(h, p, map, pl, c, stream, pdl) : dispatch<1>(h, p, map, pl, c, stream, pdl);
  if (st == SP_OK) h->weights_written = 0;
  return st;
}

}  // namespace sp
