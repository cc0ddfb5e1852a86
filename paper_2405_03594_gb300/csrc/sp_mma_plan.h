// sp_mma_plan.h -- how linear_mma_kernel (sp_linear_mma.cu) is launched for a matrix and a batch:
// its form, split and shared-memory layout.  Host only and without CUDA calls, so that the
// layout can be checked on the CPU for every chunk size.
#pragma once

#include <algorithm>

#include "sp_internal.cuh"

namespace sp {
namespace mma {

constexpr int kMaxSlots = 16;

// Token tiles, rows per warp, consumer warps, CTAs per SM (at most) and per row block.
struct MmaChoice {
  int nt, rw, cw, occ, cluster;
};
struct MmaPlan {
  int slots, cluster;
  uint32_t chunk_region, ring_off, tab_off, bar_off, lut_off, rx_off;
  size_t smem;
};

// Largest cluster size of 2 .. 8 and 16 (9 .. 15 place badly) that keeps rb * S within `cap` CTAs
// and leaves a CTA at least `cmin` of the T K-tiles; 1 (a CTA per row block) otherwise.
inline int cluster_size(int64_t rb, int64_t T, int64_t cap, int cmin) {
  for (int64_t S = std::min<int64_t>(16, cap / rb); S > 1; --S)
    if ((S <= 8 || S == 16) && T / S >= cmin) return (int)S;
  return 1;
}

// A grid overlaps well with the launches around it if it fills the CTA slots to 80 % (the next
// grid's CTAs then follow its exits evenly) or leaves half of them free (the next grid fits
// beside it whole).  In between, part of the next grid gets in and the rest waits for the
// tail: such a grid keeps the next launch out until it exits.  Measured at M = 4, 70 %, next
// launch released early / at exit: 256 CTAs of 912 slots 8.5 / 10.3 us (o), 860 of 912
// 28.6 / 29.2 us (gate/up), but 512 of 912 22.1 / 18.3 us (down).
inline bool fills(int64_t grid, int64_t slots) { return grid * 5 >= slots * 4; }
inline bool overlaps(int64_t grid, int64_t slots) { return grid * 2 <= slots || fills(grid, slots); }

// More than 20 chunks per SM: throughput counts, below mostly latency.
inline bool large(const sp_matrix* h) { return (int64_t)h->RB * h->T > 20 * (int64_t)h->num_sms; }

// Ring slots and shared-memory layout for c.occ CTAs per SM; false if the ring does not hold a
// slot per chunk in work and one more (a dense matrix's chunks are ~17 KB).
inline bool mma_plan(const sp_matrix* h, int M, const MmaChoice& c, MmaPlan* pl) {
  const int groups = c.cw * c.rw / kRows;
  const int min_slots = groups < 4 ? groups + 1 : groups;
  pl->cluster = c.cluster;
  pl->chunk_region = (uint32_t)((h->max_chunk + 127) / 128 * 128);
  const size_t budget = ((size_t)(227 * 1024) / c.occ - 1024) / 128 * 128;  // all of it is asked for
  const size_t tab = (size_t)c.cw * c.rw * 16;
  const int S = pl->cluster;
  const size_t rx = c.nt == 1 && c.cw == 8 && S > 1 ? (size_t)(M + S - 1) / S * S * kRows * sizeof(float) : 0;  // receive area
  const size_t ctl = (size_t)kMaxSlots * (8 + 8 + 8 + 4) + 64 + rx;  // barriers, tags, table, receive area
  const size_t per_slot = (size_t)c.nt * 1024 + pl->chunk_region;
  if (budget < tab + ctl + min_slots * per_slot) return false;
  const int items = (h->T + pl->cluster - 1) / pl->cluster;
  pl->slots = (int)std::min<size_t>(std::min<size_t>(kMaxSlots, std::max(items, min_slots)),
                                    (budget - tab - ctl) / per_slot);
  pl->ring_off = (uint32_t)(pl->slots * c.nt * 1024);
  const size_t sums = (size_t)(c.cw * c.rw / kRows) * M * kRows * sizeof(float);  // on the ring
  const size_t ring_end = std::max<size_t>(pl->ring_off + (size_t)pl->slots * pl->chunk_region, (sums + 127) / 128 * 128);
  pl->tab_off = (uint32_t)ring_end;
  pl->bar_off = (uint32_t)(ring_end + tab);
  pl->lut_off = (uint32_t)(pl->bar_off + kMaxSlots * (8 + 8 + 8 + 4));  // a multiple of 64
  pl->rx_off = (uint32_t)(pl->bar_off + ctl - rx);
  if (pl->bar_off + ctl > budget) return false;
  // The whole share of shared memory, whatever the chunks need: CTAs of consecutive launches
  // then fit the holes that each other's leave.  Sizes following the largest chunk cost 33.2
  // instead of 27.9 us (gate/up, M = 4) between matrices 128 bytes apart, because the larger
  // CTA does not fit where the smaller one was.
  pl->smem = budget;
  return true;
}

// The launch of a batch of M <= kMmaMaxRows rows.  Two forms per token count: four consumer
// warps at a high occupancy, and eight, whose share of a row block per warp is shorter.
//  * Small matrices: best is one eight-warp CTA per SM
//    with as large a cluster as that allows, which also leaves room for the whole next grid:
//    o (32 row blocks) 8.4 -> 7.8 us at M = 2 against 256 four-warp CTAs, 8192 x 2048 8.4 -> 7.9.
//    With more row blocks than SMs, four warps and the largest cluster whose grid overlaps:
//    22016 x 512 8.3 -> 6.1 us against a CTA per row block released at exit.
//  * Larger matrices want every CTA slot full: eight warps where their grid fills the slots,
//    else four.  q/k/v (96 row blocks) 17.8 us with eight, 18.5 with four at M = 4, 20.3 / 21.5
//    at M = 16; down (32) 16.5 / 17.2 at M = 2 (80 %), 19.5 / 20.9 at M = 16; gate/up (172, eight
//    warps leave a quarter of the slots empty) 30.8 / 28.6 at M = 4, 41.0 / 32.4 at M = 16.
//  * Both at the largest occupancy whose share of shared memory holds the ring.  A large matrix
//    takes the cluster for that occupancy's slots: at 50 % with rows of uneven length (12 KB
//    chunks, five CTAs per SM instead of six) gate/up's 860 CTAs of a split for six ran as two
//    waves, 43.5 us at M = 4 against 34.0, and q/k/v of dense rows 78.6 / 59; gate/up of dense
//    rows (16-way bank conflicts, 516 CTAs in 608 slots) loses, 109 / 113.  A small one keeps
//    the wider split (22016 x 512, uneven 40 %, 8.7 us against 9.1).
inline bool choose(const sp_matrix* h, int M, MmaChoice* out, MmaPlan* pl) {
  const int nt = M <= 8 ? 1 : M <= 16 ? 2 : 4;
  const MmaChoice few = nt == 1 ? MmaChoice{1, 64, 4, 6, 1} : nt == 2 ? MmaChoice{2, 32, 4, 5, 1} : MmaChoice{4, 32, 4, 4, 1};
  const MmaChoice many = nt == 1 ? MmaChoice{1, 64, 8, 3, 1} : nt == 2 ? MmaChoice{2, 64, 8, 2, 1} : MmaChoice{4, 32, 8, 2, 1};
  const int64_t rb = std::max<int32_t>(h->RB, 1), T = h->T, sms = h->num_sms;
  MmaChoice& c = *out;
  if (!large(h) && rb <= sms) {
    c = many;
    c.cluster = cluster_size(rb, T, sms, 2);
    for (c.occ = 2; c.occ >= 1; --c.occ)
      if (mma_plan(h, M, c, pl)) return true;
    return false;
  }
  if (large(h))
    for (int occ = many.occ; occ >= 2; --occ) {
      c = many;
      c.occ = occ;
      c.cluster = cluster_size(rb, T, occ * sms, 8);
      const int64_t grid = rb * c.cluster;
      if (fills(grid, occ * sms) && grid <= occ * sms && mma_plan(h, M, c, pl)) return true;
    }
  int64_t wide = 1;  // the small matrix's cluster, by the kernel's own occupancy
  for (int64_t S = std::min<int64_t>(8, few.occ * sms / rb); S > 1 && wide == 1; --S)
    if (T / S >= 2 && overlaps(rb * S, few.occ * sms)) wide = S;
  for (int occ = few.occ; occ >= 1; --occ) {
    c = few;
    c.occ = occ;
    c.cluster = large(h) ? cluster_size(rb, T, occ * sms, 8) : (int)wide;
    if (mma_plan(h, M, c, pl)) return true;
  }
  return false;
}

}  // namespace mma
}  // namespace sp
