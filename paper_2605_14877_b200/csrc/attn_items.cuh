// What the two tensor-memory attention kernels share: tile sizes, tensor maps, key half-tiles and the cache update of their spare warps.
#pragma once
#include "append_device.cuh"
#include "tc_common.cuh"

namespace heatkv {
namespace tc {

constexpr int BM = 128;                 // rows per Q tile
constexpr int BN = 128;                 // keys per tile (two 64-row half-tiles)
constexpr int HALF = 64;
constexpr int STORE_COUNTER_WORD = 17;                         // word of the status region that hands out the cache-update items

struct Maps {
  CUtensorMap q, k_own, v_own, k_pool, v_pool, out;
};

// One key half-tile: where it comes from and how many of its 64 rows are real.
struct Slot {
  int pool_row;     // >= 0: row in the pool; < 0: own-scale tokens starting at -(pool_row + 1)
  int n_valid;
  int seg;
};

// FULL (calibration with an attention output): every key comes from the caller's tensor, and the descriptors, cut at
// source-scale borders, number its rows.
template <bool FULL>
__device__ __forceinline__ Slot get_slot(int i, const int2* descs, int n_desc, int n_slots, int64_t base_row,
                                         int t_own, int step) {
  Slot s;
  int valid = i < n_slots;
  if (!valid) i = n_slots - 1;                      // padding half-tile: re-read finite data, mask everything
  if (i < n_desc) {
    int2 d = descs[i];
    s.pool_row = FULL ? -(d.x + 1) : (int)(base_row + d.x);
    s.n_valid = d.y & 0xff;
    s.seg = (d.y >> 8) & 0xff;
  } else {
    int tok0 = (i - n_desc) * HALF;
    s.pool_row = -(tok0 + 1);
    s.n_valid = min(HALF, t_own - tok0);
    s.seg = step;
  }
  if (!valid) s.n_valid = 0;
  return s;
}

// Cache update by one warp: destination half-tiles of (sequence, head) units from a counter of its own.  Every store warp of the
// launch ends with one fetch past the end; the last of those store_items + n_warps fetches resets the counter.
template <int D>
__device__ __forceinline__ void store_rows_loop(const AttnParams& p, uint32_t n_warps, int lane) {
  const int u = (p.step * p.L + p.layer) * p.H;
  uint32_t* store_counter = p.status + STORE_COUNTER_WORD;
  const uint32_t fetches = (uint32_t)p.store_items + n_warps;
  for (;;) {
    uint32_t old = 0;
    if (lane == 0) {
      old = atomicAdd(store_counter, 1u);
      if (old == fetches - 1u) *reinterpret_cast<volatile uint32_t*>(store_counter) = 0;
    }
    const int a = (int)__shfl_sync(0xffffffffu, old, 0);
    if (a >= p.store_items) break;
    const int sq = a % p.n_seq, hd = (a / p.n_seq) % p.H, j = a / (p.n_seq * p.H);
    const int64_t src = sq * p.kv_seq + hd * p.kv_head;
    append_half_tile(append_place(p.seqs[sq].plan, p.seqs[sq].base_row, u + hd, j), p.k_new + src, p.v_new + src, p.kv_tok,
                     const_cast<__nv_bfloat16*>(p.k_pool), const_cast<__nv_bfloat16*>(p.v_pool), D, lane, 32);
  }
}

}  // namespace tc
}  // namespace heatkv
