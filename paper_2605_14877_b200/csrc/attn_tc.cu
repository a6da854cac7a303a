// Tensor-memory attention kernel for the large scale steps (head_dim 128 or 64).
//
// The launch is a list of work items handed out through a counter: one CTA per SM stays resident and takes
// item after item, so the loads and first products of the next item run under the epilogue of the current
// one.  An attention item is 256 queries of one (sequence, head) as two 128-row tiles A and B that share
// the key/value stream, over the head's whole key range or one piece of it.  When the call carries the
// cache update, the rows of the step's own K/V are copied by two otherwise idle warps, which take
// destination half-tiles from a counter of their own.  Warp roles:
//   warp 0      fetches and decodes items (a two-entry ring in shared memory) and is the TMA producer:
//               Q tiles once per item, then K and V half-tiles (64 rows x 128 dims each) gathered
//               through the plan's page table, followed by the step's own keys.
//   warp 1      MMA issuer: S = Q K^T and O += P V with tcgen05.mma, accumulators in TMEM.
//   warps 2-3   cache update (only when the call carries it).
//   warps 4-7   softmax of tile A, warps 8-11 softmax of tile B: one thread per query row
//               reads its row of S from TMEM, keeps the running max / sum, writes P (bf16)
//               back into the columns S occupied, and rescales O only when the row max grew
//               by more than 2^32 since the last reference (the sum keeps the same reference,
//               so the result is exact).  The same warps write the item's result.
// Times of whole cases in this file's comments are GPU time of short bursts (SM clock 1.6 to 1.9 GHz), both sides in turn on
// one box; back to back, under the power limit, the same passes take 6 to 14 % longer.
// TMEM columns: S_A/P_A 0..127, S_B/P_B 128..255, O_A 256..383, O_B 384..511.
// The MMA order S_A S_B (PV_A S_A' PV_B S_B')* lets the softmax of one tile overlap the
// tensor work of the other.  The host may cut a head's key range into pieces (a count per head); their
// unnormalised results meet in a scratch region, where, for every group of 32 rows, the warp that arrives
// last adds them up in piece order.  An item may also be a single query tile (the host's choice for launches that leave SMs idle, and the
// odd last tile of a head beside those): then A and B are its even and its odd key tiles, so that one's softmax runs under the
// other's products as it does for two query tiles, and the two results meet in the CTA.  All barrier phases run on across items.  Every wait is bounded; on expiry the
// CTA records a status word, drains its own copies and leaves.
#include <algorithm>
#include <climits>

#include "attn_items.cuh"
#include "internal.h"

namespace heatkv {

namespace tc {

constexpr int THREADS = 384;
constexpr int KV_STAGES = 2;
// Registers are handed from the four utility warps to the eight softmax warps.  setmaxnreg only moves
// registers inside the CTA's own allocation (threads x registers at launch), so the two budgets must fit
// in it; an increase that cannot be served would block for ever.
constexpr int REGS_LAUNCH = 168;        // what ptxas assigns under __launch_bounds__(384, 1)
constexpr int REGS_SMALL = 72;
constexpr int REGS_SOFTMAX = 216;
static_assert(128 * REGS_SMALL + 256 * REGS_SOFTMAX <= THREADS * REGS_LAUNCH, "register hand-over exceeds the CTA's allocation");
constexpr uint32_t HALF_COLS_BYTES = 128 * 128;        // one 64-column half of a 128-row tile: 16 KB
constexpr uint32_t SLOT_BYTES = HALF * 128;            // 64 rows x 128 B inside one column half
constexpr uint32_t STAGE_BYTES = 4096;                 // per softmax warp: two buffers of 32 rows x 64 B for the output rows

// Sizes that follow the head dimension D (64 or 128): a 128-row tile is D / 64 column halves of 16 KB.
template <int D>
struct Layout {
  static_assert(D == 64 || D == 128, "head dimension");
  static constexpr int NCH = D / 64;                             // 64-column halves per row
  static constexpr uint32_t TILE_BYTES = NCH * HALF_COLS_BYTES;  // 16 or 32 KB
  // shared memory map (bytes from a 1024-aligned base)
  static constexpr uint32_t SM_Q = 0;                                   // 2 tiles
  static constexpr uint32_t SM_K = SM_Q + 2 * TILE_BYTES;               // KV_STAGES tiles
  static constexpr uint32_t SM_V = SM_K + KV_STAGES * TILE_BYTES;       // KV_STAGES tiles
  static constexpr uint32_t SM_OUT = SM_V + KV_STAGES * TILE_BYTES;     // output staging of the eight softmax warps
  static constexpr uint32_t SM_BAR = SM_OUT + 8 * STAGE_BYTES;          // barriers + scalars + item ring
  static constexpr uint32_t SM_TOTAL = SM_BAR + 512;
  static constexpr uint32_t SM_ALLOC = SM_TOTAL + 1024;                 // slack for manual alignment
  static_assert(SM_ALLOC <= 227 * 1024, "shared memory of one CTA");
  // One partial result of a split head: unnormalised O of both query tiles (fp32, groups of four columns
  // outermost so that a warp's 32 rows touch consecutive 16-byte words), then the rows' running references
  // and row sums.
  static constexpr int SPLIT_SLOT_FLOATS = 2 * BM * D + 2 * 2 * BM;
};

// barrier slots (8 bytes each) inside SM_BAR
enum Bar : uint32_t {
  Q_FULL = 0, Q_EMPTY = 2,      // +x
  K_FULL = 4, K_EMPTY = 6,      // +stage
  V_FULL = 8, V_EMPTY = 10,     // +stage
  S_FULL = 12,                  // +x  S_x of the tile is in TMEM
  P_FULL = 14,                  // +2x+h  half h (keys 64h..64h+63) of P_x of the tile is in TMEM (128 arrivals)
  PV_DONE = 18,                 // +x  O_x includes the item's last tile (one completion per item)
  ITEM_FULL = 20, ITEM_EMPTY = 22,  // +ring entry; EMPTY takes one arrival from the MMA warp and each softmax warp
  MEET = 24,                    // +w  the two softmax warps of 32 rows in an item of one query tile: two phases per item
  N_BARS = 28
};
constexpr uint32_t BAR_TMEM_PTR = N_BARS * 8;                  // offsets inside the barrier region
constexpr uint32_t BAR_ABORT = BAR_TMEM_PTR + 4;
constexpr uint32_t BAR_RING = 256;                             // 2 entries x int32[16]
constexpr float SUM_LIMIT = 4294967296.f;                      // 2^RESCALE_THRESHOLD: no term of a sum below it is above it
// FULL: items of at most so many key tiles (the largest such step of a 1024 x 1024 image has 1024 queries) move the reference
// with every rise of a maximum.  P is rounded to bf16 relative to it, and the few keys that carry a short row are
// rounded best just below a power of two: output error against 64 bits, 64 queries 2.31e-3 -> 2.12e-3 of the norm, 1024:
// 2.36e-3 -> 2.27e-3, a pass of 13 scales 2.177e-3 -> 2.107e-3 (warp-level kernel 2.13e-3, 2.27e-3, 2.094e-3) for 3 % of its
// time.  In longer rows no few keys matter that much (4096 queries 2.35e-3, 2.30e-3 on the warp-level kernel) and following
// cost 15 to 20 %.
constexpr int FOLLOW_TILES = 24;
enum ItemKind : int { ATTENTION = 0, STOP = 2, NOTHING = 3 };
// ring entry words
enum ItemWord : int { W_KIND = 0, W_HEAD, W_SEQ, W_TILES, W_NSPLIT, W_SUB, W_SLOT, W_CTR, W_DESC, W_NDESC };

constexpr int WORK_COUNTER_WORD = 16;                          // word of the status region that hands out the attention items


// What every role derives from a ring entry of kind ATTENTION.
struct Item {
  int head, seq, n_split, sub, piece, qp, q0, nq, j0, n_tiles, slot_base, ctr_base, n_desc, n_slots, desc_begin;
  // One query tile, its key tiles taken by the two softmax warpgroups in turn (S_A, O_A: tiles 0, 2, ..; S_B, O_B: 1, 3, ..)
  bool shared;
};
// (the shuffle makes a word provably warp-uniform)
__device__ __forceinline__ int ring_word(const volatile int32_t* ring, int word) {
  return __shfl_sync(0xffffffffu, ring[word], 0);
}
template <bool FULL, bool LONE>
__device__ __forceinline__ Item read_item(const volatile int32_t* ring, const AttnParams& p, int n_qp) {
  Item it;
  it.head = ring_word(ring, W_HEAD);
  it.seq = ring_word(ring, W_SEQ);
  it.n_split = ring_word(ring, W_NSPLIT);
  it.sub = ring_word(ring, W_SUB);
  it.slot_base = ring_word(ring, W_SLOT);
  it.ctr_base = ring_word(ring, W_CTR);
  it.desc_begin = ring_word(ring, W_DESC);
  it.n_desc = ring_word(ring, W_NDESC);
  const int tiles = ring_word(ring, W_TILES);
  const bool one = LONE && it.n_split < 0;          // the head's items are single query tiles
  it.piece = LONE ? 0 : it.sub / n_qp;
  it.qp = LONE ? it.sub : it.sub % n_qp;
  it.q0 = it.qp * (one ? BM : 2 * BM);
  it.nq = (!one && it.q0 + BM < p.t_q) ? 2 : 1;     // does tile B hold any query?
  if (FULL) {                                       // one query tile of the pair (W_SLOT: 0 both, 1 the first, 2 the second)
    const int single = ring_word(ring, W_SLOT);
    if (single > 0) it.nq = 1;
    if (single == 2) it.q0 += BM;
  }
  it.shared = LONE && it.nq == 1;
  it.n_slots = FULL ? it.n_desc : it.n_desc + (p.n_own + HALF - 1) / HALF;
  // this item's run of key tiles: [j0, j0 + n_tiles) of the head's ceil(n_slots / 2)
  const int piece_tiles = LONE ? tiles : (tiles + it.n_split - 1) / it.n_split;
  it.j0 = it.piece * piece_tiles;
  it.n_tiles = min(tiles, it.j0 + piece_tiles) - it.j0;
  return it;
}

// LONE: some of the launch's items are a single query tile, none is a piece of a head.  An instantiation of its own, because
// each way of ending an item costs the others: with the pieces' code beside it a launch took 1.5 us more (from the second
// kind of item in a launch on, the instruction caches hold neither), and one kernel for everything 0.3 to 1.5 us more everywhere.
// What bounds such an item is what bounds a pair: 28 heads x 576 queries, 0.80 us per key tile where a pair takes 1.52; filled SMs
// 1.02 and 1.83.  Keys come one tile ahead of the values here, a step is half as long (in the pair's order 1.35 us).
// FULL: heatkv_calibrate_scores with an attention output.  The softmax warps also keep, for every query row, the
// probability mass of each source scale (a half-tile lies inside one scale; finished scales are parked in the warp's
// output staging buffer) and add the step's row of beta (Eq. 2) at the end of the item.  The masses are fp32 results, so all
// exponentials are ex2's here: with one pair in four from the cubic beta was off by 3.8e-7 on average (13 scales, against 64
// bits), with none by 1.0e-7 (warp-level kernel 1.3e-7), for 1 % of the time.
template <int D, bool FULL, bool LONE>
__global__ void __launch_bounds__(THREADS, 1)
attn_tc_kernel(const __grid_constant__ AttnParams p, const __grid_constant__ Maps maps) {
  using L = Layout<D>;
  constexpr int NCH = L::NCH;
  // Where the softmax itself weighs most: half the tensor work per exponential (64-wide heads), or masses to keep besides
  // (FULL).  Measured: generation with 64-wide heads 1.673 -> 1.629 ms, calibration with output (128-wide) 1.186 -> 1.142;
  // 128-wide generation, where a product's latency is the larger part of the chain, was 0.3 to 0.8 % slower with it.
  constexpr bool SPECULATE = FULL || D == 64;
  constexpr uint32_t TILE_BYTES = L::TILE_BYTES, SM_Q = L::SM_Q, SM_K = L::SM_K, SM_V = L::SM_V, SM_OUT = L::SM_OUT,
                     SM_BAR = L::SM_BAR, SM_TMEM_PTR = L::SM_BAR + BAR_TMEM_PTR, SM_ABORT = L::SM_BAR + BAR_ABORT,
                     SM_RING = L::SM_BAR + BAR_RING;
  constexpr int SPLIT_SLOT_FLOATS = L::SPLIT_SLOT_FLOATS;
  extern __shared__ unsigned char smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t sbase = (raw + 1023u) & ~1023u;
  unsigned char* sgen = smem_raw + (sbase - raw);
  volatile uint32_t* abort_flag = reinterpret_cast<volatile uint32_t*>(sgen + SM_ABORT);
  volatile uint32_t* tmem_ptr_smem = reinterpret_cast<volatile uint32_t*>(sgen + SM_TMEM_PTR);
  volatile int32_t* ring_base = reinterpret_cast<volatile int32_t*>(sgen + SM_RING);
  auto bar = [&](uint32_t which) { return sbase + SM_BAR + which * 8; };

  // the shuffle makes the warp index provably warp-uniform, so role code stays on the uniform datapath
  const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
  const int u = (p.step * p.L + p.layer) * p.H;
  const int n_qp = (p.t_q + 2 * BM - 1) / (2 * BM);

  pdl_trigger();
  if (threadIdx.x == 0) {
    *abort_flag = *reinterpret_cast<volatile uint32_t*>(p.status) != 0;   // an earlier CTA gave up: do not wait again
    for (int x = 0; x < 2; ++x) {
      mbar_init(bar(Q_FULL + x), 1);
      mbar_init(bar(Q_EMPTY + x), 1);
      mbar_init(bar(S_FULL + x), 1);
      mbar_init(bar(P_FULL + 2 * x), BM);
      mbar_init(bar(P_FULL + 2 * x + 1), BM);
      mbar_init(bar(PV_DONE + x), 1);
      mbar_init(bar(ITEM_FULL + x), 1);
      mbar_init(bar(ITEM_EMPTY + x), 9);
    }
    for (int w = 0; w < 4; ++w) mbar_init(bar(MEET + w), 2);
    for (int s = 0; s < KV_STAGES; ++s) {
      mbar_init(bar(K_FULL + s), 1);
      mbar_init(bar(K_EMPTY + s), 1);
      mbar_init(bar(V_FULL + s), 1);
      mbar_init(bar(V_EMPTY + s), 1);
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 0) {
    __syncwarp();
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(sbase + SM_TMEM_PTR), "r"(512u)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = __shfl_sync(0xffffffffu, *tmem_ptr_smem, 0);
  // (every role waits for the launches before this one where it first touches what they may still use, and before its first
  // wait for another role: the tries of a bounded wait are for this CTA's own copies and products, not for a launch that is
  // still running)

  // register budget per warpgroup: 128*72 + 256*216 <= 64K
  if (warp < 4) {
    reg_dealloc<REGS_SMALL>();
  if (warp == 0) {
    // ------------------------------------------------------------------ item fetch + TMA producer
    const bool leader = elect_one();
    const int own_slots = (p.n_own + HALF - 1) / HALF;
    uint32_t* work_counter = p.status + WORK_COUNTER_WORD;
    uint32_t g = 0;                                    // key tiles handed to the copy engine so far (all items)
    uint32_t iq[2] = {0, 0};                           // items that loaded query tile x so far
    uint32_t armed_k = 0, armed_v = 0, armed_q = 0;    // bit per barrier: a copy was issued at least once
    uint32_t par_k = 0, par_v = 0, par_q = 0;          // bit per barrier: parity of the phase its last copy completes
    bool ok = true;
    for (uint32_t it = 0; ok; ++it) {
      // The first item of a CTA is its block index; later ones come from the counter.  Every CTA ends with
      // one fetch past the end, so the launch makes exactly attn_items fetches and the last resets the counter.
      int idx = blockIdx.x;
      if (it > 0) {
        if (it == 1) pdl_wait();
        uint32_t old = 0;
        if (lane == 0) {
          old = atomicAdd(work_counter, 1u);
          if (old == (uint32_t)p.attn_items - 1u) *reinterpret_cast<volatile uint32_t*>(work_counter) = 0;
        }
        idx = (int)gridDim.x + (int)__shfl_sync(0xffffffffu, old, 0);
      }
      const uint32_t slot = it & 1;
      volatile int32_t* ring = ring_base + slot * 16;
      if (it >= 2) ok = warp_wait(bar(ITEM_EMPTY + slot), ((it >> 1) - 1) & 1, abort_flag, p.status);
      if (!ok) break;
      if (idx >= p.attn_items) {
        if (lane == 0) ring[W_KIND] = STOP;
        __syncwarp();
        if (leader) mbar_arrive(bar(ITEM_FULL + slot));
        break;
      }
      // Attention items: sequences interleaved; the items of one sequence run over its heads by descending
      // key count (the plan's order); a head may be cut into equal pieces of its key range (the count comes
      // from the host's table, else from the launch's longest run), and every (piece, query tile pair) is
      // one item, pieces outermost.  A prefix sum over the
      // heads finds the item.
      // (FULL: past full_whole the items are single query tiles, so that the last round of CTAs is not half empty)
      const int pair = FULL && idx > p.full_whole ? p.full_whole + (idx - p.full_whole) / 2 : idx;
      const int seq = pair % p.n_seq;
      const int item = pair / p.n_seq;
      if (lane == 0) {
        ring[W_KIND] = FULL ? ATTENTION : NOTHING;      // sequences of a call may differ in item count
        if (FULL) {                                     // all heads alike: query tile pair fastest
          ring[W_HEAD] = item / n_qp;
          ring[W_SEQ] = seq;
          ring[W_TILES] = (p.full_slots + 1) >> 1;
          ring[W_NSPLIT] = 1;
          ring[W_SUB] = item % n_qp;
          ring[W_CTR] = ring[W_DESC] = 0;
          ring[W_SLOT] = idx < p.full_whole ? 0 : 1 + ((idx - p.full_whole) & 1);
          if (ring[W_SLOT] == 2 && item % n_qp * (2 * BM) + BM >= p.t_q) ring[W_KIND] = NOTHING;
          ring[W_NDESC] = p.full_slots;
        }
      }
      __syncwarp();
      if (!FULL) {
        PlanView pv(p.seqs[seq].plan);
        int before = 0, slots_before = 0, ctrs_before = 0;
        for (int base = 0; base < p.H; base += 32) {
          const int i = base + lane;
          int h = 0, tiles = 0, ns = 0, cnt = 0;
          if (i < p.H) {
            if (p.table_heads > 0) {                            // the host put the per-head table into the launch parameters
              h = p.table_head[i];
              tiles = p.table_tiles[i];
              ns = p.table_split[i];
            } else {
              h = pv.order()[u + i];
              tiles = (pv.attn_cnt(p.runs)[u + h] + own_slots + 1) >> 1;
              ns = p.split_tiles > 0 ? (tiles + p.split_tiles - 1) / p.split_tiles : 1;
              if (LONE && p.lone == 2) ns = -ns;
            }
            cnt = !LONE ? n_qp * ns : ns > 0 ? n_qp : (p.t_q + BM - 1) / BM;    // below 0: the head's query tiles one by one
          }
          const int scnt = !LONE && ns > 1 ? cnt : 0, ccnt = !LONE && ns > 1 ? n_qp : 0;
          int inc = cnt, sinc = scnt, cinc = ccnt;
#pragma unroll
          for (int o = 1; o < 32; o <<= 1) {
            const int v0 = __shfl_up_sync(0xffffffffu, inc, o), v1 = __shfl_up_sync(0xffffffffu, sinc, o),
                      v2 = __shfl_up_sync(0xffffffffu, cinc, o);
            if (lane >= o) { inc += v0; sinc += v1; cinc += v2; }
          }
          const int excl = before + inc - cnt;
          const bool mine = cnt > 0 && item >= excl && item < excl + cnt;
          if (mine) {
            ring[W_HEAD] = h;
            ring[W_SEQ] = seq;
            ring[W_TILES] = tiles;
            ring[W_NSPLIT] = ns;
            ring[W_SUB] = item - excl;                        // piece * n_qp + query tile pair, or (no pieces) query tile
            ring[W_SLOT] = slots_before + sinc - scnt;        // first partial slot of this head
            ring[W_CTR] = ctrs_before + cinc - ccnt;          // first arrival counter group of this head
            ring[W_DESC] = p.table_heads > 0 ? p.table_desc_begin[i] : pv.w[p.runs ? 18 : 4] + 2 * pv.attn_begin(p.runs)[u + h];
            ring[W_NDESC] = p.table_heads > 0 ? (int)p.table_ndesc[i] : pv.attn_cnt(p.runs)[u + h];
            ring[W_KIND] = ATTENTION;
          }
          const bool any = __any_sync(0xffffffffu, mine);
          before += __shfl_sync(0xffffffffu, inc, 31);
          slots_before += __shfl_sync(0xffffffffu, sinc, 31);
          ctrs_before += __shfl_sync(0xffffffffu, cinc, 31);
          if (any) break;
        }
        __syncwarp();
      }
      const bool is_attn = ring_word(ring, W_KIND) == ATTENTION;
      Item im;
      if (is_attn) im = read_item<FULL, LONE>(ring, p, n_qp);
      __syncwarp();
      if (leader) mbar_arrive(bar(ITEM_FULL + slot));
      if (!is_attn) continue;
      const int2* descs = FULL ? p.full_descs : reinterpret_cast<const int2*>(p.seqs[seq].plan + im.desc_begin);
      const int64_t base_row = FULL ? 0 : p.seqs[seq].base_row;
      const int q_head = im.head & p.q_head_mask, q_seq = seq & p.q_seq_mask;
      const int kv_head = im.head & p.kv_head_mask, kv_seq = seq & p.kv_seq_mask;
      if (g == 0 && leader) {
        // What the first item's first copies will fetch, sent for while the launch before may still run (10 steps x 16 layers of a
        // pair of images 1741 -> 1723 us, 7 steps x 32 layers, of which one runs on CTA pairs, 1186 -> 1171)
        for (int hf = 0; hf < 2; ++hf) {
          const int row = get_slot<FULL>(2 * im.j0 + hf, descs, im.n_desc, im.n_slots, base_row, p.n_own, p.step).pool_row;
          for (int ch = 0; ch < NCH; ++ch) {
            if (row >= 0 && p.k8_pool) {                      // staging rows: the launch before is writing them
            } else if (row >= 0) {
              tma_prefetch_2d(&maps.k_pool, ch * 64, row);
              tma_prefetch_2d(&maps.v_pool, ch * 64, row);
            } else {
              tma_prefetch_4d(&maps.k_own, ch * 64, -row - 1, kv_head, kv_seq);
              tma_prefetch_4d(&maps.v_own, ch * 64, -row - 1, kv_head, kv_seq);
            }
            for (int x = 0; x < im.nq; ++x)
              tma_prefetch_4d(&maps.q, ch * 64, im.q0 + x * BM + hf * HALF, q_head, q_seq);
          }
        }
      }
      __syncwarp();
      if (LONE && im.shared) {
        // Pool rows of 32 half-tiles at a time, one per lane (a look-up per tile would be a chain of its own).
        const int first_slot = 2 * im.j0;
        int rows = 0, rows_at = -32;
        auto half_tile = [&](int i) {
          if (i >= rows_at + 32) {
            rows_at = i;
            rows = get_slot<FULL>(first_slot + i + lane, descs, im.n_desc, im.n_slots, base_row, p.n_own, p.step).pool_row;
          }
          return __shfl_sync(0xffffffffu, rows, i - rows_at);
        };
        auto load = [&](uint32_t smem, const CUtensorMap* pool, const CUtensorMap* own, int row0, int row1, uint32_t full) {
          if (!leader) return;
          mbar_expect_tx(full, TILE_BYTES);
          for (int hf = 0; hf < 2; ++hf)
            for (int ch = 0; ch < NCH; ++ch) {
              const int row = hf == 0 ? row0 : row1;
              const uint32_t dst = smem + ch * HALF_COLS_BYTES + hf * SLOT_BYTES;
              if (row >= 0) tma_load_2d(dst, pool, ch * 64, row, full);
              else tma_load_4d(dst, own, ch * 64, -row - 1, kv_head, kv_seq, full);
            }
        };
        auto load_k = [&](uint32_t t, int row0, int row1) {             // t: key tiles before it, over all items
          const uint32_t st = t % KV_STAGES, use = t / KV_STAGES;
          if (use > 0) ok = warp_wait(bar(K_EMPTY + st), (use - 1) & 1, abort_flag, p.status);
          if (!ok) return;
          armed_k |= 1u << st;
          par_k = (par_k & ~(1u << st)) | ((use & 1) << st);
          load(sbase + SM_K + st * TILE_BYTES, &maps.k_pool, &maps.k_own, row0, row1, bar(K_FULL + st));
        };
        int next0 = 0, next1 = 0;                                       // half-tiles of the tile whose keys came ahead
        for (int j = 0; j < im.n_tiles && ok; ++j, ++g) {
          const int row0 = j > 0 ? next0 : half_tile(0), row1 = j > 0 ? next1 : half_tile(1);
          // the first item is decoded and its descriptors are read while the launch before may still run
          if (g == 0) pdl_wait();
          // K first: the S product of the next tile needs it earliest
          if (j == 0) load_k(g, row0, row1);
          if (!ok) break;
          if (j == 0) {
            if (iq[0] > 0) ok = warp_wait(bar(Q_EMPTY), (iq[0] - 1) & 1, abort_flag, p.status);
            if (!ok) break;
            armed_q |= 1u;
            par_q = (par_q & ~1u) | (iq[0] & 1);
            ++iq[0];
            if (leader) {
              mbar_expect_tx(bar(Q_FULL), TILE_BYTES);
              for (int ch = 0; ch < NCH; ++ch)
                for (int hf = 0; hf < 2; ++hf)
                  tma_load_4d(sbase + SM_Q + ch * HALF_COLS_BYTES + hf * SLOT_BYTES, &maps.q, ch * 64, im.q0 + hf * HALF, q_head, q_seq,
                              bar(Q_FULL));
            }
          }
          if (j + 1 < im.n_tiles) {             // the step is half as long: the next keys do not wait behind these values
            next0 = half_tile(2 * j + 2);
            next1 = half_tile(2 * j + 3);
            load_k(g + 1, next0, next1);
            if (!ok) break;
          }
          const uint32_t st = g % KV_STAGES, use = g / KV_STAGES;
          if (use > 0) ok = warp_wait(bar(V_EMPTY + st), (use - 1) & 1, abort_flag, p.status);
          if (!ok) break;
          armed_v |= 1u << st;
          par_v = (par_v & ~(1u << st)) | ((use & 1) << st);
          load(sbase + SM_V + st * TILE_BYTES, &maps.v_pool, &maps.v_own, row0, row1, bar(V_FULL + st));
          __syncwarp();
        }
      } else {
        for (int j = 0; j < im.n_tiles && ok; ++j, ++g) {
          const uint32_t st = g % KV_STAGES;
          const uint32_t use = g / KV_STAGES;
          Slot sl[2];
          for (int hf = 0; hf < 2; ++hf)
            sl[hf] = get_slot<FULL>(2 * (im.j0 + j) + hf, descs, im.n_desc, im.n_slots, base_row, p.n_own, p.step);
          // the first item is decoded and its descriptors are read while the launch before may still run
          if (g == 0) pdl_wait();
          // K first: the S product of the next tile needs it earliest
          if (use > 0) ok = warp_wait(bar(K_EMPTY + st), (use - 1) & 1, abort_flag, p.status);
          if (!ok) break;
          armed_k |= 1u << st;
          par_k = (par_k & ~(1u << st)) | ((use & 1) << st);
          if (leader) {
            mbar_expect_tx(bar(K_FULL + st), TILE_BYTES);
            for (int hf = 0; hf < 2; ++hf)
              for (int ch = 0; ch < NCH; ++ch) {
                uint32_t dst = sbase + SM_K + st * TILE_BYTES + ch * HALF_COLS_BYTES + hf * SLOT_BYTES;
                if (sl[hf].pool_row >= 0) tma_load_2d(dst, &maps.k_pool, ch * 64, sl[hf].pool_row, bar(K_FULL + st));
                else tma_load_4d(dst, &maps.k_own, ch * 64, -sl[hf].pool_row - 1, kv_head, kv_seq, bar(K_FULL + st));
              }
          }
          if (j == 0) {
            // the item's query tiles, once the last S product of the previous item has read the old ones
#pragma unroll
            for (int x = 0; x < 2; ++x) {
              if (x >= im.nq || !ok) continue;
              if (iq[x] > 0) ok = warp_wait(bar(Q_EMPTY + x), (iq[x] - 1) & 1, abort_flag, p.status);
              if (!ok) continue;
              armed_q |= 1u << x;
              par_q = (par_q & ~(1u << x)) | ((iq[x] & 1) << x);
              ++iq[x];
              if (leader) {
                mbar_expect_tx(bar(Q_FULL + x), TILE_BYTES);
                for (int ch = 0; ch < NCH; ++ch)
                  for (int hf = 0; hf < 2; ++hf)
                    tma_load_4d(sbase + SM_Q + x * TILE_BYTES + ch * HALF_COLS_BYTES + hf * SLOT_BYTES, &maps.q, ch * 64,
                                im.q0 + x * BM + hf * HALF, q_head, q_seq, bar(Q_FULL + x));
              }
            }
            if (!ok) break;
          }
          if (use > 0) ok = warp_wait(bar(V_EMPTY + st), (use - 1) & 1, abort_flag, p.status);
          if (!ok) break;
          armed_v |= 1u << st;
          par_v = (par_v & ~(1u << st)) | ((use & 1) << st);
          if (leader) {
            mbar_expect_tx(bar(V_FULL + st), TILE_BYTES);
            for (int hf = 0; hf < 2; ++hf)
              for (int ch = 0; ch < NCH; ++ch) {
                uint32_t dst = sbase + SM_V + st * TILE_BYTES + ch * HALF_COLS_BYTES + hf * SLOT_BYTES;
                if (sl[hf].pool_row >= 0) tma_load_2d(dst, &maps.v_pool, ch * 64, sl[hf].pool_row, bar(V_FULL + st));
                else tma_load_4d(dst, &maps.v_own, ch * 64, -sl[hf].pool_row - 1, kv_head, kv_seq, bar(V_FULL + st));
              }
          }
          __syncwarp();
        }
      }
      __syncwarp();
    }
    if (!ok || *abort_flag) {
      // leaving early: let every copy this warp started land before the CTA exits
      for (int s = 0; s < KV_STAGES; ++s) {
        if (armed_k & (1u << s))
          for (uint32_t t = 0; t < WAIT_LIMIT && !mbar_try(bar(K_FULL + s), (par_k >> s) & 1); ++t) {}
        if (armed_v & (1u << s))
          for (uint32_t t = 0; t < WAIT_LIMIT && !mbar_try(bar(V_FULL + s), (par_v >> s) & 1); ++t) {}
      }
      for (int x = 0; x < 2; ++x)
        if (armed_q & (1u << x))
          for (uint32_t t = 0; t < WAIT_LIMIT && !mbar_try(bar(Q_FULL + x), (par_q >> x) & 1); ++t) {}
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------------ MMA issuer
    // This warp's instruction stream is part of every key tile's chain (P handed over -> PV, next S -> softmax), so it is kept
    // short: item words and the TMEM base come through a shuffle and are provably uniform, and the products are predicated on
    // one lane instead of branched around.  Measured: a pair generated at 20x 2.395 -> 2.339 ms of GPU time, the largest
    // model's batch 7.025 -> 6.763 ms, 64-wide heads unchanged (1.66 ms); one thread running the whole role lost 5 %.  The lane is
    // elected anew for every tile and the descriptors are a base and a constant: 65 instructions less per tile, 1024 queries x 296
    // heads x 24 tiles 369.4 -> 363.5 us in a burst (64-wide heads 306.7 -> 302.7), 449.0 -> 446.4 under the power limit.  What matters is that the compiler knows the warp to be
    // converged: where it does not (a `continue` past the __syncwarp at the loop's end, a lane mask that a failed wait may clear) it
    // branches around every product, 33 branches and 350 instructions more per tile, and the kernel is 6 % slower.
    const uint32_t lead = elect_one();
    constexpr uint32_t IDESC_S = instr_desc(BM, BN, 0, 0);     // Q, K both K-major
    constexpr uint32_t IDESC_PV = instr_desc(BM, D, 0, 1);     // P from TMEM, V MN-major
    pdl_wait();
    bool ok = true;
    // 64-wide heads wait with the vote in the loop (1.621 -> 1.588 ms); for 128-wide ones it measured 1 to 2 % slower
    auto mma_wait = [&](uint32_t b, uint32_t parity) {
      return D == 64 ? warp_wait_vote(b, parity, abort_flag, p.status) : warp_wait(b, parity, abort_flag, p.status);
    };
    const uint32_t q_lo = desc_lo(sbase + SM_Q, 16), k_lo = desc_lo(sbase + SM_K, 16), v_lo = desc_lo(sbase + SM_V, HALF_COLS_BYTES);
    auto issue_s = [&](uint32_t lead, int qx, int x, int st) {                // S_x = Q_qx K^T
      const uint32_t qa = q_lo + qx * (TILE_BYTES >> 4), ka = k_lo + st * (TILE_BYTES >> 4);
#pragma unroll
      for (int ks = 0; ks < D / 16; ++ks) {
        const uint32_t off = ((ks >> 2) * HALF_COLS_BYTES + (ks & 3) * 32) >> 4;
        mma_ss(lead, tmem + x * 128, qa + off, ka + off, IDESC_S, ks > 0);
      }
    };
    // keys 64h .. 64h+63 of the tile: four K=16 steps
    auto issue_pv = [&](uint32_t lead, int x, int st, int h, bool first) {
      const uint32_t va = v_lo + st * (TILE_BYTES >> 4);
#pragma unroll
      for (int ks = 4 * h; ks < 4 * h + 4; ++ks)
        mma_ts(lead, tmem + 256 + x * 128, tmem + x * 128 + ks * 8, va + ks * (2048 >> 4), IDESC_PV, !(first && ks == 0));
    };
    uint32_t g = 0;                                    // key tiles consumed so far (all items)
    uint32_t cx[2] = {0, 0};                           // key tiles of query tile x so far
    uint32_t iq[2] = {0, 0};                           // items with query tile x so far
    for (uint32_t it = 0; ok; ++it) {
      const uint32_t slot = it & 1;
      volatile int32_t* ring = ring_base + slot * 16;
      ok = mma_wait(bar(ITEM_FULL + slot), (it >> 1) & 1);
      if (!ok) break;
      const int kind = ring_word(ring, W_KIND);
      if (kind == STOP) break;
      if (kind == ATTENTION) {
        const Item im = read_item<FULL, LONE>(ring, p, n_qp);
        const int nq = im.nq, n_tiles = im.n_tiles;
        const uint32_t st0 = g % KV_STAGES, par0 = (g / KV_STAGES) & 1;
        if (LONE && im.shared) {
          // One query tile: key tile t goes through S, P and O number t & 1, so that the softmax of one tile overlaps the
          // products of the next as it does with two query tiles.
          static_assert(KV_STAGES == 2, "tile t + 2 takes the stage of tile t");
          ok = mma_wait(bar(Q_FULL), iq[0] & 1);
          for (int t = 0; t < min(n_tiles, 2) && ok; ++t) {
            const uint32_t st = (g + t) % KV_STAGES;
            ok = mma_wait(bar(K_FULL + st), ((g + t) / KV_STAGES) & 1);
            if (!ok) break;
            tc_fence_after();
            issue_s(lead, 0, t, st);
            tc_commit(lead, bar(S_FULL + t));
            tc_commit(lead, bar(K_EMPTY + st));
            if (t + 1 == n_tiles) tc_commit(lead, bar(Q_EMPTY));
          }
#pragma unroll 1
          for (int t = 0; t < n_tiles && ok; ++t) {
            const uint32_t x = t & 1, st = (g + t) % KV_STAGES, par = ((g + t) / KV_STAGES) & 1;
            const uint32_t ph = ((x ? cx[1] : cx[0]) + (t >> 1)) & 1;
            const bool more = t + 2 < n_tiles;
            ok = mma_wait(bar(V_FULL + st), par);
            if (ok) ok = mma_wait(bar(P_FULL + 2 * x), ph);
            if (!ok) break;
            tc_fence_after();
            issue_pv(lead, x, st, 0, t < 2);
            if (more) ok = mma_wait(bar(K_FULL + st), par ^ 1);
            if (ok) ok = mma_wait(bar(P_FULL + 2 * x + 1), ph);
            if (!ok) break;
            tc_fence_after();
            issue_pv(lead, x, st, 1, false);
            tc_commit(lead, bar(V_EMPTY + st));
            if (more) {
              issue_s(lead, 0, x, st);
              tc_commit(lead, bar(S_FULL + x));
              tc_commit(lead, bar(K_EMPTY + st));
              if (t + 3 == n_tiles) tc_commit(lead, bar(Q_EMPTY));
            }
          }
          if (ok) {
            tc_commit(lead, bar(PV_DONE));
            tc_commit(lead, bar(PV_DONE + 1));
          }
          g += n_tiles;
          cx[0] += (n_tiles + 1) >> 1;
          cx[1] += n_tiles >> 1;
          ++iq[0];
        } else {
#pragma unroll
        for (int x = 0; x < 2; ++x)
          if (x < nq && ok) ok = mma_wait(bar(Q_FULL + x), iq[x] & 1);
        if (ok) ok = mma_wait(bar(K_FULL + st0), par0);
        if (ok) {
          tc_fence_after();
          for (int x = 0; x < nq; ++x) {
            issue_s(lead, x, x, st0);
            tc_commit(lead, bar(S_FULL + x));
            if (n_tiles == 1) tc_commit(lead, bar(Q_EMPTY + x));
          }
          tc_commit(lead, bar(K_EMPTY + st0));
        }
        // Waits for K and V sit where the tensor pipe still has queued work: the next tile's V at the end
        // of an iteration, the next tile's K between the two halves of PV_A.  The hand-over of P is then
        // the only wait between the last S product of one tile and the first PV product of the next.
        if (ok) ok = mma_wait(bar(V_FULL + st0), par0);
        for (int j = 0; j < n_tiles && ok; ++j) {
          const uint32_t st = (g + j) % KV_STAGES, stn = (g + j + 1) % KV_STAGES;
          const uint32_t parn = ((g + j + 1) / KV_STAGES) & 1;
          const bool more = j + 1 < n_tiles;
          const uint32_t lead = elect_one();
#pragma unroll
          for (int x = 0; x < 2; ++x) {
            if (x >= nq || !ok) continue;
            const uint32_t ph = (cx[x] + j) & 1;
            ok = mma_wait(bar(P_FULL + 2 * x), ph);
            if (!ok) continue;
            tc_fence_after();
            issue_pv(lead, x, st, 0, j == 0);
            // the next tile's keys are waited for here, off the path between the last half of P and the next S
            if (more && x == 0) ok = mma_wait(bar(K_FULL + stn), parn);
            if (!ok) continue;
            ok = mma_wait(bar(P_FULL + 2 * x + 1), ph);
            if (!ok) continue;
            tc_fence_after();
            issue_pv(lead, x, st, 1, false);
            if (more) {
              issue_s(lead, x, x, stn);
              tc_commit(lead, bar(S_FULL + x));
              if (j + 2 == n_tiles) tc_commit(lead, bar(Q_EMPTY + x));     // the item's last product that reads Q_x
            } else {
              tc_commit(lead, bar(PV_DONE + x));                     // only the epilogue waits for it
            }
          }
          if (ok) {
            tc_commit(lead, bar(V_EMPTY + st));
            if (more) tc_commit(lead, bar(K_EMPTY + stn));
          }
          if (ok && more) ok = mma_wait(bar(V_FULL + stn), parn);
        }
        g += n_tiles;
#pragma unroll
        for (int x = 0; x < 2; ++x)
          if (x < nq) {
            cx[x] += n_tiles;
            ++iq[x];
          }
        }
      }
      __syncwarp();
      if (ok && lead) mbar_arrive(bar(ITEM_EMPTY + slot));
    }
  } else if (p.store_items > 0) {
    // ------------------------------------------------------------------ cache update (warps 2 and 3)
    // their rows are copied while the other warps work on attention items
    pdl_wait();
    store_rows_loop<D>(p, 2u * gridDim.x, lane);
  }
  } else {
    reg_alloc<REGS_SOFTMAX>();
    // ------------------------------------------------------------------ softmax + epilogue + cache-update items
    const int x = (warp - 4) >> 2;                      // 0: tile A, 1: tile B
    const int row = (warp & 3) * 32 + lane;             // row inside the tile == TMEM lane
    const uint32_t lane_base = (uint32_t)((warp & 3) * 32) << 16;
    const uint32_t t_s = tmem + lane_base + x * 128;
    const uint32_t t_o = tmem + lane_base + 256 + x * 128;
    unsigned char* stage = sgen + SM_OUT + (warp - 4) * STAGE_BYTES;
    const float LOG2E = 1.4426950408889634f;
    uint32_t cx = 0;                                    // key tiles of this query tile so far (all items)
    uint32_t items_x = 0;                               // items in which this query tile held rows so far
    pdl_wait();
    bool ok = true;
    for (uint32_t it = 0; ok; ++it) {
      const uint32_t slot = it & 1;
      volatile int32_t* ring = ring_base + slot * 16;
      ok = __all_sync(0xffffffffu, mbar_wait(bar(ITEM_FULL + slot), (it >> 1) & 1, abort_flag, p.status));
      if (!ok) break;
      const int kind = ring_word(ring, W_KIND);
      if (kind == STOP) break;
      if (kind == ATTENTION) {
        // Only what the tile loop needs stays in registers; the epilogue reads the ring entry again.
        int n_tiles, nq;
        {
          const Item im = read_item<FULL, LONE>(ring, p, n_qp);
          n_tiles = im.shared ? (im.n_tiles + 1 - x) >> 1 : im.n_tiles;      // those this warpgroup takes
          nq = im.shared ? 2 : im.nq;
        }
        if (x < nq) {
          int j0, n_desc, n_slots, q0, stride, piece = INT_MAX, in_piece = 2, first_looks = 1;
          const int2* descs;
          const float* bias_h;
          {
            const Item im = read_item<FULL, LONE>(ring, p, n_qp);
            stride = im.shared ? 2 : 1;
            j0 = im.shared ? x : im.j0; n_desc = im.n_desc; n_slots = im.n_slots; q0 = im.q0;
            if (!FULL && LONE && abs(im.n_split) > 1) {                        // the pieces the head would be cut into (`look` below)
              piece = (im.n_tiles + abs(im.n_split) - 1) / abs(im.n_split);
              in_piece = j0;
              first_looks = stride;
            }
            descs = FULL ? p.full_descs : reinterpret_cast<const int2*>(p.seqs[im.seq].plan + im.desc_begin);
            bias_h = p.seg_bias ? p.seg_bias + im.head * p.K : nullptr;
          }
          float m_ref = NO_MAX, l_sum = 0.f;
          // FULL: the scale whose mass is being collected (warp-uniform; scales arrive in ascending order, each as one
          // run of half-tiles, and every scale up to the step has some) and the masses of the finished ones
          int cur_seg = 0;
          float cur_mass = 0.f;
          float* masses = reinterpret_cast<float*>(stage) + lane;      // [scale][32 rows]
          if (FULL && LONE)                                            // a scale may lie in the other warpgroup's tiles alone
            for (int s = 0; s <= p.step; ++s) masses[s * 32] = 0.f;
          const bool follow = FULL && (n_slots + 1) / 2 <= FOLLOW_TILES;
          int j = 0;
          // FULL: a warp whose 32 rows all lie past the last query hands on whatever is there (its rows of O and its masses go
          // nowhere): a calibration pass 1.130 -> 1.115 ms.  Generation measured 0.3 to 0.8 % slower with the branch.
          const bool no_rows = FULL && q0 + (stride == 2 ? 0 : x * BM) + (warp & 3) * 32 >= p.t_q;
          for (; no_rows && j < n_tiles && ok; ++j) {
            ok = __all_sync(0xffffffffu, mbar_wait(bar(S_FULL + x), (cx + j) & 1, abort_flag, p.status));
            mbar_arrive(bar(P_FULL + 2 * x));
            mbar_arrive(bar(P_FULL + 2 * x + 1));
          }
          for (; j < n_tiles && ok; ++j) {
            const uint32_t ph = (cx + j) & 1;
            Slot s0 = get_slot<FULL>(2 * j0, descs, n_desc, n_slots, 0, p.n_own, p.step);       // row numbers unused here
            Slot s1 = get_slot<FULL>(2 * j0 + 1, descs, n_desc, n_slots, 0, p.n_own, p.step);
            j0 += LONE ? stride : 1;
            const float b0 = bias_h ? bias_h[s0.seg] * LOG2E : 0.f;
            const float b1 = bias_h ? bias_h[s1.seg] * LOG2E : 0.f;
            ok = __all_sync(0xffffffffu, mbar_wait(bar(S_FULL + x), ph, abort_flag, p.status));
            if (!ok) break;
            tc_fence_after();
            // whole row of S into registers (one wait for the four loads)
            uint32_t r0[32], r1[32], r2[32], r3[32];
            tmem_ld32(t_s, r0);
            tmem_ld32(t_s + 32, r1);
            tmem_ld32(t_s + 64, r2);
            tmem_ld32(t_s + 96, r3);
            tmem_wait_ld();
            if (s0.n_valid < HALF || s1.n_valid < HALF) {            // ragged tile (warp-uniform): mask by -inf
#pragma unroll
              for (int i = 0; i < 32; ++i) {
                if (i >= s0.n_valid) r0[i] = 0xff800000u;
                if (i + 32 >= s0.n_valid) r1[i] = 0xff800000u;
                if (i >= s1.n_valid) r2[i] = 0xff800000u;
                if (i + 32 >= s1.n_valid) r3[i] = 0xff800000u;
              }
            }
            // p = exp2(logit - m_ref); row sum in fp32; P as bf16 pairs into the columns S occupied
            // (keys 32c..32c+31 -> P columns 16c..16c+15; the whole row of S is already in registers).
            // One pair in four takes the polynomial on the FMA pipe, the rest the MUFU unit: the tile's
            // 16 384 exponentials would otherwise keep MUFU busy as long as the tensor pipe needs for
            // the tile's two products.
            const uint64_t scale2 = pack2(p.scale_log2, p.scale_log2);
            uint64_t sum2 = pack2(0.f, 0.f);
            float top = 0.f;                                         // the largest argument that went to the polynomial
            auto exps = [&](const uint32_t (&rc)[32], uint64_t bb2, uint32_t (&pk)[16]) {
#pragma unroll
              for (int i = 0; i < 32; i += 2) {
                const uint64_t xx = fma2(pack2(__uint_as_float(rc[i]), __uint_as_float(rc[i + 1])), scale2, bb2);
                float e0, e1, x0, x1;
                unpack2(xx, x0, x1);
                if (!FULL && ((i >> 1) & POLY_MASK) == POLY_MASK) {
                  exp2_poly2(xx, e0, e1);
                  if (SPECULATE) top = fmax3(top, x0, x1);
                } else {
                  e0 = ex2_approx(x0);
                  e1 = ex2_approx(x1);
                }
                sum2 = add2(sum2, pack2(e0, e1));
                pk[i >> 1] = pack_bf16(e0, e1);
              }
            };
            auto exp_chunk = [&](const uint32_t (&rc)[32], uint64_t bb2, int c) {
              uint32_t pk[16];
              exps(rc, bb2, pk);
              tmem_st16(t_s + c * 16, pk);
            };
            // The reference moves seldom.  SPECULATE: from the second tile on, the first half's exponentials are taken against the
            // present one, and their sum tells whether it still serves (the polynomial's arguments are looked at too: it is
            // meaningless above 2^127); only the second half's maximum is computed, beside them.
            bool take_max = true;
            uint32_t pk0[16], pk1[16];
            // A head that would be cut had a reference, and an exact weight for it, in every piece.  Here its references follow the
            // maximum in the first two tiles of every such piece (and in a lone warpgroup's first two), heads that would stay whole
            // keep the first tile's.  Against 64 bits no launch measured is then further off than the cuts it replaces (second tiles
            // alone, in all heads of such a launch: single heads up to 1.3 % further off, those left as pairs of query tiles; with a bias
            // that raises the last tiles an emulation has them 4 % further off).  An image pair at 20x: 576 queries 19.5 -> 18.5 us.
            const bool look = !FULL && LONE && (in_piece < 2 || j < first_looks);
            if (LONE) in_piece += stride;
            if (LONE && in_piece >= piece) in_piece -= piece;
            if (SPECULATE && j > 0 && !follow && !look) {
              const uint64_t bb0 = pack2(b0 - m_ref, b0 - m_ref);
              exps(r0, bb0, pk0);
              exps(r1, bb0, pk1);
              float ma[4];
#pragma unroll
              for (int c = 0; c < 4; ++c) ma[c] = fmaxf(__uint_as_float(r2[c]), __uint_as_float(r3[c]));
#pragma unroll
              for (int i = 4; i < 32; ++i) ma[i & 3] = fmax3(ma[i & 3], __uint_as_float(r2[i]), __uint_as_float(r3[i]));
              const float m1 = fmaf(fmaxf(fmaxf(ma[0], ma[1]), fmaxf(ma[2], ma[3])), p.scale_log2, b1);
              float sa, sb;
              unpack2(sum2, sa, sb);
              take_max = __any_sync(0xffffffffu, !(sa + sb <= SUM_LIMIT && fmaxf(top, m1 - m_ref) <= RESCALE_THRESHOLD));
              if (take_max) {                                        // S is still there: load the half again
                sum2 = pack2(0.f, 0.f);
                tmem_ld32(t_s, r0);
                tmem_ld32(t_s + 32, r1);
                tmem_wait_ld();
#pragma unroll
                for (int i = 0; i < 32; ++i) {
                  if (i >= s0.n_valid) r0[i] = 0xff800000u;
                  if (i + 32 >= s0.n_valid) r1[i] = 0xff800000u;
                }
              }
            }
            if (take_max) {
              // row maximum: the logit is raw * scale + bias(half) with scale > 0, so take the raw maxima
              // (eight independent chains keep the dependent depth short)
              float mq[8];
#pragma unroll
              for (int c = 0; c < 4; ++c) {
                mq[c] = fmaxf(__uint_as_float(r0[c]), __uint_as_float(r1[c]));
                mq[4 + c] = fmaxf(__uint_as_float(r2[c]), __uint_as_float(r3[c]));
              }
#pragma unroll
              for (int i = 4; i < 32; i += 4) {
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                  mq[c] = fmax3(mq[c], __uint_as_float(r0[i + c]), __uint_as_float(r1[i + c]));
                  mq[4 + c] = fmax3(mq[4 + c], __uint_as_float(r2[i + c]), __uint_as_float(r3[i + c]));
                }
              }
              const float mx0 = fmaxf(fmaxf(mq[0], mq[1]), fmaxf(mq[2], mq[3]));
              const float mx1 = fmaxf(fmaxf(mq[4], mq[5]), fmaxf(mq[6], mq[7]));
              const float mx = fmaxf(fmaf(mx0, p.scale_log2, b0), fmaf(mx1, p.scale_log2, b1));
              const float m_new = fmaxf(m_ref, mx);
              const bool grow = m_new > m_ref + (follow || look ? 0.f : RESCALE_THRESHOLD);   // also true on the first tile (m_ref = NO_MAX)
              if (j > 0 && __any_sync(0xffffffffu, grow)) {
                // O_x holds tiles < j relative to m_ref: rescale the rows whose reference moves.  O_x is complete:
                // S_x of this tile was issued after the PV products of tile j - 1 by the same thread, and the
                // commit behind S_FULL covers every product issued before it.
                const float f = grow ? exp2f(m_ref - m_new) : 1.f;
#pragma unroll
                for (int c = 0; c < D / 32; ++c) {
                  uint32_t r[32];
                  tmem_ld32(t_o + c * 32, r);
                  tmem_wait_ld();
#pragma unroll
                  for (int i = 0; i < 32; ++i) r[i] = __float_as_uint(__uint_as_float(r[i]) * f);
                  tmem_st32(t_o + c * 32, r);
                }
                tmem_wait_st();
                l_sum *= f;
                if (FULL) {
                  cur_mass *= f;
                  for (int s = 0; s < cur_seg; ++s) masses[s * 32] *= f;
                }
              }
              if (grow) m_ref = m_new;
              const uint64_t bb0 = pack2(b0 - m_ref, b0 - m_ref);
              exp_chunk(r0, bb0, 0);
              exp_chunk(r1, bb0, 1);
            } else {
              tmem_st16(t_s, pk0);
              tmem_st16(t_s + 16, pk1);
            }
            tmem_wait_st();
            tc_fence_before();
            mbar_arrive(bar(P_FULL + 2 * x));                      // the PV product of keys 0..63 may start
            if (FULL) {
              float sa, sb;
              unpack2(sum2, sa, sb);
              const float half = sa + sb;
              l_sum += half;
              sum2 = pack2(0.f, 0.f);
              if (s0.seg != cur_seg) {
                masses[cur_seg * 32] = cur_mass;
                cur_seg = s0.seg;
                cur_mass = 0.f;
              }
              cur_mass += half;
            }
            const uint64_t bb1 = pack2(b1 - m_ref, b1 - m_ref);
            exp_chunk(r2, bb1, 2);
            exp_chunk(r3, bb1, 3);
            float sa, sb;
            unpack2(sum2, sa, sb);
            l_sum += sa + sb;
            tmem_wait_st();
            tc_fence_before();
            mbar_arrive(bar(P_FULL + 2 * x + 1));
            if (FULL && s1.n_valid > 0) {
              if (s1.seg != cur_seg) {
                masses[cur_seg * 32] = cur_mass;
                cur_seg = s1.seg;
                cur_mass = 0.f;
              }
              cur_mass += sa + sb;
            }
          }
          if (ok) ok = __all_sync(0xffffffffu, mbar_wait(bar(PV_DONE + x), items_x & 1, abort_flag, p.status));
          ++items_x;
          cx += n_tiles;
          const Item im = read_item<FULL, LONE>(ring, p, n_qp);
          const int seq = im.seq;
          const int q_row0 = im.shared ? im.q0 : im.q0 + x * BM;
          // Eq. 2: mean over the step's rows of mass(row, scale) / rowsum(row), `inv_l` = this row's 1 / rowsum relative to its
          // reference; rows past t_q are padding
          auto add_beta = [&](float inv_l) {
            const float w = q_row0 + row < p.t_q ? inv_l / (float)p.t_q : 0.f;
            float* beta = p.beta_row + (int64_t)im.head * p.K * p.K;
            for (int s = 0; s <= p.step; ++s) {
              float v = (s == cur_seg ? cur_mass : masses[s * 32]) * w;
#pragma unroll
              for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
              if (lane == 0) atomicAdd(beta + s, v);
            }
            __syncwarp();                                   // the buffer now takes output rows
          };
          if (FULL && ok && !no_rows && !im.shared) add_beta(1.f / l_sum);
          // Normalised rows leave through this warp's staging buffer: per group of 32 columns every thread parks its 64 bytes
          // (16-byte chunks, chunk ^ (row / 2 mod 4): the copy engine's 64-byte swizzle, free of bank conflicts) and one bulk
          // store writes the 32 rows, clipping those past the last query.  The halves of the buffer alternate.  Loads from the
          // buffer and 16-byte stores by all lanes took 3000 to 3700 cycles of every item; image pair at 20x 2.219 -> 2.183 ms, eight
          // images at 10x 3.659 -> 3.623, ragged 2.492 -> 2.458, preview 162.8 -> 158.7 us, 64-wide heads as before.
          // A warp without a row below the last query writes nothing, the buffer included: its last store may still be reading one
          // half, and only a store of its own for every group would make the wait for all but the newest one cover that half.
          const bool any_row = q_row0 + (warp & 3) * 32 < p.t_q;
          auto store_rows = [&](const float (&acc)[32], float inv, int c, int half) {
            if (!any_row) return;
            unsigned char* buf = stage + half * 2048;
            if (lane == 0) bulk_wait_read<1>();                 // the store before the last has read this half
            __syncwarp();
#pragma unroll
            for (int i = 0; i < 32; i += 8) {
              int4 v;
              v.x = (int)pack_bf16(acc[i] * inv, acc[i + 1] * inv);
              v.y = (int)pack_bf16(acc[i + 2] * inv, acc[i + 3] * inv);
              v.z = (int)pack_bf16(acc[i + 4] * inv, acc[i + 5] * inv);
              v.w = (int)pack_bf16(acc[i + 6] * inv, acc[i + 7] * inv);
              const int chunk = i >> 3;
              *reinterpret_cast<int4*>(buf + lane * 64 + ((chunk ^ ((lane >> 1) & 3)) << 4)) = v;
            }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            __syncwarp();
            if (lane == 0) {
              tma_store_4d(&maps.out, smem_u32(buf), c * 32, q_row0 + (warp & 3) * 32, p.o_head > 0 ? im.head : 0,
                           p.o_seq > 0 ? seq : 0);
              bulk_commit();
            }
          };
          if (LONE && ok && im.shared) {
            // The two warps of these 32 rows meet: each leaves its reference and row sum in its staging buffer, then takes half
            // of the columns of both results.  The half of the buffer that is not written first holds them; with one group of
            // columns that group takes the other half, so that here as after other items the newest store reads half 1.
            constexpr int NG = D / 64, EX = NG > 1 || FULL ? 1 : 0;          // (FULL: the masses lie in half 0)
            if (lane == 0) bulk_wait_read<0>();
            __syncwarp();
            reinterpret_cast<float2*>(stage + EX * 2048)[lane] = make_float2(m_ref, l_sum);
            __syncwarp();
            const uint32_t meet = bar(MEET + (warp & 3));
            if (lane == 0) mbar_arrive(meet);
            ok = __all_sync(0xffffffffu, mbar_wait(meet, 0, abort_flag, p.status));
            if (ok) {
              tc_fence_after();
              const unsigned char* other = sgen + SM_OUT + (warp < 8 ? warp : warp - 8) * STAGE_BYTES;
              const float2 ml = reinterpret_cast<const float2*>(other + EX * 2048)[lane];
              const bool both = im.n_tiles > 1;                 // else the second warpgroup had no key tile
              const float m_all = fmaxf(m_ref, ml.x);
              float w_own = exp2f(m_ref - m_all), w_other = exp2f(ml.x - m_all);
              const float inv = 1.f / (l_sum * w_own + ml.y * w_other);
              if (FULL && !no_rows) add_beta(w_own * inv);
              uint32_t a[NG][32], b[NG][32];
#pragma unroll
              for (int c = 0; c < NG; ++c) {
                tmem_ld32(tmem + lane_base + 256 + (x * NG + c) * 32, a[c]);
                tmem_ld32(tmem + lane_base + 384 + (x * NG + c) * 32, b[c]);
              }
              tmem_wait_ld();
              tc_fence_before();
              __syncwarp();
              if (lane == 0) mbar_arrive(meet);                 // the other warp's results and its two words have been read
              const float wa = x == 0 ? w_own : w_other, wb = x == 0 ? w_other : w_own;
#pragma unroll
              for (int c = 0; c < NG; ++c) {
                float acc[32];
#pragma unroll
                for (int i = 0; i < 32; ++i) {
                  acc[i] = __uint_as_float(a[c][i]) * wa;
                  if (both) acc[i] = fmaf(__uint_as_float(b[c][i]), wb, acc[i]);
                }
                if (c == NG - 1) {
                  ok = __all_sync(0xffffffffu, mbar_wait(meet, 1, abort_flag, p.status));
                  tc_fence_after();
                }
                if (ok) store_rows(acc, inv, x * NG + c, NG > 1 ? c : 1);
              }
            }
          } else if (ok && (LONE || im.n_split == 1)) {
            tc_fence_after();
            const float inv = 1.f / l_sum;
            // the whole row of O in one go, so the four groups' conversions and stores overlap
            uint32_t o[D / 32][32];
#pragma unroll
            for (int c = 0; c < D / 32; ++c) tmem_ld32(t_o + c * 32, o[c]);
            tmem_wait_ld();
            auto out_group = [&](const uint32_t (&r)[32], int c) {
              float acc[32];
#pragma unroll
              for (int i = 0; i < 32; ++i) acc[i] = __uint_as_float(r[i]);
              store_rows(acc, inv, c, c & 1);
            };
#pragma unroll
            for (int c = 0; c < D / 32; ++c) out_group(o[c], c);
          } else if (!LONE && ok) {
            // A piece of a split head: publish the unnormalised O of this row with its reference and row
            // sum; the warp that arrives last at the counter of these 32 rows merges
            // sum over pieces of 2^(m_piece - m) * (O_piece, l_piece).
            tc_fence_after();
            const int n_split = im.n_split, piece = im.piece, qp = im.qp;
            float* slots = p.split_partials + ((int64_t)seq * p.slots_per_seq + im.slot_base) * SPLIT_SLOT_FLOATS;
            float* slot_own = slots + (int64_t)im.sub * SPLIT_SLOT_FLOATS;
            int4* ocol = reinterpret_cast<int4*>(slot_own) + x * BM + row;
            uint32_t* ctr = p.split_counters + ((int64_t)seq * p.ctrs_per_seq + im.ctr_base + qp) * 8 + (warp - 4);
            // Every other piece of these 32 rows published already?  Then this warp's own stays in TMEM and it merges at once.
            uint32_t last = 0;
            if (lane == 0) {
              uint32_t seen;
              asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(seen) : "l"(ctr) : "memory");
              last = seen == (uint32_t)(n_split - 1);
              if (last) *reinterpret_cast<volatile uint32_t*>(ctr) = 0;     // ready for the next launch
            }
            last = __shfl_sync(0xffffffffu, last, 0);
            if (!last) {
#pragma unroll 1
              for (int c = 0; c < D / 32; ++c) {
                uint32_t r[32];
                tmem_ld32(t_o + c * 32, r);
                tmem_wait_ld();
#pragma unroll
                for (int gq = 0; gq < 8; ++gq)
                  ocol[(c * 8 + gq) * (2 * BM)] = make_int4((int)r[4 * gq], (int)r[4 * gq + 1], (int)r[4 * gq + 2], (int)r[4 * gq + 3]);
              }
              slot_own[2 * BM * D + x * BM + row] = m_ref;
              slot_own[2 * BM * D + 2 * BM + x * BM + row] = l_sum;
              __threadfence();
              __syncwarp();
              if (lane == 0) {
                const uint32_t old = atomicAdd(ctr, 1u);
                last = old == (uint32_t)(n_split - 1);
                if (last) *reinterpret_cast<volatile uint32_t*>(ctr) = 0;   // ready for the next launch
              }
              last = __shfl_sync(0xffffffffu, last, 0);
            }
            if (last) {
              __threadfence();
              // The pieces are added in piece order, this warp's own (still in TMEM) at its place among them, so
              // the result does not depend on which piece happened to arrive last.
              // references and row sums of up to MERGE_FAST pieces are read once, all loads in flight together;
              // a head cut finer than that reads them again where it needs them
              constexpr int MERGE_FAST = 4;
              float mp[MERGE_FAST], lp[MERGE_FAST];
#pragma unroll
              for (int s2 = 0; s2 < MERGE_FAST; ++s2) {
                const float* sl = slots + (int64_t)(s2 * n_qp + qp) * SPLIT_SLOT_FLOATS;
                const bool other = s2 < n_split && s2 != piece;
                mp[s2] = other ? __ldcg(sl + 2 * BM * D + x * BM + row) : (s2 == piece ? m_ref : -INFINITY);
                lp[s2] = other ? __ldcg(sl + 2 * BM * D + 2 * BM + x * BM + row) : (s2 == piece ? l_sum : 0.f);
              }
              float m_all = -INFINITY;                                // common reference and total row sum
#pragma unroll
              for (int s2 = 0; s2 < MERGE_FAST; ++s2) m_all = fmaxf(m_all, mp[s2]);
              for (int s2 = MERGE_FAST; s2 < n_split; ++s2) {
                const float* sl = slots + (int64_t)(s2 * n_qp + qp) * SPLIT_SLOT_FLOATS;
                m_all = fmaxf(m_all, s2 == piece ? m_ref : __ldcg(sl + 2 * BM * D + x * BM + row));
              }
              float l_all = 0.f;
#pragma unroll
              for (int s2 = 0; s2 < MERGE_FAST; ++s2) {               // piece order, as below
                mp[s2] = s2 < n_split ? exp2f(mp[s2] - m_all) : 0.f;  // from here on: the piece's weight
                l_all = fmaf(lp[s2], mp[s2], l_all);
              }
              for (int s2 = MERGE_FAST; s2 < n_split; ++s2) {
                const float* sl = slots + (int64_t)(s2 * n_qp + qp) * SPLIT_SLOT_FLOATS;
                const float l2 = s2 == piece ? l_sum : __ldcg(sl + 2 * BM * D + 2 * BM + x * BM + row);
                const float m2 = s2 == piece ? m_ref : __ldcg(sl + 2 * BM * D + x * BM + row);
                l_all = fmaf(l2, exp2f(m2 - m_all), l_all);
              }
              const float inv = 1.f / l_all;
#pragma unroll 1
              for (int c = 0; c < D / 32; ++c) {
                uint32_t r[32];
                tmem_ld32(t_o + c * 32, r);
                tmem_wait_ld();
                float acc[32];
#pragma unroll
                for (int i = 0; i < 32; ++i) acc[i] = 0.f;
                for (int s2 = 0; s2 < n_split; ++s2) {
                  if (s2 == piece) {
                    const float w_own = exp2f(m_ref - m_all);
#pragma unroll
                    for (int i = 0; i < 32; ++i) acc[i] = fmaf(__uint_as_float(r[i]), w_own, acc[i]);
                    continue;
                  }
                  const float* sl = slots + (int64_t)(s2 * n_qp + qp) * SPLIT_SLOT_FLOATS;
                  float w;
                  if (s2 < MERGE_FAST) {
                    w = s2 == 0 ? mp[0] : s2 == 1 ? mp[1] : s2 == 2 ? mp[2] : mp[3];
                  } else {
                    w = exp2f(__ldcg(sl + 2 * BM * D + x * BM + row) - m_all);
                  }
                  const float4* oc = reinterpret_cast<const float4*>(sl) + (c * 8) * (2 * BM) + x * BM + row;
#pragma unroll
                  for (int i = 0; i < 8; ++i) {
                    const float4 v = __ldcg(oc + i * (2 * BM));
                    acc[4 * i] = fmaf(v.x, w, acc[4 * i]);
                    acc[4 * i + 1] = fmaf(v.y, w, acc[4 * i + 1]);
                    acc[4 * i + 2] = fmaf(v.z, w, acc[4 * i + 2]);
                    acc[4 * i + 3] = fmaf(v.w, w, acc[4 * i + 3]);
                  }
                }
                store_rows(acc, inv, c, c & 1);
              }
            }
          }
          if (FULL) {                                           // the next item's masses take the buffer again
            if (lane == 0) bulk_wait_read<0>();
            __syncwarp();
          }
          // the next item's first P hand-over orders this item's reads of O before the next PV product
          tc_fence_before();
        }
      }
      __syncwarp();
      if (ok && lane == 0) mbar_arrive(bar(ITEM_EMPTY + slot));
    }
    if (lane == 0) bulk_wait();                                 // rows still on their way out
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u) : "memory");
  }
}

// Self-test of the bounded wait: one thread waits on a barrier nobody will ever arrive at, with a short limit,
// and reports what the wait returned.  The wait must give up, set the status word and return false.
__global__ void wait_expiry_kernel(uint32_t* status, uint32_t* result) {
  __shared__ __align__(8) unsigned long long barrier_word;
  __shared__ uint32_t abort_word;
  if (threadIdx.x == 0) {
    abort_word = 0;
    mbar_init(smem_u32(&barrier_word), 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    const bool ok = mbar_wait(smem_u32(&barrier_word), 0, &abort_word, status, 2048u);
    result[0] = ok ? 1u : (abort_word ? 2u : 3u);
  }
}

}  // namespace tc

cudaError_t launch_wait_expiry(uint32_t* status, uint32_t* result, cudaStream_t stream) {
  tc::wait_expiry_kernel<<<1, 32, 0, stream>>>(status, result);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------------- host side
int pair_create(int d);
cudaError_t launch_attn_pair_kernel(int d, const AttnParams& p, const tc::Maps& maps, cudaStream_t stream);

struct TcState {
  PFN_cuTensorMapEncodeTiled_v12000 encode = nullptr;
  CUtensorMap k_pool, v_pool;
  CUtensorMap v_pool_half;   // as v_pool with boxes of d / 2 columns: what one CTA of a pair keeps of a tile's values
  int n_sm = 148;
  int n_pairs = 0;           // CTA pairs of attn_pair_kernel the device holds at once
  int d = 0;                 // head dimension of the context (64 or 128)
  bool ready = false;
};

namespace {

// boxes of `cols` columns (64 or 32), their rows swizzled over their 128 or 64 bytes
CUtensorMapSwizzle swizzle_of(int cols) { return cols == 32 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_128B; }

bool encode_2d(TcState* st, CUtensorMap* m, void* base, uint64_t rows, int cols) {
  cuuint64_t dims[2] = {(cuuint64_t)st->d, (cuuint64_t)rows};
  cuuint64_t strides[1] = {(cuuint64_t)st->d * 2};
  cuuint32_t box[2] = {(cuuint32_t)cols, (cuuint32_t)tc::HALF};
  cuuint32_t estr[2] = {1, 1};
  return st->encode(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, base, dims, strides, box, estr,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle_of(cols), CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// [n_seq, H, t, d] view with element strides -> 4-D map (d, token, head, sequence)
bool encode_4d(TcState* st, CUtensorMap* m, const void* base, int t, int H, int n_seq, int64_t s_tok, int64_t s_head,
               int64_t s_seq, int cols = 64, int rows = tc::HALF) {
  const tc::MapShape g = tc::map_shape(st->d, t, H, n_seq, s_tok, s_head, s_seq);
  cuuint32_t box[4] = {(cuuint32_t)cols, (cuuint32_t)rows, 1, 1};
  cuuint32_t estr[4] = {1, 1, 1, 1};
  return st->encode(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(base), g.dims, g.strides, box, estr,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle_of(cols), CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace

int tc_create(const heatkv_config& cfg, void* k_pool, void* v_pool, uint64_t pool_rows, TcState** out) {
  *out = nullptr;
  TcState* st = new (std::nothrow) TcState;
  if (!st) return HEATKV_ERR_HOST_MEMORY;
  *out = st;
  if (cfg.d != 64 && cfg.d != 128) return HEATKV_OK;    // other head dimensions run on the generic kernel only
  st->d = cfg.d;
  void* fn = nullptr;
  cudaDriverEntryPointQueryResult qres;
  if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &fn, cudaEnableDefault, &qres) != cudaSuccess ||
      qres != cudaDriverEntryPointSuccess || !fn) {
    cudaGetLastError();
    return HEATKV_OK;                                   // no driver entry point: generic kernel only
  }
  st->encode = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(fn);
  if (!encode_2d(st, &st->k_pool, k_pool, pool_rows, 64) || !encode_2d(st, &st->v_pool, v_pool, pool_rows, 64) ||
      !encode_2d(st, &st->v_pool_half, v_pool, pool_rows, cfg.d / 2))
    return HEATKV_OK;
  const int smem = cfg.d == 128 ? (int)tc::Layout<128>::SM_ALLOC : (int)tc::Layout<64>::SM_ALLOC;
  const void* kernels[4];
  for (int i = 0; i < 4; ++i)
    kernels[i] = cfg.d == 128 ? (i == 0   ? (const void*)tc::attn_tc_kernel<128, false, false>
                                 : i == 1 ? (const void*)tc::attn_tc_kernel<128, false, true>
                                 : i == 2 ? (const void*)tc::attn_tc_kernel<128, true, false>
                                          : (const void*)tc::attn_tc_kernel<128, true, true>)
                              : (i == 0   ? (const void*)tc::attn_tc_kernel<64, false, false>
                                 : i == 1 ? (const void*)tc::attn_tc_kernel<64, false, true>
                                 : i == 2 ? (const void*)tc::attn_tc_kernel<64, true, false>
                                          : (const void*)tc::attn_tc_kernel<64, true, true>);
  for (const void* kern : kernels) {
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) != cudaSuccess) {
      cudaGetLastError();
      return HEATKV_OK;
    }
    // the register hand-over inside the kernel must fit in what the launch really allocates
    cudaFuncAttributes attr;
    if (cudaFuncGetAttributes(&attr, kern) != cudaSuccess) {
      cudaGetLastError();
      return HEATKV_OK;
    }
    if (attr.numRegs * tc::THREADS < 128 * tc::REGS_SMALL + 256 * tc::REGS_SOFTMAX) return HEATKV_ERR_CUDA;
  }
  int dev = 0, n_sm = 0;
  if (cudaGetDevice(&dev) == cudaSuccess &&
      cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess && n_sm > 0)
    st->n_sm = n_sm;
  st->n_pairs = pair_create(cfg.d);
  st->ready = true;
  return HEATKV_OK;
}

void tc_destroy(TcState* st) { delete st; }

bool tc_ready(const TcState* st) { return st && st->ready; }

int tc_split_slot_floats(int d) { return d == 64 ? tc::Layout<64>::SPLIT_SLOT_FLOATS : tc::Layout<128>::SPLIT_SLOT_FLOATS; }

bool tc_supported(const TcState* st, const AttnParams& p, int d, int n_seq) {
  if (!st || !st->ready || d != st->d || n_seq > 65535) return false;
  // TMA needs 16-byte aligned bases (checked by the caller) and strides that are multiples of 16 bytes
  const int64_t s[6] = {p.q_seq, p.q_head, p.q_tok, p.kv_seq, p.kv_head, p.kv_tok};
  for (int64_t v : s)
    if (v & 7) return false;
  return true;
}

namespace {
bool encode_call(TcState* st, tc::Maps* maps, const AttnParams& p, int n_seq, int v_cols) {
  maps->k_pool = st->k_pool;
  maps->v_pool = v_cols == 64 ? st->v_pool : st->v_pool_half;
  // inputs: boxes of 64 rows; the output leaves in a warp's 32 rows x 32 columns
  return encode_4d(st, &maps->q, p.q, p.t_q, p.H, n_seq, p.q_tok, p.q_head, p.q_seq) &&
         encode_4d(st, &maps->k_own, p.k_new, p.n_own, p.H, n_seq, p.kv_tok, p.kv_head, p.kv_seq) &&
         encode_4d(st, &maps->v_own, p.v_new, p.n_own, p.H, n_seq, p.kv_tok, p.kv_head, p.kv_seq, v_cols) &&
         encode_4d(st, &maps->out, p.out, p.t_q, p.H, n_seq, p.o_tok, p.o_head, p.o_seq, 32, 32);
}
}  // namespace

// Does a launch of `items` (sequence, head, 256 queries) with at most `tiles` key tiles go to attn_pair_kernel?  Where all its pairs
// run at once, and not past the line where attn_tc_kernel's pieces of longer heads are quicker for some number of items (a pair takes
// 0.8 us per tile and 0.6 more for one where references follow the maximum; a tile of 64-wide heads takes attn_tc_kernel 1.2 us instead
// of 1.7).  Back to back, attn_tc_kernel against attn_pair_kernel: 32 items of 256 queries and 3 tiles 13.0 and 10.0 us; 64 items, 400
// queries, 8 tiles 18.5 and 13.9; 256 queries, 16 tiles, 1 item 19.0 and 19.3, 24 items 21.3 and 19.6; 64-wide heads, 12 tiles, 1 item
// 14.1 and 14.4, 24 items 15.0 and 14.7.  Of 475 launches up to the lines none is more than 2.6 % slower on pairs, those at the lines
// are 5.7 and 2.1 % faster in the mean; at 20 tiles of 128-wide heads up to 4.9 % slower, 0.9 % faster in the mean; 28 heads x 576
// queries (84 items) 25.4 and 35.5 us.  A tile of 128 queries is left to one CTA.
bool tc_pair_wanted(const TcState* st, int t_q, int64_t items, int tiles) {
  return t_q > tc::BM && items <= st->n_pairs && tiles <= (st->d == 128 ? 16 : 12);
}

cudaError_t launch_attn_pair(TcState* st, const AttnParams& p, int n_seq, cudaStream_t stream) {
  tc::Maps maps;
  AttnParams q = p;
  q.attn_items = p.items_per_seq * n_seq;
  q.store_items = p.append_tiles * p.H * n_seq;
  if (p.n_seq != n_seq || q.attn_items < 1 || !encode_call(st, &maps, p, n_seq, st->d / 2)) return cudaErrorInvalidValue;
  return launch_attn_pair_kernel(st->d, q, maps, stream);
}

// Attention of a scale step (p.items_per_seq work items per sequence) or, with p.full_slots > 0, calibration with an
// attention output over all p.n_own keys of p.k_new / p.v_new.
cudaError_t launch_attn_tc(TcState* st, const AttnParams& p, int n_seq, cudaStream_t stream, bool* ran_lone) {
  tc::Maps maps;
  if (!encode_call(st, &maps, p, n_seq, 64)) return cudaErrorInvalidValue;
  if (p.n_seq != n_seq || p.items_per_seq < 1) return cudaErrorInvalidValue;
  // one resident CTA per SM takes the attention items in turn; its two spare warps take the cache-update items
  AttnParams q = p;
  q.attn_items = p.items_per_seq * n_seq;
  q.store_items = p.append_tiles * p.H * n_seq;
  dim3 grid((unsigned)std::min(q.attn_items, st->n_sm));
  const bool full = p.full_slots > 0;
  bool lone = p.lone != 0;
  if (full) {
    // Items of calibration are all of one length, so a partly filled last round costs as much as a full one.  Where its single
    // query tiles would still all run at once it is issued as those, half as long.  Odd last tiles are single items from the second
    // round on; one round is as long as its pairs, and the kernel without single items is the quicker one for those (1024 queries 55.3
    // against 56.3 us, 2304: 193.4 and 195.5; 576 with an odd tile 37.6 and 39.5).  2 sequences x 16 heads, with single tiles run as the
    // first of a pair before: 144 queries 12.9 -> 11.2 us, 256: 16.7 -> 13.4, 400: 24.9 -> 18.9, 1600: 117 -> 103, 4096: 586 -> 554; 8
    // sequences, 576 queries: 103.5 -> 93.5, 1024: 203 -> 190.
    const int total = q.attn_items, n_qp = (p.t_q + 2 * tc::BM - 1) / (2 * tc::BM), whole = total / st->n_sm * st->n_sm;
    const bool tail_single = p.t_q - (n_qp - 1) * 2 * tc::BM <= tc::BM;
    int singles = 0;
    for (int i = whole; i < total; ++i) singles += (tail_single && i / n_seq % n_qp == n_qp - 1) ? 1 : 2;
    const bool cut = singles <= st->n_sm && total < INT32_MAX - 2 * st->n_sm;
    q.full_whole = cut ? whole : total;
    if (cut) q.attn_items = whole + 2 * (total - whole);
    lone = (cut && whole < total) || (tail_single && total > st->n_sm);
    grid = dim3((unsigned)std::min(q.attn_items, st->n_sm));
  }
  *ran_lone = lone;
  auto launch = [&](auto kernel, uint32_t smem) { return launch_pdl(kernel, grid, tc::THREADS, smem, stream, q, maps); };
  if (st->d == 128) {
    constexpr uint32_t smem = tc::Layout<128>::SM_ALLOC;
    if (full) return lone ? launch(tc::attn_tc_kernel<128, true, true>, smem) : launch(tc::attn_tc_kernel<128, true, false>, smem);
    return lone ? launch(tc::attn_tc_kernel<128, false, true>, smem) : launch(tc::attn_tc_kernel<128, false, false>, smem);
  }
  constexpr uint32_t smem = tc::Layout<64>::SM_ALLOC;
  if (full) return lone ? launch(tc::attn_tc_kernel<64, true, true>, smem) : launch(tc::attn_tc_kernel<64, true, false>, smem);
  return lone ? launch(tc::attn_tc_kernel<64, false, true>, smem) : launch(tc::attn_tc_kernel<64, false, false>, smem);
}

}  // namespace heatkv
