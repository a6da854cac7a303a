// Tensor-memory attention kernel for launches that cannot fill the GPU (head_dim 128 or 64): one pair of CTAs, on two SMs, per
// 256 queries of a (sequence, head), over the head's whole key range.
//
// attn_tc_kernel gives such a launch one SM per 256 queries, and a key tile there is a chain S, softmax, P, PV, next S of 2900
// cycles (1.85 us where a CTA has nothing else to overlap it with).  Here each CTA of a cluster of two holds 128 of the queries,
// the products are issued for both at once (cta_group::2, M = 256; a CTA keeps one half of K's rows and of V's columns, so every
// key is loaded once per pair) and the chain is cut: two softmax warpgroups take the key tiles in turn, S has two
// buffers, P columns of its own, and S of tile j + 2 is issued as soon as tile j has been read into registers.  About 1400 cycles
// per key tile.  Launches that do fill the GPU are better off with attn_tc_kernel: there two pairs of these take 12 % longer
// than one CTA with two query tiles (both softmax warpgroups are then busy throughout and share their sub-partition's issue slots).
// Warp roles:
//   warp 0      copies: the CTA's queries, its 64 keys of every tile and its D / 2 columns of the tile's values.  They complete on
//               barriers of CTA 0, where the issuers wait for both CTAs' at once.
//   warp 1      CTA 0: issues S = Q K^T for the pair.
//   warp 2      CTA 0: issues O += P V for the pair (an issuer of its own: with one for both, its waits alone took 2500 cycles per
//               tile).
//   warp 3 and warps 1 to 3 of CTA 1   cache update (only when the call carries it).
//   warps 4-7   softmax of even key tiles, warps 8-11 of odd ones, one thread per query row.  A row's reference is common to
//               both and handed from tile to tile through shared memory; the sums meet at the end, where the warpgroup of the
//               last tile writes the result.
// TMEM columns of either CTA: S 0..127 and 128..255 (even and odd tiles), O 256..383, P 384..447 and 448..511.
// Every wait is bounded, as in attn_tc_kernel.  (Cluster barriers are hardware waits that both CTAs always reach.)
#include <algorithm>

#include "attn_items.cuh"
#include "internal.h"

namespace heatkv {
namespace pair {

using namespace tc;

constexpr int THREADS = 384;
constexpr int STAGES = 4;               // of K and of V
// What ptxas assigns under __launch_bounds__(384, 1), for either head size; 44 bytes a thread spilled (11 stores, 36 loads), in all
// roles together.
constexpr int REGS_LAUNCH = 168;
constexpr int REGS_SMALL = 72, REGS_SOFTMAX = 216;
static_assert(128 * REGS_SMALL + 256 * REGS_SOFTMAX <= THREADS * REGS_LAUNCH, "register hand-over exceeds the CTA's allocation");
constexpr uint32_t OUT_BYTES = 4096;    // per softmax warp: two buffers of 32 rows x 64 B for the output rows
constexpr uint32_t T_O = 256, T_P = 384;

template <int D>
struct Layout {
  static_assert(D == 64 || D == 128, "head dimension");
  static constexpr int NCH = D / 64;                            // 64-column halves per row
  static constexpr uint32_t Q_BYTES = NCH * BM * 128;           // this CTA's 128 query rows
  static constexpr uint32_t K_BYTES = NCH * HALF * 128;         // its 64 keys of a tile
  static constexpr uint32_t V_BYTES = BN * D;                   // its D / 2 columns of the tile's 128 rows
  static constexpr uint32_t SM_Q = 0;
  static constexpr uint32_t SM_K = SM_Q + Q_BYTES;
  static constexpr uint32_t SM_V = SM_K + STAGES * K_BYTES;
  static constexpr uint32_t SM_OUT = SM_V + STAGES * V_BYTES;
  static constexpr uint32_t SM_SUM = SM_OUT + 8 * OUT_BYTES;    // float2[128 rows]: row sum and reference of the other warpgroup
  static constexpr uint32_t SM_REF = SM_SUM + BM * 8;           // float[128 rows]: the reference so far
  static constexpr uint32_t SM_BAR = SM_REF + BM * 4;           // barriers and scalars
  static constexpr uint32_t SM_ALLOC = SM_BAR + 512 + 1024;     // slack for manual alignment
  static_assert(SM_ALLOC <= 227 * 1024, "shared memory of one CTA");
};

enum Bar : uint32_t {
  Q_FULL = 0,                         // Q_FULL, K_FULL, V_FULL: in CTA 0, for the copies of both
  K_FULL = 1, K_EMPTY = 5, V_FULL = 9, V_EMPTY = 13,  // + stage
  S_FULL = 17, S_READ = 19,           // + tile & 1
  P_FULL = 21,                        // + 2 (tile & 1) + half
  P_EMPTY = 25,                       // + tile & 1   the tile's PV product is done
  REF = 27,                           // + 4 warpgroup + warp   the reference after a tile of that warpgroup is published
  SUMS = 35,                          // + warp
  DRAIN = 39,                         // + issuer   its last product is done
  N_BARS = 41
};
constexpr uint32_t BAR_TMEM_PTR = N_BARS * 8, BAR_ABORT = BAR_TMEM_PTR + 4;

// ---- what cluster launches add to the wrappers of tc_common.cuh
__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
// The address in CTA 0 of what has the address `addr` in this CTA.
__device__ __forceinline__ uint32_t in_cta0(uint32_t addr) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(r) : "r"(addr));
  return r;
}
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// A hand-over of tensor memory to an issuer in CTA 0, which waits with mbar_try_cluster.  Relaxed: tcgen05.fence on either side orders
// the tensor memory, nothing else is handed over.  (With release and acquire here and for CTA 1's copies, passed on by a warp of
// it, a preview pair took 161 us, with them for the copies alone 156; so 150.)
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t cluster_bar) {
  asm volatile("mbarrier.arrive.relaxed.cluster.shared::cluster.b64 _, [%0];" ::"r"(cluster_bar) : "memory");
}
// Copies into this CTA's shared memory that complete on a barrier of either CTA of the pair.
__device__ __forceinline__ void tma_load_2d_pair(uint32_t dst, const CUtensorMap* map, int c0, int c1, uint32_t cluster_bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
      ::"r"(dst), "l"(map), "r"(c0), "r"(c1), "r"(cluster_bar)
      : "memory");
}
__device__ __forceinline__ void tma_load_4d_pair(uint32_t dst, const CUtensorMap* map, int c0, int c1, int c2, int c3,
                                                 uint32_t cluster_bar) {
  asm volatile(
      "cp.async.bulk.tensor.4d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], [%6];"
      ::"r"(dst), "l"(map), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(cluster_bar)
      : "memory");
}
__device__ __forceinline__ bool mbar_test(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}
// Completion of every product this thread has issued, signalled at the same barrier of both CTAs.
__device__ __forceinline__ void tc_commit_pair(uint32_t lead, uint32_t bar) {
  asm volatile(
      "{\n\t.reg .pred q;\n\t.reg .b16 m;\n\tmov.b16 m, 3;\n\tsetp.ne.b32 q, %1, 0;\n\t"
      "@q tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], m;\n\t}"
      ::"r"(bar), "r"(lead)
      : "memory");
}
// Shared-memory matrix descriptors in two words: the lower holds the address, the upper the stride between groups of eight rows
// and the swizzle, of 128-byte rows (queries, keys, 64 value columns) or 64-byte rows (32 value columns).  Version 1.
__device__ __forceinline__ uint32_t desc_lo(uint32_t addr) { return (addr & 0x3ffffu) >> 4 | 1u << 16; }
constexpr uint32_t DESC_HI_128 = (1024 >> 4) | 1u << 14 | 2u << 29, DESC_HI_64 = (512 >> 4) | 1u << 14 | 4u << 29;
// D (+)= A B over the pair: M = 256, rows 0..127 and their operands in CTA 0, rows 128..255 in CTA 1; B split along N.
__device__ __forceinline__ void mma_ss_pair(uint32_t lead, uint32_t d_tmem, uint32_t a_lo, uint32_t b_lo, uint32_t hi, uint32_t idesc,
                                            uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t.reg .b64 a, b;\n\tmov.b64 a, {%1, %6};\n\tmov.b64 b, {%2, %6};\n\t"
      "setp.ne.b32 p, %4, 0;\n\tsetp.ne.b32 q, %5, 0;\n\t"
      "@q tcgen05.mma.cta_group::2.kind::f16 [%0], a, b, %3, p;\n\t}"
      ::"r"(d_tmem), "r"(a_lo), "r"(b_lo), "r"(idesc), "r"(acc), "r"(lead), "r"(hi)
      : "memory");
}
__device__ __forceinline__ void mma_ts_pair(uint32_t lead, uint32_t d_tmem, uint32_t a_tmem, uint32_t b_lo, uint32_t hi, uint32_t idesc,
                                            uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t.reg .b64 b;\n\tmov.b64 b, {%2, %6};\n\t"
      "setp.ne.b32 p, %4, 0;\n\tsetp.ne.b32 q, %5, 0;\n\t"
      "@q tcgen05.mma.cta_group::2.kind::f16 [%0], [%1], b, %3, p;\n\t}"
      ::"r"(d_tmem), "r"(a_tmem), "r"(b_lo), "r"(idesc), "r"(acc), "r"(lead), "r"(hi)
      : "memory");
}

template <int D>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(THREADS, 1)
attn_pair_kernel(const __grid_constant__ AttnParams p, const __grid_constant__ Maps maps) {
  using L = Layout<D>;
  constexpr int NCH = L::NCH;
  constexpr uint32_t SM_BAR = L::SM_BAR;
  extern __shared__ unsigned char smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t sbase = (raw + 1023u) & ~1023u;
  unsigned char* sgen = smem_raw + (sbase - raw);
  volatile uint32_t* abort_flag = reinterpret_cast<volatile uint32_t*>(sgen + SM_BAR + BAR_ABORT);
  auto bar = [&](uint32_t which) { return sbase + SM_BAR + which * 8; };

  const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
  const uint32_t rank = __shfl_sync(0xffffffffu, cluster_rank(), 0);

  pdl_trigger();
  // ---- what this pair works on: pairs of one head follow one another, sequences interleaved (plans may be read before pdl_wait)
  const int pair = blockIdx.x >> 1;
  const int n_qp = (p.t_q + 2 * BM - 1) / (2 * BM);
  const int seq = pair % p.n_seq, place = pair / p.n_seq / n_qp;          // place of the head in the plan's order
  const int q_row0 = (pair / p.n_seq % n_qp) * (2 * BM) + (int)rank * BM; // first query of this CTA
  int head, n_desc;
  const int2* descs;
  if (p.table_heads > 0) {                             // the host put the per-head table into the launch parameters
    head = p.table_head[place];
    n_desc = p.table_ndesc[place];
    descs = reinterpret_cast<const int2*>(p.seqs[seq].plan + p.table_desc_begin[place]);
  } else {
    const PlanView pv(p.seqs[seq].plan);
    const int u = (p.step * p.L + p.layer) * p.H;
    head = pv.order()[u + place];
    n_desc = pv.attn_cnt(p.runs)[u + head];
    descs = pv.attn_descs(p.runs) + pv.attn_begin(p.runs)[u + head];
  }
  const int n_slots = n_desc + (p.n_own + HALF - 1) / HALF, n_tiles = (n_slots + 1) >> 1;
  if (n_desc > 0) asm volatile("prefetch.global.L1 [%0];" ::"l"(descs));

  // One barrier a thread, while warp 0 asks for tensor memory.  (With one thread for all of them and the item looked up behind the
  // cluster barrier, a launch took 0.3 to 0.6 us more: 256 queries, 32 items 10.5, now 10.0 us.)
  if (threadIdx.x - 32u < N_BARS) {
    const uint32_t i = threadIdx.x - 32u;
    const bool warps = i >= S_READ && i < P_EMPTY;     // S_READ, P_FULL (used in CTA 0): a warpgroup's warps in both CTAs
    mbar_init(bar(i), warps ? 8 : 1);
    if (i == 0) *abort_flag = *reinterpret_cast<volatile uint32_t*>(p.status) != 0;   // an earlier CTA gave up: do not wait again
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 0) {
    __syncwarp();
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(sbase + SM_BAR + BAR_TMEM_PTR), "r"(512u)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync();                                      // the other CTA's barriers are there
  tc_fence_after();
  const uint32_t tmem = __shfl_sync(0xffffffffu, *reinterpret_cast<volatile uint32_t*>(sgen + SM_BAR + BAR_TMEM_PTR), 0);

  auto slot_of = [&](int i, int64_t base_row) { return get_slot<false>(i, descs, n_desc, n_slots, base_row, p.n_own, p.step); };

  auto warp_wait = [&](uint32_t b, uint32_t parity) { return tc::warp_wait(b, parity, abort_flag, p.status); };
  // for the issuers: both CTAs' softmax warps arrive there
  auto warp_wait_cluster = [&](uint32_t b, uint32_t parity) {
    return (bool)__all_sync(0xffffffffu, mbar_wait<Try::CLUSTER>(b, parity, abort_flag, p.status));
  };
  // for roles that have time: a suspended warp leaves its issue slots to the softmax
  auto warp_wait_idle = [&](uint32_t b, uint32_t parity) {
    return (bool)__all_sync(0xffffffffu, mbar_wait_hint(b, parity, abort_flag, p.status));
  };
  bool ok = true;
  if (warp < 4) {
    reg_dealloc<REGS_SMALL>();
    if (warp == 0) {
      // ------------------------------------------------------------------ copies
      const bool leader = elect_one();
      const int64_t base_row = p.seqs[seq].base_row;
      const int kv_head = head & p.kv_head_mask, kv_seq = seq & p.kv_seq_mask;
      auto landed = [&](uint32_t which, uint32_t bytes) {     // the barrier in CTA 0, which expects as much from CTA 1
        if (rank == 0) mbar_expect_tx(bar(which), 2 * bytes);
        return in_cta0(bar(which));
      };
      auto load_k = [&](int j) {                       // this CTA's 64 keys of tile j
        const uint32_t st = j % STAGES, use = j / STAGES;
        const Slot sl = slot_of(2 * j + (int)rank, base_row);
        if (j == 0) pdl_wait();                        // the first descriptors are read while the launch before may still run
        if (use > 0) ok = warp_wait_idle(bar(K_EMPTY + st), (use - 1) & 1);
        if (ok && leader) {
          const uint32_t full = landed(K_FULL + st, L::K_BYTES);
#pragma unroll
          for (int ch = 0; ch < NCH; ++ch) {
            const uint32_t dst = sbase + L::SM_K + st * L::K_BYTES + ch * (HALF * 128);
            if (sl.pool_row >= 0) tma_load_2d_pair(dst, &maps.k_pool, ch * 64, sl.pool_row, full);
            else tma_load_4d_pair(dst, &maps.k_own, ch * 64, -sl.pool_row - 1, kv_head, kv_seq, full);
          }
        }
        __syncwarp();
      };
      auto load_v = [&](int j) {                       // its D / 2 columns of the tile's values
        const uint32_t st = j % STAGES, use = j / STAGES;
        const Slot sl[2] = {slot_of(2 * j, base_row), slot_of(2 * j + 1, base_row)};
        if (use > 0) ok = warp_wait_idle(bar(V_EMPTY + st), (use - 1) & 1);
        if (ok && leader) {
          const uint32_t full = landed(V_FULL + st, L::V_BYTES);
          const int col = (int)rank * (D / 2);
#pragma unroll
          for (int hf = 0; hf < 2; ++hf) {
            const uint32_t dst = sbase + L::SM_V + st * L::V_BYTES + hf * (HALF * D);
            if (sl[hf].pool_row >= 0) tma_load_2d_pair(dst, &maps.v_pool, col, sl[hf].pool_row, full);
            else tma_load_4d_pair(dst, &maps.v_own, col, -sl[hf].pool_row - 1, kv_head, kv_seq, full);
          }
        }
        __syncwarp();
      };
      // What the first copies will fetch, sent for while the launch before may still run.  Where the update is a call of its own that
      // launch is a small one that ends first, and the requests only queue ahead of the copies (3 heads, 10 steps: 102.6 us a pass, with
      // them 104.5; as one call, 16 heads x 2 sequences, 7 steps, 4 layers: 146.8 us with them, 148.9 without).
      if (leader && p.carries_update) {
        const bool pool = !p.k8_pool;                    // (staging rows: the launch before is writing them)
        const Slot k0 = slot_of((int)rank, base_row);
        for (int ch = 0; ch < NCH; ++ch)
          if (k0.pool_row >= 0 && !pool) continue;
          else if (k0.pool_row >= 0) tma_prefetch_2d(&maps.k_pool, ch * 64, k0.pool_row);
          else tma_prefetch_4d(&maps.k_own, ch * 64, -k0.pool_row - 1, kv_head, kv_seq);
        for (int i = 0; i < 2 * NCH; ++i)
          tma_prefetch_4d(&maps.q, (i >> 1) * 64, q_row0 + (i & 1) * HALF, head & p.q_head_mask, seq & p.q_seq_mask);
        for (int hf = 0; hf < 2; ++hf) {
          const Slot v0 = slot_of(hf, base_row);
          if (v0.pool_row >= 0 && !pool) continue;
          else if (v0.pool_row >= 0) tma_prefetch_2d(&maps.v_pool, (int)rank * (D / 2), v0.pool_row);
          else tma_prefetch_4d(&maps.v_own, (int)rank * (D / 2), -v0.pool_row - 1, kv_head, kv_seq);
        }
      }
      __syncwarp();
      // keys run two tiles ahead of the values, as the products do
      int j = 0;
#pragma unroll 1
      for (; j < n_tiles + 2; ++j) {
        if (j < n_tiles) load_k(j);
        if (!ok) break;
        if (j == 0) {
          if (leader) {
            const uint32_t full = landed(Q_FULL, L::Q_BYTES);
            for (int i = 0; i < 2 * NCH; ++i)          // 64-column half i / 2, rows 64 (i & 1) ..
              tma_load_4d_pair(sbase + L::SM_Q + i * (HALF * 128), &maps.q, (i >> 1) * 64, q_row0 + (i & 1) * HALF,
                               head & p.q_head_mask, seq & p.q_seq_mask, full);
          }
          __syncwarp();
        }
        if (j >= 2) load_v(j - 2);
        if (!ok) break;
      }
      // The products read and signal both CTAs: neither leaves before the last of either issuer, complete run or not.  (Whoever
      // gave up has left its reason in the status word.)
#pragma unroll 1
      for (int i = 0; i < 2; ++i)
#pragma unroll 1
        for (uint32_t t = 0; t < WAIT_LIMIT && !mbar_try_hint(bar(DRAIN + i), 0); ++t) {}
      if (rank == 0 && (!ok || *abort_flag)) {
        // leaving early: let every copy of either CTA land before they exit (tiles 0 .. j of K and 0 .. j - 2 of V at most).  What
        // CTA 1 still lacks runs into the bound; an issuer that gives up over it sets this CTA's flag before its last commit.
        auto drain = [&](uint32_t first, int tiles) {
#pragma unroll 1
          for (int i = max(0, tiles - STAGES); i < tiles; ++i)
#pragma unroll 1
            for (uint32_t t = 0; t < WAIT_LIMIT / 16 && !mbar_try(bar(first + i % STAGES), (i / STAGES) & 1); ++t) {}
        };
        drain(K_FULL, min(j + 1, n_tiles));
        drain(V_FULL, min(max(j - 1, 0), n_tiles));
        drain(Q_FULL, 1);
      }
    } else if (warp < 3 && rank == 0) {
      // ------------------------------------------------------------------ MMA issuers (CTA 0, for the pair)
      const uint32_t lead = elect_one();
      pdl_wait();
      if (warp == 1) {
        constexpr uint32_t IDESC = instr_desc(2 * BM, BN, 0, 0);     // Q, K both K-major
        ok = warp_wait(bar(Q_FULL), 0);
        const uint32_t qa = desc_lo(sbase + L::SM_Q);
#pragma unroll 1
        for (int j = 0; j < n_tiles && ok; ++j) {
          const uint32_t b = j & 1, st = j % STAGES;
          if (j >= 2) ok = warp_wait_cluster(bar(S_READ + b), ((j >> 1) - 1) & 1);
          if (ok) ok = warp_wait(bar(K_FULL + st), (j / STAGES) & 1);
          if (!ok) break;
          tc_fence_after();
          const uint32_t ka = desc_lo(sbase + L::SM_K + st * L::K_BYTES);
#pragma unroll
          for (int ks = 0; ks < D / 16; ++ks)
            mma_ss_pair(lead, tmem + b * BN, qa + (((ks >> 2) * (BM * 128) + (ks & 3) * 32) >> 4),
                        ka + (((ks >> 2) * (HALF * 128) + (ks & 3) * 32) >> 4), DESC_HI_128, IDESC, ks > 0);
          tc_commit_pair(lead, bar(S_FULL + b));
          tc_commit_pair(lead && j + STAGES < n_tiles, bar(K_EMPTY + st));   // a stage nobody fills again has no one waiting
        }
      } else {
        constexpr uint32_t IDESC = instr_desc(2 * BM, D, 0, 1);      // P from TMEM, V MN-major
        constexpr uint32_t HI = D == 128 ? DESC_HI_128 : DESC_HI_64;
#pragma unroll 1
        for (int j = 0; j < n_tiles && ok; ++j) {
          const uint32_t b = j & 1, st = j % STAGES;
          ok = warp_wait(bar(V_FULL + st), (j / STAGES) & 1);
          const uint32_t va = desc_lo(sbase + L::SM_V + st * L::V_BYTES), pa = tmem + T_P + b * 64;
#pragma unroll
          for (int h = 0; h < 2; ++h) {                // keys 64 h .. 64 h + 63
            if (ok) ok = warp_wait_cluster(bar(P_FULL + 2 * b + h), (j >> 1) & 1);
            if (!ok) break;
            tc_fence_after();
#pragma unroll
            for (int ks = 4 * h; ks < 4 * h + 4; ++ks)
              mma_ts_pair(lead, tmem + T_O, pa + ks * 8, va + ks * (16 * D >> 4), HI, IDESC, ks > 0 || j > 0);
          }
          if (!ok) break;
          tc_commit_pair(lead, bar(P_EMPTY + b));
          tc_commit_pair(lead && j + STAGES < n_tiles, bar(V_EMPTY + st));
        }
      }
      tc_commit_pair(lead, bar(DRAIN + warp - 1));
    } else if (p.store_items > 0) {
      // ------------------------------------------------------------------ cache update (four warps of a pair)
      pdl_wait();
      store_rows_loop<D>(p, 2u * gridDim.x, lane);
    }
  } else {
    reg_alloc<REGS_SOFTMAX>();
    // ------------------------------------------------------------------ softmax: warpgroup w takes every second key tile
    const int w = (warp - 4) >> 2, wr = warp & 3;
    const int row = wr * 32 + lane;                     // row inside the CTA's query tile == TMEM lane
    const uint32_t lanes = tmem + ((uint32_t)(wr * 32) << 16);
    const uint32_t t_s = lanes + w * BN, t_p = lanes + T_P + w * 64, t_o = lanes + T_O;
    volatile float* ref_smem = reinterpret_cast<volatile float*>(sgen + L::SM_REF) + row;
    const float LOG2E = 1.4426950408889634f;
    const float* bias_h = p.seg_bias ? p.seg_bias + head * p.K : nullptr;
    // where the issuers are told (CTA 0)
    const uint32_t s_read = in_cta0(bar(S_READ + w)), p_full = in_cta0(bar(P_FULL + 2 * w));
    const bool no_rows = q_row0 + wr * 32 >= p.t_q;     // nothing below the last query: hand on whatever is there
    // The reference follows the maximum in the first two tiles and in every fourth, where the pieces of a cut head would start, if
    // attn_tc_kernel would cut any of the launch's heads: a row's largest weight rounds to bf16 without error where it is its reference,
    // and a cut head has a reference per piece.  Error of the output against 64 bits, of its norm, x 1e-3, cut / on pairs / on pairs
    // with the first tile's reference throughout: 48 heads x 256 queries, 7 tiles 2.298 / 2.287 / 2.326, 10 tiles
    // 2.290 / 2.287 / 2.329, 13 tiles 2.308 / 2.300 / 2.336; the same as times: 400 queries x 32 heads, 8 tiles 18.5 / 13.9 / 12.6 us.
    const bool follows = p.longest_piece >= 2 * SPLIT_MIN_PIECE - 1;
    float m_ref = NO_MAX, l_sum = 0.f;
    int j = w;
    pdl_wait();
#pragma unroll 1
    for (; no_rows && j < n_tiles && ok; j += 2) {
      const int n = j >> 1;
      ok = warp_wait(bar(S_FULL + w), n & 1);
      if (ok && n > 0) ok = warp_wait(bar(P_EMPTY + w), (n - 1) & 1);      // (the arrivals below are for this tile, not the last)
      if (ok && lane == 0) {
        mbar_arrive_cluster(s_read);
        mbar_arrive_cluster(p_full);
        mbar_arrive_cluster(p_full + 8);
      }
      __syncwarp();
    }
#pragma unroll 1
    for (; j < n_tiles && ok; j += 2) {
      const int n = j >> 1;
      const Slot s0 = slot_of(2 * j, 0), s1 = slot_of(2 * j + 1, 0);       // row numbers unused here
      const float b0 = bias_h ? bias_h[s0.seg] * LOG2E : 0.f;
      const float b1 = bias_h ? bias_h[s1.seg] * LOG2E : 0.f;
      ok = warp_wait(bar(S_FULL + w), n & 1);
      if (!ok) break;
      tc_fence_after();
      uint32_t r0[32], r1[32], r2[32], r3[32];
      tmem_ld32(t_s, r0);
      tmem_ld32(t_s + 32, r1);
      tmem_ld32(t_s + 64, r2);
      tmem_ld32(t_s + 96, r3);
      // looked at here, needed below: the answers come while the maxima and exponentials are computed
      const bool ref_there = j > 0 && mbar_test(bar(REF + 4 * (w ^ 1) + wr), ((j - 1) >> 1) & 1);
      float ref = NO_MAX;
      if (j > 0) ref = *ref_smem;
      const bool p_free = n > 0 && mbar_test(bar(P_EMPTY + w), (n - 1) & 1);
      tmem_wait_ld();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive_cluster(s_read);
      if (s0.n_valid < HALF || s1.n_valid < HALF) {            // ragged tile (warp-uniform): mask by -inf
#pragma unroll
        for (int i = 0; i < 32; ++i) {
          if (i >= s0.n_valid) r0[i] = 0xff800000u;
          if (i + 32 >= s0.n_valid) r1[i] = 0xff800000u;
          if (i >= s1.n_valid) r2[i] = 0xff800000u;
          if (i + 32 >= s1.n_valid) r3[i] = 0xff800000u;
        }
      }
      // row maximum: the logit is raw * scale + bias(half) with scale > 0, so raw maxima will do
      float mq[8];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        mq[i] = fmaxf(__uint_as_float(r0[i]), __uint_as_float(r1[i]));
        mq[4 + i] = fmaxf(__uint_as_float(r2[i]), __uint_as_float(r3[i]));
      }
#pragma unroll
      for (int i = 4; i < 32; ++i) {
        mq[i & 3] = fmax3(mq[i & 3], __uint_as_float(r0[i]), __uint_as_float(r1[i]));
        mq[4 + (i & 3)] = fmax3(mq[4 + (i & 3)], __uint_as_float(r2[i]), __uint_as_float(r3[i]));
      }
      const float mx0 = fmaxf(fmaxf(mq[0], mq[1]), fmaxf(mq[2], mq[3])), mx1 = fmaxf(fmaxf(mq[4], mq[5]), fmaxf(mq[6], mq[7]));
      const float mx = fmaxf(fmaf(mx0, p.scale_log2, b0), fmaf(mx1, p.scale_log2, b1));
      // the reference after the tile before this one, from the other warpgroup
      if (j > 0 && !__all_sync(0xffffffffu, ref_there)) {
        ok = warp_wait(bar(REF + 4 * (w ^ 1) + wr), ((j - 1) >> 1) & 1);
        if (!ok) break;
        ref = *ref_smem;
      }
      float m_new = fmaxf(ref, mx);
      const bool grow = m_new > ref + (follows && (j < 2 || (j & 3) == 0) ? 0.f : RESCALE_THRESHOLD);   // (true on the first tile: NO_MAX)
      if (!grow) m_new = ref;
      if (grow || j == 0) *ref_smem = m_new;
      __syncwarp();
      if (lane == 0) mbar_arrive(bar(REF + 4 * w + wr));
      if (__any_sync(0xffffffffu, m_new != m_ref)) {
        if (j > 0 && __any_sync(0xffffffffu, grow)) {
          // O holds the tiles before this one relative to ref: rescale the rows whose reference moves, once the last of their
          // products are done (none of a later tile is issued before P of this one is handed over).  The tile before that comes
          // first: only then is the other buffer's barrier at most one phase behind, and its parity means what it says.
          if (n > 0) ok = warp_wait(bar(P_EMPTY + w), (n - 1) & 1);
          if (ok) ok = warp_wait(bar(P_EMPTY + (w ^ 1)), ((j - 1) >> 1) & 1);
          if (!ok) break;
          tc_fence_after();
          const float f = grow ? exp2f(ref - m_new) : 1.f;
#pragma unroll
          for (int k = 0; k < D / 32; ++k) {
            uint32_t r[32];
            tmem_ld32(t_o + k * 32, r);
            tmem_wait_ld();
#pragma unroll
            for (int i = 0; i < 32; ++i) r[i] = __float_as_uint(__uint_as_float(r[i]) * f);
            tmem_st32(t_o + k * 32, r);
          }
          tmem_wait_st();
        }
        l_sum *= exp2f(m_ref - m_new);                         // (0 on the warpgroup's first tile)
        m_ref = m_new;
      }
      // p = exp2(logit - m_ref); row sum in fp32; P as bf16 pairs (keys 32k .. 32k+31 -> P columns 16k .. 16k+15).  One pair in
      // four takes the polynomial on the FMA pipe, as in attn_tc_kernel.
      const uint64_t scale2 = pack2(p.scale_log2, p.scale_log2);
      uint64_t sum2 = pack2(0.f, 0.f);
      auto exps = [&](const uint32_t (&rc)[32], uint64_t bb2, uint32_t (&pk)[16]) {
#pragma unroll
        for (int i = 0; i < 32; i += 2) {
          const uint64_t xx = fma2(pack2(__uint_as_float(rc[i]), __uint_as_float(rc[i + 1])), scale2, bb2);
          float e0, e1;
          if (((i >> 1) & POLY_MASK) == POLY_MASK) {
            exp2_poly2(xx, e0, e1);
          } else {
            float x0, x1;
            unpack2(xx, x0, x1);
            e0 = ex2_approx(x0);
            e1 = ex2_approx(x1);
          }
          sum2 = add2(sum2, pack2(e0, e1));
          pk[i >> 1] = pack_bf16(e0, e1);
        }
      };
      const uint64_t bb0 = pack2(b0 - m_ref, b0 - m_ref), bb1 = pack2(b1 - m_ref, b1 - m_ref);
      uint32_t pk0[16], pk1[16];
      exps(r0, bb0, pk0);
      exps(r1, bb0, pk1);
      if (n > 0 && !__all_sync(0xffffffffu, p_free)) {         // the product before has read P
        ok = warp_wait(bar(P_EMPTY + w), (n - 1) & 1);
        if (!ok) break;
      }
      tc_fence_after();
      tmem_st16(t_p, pk0);
      tmem_st16(t_p + 16, pk1);
      tmem_wait_st();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive_cluster(p_full);              // the PV product of keys 0..63 may start
      exps(r2, bb1, pk0);
      tmem_st16(t_p + 32, pk0);
      exps(r3, bb1, pk0);
      tmem_st16(t_p + 48, pk0);
      float sa, sb;
      unpack2(sum2, sa, sb);
      l_sum += sa + sb;
      tmem_wait_st();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive_cluster(p_full + 8);
    }
    // ---- the two warpgroups' row sums meet; the one with the last tile writes the result
    volatile float2* sums = reinterpret_cast<volatile float2*>(sgen + L::SM_SUM) + row;
    const bool writes = ((n_tiles - 1) & 1) == w;
    if (ok && !no_rows && !writes) {                           // (a warpgroup without a tile: 0 and NO_MAX)
      sums->x = l_sum;
      sums->y = m_ref;
      __syncwarp();
      if (lane == 0) mbar_arrive(bar(SUMS + wr));
    }
    // with rows or without: the product of this warpgroup's last tile signals its barrier in both CTAs
    if (ok && n_tiles > w) ok = warp_wait(bar(P_EMPTY + w), ((n_tiles - 1 - w) >> 1) & 1);
    if (ok && !no_rows && writes) {
      ok = warp_wait(bar(SUMS + wr), 0);
      if (ok) {
        tc_fence_after();
        l_sum = fmaf(sums->x, exp2f(sums->y - m_ref), l_sum);  // (references only rise, so this one is the higher)
        const float inv = 1.f / l_sum;
        unsigned char* stage = sgen + L::SM_OUT + (warp - 4) * OUT_BYTES;
        uint32_t o[D / 32][32];
#pragma unroll
        for (int c = 0; c < D / 32; ++c) tmem_ld32(t_o + c * 32, o[c]);
        tmem_wait_ld();
        // per group of 32 columns a bulk store of the warp's 32 rows (64-byte swizzle), clipped below the last query
#pragma unroll
        for (int c = 0; c < D / 32; ++c) {
          unsigned char* buf = stage + (c & 1) * 2048;
          if (c >= 2) {
            if (lane == 0) bulk_wait_read<1>();                // the store before the last has read this half
            __syncwarp();
          }
#pragma unroll
          for (int i = 0; i < 32; i += 8) {
            uint32_t v[4];
#pragma unroll
            for (int k = 0; k < 4; ++k)
              v[k] = pack_bf16(__uint_as_float(o[c][i + 2 * k]) * inv, __uint_as_float(o[c][i + 2 * k + 1]) * inv);
            *reinterpret_cast<int4*>(buf + lane * 64 + (((i >> 3) ^ ((lane >> 1) & 3)) << 4)) =
                make_int4((int)v[0], (int)v[1], (int)v[2], (int)v[3]);
          }
          asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
          __syncwarp();
          if (lane == 0) {
            tma_store_4d(&maps.out, smem_u32(buf), c * 32, q_row0 + wr * 32, p.o_head > 0 ? head : 0, p.o_seq > 0 ? seq : 0);
            bulk_commit();
          }
        }
        if (lane == 0) bulk_wait();
      }
    }
    __syncwarp();
  }

  tc_fence_before();
  __syncthreads();
  cluster_sync();      // nobody reads or signals this CTA any more: what the products signal was waited for in both
  if (warp == 0) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u) : "memory");
  }
}

}  // namespace pair

// ---------------------------------------------------------------------------------- host side
// Sets the kernel up on the current device: the pairs of CTAs it holds at once.  0: it cannot run them, attn_tc_kernel takes all.
int pair_create(int d) {
  const void* kern = d == 128 ? (const void*)pair::attn_pair_kernel<128> : (const void*)pair::attn_pair_kernel<64>;
  const int smem = d == 128 ? (int)pair::Layout<128>::SM_ALLOC : (int)pair::Layout<64>::SM_ALLOC;
  cudaFuncAttributes attr;
  if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) != cudaSuccess ||
      cudaFuncGetAttributes(&attr, kern) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  // the register hand-over inside the kernel must fit in what the launch really allocates
  if (attr.numRegs * pair::THREADS < 128 * pair::REGS_SMALL + 256 * pair::REGS_SOFTMAX) return 0;
  cudaLaunchConfig_t lc = {};
  lc.gridDim = dim3(2);
  lc.blockDim = dim3(pair::THREADS);
  lc.dynamicSmemBytes = smem;
  int n_pairs = 0;
  if (cudaOccupancyMaxActiveClusters(&n_pairs, kern, &lc) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return n_pairs;
}

cudaError_t launch_attn_pair_kernel(int d, const AttnParams& p, const tc::Maps& maps, cudaStream_t stream) {
  const dim3 grid((unsigned)(2 * p.attn_items));
  if (d == 128) return launch_pdl(pair::attn_pair_kernel<128>, grid, pair::THREADS, pair::Layout<128>::SM_ALLOC, stream, p, maps);
  return launch_pdl(pair::attn_pair_kernel<64>, grid, pair::THREADS, pair::Layout<64>::SM_ALLOC, stream, p, maps);
}

}  // namespace heatkv
