// Generic ragged attention kernel (warp-level MMA, online softmax), used for the small,
// bandwidth / latency bound scale steps and for calibration.
//
// One CTA = 64 queries of one (sequence, head); 4 warps x 16 query rows, or two such groups of warps that take the key
// half-tiles in turn and meet at the end.  Keys arrive as a
// sequence of half-tiles of up to 64 rows: first the head's retained prior keys, listed by
// the plan's page table (Sec. 3.3: the head-scales not in A_k), then the step's own keys
// from k_new.  In calibration mode (Eq. 2) every key comes from k_full and the per-row
// probability mass of every source scale is accumulated next to the online softmax, so the
// attention matrix alpha is never formed.
#include <atomic>
#include "append_device.cuh"

namespace heatkv {

constexpr int GM = 64;    // queries per CTA
constexpr int GN = 64;    // keys per half-tile
constexpr int GTHREADS = 128; // threads of one group
constexpr int GSTAGES = 2;   // key/value half-tiles in flight or in use per CTA (3 measured no faster: the small steps are bound by the warp-level MMA rate)

template <int D, int GROUPS = 1>
struct GenericSmem {
  static constexpr int TILE_BYTES = GN * D * 2;
  // q | per group: k[GSTAGES] | v[GSTAGES] | then seg_sum[GM][16] | seg_ref[GM][16]
  static constexpr int Q_OFF = 0;
  static constexpr int K_OFF = GM * D * 2;
  static constexpr int V_OFF = K_OFF + GSTAGES * TILE_BYTES;
  static constexpr int GROUP_BYTES = 2 * GSTAGES * TILE_BYTES;
  static constexpr int SEG_OFF = K_OFF + GROUPS * GROUP_BYTES;
  static constexpr int BYTES = SEG_OFF + 2 * GM * HEATKV_MAX_K * 4;
  static constexpr int ATTN_BYTES = SEG_OFF;             // without the calibration sums: two CTAs of head_dim 128 fit an SM
};

// byte offset of 16-byte chunk `ch` of row `r` in a [rows][D] bf16 tile (XOR swizzle)
template <int D>
__device__ __forceinline__ uint32_t tile_off(int r, int ch) {
  return (uint32_t)((r * (D / 8) + (ch ^ (r & 7))) * 16);
}

// copies n_valid rows (row-major, D bf16 each, `stride` elements apart) into a swizzled tile; the rows behind them that the
// products read are zero-filled: all of the tile's (WHOLE), or those up to the next multiple of 16.
template <int D, bool WHOLE, int THREADS = GTHREADS>
__device__ __forceinline__ void load_tile(uint32_t smem_base, const __nv_bfloat16* src, int64_t stride,
                                          int n_valid, int tid) {
  constexpr int CH = D / 8;
  constexpr int ROWS_PER_PASS = THREADS / CH;
  const int ch = tid % CH;
  const int r0 = tid / CH;
  const int rows = (n_valid + 15) & ~15;
#pragma unroll
  for (int r = r0; r < GN; r += ROWS_PER_PASS) {
    if (!WHOLE && r >= rows) break;
    const bool ok = r < n_valid;
    const __nv_bfloat16* p = ok ? src + (int64_t)r * stride + ch * 8 : src;
    cp_async16(smem_base + tile_off<D>(r, ch), p, ok ? 16 : 0);
  }
}

// Scratch of heatkv_calibrate_scores_static: one partial mass per (CTA, warp, source scale).  It lives in
// the library image, so that entry point needs no allocation; every GPU that loads the library holds
// these 4 MiB until the process exits.
constexpr int STATIC_PARTIAL_FLOATS = 1 << 20;
static __device__ __align__(256) float g_static_partials[STATIC_PARTIAL_FLOATS];

__device__ __forceinline__ void group_sync(int grp) {
  asm volatile("bar.sync %0, %1;" ::"r"(grp + 1), "n"(GTHREADS) : "memory");
}

// GROUPS = 2: a launch that leaves SMs idle is a chain of key half-tiles (1.4 to 2 us each: copies, products at the
// warp-level rate, softmax) per CTA; two groups of warps halve it.  Back to back, 2 sequences x 16 heads:
// 144 queries 19.8 us with one group and 12.4 with two, 64: 11.6 and 8.8, 36: 8.7 and 6.8.
template <int D, bool CALIB, bool PARTIALS = false, int GROUPS = 1>
__global__ void __launch_bounds__(GTHREADS * GROUPS, 2 / GROUPS) attn_generic_kernel(const __grid_constant__ AttnParams p) {
  extern __shared__ __align__(128) unsigned char smem[];
  using SM = GenericSmem<D, GROUPS>;
  // Two groups run a launch that is bound by latency: there the empty 16-key groups of a short tile, and warps without query
  // rows, are skipped.  With one group the launch fills the GPU, and the branches cost more than they save: 1024 queries
  // x 512 units 1951 -> 1287 us without them, allocation-free calibration over 13 scales 6.73 -> 4.70 ms, 64 queries
  // x 512 units 22.1 -> 17.8 us.
  constexpr bool SKIP = GROUPS == 2;
  static_assert(GROUPS == 1 || !CALIB, "the scale masses are kept by one group");
  const int grp = GROUPS == 1 ? 0 : __shfl_sync(0xffffffffu, (int)threadIdx.x / GTHREADS, 0);
  const int tid = threadIdx.x - grp * GTHREADS, warp = tid >> 5, lane = tid & 31;
  if (!PARTIALS) pdl_trigger();                        // (its follower, one small reduction, took SM slots from the tail: 64-wide heads 3 %)
  const int g = lane >> 2, qd = lane & 3;
  // attention: grid = (query tiles, sequences, heads by descending key count), so the heaviest heads of
  // every sequence are dispatched first; calibration: grid = (query tiles, heads, sequences)
  if (!CALIB && (int)blockIdx.x >= (p.t_q + GM - 1) / GM) {
    // cache update riding on this launch: one CTA per (destination half-tile, sequence, head)
    append_cta<D>(p, blockIdx.y, blockIdx.z, blockIdx.x - (p.t_q + GM - 1) / GM, threadIdx.x, GTHREADS * GROUPS);
    return;
  }
  const int seq = CALIB ? blockIdx.z : blockIdx.y;
  int head = CALIB ? blockIdx.y : blockIdx.z;
  // What a CTA works on comes from the launch parameters; a calibration launch may cover several steps
  // (heatkv_calibrate_scores_steps), its query tiles laid side by side along grid.x.
  int t_q = p.t_q, n_own = p.n_own, step = p.step, q0 = blockIdx.x * GM;
  const __nv_bfloat16* q_base = p.q;
  float* beta_row = p.beta_row;
  const float* seg_bias = p.seg_bias;
  if (CALIB && p.cal_n > 0) {
    int e = 0;
    while (e + 1 < p.cal_n && (int)blockIdx.x >= p.cal_tile_begin[e + 1]) ++e;
    step = p.cal_step[e];
    n_own = p.c[step];
    t_q = n_own - (step > 0 ? p.c[step - 1] : 0);
    q0 = ((int)blockIdx.x - p.cal_tile_begin[e]) * GM;
    q_base = p.q + (int64_t)(n_own - t_q) * p.q_tok;        // the step's queries on the token axis of all scales
    beta_row = p.beta_row + (int64_t)step * p.K;              // p.beta_row is beta_accum[layer][0][0] here
    if (seg_bias) seg_bias += (int64_t)step * p.cal_bias_stride;
  }

  const int2* descs = nullptr;
  int n_desc = 0;
  int64_t base_row = 0;
  if (!CALIB) {
    if (p.table_heads > 0) {
      // one schedule for the whole call: the host listed, per head in dispatch order, where its descriptors
      // start, so the first key tile is two dependent loads away instead of four
      head = p.table_head[blockIdx.z];
      descs = reinterpret_cast<const int2*>(p.seqs[seq].plan + p.table_desc_begin[blockIdx.z]);
      n_desc = p.table_ndesc[blockIdx.z];
    } else {
      PlanView pv(p.seqs[seq].plan);
      const int u = (p.step * p.L + p.layer) * p.H;
      head = pv.order()[u + blockIdx.z];                   // heavy heads first
      descs = pv.attn_descs(p.runs) + pv.attn_begin(p.runs)[u + head];
      n_desc = pv.attn_cnt(p.runs)[u + head];
    }
    base_row = p.seqs[seq].base_row;
  }
  const int n_own_tiles = (n_own + GN - 1) / GN;
  const int n_tiles = n_desc + n_own_tiles;

  const uint32_t sbase = smem_u32(smem);
  const uint32_t gbase = sbase + grp * SM::GROUP_BYTES;    // K_OFF / V_OFF of this group's stages count from here
  float* seg_sum = reinterpret_cast<float*>(smem + SM::SEG_OFF);
  float* seg_ref = seg_sum + GM * HEATKV_MAX_K;

  const __nv_bfloat16* kown = p.k_new + seq * p.kv_seq + head * p.kv_head;
  const __nv_bfloat16* vown = p.v_new ? p.v_new + seq * p.kv_seq + head * p.kv_head : nullptr;

  // descriptors are fetched one tile ahead of the copy they steer: `dsc_next` belongs to the tile issued next.
  // The group's i-th tile is tile grp + i * GROUPS of the CTA.
  int2 dsc_next = n_desc > grp ? descs[grp] : make_int2(0, 0);
  auto issue_tile = [&](int j, int stage) {
    const __nv_bfloat16 *ks, *vs;
    int64_t stride;
    int nv;
    if (j < n_desc) {
      int2 dsc = dsc_next;
      int64_t row = base_row + dsc.x;
      ks = p.k_pool + row * D;
      vs = p.v_pool + row * D;
      stride = D;
      nv = dsc.y & 0xff;
    } else {
      int jj = j - n_desc;
      ks = kown + (int64_t)jj * GN * p.kv_tok;
      vs = vown ? vown + (int64_t)jj * GN * p.kv_tok : nullptr;
      stride = p.kv_tok;
      nv = min(GN, n_own - jj * GN);
    }
    load_tile<D, !SKIP>(gbase + SM::K_OFF + stage * SM::TILE_BYTES, ks, stride, nv, tid);
    if (vs) load_tile<D, !SKIP>(gbase + SM::V_OFF + stage * SM::TILE_BYTES, vs, stride, nv, tid);
    if (j + GROUPS < n_desc) dsc_next = descs[j + GROUPS];
  };

  pdl_wait();
  // ---- prologue: Q tile and the first GSTAGES - 1 key tiles, one copy group each (empty groups keep the count)
  {
    const __nv_bfloat16* qsrc = q_base + seq * p.q_seq + head * p.q_head + (int64_t)q0 * p.q_tok;
    load_tile<D, !SKIP, GTHREADS * GROUPS>(sbase + SM::Q_OFF, qsrc, p.q_tok, min(GM, t_q - q0), threadIdx.x);
    cp_async_commit();
    for (int i = 0; i < GSTAGES - 1; ++i) {
      if (grp + i * GROUPS < n_tiles) issue_tile(grp + i * GROUPS, i);
      cp_async_commit();
    }
  }
  if (CALIB) {
    for (int i = tid; i < GM * HEATKV_MAX_K; i += GTHREADS) {
      seg_sum[i] = 0.f;
      seg_ref[i] = -INFINITY;
    }
  }
  cp_async_wait<GSTAGES - 1>();                        // Q has landed
  __syncthreads();

  uint32_t qf[D / 16][4];
#pragma unroll
  for (int ks = 0; ks < D / 16; ++ks) {
    int r = warp * 16 + (lane & 7) + ((lane >> 3) & 1) * 8;
    int ch = ks * 2 + (lane >> 4);
    ldmatrix_x4(qf[ks], sbase + SM::Q_OFF + tile_off<D>(r, ch));
  }

  float o[D / 8][4];
#pragma unroll
  for (int i = 0; i < D / 8; ++i) o[i][0] = o[i][1] = o[i][2] = o[i][3] = 0.f;
  float m_run[2] = {NO_MAX, NO_MAX};
  float l_run[2] = {0.f, 0.f};

  const bool has_rows = !SKIP || q0 + warp * 16 < t_q;  // SKIP: a warp without query rows only helps with the copies
  for (int i = 0, j = grp; j < n_tiles; ++i, j += GROUPS) {
    const int stage = i % GSTAGES;
    cp_async_wait<GSTAGES - 2>();                      // all groups but the newest GSTAGES - 2: tile j is among them
    if (GROUPS == 1) __syncthreads();                  // tile j landed for everyone; everyone left the tile before
    else group_sync(grp);
    if (j + (GSTAGES - 1) * GROUPS < n_tiles)          // into the stage of the tile before
      issue_tile(j + (GSTAGES - 1) * GROUPS, (i + GSTAGES - 1) % GSTAGES);
    cp_async_commit();
    if (!has_rows) continue;

    // tile attributes (warp-uniform)
    int nv, seg_lo, seg_hi, col0 = 0;
    if (j < n_desc) {
      int2 dsc = descs[j];
      nv = dsc.y & 0xff;
      seg_lo = seg_hi = (dsc.y >> 8) & 0xff;
    } else {
      int jj = j - n_desc;
      nv = min(GN, n_own - jj * GN);
      col0 = jj * GN;
      seg_lo = seg_hi = step;
      if (CALIB) {
        seg_lo = 0;
        while (p.c[seg_lo] <= col0) ++seg_lo;
        seg_hi = seg_lo;
        while (p.c[seg_hi] < col0 + nv) ++seg_hi;
      }
    }

    // ---- S = Q K^T
    float s[GN / 8][4];
#pragma unroll
    for (int i = 0; i < GN / 8; ++i) s[i][0] = s[i][1] = s[i][2] = s[i][3] = 0.f;
    const uint32_t kbase = gbase + SM::K_OFF + stage * SM::TILE_BYTES;
#pragma unroll
    for (int ks = 0; ks < D / 16; ++ks) {
#pragma unroll
      for (int np = 0; np < GN / 16; ++np) {
        if (SKIP && np * 16 >= nv) break;
        uint32_t b[4];
        int r = np * 16 + (lane & 7) + (lane >> 4) * 8;
        int ch = ks * 2 + ((lane >> 3) & 1);
        ldmatrix_x4(b, kbase + tile_off<D>(r, ch));
        mma_bf16(s[2 * np], qf[ks], b[0], b[1]);
        mma_bf16(s[2 * np + 1], qf[ks], b[2], b[3]);
      }
    }

    // ---- scale, bias, mask, online softmax
    const float* bias_h = seg_bias ? seg_bias + head * p.K : nullptr;
    const float LOG2E = 1.4426950408889634f;
    float tile_bias = bias_h ? bias_h[seg_lo] * LOG2E : 0.f;
    float mx[2] = {-INFINITY, -INFINITY};
#pragma unroll
    for (int n = 0; n < GN / 8; ++n) {
      if (SKIP && (n & ~1) * 8 >= nv) break;
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        int col = n * 8 + qd * 2 + (e & 1);
        float bias = tile_bias;
        if (CALIB && bias_h && seg_lo != seg_hi) {
          int sg = seg_lo;
          while (p.c[sg] <= col0 + col && sg < seg_hi) ++sg;
          bias = bias_h[sg] * LOG2E;
        }
        float v = col < nv ? fmaf(s[n][e], p.scale_log2, bias) : -INFINITY;
        s[n][e] = v;
        mx[e >> 1] = fmaxf(mx[e >> 1], v);
      }
    }
    float corr[2];
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      mx[r] = fmaxf(mx[r], __shfl_xor_sync(0xffffffffu, mx[r], 1));
      mx[r] = fmaxf(mx[r], __shfl_xor_sync(0xffffffffu, mx[r], 2));
      float m_new = fmaxf(m_run[r], mx[r]);
      corr[r] = exp2f(m_run[r] - m_new);
      m_run[r] = m_new;
      l_run[r] *= corr[r];
    }
    float psum[2] = {0.f, 0.f};
#pragma unroll
    for (int n = 0; n < GN / 8; ++n) {
      if (SKIP && (n & ~1) * 8 >= nv) break;
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        float pv = exp2f(s[n][e] - m_run[e >> 1]);
        s[n][e] = pv;
        psum[e >> 1] += pv;
      }
    }
    l_run[0] += psum[0];
    l_run[1] += psum[1];

    if (CALIB) {
      // per-row mass of every source scale that intersects this tile, kept as (sum, reference max)
      for (int sg = seg_lo; sg <= seg_hi; ++sg) {
        const int lo = sg > 0 ? p.c[sg - 1] : 0, hi = p.c[sg];
        float part[2] = {0.f, 0.f};
#pragma unroll
        for (int n = 0; n < GN / 8; ++n) {
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            int col = col0 + n * 8 + qd * 2 + (e & 1);
            if (col >= lo && col < hi) part[e >> 1] += s[n][e];
          }
        }
#pragma unroll
        for (int r = 0; r < 2; ++r) {
          part[r] += __shfl_xor_sync(0xffffffffu, part[r], 1);
          part[r] += __shfl_xor_sync(0xffffffffu, part[r], 2);
          if (qd == 0) {
            int row = warp * 16 + g + r * 8;
            float old = seg_sum[row * HEATKV_MAX_K + sg];
            float ref = seg_ref[row * HEATKV_MAX_K + sg];
            seg_sum[row * HEATKV_MAX_K + sg] = old * exp2f(ref - m_run[r]) + part[r];
            seg_ref[row * HEATKV_MAX_K + sg] = m_run[r];
          }
        }
      }
    }

    // ---- O = O * corr + P V
    if (!CALIB || p.out) {
#pragma unroll
      for (int i = 0; i < D / 8; ++i) {
        o[i][0] *= corr[0];
        o[i][1] *= corr[0];
        o[i][2] *= corr[1];
        o[i][3] *= corr[1];
      }
      const uint32_t vbase = gbase + SM::V_OFF + stage * SM::TILE_BYTES;
#pragma unroll
      for (int kk = 0; kk < GN / 16; ++kk) {
        if (SKIP && kk * 16 >= nv) break;
        uint32_t pa[4];
        pa[0] = pack_bf16(s[2 * kk][0], s[2 * kk][1]);
        pa[1] = pack_bf16(s[2 * kk][2], s[2 * kk][3]);
        pa[2] = pack_bf16(s[2 * kk + 1][0], s[2 * kk + 1][1]);
        pa[3] = pack_bf16(s[2 * kk + 1][2], s[2 * kk + 1][3]);
#pragma unroll
        for (int dp = 0; dp < D / 16; ++dp) {
          uint32_t b[4];
          int r = kk * 16 + (lane & 7) + ((lane >> 3) & 1) * 8;
          int ch = dp * 2 + (lane >> 4);
          ldmatrix_x4_trans(b, vbase + tile_off<D>(r, ch));
          mma_bf16(o[2 * dp], pa, b[0], b[1]);
          mma_bf16(o[2 * dp + 1], pa, b[2], b[3]);
        }
      }
    }
  }
  cp_async_wait<0>();

  if (GROUPS == 2) {
    // ---- the second group's partial result joins the first's (through the copy stages, which nobody reads any more)
    __syncthreads();
    float* part = reinterpret_cast<float*>(smem + SM::K_OFF) + tid;
    constexpr int STAT = D / 8 * 4 * GTHREADS;
    if (grp == 1) {
      if (has_rows) {
#pragma unroll
        for (int i = 0; i < D / 8; ++i)
#pragma unroll
          for (int e = 0; e < 4; ++e) part[(i * 4 + e) * GTHREADS] = o[i][e];
#pragma unroll
        for (int r = 0; r < 2; ++r) {
          part[STAT + r * GTHREADS] = m_run[r];
          part[STAT + (2 + r) * GTHREADS] = l_run[r];
        }
      }
    }
    __syncthreads();
    if (grp == 0 && has_rows) {
      float w0[2], w1[2];
#pragma unroll
      for (int r = 0; r < 2; ++r) {
        const float m1 = part[STAT + r * GTHREADS];     // NO_MAX when the second group had no tile
        const float m = fmaxf(m_run[r], m1);
        w0[r] = exp2f(m_run[r] - m);
        w1[r] = exp2f(m1 - m);
        l_run[r] = l_run[r] * w0[r] + part[STAT + (2 + r) * GTHREADS] * w1[r];
      }
#pragma unroll
      for (int i = 0; i < D / 8; ++i)
#pragma unroll
        for (int e = 0; e < 4; ++e)
          o[i][e] = o[i][e] * w0[e >> 1] + part[(i * 4 + e) * GTHREADS] * w1[e >> 1];
    }
  }

  // ---- epilogue
  float inv_l[2];
#pragma unroll
  for (int r = 0; r < 2; ++r) {
    float l = l_run[r];
    l += __shfl_xor_sync(0xffffffffu, l, 1);
    l += __shfl_xor_sync(0xffffffffu, l, 2);
    inv_l[r] = 1.f / l;
  }

  if (CALIB) {
    // beta[step][sg] += (1/t) * sum over rows of mass(row, sg) / l(row)     (Eq. 2)
    float* beta = beta_row + (int64_t)head * p.K * p.K;
    for (int sg = 0; sg <= step; ++sg) {
      float acc = 0.f;
      if (qd == 0) {
#pragma unroll
        for (int r = 0; r < 2; ++r) {
          int row = warp * 16 + g + r * 8;
          if (q0 + row < t_q)
            acc += seg_sum[row * HEATKV_MAX_K + sg] * exp2f(seg_ref[row * HEATKV_MAX_K + sg] - m_run[r]) * inv_l[r];
        }
      }
      acc += __shfl_xor_sync(0xffffffffu, acc, 4);
      acc += __shfl_xor_sync(0xffffffffu, acc, 8);
      acc += __shfl_xor_sync(0xffffffffu, acc, 16);
      if (PARTIALS) {
        // slot of (CTA, warp, source scale); reduce_partials_kernel adds them up in a fixed order
        const int64_t cta = blockIdx.x + (int64_t)gridDim.x * (blockIdx.y + (int64_t)gridDim.y * blockIdx.z);
        if (lane == 0) p.partials[(cta * (GTHREADS / 32) + warp) * HEATKV_MAX_K + sg] = acc / (float)t_q;
      } else {
        if (lane == 0) atomicAdd(beta + sg, acc / (float)t_q);
      }
    }
  }

  if (p.out) {
    __syncthreads();                                   // all warps are done with the K/V stages
    // stage the bf16 tile in shared memory (reusing the Q region), then 16-byte row stores
    if (grp == 0 && has_rows) {
#pragma unroll
    for (int n = 0; n < D / 8; ++n) {
      int r0 = warp * 16 + g;
      uint32_t lo = pack_bf16(o[n][0] * inv_l[0], o[n][1] * inv_l[0]);
      uint32_t hi = pack_bf16(o[n][2] * inv_l[1], o[n][3] * inv_l[1]);
      *reinterpret_cast<uint32_t*>(smem + SM::Q_OFF + tile_off<D>(r0, n) + qd * 4) = lo;
      *reinterpret_cast<uint32_t*>(smem + SM::Q_OFF + tile_off<D>(r0 + 8, n) + qd * 4) = hi;
    }
    }
    __syncthreads();
    constexpr int CH = D / 8;
    __nv_bfloat16* dst = p.out + seq * p.o_seq + head * p.o_head + (int64_t)q0 * p.o_tok;
    for (int i = threadIdx.x; i < GM * CH; i += GTHREADS * GROUPS) {
      int r = i / CH, ch = i % CH;
      if (q0 + r < t_q) {
        int4 v = *reinterpret_cast<const int4*>(smem + SM::Q_OFF + tile_off<D>(r, ch));
        *reinterpret_cast<int4*>(dst + (int64_t)r * p.o_tok + ch * 8) = v;
      }
    }
  }
}

// ---------------------------------------------------------------------------------- attention of the small steps
// What bounds a small scale step is the chain of one CTA: descriptors, the first copies, then per key half-tile the
// products at the warp-level rate (a 16 x 16 x 128 chunk, S and PV, takes a warp about 0.5 us) and the softmax.  So a CTA
// is 16 queries and four warps, one per SM sub-partition, that take 16 keys of every half-tile each and meet once at the
// end in shared memory, where all threads normalise and write.  The step's own keys, whose place needs no descriptor,
// come first.  2 sequences x 16 heads, back to back, against 64 queries per CTA with two groups of four warps:
// 4 queries 3.3 against 4.0 us, 36: 6.4 against 6.8, 64: 7.9 against 8.8, 144: 11.7 against 12.4.  K and V are read once per
// 16 queries, so a launch that fills the SMs is better off with the 64-query CTAs (8 sequences, 64 queries: 12.4 against
// 9.1 us).
constexpr int SKEYS = 16;      // keys of a half-tile one warp takes
constexpr int SGROUPS = GN / SKEYS;
constexpr int SSTAGES = 3;

template <int D>
struct SmallSmem {
  static constexpr int ROWS = 16;
  static constexpr int CHUNK_BYTES = SKEYS * D * 2;                 // K or V of one warp and stage
  static constexpr int Q_OFF = 0;
  static constexpr int KV_OFF = ROWS * D * 2;                       // [warp][stage][K | V]
  static constexpr int KV_BYTES = SGROUPS * SSTAGES * 2 * CHUNK_BYTES;
  static constexpr int PART_STRIDE = D + 8;                         // floats per row of a partial O (8: no bank conflicts)
  static constexpr int PART_BYTES = SGROUPS * ROWS * PART_STRIDE * 4;      // takes the place of the copy stages
  static_assert(PART_BYTES <= KV_BYTES, "partial results");
  static constexpr int STAT_OFF = KV_OFF + KV_BYTES;   // [reference | sum][warp][row]
  static constexpr int BYTES = STAT_OFF + 2 * SGROUPS * ROWS * 4;
};

// FP8: the cached keys are read from the code pools themselves (a chunk's codes land in its place in shared memory and are
// widened there), so a small step of such a context needs no expansion launch before it (4 x 16 units, 4 queries: 6.4 -> 3.5 us,
// 64 queries: 12.3 -> 8.1).
template <int D, bool FP8>
__global__ void __launch_bounds__(GTHREADS, 2) attn_small_kernel(const __grid_constant__ AttnParams p) {
  using SM = SmallSmem<D>;
  extern __shared__ __align__(128) unsigned char smem[];
  pdl_trigger();
  const int q_tiles = (p.t_q + SM::ROWS - 1) / SM::ROWS;
  if ((int)blockIdx.x >= q_tiles) {
    // cache update riding on this launch: one CTA per (destination half-tile, sequence, head)
    append_cta<D>(p, blockIdx.y, blockIdx.z, blockIdx.x - q_tiles, threadIdx.x, GTHREADS);
    return;
  }
  const int grp = __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
  const int g = lane >> 2, qd = lane & 3;
  const int seq = blockIdx.y, q0 = blockIdx.x * SM::ROWS;
  int head, n_desc;
  const int2* descs;
  if (p.table_heads > 0) {
    head = p.table_head[blockIdx.z];
    descs = reinterpret_cast<const int2*>(p.seqs[seq].plan + p.table_desc_begin[blockIdx.z]);
    n_desc = p.table_ndesc[blockIdx.z];
  } else {
    PlanView pv(p.seqs[seq].plan);
    const int u = (p.step * p.L + p.layer) * p.H;
    head = pv.order()[u + blockIdx.z];                   // heavy heads first
    descs = pv.attn_descs(p.runs) + pv.attn_begin(p.runs)[u + head];
    n_desc = pv.attn_cnt(p.runs)[u + head];
  }
  const int64_t base_row = FP8 ? p.pool_base[seq] : p.seqs[seq].base_row;
  const int n_own_tiles = (p.n_own + GN - 1) / GN, n_tiles = n_own_tiles + n_desc;
  const uint32_t sbase = smem_u32(smem);
  const uint32_t kvbase = sbase + SM::KV_OFF + grp * (SSTAGES * 2 * SM::CHUNK_BYTES);
  const __nv_bfloat16* kown = p.k_new + seq * p.kv_seq + head * p.kv_head;
  const __nv_bfloat16* vown = p.v_new + seq * p.kv_seq + head * p.kv_head;

  const int32_t* src_rows = nullptr;                     // FP8: the pool rows behind the head's descriptors
  if (FP8) {
    const int32_t* plan = p.seqs[seq].plan;
    const int off_desc = p.table_heads > 0 ? p.off_desc : plan[p.runs ? 18 : 4];
    const int off_src = p.table_heads > 0 ? p.off_src : plan[p.runs ? 21 : 17];
    src_rows = plan + off_src + (reinterpret_cast<const int32_t*>(descs) - (plan + off_desc)) / 2;
  }

  // This warp's keys of tile j: rows [16 sub, 16 sub + n) of it.  The assignment turns with the tile, so that short tiles
  // do not all fall to the same warps.  `dsc` is the tile's descriptor (used past the own tiles).
  auto part_of = [&](int j, int2 dsc, int& sub) {
    sub = (grp + 2 * j) & (SGROUPS - 1);
    const int nv = j < n_own_tiles ? p.n_own - j * GN : dsc.y & 0xff;
    return min(SKEYS, max(0, nv - sub * SKEYS));
  };
  auto load_chunk = [&](uint32_t dst, const __nv_bfloat16* src, int64_t stride, int n) {
    constexpr int CH = D / 8;
#pragma unroll
    for (int i = lane; i < SKEYS * CH; i += 32) {
      const int r = i / CH, ch = i % CH;
      const bool ok = r < n;
      cp_async16(dst + tile_off<D>(r, ch), ok ? src + (int64_t)r * stride + ch * 8 : src, ok ? 16 : 0);
    }
  };
  auto load_codes = [&](uint32_t dst, const uint8_t* src, int n) {          // rows of D codes, one after the other
    constexpr int CH = D / 16;
#pragma unroll
    for (int i = lane; i < SKEYS * CH; i += 32) {
      const bool ok = i / CH < n;
      cp_async16(dst + i * 16, ok ? src + i * 16 : src, ok ? 16 : 0);
    }
  };
  // FP8: exponent byte of K row `lane` (lanes 0..15) or V row `lane - 16` of the chunk
  auto issue = [&](int j, int2 dsc, int stage, int& exponent) {
    int sub;
    const int n = part_of(j, dsc, sub);
    if (n <= 0) return;
    const uint32_t dst = kvbase + stage * 2 * SM::CHUNK_BYTES;
    if (j < n_own_tiles) {
      const int64_t off = (int64_t)(j * GN + sub * SKEYS) * p.kv_tok;
      load_chunk(dst, kown + off, p.kv_tok, n);
      load_chunk(dst + SM::CHUNK_BYTES, vown + off, p.kv_tok, n);
    } else if (FP8) {
      const int64_t r0 = base_row + dsc.x + sub * SKEYS;
      load_codes(dst, p.k8_pool + r0 * D, n);
      load_codes(dst + SM::CHUNK_BYTES, p.v8_pool + r0 * D, n);
      const int r = lane & 15;
      exponent = r < n ? (lane < 16 ? p.k_exp : p.v_exp)[r0 + r] : 0;
    } else {
      const int64_t off = (base_row + dsc.x + sub * SKEYS) * D;
      load_chunk(dst, p.k_pool + off, D, n);
      load_chunk(dst + SM::CHUNK_BYTES, p.v_pool + off, D, n);
    }
  };
  // codes of a chunk -> bf16 rows in the swizzled layout, in place
  auto widen = [&](unsigned char* chunk, int exponent, int first_lane) {
    constexpr int CH = D / 8, PER_LANE = SKEYS * CH / 32;
    uint2 c[PER_LANE];
#pragma unroll
    for (int i = 0; i < PER_LANE; ++i) c[i] = *reinterpret_cast<const uint2*>(chunk + (lane + 32 * i) * 8);
    __syncwarp();
#pragma unroll
    for (int i = 0; i < PER_LANE; ++i) {
      const int r = (lane + 32 * i) / CH, ch = (lane + 32 * i) % CH;
      const float scale = pow2f(__shfl_sync(0xffffffffu, exponent, first_lane + r));
      const uint32_t w[4] = {c[i].x & 0xffffu, c[i].x >> 16, c[i].y & 0xffffu, c[i].y >> 16};
      uint32_t o[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        float lo, hi;
        from_e4m3x2(w[q], lo, hi);
        o[q] = pack_bf16(lo * scale, hi * scale);          // exact, as in the expansion kernel
      }
      *reinterpret_cast<int4*>(chunk + tile_off<D>(r, ch)) = make_int4((int)o[0], (int)o[1], (int)o[2], (int)o[3]);
    }
  };
  auto desc_of = [&](int j) {
    if (j < n_own_tiles || j >= n_tiles) return make_int2(0, 0);
    int2 d = descs[j - n_own_tiles];
    if (FP8) d.x = src_rows[j - n_own_tiles];
    return d;
  };

  // descriptors run SSTAGES tiles ahead of the products: ahead[i] belongs to the i-th tile from the current one
  int2 ahead[SSTAGES];
  int exps[SSTAGES] = {};
#pragma unroll
  for (int i = 0; i < SSTAGES; ++i) ahead[i] = desc_of(i);
  pdl_wait();
  {
    constexpr int CH = D / 8;
    const __nv_bfloat16* qsrc = p.q + seq * p.q_seq + head * p.q_head + (int64_t)q0 * p.q_tok;
#pragma unroll
    for (int i = threadIdx.x; i < SM::ROWS * CH; i += GTHREADS) {
      const int r = i / CH, ch = i % CH;
      const bool ok = q0 + r < p.t_q;
      cp_async16(sbase + SM::Q_OFF + tile_off<D>(r, ch), ok ? qsrc + (int64_t)r * p.q_tok + ch * 8 : qsrc, ok ? 16 : 0);
    }
  }
  cp_async_commit();
#pragma unroll
  for (int i = 0; i < SSTAGES - 1; ++i) {
    if (i < n_tiles) issue(i, ahead[i], i, exps[i]);
    cp_async_commit();
  }
  cp_async_wait<SSTAGES - 1>();                          // Q has landed
  __syncthreads();
  uint32_t qf[D / 16][4];
#pragma unroll
  for (int ks = 0; ks < D / 16; ++ks)
    ldmatrix_x4(qf[ks], sbase + SM::Q_OFF + tile_off<D>((lane & 7) + ((lane >> 3) & 1) * 8, ks * 2 + (lane >> 4)));

  float o[D / 8][4];
#pragma unroll
  for (int i = 0; i < D / 8; ++i) o[i][0] = o[i][1] = o[i][2] = o[i][3] = 0.f;
  float m_run[2] = {NO_MAX, NO_MAX}, l_run[2] = {0.f, 0.f};
  const float LOG2E = 1.4426950408889634f;
  const float* bias_h = p.seg_bias ? p.seg_bias + head * p.K : nullptr;

  for (int j = 0; j < n_tiles; ++j) {
    const int stage = j % SSTAGES;
    const int2 dsc = ahead[0];
#pragma unroll
    for (int i = 0; i + 1 < SSTAGES; ++i) ahead[i] = ahead[i + 1];
    ahead[SSTAGES - 1] = desc_of(j + SSTAGES);
    const int exponent = exps[0];
#pragma unroll
    for (int i = 0; i + 1 < SSTAGES; ++i) exps[i] = exps[i + 1];
    cp_async_wait<SSTAGES - 2>();
    __syncwarp();                                        // the warp's chunk landed; every lane left the one before
    if (j + SSTAGES - 1 < n_tiles) issue(j + SSTAGES - 1, ahead[SSTAGES - 2], (j + SSTAGES - 1) % SSTAGES, exps[SSTAGES - 2]);
    cp_async_commit();
    int sub;
    const int n = part_of(j, dsc, sub);
    if (n <= 0) continue;

    const uint32_t kb = kvbase + stage * 2 * SM::CHUNK_BYTES, vb = kb + SM::CHUNK_BYTES;
    if (FP8 && j >= n_own_tiles) {
      widen(smem + (kb - sbase), exponent, 0);
      widen(smem + (vb - sbase), exponent, 16);
      __syncwarp();
    }
    float s[2][4] = {};
#pragma unroll
    for (int ks = 0; ks < D / 16; ++ks) {
      uint32_t b[4];
      ldmatrix_x4(b, kb + tile_off<D>((lane & 7) + (lane >> 4) * 8, ks * 2 + ((lane >> 3) & 1)));
      mma_bf16(s[0], qf[ks], b[0], b[1]);
      mma_bf16(s[1], qf[ks], b[2], b[3]);
    }
    const float bias = bias_h ? bias_h[j < n_own_tiles ? p.step : (dsc.y >> 8) & 0xff] * LOG2E : 0.f;
    float mx[2] = {-INFINITY, -INFINITY}, psum[2] = {0.f, 0.f}, corr[2];
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const float v = i * 8 + qd * 2 + (e & 1) < n ? fmaf(s[i][e], p.scale_log2, bias) : -INFINITY;
        s[i][e] = v;
        mx[e >> 1] = fmaxf(mx[e >> 1], v);
      }
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      mx[r] = fmaxf(mx[r], __shfl_xor_sync(0xffffffffu, mx[r], 1));
      mx[r] = fmaxf(mx[r], __shfl_xor_sync(0xffffffffu, mx[r], 2));
      const float m_new = fmaxf(m_run[r], mx[r]);
      corr[r] = exp2f(m_run[r] - m_new);
      m_run[r] = m_new;
    }
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        s[i][e] = exp2f(s[i][e] - m_run[e >> 1]);
        psum[e >> 1] += s[i][e];
      }
    l_run[0] = l_run[0] * corr[0] + psum[0];
    l_run[1] = l_run[1] * corr[1] + psum[1];
    if (__any_sync(0xffffffffu, corr[0] != 1.f || corr[1] != 1.f)) {
#pragma unroll
      for (int i = 0; i < D / 8; ++i) {
        o[i][0] *= corr[0];
        o[i][1] *= corr[0];
        o[i][2] *= corr[1];
        o[i][3] *= corr[1];
      }
    }
    uint32_t pa[4] = {pack_bf16(s[0][0], s[0][1]), pack_bf16(s[0][2], s[0][3]), pack_bf16(s[1][0], s[1][1]),
                      pack_bf16(s[1][2], s[1][3])};
#pragma unroll
    for (int dp = 0; dp < D / 16; ++dp) {
      uint32_t b[4];
      ldmatrix_x4_trans(b, vb + tile_off<D>((lane & 7) + ((lane >> 3) & 1) * 8, dp * 2 + (lane >> 4)));
      mma_bf16(o[2 * dp], pa, b[0], b[1]);
      mma_bf16(o[2 * dp + 1], pa, b[2], b[3]);
    }
  }
  cp_async_wait<0>();
  __syncthreads();                                       // the copy stages are free: the partial results take their place

  float* part = reinterpret_cast<float*>(smem + SM::KV_OFF);
  float* stat = reinterpret_cast<float*>(smem + SM::STAT_OFF);
#pragma unroll
  for (int r = 0; r < 2; ++r) {
    const int row = g + r * 8;
    float l = l_run[r];
    l += __shfl_xor_sync(0xffffffffu, l, 1);
    l += __shfl_xor_sync(0xffffffffu, l, 2);
    if (qd == 0) {
      stat[grp * SM::ROWS + row] = m_run[r];
      stat[(SGROUPS + grp) * SM::ROWS + row] = l;
    }
    float* dst = part + (grp * SM::ROWS + row) * SM::PART_STRIDE + qd * 2;
#pragma unroll
    for (int i = 0; i < D / 8; ++i) *reinterpret_cast<float2*>(dst + i * 8) = make_float2(o[i][2 * r], o[i][2 * r + 1]);
  }
  __syncthreads();
  constexpr int CH = D / 8;
  __nv_bfloat16* out = p.out + seq * p.o_seq + head * p.o_head + (int64_t)q0 * p.o_tok;
#pragma unroll
  for (int i = threadIdx.x; i < SM::ROWS * CH; i += GTHREADS) {
    const int row = i / CH, ch = i % CH;
    if (q0 + row >= p.t_q) continue;
    // a warp without keys (reference NO_MAX, sum 0) weighs nothing
    float w[SGROUPS], m = -INFINITY, l = 0.f, acc[8] = {};
#pragma unroll
    for (int k = 0; k < SGROUPS; ++k) m = fmaxf(m, stat[k * SM::ROWS + row]);
#pragma unroll
    for (int k = 0; k < SGROUPS; ++k) {
      w[k] = exp2f(stat[k * SM::ROWS + row] - m);
      l = fmaf(stat[(SGROUPS + k) * SM::ROWS + row], w[k], l);
    }
    const float inv = 1.f / l;
#pragma unroll
    for (int k = 0; k < SGROUPS; ++k) {
      const float4* src = reinterpret_cast<const float4*>(part + (k * SM::ROWS + row) * SM::PART_STRIDE + ch * 8);
      const float4 a = src[0], b = src[1];
      const float v[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
#pragma unroll
      for (int e = 0; e < 8; ++e) acc[e] = fmaf(v[e], w[k], acc[e]);
    }
    *reinterpret_cast<int4*>(out + (int64_t)row * p.o_tok + ch * 8) =
        make_int4((int)pack_bf16(acc[0] * inv, acc[1] * inv), (int)pack_bf16(acc[2] * inv, acc[3] * inv),
                  (int)pack_bf16(acc[4] * inv, acc[5] * inv), (int)pack_bf16(acc[6] * inv, acc[7] * inv));
  }
}

// beta[head][step][sg] += sum of the partials of that head in the order (sequence, query tile, warp):
// one thread per (head, source scale), so the result does not depend on scheduling.
__global__ void reduce_partials_kernel(const float* partials, float* beta_row, int n_qtiles, int H, int n_seq, int K,
                                       int step) {
  const int head = blockIdx.x, sg = threadIdx.x;
  pdl_trigger();
  pdl_wait();
  if (sg > step) return;
  float acc = 0.f;
  for (int seq = 0; seq < n_seq; ++seq)
    for (int qt = 0; qt < n_qtiles; ++qt) {
      const int64_t cta = qt + (int64_t)n_qtiles * (head + (int64_t)H * seq);
      for (int w = 0; w < GTHREADS / 32; ++w) acc += partials[(cta * (GTHREADS / 32) + w) * HEATKV_MAX_K + sg];
    }
  beta_row[(int64_t)head * K * K + sg] += acc;
}

constexpr int MAX_DEVICES = 64;

// the attribute belongs to the (function, device) pair: set it once on every device that launches
template <auto KERN>
static cudaError_t allow_smem(int bytes) {
  static std::atomic<bool> configured[MAX_DEVICES];
  int dev = -1;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= MAX_DEVICES) return cudaErrorInvalidDevice;
  if (!configured[dev].load(std::memory_order_acquire)) {
    e = cudaFuncSetAttribute(KERN, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (e != cudaSuccess) return e;
    configured[dev].store(true, std::memory_order_release);
  }
  return cudaSuccess;
}

template <int D, bool CALIB, int GROUPS = 1>
static cudaError_t launch_one(const AttnParams& p, int n_seq, cudaStream_t stream) {
  constexpr auto kern = attn_generic_kernel<D, CALIB, false, GROUPS>;
  constexpr int bytes = CALIB ? GenericSmem<D>::BYTES : GenericSmem<D, GROUPS>::ATTN_BYTES;
  cudaError_t e = allow_smem<kern>(bytes);
  if (e != cudaSuccess) return e;
  const int q_tiles = CALIB && p.cal_n > 0 ? p.cal_tile_begin[p.cal_n] : (p.t_q + GM - 1) / GM;
  dim3 grid(q_tiles + (CALIB ? 0 : p.append_tiles), CALIB ? p.H : n_seq, CALIB ? n_seq : p.H);
  return launch_pdl(kern, grid, GTHREADS * GROUPS, bytes, stream, p);
}

template <int D, bool FP8>
static cudaError_t launch_small(const AttnParams& p, int n_seq, cudaStream_t stream) {
  constexpr auto kern = attn_small_kernel<D, FP8>;
  constexpr int bytes = SmallSmem<D>::BYTES;
  cudaError_t e = allow_smem<kern>(bytes);
  if (e != cudaSuccess) return e;
  dim3 grid((p.t_q + SmallSmem<D>::ROWS - 1) / SmallSmem<D>::ROWS + p.append_tiles, n_seq, p.H);
  return launch_pdl(kern, grid, GTHREADS, bytes, stream, p);
}

// Calibration pass whose scratch is the static array above.  Returns cudaErrorInvalidValue when the
// launch would need more partial slots than the array has.  The array's device address is looked up
// once per device (cudaGetSymbolAddress; the symbol's name itself is only a host-side handle).
cudaError_t launch_calibrate_static(const AttnParams& p_in, int d, int n_seq, cudaStream_t stream, bool* too_large) {
  *too_large = false;
  const int n_qtiles = (p_in.t_q + GM - 1) / GM;
  const int64_t slots = (int64_t)n_qtiles * p_in.H * n_seq * (GTHREADS / 32) * HEATKV_MAX_K;
  if (slots > STATIC_PARTIAL_FLOATS) {
    *too_large = true;
    return cudaErrorInvalidValue;
  }
  static std::atomic<float*> scratch_of_device[MAX_DEVICES];
  static std::atomic<bool> configured[MAX_DEVICES][2];
  int dev = -1;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= MAX_DEVICES) return cudaErrorInvalidDevice;
  float* scratch = scratch_of_device[dev].load(std::memory_order_acquire);
  if (!scratch) {
    e = cudaGetSymbolAddress(reinterpret_cast<void**>(&scratch), g_static_partials);
    if (e != cudaSuccess) return e;
    scratch_of_device[dev].store(scratch, std::memory_order_release);
  }
  AttnParams p = p_in;
  p.partials = scratch;
  p.out = nullptr;
  p.v_new = nullptr;
  const int which = d == 128 ? 1 : 0;
  dim3 grid(n_qtiles, p.H, n_seq);
  if (d == 128) {
    auto kern = attn_generic_kernel<128, true, true>;
    if (!configured[dev][which].load(std::memory_order_acquire)) {
      e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, GenericSmem<128>::BYTES);
      if (e != cudaSuccess) return e;
      configured[dev][which].store(true, std::memory_order_release);
    }
    e = launch_pdl(kern, grid, GTHREADS, GenericSmem<128>::BYTES, stream, p);
  } else if (d == 64) {
    auto kern = attn_generic_kernel<64, true, true>;
    if (!configured[dev][which].load(std::memory_order_acquire)) {
      e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, GenericSmem<64>::BYTES);
      if (e != cudaSuccess) return e;
      configured[dev][which].store(true, std::memory_order_release);
    }
    e = launch_pdl(kern, grid, GTHREADS, GenericSmem<64>::BYTES, stream, p);
  } else {
    return cudaErrorInvalidValue;
  }
  if (e != cudaSuccess) return e;
  return launch_pdl(reduce_partials_kernel, p.H, HEATKV_MAX_K, 0, stream, (const float*)p.partials, p.beta_row, n_qtiles, p.H,
                    n_seq, p.K, p.step);
}

// Does the small-step kernel take an attention launch of t_q queries and `units` (sequence, head) pairs?  16-query CTAs while two of them per SM hold the launch (or the step has no more queries than
// that: then nothing is read twice); else two groups of warps per 64-query CTA while every CTA has an SM to itself and heads
// see more than one key half-tile; a fuller launch keeps two single-group CTAs per SM (the same warps per SM, and nothing
// to merge).
bool attn_is_small(int t_q, int64_t units, int n_sm) { return t_q <= 16 || (t_q + 15) / 16 * units <= 2 * n_sm; }

// `n_sm`: SMs of the device.
cudaError_t launch_attn_generic(const AttnParams& p, int d, int n_seq, bool calib, int n_sm, cudaStream_t stream) {
  if (d != 64 && d != 128) return cudaErrorInvalidValue;
  if (calib) return d == 128 ? launch_one<128, true>(p, n_seq, stream) : launch_one<64, true>(p, n_seq, stream);
  const int64_t units = (int64_t)n_seq * p.H;
  if (attn_is_small(p.t_q, units, n_sm))                    // (direct8 is set under this same rule)
    return p.direct8 ? (d == 128 ? launch_small<128, true>(p, n_seq, stream) : launch_small<64, true>(p, n_seq, stream))
                     : (d == 128 ? launch_small<128, false>(p, n_seq, stream) : launch_small<64, false>(p, n_seq, stream));
  if (p.step > 0 && (p.t_q + GM - 1) / GM * units <= n_sm)
    return d == 128 ? launch_one<128, false, 2>(p, n_seq, stream) : launch_one<64, false, 2>(p, n_seq, stream);
  return d == 128 ? launch_one<128, false>(p, n_seq, stream) : launch_one<64, false>(p, n_seq, stream);
}

}  // namespace heatkv
