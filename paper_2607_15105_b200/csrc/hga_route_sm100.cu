// hga_route for sm_100a: chunk selection and group selection (Section 2.1 items 1-2) as one
// fused tcgen05 kernel per item (b, kv head, query block).
//
// Scores are the max (or mean / log-sum-exp, HGA_FLAG_SCORE_*) over the item's G*Bq query rows of q . summary.  The GEMM
// puts 128 summaries on the MMA M dimension (= TMEM lanes) and the query rows on N (= TMEM columns), so the
// reduction over rows is an in-thread reduction over the columns a thread reads back with
// tcgen05.ld: thread = summary.
//   phase 1  candidate chunk summaries, 128 per tile, streamed by TMA
//   select   the k_c best chunks by score, ties to the lowest index, in ascending order
//   phase 2  the opened chunks' group summaries (c/g = 8 or 16 consecutive rows per chunk, i.e.
//            one or two octets each) gathered by TMA, same GEMM, then top-kg_eff inside each chunk
// bf16 x bf16 products are exact in fp32; only the accumulation order differs from an exact sum.
//
// Pipeline.  The query rows are taken in parts of up to 128 columns, each with an accumulator of its own, so that the
// readers work on one part while the tensor pipe works on the next.  A summary tile arrives in slabs of 64 elements
// (16 KB); a slab is free as soon as every part has used it, so the next tile's first slab is copied during the second
// half of this tile's GEMMs.  Where Q, two slabs and the scores fit half of an SM (up to 256 query rows at head_dim 128)
// two CTAs share it and one's serial phases hide behind the other's GEMMs; four slabs where they fit; larger row
// counts take a whole SM with four accumulators.
//
// Code size: a CTA of a small problem runs most of this once, on instruction caches that other kernels have filled meanwhile, so
// loops that are not hot are not unrolled (left to itself the compiler made 127 KB of it, now 67): whole steps, 16K layer
// 147.1 -> 145.6 us, one / 32 tokens of a generation 16.6 -> 15.4 and 36.9 -> 35.1, tiny layer 43.6 -> 42.7, 128K 90.2 -> 89.4.
#include <algorithm>
#include <cfloat>
#include <type_traits>

#include "hga_common.cuh"
#include "hga_sm100.cuh"

namespace hga {

using namespace sm100;

namespace {

constexpr int kRtThreads = 256;     // warp 0 producer, warp 1 MMA, warps 2-5 readers, 6-7 help in select
constexpr int kRtWarps = kRtThreads / 32, kRtCopyWarps = kRtWarps - 2;
constexpr int kSlab = 128 * 128;    // bytes of 128 summaries x 64 elements
constexpr int kRankMax = kRtThreads;      // up to here a candidate's rank is counted directly, by a thread each
constexpr int kMostFinal = 64;            // up to so many chunks to select the warps pick their best first

template <int NSTG, int ACCS>
struct RouteSmem {
  alignas(1024) uint8_t a[NSTG][kSlab];
  uint64_t q_full, a_full[NSTG], a_empty[NSTG], acc_full[ACCS], acc_free[ACCS];
  uint64_t drain;              // give-up path only: completes when the tensor pipe has run dry
  uint32_t tmem_base;
  volatile int abort;
  // dynamic tail (see RouteLayout): Q rows (B operand, 1024-aligned), scores, bitmap, selected chunks, group scores
};

// Query rows of an item on the MMA N dimension: equal parts of at most 128 columns, each a multiple of 32
struct RouteLayout {
  int parts, part_cols, q_bytes, n_keys, n_final;
  __host__ __device__ RouteLayout(const Dims& dm, int max_cand) {
    const int rows = rows_padded(dm);
    parts = (rows + 127) / 128;
    part_cols = ((rows + parts - 1) / parts + 31) & ~31;
    q_bytes = parts * part_cols * dm.d * 2;
    n_keys = (max_cand + 7) & ~3;
    n_final = max_cand > kRankMax && dm.kc <= kMostFinal ? kRtWarps * dm.kc : 0;
  }
  size_t tail(const Dims& dm) const {
    return 1024 + (size_t)q_bytes + 4 * ((size_t)n_keys + 2 * n_final + 128 + dm.kc + (size_t)dm.kc * dm.per + 8);
  }
};

__device__ __forceinline__ bool rt_wait(uint64_t* bar, uint32_t parity, volatile int* abort) {
  return mbar_wait_bounded(bar, parity, abort);
}

__device__ __forceinline__ uint32_t rt_orderable(float f) {
  const uint32_t u = __float_as_uint(f);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float rt_score(uint32_t key) {
  return __uint_as_float((key & 0x80000000u) ? key ^ 0x80000000u : ~key);
}

// The k largest of n keys (k <= n), ties to the lowest position, by one warp: emit(position, rank by position, key) for each.  The
// k-th largest is found bit by bit below the bits that all keys share.  KPL: keys that a lane keeps in registers
// (n <= 32 KPL), 0 = they are read again in every round.
template <int KPL, class F>
__device__ __forceinline__ void warp_select(const uint32_t* keys, int n, int k, F emit) {
  const unsigned full = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  uint32_t own[KPL > 0 ? KPL : 1];
  if constexpr (KPL > 0) {
#pragma unroll
    for (int q = 0; q < KPL; ++q) own[q] = 32 * q + lane < n ? keys[32 * q + lane] : 0u;
  }
  auto each = [&](auto f) {              // f(key), padding keys among them as 0
    if constexpr (KPL > 0) {
#pragma unroll
      for (int q = 0; q < KPL; ++q) f(own[q]);
    } else {
#pragma unroll 4
      for (int i = lane; i < n; i += 32) f(keys[i]);
    }
  };
  uint32_t hi = 0, both = 0xffffffffu, any = 0;      // bits that are one / not zero in all keys
  each([&](uint32_t key) { hi = max(hi, key); });
#pragma unroll 1
  for (int i = lane; i < n; i += 32) {
    const uint32_t key = keys[i];
    both &= key;
    any |= key;
  }
  hi = __reduce_max_sync(full, hi);
  const uint32_t differ = __reduce_or_sync(full, any) ^ __reduce_and_sync(full, both);
  uint32_t kth = hi;                    // in the end the largest value that at least k keys reach
  if (differ != 0) {
    uint32_t bit = 0x80000000u >> __clz(differ);
    kth = hi & ~(2 * bit - 1);          // (2 * bit wraps to 0 at the top bit: nothing is shared)
#pragma unroll 1
    for (int reach = n; bit != 0 && reach != k; bit >>= 1) {
      const uint32_t t = kth | bit;
      int c = 0;
      each([&](uint32_t key) { c += key >= t ? 1 : 0; });
      c = __reduce_add_sync(full, c);
      if (c >= k) { kth = t; reach = c; }
    }
  }
  int above = 0;
  each([&](uint32_t key) { above += key > kth ? 1 : 0; });
  int ties = k - __reduce_add_sync(full, above), rank = 0;      // of the keys equal to it, how many are still to be taken
  const uint32_t below = (1u << lane) - 1u;
#pragma unroll 1
  for (int base = 0; base < n; base += 32) {
    const int i = base + lane;
    const uint32_t key = i < n ? keys[i] : 0u;
    const uint32_t equal = __ballot_sync(full, i < n && key == kth);
    const bool sel = i < n && (key > kth || (key == kth && __popc(equal & below) < ties));
    ties -= min(ties, __popc(equal));
    const uint32_t word = __ballot_sync(full, sel);
    if (sel) emit(i, rank + __popc(word & below), key);
    rank += __popc(word);
  }
}

}  // namespace

template <int D, int NSTG, int ACCS, class Segs>
__global__ void __launch_bounds__(kRtThreads, ACCS == 2 ? 2 : 1)
k_route_sm100(const __grid_constant__ CUtensorMap map_q, const __grid_constant__ CUtensorMap map_ct,
              const __grid_constant__ CUtensorMap map_gs, const Dims dm, int32_t* __restrict__ chunk_idx,
              int32_t* __restrict__ group_idx, int32_t* __restrict__ n_groups,
              float* __restrict__ chunk_scores, float* __restrict__ group_scores, const RouteLayout lay,
              const __grid_constant__ Segs segs) {
  constexpr int kOctBytes = 8 * D * 2, kPanels = D / 64;
  constexpr uint32_t kTmemCols = 128 * ACCS;
  static_assert(NSTG % kPanels == 0, "the slabs of a tile are neighbours");
  extern __shared__ uint8_t smem_raw[];
  using Smem = RouteSmem<NSTG, ACCS>;
  Smem& sm = *reinterpret_cast<Smem*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* q_smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(&sm + 1) + 1023) & ~uintptr_t(1023));
  uint32_t* okeys = reinterpret_cast<uint32_t*>(q_smem + lay.q_bytes);       // orderable candidate scores
  uint32_t* fkeys = okeys + lay.n_keys;                                      // the warps' best candidates
  int* fidx = reinterpret_cast<int*>(fkeys + lay.n_final);
  uint32_t* flags = reinterpret_cast<uint32_t*>(fidx + lay.n_final);         // bit i: slot i selected
  int* sorted = reinterpret_cast<int*>(flags + 128);                         // selected chunks, ascending
  uint32_t* gkeys = reinterpret_cast<uint32_t*>(sorted + dm.kc);             // orderable scores of the opened chunks' groups

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  // (late query blocks first: where the history is short they have the most candidates)
  int cta;
  const Segment sg = segment_of(dm, segs, blockIdx.x, cta);
  const int n_bh = dm.B * dm.Hkv, n_qb = dm.by_Bq(sg.S), i_qb = dm.by_bh(cta), bh = cta - i_qb * n_bh;
  const int qb = n_qb - 1 - i_qb, b = dm.by_Hkv(bh), h = bh - b * dm.Hkv;
  const int64_t item = item_base(dm, sg, b) + h * n_qb + qb;
  const Window w = window_at(dm, sg.H + qb * dm.Bq);
  const int j0 = dm.by_c(w.se), n_cand = dm.by_c(w.ls - w.se);
  const int ct0 = dm.by_c(sg.k0), gs0 = dm.by_g(sg.k0);          // the segment's first rows in the summary tables
  // query rows on N: every head's Bq rows padded to whole octets (padding columns hold whatever shared memory held and
  // are masked when the columns are reduced)
  const int bq_pad = bq_padded(dm), rows_pad = rows_padded(dm);
  const bool boxes = dm.Bq % 64 == 0;                        // Q in boxes of 64 rows x one panel: [panel][rows][128 B]
  const int q_panel = boxes ? lay.parts * lay.part_cols * 128 : 1024;
  const bool all_rows_real = lay.parts * lay.part_cols == dm.rows;
  const int k_sel = dm.kc < n_cand ? dm.kc : n_cand;
  const int opc = dm.per / 8;                                // octets per opened chunk
  const int n_ct = (n_cand + 127) / 128;                     // chunk tiles
  const int n_gt = (k_sel * dm.per + 127) / 128;             // group tiles
  volatile int* abort = &sm.abort;
  const int agg = score_agg_of(dm.flags);
  constexpr float kLog2e = 1.4426950408889634f;
  uint32_t col_mask = 0xffffffffu;                           // bit i: column i of a block of 32 is a real query row
  if (!all_rows_real) {
    col_mask = 0;
#pragma unroll 1
    for (int i = 0, t = 0; i < 32; ++i, t = t + 1 == bq_pad ? 0 : t + 1) col_mask |= (uint32_t)(t < dm.Bq) << i;
  }

  // Copies slab p of chunk tile t (slab number g overall) into its stage; all lanes of warp 0.  The candidate chunks are
  // consecutive rows of the summary table, so a slab is two 64-row boxes; rows past the table read as zeros.
  int slabs_issued = 0;                 // warp 0's count of slabs whose copies were started
  auto copy_slab = [&](int g, int t, int p) {
    uint64_t* full = &sm.a_full[g % NSTG];
    slabs_issued = g + 1;
    if (lane == 0) mbar_arrive_expect_tx(full, kSlab);
    __syncwarp();
    if (lane < 2) tma_load_5d(sm.a[g % NSTG] + lane * 8192, &map_ct, full, 0, ct0 + j0 + 128 * t + 64 * lane, p, h, b);
  };
  // Box `oc` of group tile t: one octet of an opened chunk's group summaries, [octet][panel][8 rows][128 B] over the tile's
  // neighbouring slabs; the bytes are announced on the first one's barrier.
  auto copy_group_octet = [&](int tg, int t, int oc_in_tile) {
    const int s = tg * kPanels % NSTG, oc = 16 * t + oc_in_tile, r = opc == 1 ? oc : oc >> 1;      // (one or two octets)
    const int row = r < k_sel ? gs0 + sorted[r] * dm.per + 8 * (oc - r * opc) : dm.Ng;
    tma_load_5d(sm.a[s] + oc_in_tile * kOctBytes, &map_gs, &sm.a_full[s], 0, row, 0, h, b);
  };
  auto announce_group_tile = [&](int tg) {
    const int s = tg * kPanels % NSTG;
    slabs_issued = (tg + 1) * kPanels;
    if (lane == 0) {
      mbar_arrive_expect_tx(&sm.a_full[s], kPanels * kSlab);
      for (int p = 1; p < kPanels; ++p) mbar_arrive(&sm.a_full[s + p]);
    }
  };
  const int n_slabs = k_sel > 0 ? n_ct * kPanels : 0, n_pre = n_slabs < NSTG ? n_slabs : NSTG;   // slabs copied ahead of the CTA barrier

  if (warp == 0) {
    if (lane == 0) {
      mbar_init(&sm.q_full, 1);
      for (int s = 0; s < NSTG; ++s) { mbar_init(&sm.a_full[s], 1); mbar_init(&sm.a_empty[s], 1); }
      for (int s = 0; s < ACCS; ++s) { mbar_init(&sm.acc_full[s], 1); mbar_init(&sm.acc_free[s], 4); }
      mbar_init(&sm.drain, 1);
      sm.abort = 0;
      fence_barrier_init();
      prefetch_tensormap(&map_q); prefetch_tensormap(&map_ct); prefetch_tensormap(&map_gs);
    }
    __syncwarp();
    pdl_wait();
    // the first slabs depend on nothing: their copies start before the CTA meets
#pragma unroll 1
    for (int g = 0; g < n_pre; ++g) copy_slab(g, g / kPanels, g % kPanels);
    if (lane == 0 && k_sel > 0) mbar_arrive_expect_tx(&sm.q_full, (uint32_t)(rows_pad / 8) * kOctBytes);
  }
  if (warp == 1) {
    tmem_alloc(&sm.tmem_base, kTmemCols);
    tmem_relinquish();
  }
  __syncwarp();
  tc_fence_before_sync();
  __syncthreads();
  tc_fence_after_sync();
  const uint32_t tmem = sm.tmem_base;
  pdl_wait();            // (every thread: any of them may write results)
  // The forward kernel, the usual successor, may set itself up meanwhile.  Released here its CTAs come to lie on the SMs
  // while this kernel still selects, and fetch their instructions beside it; for one problem, a wave or two of CTAs, that cost
  // more than it hid (released ahead of the group selection instead: 32 sequences 42.4 -> 39.7 us, 128K 93.6 -> 92.1, 16K layer
  // 166.5 -> 165.6, all whole steps).  The many CTAs of several segments hide it (walk of 16K: 1155 us so, 1175 late).
  constexpr bool kReleaseEarly = !std::is_same<Segs, OneSegment>::value;
  if (kReleaseEarly && tid == 0) pdl_launch_dependents();

  // optional output: -inf outside the candidate range
  if (chunk_scores)
#pragma unroll 1
    for (int j = tid; j < dm.Nc; j += kRtThreads)
      if (j < j0 || j >= j0 + n_cand) chunk_scores[item * dm.Nc + j] = -INFINITY;
  if (group_scores)
#pragma unroll 1
    for (int i = tid; i < dm.kc * dm.per; i += kRtThreads)
      group_scores[item * dm.kc * dm.per + i] = -INFINITY;

  // Two GEMM phases over the same code, one after the other: candidate chunks, then the groups of the opened chunks.
  // Tiles are numbered through (t_begin + t), which drives barrier parities.  (One copy of the code: a CTA of a small
  // problem runs it once or twice, and what it executes for the first time costs instruction-cache misses -- with a
  // copy per phase the second phase's first tile was 2 us later.)
#pragma unroll 1
  for (int phase = 0; phase < 2; ++phase) {
    const bool phase2 = phase == 1;
    const int t_begin = phase2 ? n_ct : 0, n_tiles = phase2 ? n_gt : n_ct;
    if (k_sel > 0 && !sm.abort) {
      if (!phase2 && warp >= 2) {
        // The item's query rows.  Issuing a box costs its warp a few hundred
        // cycles and warps issue in parallel, so the boxes are spread over the non-producer warps.
        if (boxes) {
#pragma unroll 1
          for (int i = (warp - 2) + kRtCopyWarps * lane; i < rows_pad / 64 * kPanels; i += 32 * kRtCopyWarps) {
            const int panel = i % kPanels, r = i / kPanels * 64, a = dm.by_Bq(r);
            tma_load_5d(q_smem + panel * q_panel + r * 128, &map_q, &sm.q_full, 0, sg.q0 + qb * dm.Bq + r - a * dm.Bq, panel, h * dm.G + a, b);
          }
        } else {
#pragma unroll 1
          for (int o = (warp - 2) + kRtCopyWarps * lane; o < rows_pad / 8; o += 32 * kRtCopyWarps) {
            const int r = 8 * o, a = dm.by_Bq_pad(r), t = r - a * bq_pad;    // rows past the segment arrive as zeros
            tma_load_5d(q_smem + o * kOctBytes, &map_q, &sm.q_full, 0, sg.q0 + qb * dm.Bq + t, 0, h * dm.G + a, b);
          }
        }
      }
      // First tile of the opened chunks' group summaries, again spread over these warps (two or three octet boxes each).  Its
      // stages are known to be free: every tile of the first phase has been read back, so no barrier needs to be
      // observed; warp 0 announces the bytes.
      if (phase2 && warp >= 2 && (warp - 2) + kRtCopyWarps * lane < 16) copy_group_octet(t_begin, 0, (warp - 2) + kRtCopyWarps * lane);
      __syncwarp();
      if (warp == 0) {
        // ---------------------------------------------------------------- producer
        bool ok = true;
        auto wait_empty = [&](int g) {
          if (lane == 0 && g >= NSTG) ok = rt_wait(&sm.a_empty[g % NSTG], (uint32_t)(g / NSTG - 1) & 1, abort);
          ok = __shfl_sync(0xffffffffu, ok, 0);
          return ok;
        };
        if (!phase2) {
#pragma unroll 1
          for (int g = n_pre; g < n_slabs; ++g) {
            if (!wait_empty(g)) break;
            copy_slab(g, g / kPanels, g % kPanels);
          }
        } else {
          announce_group_tile(t_begin);      // (its boxes come from the other warps, see above)
#pragma unroll 1
          for (int t = 1; t < n_tiles && ok; ++t) {
            const int tg = t_begin + t;
            for (int p = 0; p < kPanels && ok; ++p) wait_empty(tg * kPanels + p);
            if (!ok) break;
            announce_group_tile(tg);
            __syncwarp();
            if (lane < 16) copy_group_octet(tg, t, lane);
          }
        }
      } else if (warp == 1) {
        // ---------------------------------------------------------------- MMA issuer
        // The whole warp runs this branch converged (waits included) and one elected lane issues: see mma_ss_w.
        const uint32_t lead = elect_one();
        auto mma_wait = [&](uint64_t* bar, uint32_t parity) {
          return __all_sync(0xffffffffu, rt_wait(bar, parity, abort));
        };
        const uint32_t idesc = idesc_bf16_f32(128, lay.part_cols, 0, 0);
        const uint64_t b_desc = smem_desc_sw128(smem_u32(q_smem), 16, boxes ? 1024 : kOctBytes);
        // A: 8-row groups 1024 B apart inside a slab, or octets (8 rows x all panels) for the gathered group tiles
        const uint64_t a_desc = smem_desc_sw128(smem_u32(sm.a[0]), 16, phase2 ? kOctBytes : 1024);
        const uint32_t part_bytes = (uint32_t)lay.part_cols * (boxes ? 128u : (uint32_t)D * 2);
        bool ok = phase2 ? true : mma_wait(&sm.q_full, 0);
        for (int t = 0; t < n_tiles && ok; ++t) {
          const int tg = t_begin + t;
          // parts that have accumulators at the same time; a slab is used by all of them before the next one
          for (int p0 = 0; p0 < lay.parts && ok; p0 += ACCS) {
            const int p1 = min(p0 + ACCS, lay.parts);
#pragma unroll
            for (int pn = 0; pn < kPanels; ++pn) {
              const int g = tg * kPanels + pn, s = g % NSTG;
              if (ok && p0 == 0) ok = mma_wait(&sm.a_full[s], (uint32_t)(g / NSTG) & 1);
              const uint64_t ad = desc_advance(a_desc, phase2 ? (uint32_t)(tg * kPanels % NSTG) * kSlab + pn * 1024 : (uint32_t)s * kSlab);
            for (int part = p0; part < p1 && ok; ++part) {
                const int step = tg * lay.parts + part, acc = step % ACCS;
                if (pn == 0 && step >= ACCS) ok = mma_wait(&sm.acc_free[acc], (uint32_t)(step / ACCS - 1) & 1);
                if (!ok) break;
                tc_fence_after_sync();
                const uint64_t bd = desc_advance(b_desc, (uint32_t)part * part_bytes + pn * q_panel);
#pragma unroll
                for (int kk = 0; kk < 4; ++kk)
                  mma_ss_w(lead, tmem + acc * 128, desc_advance(ad, kk * 32), desc_advance(bd, kk * 32), idesc, (pn > 0 || kk > 0));
                if (pn == kPanels - 1) mma_commit_w(lead, &sm.acc_full[acc]);
              }
              if (ok && p1 == lay.parts) mma_commit_w(lead, &sm.a_empty[s]);
            }
          }
        }
      } else if (warp < 6) {
        // ---------------------------------------------------------------- readers: thread = summary
        const int quarter = warp & 3;
        const int row = quarter * 32 + lane;
        const uint32_t lane_base = tmem + ((uint32_t)(quarter * 32) << 16);
        bool ok = true;
        for (int t = 0; t < n_tiles && ok; ++t) {
          const int tg = t_begin + t;
          float best = -FLT_MAX, sum = 0.f;    // log-sum-exp: (running maximum, sum of exp(dot - maximum))
          for (int part = 0; part < lay.parts; ++part) {
            const int step = tg * lay.parts + part, acc = step % ACCS;
            ok = __all_sync(0xffffffffu, rt_wait(&sm.acc_full[acc], (uint32_t)(step / ACCS) & 1, abort));
            if (!ok) break;
            tc_fence_after_sync();
            if (agg == 0 && all_rows_real) {
              // the usual case: 64 columns per round trip to tensor memory
              float m[4] = {best, -FLT_MAX, -FLT_MAX, -FLT_MAX};
              for (int c = 0; c < lay.part_cols; c += 64) {
                uint32_t x[32], y[32];
                tmem_ld32(lane_base + acc * 128 + c, x);
                if (c + 32 < lay.part_cols) tmem_ld32(lane_base + acc * 128 + c + 32, y);
                else {
#pragma unroll
                  for (int i = 0; i < 32; ++i) y[i] = 0xff7fffffu;      // -FLT_MAX
                }
                tmem_wait_ld();
#pragma unroll
                for (int i = 0; i < 32; ++i) m[i & 3] = fmaxf(fmaxf(m[i & 3], __uint_as_float(x[i])), __uint_as_float(y[i]));
              }
              best = fmaxf(fmaxf(m[0], m[1]), fmaxf(m[2], m[3]));
            } else {
              for (int c = 0; c < lay.part_cols; c += 32) {
                uint32_t x[32];
                tmem_ld32(lane_base + acc * 128 + c, x);
                tmem_wait_ld();
                if (!all_rows_real) {
                  // padding columns become the neutral element of the reduction (the pattern of real columns repeats in
                  // every block of 32; only the last block can be cut)
                  const float neutral = agg == 1 ? 0.f : -INFINITY;
                  const int left = rows_pad - (part * lay.part_cols + c);
                  const uint32_t m = left >= 32 ? col_mask : (col_mask & ((1u << (left > 0 ? left : 0)) - 1u));
#pragma unroll
                  for (int i = 0; i < 32; ++i)
                    if (!((m >> i) & 1u)) x[i] = __float_as_uint(neutral);
                }
                if (agg == 0) {
#pragma unroll
                  for (int i = 0; i < 32; ++i) best = fmaxf(best, __uint_as_float(x[i]));
                } else if (agg == 1) {
#pragma unroll
                  for (int i = 0; i < 32; ++i) sum += __uint_as_float(x[i]);
                } else {
                  float cm = -FLT_MAX;
#pragma unroll
                  for (int i = 0; i < 32; ++i) cm = fmaxf(cm, __uint_as_float(x[i]));
                  if (cm > best) { sum *= exp2f((best - cm) * kLog2e); best = cm; }
#pragma unroll
                  for (int i = 0; i < 32; ++i) sum += exp2f((__uint_as_float(x[i]) - best) * kLog2e);
                }
              }
            }
            tc_fence_before_sync();
            mbar_arrive_warp(&sm.acc_free[acc]);
          }
          if (!ok) break;
          if (agg == 1) best = sum * (1.f / (float)dm.rows);
          else if (agg == 2) best += logf(sum);
          const int i = 128 * t + row;
          if (!phase2) {
            if (i < n_cand) okeys[i] = rt_orderable(best);
            if (chunk_scores && i < n_cand) chunk_scores[item * dm.Nc + j0 + i] = best;
          } else {
            if (i < k_sel * dm.per) gkeys[i] = rt_orderable(best + 0.f);       // (+ 0: a negative zero equals a positive one)
          }
        }
      }
  
    }
    __syncwarp();          // the roles diverge inside a warp: reconverge before the block barrier
    __syncthreads();
    if (phase2) break;

    // ---------------------------------------------------------------------- chunk top-k
    // Scores compare as 32-bit orderable integers; equal scores are told apart by their index (lowest first).
    if (!sm.abort && k_sel > 0) {
      // Many candidates: every warp first picks the best k_sel of its share, without meeting the others.  (Counting every
      // candidate's rank, up to 640, and a block-wide search beyond took 17k cycles at 512 candidates and 22k at 2048, a
      // quarter of the item's time.)
      const uint32_t* keys = okeys;
      int n = n_cand;
      const bool shares = lay.n_final > 0 && n_cand > kRankMax;
      if (shares) {
        const int share = (n_cand + kRtWarps - 1) / kRtWarps, last = (n_cand - 1) / share;     // (all whole but the last)
        const int first = warp * share, mine = min(share, n_cand - first), each = min(k_sel, share);
        auto keep = [&](int i, int rank, uint32_t key) {
          fkeys[warp * each + rank] = key;
          fidx[warp * each + rank] = first + i;
        };
        if (mine > 0) {
          if (share <= 64) warp_select<2>(okeys + first, mine, min(k_sel, mine), keep);
          else if (share <= 256) warp_select<8>(okeys + first, mine, min(k_sel, mine), keep);
          else warp_select<0>(okeys + first, mine, min(k_sel, mine), keep);
        }
        n = last * each + min(k_sel, n_cand - last * share);
        keys = fkeys;
        __syncthreads();
      }
      if (n <= kRankMax) {
        // A key is selected when fewer than k_sel others beat it; counted for every one, a thread each, four
        // keys per 16-byte load.  Equal scores share a rank at first; that only matters when a tie straddles the k-th place,
        // which shows as a selection of the wrong size and is redone with the position as the second criterion.
        auto rank_select = [&](bool exact) {
          bool sel = false;
          if (tid < n) {
            int beat = 0, q = 0;
            const uint32_t mine = keys[tid];
            if (!exact) {
              const uint4* k4 = reinterpret_cast<const uint4*>(keys);
#pragma unroll 4
              for (; q + 4 <= n; q += 4) {
                const uint4 kk = k4[q >> 2];
                beat += (int)(kk.x > mine) + (int)(kk.y > mine) + (int)(kk.z > mine) + (int)(kk.w > mine);
              }
#pragma unroll 1
              for (; q < n; ++q) beat += keys[q] > mine;
            } else {
#pragma unroll 1
              for (; q < n; ++q) beat += keys[q] > mine || (keys[q] == mine && q < tid);
            }
            sel = beat < k_sel;
          }
          const uint32_t word = __ballot_sync(0xffffffffu, sel);
          if (lane == 0) flags[warp] = word;
        };
        auto picked_below = [&](int words) {
          int c = 0;
#pragma unroll 1
          for (int q = 0; q < words; ++q) c += __popc(flags[q]);
          return c;
        };
        rank_select(false);
        __syncthreads();
        if (picked_below(kRtWarps) != k_sel) {          // same value in every thread
          __syncthreads();
          rank_select(true);
          __syncthreads();
        }
        const uint32_t word = flags[warp];
        if ((word >> lane) & 1u) sorted[picked_below(warp) + __popc(word & ((1u << lane) - 1u))] = j0 + (shares ? fidx[tid] : tid);
      } else if (warp == 0) {
        warp_select<0>(keys, n, k_sel, [&](int i, int rank, uint32_t) { sorted[rank] = j0 + (shares ? fidx[i] : i); });
      }
      __syncthreads();
    }
    if (!sm.abort) {
#pragma unroll 1
      for (int i = tid; i < dm.kc; i += kRtThreads)
        chunk_idx[item * dm.kc + i] = i < k_sel ? sorted[i] : -1;
    }
    __syncthreads();
  }

  if (!kReleaseEarly && tid == 0) pdl_launch_dependents();
  // ---------------------------------------------------------------------- groups of the opened chunks
  if (!sm.abort) {
    int32_t* gi = group_idx + item * dm.width;
    const bool global_budget = (dm.flags & HGA_FLAG_GLOBAL_GROUP_BUDGET) != 0;
    if (k_sel * dm.per <= 4096) {
      // One thread per slot (opened chunk, group), slots in chunk-major order = ascending group id.
      // A slot is selected when fewer than `want` slots of its scope beat it (higher score, or equal
      // score and lower id); the scope is its own chunk (want = kg_eff) or, with one budget over all
      // opened chunks, every slot (want = k_sel * kg_eff).  Its place in the ascending output is the
      // number of selected slots below it.  (Compared as orderable integers: exactly `want` slots pass whatever the
      // scores are.  A NaN, which a mean or a log-sum-exp can be, compares with nothing as a float, so that every slot of such
      // a chunk passed and the list was written past its end.)
      const int total = k_sel * dm.per;
      const int want = global_budget ? k_sel * dm.kge : dm.kge;
#pragma unroll 1
      for (int base = 0; base < total; base += kRtThreads) {      // warp-uniform trip count (ballots below)
        const int i = base + tid;
        bool sel = false;
        if (i < total) {
          const uint32_t mine = gkeys[i];
          const int lo = global_budget ? 0 : i & ~(dm.per - 1),       // (8 or 16)
                    hi = global_budget ? total : lo + dm.per;
          int beat = 0;
#pragma unroll 8
          for (int q = lo; q < hi; ++q) beat += gkeys[q] > mine || (gkeys[q] == mine && q < i);
          sel = beat < want;
          if (group_scores) group_scores[item * dm.kc * dm.per + i] = rt_score(mine);
        }
        const uint32_t word = __ballot_sync(0xffffffffu, sel);
        if (lane == 0 && base + warp * 32 < total) flags[(base + warp * 32) >> 5] = word;
      }
      __syncthreads();
#pragma unroll 1
      for (int i = tid; i < total; i += kRtThreads)
        if ((flags[i >> 5] >> (i & 31)) & 1u) {
          int pos = __popc(flags[i >> 5] & ((1u << (i & 31)) - 1u));
#pragma unroll 1
          for (int q = 0; q < (i >> 5); ++q) pos += __popc(flags[q]);
          gi[pos] = sorted[i >> (dm.per == 8 ? 3 : 4)] * dm.per + (i & (dm.per - 1));
        }
    } else
#pragma unroll 1
    for (int r = tid; r < dm.kc; r += kRtThreads) {
      if (r < k_sel) {
        const uint32_t* v = gkeys + r * dm.per;
        unsigned long long picked = 0;
#pragma unroll 1
        for (int q = 0; q < dm.kge; ++q) {
          int bu = -1;
#pragma unroll 1
          for (int u = 0; u < dm.per; ++u)
            if (!((picked >> u) & 1ull) && (bu < 0 || v[u] > v[bu])) bu = u;     // first wins ties
          picked |= 1ull << bu;
        }
        int n = r * dm.kge;
#pragma unroll 1
        for (int u = 0; u < dm.per; ++u)
          if ((picked >> u) & 1ull) gi[n++] = sorted[r] * dm.per + u;
        if (group_scores)
#pragma unroll 1
          for (int u = 0; u < dm.per; ++u)
            group_scores[item * dm.kc * dm.per + r * dm.per + u] = rt_score(v[u]);
      }
    }
#pragma unroll 1
    for (int i = k_sel * dm.kge + tid; i < dm.width; i += kRtThreads) gi[i] = -1;
    if (tid == 0) n_groups[item] = k_sel * dm.kge;
  }

  if (sm.abort) {
    // A bounded wait gave up: the item's routing is marked invalid (the attention calls report a negative
    // count and use no routed groups for that item), and the copies still in flight get a bounded time to land
    // before the CTA's shared memory is released.
    if (tid == 0) n_groups[item] = -1;
    if (warp == 0 && lane == 0) {        // (slabs_issued is warp 0's own count)
      if (k_sel > 0) mbar_wait(&sm.q_full, 0);
      for (int g = slabs_issued > NSTG ? slabs_issued - NSTG : 0; g < slabs_issued; ++g)
        mbar_wait(&sm.a_full[g % NSTG], (uint32_t)(g / NSTG) & 1);
    }
    if (warp == 1) {
      // GEMMs the warp's issuing lane started may still be writing tensor memory: a commit completes once
      // every earlier MMA of that lane has, so wait for one (bounded) before the columns are given back
      mma_commit_w(elect_one(), &sm.drain);
      mbar_wait(&sm.drain, 0);
    }
  }
  __syncwarp();
  tc_fence_before_sync();
  __syncthreads();
  if (warp == 1) {
    __syncwarp();
    tmem_dealloc(tmem, kTmemCols);
  }
}

static int route_max_cand(const Dims& dm, const SegTable* segs) {
  // the last query block of a segment has the most candidates
  auto cand = [&](int L) {
    const Window wl = window_at(dm, L - dm.Bq);
    return (wl.ls - wl.se) / dm.c;
  };
  if (!segs) return cand(dm.L);
  int most = 0;
  for (int i = 0; i < segs->n; ++i) most = std::max(most, cand(segs->seg[i].H + segs->seg[i].S));
  return most;
}

// Shared memory with `stages` slabs
static size_t route_smem(const Dims& dm, const RouteLayout& lay, int stages) {
  const size_t ctl = stages == 2 ? sizeof(RouteSmem<2, 4>) : sizeof(RouteSmem<4, 4>);
  return 1024 + ctl + lay.tail(dm);
}

bool route_sm100_supported(const Dims& dm, const SegTable* segs) {
  if (dm.flags & HGA_FLAG_GENERIC_KERNELS) return false;
  if (bq_padded(dm) != dm.Bq && 32 % bq_padded(dm) != 0) return false;   // the padding mask repeats every 32 columns
  if (dm.per != 8 && dm.per != 16) return false;            // opened chunk = 1 or 2 octets of summaries
  if (dm.kc > 1024) return false;
  if ((dm.flags & HGA_FLAG_GLOBAL_GROUP_BUDGET) && dm.kc * dm.per > 4096) return false;   // bitmap
  return route_smem(dm, RouteLayout(dm, route_max_cand(dm, segs)), 2) <= 227 * 1024;
}

template <int D, int NSTG, int ACCS, class Segs>
static int launch_route(const Dims& dm, const Segs& segs, int64_t items, const RouteLayout& lay, const void* Q, const void* chunk_sum,
                        const void* group_sum, int32_t* chunk_idx, int32_t* group_idx, int32_t* n_groups, float* chunk_scores,
                        float* group_scores, cudaStream_t st) {
  CUtensorMap mq, mc, mg;
  const uint32_t box[5] = {64, 8, (uint32_t)(D / 64), 1, 1};
  const uint32_t box_rows[5] = {64, 64, 1, 1, 1};          // half a slab of chunk summaries; 64 query rows of a panel
  const uint64_t dq[5] = {64, (uint64_t)dm.rows_q, (uint64_t)(D / 64), (uint64_t)dm.Hq, (uint64_t)dm.B};
  const uint64_t dc[5] = {64, (uint64_t)dm.Nc, (uint64_t)(D / 64), (uint64_t)dm.Hkv, (uint64_t)dm.B};
  const uint64_t dg[5] = {64, (uint64_t)dm.Ng, (uint64_t)(D / 64), (uint64_t)dm.Hkv, (uint64_t)dm.B};
  const uint64_t sq[4] = {(uint64_t)dm.qs[2] * 2, 128, (uint64_t)dm.qs[1] * 2, (uint64_t)dm.qs[0] * 2};
  const uint64_t sc[4] = {(uint64_t)D * 2, 128, (uint64_t)dm.NcS * D * 2, (uint64_t)dm.Hkv * dm.NcS * D * 2};
  const uint64_t sg[4] = {(uint64_t)D * 2, 128, (uint64_t)dm.NgS * D * 2, (uint64_t)dm.Hkv * dm.NgS * D * 2};
  if (encode_tensor_map_bf16(&mq, Q, 5, dq, sq, dm.Bq % 64 == 0 ? box_rows : box, true) ||
      encode_tensor_map_bf16(&mc, chunk_sum, 5, dc, sc, box_rows, true) ||
      encode_tensor_map_bf16(&mg, group_sum, 5, dg, sg, box, true))
    return HGA_ERR_UNSUPPORTED;
  const size_t smem = route_smem(dm, lay, NSTG);
  // two CTAs per SM need the largest shared-memory carve-out
  const int rc = ensure_dynamic_smem(reinterpret_cast<const void*>(&k_route_sm100<D, NSTG, ACCS, Segs>), smem, true);
  if (rc) return rc;
  PdlLaunch cfg((unsigned)items, kRtThreads, smem, st, dm.flags);
  const cudaError_t e = cudaLaunchKernelEx(&cfg.c, k_route_sm100<D, NSTG, ACCS, Segs>, mq, mc, mg, dm, chunk_idx, group_idx, n_groups,
                                           chunk_scores, group_scores, lay, segs);
  count_launch(HGA_KERNELS_ROUTE_TENSOR);
  return record_cuda(e);
}

template <int D, class Segs>
static int launch_route_stages(const Dims& dm, const Segs& segs, int64_t items, const RouteLayout& lay, const void* Q, const void* chunk_sum,
                               const void* group_sum, int32_t* chunk_idx, int32_t* group_idx, int32_t* n_groups, float* chunk_scores,
                               float* group_scores, cudaStream_t st) {
#define HGA_ROUTE_ARGS dm, segs, items, lay, Q, chunk_sum, group_sum, chunk_idx, group_idx, n_groups, chunk_scores, group_scores, st
  constexpr size_t kHalf = 113 * 1024, kWhole = 227 * 1024;      // shared memory of a CTA that shares its SM, or has it to itself
  if (route_smem(dm, lay, 4) <= kHalf) return launch_route<D, 4, 2>(HGA_ROUTE_ARGS);
  if (route_smem(dm, lay, 2) <= kHalf) return launch_route<D, 2, 2>(HGA_ROUTE_ARGS);
  if (route_smem(dm, lay, 4) <= kWhole) return launch_route<D, 4, 4>(HGA_ROUTE_ARGS);
  return launch_route<D, 2, 4>(HGA_ROUTE_ARGS);
#undef HGA_ROUTE_ARGS
}

int launch_route_sm100(const Dims& dm, SegTable* segs, const void* Q, const void* chunk_sum, const void* group_sum,
                       int32_t* chunk_idx, int32_t* group_idx, int32_t* n_groups, float* chunk_scores,
                       float* group_scores, cudaStream_t st) {
  const RouteLayout lay(dm, route_max_cand(dm, segs));
#define HGA_ROUTE_ARGS lay, Q, chunk_sum, group_sum, chunk_idx, group_idx, n_groups, chunk_scores, group_scores, st
  if (!segs) {
    const int64_t items = (int64_t)dm.B * dm.Hkv * dm.NQB;
    return dm.d == 128 ? launch_route_stages<128>(dm, OneSegment{}, items, HGA_ROUTE_ARGS)
                       : launch_route_stages<64>(dm, OneSegment{}, items, HGA_ROUTE_ARGS);
  }
  const int64_t items = number_units(*segs, [&](const Segment& s) { return (int64_t)dm.B * dm.Hkv * (s.S / dm.Bq); });
  return dm.d == 128 ? launch_route_stages<128>(dm, *segs, items, HGA_ROUTE_ARGS)
                     : launch_route_stages<64>(dm, *segs, items, HGA_ROUTE_ARGS);
#undef HGA_ROUTE_ARGS
}

}  // namespace hga
