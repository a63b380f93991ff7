// hga_attn_bwd for sm_100a (head_dim 128, items of whole 128-row M-tiles): backward of routed exact-token attention with the
// routing frozen (Section 2.1, last paragraph) and history K/V detached (Section 2.2).
//
// Unit of work: one 128-row M-tile of one item (b, kv head, query block), swept over the item's routed keys in PAIRS of
// 64-key tiles (128 keys, 16 octets of 8 consecutive tokens, one TMA box each for K and for V).  Per pair
//      S(u)  = Q K^T, dP(u) = dO V^T                 (N = 128: a tcgen05.mma with N = 64 runs at little more than half the rate)
//      phase 1 of the row threads: P = 2^(S*c - LSE*log2e), kept as packed bf16 in registers;
//      phase 2: dS = scale * P o (dP - delta), written as bf16 over the dP columns already read;
//      dQ += dS K                                    (A = dS from TMEM, B = the K stage, MN-major)
// Far keys (sink, selected groups) of the active segment also get dK and dV from here (those of the local window and the causal
// block come from k_attn_bwd_band_sm100, which precedes this kernel).  Their octets, eight to a pair, are in the first tiles of
// n_a pairs; P and dS of such a first tile go to shared memory as well:
//      dV^T = dO^T P, dK^T = Q^T dS                  (M = head_dim, N = 64 keys, K = 128 rows) over the S columns read by then,
// and four warps add the two to global memory straight from tensor memory.
//
// Persistent CTAs: a CTA takes over the next one of the grid that has not started (cluster launch control), and
// every role goes on to the next unit by itself, so that its list, Q, dO, K, V, delta and first GEMMs come while the
// last pairs of the one before are still at work.  With one CTA per unit 16k of its 35k cycles (16K layer, six pairs) were
// set-up, list, first copies, epilogue and the change of CTAs.
//
// Three 128-column TMEM regions rotate: S(u+1) is issued while the row threads still work on pair u, dP(u+1) goes into S(u)'s
// region as soon as they have read it, S(u+2) into that of dS(u) behind dQ(u).  After a pair with dK/dV, whose S region these
// take, the next dP follows dQ(u) in the region of dS(u), and the S after that waits until dK has been read.
//
// Code size: the roles run side by side, and what they execute per pair and unit has to stay in the instruction caches.  The same
// kernel with everything in line (138 KB of code, now 62) was slower than one CTA per unit: 16K layer (whole step) 161 us with
// one CTA per unit, 185 persistent with 138 KB, 155 with 79, 147 with 62; 3 KB of unrolling more cost 2.5 us.  Hence the waits
// by call, one copy of the code for S and dP and rolled loops wherever a role has time.
//
// What bounds it: the row threads, ~2.7k cycles per pair (1.0k of exponentials; tensor-memory loads and barrier hand-offs), a unit's
// first pair, which waits for dO (its buffer is free only behind the last pair's dP), and a pair with dK/dV, whose place costs the K
// ring its third stage.  Whole steps, one CTA per unit -> persistent: 16K layer 161 -> 147 us, walk of 16K 1147 -> 1076; 2K layer,
// nearly all of whose pairs have dK/dV, 149 -> 139; twelve packed sequences 369 -> 334.  The 2K layer's additions (133 MB of
// fp32) are what it waits for.
//
// Warp roles (640 threads, 96 registers):
//   0, 3     K octets 0-7 / 8-15 of every pair (a box costs its issuing warp ~100 cycles)      16, 17   the same for V
//   1        issues S and dP              2    issues dQ, dV, dK (one warp issuing all took longer over it than the tensor pipe)
//   4-11     one thread per query row and tile of a pair
//   12-15    statistics (LSE, delta = rowsum(dO o O)) of the next unit, dK/dV reduction, dQ epilogue
//   18       planner: which unit is next, its routing list               19   Q and dO tiles
// TMEM (512 columns): dQ | three regions.  Shared memory: Q, dO (32 KB each), K ring of three 32 KB stages, V ring of two.  A
// pair with dK/dV takes two items of the K ring: K(u), then P | dS of its first tile.  (With P | dS in a V stage, and the next
// pairs' V tiles taking turns in the other one, the 2K layer, nearly all of whose pairs are such, took 9 us more.)
#include "hga_bwd_sm100.cuh"
#include "hga_common.cuh"
#include "hga_octets.cuh"
#include "hga_sm100.cuh"

#include <algorithm>

namespace hga {

using namespace sm100;

namespace {

constexpr int kBwdThreads = 640;
constexpr int kBwdD = 128;
constexpr int kOct = 8 * kBwdD * 2;             // bytes of one octet of K/V rows: [panel][8 rows][128 B]
constexpr int kStage = 16 * kOct;               // bytes of one stage: the octets of a pair
constexpr int kKStages = 3, kVStages = 2;
constexpr int kInfoReaders = 19;                // warps that read a unit's description (all but the planner)
constexpr int kMostRoutedTokens = 3327;         // wider items keep the CUDA-core kernel's precision (see launch_sweep)

struct Unit {
  int n_pairs;                                  // none: there is no further unit
  int a_begin, n_a;                             // pairs [a_begin, a_begin + n_a) also give dK/dV
  int n_act, n_hist, n_other;                   // octets that get it; far octets of the history; these and the local ones
  int vis;                                      // tokens of the latter that the block's first row sees
  int b, h;                                     // batch entry, kv head
  int head[2], token[2], pos[2];                // query head, token row in Q, O, dO and dQ, and position in the block at rows 0 and 64
  int k0, ls, se, ng, clean;                    // first row of the segment in K / V; see FarList
  int64_t list, lse[2];                         // first entry of its list; LSE of rows 0 and 64
  int64_t grad_row;                             // row of position 0 of its kv head in dK and dV (rows of 128 floats)
};

// Which octets pair u holds: a pair with_grads starts with up to eight that get dK/dV, everything else is filled up with the
// others in their order
struct Pairs {
  int a_begin, n_a, n_act, n_other;
  __device__ explicit Pairs(const Unit& un) : a_begin(un.a_begin), n_a(un.n_a), n_act(un.n_act), n_other(un.n_other) {}
  __device__ bool with_grads(int u) const { return (unsigned)(u - a_begin) < (unsigned)n_a; }
  // number of the pair's first octet among those that get dK/dV (a pair behind the last such: their number), and how many it holds
  __device__ int first_act(int u) const { return min(n_act, 8 * max(u - a_begin, 0)); }
  __device__ int acts(int u) const { return with_grads(u) ? min(8, n_act - 8 * (u - a_begin)) : 0; }
  // number among the others of the first of them in tile `tile` of the pair (behind the `acts` in the first one)
  __device__ int first_other(int u, int tile) const { return 16 * u - first_act(u) + (tile ? 8 - acts(u) : 0); }
};

// A stage of the K ring and the parity of its next "full": every role that has to do with the ring follows along
struct KStage {
  uint32_t at = 0, parity = 0;
  __device__ void next() { if (++at == kKStages) { at = 0; parity ^= 1; } }
};

struct BwdSmem {
  alignas(1024) uint8_t q[128 * kBwdD * 2];     // [panel][128 rows][128 B]
  alignas(1024) uint8_t dO[128 * kBwdD * 2];
  alignas(1024) uint8_t k[kKStages][kStage];    // K: [octet][panel][8 rows][128 B]; P | dS of a tile of 64 keys: [128 rows][128 B] each
  alignas(1024) uint8_t v[kVStages][kStage];    // V, like K
  float nlse[128], nds[128];                    // of the unit's rows: -LSE * log2(e), -delta * scale
  Unit unit[2];
  alignas(16) uint4 cancelled;                  // answer of the launch control
  uint64_t info_full[2], info_empty[2], plan, cancel_full;
  uint64_t q_full, q_empty, do_full, do_empty;
  // Ring items: full by copy (or, a place of P and dS, as soon as it is free), empty by the GEMMs that read them
  uint64_t k_full[kKStages], k_empty[kKStages], v_full[kVStages], v_empty[kVStages];
  // Per pair, alternately (every completion has to depend on its waiter having observed the one before on the same barrier:
  // S(u+1) and dP(u+1) are issued before the row threads' arrivals of pair u have been waited for)
  uint64_t s_full[2], dp_full[2], s_read[2], ds_full[2], step_done[2];
  uint64_t acc_full[2], acc_read[2];            // pairs with dK/dV, counted by themselves
  uint64_t lse_full, stat_full, stat_empty, dq_done, dq_free;
  uint64_t drain[2];
  uint32_t tmem_base;
  volatile int abort;
};
static_assert(sizeof(BwdSmem) + 1024 <= 227 * 1024, "one CTA per SM");

// Requests the next CTA of the grid that has not started instead of its launch; the answer (16 bytes) arrives on `bar`
__device__ __forceinline__ void request_next_cta(void* answer, uint64_t* bar) {
  asm volatile("clusterlaunchcontrol.try_cancel.async.shared::cta.mbarrier::complete_tx::bytes.b128 [%0], [%1];"
               ::"r"(smem_u32(answer)), "r"(smem_u32(bar)) : "memory");
}
// The CTA that the answer hands over, or -1
__device__ __forceinline__ int next_cta_of(const void* answer) {
  uint32_t given, x;
  asm volatile(
      "{\n\t.reg .b128 a;\n\t.reg .pred p;\n\t"
      "ld.shared.b128 a, [%2];\n\t"
      "clusterlaunchcontrol.query_cancel.is_canceled.pred.b128 p, a;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t"
      "mov.u32 %1, 0;\n\t"
      "@p clusterlaunchcontrol.query_cancel.get_first_ctaid::x.b32.b128 %1, a;\n\t}"
      : "=r"(given), "=r"(x)
      : "r"(smem_u32(answer))
      : "memory");
  return given ? (int)x : -1;
}

__device__ __forceinline__ void red_add(float* to, float x) {
  asm volatile("red.relaxed.gpu.global.add.f32 [%0], %1;" ::"l"(__cvta_generic_to_global(to)), "f"(x) : "memory");
}

// The units of a segment in launch order.  The first blocks see no routed key of the active segment: they come first, for the
// SMs that the band kernel leaves idle, where a dK/dV addition would wait for its end.  Then late blocks first: they have the
// most such keys, so the cheapest units are the ones that fill the last round.
__device__ __forceinline__ int block_in_order(const Dims& dm, int i, int n_qb) {
  const int lead = dm.by_Bq(dm.local + dm.c - 1) + 1;
  return i < lead ? i : n_qb - 1 - (i - lead);
}

}  // namespace

template <class Segs>
__global__ void __launch_bounds__(kBwdThreads, 1)
k_attn_bwd_sm100(const __grid_constant__ CUtensorMap map_q, const __grid_constant__ CUtensorMap map_do,
                 const __grid_constant__ CUtensorMap map_k, const __grid_constant__ CUtensorMap map_v,
                 const uint16_t* __restrict__ O, const float* __restrict__ LSE, const int32_t* __restrict__ group_idx,
                 const int32_t* __restrict__ n_groups, const Dims dm, uint16_t* __restrict__ dQ, float* __restrict__ dK,
                 float* __restrict__ dV, int32_t* status_word, const __grid_constant__ Segs segs) {
  constexpr int D = kBwdD;
  auto region = [](uint32_t r) -> uint32_t { return 128 + 128 * r; };       // dQ: columns 0 .. 127
  // regions of the next pair's S and dP from a pair's (see above): S goes into the third one
  auto next_regions = [](bool with_grads, uint32_t& s, uint32_t& p) {
    const uint32_t s0 = s;
    s = 3 - s - p;
    if (!with_grads) p = s0;
  };
  extern __shared__ uint8_t smem_raw[];
  BwdSmem& sm = *reinterpret_cast<BwdSmem*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  HGA_TRACE_DECL(512);
  volatile int* abort = &sm.abort;

  if (tid == 0) {
    for (int s = 0; s < 2; ++s) {
      mbar_init(&sm.info_full[s], 1); mbar_init(&sm.info_empty[s], kInfoReaders);
      mbar_init(&sm.s_full[s], 1); mbar_init(&sm.dp_full[s], 1); mbar_init(&sm.s_read[s], 8); mbar_init(&sm.ds_full[s], 8);
      mbar_init(&sm.step_done[s], 1); mbar_init(&sm.drain[s], 1);
      mbar_init(&sm.acc_full[s], 1); mbar_init(&sm.acc_read[s], 4);
    }
    mbar_init(&sm.plan, 1); mbar_init(&sm.cancel_full, 1);
    mbar_init(&sm.q_full, 1); mbar_init(&sm.do_full, 1);
    // S (dP) of the last pair and the dK (dV) GEMMs; of dO also the four statistics warps.  Both issuing warps arrive by commits
    // only, the second one for units without dK/dV too: a commit stands behind all GEMMs that its warp has issued, so it cannot
    // be counted for the unit before while that unit's dK and dV still read Q and dO, as a plain arrival could.
    mbar_init(&sm.q_empty, 2);
    mbar_init(&sm.do_empty, 6);
    for (int s = 0; s < kKStages; ++s) { mbar_init(&sm.k_full[s], 2); mbar_init(&sm.k_empty[s], 1); }
    for (int s = 0; s < kVStages; ++s) { mbar_init(&sm.v_full[s], 2); mbar_init(&sm.v_empty[s], 1); }
    mbar_init(&sm.lse_full, 4); mbar_init(&sm.stat_full, 4); mbar_init(&sm.stat_empty, 8);
    mbar_init(&sm.dq_done, 1); mbar_init(&sm.dq_free, 4);
    sm.abort = 0;
    fence_barrier_init();
  }
  if (warp == 1) {
    tmem_alloc(&sm.tmem_base, 512);
    tmem_relinquish();
    // the next kernel's launch may overlap this grid's tail (the conversion of bf16 outputs, the next step's summaries)
    if (lane == 0) pdl_launch_dependents();
  }
  __syncwarp();
  tc_fence_before_sync();
  __syncthreads();
  tc_fence_after_sync();
  const uint32_t tmem = sm.tmem_base;
  HGA_TRACE_POINT(1);

  bool ok = true;
  // all lanes poll (one lane and a shuffle took longer)
  auto wait = [&](uint64_t* bar, uint32_t parity, int line = __builtin_LINE()) {
    ok = __all_sync(0xffffffffu, bwd_wait_(bar, parity & 1, abort, HGA_WAIT_CODE(line)));
    return ok;
  };
  // ... out of line, for the roles that can spare the call (the row threads cannot: 1 us of the 16K layer)
  auto wait_by_call = [&](uint64_t* bar, uint32_t parity, int line = __builtin_LINE()) { return ok = wait_out_of_line(bar, parity, abort, line); };
  // Description of the CTA's n-th unit; done_with_info() once its fields have been read
  auto unit_info = [&](int n, int line = __builtin_LINE()) -> const Unit& { wait_by_call(&sm.info_full[n & 1], n >> 1, line); return sm.unit[n & 1]; };
  auto done_with_info = [&](int n) { mbar_arrive_warp(&sm.info_empty[n & 1]); };

  if (warp == 18) {
    // ------------------------------------------------------------------ planner
    int id = blockIdx.x;
    for (int n = 0; ok; ++n) {
      if (n >= 2 && !wait_by_call(&sm.info_empty[n & 1], (n >> 1) - 1)) break;
      Unit& un = sm.unit[n & 1];
      if (id < 0) {
        if (lane == 0) { un.n_pairs = 0; mbar_arrive(&sm.info_full[n & 1]); }
        break;
      }
      int cta;
      const Segment sg = segment_of(dm, segs, id, cta);
      const int n_mt = dm.rows / 128, n_bh = dm.B * dm.Hkv, n_qb = dm.by_Bq(sg.S);
      const int unit = dm.by_mt(cta), mt = cta - unit * n_mt, i = dm.by_bh(unit), bh = unit - i * n_bh;
      const int qb = block_in_order(dm, i, n_qb), b = dm.by_Hkv(bh), h = bh - b * dm.Hkv;
      const int64_t item = item_base(dm, sg, b) + h * n_qb + qb;
      const Window w = window_at(dm, sg.H + qb * dm.Bq);
      FarList far(dm, w, group_idx + item * dm.width);
      far.check(dm, n_groups + item, sg.H);       // (invalid entries are skipped as in the forward kernel, which reports them)
      if (lane == 0) {
        const int n_hist = min(far.first_active, far.n_far), n_act = far.n_far - n_hist, n_other = n_hist + (w.p0 + dm.Bq - w.ls) / 8;
        const int n_a = (n_act + 7) / 8, n_pairs = max(n_a, (n_act + n_other + 15) / 16);
        un.n_pairs = n_pairs;
        // (in the middle: the next unit's Q and dO are copied behind the last GEMM that reads these)
        un.a_begin = (n_pairs - n_a) / 2; un.n_a = n_a;
        un.n_act = n_act; un.n_hist = n_hist; un.n_other = n_other;
        un.vis = 8 * n_hist + w.p0 - w.ls + 1;
        un.b = b; un.h = h;
        // (Bq is a multiple of 64: 64 rows are of one head)
#pragma unroll 1
        for (int half = 0; half < 2; ++half) {
          const int r = mt * 128 + 64 * half, a = dm.by_Bq(r), t = r - a * dm.Bq;
          un.head[half] = h * dm.G + a;
          un.pos[half] = t;
          un.token[half] = sg.q0 + qb * dm.Bq + t;
          un.lse[half] = row_base(dm, sg, b) * dm.Hq + (int64_t)(h * dm.G + a) * sg.S + qb * dm.Bq + t;
        }
        un.k0 = sg.k0; un.ls = w.ls; un.se = w.se; un.ng = far.ng; un.clean = far.clean;
        un.list = item * dm.width;
        un.grad_row = row_base(dm, sg, b) * dm.Hkv + (int64_t)h * sg.S - sg.H;
        mbar_arrive(&sm.info_full[n & 1]);
      }
      __syncwarp();
      // the next one is asked for only when this one's last K pairs are being fetched: asked for earlier, it might wait here
      // while another SM has run out of work
      if (!wait_by_call(&sm.plan, n)) break;
      if (lane == 0) {
        fence_proxy_async_smem();                 // (the last answer has been read)
        mbar_arrive_expect_tx(&sm.cancel_full, 16);
        request_next_cta(&sm.cancelled, &sm.cancel_full);
      }
      __syncwarp();
      // (not cut short by the abort flag: the answer has to land before the CTA's shared memory is released)
      ok = __all_sync(0xffffffffu, mbar_wait(&sm.cancel_full, n & 1));
      id = ok ? next_cta_of(&sm.cancelled) : -1;
      __syncwarp();
    }
    if (!ok && lane == 0 && *abort == 0) *abort = 1;
  } else if (warp == 0 || warp == 3 || warp == 16 || warp == 17) {
    // ------------------------------------------------------------------ K and V tiles
    const bool is_v = warp >= 16;
    const int part = warp == 3 || warp == 17 ? 1 : 0;      // tile of a pair
    const CUtensorMap* map = is_v ? &map_v : &map_k;
    uint64_t *const full = is_v ? sm.v_full : sm.k_full, *const empty = is_v ? sm.v_empty : sm.k_empty;
    if (lane == 0) prefetch_tensormap(map);
    const int n_stages = is_v ? kVStages : kKStages;
    int st = 0;                                   // stage of the next ring item
    uint32_t used = 0, phase = 0;                 // per stage
    auto take_stage = [&]() {                     // waits until it is free
      const uint32_t bit = 1u << st;
      if (used & bit) { wait_by_call(&empty[st], phase >> st); phase ^= bit; }
      used |= bit;
      return ok;
    };
    auto next_stage = [&]() { st = st + 1 == n_stages ? 0 : st + 1; };
    for (int n = 0; ok; ++n) {
      const Unit& un = unit_info(n);
      const int n_pairs = ok ? un.n_pairs : 0;
      if (n_pairs == 0) break;
      const Pairs pairs(un);
      const int n_hist = un.n_hist, ls = un.ls, k0 = un.k0, h = un.h, b = un.b;
      FarList far(dm, Window{0, un.ls, un.se}, group_idx + un.list);
      far.ng = un.ng; far.n_far = un.n_hist + un.n_act; far.clean = un.clean;
      done_with_info(n);
      auto row_of = [&](int u) {                  // row of this lane's octet of pair u in K / V; none: out of range, zeros
        const int i = lane & 7, acts = part == 0 ? pairs.acts(u) : 0, o = pairs.first_other(u, part) + i - acts;
        if (i >= acts && o >= n_hist) return o < pairs.n_other ? k0 + ls + 8 * (o - n_hist) : dm.rows_k;
        return k0 + far.row(i < acts ? n_hist + pairs.first_act(u) + i : o);
      };
      // (looked up one pair ahead)
      for (int u = -1, row = 0; u < n_pairs; ++u) {
        const int next_row = u + 1 < n_pairs ? row_of(u + 1) : 0;
        if (u >= 0) {
          if (warp == 0 && lane == 0 && u == max(0, n_pairs - 3)) mbar_arrive(&sm.plan);
          if (!take_stage()) break;
          if (lane == 0) mbar_arrive_expect_tx(&full[st], 8 * kOct);
          __syncwarp();
          if (lane < 8) tma_load_5d((is_v ? sm.v[st] : sm.k[st]) + (8 * part + lane) * kOct, map, &full[st], 0, row, 0, h, b);
          HGA_TRACE_POINT(2);
          next_stage();
          if (!is_v && pairs.with_grads(u)) {     // the place of P and dS
            if (!take_stage()) break;
            mbar_arrive_warp(&full[st]);
            next_stage();
          }
        }
        row = next_row;
      }
    }
  } else if (warp == 19) {
    // ------------------------------------------------------------------ Q and dO tiles
    if (lane == 0) { prefetch_tensormap(&map_q); prefetch_tensormap(&map_do); }
    for (int n = 0; ok; ++n) {
      const Unit& un = unit_info(n);
      if (!ok || un.n_pairs == 0) break;
      // four boxes of 64 rows x one 64-element panel per tensor
      const int half = lane & 1, panel = (lane >> 1) & 1, row = un.token[half], head = un.head[half], b = un.b;
      done_with_info(n);
#pragma unroll 1
      for (int is_do = 0; is_do < 2; ++is_do) {
        uint64_t* full = is_do ? &sm.do_full : &sm.q_full;
        if (n > 0 && !wait_by_call(is_do ? &sm.do_empty : &sm.q_empty, n - 1)) break;
        if (lane == 0) mbar_arrive_expect_tx(full, 128 * D * 2);
        __syncwarp();
        if (lane < 4) tma_load_5d((is_do ? sm.dO : sm.q) + panel * 16384 + half * 8192, is_do ? &map_do : &map_q, full, 0, row, panel, head, b);
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------------ S and dP
    // The whole warp runs this branch converged (waits included) and one elected lane issues: see mma_ss_w.
    const uint32_t lead = elect_one();
    constexpr uint32_t idesc = idesc_bf16_f32(128, 128, 0, 0);             // rows x keys, both K-major
    // Descriptors are built once; inside the loops an MMA costs two integer adds.
    const uint64_t q_k = smem_desc_sw128(smem_u32(sm.q), 16, 1024), do_k = smem_desc_sw128(smem_u32(sm.dO), 16, 1024);
    const uint64_t k_k = smem_desc_sw128(smem_u32(sm.k[0]), 16, kOct), v_k = smem_desc_sw128(smem_u32(sm.v[0]), 16, kOct);
    auto issue = [&](uint32_t acc, uint64_t a, uint64_t b) {
#pragma unroll
      for (int kk = 0; kk < D / 16; ++kk)
        mma_ss_w(lead, acc, desc_advance(a, (kk >> 2) * 16384 + (kk & 3) * 32), desc_advance(b, (kk >> 2) * 1024 + (kk & 3) * 32), idesc, kk > 0);
    };
    uint32_t U = 0, vs = 0, vp = 0;               // pairs so far; V stage and its parity
    KStage k;
    uint32_t rs = 0, rp = 1;              // regions of the next S and of the dP with it
    uint32_t n_grads = 0;                         // pairs with dK/dV so far
    bool a1 = false, a2 = false;                  // whether the last pair, and the one before, were such
    for (int n = 0; ok; ++n) {
      const Unit& un = unit_info(n);
      const int n_pairs = ok ? un.n_pairs : 0;
      if (n_pairs == 0) break;
      const Pairs pairs(un);
      done_with_info(n);
      for (int u = 0; u < n_pairs; ++u, ++U) {
        // (one copy of the code for both)
#pragma unroll 1
        for (int dp = 0; dp < 2; ++dp) {
          // S: its region held dS of the pair before the last, or that pair's dV and dK.  dP: its region held S of the last pair,
          // or that pair's dS if its S region has gone to dV and dK
          const uint32_t g2 = n_grads - 1 - (a1 ? 1 : 0), back = dp ? 1 : 2;     // (g2: number of the pair before the last among its kind)
          uint64_t* const held = dp ? (a1 ? sm.step_done : sm.s_read) : a2 ? sm.acc_read : sm.step_done;
          const uint32_t by = !dp && a2 ? g2 : U - back;
          if (!wait_by_call(dp ? &sm.v_full[vs] : &sm.k_full[k.at], dp ? vp : k.parity) ||
              (u == 0 && !wait_by_call(dp ? &sm.do_full : &sm.q_full, n)) || (U >= back && !wait_by_call(&held[by & 1], by >> 1)))
            break;
          tc_fence_after_sync();
          issue(tmem + region(dp ? rp : rs), dp ? do_k : q_k, dp ? desc_advance(v_k, vs * kStage) : desc_advance(k_k, k.at * kStage));
          mma_commit_w(lead, dp ? &sm.dp_full[U & 1] : &sm.s_full[U & 1]);
          if (dp) mma_commit_w(lead, &sm.v_empty[vs]);
          if (u + 1 == n_pairs) mma_commit_w(lead, dp ? &sm.do_empty : &sm.q_empty);
          HGA_TRACE_POINT(6 + 2 * dp);
        }
        if (!ok) break;
        a2 = a1;
        a1 = pairs.with_grads(u);
        n_grads += a1;
        k.next();
        if (a1) k.next();
        vs ^= 1;
        if (vs == 0) vp ^= 1;
        next_regions(a1, rs, rp);
      }
    }
  } else if (warp == 2) {
    // ------------------------------------------------------------------ dQ, dV, dK
    const uint32_t lead = elect_one();
    constexpr uint32_t idesc_dq = idesc_bf16_f32(128, D, 0, 1);            // dS K-major, K tile MN-major
    constexpr uint32_t idesc_t = idesc_bf16_f32(D, 64, 1, 1);              // dO^T or Q^T, P or dS (keys along N): both MN-major
    const uint64_t k_mn = smem_desc_sw128(smem_u32(sm.k[0]), 1024, kOct);
    const uint64_t q_mn = smem_desc_sw128(smem_u32(sm.q), 16384, 1024), do_mn = smem_desc_sw128(smem_u32(sm.dO), 16384, 1024);
    const uint64_t p_mn = smem_desc_sw128(smem_u32(sm.k[0]), 16, 1024);
    uint32_t U = 0, n_grads = 0, rs = 0, rp = 1;
    KStage k;
    for (int n = 0; ok; ++n) {
      const Unit& un = unit_info(n);
      const int n_pairs = ok ? un.n_pairs : 0;
      if (n_pairs == 0) break;
      const Pairs pairs(un);
      done_with_info(n);
      if (pairs.n_a == 0) { mma_commit_w(lead, &sm.q_empty); mma_commit_w(lead, &sm.do_empty); }
      for (int u = 0; u < n_pairs; ++u, ++U) {
        if (!wait_by_call(&sm.ds_full[U & 1], U >> 1) || (u == 0 && n > 0 && !wait_by_call(&sm.dq_free, n - 1))) break;
        tc_fence_after_sync();
        HGA_TRACE_POINT(5);
        // bf16 dS from TMEM: first tile at columns 0-31 of its region, second tile at 64-95
        const uint64_t kb = desc_advance(k_mn, k.at * kStage);
        const uint32_t ds = tmem + region(rp);
#pragma unroll
        for (int kk = 0; kk < 8; ++kk)            // 16 keys per instruction
          mma_ts_w(lead, tmem, ds + (kk < 4 ? 8 * kk : 64 + 8 * (kk - 4)), desc_advance(kb, kk * 2 * kOct), idesc_dq, u > 0 || kk > 0);
        mma_commit_w(lead, &sm.step_done[U & 1]);
        mma_commit_w(lead, &sm.k_empty[k.at]);
        if (u + 1 == n_pairs) mma_commit_w(lead, &sm.dq_done);
        HGA_TRACE_POINT(7);
        k.next();
        const bool with_grads = pairs.with_grads(u);
        if (with_grads) {
          const uint32_t acc = tmem + region(rs);
          const uint64_t p = desc_advance(p_mn, k.at * kStage);
#pragma unroll 1
          for (uint32_t which = 0; which < 2; ++which)
#pragma unroll
            for (int kk = 0; kk < 8; ++kk)        // 16 query rows per instruction
              mma_ss_w(lead, acc + 64 * which, desc_advance(which ? q_mn : do_mn, kk * 2048), desc_advance(p, which * 16384 + kk * 2048), idesc_t, kk > 0);
          mma_commit_w(lead, &sm.acc_full[n_grads++ & 1]);
          mma_commit_w(lead, &sm.k_empty[k.at]);
          if (u + 1 == pairs.a_begin + pairs.n_a) { mma_commit_w(lead, &sm.q_empty); mma_commit_w(lead, &sm.do_empty); }
          k.next();
        }
        next_regions(with_grads, rs, rp);
      }
    }
  } else if (warp < 12) {
    // ------------------------------------------------------------------ one thread per query row and tile of a pair
    const int wg = (warp - 4) >> 2, quarter = warp & 3, row = quarter * 32 + lane;
    const uint32_t lane_base = tmem + ((uint32_t)(quarter * 32) << 16);
    const float sl2 = dm.scale * 1.4426950408889634f;
    const uint64_t sl2_2 = pack_f32x2(sl2, sl2);
    const uint32_t key = (uint32_t)(row & 7);
    uint32_t U = 0, rs = 0, rp = 1;
    KStage k;
    for (int n = 0; ok; ++n) {
      const Unit& un = unit_info(n);
      const int n_pairs = ok ? un.n_pairs : 0;
      if (n_pairs == 0) break;
      if (!wait(&sm.lse_full, n)) break;
      const float neg_lse2 = sm.nlse[row];
      const uint64_t neg_lse2_2 = pack_f32x2(neg_lse2, neg_lse2);
      float nds = 0.f;
      for (int u = 0; u < n_pairs; ++u, ++U) {
        const uint32_t s_addr = lane_base + region(rs) + wg * 64, dp_addr = lane_base + region(rp) + wg * 64;
        const Pairs pairs(un);                    // (read again for every pair: registers are short)
        const bool with_grads = pairs.with_grads(u);
        // how many of this thread's keys are visible: all of the far ones, of the local ones those up to the row's own
        const int see = un.vis + un.pos[row >> 6] + (row & 63);
        const int vis = (wg == 0 ? 8 * pairs.acts(u) : 0) + max(0, see - 8 * pairs.first_other(u, wg));
        uint32_t pk[32];                          // P of this row, 64 keys, packed bf16
        if (!wait(&sm.s_full[U & 1], U >> 1)) break;
        tc_fence_after_sync();
        HGA_TRACE_POINT(11);
        auto exponents = [&](uint32_t s0, uint32_t s1, float& a0, float& a1) {       // of two neighbouring keys
          unpack_f32x2(fma_f32x2(pack_f32x2(__uint_as_float(s0), __uint_as_float(s1)), sl2_2, neg_lse2_2), a0, a1);
        };
        if (!with_grads) {
#pragma unroll
          for (int q4 = 0; q4 < 4; ++q4) {
            uint32_t sv[16];
            tmem_ld16(s_addr + q4 * 16, sv);
            tmem_wait_ld();
#pragma unroll
            for (int i = 0; i < 8; ++i) {
              float a0, a1;
              exponents(sv[2 * i], sv[2 * i + 1], a0, a1);
              pk[8 * q4 + i] = pack_bf16(fast_exp2(a0), fast_exp2(a1));
            }
          }
          // (at the diagonal and the list's end only: two comparisons and selections per element in the loop above bound it by
          // instruction issue, and a copy of it costs more instruction fetch than this)
          if (__any_sync(0xffffffffu, vis < 64)) {
#pragma unroll
            for (int i = 0; i < 32; ++i) pk[i] = 2 * i + 1 < vis ? pk[i] : 2 * i < vis ? pk[i] & 0xffffu : 0u;
          }
        } else {
          // a pair with dK/dV: dS comes from the unrounded P, which takes the place of S (the next dP does not go there)
#pragma unroll 1
          for (int q4 = 0; q4 < 4; ++q4) {
            uint32_t sv[16];
            tmem_ld16(s_addr + q4 * 16, sv);
            tmem_wait_ld();
#pragma unroll
            for (int i = 0; i < 8; ++i) {
              float a0, a1;
              exponents(sv[2 * i], sv[2 * i + 1], a0, a1);
              sv[2 * i] = 16 * q4 + 2 * i < vis ? __float_as_uint(fast_exp2(a0)) : 0u;
              sv[2 * i + 1] = 16 * q4 + 2 * i + 1 < vis ? __float_as_uint(fast_exp2(a1)) : 0u;
            }
            tmem_st16(s_addr + q4 * 16, sv);
          }
          tmem_wait_st();
        }
        tc_fence_before_sync();
        mbar_arrive_warp(&sm.s_read[U & 1]);      // S has been read: its region may take the next pair's dP
        if (!wait(&sm.dp_full[U & 1], U >> 1)) break;
        if (u == 0) {
          if (!wait(&sm.stat_full, n)) break;
          nds = sm.nds[row];
          mbar_arrive_warp(&sm.stat_empty);
        }
        tc_fence_after_sync();
        HGA_TRACE_POINT(13);
        k.next();
        const uint64_t scale_2 = pack_f32x2(dm.scale, dm.scale), neg_delta_s_2 = pack_f32x2(nds, nds);
        auto gradient = [&](uint64_t p2, uint32_t dp0, uint32_t dp1) {               // dS of two neighbouring keys, rounded
          float d0, d1;
          unpack_f32x2(mul_f32x2(p2, fma_f32x2(pack_f32x2(__uint_as_float(dp0), __uint_as_float(dp1)), scale_2, neg_delta_s_2)), d0, d1);
          return pack_bf16(d0, d1);
        };
        // bf16 dS goes over the dP columns already read (8 columns per 16 keys): the A operand of dQ
        if (!with_grads) {
#pragma unroll
          for (int q4 = 0; q4 < 4; ++q4) {        // 16 keys at a time
            uint32_t dp[16], dk[8];
            tmem_ld16(dp_addr + q4 * 16, dp);
            tmem_wait_ld();
#pragma unroll
            for (int i = 0; i < 8; ++i)
              dk[i] = gradient(pack_f32x2(__uint_as_float(pk[8 * q4 + i] << 16), __uint_as_float(pk[8 * q4 + i] & 0xffff0000u)), dp[2 * i], dp[2 * i + 1]);
            tmem_st8(dp_addr + q4 * 8, dk);
          }
        } else {
          if (wg == 0 && !wait(&sm.k_full[k.at], k.parity)) break;
          const uint32_t p_line = smem_u32(sm.k[k.at]) + (uint32_t)row * 128;      // this row's 128-byte line of P (dS's: 16 KB on), 16-byte chunks XOR-swizzled
#pragma unroll 1
          for (int q4 = 0; q4 < 4; ++q4) {
            uint32_t p[16], dp[16], dk[8];
            tmem_ld16(s_addr + q4 * 16, p);
            tmem_ld16(dp_addr + q4 * 16, dp);
            tmem_wait_ld();
#pragma unroll
            for (int i = 0; i < 8; ++i)
              dk[i] = gradient(pack_f32x2(__uint_as_float(p[2 * i]), __uint_as_float(p[2 * i + 1])), dp[2 * i], dp[2 * i + 1]);
            tmem_st8(dp_addr + q4 * 8, dk);
            if (wg == 0) {
#pragma unroll
              for (int cc = 0; cc < 2; ++cc) {    // 8 keys
                const uint32_t at = p_line + ((uint32_t)(2 * q4 + cc) ^ key) * 16;
                auto rounded = [&](int i) { return pack_bf16(__uint_as_float(p[8 * cc + 2 * i]), __uint_as_float(p[8 * cc + 2 * i + 1])); };
                st_shared_v4(at, rounded(0), rounded(1), rounded(2), rounded(3));
                st_shared_v4(at + 16384, dk[4 * cc], dk[4 * cc + 1], dk[4 * cc + 2], dk[4 * cc + 3]);
              }
            }
          }
          fence_proxy_async_smem();
        }
        tmem_wait_st();
        tc_fence_before_sync();
        mbar_arrive_warp(&sm.ds_full[U & 1]);
        HGA_TRACE_POINT(14);
        if (with_grads) k.next();
        next_regions(with_grads, rs, rp);
      }
      done_with_info(n);
    }
  } else {
    // ------------------------------------------------------------------ statistics, dK / dV reduction, dQ epilogue
    const int quarter = warp & 3, row = quarter * 32 + lane;
    const uint32_t lane_base = tmem + ((uint32_t)(quarter * 32) << 16), key = (uint32_t)(row & 7);
    uint32_t n_grads = 0, rs = 0, rp = 1;
    bool band_done = false;
    // -LSE and -delta of unit n's rows: a thread each (O from global memory, dO from the tile in shared memory)
    auto statistics = [&](int n, const Unit& un) {
      const int half = row >> 6;
      const float lse = LSE[un.lse[half] + (row & 63)];
      const uint4* op = reinterpret_cast<const uint4*>(O + un.b * dm.os[0] + un.head[half] * dm.os[1] + (un.token[half] + (row & 63)) * dm.os[2]);
      uint4 o[4], o1[4];                          // 16-byte pieces of the row, four at a time
#pragma unroll
      for (int i = 0; i < 4; ++i) { o[i] = __ldg(op + i); o1[i] = __ldg(op + 4 + i); }
      if (n > 0 && !wait_by_call(&sm.stat_empty, n - 1)) return;       // the row threads have read the last unit's
      sm.nlse[row] = -lse * 1.4426950408889634f;
      mbar_arrive_warp(&sm.lse_full);
      if (!wait_by_call(&sm.do_full, n)) return;
      const uint32_t do_line = smem_u32(sm.dO) + (uint32_t)row * 128;
      uint64_t acc0 = 0, acc1 = 0;
#pragma unroll 1
      for (int q = 0; q < 4; ++q) {
        uint4 o2[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) o2[i] = q < 2 ? __ldg(op + 4 * q + 8 + i) : make_uint4(0, 0, 0, 0);
        const uint32_t panel = do_line + (uint32_t)(q >> 1) * 16384;
#pragma unroll
        for (int i = 0; i < 4; ++i) {             // (XOR-swizzled)
          uint32_t ys[4];
          ld_shared_v4(panel + (((uint32_t)(4 * (q & 1) + i) ^ key) * 16), ys[0], ys[1], ys[2], ys[3]);
          const uint32_t xs[4] = {o[i].x, o[i].y, o[i].z, o[i].w};
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            uint64_t& acc = e & 1 ? acc1 : acc0;
            acc = fma_f32x2(pack_f32x2(__uint_as_float(xs[e] << 16), __uint_as_float(xs[e] & 0xffff0000u)),
                            pack_f32x2(__uint_as_float(ys[e] << 16), __uint_as_float(ys[e] & 0xffff0000u)), acc);
          }
          o[i] = o1[i];
          o1[i] = o2[i];
        }
      }
      float acc[4];
      unpack_f32x2(acc0, acc[0], acc[1]);
      unpack_f32x2(acc1, acc[2], acc[3]);
      mbar_arrive_warp(&sm.do_empty);
      sm.nds[row] = -((acc[0] + acc[1]) + (acc[2] + acc[3])) * dm.scale;
      mbar_arrive_warp(&sm.stat_full);
      HGA_TRACE_POINT(10);
    };
    for (int n = 0; ok; ++n) {
      const Unit& un = unit_info(n);
      if (!ok) break;
      const bool more = un.n_pairs > 0;
      if (more) statistics(n, un);
      if (!ok) break;
      if (n > 0) {                                // dQ of the unit before
        const Unit& last = sm.unit[(n - 1) & 1];
        if (!wait_by_call(&sm.dq_done, n - 1)) break;
        tc_fence_after_sync();
        HGA_TRACE_POINT(20);
        const int half = row >> 6;
        uint16_t* const dq_out = dQ + last.b * dm.qs[0] + last.head[half] * dm.qs[1] + (last.token[half] + (row & 63)) * dm.qs[2];
        done_with_info(n - 1);
#pragma unroll 1
        for (int c = 0; c < 8; ++c) {
          uint32_t x[16];
          tmem_ld16(lane_base + 16 * c, x);
          tmem_wait_ld();
          if (c == 7) {
            tc_fence_before_sync();
            mbar_arrive_warp(&sm.dq_free);
          }
#pragma unroll
          for (int i = 0; i < 2; ++i)
            *reinterpret_cast<uint4*>(dq_out + 16 * c + 8 * i) =
                make_uint4(pack_bf16(__uint_as_float(x[8 * i]), __uint_as_float(x[8 * i + 1])), pack_bf16(__uint_as_float(x[8 * i + 2]), __uint_as_float(x[8 * i + 3])),
                           pack_bf16(__uint_as_float(x[8 * i + 4]), __uint_as_float(x[8 * i + 5])), pack_bf16(__uint_as_float(x[8 * i + 6]), __uint_as_float(x[8 * i + 7])));
        }
        HGA_TRACE_POINT(21);
      }
      if (!more) break;
#pragma unroll 1
      for (int u = 0; u < un.a_begin; ++u) next_regions(false, rs, rp);
#pragma unroll 1
      for (int first = 0; first < un.n_act; first += 8) {
        int mine;                                 // lane = octet: its position, -1 where it gets nothing from here
        {
          FarList far(dm, Window{0, un.ls, un.se}, group_idx + un.list);
          far.ng = un.ng; far.n_far = un.n_hist + un.n_act; far.clean = un.clean;
          mine = lane < 8 && first + lane < un.n_act ? far.row(un.n_hist + first + lane) : -1;
        }
        if (!wait_by_call(&sm.acc_full[n_grads & 1], n_grads >> 1)) break;
        tc_fence_after_sync();
        HGA_TRACE_POINT(16);
        // The band kernel, which precedes this one in the stream, stores its dK/dV rows plainly: these additions must come
        // after it.  Nothing else in this kernel depends on it (what is read was complete when that kernel let this one start).
        if (!band_done) { pdl_wait(); band_done = true; }
        // lane = element, column = key: 128 consecutive bytes per warp and addition
        // (staged in shared memory as key rows and added 512 bytes or 4 KB at a time, the additions held the place of P and
        // dS, and with it the K ring, for 5k cycles a pair)
#pragma unroll 1
        for (int part = 0; part < 4; ++part) {    // dV of octets 0-3 and 4-7, dK of the same
          uint32_t x[32];
          tmem_ld32(lane_base + region(rs) + 32 * part, x);
          tmem_wait_ld();
          if (part == 3) {
            tc_fence_before_sync();
            mbar_arrive_warp(&sm.acc_read[n_grads & 1]);
          }
#pragma unroll
          for (int o = 0; o < 4; ++o) {
            const int at = __shfl_sync(0xffffffffu, mine, 4 * (part & 1) + o);
            if (at >= 0) {
              float* const to = (part >= 2 ? dK : dV) + (un.grad_row + at) * D + row;
#pragma unroll
              for (int i = 0; i < 8; ++i) red_add(to + i * D, __uint_as_float(x[8 * o + i]));
            }
          }
        }
        if (!ok) break;
        HGA_TRACE_POINT(18);
        ++n_grads;
        next_regions(true, rs, rp);
      }
      if (!ok) break;
#pragma unroll 1
      for (int u = un.a_begin + un.n_a; u < un.n_pairs; ++u) next_regions(false, rs, rp);
    }
    // the end of this grid has to imply the end of the band kernel's, even where there was nothing to add
    if (!band_done) pdl_wait();
  }
  HGA_TRACE_POINT(30);

  // Common exit.  Roles leave their warps diverged, so every warp reconverges first: a block barrier reached by
  // part of a warp would count that warp as arrived.
  __syncwarp();
  tc_fence_before_sync();
  __syncthreads();
  HGA_TRACE_POINT(31);
  HGA_TRACE_DUMP;
  if (sm.abort) {
    // Given up (known for certain behind the barrier, and the same in every thread).  GEMMs already issued, by either issuing
    // warp, may still be reading shared and writing tensor memory: wait (bounded) until the tensor pipe has run dry, and give
    // the copies in flight time to land (their barriers may never complete, hence a bounded sleep).
    if (tid == 0 && status_word) atomicOr(status_word, HGA_ABORT_CODE(3, sm.abort));
    if (warp == 1 || warp == 2) {
      mma_commit_w(elect_one(), &sm.drain[warp - 1]);
      mbar_wait(&sm.drain[warp - 1], 0);
    }
    if (tid == 0)
      for (int it = 0; it < 64; ++it) __nanosleep(1000);
    __syncwarp();
    __syncthreads();
  }
  if (warp == 1) tmem_dealloc(tmem, 512);
}

bool attn_bwd_sm100_supported(const Dims& dm) {
  if (dm.flags & HGA_FLAG_GENERIC_KERNELS) return false;
  if (dm.g % 8 != 0 || !attn_bwd_band_sm100_supported(dm)) return false;
  // The smallest layers of head_dim 64 (fewer than eight M-tiles, few keys) keep the CUDA-core kernel, whose dV is 1.2e-7 closer
  // to fp64, for two microseconds: 4 tiles of 320 keys 16.4 us, 14.5 here.  Its time grows with the keys faster than this path's
  // (one CTA per eight rows: 704 keys 35 us, 24 here; 2240 keys 92, 63; 4288 keys 167, 116; 1 to 8 tiles alike on both sides).
  if (dm.d == 64 && dm.B * dm.Hkv * dm.NQB * ((dm.rows + 127) / 128) < 8 && max_routed_tokens(dm) <= 512) return false;
  return true;
}

template <class Segs>
static int launch_sweep(const Dims& dm, SegTable* table, const Segs& segs, int64_t units, const void* Q, const void* K, const void* V,
                        const void* O, const float* LSE, const void* dO, const int32_t* group_idx,
                        const int32_t* n_groups, void* dQ, float* dK, float* dV, int32_t* status_word, cudaStream_t st) {
  // Nothing here depends on the width; the line is one of precision.  The CUDA-core kernel, which the wider items were given by an
  // earlier sweep that had no room for their table, holds P and dS in fp32, and their callers have had its errors since.  Against fp64
  // (dQ / dK / dV), 16 items of 256 rows and 4.5K keys: CUDA cores 1.67e-3 / 5.9e-5 / 5.6e-7 in 1359 us, this kernel 2.86e-3 / 2.00e-3 /
  // 1.65e-3 in 76 us, k_attn_bwd_terms_sm100 1.67e-3 / 5.9e-5 / 1.30e-6 in 164 us.  Narrower items have this kernel's errors:
  // 3.2K keys 2.86e-3 / 2.02e-3 / 1.67e-3, 56 us.
  if ((int64_t)dm.sink + (int64_t)dm.width * dm.g + dm.local + dm.Bq + dm.c > kMostRoutedTokens) return HGA_ERR_UNSUPPORTED;
  CUtensorMap mq, mdo, mk, mv;
  const uint32_t box[5] = {64, 8, 2, 1, 1};
  const uint32_t box_q[5] = {64, 64, 1, 1, 1};
  const uint64_t dq[5] = {64, (uint64_t)dm.rows_q, 2, (uint64_t)dm.Hq, (uint64_t)dm.B};
  const uint64_t dk[5] = {64, (uint64_t)dm.rows_k, 2, (uint64_t)dm.Hkv, (uint64_t)dm.B};
  const uint64_t sq[4] = {(uint64_t)dm.qs[2] * 2, 128, (uint64_t)dm.qs[1] * 2, (uint64_t)dm.qs[0] * 2};
  const uint64_t so[4] = {(uint64_t)dm.os[2] * 2, 128, (uint64_t)dm.os[1] * 2, (uint64_t)dm.os[0] * 2};
  const uint64_t sk[4] = {(uint64_t)dm.ks[2] * 2, 128, (uint64_t)dm.ks[1] * 2, (uint64_t)dm.ks[0] * 2};
  const uint64_t sv[4] = {(uint64_t)dm.vs[2] * 2, 128, (uint64_t)dm.vs[1] * 2, (uint64_t)dm.vs[0] * 2};
  if (encode_tensor_map_bf16(&mq, Q, 5, dq, sq, box_q, true) ||
      encode_tensor_map_bf16(&mdo, dO, 5, dq, so, box_q, true) ||
      encode_tensor_map_bf16(&mk, K, 5, dk, sk, box, true) ||
      encode_tensor_map_bf16(&mv, V, 5, dk, sv, box, true))
    return HGA_ERR_UNSUPPORTED;
  const size_t smem = sizeof(BwdSmem) + 1024;      // (slack for the manual alignment)
  int rc = ensure_dynamic_smem(reinterpret_cast<const void*>(&k_attn_bwd_sm100<Segs>), smem);
  if (rc) return rc;
  // dK/dV of the local band: written once per key tile by the key-major kernel, with plain stores that
  // cover every row of the active segment (so nothing has to be zero-filled); this kernel then adds the
  // contributions of the keys before the band atomically.  It may start on SMs the band kernel leaves idle (programmatic
  // serialization; it waits for it only before adding to dK/dV).
  rc = launch_attn_bwd_band_sm100(dm, table, Q, K, V, O, LSE, dO, dK, dV, status_word, st);
  if (rc != HGA_OK) return rc;
  if (table) units = number_units(*table, [&](const Segment& g) { return (int64_t)dm.B * dm.Hkv * (g.S / dm.Bq) * (dm.rows / 128); });
  PdlLaunch cfg((unsigned)units, kBwdThreads, smem, st, dm.flags);
  const cudaError_t e = cudaLaunchKernelEx(&cfg.c, k_attn_bwd_sm100<Segs>, mq, mdo, mk, mv, (const uint16_t*)O, LSE, group_idx,
                                           n_groups, dm, (uint16_t*)dQ, dK, dV, status_word, segs);
  count_launch(HGA_KERNELS_BWD_TENSOR);
  return record_cuda(e);
}

// Whether two bf16 tensors of query rows (strides as in Dims) may share bytes: the spans between their first and last elements meet
static bool rows_meet(const Dims& dm, const void* a, const int64_t* sa, const void* b, const int64_t* sb) {
  auto last = [&](const void* p, const int64_t* s) {
    return (uintptr_t)p + 2 * (uintptr_t)((dm.B - 1) * s[0] + (dm.Hq - 1) * s[1] + (dm.rows_q - 1) * s[2] + dm.d - 1);
  };
  return (uintptr_t)a <= last(b, sb) && (uintptr_t)b <= last(a, sa);
}

int launch_attn_bwd_sm100(const Dims& given, SegTable* segs, const void* Q, const void* K, const void* V, const void* O,
                          const float* LSE, const void* dO, const int32_t* group_idx,
                          const int32_t* n_groups, void* dQ, float* dK, float* dV, int32_t* status_word,
                          cudaStream_t st) {
  Dims dm = given;
  // Inside a step the band kernel copies Q and dO while the forward still stores O: not where O is one of them (the gradient of
  // |O|^2 / 2 is O).
  if (rows_meet(dm, O, dm.os, dO, dm.os) || rows_meet(dm, O, dm.os, Q, dm.qs)) dm.flags &= ~kFlagChained;
  // The sweep stores dQ while the band kernel may still read other key tiles' share of the same rows of Q, dO and O: where dQ is
  // one of those, it starts behind the band kernel's end.
  if (rows_meet(dm, dQ, dm.qs, Q, dm.qs) || rows_meet(dm, dQ, dm.qs, dO, dm.os) || rows_meet(dm, dQ, dm.qs, O, dm.os)) dm.flags |= kFlagNoPdl;
  if (bwd_in_terms(dm))
    return launch_attn_bwd_terms_sm100(dm, segs, Q, K, V, O, LSE, dO, group_idx, n_groups, dQ, dK, dV, status_word, st);
  const int64_t units = (int64_t)dm.B * dm.Hkv * dm.NQB * (dm.rows / 128);
  if (!segs)
    return launch_sweep(dm, nullptr, OneSegment{}, units, Q, K, V, O, LSE, dO, group_idx, n_groups, dQ, dK, dV, status_word, st);
  return launch_sweep(dm, segs, *segs, units, Q, K, V, O, LSE, dO, group_idx, n_groups, dQ, dK, dV, status_word, st);
}

}  // namespace hga

#ifdef HGA_DEBUG_WAIT
extern "C" __attribute__((visibility("default"))) int hga_debug_dump(int* out64) {
  cudaMemcpyFromSymbol(out64, hga::g_dbg_fail, sizeof(int) * 64);
  int zero[64] = {0};
  cudaMemcpyToSymbol(hga::g_dbg_fail, zero, sizeof(zero));
  return 0;
}
#endif
