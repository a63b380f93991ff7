// hga_attn_bwd for sm_100a with fp32-grade probabilities: the query-major sweep (routing frozen, Section 2.1 last paragraph;
// history K/V detached, Section 2.2) of the shapes that the CUDA-core backward, which holds P and dS in fp32, used to take:
// head_dim 64, and query-row counts that do not fill 128-row M-tiles.
//
// bf16 operands hold P and dS to 2^-9.  Here P enters its products in three bf16 terms (p = p1 + p2 + p3, each the rounding
// of what the ones before it leave: 24 bits) and dS in two (16 bits; its error is that of delta = rowsum(dO o O), which
// comes from the rounded O, 2^-9 of a sum of many, and dQ is rounded to bf16).  Every term is a GEMM of its own.  Errors
// against fp64 (head_dim 64, 64 rows; relative, dQ / dK / dV): 1.68e-3 / 1.33e-4 / 5.0e-7, on CUDA cores 1.68e-3 / 1.33e-4 /
// 3.8e-7 (the tensor pipe cuts S and its sums off at 2^-24), with one term 2.9e-3 / 2.1e-3 / 1.6e-3; at head_dim 128 dV
// is off by 0.8e-6 to 1.8e-6 (see k_attn_bwd_band_sm100 for why not less).
// hga_attn_bwd, 16 heads of 64 rows, 512 items of 768 keys: head_dim 64 71 us (CUDA cores 918), head_dim 128 128 us (1970).
// What bounds it: the row threads, with twice the instructions per weight, and the hand-offs.
//
// Work unit (one CTA): one 128-row M-tile of one item (b, kv head, query block), swept over the item's routed
// keys in 64-key tiles (eight octets of 8 consecutive tokens, one TMA box each).  At head_dim 64 a CTA takes less than
// half of an SM (88 KB of shared memory, 256 TMEM columns, 256 threads), so two CTAs run on an SM: a tile is
// a chain of hand-offs (copy -> S -> dS -> dQ), and while one CTA is in its exponentials, its set-up, its
// dK/dV reduction or its epilogue, the other one has the tensor pipe.  At head_dim 128 it has the SM to itself.
//
// An M-tile that holds 64 rows only has them TWICE, in lanes 0-63 and 64-127, and a row's two threads take the first and the
// last 32 keys of every tile, with zeros in the columns of the others: dQ is the sum of the two lanes' in the end.  (With zero
// rows in lanes 64-127 two of the four sub-cores of an SM did all the work: 16 heads of 64 159.6 us a whole step, 146.5 so.)
//
// Order of the tiles of an item:
//   1. the local window and the causal block, [ls, p0 + Bq): known without the routing list, so their copies
//      start at once and the list is fetched and checked behind them;
//   2. "far" keys (sink, then the selected groups, ascending) of the detached history: dQ only;
//   3. far keys of the active segment, which also get dK/dV from this kernel (the local band's dK/dV are written by
//      the key-major kernel k_attn_bwd_band_sm100, which precedes this one and stores every row).
// Per tile: S = Q K^T, dP = dO V^T (smem x smem -> TMEM); one thread per query row turns them, 16 keys at a time, into
// P = e^(S*scale - LSE) and dS = scale * P o (dP - delta), and the two terms of dS go over the dP columns just read:
// dQ += dS K with A from TMEM.  Tiles of kind 3 go through shared memory in three rounds besides: p1 and p2; p3 and dS's
// first term; dS's second.  dV^T = dO^T P (over the other S buffer) and dK^T = Q^T dS (over this tile's S, dead by then) sum
// them up; the row threads stage the transposed tiles in shared memory as key rows and add them to global memory with bulk
// reductions.  At head_dim 64 one instruction does both halves, M = 128: A = [dO^T ; Q^T] (the two tiles are neighbours), of
// whose products with P and dS one half each is wanted, and a staged row is dV | dK.
// S has two buffers: S(j+1) is issued ahead of dQ(j) if its K tile is already there, dP(j+1) behind dQ(j): the in-order
// tensor pipe makes every reuse of a region safe.  A wait on S(j+1)'s K tile never holds up dQ(j), which frees the stage of
// K(j+2).
//
// Warp roles (256 threads):
//   warps 0, 7   producers: octets 0-3 / 4-7 of every K and V tile (a box costs its issuing warp ~100 cycles)
//   warp 6       Q and dO tiles, then the check of the routing list       warp 1   MMA issuer
//   warps 2-5    one thread per query row (TMEM lane = row); delta = rowsum(dO o O) of its own row
// TMEM: S 64 | dP / dS 64 | dQ head_dim | S 64.
#include "hga_bwd_sm100.cuh"
#include "hga_common.cuh"
#include "hga_octets.cuh"
#include "hga_sm100.cuh"

namespace hga {

using namespace sm100;

namespace {

constexpr int kThreads = 256;
constexpr int kKT = 64;                         // keys per tile
constexpr int kPdsTile = 128 * kKT * 2;         // bytes of one term of P or dS: [16 row octets][8 rows][128 B], 128-byte swizzle

template <int D>
struct SweepSmem {
  static constexpr int kQBytes = 128 * D * 2;   // the Q or dO tile: [panel][128 rows][128 B]
  static constexpr int kKv = kKT * D * 2;       // one K or V tile: [octet][panel][8 rows][128 B]
  alignas(1024) uint8_t dO[kQBytes];            // (dO and Q adjacent: at head_dim 64 one MN-major operand of 128 rows, see above)
  alignas(1024) uint8_t q[kQBytes];
  alignas(1024) uint8_t k[2][kKv];
  alignas(1024) uint8_t v[kKv];
  alignas(1024) uint8_t a[kPdsTile];            // dK/dV tiles: two terms at a time, then the staged key rows
  alignas(1024) uint8_t b[kPdsTile];
  uint64_t q_full, k_full[2], k_empty[2], v_full;
  uint64_t s_full[2], dp_full, ds_full;                 // per tile (S(j+1) may be complete before S(j) has been looked for)
  uint64_t round_full, round_done, acc_read, staged;    // dK/dV tiles
  uint64_t info_full, dq_done, dq_staged, drain;
  uint32_t tmem_base;
  int n_far, first_active, n_listed;                    // far octets; the first of them that belongs to the active segment; list entries (see FarList)
  bool clean;
  volatile int abort;
  int rows[4][8];                                       // token rows of the last four tiles' octets (dK/dV tiles read them back)
};
static_assert(sizeof(SweepSmem<64>) + 1024 <= 113 * 1024, "two CTAs per SM");

}  // namespace

template <int D, class Segs>
__global__ void __launch_bounds__(kThreads, D == 64 ? 2 : 1)
k_attn_bwd_terms_sm100(const __grid_constant__ CUtensorMap map_q, const __grid_constant__ CUtensorMap map_do,
                 const __grid_constant__ CUtensorMap map_k, const __grid_constant__ CUtensorMap map_v,
                 const __grid_constant__ CUtensorMap map_dq, const uint16_t* __restrict__ O,
                 const float* __restrict__ LSE, const int32_t* __restrict__ group_idx,
                 const int32_t* __restrict__ n_groups, const Dims dm,
                 float* __restrict__ dK, float* __restrict__ dV, int32_t* status_word, const __grid_constant__ Segs segs) {
  using Smem = SweepSmem<D>;
  constexpr int kOct = 8 * D * 2, kPanels = D / 64, kQBytes = Smem::kQBytes, kKv = Smem::kKv;
  constexpr uint32_t kColDP = 64, kColDQ = 128, kTmemCols = D == 64 ? 256 : 512;
  auto s_col = [](int j) -> uint32_t { return (j & 1) ? 128 + D : 0; };      // S of tile j
  extern __shared__ uint8_t smem_raw[];
  Smem& sm = *reinterpret_cast<Smem*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  HGA_TRACE_DECL(64);
  const int n_mt_item = (dm.rows + 127) / 128;
  // Launch order: late query blocks first.  They have the most routed keys inside the active segment (the
  // expensive dK/dV tiles), early ones none, so the cheapest CTAs are the ones that fill the last wave.
  int cta;
  const Segment sg = segment_of(dm, segs, blockIdx.x, cta);
  const int n_qb = dm.by_Bq(sg.S), unit = dm.by_mt(cta), n_bh = dm.B * dm.Hkv, mt = cta - unit * n_mt_item;
  const int i_qb = dm.by_bh(unit), bh = unit - i_qb * n_bh, qb = n_qb - 1 - i_qb, b = dm.by_Hkv(bh), h = bh - b * dm.Hkv;
  const int64_t item = item_base(dm, sg, b) + h * n_qb + qb;
  const bool twice = dm.rows - mt * 128 == 64;          // the M-tile's rows are there twice (Bq is a multiple of 64)
  const int qrow = sg.q0 + qb * dm.Bq;                  // the block's first row in Q, O, dO and dQ
  const Window w = window_at(dm, sg.H + qb * dm.Bq);
  const int n_local = w.p0 + dm.Bq - w.ls;              // tokens of the local window and the block (a multiple of 8)
  const int n_lt = (n_local + kKT - 1) / kKT;           // its tiles
  volatile int* abort = &sm.abort;

  // Row threads: LSE and the O row of the thread's own query row, requested
  // before anything else so that the latency hides behind the set-up.
  float row_lse = 0.f;
  int row_pos = 0;                                      // position inside the query block
  uint4 o_row[D / 8];
  if (warp >= 2 && warp < 6) {
    const int r = mt * 128 + (((warp & 3) * 32 + lane) & (twice ? 63 : 127)), a = dm.by_Bq(r);
    row_pos = r - a * dm.Bq;
    const int hq = h * dm.G + a, srow = qrow + row_pos;
    row_lse = LSE[row_base(dm, sg, b) * dm.Hq + (int64_t)hq * sg.S + (srow - sg.q0)];
    const uint4* op = reinterpret_cast<const uint4*>(O + b * dm.os[0] + hq * dm.os[1] + (int64_t)srow * dm.os[2]);
#pragma unroll
    for (int i = 0; i < D / 8; ++i) o_row[i] = __ldg(op + i);
  }
  // Octet rows of local tile j for the producers (lane < 4: octet 4 * half + lane); past the window: out of range, zeros
  const int half = warp == 7 ? 1 : 0;
  auto local_row = [&](int j) {
    const int off = kKT * j + 8 * (4 * half + lane);
    return off < n_local ? sg.k0 + w.ls + off : dm.rows_k;
  };
  auto copy_tile = [&](uint8_t* dst, const CUtensorMap* map, uint64_t* full, int row) {
    if (lane == 0) mbar_arrive_expect_tx(full, 4 * kOct);
    __syncwarp();
    if (lane < 4) tma_load_5d(dst + (4 * half + lane) * kOct, map, full, 0, row, 0, h, b);
  };
  auto note_rows = [&](int j, int row) {
    if (lane < 4) sm.rows[j & 3][4 * half + lane] = row;
  };
  if (warp == 0 && lane == 0) {
    mbar_init(&sm.q_full, 1);
    for (int s = 0; s < 2; ++s) { mbar_init(&sm.k_full[s], 2); mbar_init(&sm.k_empty[s], 1); }
    mbar_init(&sm.v_full, 2);
    mbar_init(&sm.s_full[0], 1); mbar_init(&sm.s_full[1], 1);
    mbar_init(&sm.dp_full, 1); mbar_init(&sm.ds_full, 4);
    mbar_init(&sm.round_full, 4); mbar_init(&sm.round_done, 1); mbar_init(&sm.acc_read, 4); mbar_init(&sm.staged, 4);
    mbar_init(&sm.info_full, 1); mbar_init(&sm.dq_done, 1); mbar_init(&sm.dq_staged, 4); mbar_init(&sm.drain, 1);
    sm.abort = 0;
    fence_barrier_init();
  }
  if (warp == 0 || warp >= 6) {
    // Q, dO and the first local tile depend on nothing: their copies start before the CTA meets.  Barrier 2 makes
    // the mbarrier initialisation above visible to the three issuing warps.
    asm volatile("bar.sync 2, 96;" ::: "memory");
    if (warp == 6) {
      if (lane == 0) mbar_arrive_expect_tx(&sm.q_full, 2 * kQBytes);
      __syncwarp();
      if (lane < 4 * kPanels) {
        // boxes of 64 rows x one panel, Q first, then dO
        const int is_do = lane / (2 * kPanels), hf = lane & 1, panel = (lane >> 1) % kPanels;
        const int r = mt * 128 + (twice ? 0 : 64 * hf), a = dm.by_Bq(r);
        tma_load_5d((is_do ? sm.dO : sm.q) + panel * 16384 + hf * 8192, is_do ? &map_do : &map_q, &sm.q_full, 0,
                    qrow + r - a * dm.Bq, panel, h * dm.G + a, b);
      }
    } else {
      const int row = local_row(0);
      copy_tile(sm.k[0], &map_k, &sm.k_full[0], row);
      copy_tile(sm.v, &map_v, &sm.v_full, row);
    }
    __syncwarp();
  }
  if (warp == 1) {
    tmem_alloc(&sm.tmem_base, kTmemCols);
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
  // Tile counts, once the list is known: tiles [0, n_a) are of kinds 1 and 2, tiles [n_a, n) of kind 3.
  auto counts = [&](int n_far, int first_active, int& n, int& n_a) {
    n = n_lt + (n_far + 7) / 8;
    n_a = first_active < n_far ? n_lt + first_active / 8 : n;
  };

  if (warp == 0 || warp == 7) {
    // ------------------------------------------------------------------ producers
    bool ok = true;
    FarList far(dm, w, group_idx + item * dm.width);
    int n = 0, n_a = 0;
    bool known = false;                                   // the list has been checked (warp 6) and its counts read
    auto learn = [&]() {
      ok = wait_out_of_line(&sm.info_full, 0, abort);
      far.ng = sm.n_listed; far.n_far = sm.n_far; far.first_active = sm.first_active; far.clean = sm.clean;
      counts(far.n_far, far.first_active, n, n_a);
      known = true;
      return ok;
    };
    // row of this lane's octet of tile j (any kind; rows past the item's keys are out of range)
    auto row_of = [&](int j) {
      if (j < n_lt) return local_row(j);
      const int o = 8 * (j - n_lt) + 4 * half + (lane & 3);
      return o < far.n_far ? sg.k0 + far.row(o) : dm.rows_k;
    };
    auto wait_for = [&](uint64_t* bar, uint32_t parity, int line = __builtin_LINE()) { return ok = wait_out_of_line(bar, parity, abort, line); };
    auto copy_k = [&](int j, int row) {
      note_rows(j, row);
      __syncwarp();                            // (all of them, before the arrival that publishes them)
      copy_tile(sm.k[j & 1], &map_k, &sm.k_full[j & 1], row);
    };
    // Rows of the next two tiles, looked up ahead of their use.  Tile j + 1's K has been issued when tile j is handled.
    if (n_lt < 3) learn();
    int next_row = ok ? row_of(1) : dm.rows_k, after_row = ok ? row_of(2) : dm.rows_k;
    if (ok && (n_lt > 1 || n > 1)) copy_k(1, next_row);
    // The events this loop waits for come in this order: dP(j) done, dQ(j) done, dP(j+1) done, ...
    for (int j = 0; ok; ++j) {
      if (!known && j + 3 >= n_lt && !learn()) break;
      if (known && j + 1 >= n) break;
      if (!wait_for(&sm.dp_full, j & 1)) break;                           // V(j) has been read
      copy_tile(sm.v, &map_v, &sm.v_full, next_row);                       // V(j+1)
      next_row = after_row;
      after_row = row_of(j + 3);
      if (!known || j + 2 < n) {
        if (!wait_for(&sm.k_empty[j & 1], (j >> 1) & 1)) break;           // dQ(j) is done
        copy_k(j + 2, next_row);
      }
      HGA_TRACE_POINT(2);
    }
    if (*abort && lane == 0) {
      // giving up: give the copies still in flight time to land before shared memory is released
      // (the full barriers may never complete once another role has stopped, hence a bounded sleep)
      for (int it = 0; it < 64; ++it) __nanosleep(1000);
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------------ MMA issuer
    // The whole warp runs this branch converged (waits included) and one elected lane issues: see mma_ss_w.
    const uint32_t lead = elect_one();
    auto mma_wait = [&](uint64_t* bar, uint32_t parity, int line = __builtin_LINE()) { return wait_out_of_line(bar, parity, abort, line); };
    constexpr uint32_t idesc_sdp = idesc_bf16_f32(128, kKT, 0, 0);       // rows x 64 keys, both K-major
    constexpr uint32_t idesc_dq = idesc_bf16_f32(128, D, 0, 1);          // dS K-major, K tile MN-major
    constexpr uint32_t idesc_dkv = idesc_bf16_f32(128, kKT, 1, 1);       // both MN-major
    // Descriptors are built once; inside the loops an MMA costs two integer adds.
    // Q, dO: [panel][128 rows][128 B] (8-row groups 1024 B apart, panels 16 KB apart)
    const uint64_t q_k = smem_desc_sw128(smem_u32(sm.q), 16, 1024);         // Q  as K-major A   (S)
    const uint64_t do_k = smem_desc_sw128(smem_u32(sm.dO), 16, 1024);       // dO as K-major A   (dP)
    // MN-major A of dV^T and of dK^T (two 64-element atoms 16 KB apart: the panels, or at head_dim 64 dO and Q for both)
    const uint64_t do_mn = smem_desc_sw128(smem_u32(sm.dO), 16384, 1024);
    const uint64_t q_mn = D == 64 ? do_mn : smem_desc_sw128(smem_u32(sm.q), 16384, 1024);
    const uint64_t k_k0 = smem_desc_sw128(smem_u32(sm.k[0]), 16, kOct);     // K tile, K-major B  (S)
    const uint64_t v_k = smem_desc_sw128(smem_u32(sm.v), 16, kOct);         // V tile, K-major B  (dP)
    const uint64_t k_mn0 = smem_desc_sw128(smem_u32(sm.k[0]), 1024, kOct);  // K tile, MN-major B (dQ)
    const uint64_t ad = smem_desc_sw128(smem_u32(sm.a), 16, 1024);          // a term of P or dS: MN-major B
    const uint64_t bd = smem_desc_sw128(smem_u32(sm.b), 16, 1024);
    auto issue_qk = [&](uint32_t acc, uint64_t a, uint64_t b) {
#pragma unroll
      for (int kk = 0; kk < D / 16; ++kk)
        mma_ss_w(lead, acc, desc_advance(a, (kk >> 2) * 16384 + (kk & 3) * 32), desc_advance(b, (kk >> 2) * 1024 + (kk & 3) * 32), idesc_sdp, kk > 0);
    };
    auto issue_s = [&](int j) {
      issue_qk(tmem + s_col(j), q_k, desc_advance(k_k0, (uint32_t)(j & 1) * kKv));
      mma_commit_w(lead, &sm.s_full[j & 1]);
    };
    auto issue_dp = [&]() {
      issue_qk(tmem + kColDP, do_k, v_k);
      mma_commit_w(lead, &sm.dp_full);           // also tells the producers that the V tile is free
    };
    // dV^T or dK^T: 16 query rows per MMA (2 row octets), the rows once where they are there twice
    auto issue_t = [&](uint32_t acc, uint64_t amn, uint64_t term, bool accumulate) {
#pragma unroll 1
      for (uint32_t part = 0; part < (twice ? 1 : 2); ++part)
#pragma unroll
        for (int kk = 0; kk < 4; ++kk)
          mma_ss_w(lead, acc, desc_advance(amn, part * 8192 + kk * 2048), desc_advance(term, part * 8192 + kk * 2048), idesc_dkv, accumulate || part > 0 || kk > 0);
    };
    bool ok = mma_wait(&sm.q_full, 0) && mma_wait(&sm.k_full[0], 0);
    HGA_TRACE_POINT(40);
    if (ok) { tc_fence_after_sync(); issue_s(0); ok = mma_wait(&sm.v_full, 0); }
    if (ok) { tc_fence_after_sync(); issue_dp(); }
    HGA_TRACE_POINT(3);
    int n = n_lt + 1, n_a = n_lt;                 // (bounds that do until the list is known)
    auto k_parity = [](int j) { return (uint32_t)(j >> 1) & 1; };
    for (int j = 0; j < n && ok; ++j) {
      if (j + 1 == n_lt) {
        ok = mma_wait(&sm.info_full, 0);
        if (!ok) break;
        counts(sm.n_far, sm.first_active, n, n_a);
      }
      const bool dkv = j >= n_a;
      // S(j+1) goes ahead of dQ(j) if its K tile is already there (its buffer held S(j-1), which the rows are done with); waiting
      // for the tile first would hold up dQ(j), and with it the copy of K(j+2) into the stage that dQ(j) reads
      bool s_ahead = false;
      if (!dkv && j + 1 < n) {
        s_ahead = __all_sync(0xffffffffu, mbar_test_wait(&sm.k_full[(j + 1) & 1], k_parity(j + 1)));
        if (s_ahead) {
          tc_fence_after_sync();
          issue_s(j + 1);
          HGA_TRACE_POINT(6);
        }
      }
      ok = mma_wait(&sm.ds_full, j & 1);
      if (!ok) break;
      tc_fence_after_sync();
      HGA_TRACE_POINT(5);
      const uint64_t kmn = desc_advance(k_mn0, (uint32_t)(j & 1) * kKv);
#pragma unroll
      for (int kk = 0; kk < 2 * (kKT / 16); ++kk)     // 16 keys (two octets of the K tile): 8 TMEM columns of each of dS's terms
        mma_ts_w(lead, tmem + kColDQ, tmem + kColDP + 8 * kk, desc_advance(kmn, (kk >> 1) * 2 * kOct), idesc_dq, (j > 0 || kk > 0));
      mma_commit_w(lead, &sm.k_empty[j & 1]);
      HGA_TRACE_POINT(7);
      if (dkv) {
        const uint32_t dv_acc = tmem + s_col(j + 1), dk_acc = tmem + s_col(j);
        const uint32_t phase = (uint32_t)(j - n_a) * 2;
        issue_t(dv_acc, do_mn, ad, false);                              // p1, p2
        issue_t(dv_acc, do_mn, bd, true);
        mma_commit_w(lead, &sm.round_done);
        ok = mma_wait(&sm.round_full, phase & 1);
        if (!ok) break;
        tc_fence_after_sync();
        issue_t(dv_acc, do_mn, ad, true);                               // p3, dS's first term (S(j) has been read)
        issue_t(dk_acc, q_mn, bd, false);
        mma_commit_w(lead, &sm.round_done);
        ok = mma_wait(&sm.round_full, (phase + 1) & 1);
        if (!ok) break;
        tc_fence_after_sync();
        issue_t(dk_acc, q_mn, ad, true);                                // dS's second term
        mma_commit_w(lead, &sm.round_done);
        HGA_TRACE_POINT(4);
        if (j + 1 < n) {
          ok = mma_wait(&sm.acc_read, (uint32_t)(j - n_a) & 1);         // S(j+1) takes the place of dV^T
          if (!ok) break;
        }
      }
      if (j + 1 < n) {
        if (!s_ahead) {
          ok = mma_wait(&sm.k_full[(j + 1) & 1], k_parity(j + 1));
          if (!ok) break;
          tc_fence_after_sync();
          issue_s(j + 1);
        }
        ok = mma_wait(&sm.v_full, (j + 1) & 1);
        if (!ok) break;
        tc_fence_after_sync();
        issue_dp();
        HGA_TRACE_POINT(8);
      }
    }
    if (ok) mma_commit_w(lead, &sm.dq_done);
  } else if (warp == 6) {
    // ------------------------------------------------------------------ routing list
    FarList far(dm, w, group_idx + item * dm.width);
    far.check(dm, n_groups + item, sg.H);      // (the forward call reports invalid lists)
    if (lane == 0) {
      sm.n_listed = far.ng; sm.n_far = far.n_far; sm.first_active = far.first_active; sm.clean = far.clean;
      mbar_arrive(&sm.info_full);
    }
    pdl_wait();      // (the end of this grid has to imply the end of the band kernel's, even where there is nothing to add)
  } else if (warp < 6) {
    // ------------------------------------------------------------------ one thread per query row
    const int quarter = warp & 3;
    const int row_in_tile = quarter * 32 + lane, row_of_item = row_in_tile & (twice ? 63 : 127);
    const int c_first = twice && row_in_tile >= 64 ? 2 : 0, c_end = twice ? c_first + 2 : 4;      // its 16-key chunks of a tile
    const int limit = w.p0 - w.ls + row_pos + 1;            // visible keys of the local tiles (causal inside the block)
    const uint32_t lane_base = tmem + ((uint32_t)(quarter * 32) << 16);
    const uint32_t key7 = (uint32_t)(row_in_tile & 7);
    bool ok = __all_sync(0xffffffffu, bwd_wait(&sm.q_full, 0, abort));
    // delta (dO from the tile in shared memory: 128-byte lines of 16-byte chunks, XOR-swizzled)
    float neg_delta_s = 0.f;
    if (ok) {
      float acc[4] = {0.f, 0.f, 0.f, 0.f};
      const uint32_t line = smem_u32(sm.dO) + (uint32_t)row_in_tile * 128;
#pragma unroll
      for (int i = 0; i < D / 8; ++i) {
        uint32_t ys[4];
        ld_shared_v4(line + (uint32_t)(i >> 3) * 16384 + (((uint32_t)(i & 7) ^ key7) * 16), ys[0], ys[1], ys[2], ys[3]);
        const uint32_t xs[4] = {o_row[i].x, o_row[i].y, o_row[i].z, o_row[i].w};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          acc[e] = fmaf(__uint_as_float(xs[e] << 16), __uint_as_float(ys[e] << 16), acc[e]);
          acc[e] = fmaf(__uint_as_float(xs[e] & 0xffff0000u), __uint_as_float(ys[e] & 0xffff0000u), acc[e]);
        }
      }
      neg_delta_s = -((acc[0] + acc[1]) + (acc[2] + acc[3])) * dm.scale;
    }
    HGA_TRACE_POINT(10);
    int n = n_lt + 1, n_a = n_lt, n_far_keys = 0;      // (bounds that do until the list is known)
    // (e^x as 2^(x log2 e), x = S*scale - LSE rounded once: no common factor of log2 e rounds S and LSE apart)
    const uint64_t scale_2 = pack_f32x2(dm.scale, dm.scale), neg_lse_2 = pack_f32x2(-row_lse, -row_lse);
    const uint64_t neg_delta_s_2 = pack_f32x2(neg_delta_s, neg_delta_s);
    const uint64_t log2e_2 = pack_f32x2(1.4426950408889634f, 1.4426950408889634f);
    const uint32_t dp_addr = lane_base + kColDP;
    const uint32_t a_line = smem_u32(sm.a) + (uint32_t)row_of_item * 128, b_line = smem_u32(sm.b) + (uint32_t)row_of_item * 128;
    // this row's 16 keys of chunk c (four to a tile) in a term's tile: two 16-byte pieces, XOR-swizzled
    auto put = [&](uint32_t line, int c, const uint32_t* w) {
#pragma unroll
      for (int q = 0; q < 2; ++q)
        st_shared_v4(line + (((uint32_t)(2 * c + q) ^ key7) * 16), w[4 * q], w[4 * q + 1], w[4 * q + 2], w[4 * q + 3]);
    };
    uint32_t staged_phase = 0, rounds = 0;
    for (int j = 0; j < n && ok; ++j) {
      if (j == n_lt) {
        ok = __all_sync(0xffffffffu, bwd_wait(&sm.info_full, 0, abort));
        if (!ok) break;
        counts(sm.n_far, sm.first_active, n, n_a);
        n_far_keys = sm.n_far * 8;
        if (j >= n) break;
      }
      const int vis = j < n_lt ? limit - kKT * j : n_far_keys - kKT * (j - n_lt);
      const bool dkv = j >= n_lt && j >= n_a;
      const uint32_t s_addr = lane_base + s_col(j);
      // P of two neighbouring keys
      auto weights = [&](int key, uint32_t s0, uint32_t s1, float& p0, float& p1) {
        float a0, a1;
        unpack_f32x2(mul_f32x2(fma_f32x2(pack_f32x2(__uint_as_float(s0), __uint_as_float(s1)), scale_2, neg_lse_2), log2e_2), a0, a1);
        p0 = fast_exp2(a0);
        p1 = fast_exp2(a1);
        if (vis < kKT) {           // diagonal / ragged tile only
          if (key >= vis) p0 = 0.f;
          if (key + 1 >= vis) p1 = 0.f;
        }
      };
      ok = __all_sync(0xffffffffu, bwd_wait(&sm.s_full[j & 1], (j >> 1) & 1, abort));
      HGA_TRACE_POINT(11);
      if (ok) ok = __all_sync(0xffffffffu, bwd_wait(&sm.dp_full, j & 1, abort));
      if (!ok) break;
      tc_fence_after_sync();
      HGA_TRACE_POINT(13);
      if (twice) {                           // (dS of the keys that the row's other thread takes)
        const uint32_t zero[32] = {};
        tmem_st32(dp_addr + 32 - 16 * c_first, zero);
      }
#pragma unroll 1
      for (int c0 = c_first; c0 < c_end; c0 += 2)
#pragma unroll
      for (int c = c0; c < c0 + 2; ++c) {    // 16 keys at a time
        uint32_t sv[16], dp[16], out[16], p1[8], p2[8];
        tmem_ld16(s_addr + 16 * c, sv);
        tmem_ld16(dp_addr + 16 * c, dp);
        tmem_wait_ld();
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          float x0, x1, d0, d1;
          weights(16 * c + 2 * i, sv[2 * i], sv[2 * i + 1], x0, x1);
          const uint64_t g2 = fma_f32x2(pack_f32x2(__uint_as_float(dp[2 * i]), __uint_as_float(dp[2 * i + 1])), scale_2, neg_delta_s_2);
          unpack_f32x2(mul_f32x2(pack_f32x2(x0, x1), g2), d0, d1);
          out[i] = next_term(d0, d1);
          out[8 + i] = pack_bf16(d0, d1);
          if (dkv) {
            p1[i] = next_term(x0, x1);
            p2[i] = pack_bf16(x0, x1);
          }
        }
        // dS's two terms over the dP columns just read (8 columns each): the A operands of dQ
        tmem_st16(dp_addr + 16 * c, out);
        if (dkv) {
          put(a_line, c, p1);
          put(b_line, c, p2);
        }
      }
      tmem_wait_st();
      tc_fence_before_sync();
      if (!dkv) {
        mbar_arrive_warp(&sm.ds_full);
        HGA_TRACE_POINT(14);
        continue;
      }
      // ---- dK/dV tile
      fence_proxy_async_smem();
      mbar_arrive_warp(&sm.ds_full);
      HGA_TRACE_POINT(17);
      auto round_done = [&]() {
        ok = __all_sync(0xffffffffu, bwd_wait(&sm.round_done, rounds, abort));
        rounds ^= 1u;
        if (ok) tc_fence_after_sync();
        return ok;
      };
      auto hand_over_round = [&]() {
        tc_fence_before_sync();
        fence_proxy_async_smem();
        mbar_arrive_warp(&sm.round_full);
      };
      // a term of dS from tensor memory into a tile
      auto put_ds = [&](uint32_t line, int term) {
#pragma unroll 1
        for (int c = c_first; c < c_end; ++c) {
          uint32_t ds[8];
          tmem_ld8(dp_addr + 16 * c + 8 * term, ds);
          tmem_wait_ld();
          put(line, c, ds);
        }
      };
      {
        uint32_t p3[32];                     // ready when the first round is over
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          if (c_first + k >= c_end) break;
          const int c = c_first + k;
          uint32_t sv[16];
          tmem_ld16(s_addr + 16 * c, sv);
          tmem_wait_ld();
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            float x0, x1;
            weights(16 * c + 2 * i, sv[2 * i], sv[2 * i + 1], x0, x1);
            next_term(x0, x1);
            next_term(x0, x1);
            p3[8 * k + i] = pack_bf16(x0, x1);
          }
        }
        if (!round_done()) break;
#pragma unroll
        for (int k = 0; k < 4; ++k)
          if (c_first + k < c_end) put(a_line, c_first + k, p3 + 8 * k);
      }
      put_ds(b_line, 0);
      hand_over_round();
      if (!round_done()) break;
      put_ds(a_line, 1);
      hand_over_round();
      if (!round_done()) break;
      HGA_TRACE_POINT(16);
      // (the band kernel, which precedes this one in the stream, stores its dK/dV rows plainly: the adds below must
      // come after it; a no-op unless the launch carried the programmatic-serialization attribute)
      if (j == n_a) pdl_wait();
      auto wait_staged = [&]() {           // all 128 row threads have arrived
        ok = __all_sync(0xffffffffu, bwd_wait(&sm.staged, staged_phase, abort));
        staged_phase ^= 1u;
        return ok;
      };
      // the lane's 32 columns (keys) of an accumulator, as element `row_in_tile` of key rows of 512 bytes
      auto stage = [&](uint32_t buf, uint32_t col) {
        uint32_t x[32];
        tmem_ld32(lane_base + col, x);
        tmem_wait_ld();
        const uint32_t base = buf + (uint32_t)row_in_tile * 4;
#pragma unroll
        for (int i = 0; i < 32; ++i) st_shared_b32(base + (uint32_t)i * 512, x[i]);
      };
      auto hand_over = [&]() {             // what this thread has written is complete and visible to bulk copies
        fence_proxy_async_smem();
        mbar_arrive_warp(&sm.staged);
        return wait_staged();
      };
      auto buffers_read = [&]() {          // the terms' tiles may be written again
        tma_store_wait_read();
        __syncwarp();
        mbar_arrive_warp(&sm.staged);
        return wait_staged();
      };
      const uint32_t dv_col = s_col(j + 1), dk_col = s_col(j), buf_a = smem_u32(sm.a), buf_b = smem_u32(sm.b);
      // row of octet o (of this tile) in the segment's dK and dV, -1: gets nothing from here
      auto grad_row = [&](int o) {
        const int far_o = 8 * (j - n_lt) + o;
        return far_o >= sm.first_active && far_o < sm.n_far ? sm.rows[j & 3][o] - sg.k0 - sg.H : -1;
      };
      const int64_t kv_base = row_base(dm, sg, b) * dm.Hkv + (int64_t)h * sg.S;
      if constexpr (D == 64) {
        // every GEMM is done, the terms' tiles are free: each takes 32 keys x (64 floats of dV | 64 of dK) (lanes 0-63 hold dV^T,
        // lanes 64-127 dK^T); a warp adds its half of each buffer's rows, 256 bytes per instruction
        const uint32_t col = quarter < 2 ? dv_col : dk_col;
        stage(buf_a, col);
        stage(buf_b, col + 32);
        tc_fence_before_sync();
        mbar_arrive_warp(&sm.acc_read);
        if (!hand_over()) break;
        const int hf = quarter >> 1, row = grad_row(4 * hf + (lane >> 3));
        if (row >= 0)
          bulk_reduce_add_f32(((quarter & 1) ? dK : dV) + (kv_base + row + (lane & 7)) * D, (hf ? buf_b : buf_a) + (uint32_t)lane * 512 + (quarter & 1) * 256, D * 4);
        tma_store_commit();
        if (!buffers_read()) break;
      } else {
        // dV, then dK: 64 key rows over both tiles; an octet of them is 4 KB of consecutive memory on both sides
#pragma unroll
        for (int which = 0; which < 2; ++which) {
          stage(buf_a, which ? dk_col : dv_col);
          stage(buf_b, (which ? dk_col : dv_col) + 32);
          if (which == 1) {
            tc_fence_before_sync();
            mbar_arrive_warp(&sm.acc_read);
          }
          if (!hand_over()) break;
          if (lane < 2) {
            const int o = 2 * quarter + lane, row = grad_row(o);
            if (row >= 0) bulk_reduce_add_f32((which ? dK : dV) + (kv_base + row) * D, buf_a + (uint32_t)o * 4096, 4096);
            tma_store_commit();
          }
          if (!buffers_read()) break;
        }
        if (!ok) break;
      }
      HGA_TRACE_POINT(18);
    }
    if (ok) ok = __all_sync(0xffffffffu, bwd_wait(&sm.dq_done, 0, abort));
    HGA_TRACE_POINT(20);
    if (ok) {
      // dQ epilogue through shared memory and TMA: a thread's own row is 2 D bytes away from its neighbour's, so direct
      // 16-byte stores would touch 32 different sectors per instruction.  The rows go into Q's shared memory (all
      // GEMMs that read it are complete) in the swizzled [panel][128 rows][128 B] layout and leave as boxes.
      tc_fence_after_sync();
      // the two lanes of a row meet in the terms' tiles (64 rows of 4 D bytes, 16-byte pieces XOR-swizzled)
      const uint32_t partner = smem_u32(sm.a) + (uint32_t)row_of_item * (4 * D);
      if (twice) {
        if (quarter >= 2) {
#pragma unroll 1
          for (int c = 0; c < D / 32; ++c) {
            uint32_t x[32];
            tmem_ld32(lane_base + kColDQ + 32 * c, x);
            tmem_wait_ld();
#pragma unroll
            for (int i = 0; i < 8; ++i) st_shared_v4(partner + 128 * c + (((uint32_t)i ^ key7) * 16), x[4 * i], x[4 * i + 1], x[4 * i + 2], x[4 * i + 3]);
          }
        }
        mbar_arrive_warp(&sm.staged);
        ok = __all_sync(0xffffffffu, bwd_wait(&sm.staged, staged_phase, abort));
      }
      if (!twice || quarter < 2)
#pragma unroll 1
      for (int c = 0; c < D / 32; ++c) {
        uint32_t x[32];
        tmem_ld32(lane_base + kColDQ + 32 * c, x);
        tmem_wait_ld();
        if (twice) {
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            uint32_t y[4];
            ld_shared_v4(partner + 128 * c + (((uint32_t)i ^ key7) * 16), y[0], y[1], y[2], y[3]);
#pragma unroll
            for (int e = 0; e < 4; ++e) x[4 * i + e] = __float_as_uint(__uint_as_float(x[4 * i + e]) + __uint_as_float(y[e]));
          }
        }
        const uint32_t line = smem_u32(sm.q) + (uint32_t)(c >> 1) * 16384 + (uint32_t)row_in_tile * 128;
#pragma unroll
        for (int i = 0; i < 4; ++i)
          st_shared_v4(line + (((uint32_t)(4 * (c & 1) + i) ^ key7) * 16),
                       pack_bf16(__uint_as_float(x[8 * i]), __uint_as_float(x[8 * i + 1])),
                       pack_bf16(__uint_as_float(x[8 * i + 2]), __uint_as_float(x[8 * i + 3])),
                       pack_bf16(__uint_as_float(x[8 * i + 4]), __uint_as_float(x[8 * i + 5])),
                       pack_bf16(__uint_as_float(x[8 * i + 6]), __uint_as_float(x[8 * i + 7])));
      }
      fence_proxy_async_smem();
      mbar_arrive_warp(&sm.dq_staged);
      if (warp == 2 && ok && lane < 2 * kPanels && bwd_wait(&sm.dq_staged, 0, abort)) {      // all 128 rows are in shared memory
        const int hf = lane & 1, panel = lane >> 1, r0 = mt * 128 + 64 * hf, a = dm.by_Bq(r0);
        if (r0 < dm.rows) {
          tma_store_5d(&map_dq, sm.q + panel * 16384 + hf * 8192, 0, qrow + r0 - a * dm.Bq, panel, h * dm.G + a, b);
          tma_store_commit();
          tma_store_wait_read();      // (the source tile has been read; the writes complete before the grid does)
        }
      }
    }
  }
  HGA_TRACE_POINT(30);

  // Common exit.  Roles leave their warps diverged, so every warp reconverges first: a block barrier reached by
  // part of a warp would count that warp as arrived.
  __syncwarp();
  tc_fence_before_sync();
  __syncthreads();
  HGA_TRACE_POINT(31);
  HGA_TRACE_DUMP;
  if (tid == 0 && sm.abort && status_word) atomicOr(status_word, HGA_ABORT_CODE(3, sm.abort));
  if (warp == 1) {
    __syncwarp();
    if (sm.abort) {
      // given up (known for certain behind the barrier): GEMMs already issued may still be writing tensor memory; wait
      // (bounded) until the tensor pipe has run dry before the columns are given back
      mma_commit_w(elect_one(), &sm.drain);
      mbar_wait(&sm.drain, 0);
      __syncwarp();
    }
    tmem_dealloc(tmem, kTmemCols);
  }
}

template <int D, class Segs>
static int launch_terms(const Dims& dm, SegTable* table, const Segs& segs, int64_t units, const void* Q, const void* K, const void* V, const void* O, const float* LSE,
                              const void* dO, const int32_t* group_idx, const int32_t* n_groups, void* dQ, float* dK,
                              float* dV, int32_t* status_word, cudaStream_t st) {
  CUtensorMap mq, mdo, mk, mv, mdq;
  const uint32_t box[5] = {64, 8, (uint32_t)(D / 64), 1, 1};
  const uint32_t box_q[5] = {64, 64, 1, 1, 1};
  const uint64_t dq[5] = {64, (uint64_t)dm.rows_q, (uint64_t)(D / 64), (uint64_t)dm.Hq, (uint64_t)dm.B};
  const uint64_t dk[5] = {64, (uint64_t)dm.rows_k, (uint64_t)(D / 64), (uint64_t)dm.Hkv, (uint64_t)dm.B};
  const uint64_t sq[4] = {(uint64_t)dm.qs[2] * 2, 128, (uint64_t)dm.qs[1] * 2, (uint64_t)dm.qs[0] * 2};
  const uint64_t so[4] = {(uint64_t)dm.os[2] * 2, 128, (uint64_t)dm.os[1] * 2, (uint64_t)dm.os[0] * 2};
  const uint64_t sk[4] = {(uint64_t)dm.ks[2] * 2, 128, (uint64_t)dm.ks[1] * 2, (uint64_t)dm.ks[0] * 2};
  const uint64_t sv[4] = {(uint64_t)dm.vs[2] * 2, 128, (uint64_t)dm.vs[1] * 2, (uint64_t)dm.vs[0] * 2};
  if (encode_tensor_map_bf16(&mq, Q, 5, dq, sq, box_q, true) ||
      encode_tensor_map_bf16(&mdo, dO, 5, dq, so, box_q, true) ||
      encode_tensor_map_bf16(&mdq, dQ, 5, dq, sq, box_q, true) ||
      encode_tensor_map_bf16(&mk, K, 5, dk, sk, box, true) ||
      encode_tensor_map_bf16(&mv, V, 5, dk, sv, box, true))
    return HGA_ERR_UNSUPPORTED;
  const size_t smem = sizeof(SweepSmem<D>) + 1024;
  // (two CTAs per SM need the largest shared-memory carve-out)
  int rc = ensure_dynamic_smem(reinterpret_cast<const void*>(&k_attn_bwd_terms_sm100<D, Segs>), smem, true);
  if (rc) return rc;
  // dK/dV of the local band first: plain stores that cover every row of the active segment; this kernel then adds
  // the contributions of the keys before the band.  Launched with programmatic serialization behind the band kernel: it
  // waits for it only before the first add.
  rc = launch_attn_bwd_band_sm100(dm, table, Q, K, V, O, LSE, dO, dK, dV, status_word, st);
  if (rc != HGA_OK) return rc;
  if (table) units = number_units(*table, [&](const Segment& g) { return (int64_t)dm.B * dm.Hkv * (g.S / dm.Bq) * ((dm.rows + 127) / 128); });
  PdlLaunch cfg((unsigned)units, kThreads, smem, st, dm.flags);
  const cudaError_t e = cudaLaunchKernelEx(&cfg.c, k_attn_bwd_terms_sm100<D, Segs>, mq, mdo, mk, mv, mdq, (const uint16_t*)O, LSE,
                                           group_idx, n_groups, dm, dK, dV, status_word, segs);
  count_launch(HGA_KERNELS_BWD_TENSOR);
  return record_cuda(e);
}

int launch_attn_bwd_terms_sm100(const Dims& dm, SegTable* segs, const void* Q, const void* K, const void* V, const void* O, const float* LSE,
                              const void* dO, const int32_t* group_idx, const int32_t* n_groups, void* dQ, float* dK,
                              float* dV, int32_t* status_word, cudaStream_t st) {
  const int64_t units = (int64_t)dm.B * dm.Hkv * dm.NQB * ((dm.rows + 127) / 128);
#define HGA_TERMS_ARGS(table, segs) dm, table, segs, units, Q, K, V, O, LSE, dO, group_idx, n_groups, dQ, dK, dV, status_word, st
  if (!segs)
    return dm.d == 64 ? launch_terms<64>(HGA_TERMS_ARGS(nullptr, OneSegment{})) : launch_terms<128>(HGA_TERMS_ARGS(nullptr, OneSegment{}));
  return dm.d == 64 ? launch_terms<64>(HGA_TERMS_ARGS(segs, *segs)) : launch_terms<128>(HGA_TERMS_ARGS(segs, *segs));
#undef HGA_TERMS_ARGS
}

}  // namespace hga
