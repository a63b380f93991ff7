// hga_attn_fwd for sm_100a: routed exact-token attention as a TMA-gather-fed tcgen05 / TMEM
// flash-style kernel (Section 2.1 item 3).
//
// Work unit (one CTA): one 128-row M-tile of one item (b, kv head, query block) swept over the item's routed key set
// in 128-key tiles.  A CTA takes half of an SM (98 KB of shared memory at head_dim 128, 256 TMEM columns), so two CTAs --
// usually the two M-tiles of one item, which then share their K/V gather through L2 -- run on an SM at once: one
// CTA's exponentials overlap the other's GEMMs, and one CTA's set-up and epilogue the other's main loop.
// Keys are addressed in "octets" (8 consecutive tokens = one 8-row 128-byte-swizzle atom per 64-element panel), local
// window and causal block first, then sink and selected groups: the local octets are known without the routing list,
// so their copies start at once and the list is fetched and checked behind the first tile (building a table from it
// first kept a CTA of the 16K layer from its first GEMM for 3k of its 33k cycles).  A tile is 16 octets, one TMA box
// each for K and for V; octets past the end of the set load an out-of-range row and arrive as zeros.
//
// Why 128-key tiles: an N = 64 tcgen05.mma with both operands in shared memory costs nearly as much as one with N = 128,
// so S = Q K^T over 64-key tiles bound the kernel (24 instructions a tile for the two CTAs of an SM, 1.9k cycles).
// S is single-buffered (128 of the 256 columns; O takes the rest); the chain S -> exponentials -> P V -> next S of
// one CTA is covered by the other CTA's, and kept short by TWO threads per row.  hga_attn_fwd, 64-key tiles with one
// thread per row and a running maximum -> this: 16K layer (512 CTAs of 768 keys) 45.2 -> 39.3 us, 2K layer 31.0 -> 27.3,
// 4 x 64K (2560 keys) 865 -> 830 (before the second terms, see below).
//
// What bounds it: a tile's chain takes ~4.3k cycles, of which the exponentials of both CTAs need 2.0k of the special-function
// unit and their GEMMs 2.0k of the tensor pipe, half overlapped.  At 4 x 64K the board's power limit on top.
//
// Warp roles (384 threads, 80 registers per thread):
//   warps 0, 2   producers: octets 0-7 / 8-15 of every K and V tile (a box costs its issuing warp ~100 cycles)
//   warp 1       MMA issuer: S = Q K^T (smem x smem), O += P V (P from TMEM)
//   warp 3       Q, then the check of the routing list
//   warps 4-11   softmax, two threads per row (TMEM lane = row), 32 keys each of both halves of a tile; the epilogue
// TMEM (256 columns): S (128), P (bf16) over the S columns just read, per 16 keys 8 columns and 8 of second terms | O.
//
// Softmax: every exponential of a row is taken against ONE reference, the row's maximum over the first tile (which holds
// the start of the local window, visible to every row).  bf16 and fp32 share an exponent range of 2^127 and O is divided
// by the sum in the end, so a later, larger logit costs no precision until it exceeds the reference by tens of binary
// orders; no maximum is looked for in later tiles, and no sum is ever rescaled.
// What the one reference does cost is the exactness of a dominant weight: against its own tile's maximum, which a running
// reference is raised to, it is 1, here it has a rounding error of 2^-9 like any other.  Where 32 keys of some row
// outweigh the reference by more than 64, that half of the tile gets P in TWO bf16 terms (value and remainder, 2^-17), the
// second ones a GEMM of their own; every warp stores the second terms, zeros elsewhere.  16K layer (needles in one block
// of eight: 1 % of the half-tiles): error of O against fp64 2.11e-3 with one term, 1.82e-3 so, 2.06e-3 with a running
// reference; hga_attn_fwd 39.8 -> 41.3 us (two terms everywhere: 1.66e-3, which is O's own rounding, and 43.5 us).
// kTwoTerms kernels use them everywhere (see two_terms()).  Their M-tiles of up to 64 rows have the rows TWICE, in lanes 0-63
// and 64-127; a row's lanes take the first and the second half of every tile, against the same reference, with zeros in
// the other half's columns, and O and the sums of the two are added in the end.  (With lanes 64-127 empty, half of the SM's
// sub-cores did all the exponentials: 16 heads of 64 142.3 us a whole step, 138.7 so.)
// Where that does not hold for some row of
// the M-tile (a sum past 2^80, i.e. a logit 55 nats above the first tile's; a weight past 2^16 that took V out of the fp32
// range; no finite logit in the first tile) the CTA goes over its keys again, twice: for the rows' true maxima, then
// with those as references.  That is one tile after another with nothing overlapped, but on the tensor cores and for all
// rows at once, so its cost is bounded by a small multiple of the first pass whatever the inputs are.  A row whose sum is
// not a number has no finite answer and is written as it is.
#include "hga_bwd_sm100.cuh"
#include "hga_common.cuh"
#include "hga_octets.cuh"
#include "hga_sm100.cuh"
#include "hga_trace.cuh"

#include <type_traits>

namespace hga {

using namespace sm100;

namespace {

constexpr int kFwdThreads = 384;
constexpr int kFT = 128;                      // keys per tile
constexpr float kSumLimit = 1.2e24f;          // 2^80
constexpr float kWeightLimit = 65536.f;       // (a smaller sum means that no weight exceeded it)
constexpr float kTwoTermSum = 64.f;           // 32 keys that together outweigh the reference by so much get two terms

template <int D>
struct FwdSmem {
  static constexpr int kQBytes = 128 * D * 2;
  static constexpr int kTileBytes = kFT * D * 2;
  static constexpr uint32_t kColO = 128;       // TMEM: S at 0, O at 128
  alignas(1024) uint8_t q[kQBytes];            // (the epilogue stages O here)
  alignas(1024) uint8_t k[kTileBytes];         // (and exchanges the row sums here)
  alignas(1024) uint8_t v[kTileBytes];
  float mx[2][128];                            // first tile: the two threads' maxima of a row
  uint64_t q_full, k_full, v_full, v_empty, s_full, p_full[2], info_full, o_done, o_staged, drain;
  uint64_t again_copied, again_multiplied;     // second passes
  uint32_t tmem_base;
  int n_far, n_listed;
  bool clean;
  volatile int second_terms[2];                // number (from 1) of the last tile whose half needs the weights' second terms
  volatile int again;                          // some row asks for the second passes
  volatile int abort;
};

// What a CTA works on
struct Place {
  Segment sg;
  int mt, b, h, qb, qrow;               // M-tile inside the item, item; the block's first row in Q and O
  Window w;
  template <class Segs>
  __device__ Place(const Dims& dm, const Segs& segs, int cta_id) {
    // Launch order: late query blocks first -- where the history is short they see the most keys, so the cheapest CTAs are
    // the ones that fill the last wave.
    const int n_mt_item = (rows_padded(dm) + 127) / 128, n_bh = dm.B * dm.Hkv;
    int cta;
    sg = segment_of(dm, segs, cta_id, cta);
    const int unit = dm.by_mt(cta), i = dm.by_bh(unit), bh = unit - i * n_bh;
    mt = cta - unit * n_mt_item;
    qb = dm.by_Bq(sg.S) - 1 - i;
    b = dm.by_Hkv(bh);
    h = bh - b * dm.Hkv;
    qrow = sg.q0 + qb * dm.Bq;
    w = window_at(dm, sg.H + qb * dm.Bq);
  }
  __device__ int64_t item(const Dims& dm) const { return item_base(dm, sg, b) + h * dm.by_Bq(sg.S) + qb; }
};

// Whether an M-tile's rows are there twice
template <bool kTwoTerms>
__device__ __forceinline__ bool rows_twice(const Dims& dm, const Place& pl) { return kTwoTerms && rows_padded(dm) - 128 * pl.mt <= 64; }

// The row of a softmax thread: rows of the item are every head's Bq rows padded to whole octets (padding rows compute
// garbage in their own TMEM lanes and are never stored)
struct Row {
  int hw, row, r, a, t;                 // which half of every 64 keys; TMEM lane; row inside the item = (query head, token)
  bool real;
  __device__ Row(const Dims& dm, const Place& pl, int tid, bool twice) {
    const int warp = tid >> 5;
    hw = (warp - 4) >> 2;
    row = (warp & 3) * 32 + (tid & 31);
    r = pl.mt * 128 + (twice ? row & 63 : row);
    a = dm.by_Bq_pad(r);
    t = r - a * bq_padded(dm);
    real = r < rows_padded(dm) && t < dm.Bq;
  }
};

// A thread index or block number that the compiler does not know to be the one it has already worked with: what follows
// from it is worked out afresh, instead of being kept in registers through the main loop
__device__ __forceinline__ int again_tid() { int x; asm volatile("mov.u32 %0, %%tid.x;" : "=r"(x)); return x; }
__device__ __forceinline__ int again_cta() { int x; asm volatile("mov.u32 %0, %%ctaid.x;" : "=r"(x)); return x; }

// A softmax thread's half of its row of O = (accumulators) / l_mma, and LSE from l and the reference m (log2 units).  O's columns
// (D/2)*hw .. are at head_dim 128 a panel each; rows go through Q's shared memory ([panel][128 rows][128 B], swizzled; every
// GEMM that reads Q is complete) and leave as boxes, or are stored directly where boxes do not fit.  Returns whether
// the accumulators are finite.  partner: the other lane's accumulators in shared memory (see share_row), 0 if there are none.
template <int D>
__device__ __forceinline__ bool store_row(FwdSmem<D>& sm, const Dims& dm, const Place& pl, const Row& rw, uint32_t tmem, float l, float l_mma, float m,
                                          uint16_t* O, float* LSE, uint32_t partner = 0) {
  constexpr int kCols = D / 2;
  const bool boxes = dm.Bq % 64 == 0;
  const uint32_t lane_base = tmem + ((uint32_t)(rw.row & 96) << 16);
  const float inv = 1.f / l_mma;
  const int hq = pl.h * dm.G + rw.a;
  uint16_t* const orow = O + pl.b * dm.os[0] + (int64_t)hq * dm.os[1] + (int64_t)(pl.qrow + rw.t) * dm.os[2];
  if (rw.real && rw.hw == 0)
    LSE[row_base(dm, pl.sg, pl.b) * dm.Hq + (int64_t)hq * pl.sg.S + pl.qb * dm.Bq + rw.t] = (log2f(l) + m) * 0.6931471805599453f;
  const uint32_t line = smem_u32(sm.q) + (uint32_t)(kCols * rw.hw / 64) * 16384 + (uint32_t)rw.row * 128;
  uint64_t finite = pack_f32x2(0.f, 0.f);                 // stays zero as long as every element is finite
#pragma unroll 1
  for (int c = 0; c < kCols / 32; ++c) {
    const int col = kCols * rw.hw + 32 * c;
    uint32_t y[32];
    tmem_ld32(lane_base + FwdSmem<D>::kColO + col, y);
    tmem_wait_ld();
    if (partner) {
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        uint32_t x[4];
        ld_shared_v4(partner + 4 * col + (((uint32_t)i ^ (uint32_t)(rw.row & 7)) * 16), x[0], x[1], x[2], x[3]);
#pragma unroll
        for (int e = 0; e < 4; ++e) y[4 * i + e] = __float_as_uint(__uint_as_float(y[4 * i + e]) + __uint_as_float(x[e]));
      }
    }
#pragma unroll
    for (int i = 0; i < 16; ++i)
      finite = fma_f32x2(pack_f32x2(__uint_as_float(y[2 * i]), __uint_as_float(y[2 * i + 1])), pack_f32x2(0.f, 0.f), finite);
    if (rw.real) {
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        uint32_t pk[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) pk[e] = pack_bf16(__uint_as_float(y[8 * i + 2 * e]) * inv, __uint_as_float(y[8 * i + 2 * e + 1]) * inv);
        if (boxes) st_shared_v4(line + (((uint32_t)((col & 63) / 8 + i) ^ (uint32_t)(rw.row & 7)) * 16), pk[0], pk[1], pk[2], pk[3]);
        else *reinterpret_cast<uint4*>(orow + col + 8 * i) = make_uint4(pk[0], pk[1], pk[2], pk[3]);
      }
    }
  }
  float x0, x1;
  unpack_f32x2(finite, x0, x1);
  return x0 + x1 == 0.f;
}

// Where a row's two lanes meet: 4 D bytes per row in V's shared memory, 16-byte pieces XOR-swizzled; the thread's half of the columns
template <int D>
__device__ __forceinline__ uint32_t shared_row(FwdSmem<D>& sm, const Row& rw) { return smem_u32(sm.v) + (uint32_t)(rw.row & 63) * (4 * D); }
template <int D>
__device__ __forceinline__ void share_row(FwdSmem<D>& sm, const Row& rw, uint32_t tmem) {
#pragma unroll 1
  for (int c = 0; c < D / 64; ++c) {
    const int col = D / 2 * rw.hw + 32 * c;
    uint32_t y[32];
    tmem_ld32(tmem + ((uint32_t)(rw.row & 96) << 16) + FwdSmem<D>::kColO + col, y);
    tmem_wait_ld();
#pragma unroll
    for (int i = 0; i < 8; ++i)
      st_shared_v4(shared_row(sm, rw) + 4 * col + (((uint32_t)i ^ (uint32_t)(rw.row & 7)) * 16), y[4 * i], y[4 * i + 1], y[4 * i + 2], y[4 * i + 3]);
  }
}

// The staged M-tile as boxes of 64 rows x one panel (the first lanes of one warp, after every row has been staged)
template <int D>
__device__ __forceinline__ void store_boxes(FwdSmem<D>& sm, const Dims& dm, const Place& pl, const CUtensorMap& map_o, int lane) {
  const int hf = lane & 1, panel = lane >> 1, r0 = pl.mt * 128 + 64 * hf, a = dm.by_Bq(r0);
  if (lane < 2 * (D / 64) && r0 < dm.rows) {
    tma_store_5d(&map_o, sm.q + panel * 16384 + hf * 8192, 0, pl.qrow + r0 - a * dm.Bq, panel, pl.h * dm.G + a, pl.b);
    tma_store_commit();
    tma_store_wait_read();      // (the source has been read; the writes complete before the grid does)
  }
}

// Q's rows: boxes of 64 rows x one panel, [panel][128 rows][128 B], or octets, [octet][panel][8 rows][128 B], up to 64 of them
// twice if asked for; `lane`s of one warp, bytes announced by the caller
template <int D>
__device__ __forceinline__ void copy_q(FwdSmem<D>& sm, const Dims& dm, const Place& pl, const CUtensorMap& map_q, uint64_t* bar, int q_oct, bool twice, int lane) {
  constexpr int kOct = 8 * D * 2, kPanels = D / 64;
  if (dm.Bq % 64 == 0) {
    if (lane < 2 * kPanels && (twice || 8 * (lane & 1) < q_oct)) {
      const int hf = lane & 1, panel = lane >> 1, r = pl.mt * 128 + (twice ? 0 : 64 * hf), a = dm.by_Bq(r);
      tma_load_5d(sm.q + panel * 16384 + hf * 8192, &map_q, bar, 0, pl.qrow + r - a * dm.Bq, panel, pl.h * dm.G + a, pl.b);
    }
  } else if (lane < (twice ? 2 : 1) * q_oct) {
    const int again = lane >= q_oct, oct = lane - again * q_oct;
    const int bq_pad = bq_padded(dm), r = pl.mt * 128 + 8 * oct, a = dm.by_Bq_pad(r);
    tma_load_5d(sm.q + (oct + 8 * again) * kOct, &map_q, bar, 0, pl.qrow + r - a * bq_pad, 0, pl.h * dm.G + a, pl.b);
  }
}

// The M-tile once more, for rows whose exponentials left the range of the first tile's reference: all 384 threads, one tile
// at a time (a block barrier behind every hand-off), first S alone for the rows' maxima, then everything against those.
// The main pass is complete: no copy, GEMM or store of it is in flight, and sm.n_far etc. hold the checked list.
template <int D, class Segs>
__device__ __forceinline__ void passes_with_true_maxima(FwdSmem<D>& sm, const CUtensorMap& map_q, const CUtensorMap& map_k, const CUtensorMap& map_v,
                                                        const CUtensorMap& map_o, const int32_t* group_idx, const Dims& dm, uint16_t* O, float* LSE,
                                                        const Segs& segs, uint32_t tmem) {
  constexpr int kOct = 8 * D * 2;
  const int tid = again_tid(), warp = tid >> 5, lane = tid & 31;
  volatile int* abort = &sm.abort;
  const bool softmax = warp >= 4, boxes = dm.Bq % 64 == 0;
  const int hw = (warp - 4) >> 2, row = (warp & 3) * 32 + lane;         // (as in Row)
  const uint32_t lane_base = tmem + ((uint32_t)(row & 96) << 16);
  const float sl2 = dm.scale * 1.4426950408889634f;
  int n_loc_oct, limit;                              // as in the main pass
  {
    const Place pl(dm, segs, again_cta());
    n_loc_oct = (pl.w.p0 + dm.Bq - pl.w.ls + 7) / 8;
    limit = pl.w.p0 - pl.w.ls + Row(dm, pl, tid, false).t + 1;
  }
  const int n_oct = n_loc_oct + sm.n_far, n_tiles = (n_oct + 15) / 16;

  uint32_t copies = 0, multiplications = 0;          // phases of the two barriers
  bool ok = true;
  auto copied = [&]() { ok = ok && __all_sync(0xffffffffu, bwd_wait(&sm.again_copied, copies++ & 1, abort)); };
  auto multiplied = [&]() { ok = ok && __all_sync(0xffffffffu, bwd_wait(&sm.again_multiplied, multiplications++ & 1, abort)); };
  // a thread that gave up has the others leave behind the next barrier, and the copies in flight a bounded time to land
  auto all_fine = [&]() {
    if (!__syncthreads_or(!ok)) return true;
    if (warp == 0 && lane == 0)
      for (int it = 0; it < 64; ++it) __nanosleep(1000);
    return false;
  };
  // the copies below overwrite what the epilogue has written into Q's and K's place
  fence_proxy_async_smem();
  __syncthreads();
  float m = -INFINITY, l = 0.f, l_mma = 0.f;
#pragma unroll 1
  for (int step = 0; step < 2 * n_tiles; ++step) {
    const bool sums = step >= n_tiles;
    const int j = sums ? step - n_tiles : step;
    if (step == n_tiles) {
      // the row's true maximum, in log2 units
      if (softmax) sm.mx[hw][row] = m;
      __syncthreads();
      if (softmax) m = fmaxf(m, sm.mx[hw ^ 1][row]) * sl2;
    }
    if (warp == 0) {
      const Place pl(dm, segs, again_cta());
      const int q_oct = min(16, rows_padded(dm) / 8 - 16 * pl.mt);
      if (lane == 0) mbar_arrive_expect_tx(&sm.again_copied, (uint32_t)(16 * (sums ? 2 : 1) + (step == 0 ? q_oct : 0)) * kOct);
      __syncwarp();
      if (lane < 16) {
        FarList far(dm, pl.w, group_idx + pl.item(dm) * dm.width);
        far.ng = sm.n_listed; far.n_far = sm.n_far; far.clean = sm.clean;
        const int o = 16 * j + lane;
        const int krow = o < n_loc_oct ? pl.sg.k0 + pl.w.ls + 8 * o : o < n_oct ? pl.sg.k0 + far.row(o - n_loc_oct) : dm.rows_k;
        tma_load_5d(sm.k + lane * kOct, &map_k, &sm.again_copied, 0, krow, 0, pl.h, pl.b);
        if (sums) tma_load_5d(sm.v + lane * kOct, &map_v, &sm.again_copied, 0, krow, 0, pl.h, pl.b);
      }
      if (step == 0) copy_q(sm, dm, pl, map_q, &sm.again_copied, q_oct, false, lane);       // (O may have been staged over Q)
      __syncwarp();
    }
    copied();
    if (warp == 1 && ok) {
      tc_fence_after_sync();
      const uint32_t lead = elect_one();
      const uint64_t q_desc = smem_desc_sw128(smem_u32(sm.q), 16, boxes ? 1024 : kOct), k_desc = smem_desc_sw128(smem_u32(sm.k), 16, kOct);
      const uint32_t q_panel = boxes ? 16384 : 1024;
#pragma unroll 1
      for (int kk = 0; kk < D / 16; ++kk)
        mma_ss_w(lead, tmem, desc_advance(q_desc, (kk >> 2) * q_panel + (kk & 3) * 32), desc_advance(k_desc, (kk >> 2) * 1024 + (kk & 3) * 32),
                 idesc_bf16_f32(128, kFT, 0, 0), kk > 0);
      mma_commit_w(lead, &sm.again_multiplied);
    }
    multiplied();
    if (softmax && ok) {
      tc_fence_after_sync();
      float tile_l = 0.f, tile_l_mma = 0.f;
#pragma unroll 1
      for (int c = 0; c < 4; ++c) {                   // 16 keys at a time
        const int first = 64 * (c >> 1) + 32 * hw + 16 * (c & 1), lo = limit - kFT * j - first, hi = 8 * n_loc_oct - kFT * j - first, end = 8 * n_oct - kFT * j - first;
        uint32_t x[16], pk[16];
        tmem_ld16(lane_base + first, x);
        tmem_wait_ld();
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          float p[2];
#pragma unroll
          for (int u = 0; u < 2; ++u) {
            const int k = 2 * i + u;
            const bool see = (k < lo || k >= hi) && k < end;
            if (!sums && see) m = fmaxf(m, __uint_as_float(x[k]));
            p[u] = see ? fast_exp2(fmaf(__uint_as_float(x[k]), sl2, -m)) : 0.f;
            tile_l += p[u];
          }
          pk[i] = pack_bf16(p[0], p[1]);                // (two terms per weight, see the main pass)
          pk[8 + i] = pack_bf16(p[0] - __uint_as_float(pk[i] << 16), p[1] - __uint_as_float(pk[i] & 0xffff0000u));
#pragma unroll
          for (int u = 0; u < 2; ++u) tile_l_mma += __uint_as_float(pk[8 * u + i] << 16) + __uint_as_float(pk[8 * u + i] & 0xffff0000u);
        }
        if (sums) tmem_st16(lane_base + first, pk);
      }
      if (sums) {
        l += tile_l;
        l_mma += tile_l_mma;
        tmem_wait_st();
      }
      tc_fence_before_sync();
    }
    // (also: S has been read, K may be overwritten)
    if (!all_fine()) return;
    if (!sums) continue;
    if (warp == 1) {
      tc_fence_after_sync();
      const uint32_t lead = elect_one();
      const uint64_t v_desc = smem_desc_sw128(smem_u32(sm.v), 1024, kOct);
#pragma unroll 1
      for (int kk = 0; kk < 2 * (kFT / 16); ++kk)
        mma_ts_w(lead, tmem + FwdSmem<D>::kColO, tmem + 8 * kk, desc_advance(v_desc, (uint32_t)(kk >> 1) * 2 * kOct),
                 idesc_bf16_f32(128, D, 0, 1), j > 0 || kk > 0);
      mma_commit_w(lead, &sm.again_multiplied);
    }
    multiplied();
    if (!all_fine()) return;
  }
  // the row's two sums meet, then the epilogue of the main pass
  float* const xchg = reinterpret_cast<float*>(sm.k);
  if (softmax) {
    xchg[hw * 256 + row] = l;
    xchg[hw * 256 + 128 + row] = l_mma;
  }
  __syncthreads();
  const Place pl(dm, segs, again_cta());
  if (softmax) {
    tc_fence_after_sync();
    l += xchg[(hw ^ 1) * 256 + row];
    l_mma += xchg[(hw ^ 1) * 256 + 128 + row];
    store_row(sm, dm, pl, Row(dm, pl, tid, false), tmem, l, l_mma, m, O, LSE);
    fence_proxy_async_smem();
    tc_fence_before_sync();
  }
  __syncthreads();
  if (boxes && warp == 4) store_boxes(sm, dm, pl, map_o, lane);
  __syncwarp();
}

}  // namespace

template <int D, bool kTwoTerms, class Segs>
__global__ void __launch_bounds__(kFwdThreads, 2)
k_attn_fwd_sm100(const __grid_constant__ CUtensorMap map_q, const __grid_constant__ CUtensorMap map_k,
                 const __grid_constant__ CUtensorMap map_v, const __grid_constant__ CUtensorMap map_o,
                 const int32_t* __restrict__ group_idx, const int32_t* __restrict__ n_groups, const Dims dm,
                 uint16_t* __restrict__ O, float* __restrict__ LSE, int32_t* status_word, const __grid_constant__ Segs segs) {
  constexpr int kOct = 8 * D * 2;
  constexpr uint32_t kTmemCols = 256;
  extern __shared__ uint8_t smem_raw[];
  FwdSmem<D>& sm = *reinterpret_cast<FwdSmem<D>*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  HGA_TRACE_DECL(256);
  const Place pl(dm, segs, blockIdx.x);
  const Segment& sg = pl.sg;
  const Window& w = pl.w;
  const int b = pl.b, h = pl.h;
  const int n_local = w.p0 + dm.Bq - w.ls;              // tokens of the local window and the block
  const int n_loc_oct = (n_local + 7) / 8;              // (the last octet may be partial in generation shapes)
  const int n_pre = n_loc_oct / 16;                     // tiles that hold local octets only
  // 64 rows of an M-tile are 64 rows of one head: Q and O travel in boxes of 64 rows x one panel
  const bool boxes = dm.Bq % 64 == 0;
  volatile int* abort = &sm.abort;
  const bool twice = rows_twice<kTwoTerms>(dm, pl);
  FarList far(dm, w, group_idx + pl.item(dm) * dm.width);
  auto n_octets = [&](int n_far) { return n_loc_oct + n_far; };

  if (warp == 0 && lane == 0) {
    mbar_init(&sm.q_full, 1);
    mbar_init(&sm.k_full, 2); mbar_init(&sm.v_full, 2); mbar_init(&sm.v_empty, 1);
    mbar_init(&sm.s_full, 1); mbar_init(&sm.p_full[0], 8); mbar_init(&sm.p_full[1], 8);
    mbar_init(&sm.info_full, 1); mbar_init(&sm.o_done, 1); mbar_init(&sm.o_staged, 8); mbar_init(&sm.drain, 1);
    mbar_init(&sm.again_copied, 1); mbar_init(&sm.again_multiplied, 1);
    sm.second_terms[0] = sm.second_terms[1] = 0;
    sm.again = 0;
    sm.abort = 0;
    fence_barrier_init();
  }
  // Tile j's octet of this lane for the producers (lane < 8), as a row of the K / V tensors
  const int half = warp == 2 ? 1 : 0;
  auto row_of = [&](int j) {
    const int o = 16 * j + 8 * half + (lane & 7);
    if (o < n_loc_oct) return sg.k0 + w.ls + 8 * o;
    return o - n_loc_oct < far.n_far ? sg.k0 + far.row(o - n_loc_oct) : dm.rows_k;     // past the end: out of range -> zeros
  };
  // this producer's boxes of a tile (a tile of up to eight octets needs the first producer only)
  auto copy_tile = [&](uint8_t* dst, const CUtensorMap* map, uint64_t* full, int row, bool any) {
    if (lane == 0) {
      if (any) mbar_arrive_expect_tx(full, 8 * kOct);
      else mbar_arrive(full);
    }
    __syncwarp();
    if (any && lane < 8) tma_load_5d(dst + (8 * half + lane) * kOct, map, full, 0, row, 0, h, b);
  };
  if (warp == 0 || warp == 2 || warp == 3) {
    // Q and a first tile of local octets do not depend on the routing: their copies start before the CTA meets.  Barrier 2
    // makes the mbarrier initialisation above visible to the issuing warps.
    asm volatile("bar.sync 2, 96;" ::: "memory");
    const bool chained = dm.flags & kFlagChained;
    if (!chained) pdl_wait();
    if (warp == 3) {
      const int q_oct = min(16, rows_padded(dm) / 8 - 16 * pl.mt);   // octets of real rows in this M-tile
      if (lane == 0) mbar_arrive_expect_tx(&sm.q_full, (uint32_t)(twice ? 2 * q_oct : q_oct) * kOct);
      __syncwarp();
      copy_q(sm, dm, pl, map_q, &sm.q_full, q_oct, twice, lane);
    } else if (n_pre > 0) {
      const int row = row_of(0);
      copy_tile(sm.k, &map_k, &sm.k_full, row, true);
      copy_tile(sm.v, &map_v, &sm.v_full, row, true);
    }
    __syncwarp();
    if (chained) pdl_wait();                       // (the routing list)
  }
  if (warp == 1) {
    tmem_alloc(&sm.tmem_base, kTmemCols);
    tmem_relinquish();
  }
  __syncwarp();
  tc_fence_before_sync();
  __syncthreads();
  tc_fence_after_sync();
  if (tid == 0) pdl_launch_dependents();

  const uint32_t tmem = sm.tmem_base;
  HGA_TRACE_POINT(1);

  if (warp == 0 || warp == 2) {
    // ------------------------------------------------------------------ producers
    bool ok = true, known = false;
    int n_oct = 16 * n_pre + 1;                    // (enough until the list is known)
    auto wait_for = [&](uint64_t* bar, uint32_t parity, int line = __builtin_LINE()) { return ok = wait_out_of_line(bar, parity, abort, line); };
    auto learn = [&]() {
      known = true;
      if (!wait_for(&sm.info_full, 0)) return false;
      far.ng = sm.n_listed; far.n_far = sm.n_far; far.clean = sm.clean;
      n_oct = n_octets(far.n_far);
      return true;
    };
    auto any_of = [&](int j) { return 16 * j + 8 * half < n_oct; };
    if (n_pre == 0 && learn()) {
      const int row = row_of(0);
      copy_tile(sm.k, &map_k, &sm.k_full, row, any_of(0));
      copy_tile(sm.v, &map_v, &sm.v_full, row, any_of(0));
    }
    for (int j = 1; ok; ++j) {                     // tile j: K behind S(j-1), V behind P V of tile j-1
      if (j >= n_pre && !known && !learn()) break;
      if (16 * j >= n_oct) break;
      const int row = row_of(j);
      const bool any = any_of(j);
      if (!wait_for(&sm.s_full, (j - 1) & 1)) break;
      copy_tile(sm.k, &map_k, &sm.k_full, row, any);
      if (!wait_for(&sm.v_empty, (j - 1) & 1)) break;
      copy_tile(sm.v, &map_v, &sm.v_full, row, any);
      HGA_TRACE_POINT(2);
    }
    if (*abort && lane == 0) {
      // giving up: give the copies still in flight time to land before shared memory is released
      for (int it = 0; it < 64; ++it) __nanosleep(1000);
    }
  } else if (warp == 3) {
    // ------------------------------------------------------------------ routing list
    const bool bad = far.check(dm, n_groups + pl.item(dm), sg.H);
    if (lane == 0) {
      sm.n_listed = far.ng; sm.n_far = far.n_far; sm.clean = far.clean;
      mbar_arrive(&sm.info_full);
      if (bad && status_word) atomicOr(status_word, HGA_STATUS_BAD_INDEX);
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------------ MMA issuer
    // The whole warp runs this branch converged (waits included) and one elected lane issues: see mma_ss_w.
    const uint32_t lead = elect_one();
    auto mma_wait = [&](uint64_t* bar, uint32_t parity) {
      return __all_sync(0xffffffffu, bwd_wait(bar, parity, abort));
    };
    constexpr uint32_t idesc_s = idesc_bf16_f32(128, kFT, 0, 0), idesc_s_half = idesc_bf16_f32(128, kFT / 2, 0, 0);
    constexpr uint32_t idesc_o = idesc_bf16_f32(128, D, 0, 1);
    // Descriptors are built once; inside the loops an MMA costs two integer adds.
    const uint64_t q_desc = smem_desc_sw128(smem_u32(sm.q), 16, boxes ? 1024 : kOct);
    const uint32_t q_panel = boxes ? 16384 : 1024;
    const uint64_t k_desc = smem_desc_sw128(smem_u32(sm.k), 16, kOct);         // K-major B of S = Q K^T
    const uint64_t v_desc = smem_desc_sw128(smem_u32(sm.v), 1024, kOct);       // MN-major B of O += P V
    const uint32_t o_acc = tmem + FwdSmem<D>::kColO;
    auto issue_s = [&](bool whole) {
      const uint32_t idesc = whole ? idesc_s : idesc_s_half;
#pragma unroll
      for (int kk = 0; kk < D / 16; ++kk)
        mma_ss_w(lead, tmem, desc_advance(q_desc, (kk >> 2) * q_panel + (kk & 3) * 32), desc_advance(k_desc, (kk >> 2) * 1024 + (kk & 3) * 32),
                 idesc, kk > 0);
      mma_commit_w(lead, &sm.s_full);                    // also tells the producers that the K tile is free
    };
    // half hf of tile j: 16 keys per step; P of keys 16i .. 16i+15 sits at columns 16i .. 16i+7, its second terms behind it
    auto issue_pv = [&](int hf, int j, bool accumulate) {
#pragma unroll
      for (int kk = 0; kk < 4; ++kk)
        mma_ts_w(lead, o_acc, tmem + 64 * hf + 16 * kk, desc_advance(v_desc, (uint32_t)(4 * hf + kk) * 2 * kOct), idesc_o,
                 (accumulate || kk > 0));
      if (kTwoTerms || sm.second_terms[hf] == j + 1) {
#pragma unroll
        for (int kk = 0; kk < 4; ++kk)
          mma_ts_w(lead, o_acc, tmem + 64 * hf + 16 * kk + 8, desc_advance(v_desc, (uint32_t)(4 * hf + kk) * 2 * kOct), idesc_o, 1);
      }
    };
    int n_oct = 16 * n_pre + 1;                    // (enough until the list is known)
    bool ok = true;
    if (n_pre == 0) {
      ok = mma_wait(&sm.info_full, 0);
      n_oct = n_octets(sm.n_far);
    }
    ok = ok && mma_wait(&sm.q_full, 0) && mma_wait(&sm.k_full, 0);
    if (ok) {
      tc_fence_after_sync();
      issue_s(n_oct > 8);
    }
    HGA_TRACE_POINT(3);
    for (int j = 0; ok; ++j) {
      if (j + 1 == n_pre) {
        ok = mma_wait(&sm.info_full, 0);
        if (!ok) break;
        n_oct = n_octets(sm.n_far);
      }
      const bool more = 16 * (j + 1) < n_oct, whole = n_oct - 16 * j > 8;
      ok = mma_wait(&sm.v_full, j & 1) && mma_wait(&sm.p_full[0], j & 1);
      if (!ok) break;
      tc_fence_after_sync();
      HGA_TRACE_POINT(5);
      issue_pv(0, j, j > 0);
      if (whole) {
        ok = mma_wait(&sm.p_full[1], j & 1);
        if (!ok) break;
        tc_fence_after_sync();
        issue_pv(1, j, true);
      }
      mma_commit_w(lead, more ? &sm.v_empty : &sm.o_done);
      HGA_TRACE_POINT(7);
      if (!more) break;
      ok = mma_wait(&sm.k_full, (j + 1) & 1);      // S(j+1) takes the columns P(j) sat in: ordered after P V of tile j
      if (!ok) break;
      tc_fence_after_sync();
      issue_s(n_oct - 16 * (j + 1) > 8);
      HGA_TRACE_POINT(8);
    }
  } else {
    // ------------------------------------------------------------------ softmax + epilogue
    const Row rw(dm, pl, tid, twice);
    const int hw = rw.hw, row = rw.row;                 // keys 32*hw .. and 64 + 32*hw .. of every tile
    // a warp whose 32 lanes are all padding only keeps the barriers moving
    const bool warp_real = __any_sync(0xffffffffu, rw.real);
    const uint32_t lane_base = tmem + ((uint32_t)(row & 96) << 16);      // the TMEM lanes this warp may touch
    const float sl2 = dm.scale * 1.4426950408889634f;   // softmax scale in log2 units
    const uint64_t sl2_2 = pack_f32x2(sl2, sl2);
    // Column c of tile j is slot 128*j + c of the set: visible below `limit` (causal), masked from there to the end of the
    // local octets, visible again up to the end of the set.
    const int limit = w.p0 - w.ls + rw.t + 1;
    int n_oct = 16 * n_pre + 1;                         // (enough until the list is known)
    uint64_t neg_m2 = pack_f32x2(0.f, 0.f);             // minus the reference (log2 units), twice
    float l = 0.f, l_mma = 0.f;
    bool ok = true;
    for (int j = 0; 16 * j < n_oct; ++j) {
      if (j == n_pre) {
        ok = __all_sync(0xffffffffu, bwd_wait(&sm.info_full, 0, abort));
        if (ok) n_oct = n_octets(sm.n_far);
        if (ok && 16 * j >= n_oct) break;
      }
      if (ok) ok = __all_sync(0xffffffffu, bwd_wait(&sm.s_full, j & 1, abort));
      if (!ok && j > 0) break;
      tc_fence_after_sync();
      HGA_TRACE_POINT(11);
      const bool whole = 8 * n_oct - kFT * j > 64;
      if (j == 0) {
        // the row's reference: its maximum over the first tile (ok or not, every softmax thread meets here once)
        float mx[2] = {-INFINITY, -INFINITY};
        if (ok && warp_real) {
#pragma unroll 1
          for (int c = 0; c < (whole ? 2 : 1); ++c) {
            uint32_t x[32];
            tmem_ld32(lane_base + 64 * c + 32 * hw, x);
            tmem_wait_ld();
            // slots relative to the first of this thread's 32 columns
            const int first = kFT * j + 64 * c + 32 * hw, lo_c = limit - first, hi_c = 8 * n_loc_oct - first, end_c = 8 * n_oct - first;
            if (__all_sync(0xffffffffu, (lo_c >= 32 || hi_c <= 0) && end_c >= 32)) {
#pragma unroll
              for (int i = 0; i < 32; ++i) mx[i & 1] = fmaxf(mx[i & 1], __uint_as_float(x[i]));
            } else {
#pragma unroll
              for (int i = 0; i < 32; ++i)
                if ((i < lo_c || i >= hi_c) && i < end_c) mx[i & 1] = fmaxf(mx[i & 1], __uint_as_float(x[i]));
            }
          }
        }
        const float m = fmaxf(mx[0], mx[1]);
        sm.mx[hw][row] = m;
        asm volatile("bar.sync 1, 256;" ::: "memory");
        const float neg_m = -fmaxf(m, sm.mx[hw ^ 1][row]) * sl2;
        neg_m2 = pack_f32x2(neg_m, neg_m);
        HGA_TRACE_POINT(13);
        if (!ok) break;
      }
      // p = 2^(x*c - m), bf16, over columns already read.  l sums the exact probabilities (for LSE), l_mma the rounded ones
      // the MMA really applies: normalising O by THEIR sum makes the rounding of a dominant weight cancel.
      uint64_t lsum = pack_f32x2(0.f, 0.f), rsum = pack_f32x2(0.f, 0.f);
      // (one copy of the code for both halves: a CTA of a few tiles pays for every line of it once in instruction-cache misses)
#pragma unroll 1
      for (int c = 0; c < 2; ++c) {
        if (c == 1 && !whole) break;
        if (twice && c != row >> 6) {                // (the row's other lane has this half)
          const uint32_t zero[32] = {};
          tmem_st32(lane_base + 64 * c + 32 * hw, zero);
          tmem_wait_st();
        } else if (warp_real) {
          const int first = kFT * j + 64 * c + 32 * hw, lo_c = limit - first, hi_c = 8 * n_loc_oct - first, end_c = 8 * n_oct - first;
          const uint32_t s_addr = lane_base + 64 * c + 32 * hw;
          // Logits of keys that the row does not see become -inf, in a pass of its own where there are any.  (A compare per element in
          // the common code doubled its time; a masked copy of it is that much more for the roles to fetch.)
          const bool masked = !__all_sync(0xffffffffu, (lo_c >= 32 || hi_c <= 0) && end_c >= 32);
          uint32_t see = 0xffffffffu;                  // bit k: key k of the 32 is visible
          if (masked) {
            auto below = [](int n) { return n >= 32 ? 0xffffffffu : n <= 0 ? 0u : (1u << n) - 1u; };
            see = (below(lo_c) | ~below(hi_c)) & below(end_c);
          }
          auto hide = [](uint32_t bits, auto& x) {
#pragma unroll
            for (int i = 0; i < (int)(sizeof(x) / 4); ++i)
              if (!((bits >> i) & 1u)) x[i] = 0xff800000u;
          };
          {
            // weights of two neighbouring keys
            auto weights = [&](uint32_t x0, uint32_t x1, float& p0, float& p1) {
              float a0, a1;
              unpack_f32x2(fma_f32x2(pack_f32x2(__uint_as_float(x0), __uint_as_float(x1)), sl2_2, neg_m2), a0, a1);
              p0 = fast_exp2(a0);
              p1 = fast_exp2(a1);
            };
            auto sum_of = [](uint32_t pk) { return pack_f32x2(__uint_as_float(pk << 16), __uint_as_float(pk & 0xffff0000u)); };
            [[maybe_unused]] bool two = kTwoTerms;
            if constexpr (!kTwoTerms) {
              uint32_t x[32], pk[16];
              uint64_t sum = pack_f32x2(0.f, 0.f);
              tmem_ld32(s_addr, x);
              tmem_wait_ld();
              if (masked) hide(see, x);
#pragma unroll
              for (int i = 0; i < 16; ++i) {
                float p0, p1;
                weights(x[2 * i], x[2 * i + 1], p0, p1);
                sum = add_f32x2(sum, pack_f32x2(p0, p1));
                pk[i] = pack_bf16(p0, p1);
                rsum = add_f32x2(rsum, sum_of(pk[i]));
              }
              lsum = add_f32x2(lsum, sum);
              float x0, x1;
              unpack_f32x2(sum, x0, x1);
              two = __any_sync(0xffffffffu, x0 + x1 > kTwoTermSum);
              if (!two) {
                const uint32_t out[32] = {pk[0], pk[1], pk[2], pk[3], pk[4], pk[5], pk[6], pk[7], 0, 0, 0, 0, 0, 0, 0, 0,
                                          pk[8], pk[9], pk[10], pk[11], pk[12], pk[13], pk[14], pk[15], 0, 0, 0, 0, 0, 0, 0, 0};
                tmem_st32(s_addr, out);
              } else if (lane == 0) {
                sm.second_terms[c] = j + 1;
              }
            }
            // 16 keys with two terms each (S is fetched again rather than kept)
            auto two_terms_of = [&](int k0, uint32_t (&x)[16]) {
              uint32_t out[16];
              if (masked) hide(see >> k0, x);
#pragma unroll
              for (int i = 0; i < 8; ++i) {
                float p0, p1;
                weights(x[2 * i], x[2 * i + 1], p0, p1);
                out[i] = pack_bf16(p0, p1);
                out[8 + i] = pack_bf16(p0 - __uint_as_float(out[i] << 16), p1 - __uint_as_float(out[i] & 0xffff0000u));
                if constexpr (kTwoTerms) lsum = add_f32x2(lsum, pack_f32x2(p0, p1));
                else rsum = add_f32x2(rsum, sum_of(out[8 + i]));
              }
              tmem_st16(s_addr + k0, out);
            };
            if constexpr (kTwoTerms) {
              uint32_t x[2][16];
              tmem_ld16(s_addr, x[0]);
              tmem_ld16(s_addr + 16, x[1]);
              tmem_wait_ld();
              two_terms_of(0, x[0]);
              two_terms_of(16, x[1]);
            } else if (two) {
#pragma unroll 1
              for (int k0 = 0; k0 < 32; k0 += 16) {
                uint32_t x[16];
                tmem_ld16(s_addr + k0, x);
                tmem_wait_ld();
                two_terms_of(k0, x);
              }
            }
          }
          tmem_wait_st();
        }
        tc_fence_before_sync();
        mbar_arrive_warp(&sm.p_full[c]);
      }
      float x0, x1;
      unpack_f32x2(lsum, x0, x1);
      l += x0 + x1;
      if constexpr (!kTwoTerms) {
        unpack_f32x2(rsum, x0, x1);
        l_mma += x0 + x1;
      }
      HGA_TRACE_POINT(14);
    }
    // the place once more (while the last GEMM runs)
    const int tid2 = again_tid();
    const Place pl2(dm, segs, again_cta());
    const bool twice2 = rows_twice<kTwoTerms>(dm, pl2);
    const Row rw2(dm, pl2, tid2, twice2);
    if (ok) ok = __all_sync(0xffffffffu, bwd_wait(&sm.o_done, 0, abort));
    HGA_TRACE_POINT(20);
    // the row's two sums meet (every GEMM has read the K tile); ok or not, every softmax thread meets here once
    float neg_m, unused;
    unpack_f32x2(neg_m2, neg_m, unused);
    float* const xchg = reinterpret_cast<float*>(sm.k);
    xchg[rw2.hw * 256 + rw2.row] = l;
    if constexpr (!kTwoTerms) xchg[rw2.hw * 256 + 128 + rw2.row] = l_mma;
    if constexpr (kTwoTerms) {
      if (twice2 && rw2.row >= 64 && ok) {
        tc_fence_after_sync();
        share_row(sm, rw2, tmem);
      }
    }
    asm volatile("bar.sync 1, 256;" ::: "memory");
    l += xchg[(rw2.hw ^ 1) * 256 + rw2.row];
    if constexpr (kTwoTerms) {
      if (twice2) l += xchg[rw2.row ^ 64] + xchg[256 + (rw2.row ^ 64)];
    }
    if constexpr (!kTwoTerms) l_mma += xchg[(rw2.hw ^ 1) * 256 + 128 + rw2.row];
    else l_mma = l;                                     // (two terms leave 2^-17 of a weight: its sum needs no counterpart)
    if (ok && __any_sync(0xffffffffu, rw2.real) && !(twice2 && rw2.row >= 64)) {
      tc_fence_after_sync();
      const bool finite = store_row(sm, dm, pl2, rw2, tmem, l, l_mma, -neg_m, O, LSE, twice2 ? shared_row(sm, rw2) : 0);
      // (a sum that is not a number passes none of these tests)
      if (rw2.real && (l >= kSumLimit || neg_m == INFINITY || (l > kWeightLimit && !finite))) sm.again = 1;
    }
    if (dm.Bq % 64 == 0) {
      fence_proxy_async_smem();
      mbar_arrive_warp(&sm.o_staged);
      if (ok && warp == 4 && bwd_wait(&sm.o_staged, 0, abort) && !sm.again) store_boxes(sm, dm, pl2, map_o, lane);   // all rows are in shared memory
    }
    HGA_TRACE_POINT(21);
  }

  // common exit: every role has either finished or given up
  HGA_TRACE_POINT(30);
  __syncwarp();
  tc_fence_before_sync();
  __syncthreads();
  HGA_TRACE_POINT(31);
  if (sm.again && !sm.abort) {
    passes_with_true_maxima<D>(sm, map_q, map_k, map_v, map_o, group_idx, dm, O, LSE, segs, sm.tmem_base);
    tc_fence_before_sync();
    __syncthreads();
  }
  HGA_TRACE_DUMP;
  if (tid == 0 && sm.abort && status_word) atomicOr(status_word, HGA_ABORT_CODE(1, sm.abort));
  if (warp == 1) {
    __syncwarp();
    if (sm.abort) {
      // given up (known for certain behind the barrier): GEMMs already issued may still be writing tensor memory; wait
      // (bounded) until the tensor pipe has run dry before the columns are given back
      mma_commit_w(elect_one(), &sm.drain);
      mbar_wait(&sm.drain, 0);
      __syncwarp();
    }
    tmem_dealloc(sm.tmem_base, kTmemCols);
  }
}

bool attn_fwd_sm100_supported(const Dims& dm) {
  if (dm.flags & HGA_FLAG_GENERIC_KERNELS) return false;
  // any number of rows: the last M-tile of an item may be partly filled (its other TMEM lanes compute garbage that is
  // never stored), which still beats the one-warp-per-row kernel by far: 16 heads of 64 rows, head_dim 64, 512 items
  // of 768 keys take 1.9 ms there
  return dm.g % 8 == 0;
}

// Row counts that do not fill M-tiles: until these kernels took them they had the warp-per-row kernel, which weighs V with
// fp32 probabilities, and they keep that precision: error of O against fp64 (head_dim 128, 64 rows) 1.66e-3, which is the
// rounding of O itself, with two terms; 2.3e-3 with one.
static bool two_terms(const Dims& dm) {
  const int rows_pad = rows_padded(dm);
  if (rows_pad > 128) return rows_pad % 128 != 0 || rows_pad != dm.rows;
  return rows_pad < 128 && !(dm.flags & HGA_FLAG_DECODE);
}

template <int D, bool kTwoTerms, class Segs>
static int launch_fwd(const Dims& dm, const Segs& segs, int64_t units, const void* Q, const void* K, const void* V,
                      const int32_t* group_idx, const int32_t* n_groups, void* O, float* LSE, int32_t* status_word, cudaStream_t st) {
  CUtensorMap mq, mk, mv, mo;
  const bool boxes = dm.Bq % 64 == 0;
  const uint32_t box[5] = {64, 8, (uint32_t)(D / 64), 1, 1}, box_rows[5] = {64, 64, 1, 1, 1};
  const uint64_t dq[5] = {64, (uint64_t)dm.rows_q, (uint64_t)(D / 64), (uint64_t)dm.Hq, (uint64_t)dm.B};
  const uint64_t dk[5] = {64, (uint64_t)dm.rows_k, (uint64_t)(D / 64), (uint64_t)dm.Hkv, (uint64_t)dm.B};
  const uint64_t sq[4] = {(uint64_t)dm.qs[2] * 2, 128, (uint64_t)dm.qs[1] * 2, (uint64_t)dm.qs[0] * 2};
  const uint64_t so[4] = {(uint64_t)dm.os[2] * 2, 128, (uint64_t)dm.os[1] * 2, (uint64_t)dm.os[0] * 2};
  const uint64_t sk[4] = {(uint64_t)dm.ks[2] * 2, 128, (uint64_t)dm.ks[1] * 2, (uint64_t)dm.ks[0] * 2};
  const uint64_t sv[4] = {(uint64_t)dm.vs[2] * 2, 128, (uint64_t)dm.vs[1] * 2, (uint64_t)dm.vs[0] * 2};
  if (encode_tensor_map_bf16(&mq, Q, 5, dq, sq, boxes ? box_rows : box, true) ||
      encode_tensor_map_bf16(&mo, O, 5, dq, so, box_rows, true) ||
      encode_tensor_map_bf16(&mk, K, 5, dk, sk, box, true) ||
      encode_tensor_map_bf16(&mv, V, 5, dk, sv, box, true))
    return HGA_ERR_UNSUPPORTED;
  const size_t smem = sizeof(FwdSmem<D>) + 1024;
  static_assert(sizeof(FwdSmem<D>) + 1024 <= 113 * 1024, "two CTAs per SM");
  // two CTAs per SM need the largest shared-memory carve-out
  const int rc = ensure_dynamic_smem(reinterpret_cast<const void*>(&k_attn_fwd_sm100<D, kTwoTerms, Segs>), smem, true);
  if (rc) return rc;
  PdlLaunch cfg((unsigned)units, kFwdThreads, smem, st, dm.flags);
  const cudaError_t e = cudaLaunchKernelEx(&cfg.c, k_attn_fwd_sm100<D, kTwoTerms, Segs>, mq, mk, mv, mo, group_idx, n_groups, dm, (uint16_t*)O,
                                           LSE, status_word, segs);
  count_launch(HGA_KERNELS_FWD_TENSOR);
  return record_cuda(e);
}

int launch_attn_fwd_sm100(const Dims& dm, SegTable* segs, const void* Q, const void* K, const void* V,
                          const int32_t* group_idx, const int32_t* n_groups, void* O, float* LSE,
                          int32_t* status_word, cudaStream_t st) {
  const int n_mt = (rows_padded(dm) + 127) / 128;
#define HGA_FWD_ARGS(segs, units) dm, segs, units, Q, K, V, group_idx, n_groups, O, LSE, status_word, st
#define HGA_FWD(segs, units)                                                                                            \
  (two_terms(dm) ? (dm.d == 128 ? launch_fwd<128, true>(HGA_FWD_ARGS(segs, units)) : launch_fwd<64, true>(HGA_FWD_ARGS(segs, units))) \
                 : (dm.d == 128 ? launch_fwd<128, false>(HGA_FWD_ARGS(segs, units)) : launch_fwd<64, false>(HGA_FWD_ARGS(segs, units))))
  if (!segs) return HGA_FWD(OneSegment{}, (int64_t)dm.B * dm.Hkv * dm.NQB * n_mt);
  const int64_t units = number_units(*segs, [&](const Segment& s) { return (int64_t)dm.B * dm.Hkv * (s.S / dm.Bq) * n_mt; });
  return HGA_FWD(*segs, units);
#undef HGA_FWD
#undef HGA_FWD_ARGS
}

}  // namespace hga
