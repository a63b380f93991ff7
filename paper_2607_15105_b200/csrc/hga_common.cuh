// Internal definitions shared by the libhga translation units (not part of the C ABI).
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "hga.h"

namespace hga {

// Block score aggregator selected by hga_params.flags: 0 maximum, 1 mean, 2 log-sum-exp over the rows.
__host__ __device__ inline int score_agg_of(int flags) {
  return (flags & HGA_FLAG_SCORE_MEAN) ? 1 : (flags & HGA_FLAG_SCORE_LSE) ? 2 : 0;
}

// Internal flag (a bit of Dims.flags that hga.h does not define and the exported calls reject): launch
// the backward's kernels without programmatic serialization.  Set by hga_step_host, whose steps are bound
// by the host link: there the early-started CTAs only get in the way of the next (batch, kv head) pair's
// kernels; and where dQ takes the place of Q, dO or O.
constexpr int kFlagNoPdl = 1 << 30;

// Division of 0 <= n < 2^31 by a number that the host knows, as a multiplication and a shift (T. Granlund, P. Montgomery:
// Division by Invariant Integers using Multiplication, 1994).  A CTA has half a dozen such divisions ahead of its first copy, one
// behind the other: 16K layer (whole step) 143.7 us with plain divisions, 140.4 so.
struct Div {
  uint32_t by, mul, shift;
  __host__ __device__ Div() : by(1), mul(1), shift(0) {}
  // 2^shift the smallest power of two >= by, mul = ceil(2^32 (2^shift - by) / by) up to the + 1 that makes it exact.  (d < 1 comes
  // from products that overflow, of sizes that no tensor can have but a size query may: any divisor does.)
  explicit Div(int d) : by(d > 0 ? (uint32_t)d : 1), mul(1), shift(0) {
    while ((1u << shift) < by) ++shift;
    mul = (uint32_t)((((uint64_t)1 << 32) * (((uint64_t)1 << shift) - by)) / by + 1);
  }
  __host__ __device__ int operator()(int n) const {
    return (int)(((uint32_t)(((uint64_t)mul * (uint32_t)n) >> 32) + (uint32_t)n) >> shift);
  }
};

// Internal flag: the kernel's predecessor in the stream is the one of this library that precedes it in a step.  That kernel has
// waited for everything before it ahead of letting this one start, and writes neither Q, K, V nor dO: their copies need not wait
// for its end.  (Behind a caller's kernel, which may let its successor start before it has written them, they do.  The backward takes
// the flag back where the caller has O, which the forward does write, share bytes with Q or dO.)
constexpr int kFlagChained = 1 << 29;

// Resolved problem description handed to kernels by value.
struct Dims {
  int B, Hq, Hkv, G, d;
  int L, S, H;          // total, active segment, history = L - S
  int c, g, Bq;         // chunk, group, query block
  int kc, kg, kge, per; // k_c, k_g, min(k_g, c/g), c/g
  int sink, local;
  int NQB, Nc, Ng;      // query blocks per sequence, chunks, groups
  int NcS, NgS;         // rows per (batch, kv head) in the chunk / group summary buffers (>= Nc, Ng)
  int rows_q, rows_k;   // token rows of the Q / O and of the K / V tensors (S and L, unless a launch covers several segments)
  int width;            // group_idx entries per item = kc * kge
  int rows;             // G * Bq query rows per item
  int flags;
  float scale;          // softmax scale
  int64_t qs[3], ks[3], vs[3], os[3];  // element strides (batch, head, token)
  Div by_Bq, by_Bq_pad, by_c, by_g, by_Hkv, by_bh, by_mt;      // query block (and padded to octets), chunk, group, kv heads, batch * kv heads, M-tiles of an item
  inline void set_divisors();          // from the fields above
};

// Window geometry of a query block (local start, sink end), see hga.h.
struct Window {
  int p0, ls, se;
};

// Window of the query block that starts at position p0
__host__ __device__ inline Window window_at(const Dims& dm, int p0) {
  Window w;
  w.p0 = p0;
  int l = w.p0 - dm.local;
  w.ls = l <= 0 ? 0 : dm.by_c(l) * dm.c;
  w.se = dm.sink < w.ls ? dm.sink : w.ls;
  return w;
}
__host__ __device__ inline Window window_of(const Dims& dm, int qb) { return window_at(dm, dm.H + qb * dm.Bq); }

// One launch can cover several segments -- the sequences of a packed batch, or the segments of one long sequence, which
// are independent problems once the summaries are built -- instead of one: a short segment's kernels are a partial wave
// each, and twelve of them one after another are mostly tails.  Segment s has S active tokens behind H resident ones; its
// query rows start at row q0 of the Q / O tensors, its position 0 is row k0 of the K / V tensors, and its summaries start
// at rows k0 / c and k0 / g.  Its routing lists, LSE and dK / dV blocks follow those of the B * q0 query rows before it.
struct Segment {
  int first;                // its first CTA (the unit of the kernel that reads the table)
  int H, S, q0, k0;
};
constexpr int kMaxSegments = 64;      // per launch: the table is a kernel parameter
struct SegTable {
  int n;
  Segment seg[kMaxSegments];
};
struct OneSegment {};                 // the usual problem: the segment of Dims, no table

// Segment of CTA `cta`, and the CTA's number inside it
__device__ __forceinline__ Segment segment_of(const Dims& dm, const OneSegment&, int cta, int& local) {
  local = cta;
  return Segment{0, dm.H, dm.S, 0, 0};
}
__device__ __forceinline__ Segment segment_of(const Dims&, const SegTable& t, int cta, int& local) {
  int lo = 0, hi = t.n;
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (t.seg[mid].first <= cta) lo = mid; else hi = mid;
  }
  local = cta - t.seg[lo].first;
  return t.seg[lo];
}
// Where a segment's routing lists (in items) and per-row outputs (in rows of one head) start for batch entry b
__device__ __forceinline__ int64_t item_base(const Dims& dm, const Segment& sg, int b) {
  return ((int64_t)dm.B * dm.by_Bq(sg.q0) + (int64_t)b * dm.by_Bq(sg.S)) * dm.Hkv;
}
__device__ __forceinline__ int64_t row_base(const Dims& dm, const Segment& sg, int b) {
  return (int64_t)dm.B * sg.q0 + (int64_t)b * sg.S;
}
// Fills in `first`, counting units_of(segment) CTAs each; returns their number (host)
template <class F>
inline int64_t number_units(SegTable& t, F units_of) {
  int64_t n = 0;
  for (int i = 0; i < t.n; ++i) { t.seg[i].first = (int)n; n += units_of(t.seg[i]); }
  return n;
}

__host__ __device__ inline void item_coords(const Dims& dm, int item, int& b, int& h, int& qb) {
  qb = item % dm.NQB;
  int bh = item / dm.NQB;
  h = bh % dm.Hkv;
  b = bh / dm.Hkv;
}

// Row layout of an item inside the tensor-core kernels: every query head's Bq rows are padded to
// whole octets (8 rows = one TMA box / swizzle atom), so row r of the item is (head r / bq_pad,
// token r % bq_pad) and rows with token >= Bq are padding.  Bq is a multiple of 8 except in
// generation-shaped problems (HGA_FLAG_DECODE), where bq_pad = 8 or 16 for 1..16 new tokens.
__host__ __device__ inline int bq_padded(const Dims& dm) { return (dm.Bq + 7) & ~7; }
__host__ __device__ inline int rows_padded(const Dims& dm) { return dm.G * bq_padded(dm); }

inline void Dims::set_divisors() {
  by_Bq = Div(Bq); by_Bq_pad = Div(bq_padded(*this)); by_c = Div(c); by_g = Div(g); by_Hkv = Div(Hkv); by_bh = Div(B * Hkv);
  by_mt = Div((rows_padded(*this) + 127) / 128);
}

// Upper bound of routed tokens per item (sink + groups + local window + the block itself).
__host__ __device__ inline int max_routed_tokens(const Dims& dm) {
  return dm.sink + dm.width * dm.g + dm.local + dm.Bq + dm.c;
}

// A launch with programmatic serialization, or a plain one with kFlagNoPdl.  The kernel may start before its predecessor in
// the stream has ended; it executes griddepcontrol.wait before it touches memory that the predecessor may write, and before
// it ends, so that "the predecessor has ended" includes all work before it.
struct PdlLaunch {
  cudaLaunchConfig_t c = {};
  cudaLaunchAttribute attr;
  PdlLaunch(dim3 grid, unsigned threads, size_t smem, cudaStream_t st, int flags) {
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    c.gridDim = grid;
    c.blockDim = dim3(threads);
    c.dynamicSmemBytes = smem;
    c.stream = st;
    c.attrs = &attr;
    c.numAttrs = (flags & kFlagNoPdl) ? 0 : 1;
  }
  PdlLaunch(const PdlLaunch&) = delete;
};

// cudaFuncSetAttribute(max dynamic shared memory [, maximal carve-out]) for `func`, cached per device (hga_tma.cu)
int ensure_dynamic_smem(const void* func, size_t bytes, bool max_carveout = false);

// Launch bookkeeping (hga_api.cu).
void count_launch(int family, int n = 1);   // family: HGA_KERNELS_*
int record_cuda(cudaError_t e);  // returns HGA_OK or HGA_ERR_CUDA and remembers the code

// Kernel launchers, one per translation unit.  All return an HGA status.
int launch_build_summaries(const Dims& dm, const void* K, int tok_begin, int tok_end,
                           void* chunk_sum, void* group_sum, cudaStream_t st);
// the active chunks of every segment of the table
int launch_build_active_summaries(const Dims& dm, SegTable& segs, const void* K, void* chunk_sum, void* group_sum, cudaStream_t st);
int launch_route_generic(const Dims& dm, const void* Q, const void* chunk_sum,
                         const void* group_sum, int32_t* chunk_idx, int32_t* group_idx,
                         int32_t* n_groups, float* chunk_scores, float* group_scores,
                         void* workspace, cudaStream_t st);
int launch_attn_fwd_generic(const Dims& dm, const void* Q, const void* K, const void* V,
                            const int32_t* group_idx, const int32_t* n_groups, void* O, float* LSE,
                            int32_t* status_word, cudaStream_t st);
int launch_attn_bwd_generic(const Dims& dm, const void* Q, const void* K, const void* V,
                            const void* O, const float* LSE, const void* dO,
                            const int32_t* group_idx, const int32_t* n_groups, void* dQ, float* dK,
                            float* dV, int32_t* status_word, cudaStream_t st);

// tensor-core (tcgen05 / TMEM / TMA) kernels; *_supported says whether the shape qualifies; segs: the segments the launch
// covers (renumbered by the call), or null for the one of dm
bool attn_fwd_sm100_supported(const Dims& dm);
int launch_attn_fwd_sm100(const Dims& dm, SegTable* segs, const void* Q, const void* K, const void* V,
                          const int32_t* group_idx, const int32_t* n_groups, void* O, float* LSE,
                          int32_t* status_word, cudaStream_t st);

// the smallest generation shapes (warp-level matrix instructions, no tiles)
bool attn_decode_supported(const Dims& dm);
int launch_attn_decode(const Dims& dm, const void* Q, const void* K, const void* V, const int32_t* group_idx,
                       const int32_t* n_groups, void* O, float* LSE, int32_t* status_word, cudaStream_t st);

bool route_sm100_supported(const Dims& dm, const SegTable* segs);
int launch_route_sm100(const Dims& dm, SegTable* segs, const void* Q, const void* chunk_sum, const void* group_sum,
                       int32_t* chunk_idx, int32_t* group_idx, int32_t* n_groups, float* chunk_scores,
                       float* group_scores, cudaStream_t st);
bool attn_bwd_sm100_supported(const Dims& dm);
int launch_attn_bwd_sm100(const Dims& dm, SegTable* segs, const void* Q, const void* K, const void* V, const void* O,
                          const float* LSE, const void* dO, const int32_t* group_idx,
                          const int32_t* n_groups, void* dQ, float* dK, float* dV, int32_t* status_word,
                          cudaStream_t st);
// The backward keeps P and dS in several bf16 terms, i.e. at fp32's precision, for the shapes that used to have the CUDA-core
// kernel; they have a sweep of their own, called by the above
inline bool bwd_in_terms(const Dims& dm) { return dm.d == 64 || dm.rows % 128 != 0; }
int launch_attn_bwd_terms_sm100(const Dims& dm, SegTable* segs, const void* Q, const void* K, const void* V, const void* O,
                                const float* LSE, const void* dO, const int32_t* group_idx,
                                const int32_t* n_groups, void* dQ, float* dK, float* dV, int32_t* status_word,
                                cudaStream_t st);
// Key-major dK/dV of the local band (plain stores covering every active-segment row); launched by the above.
bool attn_bwd_band_sm100_supported(const Dims& dm);
int launch_attn_bwd_band_sm100(const Dims& dm, SegTable* segs, const void* Q, const void* K, const void* V, const void* O,
                               const float* LSE, const void* dO, float* dK, float* dV, int32_t* status_word,
                               cudaStream_t st);

// Validates an hga_params block and fills the resolved description (hga_api.cu).
int resolve_params(const hga_params* p, Dims& dm);

size_t route_workspace_bytes(const Dims& dm);
size_t bwd_workspace_bytes(const Dims& dm);

// fp32 -> bf16 (round to nearest even): src holds n dK sums followed by n dV sums, n a multiple of 8; one
// launch for both tensors.  after_sweep: launched with programmatic serialization behind the tensor-core sweep
// (which releases it early in that mode), so that its launch overlaps the sweep's tail (hga_attn_generic.cu)
int launch_grads_to_bf16(const float* src, void* dst_k, void* dst_v, size_t n, bool after_sweep, cudaStream_t st);

}  // namespace hga
