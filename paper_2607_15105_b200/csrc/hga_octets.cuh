// Octet table of an item's routed key set, built by one warp.
//
// The routed set of an item (sink, selected groups, local window) is addressed in octets of 8
// consecutive tokens; oct_row[o] is the first token of octet o, in ascending token order.  The
// group list is validated on the way: an entry must be greater than the last accepted entry
// and lie wholly between the sink and the local window; other entries are skipped and
// reported.  The common case (a valid ascending list) is checked with one coalesced load and a
// warp vote per 32 entries; only a list that fails the vote is walked sequentially.  (None of these loops is worth
// unrolling: they are inlined into every role that looks octets up.)
#pragma once

#include "hga_common.cuh"

namespace hga {

// Must be called by all 32 lanes of one warp.  Returns the number of octets (same value in
// every lane).  *bad_out (lane-uniform) tells whether an entry was skipped.
__device__ inline int build_octet_table(const Dims& dm, const Window& w, const int32_t* __restrict__ gi,
                                        const int32_t* __restrict__ ng_ptr, int* oct_row, bool* bad_out) {
  const unsigned full = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  // the first 64 entries are fetched before the count is known, so the two loads overlap
  const int pre0 = lane < dm.width ? __ldcg(gi + lane) : 0x7fffffff;
  const int pre1 = lane + 32 < dm.width ? __ldcg(gi + lane + 32) : 0x7fffffff;
  int ng = __ldcg(ng_ptr);
  bool bad = false;
  if (ng > dm.width) { ng = dm.width; bad = true; }
  if (ng < 0) { ng = 0; bad = true; }
  const int opg = dm.g / 8;           // octets per group
  const int n_sink = w.se / 8;
  bool all_ok = true;
  int prev = -1;
#pragma unroll 1
  for (int base = 0; base < ng; base += 32) {
    const int i = base + lane;
    const int m = i >= ng ? 0x7fffffff : base == 0 ? pre0 : base == 32 ? pre1 : __ldcg(gi + i);
    int left = __shfl_up_sync(full, m, 1);
    if (lane == 0) left = prev;
    const bool ok = i >= ng || (m > left && (int64_t)m * dm.g >= w.se && ((int64_t)m + 1) * dm.g <= w.ls);
    all_ok = all_ok && __all_sync(full, ok);
    if (all_ok && i < ng)
      for (int u = 0; u < opg; ++u) oct_row[n_sink + i * opg + u] = m * dm.g + 8 * u;
    prev = __shfl_sync(full, m, 31);
  }
  int n_far = n_sink + ng * opg;
  if (!all_ok) {
    bad = true;
    int n = n_sink;
    if (lane == 0) {
      int last = -1;
#pragma unroll 1
      for (int i = 0; i < ng; ++i) {
        const int m = __ldcg(gi + i);
        if (m > last && (int64_t)m * dm.g >= w.se && ((int64_t)m + 1) * dm.g <= w.ls) {
          for (int u = 0; u < opg; ++u) oct_row[n++] = m * dm.g + 8 * u;
          last = m;
        }
      }
    }
    n_far = __shfl_sync(full, n, 0);
  }
  for (int o = lane; o < n_sink; o += 32) oct_row[o] = 8 * o;
  const int n_local = (w.p0 + dm.Bq - w.ls + 7) / 8;      // the last octet may be partial (decode shapes)
  for (int o = lane; o < n_local; o += 32) oct_row[n_far + o] = w.ls + 8 * o;
  __syncwarp();
  *bad_out = bad;
  return n_far + n_local;
}

// The "far" part of an item's routed set (sink, then selected groups) as octets, looked up in the group list
// itself: no table in shared memory.  A list is checked once, 32 entries per vote; a valid list (every entry
// ascending and wholly between sink and local window) is then read directly, an invalid one is walked, skipping the
// entries build_octet_table would skip.
struct FarList {
  const int32_t* gi;
  int ng, opg, n_sink, n_far, first_active, se, ls, g;
  bool clean;
  __device__ bool fits(int m, int last) const {
    return m > last && (int64_t)m * g >= se && ((int64_t)m + 1) * g <= ls;
  }
  __device__ FarList(const Dims& dm, const Window& w, const int32_t* list)
      : gi(list), ng(0), opg(dm.g / 8), n_sink(w.se / 8), n_far(0), first_active(0), se(w.se), ls(w.ls), g(dm.g), clean(true) {}
  // Checks the list and counts its octets (H: first position of the active segment); all 32 lanes of a warp.  Returns
  // whether the list or its count is invalid.  The loads go past the L1 cache: the kernel may have started before
  // the list was written.
  __device__ bool check(const Dims& dm, const int32_t* ng_ptr, int H) {
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const int pre0 = lane < dm.width ? __ldcg(gi + lane) : 0x7fffffff;      // (overlaps the load of the count)
    const int pre1 = lane + 32 < dm.width ? __ldcg(gi + lane + 32) : 0x7fffffff;
    const int listed = __ldcg(ng_ptr);
    ng = listed < 0 ? 0 : listed > dm.width ? dm.width : listed;
    int prev = -1, below = 0;
#pragma unroll 1
    for (int base = 0; base < ng; base += 32) {
      const int i = base + lane;
      const int m = i >= ng ? 0x7fffffff : base == 0 ? pre0 : base == 32 ? pre1 : __ldcg(gi + i);
      int left = __shfl_up_sync(full, m, 1);
      if (lane == 0) left = prev;
      clean = clean && __all_sync(full, i >= ng || fits(m, left));
      below += __popc(__ballot_sync(full, i < ng && (int64_t)m * g < H));
      prev = __shfl_sync(full, m, 31);
    }
    int n = ng;
    if (!clean) {
      n = below = 0;
      if (lane == 0) {
        int last = -1;
#pragma unroll 1
        for (int i = 0; i < ng; ++i) {
          const int m = __ldcg(gi + i);
          if (fits(m, last)) { ++n; below += (int64_t)m * g < H; last = m; }
        }
      }
      n = __shfl_sync(full, n, 0);
      below = __shfl_sync(full, below, 0);
    }
    n_far = n_sink + n * opg;
    first_active = H / 8 < n_sink ? H / 8 : n_sink + below * opg;            // (training shapes: H is a multiple of g)
    return !clean || ng != listed;
  }
  // first token of far octet o (o < n_far)
  __device__ int row(int o) const {
    if (o < n_sink) return 8 * o;
    const int k = o - n_sink, u = opg == 1 ? k : k / opg, sub = k - u * opg;
    if (clean) return __ldcg(gi + u) * g + 8 * sub;
    int last = -1, n = -1;
#pragma unroll 1
    for (int i = 0; i < ng; ++i) {
      const int m = __ldcg(gi + i);
      if (fits(m, last)) { last = m; if (++n == u) break; }
    }
    return last * g + 8 * sub;
  }
};

}  // namespace hga
