// The routed key set of an item (sink, selected groups, local window), addressed in octets of 8 consecutive tokens.
#pragma once

#include "hga_common.cuh"

namespace hga {

// The "far" part of an item's routed set (sink, then selected groups) as octets, looked up in the group list
// itself: no table in shared memory.  A list is checked once, 32 entries per vote; a valid list (every entry
// ascending and wholly between sink and local window) is then read directly, an invalid one is walked, skipping (and
// reporting) an entry that is not greater than the last accepted one or does not lie there.  (None of these loops is worth
// unrolling: they are inlined into every role that looks octets up.)
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
    if (clean && opg == 1) return __ldcg(gi + (o - n_sink)) * g;
    return row_of_group(gi, clean ? -1 : ng, o - n_sink, g, se, ls);
  }
  // (out of line: inlined into every role that looks octets up, this and the division cost the usual case, groups of eight
  // tokens in a valid list, more in instruction fetch than the call costs the others)
  static __device__ __noinline__ int row_of_group(const int32_t* gi, int n_walk, int k, int g, int se, int ls) {
    const int opg = g / 8, u = k / opg, sub = k - u * opg;
    if (n_walk < 0) return __ldcg(gi + u) * g + 8 * sub;
    int last = -1, n = -1;
#pragma unroll 1
    for (int i = 0; i < n_walk; ++i) {
      const int m = __ldcg(gi + i);
      if (m > last && (int64_t)m * g >= se && ((int64_t)m + 1) * g <= ls) { last = m; if (++n == u) break; }
    }
    return last * g + 8 * sub;
  }
};

}  // namespace hga
