// hga_attn_fwd for the smallest generation shapes (HGA_FLAG_DECODE, up to 16 query rows per kv head, few sequences): routed
// exact-token attention (Section 2.1 item 3) with warp-level matrix instructions.
//
// A step for a few sequences is bound by latency: the tensor-memory tiles of k_attn_fwd_sm100 take 128 keys at a time
// through a chain copy -> S -> exponentials -> P V -> copy, six or more times, in one CTA per item, on a nearly idle GPU.
// Here every warp works on its own, 16 keys (two octets) at a time: a lane copies (cp.async) the very 16-byte pieces
// it will use, in the layout that mma.sync.m16n8k16 wants (below), into its slots of a three-stage ring, so no barrier
// separates copies from use; an item is split over eight warps and a cluster of up to eight CTAs, whose partial
// results meet through (distributed) shared memory.  One sequence behind 5003 tokens: hga_attn_fwd 16.6 -> 8.9 us, the
// step (route + forward) 24.8 -> 18 us; 8 sequences behind 16K: 28.5 -> 24.4.  With more items than SMs both are bound by
// HBM and the tiles do as well or better (32 sequences: 21.8 us there, 26.6 here), hence the limit.
//
//   S = Q K^T      A = Q rows (16, unused ones zero), B = 8 keys; the head_dim axis is permuted alike on both sides so
//                  that a lane's 16 bytes of a K row are two instructions' worth of its B fragment
//   O^T += V^T P^T A = V^T: the lane's 16 bytes of four V rows, halves interleaved pairwise (prmt); the rows of the
//                  M axis are head_dim elements in an order of our choosing; B = P^T, which is the S fragment as it is
//
// The running maximum is raised lazily (only when it grows by more than 2^8).  l sums the exact probabilities (LSE), l_mma
// the bf16-rounded ones that multiply V and that O is divided by.
#include <cooperative_groups.h>

#include "hga_common.cuh"
#include "hga_octets.cuh"
#include "hga_sm100.cuh"

namespace hga {

using namespace sm100;

namespace {

constexpr float kRaise = 8.f;         // log2 units
constexpr int kStages = 3, kWarps = 8;

__device__ __forceinline__ void mma_16816(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
  asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
               : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
               : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
// 16 bytes global -> shared, past L1; zeros where !real
__device__ __forceinline__ void copy16(uint32_t dst, const uint16_t* src, bool real) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(real ? 16 : 0) : "memory");
}
__device__ __forceinline__ uint4 lds16(uint32_t addr) {
  uint4 v;
  asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr));
  return v;
}
__device__ __forceinline__ uint32_t word(const uint4& v, int i) { return i == 0 ? v.x : i == 1 ? v.y : i == 2 ? v.z : v.w; }
__device__ __forceinline__ uint32_t pack2(float lo, float hi) {
  const __nv_bfloat162 h = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<const uint32_t*>(&h);
}

template <int D>
constexpr int kPieces = 2 * (D / 32) + 4 * (D / 64);       // 16-byte pieces per lane and unit: two K rows' quarters, four V rows' eighths

}  // namespace

// NT: 8-row tiles of query rows (1 or 2)
template <int D, int NT>
__global__ void __launch_bounds__(32 * kWarps)
k_attn_decode(const uint16_t* __restrict__ Q, const uint16_t* __restrict__ K, const uint16_t* __restrict__ V,
              const int32_t* __restrict__ group_idx, const int32_t* __restrict__ n_groups, const Dims dm,
              uint16_t* __restrict__ O, float* __restrict__ LSE, int32_t* status_word, int n_split) {
  constexpr int kRows = 8 * NT, kChunks = D / 32, kPanels = D / 64;
  constexpr int kStageBytes = kPieces<D> * 512, kWarpBytes = kStages * kStageBytes;
  static_assert(kRows * D * 4 <= kWarpBytes, "a warp's partial O takes its ring's place");
  extern __shared__ __align__(16) uint8_t smem[];       // [warps][ring], then per warp and for the CTA: max, l, l_mma of each row
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int g = lane >> 2, q = lane & 3;
  const int split = blockIdx.x % n_split, item = blockIdx.x / n_split;
  int b, h, qb;
  item_coords(dm, item, b, h, qb);
  const Window w = window_of(dm, qb);
  const int n_loc_oct = (w.p0 + dm.Bq - w.ls + 7) / 8;
  const uint16_t* const Kb = K + b * dm.ks[0] + h * dm.ks[1] + 8 * q;
  const uint16_t* const Vb = V + b * dm.vs[0] + h * dm.vs[1] + 8 * g;
  const uint32_t ring = smem_u32(smem) + warp * kWarpBytes + lane * 16;
  pdl_wait();

  FarList far(dm, w, group_idx + (int64_t)item * dm.width);
  const bool bad = far.check(dm, n_groups + item, dm.H);
  if (bad && status_word && tid == 0) atomicOr(status_word, HGA_STATUS_BAD_INDEX);
  const int n_oct = n_loc_oct + far.n_far, n_units = (n_oct + 1) / 2;
  const int first = split * kWarps + warp, step = n_split * kWarps;         // this warp's units: first, first + step, ...
  const int n_mine = n_units > first ? (n_units - first + step - 1) / step : 0;
  // token row of octet o of the set, -1 past its end
  auto row_of = [&](int o) {
    if (o < n_loc_oct) return w.ls + 8 * o;
    return o < n_oct ? far.row(o - n_loc_oct) : -1;
  };
  // lane l holds the row of octet (l & 1) of the warp's unit number (l >> 1) of the current sixteen
  int fetch_row = -1;
  auto fetch = [&](int k, int stage) {           // the warp's k-th unit (called with k = 0, 1, 2, ...)
    if (k < n_mine) {
      if ((k & 15) == 0) fetch_row = row_of(2 * (first + (k + (lane >> 1)) * step) + (lane & 1));
      const uint32_t dst = ring + stage * kStageBytes;
#pragma unroll
      for (int o = 0; o < 2; ++o) {
        const int row = __shfl_sync(0xffffffffu, fetch_row, 2 * (k & 15) + o);
        // rows past the sequence (the unwritten tail of a cache) are never read
        const bool real = row >= 0 && row + g < dm.L;
        const uint16_t* kp = Kb + (int64_t)(real ? row + g : 0) * dm.ks[2];
#pragma unroll
        for (int i = 0; i < kChunks; ++i) copy16(dst + (o * kChunks + i) * 512, kp + 32 * i, real);
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          const int key = row + 2 * q + u;
          const bool real_v = row >= 0 && key < dm.L;
          const uint16_t* vp = Vb + (int64_t)(real_v ? key : 0) * dm.vs[2];
#pragma unroll
          for (int p = 0; p < kPanels; ++p) copy16(dst + (2 * kChunks + (2 * o + u) * kPanels + p) * 512, vp + 64 * p, real_v);
        }
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
#pragma unroll 1
  for (int k = 0; k < kStages - 1; ++k) fetch(k, k);
  pdl_launch_dependents();

  // Q fragments and the visibility limit of this lane's rows (g, and g + 8 of the second tile)
  uint4 qa[NT][kChunks];
  int pos[NT];
#pragma unroll
  for (int n = 0; n < NT; ++n) {
    const int r = 8 * n + g;
    const bool real = r < dm.rows;
    const int a = real ? dm.by_Bq(r) : 0, t = real ? r - a * dm.Bq : 0;
    pos[n] = w.p0 + t;
    const uint16_t* qp = Q + b * dm.qs[0] + (h * dm.G + a) * dm.qs[1] + (int64_t)(qb * dm.Bq + t) * dm.qs[2] + 8 * q;
#pragma unroll
    for (int i = 0; i < kChunks; ++i) qa[n][i] = real ? __ldcg(reinterpret_cast<const uint4*>(qp + 32 * i)) : make_uint4(0, 0, 0, 0);
  }
  const float sl2 = dm.scale * 1.4426950408889634f;
  float m[NT], l[NT], l_mma[NT];
  float acc[kPanels][4][NT][4];                  // O^T: [panel][t]: elements 64p + 8g + 2t, +1 of rows 2q, 2q + 1
#pragma unroll
  for (int n = 0; n < NT; ++n) { m[n] = -INFINITY; l[n] = l_mma[n] = 0.f; }
#pragma unroll
  for (int p = 0; p < kPanels; ++p)
#pragma unroll
    for (int t = 0; t < 4; ++t)
#pragma unroll
      for (int n = 0; n < NT; ++n)
#pragma unroll
        for (int i = 0; i < 4; ++i) acc[p][t][n][i] = 0.f;

  int use_row = -1;
#pragma unroll 1
  for (int k = 0, stage = 0; k < n_mine; ++k) {
    asm volatile("cp.async.wait_group %0;" ::"n"(kStages - 2) : "memory");        // this lane's pieces of unit k have landed
    if ((k & 15) == 0) use_row = row_of(2 * (first + (k + (lane >> 1)) * step) + (lane & 1));
    const uint32_t src = ring + stage * kStageBytes;
    float s[2][4];
    int row[2];
#pragma unroll
    for (int o = 0; o < 2; ++o) {
      row[o] = __shfl_sync(0xffffffffu, use_row, 2 * (k & 15) + o);
#pragma unroll
      for (int i = 0; i < 4; ++i) s[o][i] = 0.f;
    }
#pragma unroll
    for (int i = 0; i < kChunks; ++i)
#pragma unroll
      for (int o = 0; o < 2; ++o) {
        const uint4 kf = lds16(src + (o * kChunks + i) * 512);
        mma_16816(s[o], qa[0][i].x, NT == 2 ? qa[NT - 1][i].x : 0u, qa[0][i].y, NT == 2 ? qa[NT - 1][i].y : 0u, kf.x, kf.y);
        mma_16816(s[o], qa[0][i].z, NT == 2 ? qa[NT - 1][i].z : 0u, qa[0][i].w, NT == 2 ? qa[NT - 1][i].w : 0u, kf.z, kf.w);
      }
    float mx[NT];
#pragma unroll
    for (int n = 0; n < NT; ++n) {
      mx[n] = -INFINITY;
#pragma unroll
      for (int o = 0; o < 2; ++o)
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          const int key = row[o] + 2 * q + u;
          const bool see = row[o] >= 0 && key <= pos[n];         // (every key before the block is at most p0 - 1)
          float& x = s[o][2 * n + u];
          x = see ? x * sl2 : -INFINITY;
          mx[n] = fmaxf(mx[n], x);
        }
      mx[n] = fmaxf(mx[n], __shfl_xor_sync(0xffffffffu, mx[n], 1));
      mx[n] = fmaxf(mx[n], __shfl_xor_sync(0xffffffffu, mx[n], 2));
    }
    uint32_t pb[2][NT];
#pragma unroll
    for (int n = 0; n < NT; ++n) {
      const bool raise = mx[n] > m[n] + kRaise;                  // (also the first time: m = -inf)
      if (__any_sync(0xffffffffu, raise)) {
        float corr = 1.f;
        if (raise) {
          corr = fast_exp2(m[n] - mx[n]);
          m[n] = mx[n];
          l[n] *= corr;
          l_mma[n] *= corr;
        }
        // (O's rows sit in other lanes than S's: row r's factor is in lanes 4r .. 4r + 3)
        const float c0 = __shfl_sync(0xffffffffu, corr, 8 * q), c1 = __shfl_sync(0xffffffffu, corr, 8 * q + 4);
#pragma unroll
        for (int p = 0; p < kPanels; ++p)
#pragma unroll
          for (int t = 0; t < 4; ++t) {
            acc[p][t][n][0] *= c0; acc[p][t][n][1] *= c1; acc[p][t][n][2] *= c0; acc[p][t][n][3] *= c1;
          }
      }
      const float ref = m[n] == -INFINITY ? 0.f : m[n];
#pragma unroll
      for (int o = 0; o < 2; ++o) {
        const float p0 = fast_exp2(s[o][2 * n] - ref), p1 = fast_exp2(s[o][2 * n + 1] - ref);
        l[n] += p0 + p1;
        const uint32_t pk = pack2(p0, p1);
        pb[o][n] = pk;
        l_mma[n] += __uint_as_float(pk << 16) + __uint_as_float(pk & 0xffff0000u);
      }
    }
#pragma unroll
    for (int p = 0; p < kPanels; ++p) {
      uint4 vf[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) vf[j] = lds16(src + (2 * kChunks + j * kPanels + p) * 512);
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        const uint32_t x0 = word(vf[0], t), x1 = word(vf[1], t), x2 = word(vf[2], t), x3 = word(vf[3], t);
        const uint32_t a0 = __byte_perm(x0, x1, 0x5410), a1 = __byte_perm(x0, x1, 0x7632);
        const uint32_t a2 = __byte_perm(x2, x3, 0x5410), a3 = __byte_perm(x2, x3, 0x7632);
#pragma unroll
        for (int n = 0; n < NT; ++n) mma_16816(acc[p][t][n], a0, a1, a2, a3, pb[0][n], pb[1][n]);
      }
    }
    // the stage of unit k - 1 takes unit k + 2 (a lane reuses only slots that it has itself read)
    fetch(k + kStages - 1, stage == 0 ? kStages - 1 : stage - 1);
    stage = stage + 1 == kStages ? 0 : stage + 1;
  }
  // ---- the warps' partial results meet in shared memory (each O over its own warp's ring)
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  __syncwarp();
  constexpr int kStep = kWarpBytes / 4;
  float* const so = reinterpret_cast<float*>(smem);            // [warps][kStep]: [kRows][D]
  float* const sst = so + kWarps * kStep;                      // [warps][3][kRows]
#pragma unroll
  for (int n = 0; n < NT; ++n) {
    l[n] += __shfl_xor_sync(0xffffffffu, l[n], 1);
    l[n] += __shfl_xor_sync(0xffffffffu, l[n], 2);
    l_mma[n] += __shfl_xor_sync(0xffffffffu, l_mma[n], 1);
    l_mma[n] += __shfl_xor_sync(0xffffffffu, l_mma[n], 2);
    if (q == 0) {
      float* st = sst + warp * 3 * kRows + 8 * n + g;
      st[0] = m[n]; st[kRows] = l[n]; st[2 * kRows] = l_mma[n];
    }
#pragma unroll
    for (int p = 0; p < kPanels; ++p)
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        float* o0 = so + warp * kStep + (8 * n + 2 * q) * D + 64 * p + 8 * g + 2 * t;
        *reinterpret_cast<float2*>(o0) = make_float2(acc[p][t][n][0], acc[p][t][n][2]);
        *reinterpret_cast<float2*>(o0 + D) = make_float2(acc[p][t][n][1], acc[p][t][n][3]);
      }
  }
  __syncthreads();
  // sums of partial results for row r, elements d and d + 1
  struct Sum { float m, l, l_mma, x, y; };
  auto add_part = [&](Sum& a, const float* st, const float* o, int r, int d) {
    const float pm = st[r];
    if (pm == -INFINITY) return;
    const float top = fmaxf(a.m, pm), ca = fast_exp2(a.m - top), cp = fast_exp2(pm - top);
    const float2 v = *reinterpret_cast<const float2*>(o + r * D + d);
    a.l = a.l * ca + st[kRows + r] * cp;
    a.l_mma = a.l_mma * ca + st[2 * kRows + r] * cp;
    a.x = a.x * ca + v.x * cp;
    a.y = a.y * ca + v.y * cp;
    a.m = top;
  };
  // each CTA sums its warps into its first slot (a thread overwrites only what it alone has read), then the rows are
  // shared out over the CTAs of the cluster, which read the others' slots
  float* const cst = sst + kWarps * 3 * kRows;                 // [3][kRows]
#pragma unroll 1
  for (int i = tid; i < kRows * D / 2; i += blockDim.x) {
    const int r = i / (D / 2), d = i % (D / 2) * 2;
    Sum a{-INFINITY, 0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int u = 0; u < kWarps; ++u) add_part(a, sst + u * 3 * kRows, so + u * kStep, r, d);
    *reinterpret_cast<float2*>(so + r * D + d) = make_float2(a.x, a.y);
    if (d == 0) { cst[r] = a.m; cst[kRows + r] = a.l; cst[2 * kRows + r] = a.l_mma; }
  }
  auto cluster = cooperative_groups::this_cluster();
  cluster.sync();
#pragma unroll 1
  for (int i = tid + split * blockDim.x; i < kRows * D / 2; i += blockDim.x * n_split) {
    const int r = i / (D / 2), d = i % (D / 2) * 2;
    Sum a{-INFINITY, 0.f, 0.f, 0.f, 0.f};
    for (int u = 0; u < n_split; ++u) add_part(a, cluster.map_shared_rank(cst, u), cluster.map_shared_rank(so, u), r, d);
    if (r < dm.rows) {
      const int head = dm.by_Bq(r), hq = h * dm.G + head, sr = qb * dm.Bq + r - head * dm.Bq;
      const float inv = 1.f / a.l_mma;
      *reinterpret_cast<uint32_t*>(O + b * dm.os[0] + hq * dm.os[1] + (int64_t)sr * dm.os[2] + d) = pack2(a.x * inv, a.y * inv);
      if (d == 0) LSE[((int64_t)b * dm.Hq + hq) * dm.S + sr] = (a.m + log2f(a.l)) * 0.6931471805599453f;
    }
  }
  cluster.sync();                                              // (nobody leaves while its slots are read)
}

bool attn_decode_supported(const Dims& dm) {
  if (dm.flags & HGA_FLAG_GENERIC_KERNELS) return false;
  return (dm.flags & HGA_FLAG_DECODE) && dm.rows <= 16 && dm.g % 8 == 0 && (int64_t)dm.B * dm.Hkv * dm.NQB <= 148;
}

template <int D, int NT>
static int launch_decode(const Dims& dm, const void* Q, const void* K, const void* V, const int32_t* group_idx, const int32_t* n_groups,
                         void* O, float* LSE, int32_t* status_word, cudaStream_t st) {
  const int items = dm.B * dm.Hkv * dm.NQB, units = (max_routed_tokens(dm) + 15) / 16;
  // a cluster of CTAs per item until a warp has about one unit or the SMs are full
  int split = 1;
  while (split < 8 && items * split * 2 <= 148 && units > kWarps * split) split *= 2;
  const size_t smem = (size_t)kWarps * kStages * kPieces<D> * 512 + sizeof(float) * (kWarps + 1) * 3 * 8 * NT;
  // (the shared-memory carve-out of the other kernels of the path: an SM has to drain before it changes)
  const int rc = ensure_dynamic_smem(reinterpret_cast<const void*>(&k_attn_decode<D, NT>), smem, true);
  if (rc) return rc;
  PdlLaunch cfg((unsigned)(items * split), kWarps * 32, smem, st, dm.flags);
  cudaLaunchAttribute attrs[2] = {cfg.attr, {}};
  attrs[1].id = cudaLaunchAttributeClusterDimension;
  attrs[1].val.clusterDim.x = (unsigned)split;
  attrs[1].val.clusterDim.y = attrs[1].val.clusterDim.z = 1;
  cfg.c.attrs = attrs;
  cfg.c.numAttrs = 2;
  const cudaError_t e = cudaLaunchKernelEx(&cfg.c, k_attn_decode<D, NT>, (const uint16_t*)Q, (const uint16_t*)K, (const uint16_t*)V,
                                           group_idx, n_groups, dm, (uint16_t*)O, LSE, status_word, split);
  count_launch(HGA_KERNELS_FWD_TENSOR);
  return record_cuda(e);
}

int launch_attn_decode(const Dims& dm, const void* Q, const void* K, const void* V, const int32_t* group_idx, const int32_t* n_groups,
                       void* O, float* LSE, int32_t* status_word, cudaStream_t st) {
#define HGA_DECODE_ARGS dm, Q, K, V, group_idx, n_groups, O, LSE, status_word, st
  if (dm.d == 128) return dm.rows <= 8 ? launch_decode<128, 1>(HGA_DECODE_ARGS) : launch_decode<128, 2>(HGA_DECODE_ARGS);
  return dm.rows <= 8 ? launch_decode<64, 1>(HGA_DECODE_ARGS) : launch_decode<64, 2>(HGA_DECODE_ARGS);
#undef HGA_DECODE_ARGS
}

}  // namespace hga
