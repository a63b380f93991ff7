// Shape-generic CUDA-core kernels for routed exact-token attention (Section 2.1 item 3) and
// its backward under segment-wise TBPTT (Section 2.2).  Forward: one warp owns one query row, a lane owns
// d/32 consecutive elements.  Backward: one CTA owns 8 query rows of an item.  These kernels accept
// every shape hga_params allows and serve as the cross-check of the tensor-core kernels.
#include <atomic>

#include <cfloat>

#include "hga_common.cuh"

namespace hga {

constexpr int kAttnThreads = 256;
constexpr int kAttnWarps = kAttnThreads / 32;

template <int EPL>
struct Frag {
  float v[EPL];
};

// EPL consecutive bf16 -> fp32 (EPL = 2: one 32-bit load, EPL = 4: one 64-bit load)
template <int EPL>
__device__ inline Frag<EPL> load_frag(const uint16_t* p) {
  Frag<EPL> f;
  if constexpr (EPL == 2) {
    const uint32_t w = *reinterpret_cast<const uint32_t*>(p);
    f.v[0] = __uint_as_float(w << 16);
    f.v[1] = __uint_as_float(w & 0xffff0000u);
  } else {
    const uint2 w = *reinterpret_cast<const uint2*>(p);
    f.v[0] = __uint_as_float(w.x << 16);
    f.v[1] = __uint_as_float(w.x & 0xffff0000u);
    f.v[2] = __uint_as_float(w.y << 16);
    f.v[3] = __uint_as_float(w.y & 0xffff0000u);
  }
  return f;
}

template <int EPL>
__device__ inline void store_frag_bf16(uint16_t* p, const Frag<EPL>& f) {
  uint32_t w[EPL / 2];
#pragma unroll
  for (int i = 0; i < EPL / 2; ++i) {
    const __nv_bfloat162 h = __floats2bfloat162_rn(f.v[2 * i], f.v[2 * i + 1]);
    w[i] = *reinterpret_cast<const uint32_t*>(&h);
  }
  if constexpr (EPL == 2) *reinterpret_cast<uint32_t*>(p) = w[0];
  else *reinterpret_cast<uint2*>(p) = make_uint2(w[0], w[1]);
}

template <int EPL>
__device__ inline float dot_frag(const Frag<EPL>& a, const Frag<EPL>& b) {
  float s = 0.f;
#pragma unroll
  for (int i = 0; i < EPL; ++i) s = fmaf(a.v[i], b.v[i], s);
  return s;
}

__device__ inline float warp_sum(float x) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
  return x;
}

// The item's valid group ids in shared memory (vg, up to `width` entries); returns how many.  Invalid entries (not
// ascending, or not wholly between sink and local window) are skipped and reported.
__device__ int build_group_list(const Dims& dm, const Window& w, const int32_t* gi, int ng, int* vg, int* s_meta,
                                int32_t* status_word) {
  const int tid = threadIdx.x, lane = tid & 31;
  auto fits = [&](int m, int last) {
    return m > last && (int64_t)m * dm.g >= w.se && ((int64_t)m + 1) * dm.g <= w.ls;
  };
  if (tid < 32) {
    // a valid list (the common case) passes 32 entries per vote; only an invalid one is walked sequentially
    bool bad = ng < 0 || ng > dm.width;
    ng = ng < 0 ? 0 : ng > dm.width ? dm.width : ng;
    bool clean = true;
    int prev = -1;
    for (int base = 0; base < ng; base += 32) {
      const int i = base + lane;
      const int m = i < ng ? gi[i] : 0x7fffffff;
      int left = __shfl_up_sync(0xffffffffu, m, 1);
      if (lane == 0) left = prev;
      clean = clean && __all_sync(0xffffffffu, i >= ng || fits(m, left));
      if (i < ng) vg[i] = m;
      prev = __shfl_sync(0xffffffffu, m, 31);
    }
    __syncwarp();
    int n = ng;
    if (!clean && lane == 0) {
      n = 0;
      int last = -1;
      for (int i = 0; i < ng; ++i) {
        const int m = vg[i];
        if (fits(m, last)) { vg[n++] = m; last = m; }
      }
    }
    if (lane == 0) {
      s_meta[0] = n;
      if ((bad || !clean) && status_word) atomicOr(status_word, HGA_STATUS_BAD_INDEX);
    }
  }
  __syncthreads();
  return s_meta[0];
}

// Token i of the routed set (sink, valid groups, local window), n_far = sink and group tokens
__device__ inline int routed_token(const Dims& dm, const Window& w, const int* vg, int n_far, int i) {
  if (i < w.se) return i;
  if (i < n_far) return vg[(i - w.se) / dm.g] * dm.g + (i - w.se) % dm.g;
  return w.ls + (i - n_far);
}

// The item's whole token list in shared memory; returns its length, s_meta[0] receives the number of valid groups.
__device__ int build_token_list(const Dims& dm, const Window& w, const int32_t* gi, int ng,
                                int* toks, int* s_meta, int32_t* status_word) {
  int* vg = toks + max_routed_tokens(dm);
  const int n_far = w.se + build_group_list(dm, w, gi, ng, vg, s_meta, status_word) * dm.g;
  const int n_tok = n_far + (w.p0 + dm.Bq - w.ls);
  for (int i = threadIdx.x; i < n_tok; i += blockDim.x) toks[i] = routed_token(dm, w, vg, n_far, i);
  __syncthreads();
  return n_tok;
}

template <int D>
__global__ void __launch_bounds__(kAttnThreads)
k_attn_fwd_generic(const uint16_t* __restrict__ Q, const uint16_t* __restrict__ K,
                   const uint16_t* __restrict__ V, const int32_t* __restrict__ group_idx,
                   const int32_t* __restrict__ n_groups, Dims dm, uint16_t* __restrict__ O,
                   float* __restrict__ LSE, int32_t* status_word) {
  constexpr int EPL = D / 32;
  extern __shared__ int s_int[];
  __shared__ int s_meta[2];
  const int item = blockIdx.x;
  int b, h, qb;
  item_coords(dm, item, b, h, qb);
  const Window w = window_of(dm, qb);
  build_token_list(dm, w, group_idx + (int64_t)item * dm.width, n_groups[item], s_int, s_meta, status_word);
  const int n_far = w.se + s_meta[0] * dm.g;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint16_t* Kb = K + b * dm.ks[0] + h * dm.ks[1] + lane * EPL;
  const uint16_t* Vb = V + b * dm.vs[0] + h * dm.vs[1] + lane * EPL;
  for (int r = warp; r < dm.rows; r += kAttnWarps) {
    const int a = r / dm.Bq, t = r % dm.Bq;
    const int hq = h * dm.G + a, srow = qb * dm.Bq + t;
    const int pos = w.p0 + t;
    const int n_vis = n_far + (pos - w.ls + 1);
    const Frag<EPL> q = load_frag<EPL>(Q + b * dm.qs[0] + hq * dm.qs[1] + srow * dm.qs[2] + lane * EPL);
    float m = -FLT_MAX, l = 0.f;
    Frag<EPL> acc;
#pragma unroll
    for (int e = 0; e < EPL; ++e) acc.v[e] = 0.f;
    for (int i = 0; i < n_vis; i += 4) {
      float s[4];
      Frag<EPL> vv[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int idx = i + u < n_vis ? i + u : n_vis - 1;
        const int64_t tok = s_int[idx];
        s[u] = dot_frag<EPL>(q, load_frag<EPL>(Kb + tok * dm.ks[2]));
        vv[u] = load_frag<EPL>(Vb + tok * dm.vs[2]);
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) s[u] = warp_sum(s[u]) * dm.scale;
      float m_new = m;
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (i + u < n_vis) m_new = fmaxf(m_new, s[u]);
      const float corr = __expf(m - m_new);
      l *= corr;
#pragma unroll
      for (int e = 0; e < EPL; ++e) acc.v[e] *= corr;
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        if (i + u < n_vis) {
          const float p = __expf(s[u] - m_new);
          l += p;
#pragma unroll
          for (int e = 0; e < EPL; ++e) acc.v[e] = fmaf(p, vv[u].v[e], acc.v[e]);
        }
      }
      m = m_new;
    }
    const float inv = 1.f / l;
#pragma unroll
    for (int e = 0; e < EPL; ++e) acc.v[e] *= inv;
    store_frag_bf16<EPL>(O + b * dm.os[0] + hq * dm.os[1] + srow * dm.os[2] + lane * EPL, acc);
    if (lane == 0) LSE[((int64_t)b * dm.Hq + hq) * dm.S + srow] = m + logf(l);
  }
}

// Backward.  One CTA owns kBwdRows query rows of an item; its eight warps take the item's routed keys in turn, eight
// at a time, each on its own (no block barrier in the loop; the next keys' loads are in flight during the work on
// the current ones).  Per warp and eight keys:
//   S = Q K^T, dP = dO V^T   lane = one row, two keys        -> P, dS in shared memory
//   dQ += dS K               lane = one row, d/4 elements (registers; the warps' sums meet at the end)
//   dV = P^T dO, dK = dS^T Q lane = one key, d/4 elements, added to global memory 16 bytes at a time (keys of the
//                            active segment only: history keys are detached constants)
// Where that leaves half of the device idle, a cluster of two CTAs owns the rows and each takes every other round of
// keys; their dQ sums meet through distributed shared memory.
// Everything is fp32.  Taken for shapes the tensor-core kernels do not cover and for problems too small to fill
// them, so what counts is the length of one CTA's chain and how many CTAs there are; the work itself is bound by
// shared-memory reads, 216 per 640 fused multiply-adds of a warp.
constexpr int kBwdRows = 8, kBwdKeys = 8, kBwdWarps = 8;

template <int D>
struct BwdTile {
  static constexpr int kPitch = D + 4;           // floats; 16-byte aligned rows that start 4 banks apart
  float q[kBwdRows][kPitch], dO[kBwdRows][kPitch];
  struct PerWarp {
    float k[kBwdKeys][kPitch], v[kBwdKeys][kPitch];       // (at the end: the warp's dQ sums)
    float p[kBwdRows][kBwdKeys], ds[kBwdRows][kBwdKeys];
    int tok[kBwdKeys];                           // -1 past the end of the list
  } w[kBwdWarps];
  static_assert(kBwdRows <= kBwdKeys, "dQ sums fit the K tile");
};

__device__ inline void bf16x8_to_smem(float* dst, uint4 w) {
  const uint32_t x[4] = {w.x, w.y, w.z, w.w};
  float4* d4 = reinterpret_cast<float4*>(dst);
  d4[0] = make_float4(__uint_as_float(x[0] << 16), __uint_as_float(x[0] & 0xffff0000u), __uint_as_float(x[1] << 16), __uint_as_float(x[1] & 0xffff0000u));
  d4[1] = make_float4(__uint_as_float(x[2] << 16), __uint_as_float(x[2] & 0xffff0000u), __uint_as_float(x[3] << 16), __uint_as_float(x[3] & 0xffff0000u));
}
__device__ inline float dot4(float4 a, float4 b, float s) {
  return fmaf(a.x, b.x, fmaf(a.y, b.y, fmaf(a.z, b.z, fmaf(a.w, b.w, s))));
}
__device__ inline void fma4(float4& acc, float s, float4 x) {
  acc.x = fmaf(s, x.x, acc.x); acc.y = fmaf(s, x.y, acc.y); acc.z = fmaf(s, x.z, acc.z); acc.w = fmaf(s, x.w, acc.w);
}
__device__ inline float4 ld4(const float* p) { return *reinterpret_cast<const float4*>(p); }

__device__ inline uint32_t cluster_size() {
  uint32_t n;
  asm("mov.u32 %0, %%cluster_nctarank;" : "=r"(n));
  return n;
}
__device__ inline void cluster_meet() {
  __syncwarp();
  asm volatile("barrier.cluster.arrive.aligned;\n\tbarrier.cluster.wait.aligned;" ::: "memory");
}
// four floats at the same place in the shared memory of CTA `rank` of the cluster
__device__ inline float4 ld4_of_rank(const float* p, uint32_t rank) {
  uint32_t at = (uint32_t)__cvta_generic_to_shared(p);
  float4 x;
  asm volatile("mapa.shared::cluster.u32 %0, %0, %1;" : "+r"(at) : "r"(rank));
  asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(x.x), "=f"(x.y), "=f"(x.z), "=f"(x.w) : "r"(at) : "memory");
  return x;
}

template <int D>
__global__ void __launch_bounds__(32 * kBwdWarps)
k_attn_bwd_generic(const uint16_t* __restrict__ Q, const uint16_t* __restrict__ K, const uint16_t* __restrict__ V,
                   const uint16_t* __restrict__ O, const float* __restrict__ LSE, const uint16_t* __restrict__ dO,
                   const int32_t* __restrict__ group_idx, const int32_t* __restrict__ n_groups, Dims dm,
                   uint16_t* __restrict__ dQ, float* __restrict__ dK, float* __restrict__ dV, int32_t* status_word) {
  constexpr int kParts = D / 8, kLoads = kBwdKeys * kParts / 32;     // 16-byte pieces of a row; pieces per lane and tensor
  extern __shared__ __align__(16) uint8_t s_raw[];
  BwdTile<D>& sm = *reinterpret_cast<BwdTile<D>*>(s_raw);
  int* vg = reinterpret_cast<int*>(s_raw + sizeof(BwdTile<D>));      // valid group ids
  __shared__ int s_meta[2];
  __shared__ float s_lse[kBwdRows], s_delta[kBwdRows];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int slices = (dm.rows + kBwdRows - 1) / kBwdRows;
  const int n_split = (int)cluster_size(), split = (int)blockIdx.x % n_split, slice = (int)blockIdx.x / n_split;      // (1 or 2 CTAs)
  const int item = slice / slices, r0 = (slice % slices) * kBwdRows;
  int b, h, qb;
  item_coords(dm, item, b, h, qb);
  const Window w = window_of(dm, qb);

  {
    // warp = row: Q and dO to shared memory, delta = rowsum(dO o O)
    const int r = r0 + warp;
    const bool real = r < dm.rows;
    const int hq = h * dm.G + (real ? r / dm.Bq : 0), sr = qb * dm.Bq + (real ? r % dm.Bq : 0);
    const int64_t q_off = b * dm.qs[0] + hq * dm.qs[1] + sr * dm.qs[2], o_off = b * dm.os[0] + hq * dm.os[1] + sr * dm.os[2];
    float acc = 0.f;
    if (lane < kParts) {
      const uint4 zero = make_uint4(0, 0, 0, 0);
      const uint4 q8 = real ? *reinterpret_cast<const uint4*>(Q + q_off + 8 * lane) : zero;
      const uint4 g8 = real ? *reinterpret_cast<const uint4*>(dO + o_off + 8 * lane) : zero;
      bf16x8_to_smem(&sm.q[warp][8 * lane], q8);
      bf16x8_to_smem(&sm.dO[warp][8 * lane], g8);
      if (real)
        acc = dot_frag<4>(load_frag<4>(O + o_off + 8 * lane), load_frag<4>(dO + o_off + 8 * lane)) +
              dot_frag<4>(load_frag<4>(O + o_off + 8 * lane + 4), load_frag<4>(dO + o_off + 8 * lane + 4));
    }
    acc = warp_sum(acc);
    if (lane == 0) {
      s_delta[warp] = acc;
      s_lse[warp] = real ? LSE[((int64_t)b * dm.Hq + hq) * dm.S + sr] : INFINITY;      // padding rows: P = 0
    }
  }
  const int n_far = w.se + dm.g * build_group_list(dm, w, group_idx + (int64_t)item * dm.width, n_groups[item], vg, s_meta,
                                                   r0 == 0 && split == 0 ? status_word : nullptr);   // (ends with a block barrier)
  const int n_tok = n_far + (w.p0 + dm.Bq - w.ls);
  const uint16_t* Kb = K + b * dm.ks[0] + h * dm.ks[1];
  const uint16_t* Vb = V + b * dm.vs[0] + h * dm.vs[1];
  auto& tile = sm.w[warp];
  uint4 kk[kLoads], vv[kLoads];
  int tok[kLoads];
  auto fetch = [&](int t0) {                       // this lane's pieces of keys t0 .. t0+7 of the list
#pragma unroll
    for (int i = 0; i < kLoads; ++i) {
      const int key = (i * 32 + lane) / kParts, part = (i * 32 + lane) % kParts;
      tok[i] = t0 + key < n_tok ? routed_token(dm, w, vg, n_far, t0 + key) : -1;
      kk[i] = vv[i] = make_uint4(0, 0, 0, 0);
      if (tok[i] >= 0) {
        kk[i] = *reinterpret_cast<const uint4*>(Kb + (int64_t)tok[i] * dm.ks[2] + 8 * part);
        vv[i] = *reinterpret_cast<const uint4*>(Vb + (int64_t)tok[i] * dm.vs[2] + 8 * part);
      }
    }
  };
  const int row = lane >> 2, quad = lane & 3;       // S, dP and dQ: row, keys 2*quad, 2*quad+1 / elements 16*c + 4*quad ..
  const int pos = w.p0 + (r0 + row) % dm.Bq;
  const float lse = s_lse[row], delta = s_delta[row];
  float4 dq[D / 16];
#pragma unroll
  for (int c = 0; c < D / 16; ++c) dq[c] = make_float4(0.f, 0.f, 0.f, 0.f);
  bool waited = false;

  const int round = kBwdKeys * kBwdWarps * n_split;
  fetch(kBwdKeys * (warp + kBwdWarps * split));
  for (int t0 = kBwdKeys * (warp + kBwdWarps * split); t0 < n_tok; t0 += round) {
#pragma unroll
    for (int i = 0; i < kLoads; ++i) {
      const int key = (i * 32 + lane) / kParts, part = (i * 32 + lane) % kParts;
      bf16x8_to_smem(&tile.k[key][8 * part], kk[i]);
      bf16x8_to_smem(&tile.v[key][8 * part], vv[i]);
      if (part == 0) tile.tok[key] = tok[i];
    }
    __syncwarp();
    fetch(t0 + round);
    {
      float s[2] = {0.f, 0.f}, dp[2] = {0.f, 0.f};
#pragma unroll 8
      for (int e = 0; e < D; e += 4) {
        const float4 q4 = ld4(&sm.q[row][e]), g4 = ld4(&sm.dO[row][e]);
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          s[u] = dot4(q4, ld4(&tile.k[2 * quad + u][e]), s[u]);
          dp[u] = dot4(g4, ld4(&tile.v[2 * quad + u][e]), dp[u]);
        }
      }
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const int t = tile.tok[2 * quad + u];
        const float p = t >= 0 && t <= pos ? __expf(s[u] * dm.scale - lse) : 0.f;
        tile.p[row][2 * quad + u] = p;
        tile.ds[row][2 * quad + u] = p * (dp[u] - delta) * dm.scale;
      }
    }
    __syncwarp();
#pragma unroll
    for (int key = 0; key < kBwdKeys; ++key) {
      const float ds = tile.ds[row][key];
#pragma unroll
      for (int c = 0; c < D / 16; ++c) fma4(dq[c], ds, ld4(&tile.k[key][16 * c + 4 * quad]));
    }
    const int mine = tile.tok[row];                 // dK, dV: key `row` of the eight
    if (__any_sync(0xffffffffu, mine >= dm.H)) {
      float4 gk[D / 16], gv[D / 16];
#pragma unroll
      for (int c = 0; c < D / 16; ++c) gk[c] = gv[c] = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int r = 0; r < kBwdRows; ++r) {
        const float ds = tile.ds[r][row], p = tile.p[r][row];
#pragma unroll
        for (int c = 0; c < D / 16; ++c) {
          fma4(gk[c], ds, ld4(&sm.q[r][16 * c + 4 * quad]));
          fma4(gv[c], p, ld4(&sm.dO[r][16 * c + 4 * quad]));
        }
      }
      if (!waited) {
        // dK and dV are zeroed by the launch before this one, which this one may overlap
        asm volatile("griddepcontrol.wait;" ::: "memory");
        waited = true;
      }
      if (mine >= dm.H) {
        const int64_t off = (((int64_t)b * dm.Hkv + h) * dm.S + (mine - dm.H)) * D + 4 * quad;
#pragma unroll
        for (int c = 0; c < D / 16; ++c) {
          atomicAdd(reinterpret_cast<float4*>(dK + off + 16 * c), gk[c]);
          atomicAdd(reinterpret_cast<float4*>(dV + off + 16 * c), gv[c]);
        }
      }
    }
    __syncwarp();
  }
  // the warps' dQ sums meet in the K tiles
#pragma unroll
  for (int c = 0; c < D / 16; ++c) *reinterpret_cast<float4*>(&tile.k[row][16 * c + 4 * quad]) = dq[c];
  if (n_split > 1) cluster_meet();
  else __syncthreads();
  // (of a cluster every CTA writes its share of the rows)
  if (r0 + warp < dm.rows && lane < D / 4 && warp % n_split == split) {
    float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int u = 0; u < kBwdWarps; ++u) fma4(a, 1.f, ld4(&sm.w[u].k[warp][4 * lane]));
    if (n_split > 1) {
#pragma unroll
      for (int u = 0; u < kBwdWarps; ++u) fma4(a, 1.f, ld4_of_rank(&sm.w[u].k[warp][4 * lane], split ^ 1));
    }
    const int r = r0 + warp, hq = h * dm.G + r / dm.Bq, sr = qb * dm.Bq + r % dm.Bq;
    Frag<4> f;
    f.v[0] = a.x; f.v[1] = a.y; f.v[2] = a.z; f.v[3] = a.w;
    store_frag_bf16<4>(dQ + b * dm.qs[0] + hq * dm.qs[1] + sr * dm.qs[2] + 4 * lane, f);
  }
  if (n_split > 1) cluster_meet();               // (the other CTA may still be reading this one's shared memory)
}

// dK and dV to zero, one launch for both tensors (n elements each, a multiple of 8).  It waits for what is before it ahead of
// releasing the backward, which reads the forward's results at once.
__global__ void __launch_bounds__(256) k_zero_grads(float4* __restrict__ a, float4* __restrict__ b, size_t n4) {
  const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  if (i < n4) a[i] = b[i] = make_float4(0.f, 0.f, 0.f, 0.f);
}

static size_t token_smem_bytes(const Dims& dm) {
  return sizeof(int) * ((size_t)max_routed_tokens(dm) + dm.width + 4);
}

// dK/dV accumulators (fp32, adjacent: dV's follow dK's) -> the two bf16 outputs, eight elements per thread
__global__ void __launch_bounds__(256) k_grads_to_bf16(const float4* __restrict__ src, uint4* __restrict__ dst_k,
                                                       uint4* __restrict__ dst_v, size_t n8) {
  const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  // (a no-op unless launched with programmatic serialization: then the sums are complete only from here on)
  asm volatile("griddepcontrol.wait;" ::: "memory");
  if (i >= 2 * n8) return;
  const float4 a = src[2 * i], b = src[2 * i + 1];
  const __nv_bfloat162 h0 = __floats2bfloat162_rn(a.x, a.y), h1 = __floats2bfloat162_rn(a.z, a.w);
  const __nv_bfloat162 h2 = __floats2bfloat162_rn(b.x, b.y), h3 = __floats2bfloat162_rn(b.z, b.w);
  uint4* dst = i < n8 ? dst_k + i : dst_v + (i - n8);
  *dst = make_uint4(*reinterpret_cast<const uint32_t*>(&h0), *reinterpret_cast<const uint32_t*>(&h1),
                    *reinterpret_cast<const uint32_t*>(&h2), *reinterpret_cast<const uint32_t*>(&h3));
}

int launch_grads_to_bf16(const float* src, void* dst_k, void* dst_v, size_t n, bool after_sweep, cudaStream_t st) {
  const size_t n8 = n / 8;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)((2 * n8 + 255) / 256));
  cfg.blockDim = dim3(256);
  cfg.stream = st;
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &attr;
  cfg.numAttrs = after_sweep ? 1 : 0;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, k_grads_to_bf16, (const float4*)src, (uint4*)dst_k, (uint4*)dst_v, n8);
  count_launch(HGA_KERNELS_AUX);
  return record_cuda(e);
}

int launch_attn_fwd_generic(const Dims& dm, const void* Q, const void* K, const void* V,
                            const int32_t* group_idx, const int32_t* n_groups, void* O, float* LSE,
                            int32_t* status_word, cudaStream_t st) {
  const int items = dm.B * dm.Hkv * dm.NQB;
  const size_t smem = token_smem_bytes(dm);
  if (smem > 200 * 1024) return HGA_ERR_UNSUPPORTED;
  cudaError_t e;
  if (dm.d == 128) {
    e = cudaFuncSetAttribute(k_attn_fwd_generic<128>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return record_cuda(e);
    k_attn_fwd_generic<128><<<items, kAttnThreads, smem, st>>>(
        (const uint16_t*)Q, (const uint16_t*)K, (const uint16_t*)V, group_idx, n_groups, dm,
        (uint16_t*)O, LSE, status_word);
  } else {
    e = cudaFuncSetAttribute(k_attn_fwd_generic<64>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return record_cuda(e);
    k_attn_fwd_generic<64><<<items, kAttnThreads, smem, st>>>(
        (const uint16_t*)Q, (const uint16_t*)K, (const uint16_t*)V, group_idx, n_groups, dm,
        (uint16_t*)O, LSE, status_word);
  }
  count_launch(HGA_KERNELS_FWD_GENERIC);
  return record_cuda(cudaGetLastError());
}

// SMs of the current device
static int multiprocessors() {
  static std::atomic<int> known[64];
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev >= 64) return 0;
  int n = known[dev].load(std::memory_order_relaxed);
  if (n == 0 && cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess) known[dev].store(n, std::memory_order_relaxed);
  return n;
}

template <int D>
static int bwd_generic(const Dims& dm, const uint16_t* Q, const uint16_t* K, const uint16_t* V,
                       const uint16_t* O, const float* LSE, const uint16_t* dO,
                       const int32_t* group_idx, const int32_t* n_groups, uint16_t* dQ, float* dK,
                       float* dV, int32_t* status_word, cudaStream_t st) {
  const size_t smem = sizeof(BwdTile<D>) + sizeof(int) * ((size_t)dm.width + 4);
  if (smem > 227 * 1024) return HGA_ERR_UNSUPPORTED;
  const int rc = ensure_dynamic_smem(reinterpret_cast<const void*>(&k_attn_bwd_generic<D>), smem);
  if (rc) return rc;
  const bool zero = !(dm.flags & HGA_FLAG_BWD_ACCUMULATE);
  if (zero) {
    const size_t n4 = (size_t)dm.B * dm.Hkv * dm.S * D / 4;
    // (set up under the forward's end, like the tensor-core kernels: tiny layer 35.0 -> 34.1 us a whole step)
    PdlLaunch fill(dim3((unsigned)((n4 + 255) / 256)), 256, 0, st, dm.flags);
    const cudaError_t e = cudaLaunchKernelEx(&fill.c, k_zero_grads, (float4*)dK, (float4*)dV, n4);
    if (e != cudaSuccess) return record_cuda(e);
    count_launch(HGA_KERNELS_BWD_GENERIC);
  }
  // Two CTAs per eight rows where both fit the device at once and there is more than a round of keys for the second: tiny layer
  // (64 of them, five rounds) 41.5 -> 38.2 us a whole step.
  const int64_t slices = (int64_t)dm.B * dm.Hkv * dm.NQB * ((dm.rows + kBwdRows - 1) / kBwdRows);
  const bool split = 2 * slices <= multiprocessors() && max_routed_tokens(dm) > kBwdKeys * kBwdWarps;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(split ? 2 * slices : slices));
  cfg.blockDim = dim3(32 * kBwdWarps);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attrs[2];
  cfg.attrs = attrs;
  cfg.numAttrs = 0;
  if (zero) {                               // may start under the zero fill; waits for it before its first add
    attrs[cfg.numAttrs].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attrs[cfg.numAttrs++].val.programmaticStreamSerializationAllowed = 1;
  }
  if (split) {
    attrs[cfg.numAttrs].id = cudaLaunchAttributeClusterDimension;
    attrs[cfg.numAttrs].val.clusterDim.x = 2;
    attrs[cfg.numAttrs].val.clusterDim.y = attrs[cfg.numAttrs].val.clusterDim.z = 1;
    ++cfg.numAttrs;
  }
  const cudaError_t e = cudaLaunchKernelEx(&cfg, k_attn_bwd_generic<D>, Q, K, V, O, LSE, dO, group_idx, n_groups, dm, dQ, dK, dV,
                                           status_word);
  count_launch(HGA_KERNELS_BWD_GENERIC);
  return record_cuda(e);
}

int launch_attn_bwd_generic(const Dims& dm, const void* Q, const void* K, const void* V,
                            const void* O, const float* LSE, const void* dO,
                            const int32_t* group_idx, const int32_t* n_groups, void* dQ, float* dK,
                            float* dV, int32_t* status_word, cudaStream_t st) {
  if (dm.d == 128)
    return bwd_generic<128>(dm, (const uint16_t*)Q, (const uint16_t*)K, (const uint16_t*)V,
                            (const uint16_t*)O, LSE, (const uint16_t*)dO, group_idx, n_groups,
                            (uint16_t*)dQ, dK, dV, status_word, st);
  return bwd_generic<64>(dm, (const uint16_t*)Q, (const uint16_t*)K, (const uint16_t*)V,
                         (const uint16_t*)O, LSE, (const uint16_t*)dO, group_idx, n_groups,
                         (uint16_t*)dQ, dK, dV, status_word, st);
}

}  // namespace hga
