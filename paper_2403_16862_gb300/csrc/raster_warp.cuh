// raster_warp.cuh -- blending of the buckets beyond the group path's 8 GA
// fragments by one warp per pixel.
//
// Up to kCandMax fragments the warp takes the whole bucket; from there up to
// kWarpKeys it holds the bucket's depths in registers (32 per lane), finds a
// depth threshold that the nearest 72 to 128 fragments meet by an
// interpolating search over warp-wide counts, and takes those.  The fragments
// taken are sorted in registers on 32-bit keys and blended.  Where those do not
// order them (equal depths, a depth span of 2^24 FP32 values) the warp sorts a
// whole bucket on its full keys; a selection is left to the CTA path then, and
// where it does not reach t_min.  No barrier is involved, the bucket is read
// from memory once, and the pixels of a CTA's warps overlap.
//
// The transmittances are those of the CTA path bit for bit: products over
// chunks of 32 within blocks of 256 fragments, in the same order.
#pragma once

namespace inpc {
namespace {

// Lanes per fragment and channels per lane of a warp's gathers.
template <int V, int GA>
struct WarpLanes {
  static constexpr int kV = V == 1 ? 1 : 4;
  static constexpr int kL = V == 2 ? 16 : GA;
};

struct WarpCand {  // the fragments a warp works on
  unsigned long long key[kCandMax];
  float alpha[kCandMax];
  uint32_t pos[kCandMax];  // bucket position; of a whole bucket, which needs none, the sort's exchange space
};

// Blends fragments: each group of GL lanes takes one fragment's row at a
// time (lane: VL channels), 32 / GL fragments together.
template <int VL, int GL, class FT>
__device__ __forceinline__ void warp_gather(const RP& P, const FT* __restrict__ feat, uint32_t id, float wk, int take,
                                            float (&C)[VL]) {
  constexpr int kPts = 32 / GL;
  const int lane = threadIdx.x & 31, ch = (lane % GL) * VL;
#pragma unroll 4
  for (int t = 0; t * kPts < take; ++t) {
    const int src = t * kPts + lane / GL;
    const uint32_t idj = __shfl_sync(0xffffffffu, id, src & 31);
    const float wj = __shfl_sync(0xffffffffu, wk, src & 31);
    if (src < take && ch < P.F) {
      float c[VL];
      load_color<VL, FT>(P, feat, idj, ch, c);
#pragma unroll
      for (int v = 0; v < VL; ++v) C[v] = __fmaf_rn(wj, c[v], C[v]);
    }
  }
}

// Transmittance of chunk r (32 fragments) of a block of 256 in the CTA
// path's order: products within the chunk, times the product `pre` of the
// chunks in front.
__device__ __forceinline__ void chunk256(const Group<32>& G, float a, float& pre, float& Tk, float& Tn) {
  const float incl = __fmul_rn(pre, G.prod_scan(__fsub_rn(1.0f, a)));
  const float up = __shfl_up_sync(0xffffffffu, incl, 1);
  Tk = G.lg > 0 ? up : pre;
  Tn = incl;
  pre = __shfl_sync(0xffffffffu, incl, 31);
}

// Sorts the C <= 32 R candidates by depth: element 32 r + lane of the order
// is candidate k[r] & 255.  False when 32-bit keys (depth field above the
// nearest one's, candidate) do not order them: two equal depths (the point
// index decides) or a span of 2^24 FP32 values.
template <int R>
__device__ __forceinline__ bool sort_candidates(const Group<32>& G, const RP& P, const WarpCand& S, int C,
                                                uint32_t (&k)[R]) {
  uint32_t lo = 0xFFFFFFFFu, hi = 0u;
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const int e = r * 32 + G.lg;
    k[r] = e < C ? (uint32_t)(S.key[e] >> P.idb) : 0u;
    if (e < C) {
      lo = min(lo, k[r]);
      hi = max(hi, k[r]);
    }
  }
  lo = __reduce_min_sync(0xffffffffu, lo);
  hi = __reduce_max_sync(0xffffffffu, hi);
  if (hi - lo >= 0xFFFFFFu) return false;
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const int e = r * 32 + G.lg;
    k[r] = e < C ? ((k[r] - lo) << 8) | (uint32_t)e : 0xFFFFFFFFu;
  }
  reg_sort32<32, R>(G, k, C);
  bool tie = false;
#pragma unroll
  for (int r = 0; r < R; ++r) {
    uint32_t nx = __shfl_down_sync(0xffffffffu, k[r], 1);
    const uint32_t n0 = __shfl_sync(0xffffffffu, k[r + 1 < R ? r + 1 : r], 0);
    if (G.lg == 31) nx = r + 1 < R ? n0 : 0xFFFFFFFFu;
    if (r * 32 + G.lg + 1 < C && (nx >> 8) == (k[r] >> 8)) tie = true;
  }
  return !__any_sync(0xffffffffu, tie);
}

// S.pos = the C candidates in the order of their full keys (the network of
// bitonic_sort_idx, its indices by shifts and masks).
__device__ __forceinline__ void warp_sort_full(WarpCand& S, int C) {
  const int lane = threadIdx.x & 31;
  for (int e = lane; e < C; e += 32) S.pos[e] = (uint32_t)e;
  __syncwarp();
  for (int k = 2; (k >> 1) < C; k <<= 1) {
    for (int j = k >> 1; j > 0; j >>= 1) {
      const int flip = 2 * j == k ? k - 1 : j;
      for (int q = lane; 2 * q < C + k; q += 32) {
        const int lo = 2 * q - (q & (j - 1)), hi = lo ^ flip;
        if (hi < C) {
          const uint32_t a = S.pos[lo], b = S.pos[hi];
          if (S.key[a] > S.key[b]) {
            S.pos[lo] = b;
            S.pos[hi] = a;
          }
        }
      }
      __syncwarp();
    }
  }
}

// Sorts the C <= 32 R candidates (kWhole: the whole bucket) and blends
// the pixel.  False (nothing written) when a selection's sort leaves it open
// or its candidates do not reach t_min.  A selection is not sorted on full
// keys: its equal depths are rare, and such pixels become the launch's tail
// (19,200 pixels of 520 fragments, 64 channels: 84 us, 91 us with them).  Whole
// buckets are, for they may be all ties: 600,000 points in one plane of depth
// on 200 x 160 pixels, 8 channels, forward 664 us left to the CTA path, 190 us
// here; at random depths 143 and 125 us.
template <int V, int GA, class FT, int R, bool kWhole>
__device__ __forceinline__ bool blend_candidates(const Group<32>& G, const RP& P, const RasterWs& ws, uint32_t s0,
                                                 int C, long long pix, WarpCand& S,
                                                 const FT* __restrict__ feat, FT* __restrict__ image,
                                                 float* __restrict__ T_final, int32_t* __restrict__ n_contrib) {
  uint32_t k[R];
  if (!sort_candidates<R>(G, P, S, C, k)) {
    if constexpr (!kWhole) return false;
    warp_sort_full(S, C);
#pragma unroll
    for (int r = 0; r < R; ++r) k[r] = r * 32 + G.lg < C ? S.pos[r * 32 + G.lg] : 0xFFu;
  }
  uint32_t id[R];
#pragma unroll
  for (int r = 0; r < R; ++r) id[r] = r * 32 + G.lg < C ? (uint32_t)(S.key[k[r] & 255u] & P.idm) : 0u;
  if constexpr (V == 2) {
#pragma unroll
    for (int r = 0; r < (R < 2 ? R : 2); ++r)
      if (r * 32 + G.lg < C) prefetch_row64(feat, id[r]);
  }
  float wk[R];
  float pre = 1.0f, T = 1.0f;
  int cnt = 0;
  bool stop = false;
#pragma unroll
  for (int r = 0; r < R; ++r) {
    wk[r] = 0.f;
    const int b = r * 32;
    if (b < C && !stop) {
      const bool valid = b + G.lg < C;
      const float a = valid ? S.alpha[k[r] & 255u] : 0.f;
      float Tk, Tn;
      chunk256(G, a, pre, Tk, Tn);
      const unsigned st = __ballot_sync(0xffffffffu, valid && Tn < P.t_min);
      stop = st != 0;
      const int take = stop ? __ffs(st) : min(32, C - b);
      if (G.lg < take) wk[r] = __fmul_rn(Tk, a);
      cnt += take;
      T = __shfl_sync(0xffffffffu, Tn, take - 1);
    }
  }
  if (!kWhole && !stop) return false;
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const int j = r * 32 + G.lg;
    if (j < cnt) ws.order[s0 + j] = make_uint2(kWhole ? k[r] & 255u : S.pos[k[r] & 255u], id[r]);
  }
  if constexpr (V == 2) {  // F = 64
    float acc[16];
#pragma unroll
    for (int e = 0; e < 16; ++e) acc[e] = 0.f;
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const int take = min(32, cnt - 32 * r);
      if (take > 0) slots_gather(G, P, feat, id[r], wk[r], take, acc);
    }
    slots_write(G, acc, pix, image);
  } else {
    constexpr int VL = WarpLanes<V, GA>::kV, GL = WarpLanes<V, GA>::kL;
    float Cc[VL];
#pragma unroll
    for (int v = 0; v < VL; ++v) Cc[v] = 0.f;
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const int take = min(32, cnt - 32 * r);
      if (take > 0) warp_gather<VL, GL>(P, feat, id[r], wk[r], take, Cc);
    }
#pragma unroll
    for (int o = GL; o < 32; o <<= 1)
#pragma unroll
      for (int v = 0; v < VL; ++v) Cc[v] = __fadd_rn(Cc[v], __shfl_xor_sync(0xffffffffu, Cc[v], o));
    if (G.lg < GL) write_pixel<VL>(P, pix, G.lg * VL, Cc, image);
  }
  if (G.lg == 0) {
    T_final[pix] = T;
    n_contrib[pix] = cnt;
  }
  return true;
}

// A whole bucket of m <= kCandMax fragments.
template <int V, int GA, class FT>
__device__ __forceinline__ bool blend_whole(const Group<32>& G, const RP& P, const RasterWs& ws, uint32_t s0, int m,
                                            long long q, WarpCand& S, const FT* __restrict__ feat,
                                            FT* __restrict__ image, float* __restrict__ T_final,
                                            int32_t* __restrict__ n_contrib) {
  __syncwarp();
  for (int e = G.lg; e < m; e += 32) {
    S.key[e] = ws.keys[s0 + e];
    S.alpha[e] = ws.alpha[s0 + e];
  }
  __syncwarp();
  if (m <= 32) return blend_candidates<V, GA, FT, 1, true>(G, P, ws, s0, m, q, S, feat, image, T_final, n_contrib);
  if (m <= 64) return blend_candidates<V, GA, FT, 2, true>(G, P, ws, s0, m, q, S, feat, image, T_final, n_contrib);
  if (m <= 128) return blend_candidates<V, GA, FT, 4, true>(G, P, ws, s0, m, q, S, feat, image, T_final, n_contrib);
  return blend_candidates<V, GA, FT, 8, true>(G, P, ws, s0, m, q, S, feat, image, T_final, n_contrib);
}

// The fragments with a depth field of at most t, in bucket order, into S.
// d: the bucket's depth fields, element 32 r + lane (0xFFFFFFFF beyond m).
__device__ __forceinline__ void take_front(const Group<32>& G, const RasterWs& ws, uint32_t s0, const uint32_t (&d)[32],
                                           int m, uint32_t t, int C, WarpCand& S) {
  const unsigned below = (1u << G.lg) - 1u;
  int at = 0;
  __syncwarp();
#pragma unroll
  for (int r = 0; r < 32; ++r) {
    if (r * 32 < m) {
      const bool in = d[r] <= t;
      const unsigned b = __ballot_sync(0xffffffffu, in);
      if (in) S.pos[at + __popc(b & below)] = (uint32_t)(r * 32 + G.lg);
      at += __popc(b);
    }
  }
  __syncwarp();
  for (int e = G.lg; e < C; e += 32) {
    const uint32_t p = S.pos[e];
    S.key[e] = ws.keys[s0 + p];
    S.alpha[e] = ws.alpha[s0 + p];
  }
  __syncwarp();
}

// A bucket of kCandMax < m <= kWarpKeys fragments: the nearest ones only.
template <int V, int GA, class FT>
__device__ __forceinline__ bool blend_selected(const Group<32>& G, const RP& P, const RasterWs& ws, uint32_t s0, int m,
                                               long long q, WarpCand& S, const FT* __restrict__ feat,
                                               FT* __restrict__ image, float* __restrict__ T_final,
                                               int32_t* __restrict__ n_contrib) {
  // A pixel that blends more than it selects is done again by a CTA.  2.5M points
  // on 160 x 120 pixels (520 fragments each), 4 channels, forward with and
  // without the selection: alphas of 0.2 to 0.8 (64 blended) 233 and 466 us; of
  // 0.02 to 0.3 (220 blended) 1209 and 1159; of 0.001 to 0.01 (all) 1266 and 1216.
  constexpr int kLeast = 72, kMost = 128;
  uint32_t d[32];
  uint32_t lo = 0xFFFFFFFFu, hi = 0u;
#pragma unroll
  for (int r = 0; r < 32; ++r) {
    const int e = r * 32 + G.lg;
    d[r] = e < m ? (uint32_t)(ws.keys[s0 + e] >> P.idb) : 0xFFFFFFFFu;
  }
#pragma unroll
  for (int r = 0; r < 32; ++r) {
    lo = min(lo, d[r]);
    if (r * 32 + G.lg < m) hi = max(hi, d[r]);
  }
  lo = __reduce_min_sync(0xffffffffu, lo);
  hi = __reduce_max_sync(0xffffffffu, hi);
  // count(d <= a) = ca < kLeast and count(d <= b) = cb > kMost bracket the
  // threshold; a starts one below the nearest depth (its bits are positive)
  uint32_t a = lo - 1u, b = hi, t = 0;
  int ca = 0, cb = m, C = 0;
#pragma unroll 1
  for (int step = 0; step < 40 && b - a > 1u; ++step) {
    // interpolate the count between the ends, then halve
    const uint32_t span = b - a;
    uint32_t off = span >> 1;
    if (step < 6) off = (uint32_t)((float)span * ((float)((kLeast + kMost) / 2 - ca) / (float)(cb - ca)));
    t = a + min(max(off, 1u), span - 1u);
    int c = 0;
#pragma unroll
    for (int r = 0; r < 32; ++r) c += d[r] <= t ? 1 : 0;
    c = (int)__reduce_add_sync(0xffffffffu, (unsigned)c);
    if (c < kLeast) {
      a = t;
      ca = c;
    } else if (c > kMost) {
      b = t;
      cb = c;
    } else {
      C = c;
      break;
    }
  }
  if (C == 0) return false;  // equal depths make the count jump over the window
  take_front(G, ws, s0, d, m, t, C, S);
  return blend_candidates<V, GA, FT, 4, false>(G, P, ws, s0, C, q, S, feat, image, T_final, n_contrib);
}

// The warps' launch: the pixels with 8 GA < m <= kCandMax fragments (GA < 32;
// the list's back), and those with up to kWarpKeys (its front) where there
// are enough of them: few pixels are done sooner by a CTA each
// (k_blend_fwd_heavy), since one pixel's chain through this kernel takes a
// warp about 25 us with the instructions still to be fetched.
constexpr uint32_t kSelectMin = 4096;

template <int V, int GA, class FT>
__global__ void __launch_bounds__(kThreads, 3) k_blend_fwd_warp(RP P, const FT* __restrict__ feat, RasterWs ws,
                                                                FT* __restrict__ image, float* __restrict__ T_final,
                                                                int32_t* __restrict__ n_contrib) {
  start_next();
  __shared__ WarpCand cand[kWarps];
  const Group<32> G;
  WarpCand& S = cand[threadIdx.x >> 5];
  const uint32_t n_mid = *ws.select_count, n_select = n_mid >= kSelectMin ? n_mid : 0u;
  const uint32_t n_list = n_select + (GA < 32 ? *ws.warp_count : 0u);
  for (;;) {
    uint32_t h = 0;
    if (G.lg == 0) h = atomicAdd(ws.warp_next, 1u);
    h = G.bcast(h, 0);
    if (h >= n_list) break;
    const uint32_t q = h < n_select ? ws.mid[h] : ws.mid[P.n_pix - 1 - (h - n_select)];
    const uint32_t s0 = ws.pix_start[q];
    const int m = (int)(ws.pix_start[q + 1] - s0);
    bool done = false;
    if (h < n_select) {
      done = blend_selected<V, GA, FT>(G, P, ws, s0, m, q, S, feat, image, T_final, n_contrib);
    } else {
      if constexpr (GA < 32) done = blend_whole<V, GA, FT>(G, P, ws, s0, m, q, S, feat, image, T_final, n_contrib);
    }
    if (!done && G.lg == 0) ws.heavy[atomicAdd(ws.heavy_count, 1u)] = q;
  }
}

// Backward of up to 32 R blended fragments (GA < 32): transmittances as
// in blend_candidates over the blended prefix the forward recorded, then back
// to front, each lane holding one fragment of the chunk; the dot products
// c_k . g by groups of GL lanes.
template <int V, int GA, class FT, int R>
__device__ __forceinline__ void blend_bwd_warp(const Group<32>& G, const RP& P, const RasterWs& ws, uint32_t s0, int m,
                                               int nb, long long pix, const FT* __restrict__ feat,
                                               const float* __restrict__ d_image) {
  constexpr int VL = WarpLanes<V, GA>::kV, GL = WarpLanes<V, GA>::kL, kPts = 32 / GL;
  const int qy = (int)(pix / P.cam.W), qx = (int)(pix - (long long)qy * P.cam.W);
  const int ch = (G.lg % GL) * VL;
  uint32_t id[R];
  float a[R], Tk[R];
  float pre = 1.0f;
#pragma unroll
  for (int r = 0; r < R; ++r) {
    id[r] = 0;
    a[r] = Tk[r] = 0.f;
    if (r * 32 + G.lg < nb) {
      const uint2 o = order_at(P, ws, s0, m, r * 32 + G.lg);
      id[r] = o.y;
      a[r] = ws.alpha[s0 + o.x];
    }
  }
#pragma unroll
  for (int r = 0; r < R; ++r) {
    float Tn;
    if (r * 32 < nb) chunk256(G, a[r], pre, Tk[r], Tn);
  }
  float g[VL];
  if (ch < P.F) load_vec<VL>(d_image + pix * P.F + ch, g);
  else
#pragma unroll
    for (int v = 0; v < VL; ++v) g[v] = 0.f;
  float S = 0.f;  // sum over the fragments behind the chunk
#pragma unroll
  for (int r = R - 1; r >= 0; --r) {
    const int take = min(32, nb - r * 32);
    if (take <= 0) continue;
    const bool mine = G.lg < take;
    const uint32_t dst = mine ? frag_index(ws, id[r], qx, qy) : 0u;
    float mydot = 0.f;
#pragma unroll 4
    for (int t = 0; t * kPts < take; ++t) {
      const int src = t * kPts + G.lg / GL;
      const uint32_t idj = __shfl_sync(0xffffffffu, id[r], src & 31);
      float part = 0.f;
      if (src < take && ch < P.F) {
        float c[VL];
        load_color<VL, FT>(P, feat, idj, ch, c);
#pragma unroll
        for (int v = 0; v < VL; ++v) part = __fmaf_rn(c[v], g[v], part);
      }
#pragma unroll
      for (int o = GL / 2; o > 0; o >>= 1) part = __fadd_rn(part, __shfl_xor_sync(0xffffffffu, part, o));
      // fragment src's dot product goes to lane src
      const float v = __shfl_sync(0xffffffffu, part, (G.lg % kPts) * GL);
      if (G.lg / kPts == t) mydot = v;
    }
    const float wk = __fmul_rn(Tk[r], a[r]);
    const float suf = G.suffix_scan(__fmul_rn(wk, mydot));
    const float Sk = __fadd_rn(S, G.shift_down(suf));
    const float da = __fsub_rn(__fmul_rn(Tk[r], mydot), __fdiv_rn(Sk, __fsub_rn(1.0f, a[r])));
    if (mine) ws.fscal[dst] = make_float2(wk, da);
    S = __fadd_rn(S, G.bcast(suf, 0));
  }
}

}  // namespace
}  // namespace inpc
