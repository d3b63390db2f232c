// raster_small.cuh -- 64-channel blending of buckets of at most 16 fragments:
// several pixels per warp.
//
// LP lanes take one pixel (8 lanes up to 8 fragments, 16 up to 16), so a warp
// works on 32 / LP pixels at a time.  Each lane holds one fragment while the
// bucket is ordered (by rank: as many comparisons as fragments, exact on the
// full keys) and scanned, and 64 / LP channels while the rows are gathered,
// so the pixel needs no reduction over lanes.  One warp per pixel spends
// about 250 instructions on a bucket of four fragments and is bound by
// instruction issue (1M points on 1237 x 822 pixels, 78 % issue slots busy).
// The product scan over the first 16 fragments is the one of 32 lanes, so
// transmittances and counts are the same bits.
#pragma once

namespace inpc {
namespace {

// This lane's channels of a row: 64 / LP of them, kB bytes at a time.
template <class FT, int LP>
struct LaneRow {
  static constexpr int kCh = 64 / LP;                        // channels per lane
  static constexpr int kVec = sizeof(FT) == 4 ? 4 : kCh;     // channels per load (FP32: 4; BF16: 4 or 8)
  static constexpr int kLoads = kCh / kVec;
  // channel of load i, element 0
  __device__ static int channel(int sl, int i) { return kVec * (sl + LP * i); }
  __device__ static void load(const FT* __restrict__ row, int sl, float (&c)[kCh]) {
#pragma unroll
    for (int i = 0; i < kLoads; ++i) {
      const FT* p = row + channel(sl, i);
      if constexpr (kVec == 8) {
        const uint4 raw = __ldg(reinterpret_cast<const uint4*>(p));
        const uint32_t w[4] = {raw.x, raw.y, raw.z, raw.w};
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          c[2 * k] = __uint_as_float(w[k] << 16);
          c[2 * k + 1] = __uint_as_float(w[k] & 0xFFFF0000u);
        }
      } else {
        load_vec<4>(p, &c[4 * i]);
      }
    }
  }
  // FP32 values in the same channel layout
  __device__ static void load_f32(const float* __restrict__ row, int sl, float (&c)[kCh]) {
#pragma unroll
    for (int e = 0; e < kCh; e += 4) load_vec<4>(row + channel(sl, e / kVec) + e % kVec, &c[e]);
  }
  __device__ static void store(FT* __restrict__ row, int sl, const float (&c)[kCh]) {
#pragma unroll
    for (int i = 0; i < kLoads; ++i) {
      FT* p = row + channel(sl, i);
      if constexpr (sizeof(FT) == 4) {
        __stcs(reinterpret_cast<float4*>(p), make_float4(c[4 * i], c[4 * i + 1], c[4 * i + 2], c[4 * i + 3]));
      } else {
        uint32_t w[kVec / 2];
#pragma unroll
        for (int k = 0; k < kVec / 2; ++k) {
          __nv_bfloat162 v = __floats2bfloat162_rn(c[2 * k], c[2 * k + 1]);
          w[k] = *reinterpret_cast<uint32_t*>(&v);
        }
        if constexpr (kVec == 8) __stcs(reinterpret_cast<uint4*>(p), make_uint4(w[0], w[1], w[2], w[3]));
        else __stcs(reinterpret_cast<uint2*>(p), make_uint2(w[0], w[1]));
      }
    }
  }
};

// Transmittance in front of and behind this lane's fragment, and the number
// of blended fragments of its pixel (m valid lanes).
template <int LP>
__device__ __forceinline__ void small_transmittance(const Group<LP>& G, const RP& P, float a, int m, float& Tk,
                                                    float& Tn, int& take) {
  const float incl = G.prod_scan(__fsub_rn(1.0f, a));
  const float up = __shfl_up_sync(G.mask, incl, 1, LP);
  Tk = G.lg > 0 ? up : 1.0f;
  Tn = incl;
  const unsigned st = G.ballot(G.lg < m && Tn < P.t_min);
  take = st ? __ffs(st) : m;
}

// One pixel per LP lanes; m = 0: no pixel for these lanes.  Every lane of the
// warp calls it.  src: the lanes' exchange space (LP bytes per pixel).
template <class FT, int LP>
__device__ __forceinline__ void blend_fwd_small(const Group<LP>& G, const RP& P, const RasterWs& ws, uint32_t s0, int m,
                                                long long pix, uint8_t* src, const FT* __restrict__ feat,
                                                FT* __restrict__ image, float* __restrict__ T_final,
                                                int32_t* __restrict__ n_contrib) {
  using Row = LaneRow<FT, LP>;
  const bool valid = G.lg < m;
  const unsigned long long key = valid ? ws.keys[s0 + G.lg] : ~0ull;
  const float a_in = valid ? ws.alpha[s0 + G.lg] : 0.f;
  int rank = 0;
#pragma unroll
  for (int j = 0; j < LP; ++j) rank += __shfl_sync(0xffffffffu, key, j, LP) < key ? 1 : 0;
  if (valid) src[rank] = (uint8_t)G.lg;
  __syncwarp();
  const int from = valid ? src[G.lg] : 0;
  __syncwarp();
  const uint32_t id = (uint32_t)(__shfl_sync(0xffffffffu, key, from, LP) & P.idm);
  const float as = __shfl_sync(0xffffffffu, a_in, from, LP);
  const float a = valid ? as : 0.f;
  float Tk, Tn;
  int take;
  small_transmittance(G, P, a, m, Tk, Tn, take);
  const float wk = __fmul_rn(Tk, a);
  if (G.lg < take) ws.order[s0 + G.lg] = make_uint2((uint32_t)from, id);
  float C[Row::kCh];
#pragma unroll
  for (int e = 0; e < Row::kCh; ++e) C[e] = 0.f;
  const int most = (int)__reduce_max_sync(0xffffffffu, (unsigned)take);
#pragma unroll 4
  for (int j = 0; j < most; ++j) {
    const uint32_t idj = __shfl_sync(0xffffffffu, id, j, LP);
    const float wj = __shfl_sync(0xffffffffu, wk, j, LP);
    if (j < take) {
      float c[Row::kCh];
      Row::load(feat + 64ll * idj, G.lg, c);
      if (P.head && G.lg == 0) c[0] = 1.0f;
#pragma unroll
      for (int e = 0; e < Row::kCh; ++e) C[e] = __fmaf_rn(wj, c[e], C[e]);
    }
  }
  const float T = __shfl_sync(0xffffffffu, Tn, max(take, 1) - 1, LP);
  if (m > 0) {
    Row::store(image + pix * 64, G.lg, C);
    if (G.lg == 0) {
      T_final[pix] = T;
      n_contrib[pix] = take;
    }
  }
}

// The backward of nb <= LP blended fragments, as blend_bwd_slots.
template <class FT, int LP>
__device__ __forceinline__ void blend_bwd_small(const Group<LP>& G, const RP& P, const RasterWs& ws, uint32_t s0, int m,
                                                int nb, long long pix, const FT* __restrict__ feat,
                                                const float* __restrict__ d_image) {
  using Row = LaneRow<FT, LP>;
  const bool valid = G.lg < nb;
  float a = 0.f;
  uint32_t id = 0, dst = 0;
  if (valid) {
    const uint2 o = order_at(P, ws, s0, m, G.lg);
    id = o.y;
    a = ws.alpha[s0 + o.x];
    const int qy = (int)(pix / P.cam.W), qx = (int)(pix - (long long)qy * P.cam.W);
    dst = frag_index(ws, id, qx, qy);
  }
  float g[Row::kCh];
#pragma unroll
  for (int e = 0; e < Row::kCh; ++e) g[e] = 0.f;
  if (nb > 0) Row::load_f32(d_image + pix * 64, G.lg, g);
  float Tk, Tn;
  int take;
  small_transmittance(G, P, a, nb, Tk, Tn, take);
  float mydot = 0.f;
  const int most = (int)__reduce_max_sync(0xffffffffu, (unsigned)take);
#pragma unroll 4
  for (int j = 0; j < most; ++j) {
    const uint32_t idj = __shfl_sync(0xffffffffu, id, j, LP);
    float part = 0.f;
    if (j < take) {
      float c[Row::kCh];
      Row::load(feat + 64ll * idj, G.lg, c);
      if (P.head && G.lg == 0) c[0] = 1.0f;
#pragma unroll
      for (int e = 0; e < Row::kCh; ++e) part = __fmaf_rn(c[e], g[e], part);
    }
#pragma unroll
    for (int o = LP / 2; o > 0; o >>= 1) part = __fadd_rn(part, __shfl_xor_sync(0xffffffffu, part, o, LP));
    if (G.lg == j) mydot = part;
  }
  const bool mine = G.lg < take;
  const float wk = mine ? __fmul_rn(Tk, a) : 0.f;
  const float suf = G.suffix_scan(__fmul_rn(wk, mydot));  // this fragment and those behind it
  const float behind = G.shift_down(suf);
  const float da = __fsub_rn(__fmul_rn(Tk, mydot), __fdiv_rn(behind, __fsub_rn(1.0f, a)));
  if (mine) ws.fscal[dst] = make_float2(wk, da);
}

}  // namespace
}  // namespace inpc
