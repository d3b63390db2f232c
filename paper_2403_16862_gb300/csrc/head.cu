// head.cu -- the view-dependent appearance head (Sec. 3.3): spherical
// contraction of the query positions into [0, 1]^3 (mip-NeRF 360), and per
// point the opacity alpha_h = 1 - exp(-exp(h0)) with a 4D color from degree-2
// real spherical harmonics of the viewing direction on the next 36 features
// (channel c uses h[1 + 9 c + k], k < 9), plus its derivative.
//
// The head is evaluated once per point before the rasterizer (which then
// blends 4 channels with given opacities) instead of once per splat inside
// the blend: the point's 37 features are read once, not four times.
#include <cmath>
#include <type_traits>

#include <cuda_bf16.h>

#include "common.cuh"

namespace inpc {
namespace {

struct ShConsts {
  float c0, c1, c2, c20, c22;  // sqrt(1/4pi), sqrt(3/4pi), sqrt(15/4pi), sqrt(5/16pi), sqrt(15/16pi)
  double o[3];                 // camera center -R^T t
};

ShConsts make_consts(const inpc_camera& cam) {
  const double pi = std::acos(-1.0);
  ShConsts k;
  k.c0 = (float)std::sqrt(1.0 / (4.0 * pi));
  k.c1 = (float)std::sqrt(3.0 / (4.0 * pi));
  k.c2 = (float)std::sqrt(15.0 / (4.0 * pi));
  k.c20 = (float)std::sqrt(5.0 / (16.0 * pi));
  k.c22 = (float)std::sqrt(15.0 / (16.0 * pi));
  for (int a = 0; a < 3; ++a)
    k.o[a] = -((double)cam.R[a] * cam.t[0] + (double)cam.R[3 + a] * cam.t[1] + (double)cam.R[6 + a] * cam.t[2]);
  return k;
}

// The direction is formed in FP64: x - o cancels for points near a
// coordinate plane through the camera, and FP32 would lose the small
// component's relative accuracy there.  FP64 runs at a few lanes per SM and
// clock, so the three divisions and the square root are one reciprocal
// square root and three products (about 23 FP64 operations instead of 75;
// the results are rounded to FP32 either way).
__device__ __forceinline__ void sh9(const ShConsts& k, const float* p, float Y[9]) {
  const double vx = (double)p[0] - k.o[0], vy = (double)p[1] - k.o[1], vz = (double)p[2] - k.o[2];
  const double len2 = vx * vx + vy * vy + vz * vz;
  float x = 0.f, y = 0.f, z = 1.f;
  if (len2 > 0.0) {
    const double inv = rsqrt(len2);
    x = (float)(vx * inv);
    y = (float)(vy * inv);
    z = (float)(vz * inv);
  }
  Y[0] = k.c0;
  Y[1] = k.c1 * y;
  Y[2] = k.c1 * z;
  Y[3] = k.c1 * x;
  Y[4] = k.c2 * x * y;
  Y[5] = k.c2 * y * z;
  Y[6] = k.c20 * fmaf(3.f * z, z, -1.f);
  Y[7] = k.c2 * x * z;
  Y[8] = k.c22 * (x * x - y * y);
}

__device__ __forceinline__ float ldf(const float* p) { return __ldg(p); }
__device__ __forceinline__ float ldf(const __nv_bfloat16* p) {
  return __uint_as_float(((uint32_t)__ldg(reinterpret_cast<const unsigned short*>(p))) << 16);
}

__global__ void k_contract(const float* __restrict__ pos, int64_t n, float cx, float cy, float cz, float radius,
                           float* __restrict__ out) {
  for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < n; p += (int64_t)gridDim.x * blockDim.x) {
    const float y0 = __fdiv_rn(__fsub_rn(pos[3 * p + 0], cx), radius);
    const float y1 = __fdiv_rn(__fsub_rn(pos[3 * p + 1], cy), radius);
    const float y2 = __fdiv_rn(__fsub_rn(pos[3 * p + 2], cz), radius);
    const float r = __fsqrt_rn(__fmaf_rn(y2, y2, __fmaf_rn(y1, y1, __fmul_rn(y0, y0))));
    float sc = 1.0f;
    if (r > 1.0f) sc = __fdiv_rn(__fsub_rn(2.0f, __fdiv_rn(1.0f, r)), r);
    out[3 * p + 0] = __fmaf_rn(__fmul_rn(y0, sc), 0.25f, 0.5f);
    out[3 * p + 1] = __fmaf_rn(__fmul_rn(y1, sc), 0.25f, 0.5f);
    out[3 * p + 2] = __fmaf_rn(__fmul_rn(y2, sc), 0.25f, 0.5f);
  }
}

// Four features from element e of a row.
__device__ __forceinline__ float4 ld4(const float* p) { return __ldg(reinterpret_cast<const float4*>(p)); }
__device__ __forceinline__ float4 ld4(const __nv_bfloat16* p) {
  const uint2 r = __ldg(reinterpret_cast<const uint2*>(p));
  return make_float4(__uint_as_float(r.x << 16), __uint_as_float(r.x & 0xFFFF0000u), __uint_as_float(r.y << 16),
                     __uint_as_float(r.y & 0xFFFF0000u));
}

constexpr int kHeadThreads = 128;
constexpr int kHeadFeats = 37;   // opacity and 36 SH features
constexpr int kHeadStride = 41;  // shared-memory row of a point (odd: the lanes' rows start in different banks)

// How the forward reads the rows (2,000,000 FP32 points, us: a thread per point
// reading its row with twice as many threads a CTA, as before the warps; through
// shared memory 4 elements at a time; one at a time; kDirect):
//   64 features           280, 119, 182, -
//   64, at an odd offset  280, -, 182, 252
//   37                    179, -, 277 (175 unrolled), 97
//   71                    183, -, 292 (186), 131
enum class Rows {
  kVec,     // F % 4 == 0, F >= 40 and 4 elements aligned: the first 40 features, 4 at a time
  kOne,     // F % 4 == 0 otherwise: the first 37, one at a time
  kDirect,  // F % 4 != 0: each lane its own row (32 lanes' rows lie in different sectors and cache sets)
};

// A warp takes 32 consecutive points: it reads their rows' first features
// side by side into shared memory, then each lane works on its own point.  (One
// thread per point reading its row directly touched 32 lines per load: 500k
// points, 64 features, 78 us.)
template <class HT, Rows kRows>
__global__ void __launch_bounds__(kHeadThreads) k_sh_head_fwd(ShConsts k, const float* __restrict__ pos,
                                                              const HT* __restrict__ h, int64_t n, int F,
                                                              float* __restrict__ alpha, float* __restrict__ color) {
  constexpr bool kDirect = kRows == Rows::kDirect;
  __shared__ float rows_s[kHeadThreads / 32][kDirect ? 1 : 32 * kHeadStride];
  const int lane = threadIdx.x & 31;
  float* rows = rows_s[threadIdx.x >> 5];
  const int64_t n_warps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t b = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; 32 * b < n; b += n_warps) {
    const int64_t p0 = 32 * b;
    const int np = (int)min((int64_t)32, n - p0);
    __syncwarp();
    if constexpr (kRows == Rows::kVec) {
#pragma unroll
      for (int i = 0; i < 10; ++i) {
        const int pt = (i * 32 + lane) / 10, e = 4 * ((i * 32 + lane) % 10);
        if (pt < np) {
          const float4 v = ld4(h + (p0 + pt) * F + e);
          float* o = rows + pt * kHeadStride + e;
          o[0] = v.x;
          o[1] = v.y;
          o[2] = v.z;
          o[3] = v.w;
        }
      }
    } else if constexpr (kRows == Rows::kOne) {
#pragma unroll 8
      for (int i = lane; i < np * kHeadFeats; i += 32)
        rows[i / kHeadFeats * kHeadStride + i % kHeadFeats] = ldf(h + (p0 + i / kHeadFeats) * F + i % kHeadFeats);
    }
    __syncwarp();
    if (lane >= np) continue;
    const int64_t p = p0 + lane;
    float Y[9];
    sh9(k, pos + 3 * p, Y);
    const auto feat = [&](int f) { return kDirect ? ldf(h + (int64_t)F * p + f) : rows[lane * kHeadStride + f]; };
    alpha[p] = -expm1f(-expf(feat(0)));
    float c[4];
#pragma unroll
    for (int ch = 0; ch < 4; ++ch) {
      float s = 0.f;
#pragma unroll
      for (int q = 0; q < 9; ++q) s = fmaf(Y[q], feat(1 + 9 * ch + q), s);
      c[ch] = s;
    }
    reinterpret_cast<float4*>(color)[p] = make_float4(c[0], c[1], c[2], c[3]);
  }
}

// The derivative: each lane forms one point's basis and color gradient into
// shared memory, then the warp writes the 32 rows of dh side by side (kVec:
// 4 values per lane).  (Each thread writing its own row: 500k points, 64
// features, 178 us.)
template <class HT, bool kVec>
__global__ void __launch_bounds__(kHeadThreads) k_sh_head_bwd(ShConsts k, const float* __restrict__ pos,
                                                              const HT* __restrict__ h, int64_t n, int F,
                                                              const float* __restrict__ d_alpha,
                                                              const float* __restrict__ d_color,
                                                              float* __restrict__ dh) {
  constexpr int kRec = 15;  // basis (9), color gradient (4), opacity path
  __shared__ float rec_s[kHeadThreads / 32][32 * kRec];
  const int lane = threadIdx.x & 31;
  float* rec = rec_s[threadIdx.x >> 5];
  const auto value = [&](const float* r, int f) {
    if (f == 0) return r[13];
    if (f >= kHeadFeats) return 0.f;
    return r[(f - 1) % 9] * r[9 + (f - 1) / 9];
  };
  const int64_t n_warps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t b = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; 32 * b < n; b += n_warps) {
    const int64_t p0 = 32 * b;
    const int np = (int)min((int64_t)32, n - p0);
    __syncwarp();
    if (lane < np) {
      const int64_t p = p0 + lane;
      float Y[9];
      sh9(k, pos + 3 * p, Y);
      float* r = rec + lane * kRec;
#pragma unroll
      for (int q = 0; q < 9; ++q) r[q] = Y[q];
      const float4 g = reinterpret_cast<const float4*>(d_color)[p];
      r[9] = g.x;
      r[10] = g.y;
      r[11] = g.z;
      r[12] = g.w;
      const float e = expf(ldf(h + F * p));
      r[13] = d_alpha[p] * (e * expf(-e));
    }
    __syncwarp();
    float* out = dh + p0 * F;
    if (kVec) {
      const int parts = F / 4;
      for (int i = lane; i < np * parts; i += 32) {
        const float* r = rec + i / parts * kRec;
        const int f = 4 * (i % parts);
        reinterpret_cast<float4*>(out)[i] = make_float4(value(r, f), value(r, f + 1), value(r, f + 2), value(r, f + 3));
      }
    } else {
      for (int i = lane; i < np * F; i += 32) out[i] = value(rec + i / F * kRec, i % F);
    }
  }
}

unsigned grid_for_points(int64_t n) {
  return (unsigned)std::max<int64_t>(1, std::min<int64_t>(ceil_div(n, 256), (int64_t)device_sm_count() * 16));
}

unsigned grid_for_warps(int64_t n) {
  return (unsigned)std::max<int64_t>(1, std::min<int64_t>(ceil_div(n, kHeadThreads), (int64_t)device_sm_count() * 16));
}

inpc_status check_head(const inpc_camera* cam, const float* pos, const void* h, int32_t dtype, int64_t n, int32_t F) {
  if (!cam) return fail(INPC_ERR_INVALID_ARG, "camera is null");
  if (n < 0) return fail(INPC_ERR_INVALID_ARG, "n < 0");
  if (F < 37) return fail(INPC_ERR_INVALID_ARG, "the SH head needs n_channels >= 37 (1 opacity + 36 SH)");
  if (dtype != INPC_F32 && dtype != INPC_BF16) return fail(INPC_ERR_UNSUPPORTED, "dtype must be INPC_F32 or INPC_BF16");
  if (n > 0 && (!pos || !h)) return fail(INPC_ERR_INVALID_ARG, "null pointer");
  return INPC_OK;
}

}  // namespace
}  // namespace inpc

using namespace inpc;

extern "C" inpc_status inpc_contract_positions(const float* pos, int64_t n, const float* center, float radius,
                                               float* out, inpc_stream_t stream) {
  inpc::fault_arg(pos);
  if (n < 0) return fail(INPC_ERR_INVALID_ARG, "n < 0");
  if (n == 0) return INPC_OK;
  if (!pos || !center || !out) return fail(INPC_ERR_INVALID_ARG, "null pointer");
  if (!(radius > 0.0f)) return fail(INPC_ERR_INVALID_ARG, "radius must be positive");
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  k_contract<<<grid_for_points(n), 256, 0, s>>>(pos, n, center[0], center[1], center[2], radius, out);
  return check_launch("k_contract");
}

extern "C" inpc_status inpc_sh_head_fwd(const inpc_camera* cam, const float* pos, const void* h, int32_t h_dtype,
                                        int64_t n, int32_t n_channels, float* alpha_out, float* color_out,
                                        inpc_stream_t stream) {
  inpc::fault_arg(pos);
  INPC_TRY(check_head(cam, pos, h, h_dtype, n, n_channels));
  if (n == 0) return INPC_OK;
  if (!alpha_out || !color_out || !aligned(color_out, 16)) return fail(INPC_ERR_INVALID_ARG, "bad output pointer");
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  const ShConsts k = make_consts(*cam);
  const bool four = aligned(h, h_dtype == INPC_F32 ? 16 : 8);
  const Rows how = n_channels % 4 ? Rows::kDirect : four && n_channels >= 40 ? Rows::kVec : Rows::kOne;
  const auto run = [&](auto kernel, auto* rows) {
    kernel<<<grid_for_warps(n), kHeadThreads, 0, s>>>(k, pos, rows, n, n_channels, alpha_out, color_out);
  };
  const auto read = [&](auto* rows) {
    using HT = std::remove_const_t<std::remove_pointer_t<decltype(rows)>>;
    if (how == Rows::kVec) run(k_sh_head_fwd<HT, Rows::kVec>, rows);
    else if (how == Rows::kOne) run(k_sh_head_fwd<HT, Rows::kOne>, rows);
    else run(k_sh_head_fwd<HT, Rows::kDirect>, rows);
  };
  if (h_dtype == INPC_F32) read(static_cast<const float*>(h));
  else read(static_cast<const __nv_bfloat16*>(h));
  return check_launch("k_sh_head_fwd");
}

extern "C" inpc_status inpc_sh_head_bwd(const inpc_camera* cam, const float* pos, const void* h, int32_t h_dtype,
                                        int64_t n, int32_t n_channels, const float* d_alpha, const float* d_color,
                                        float* dh_out, inpc_stream_t stream) {
  inpc::fault_arg(pos);
  INPC_TRY(check_head(cam, pos, h, h_dtype, n, n_channels));
  if (n == 0) return INPC_OK;
  if (!d_alpha || !d_color || !dh_out || !aligned(d_color, 16)) return fail(INPC_ERR_INVALID_ARG, "bad pointer");
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  const ShConsts k = make_consts(*cam);
  const bool vec = n_channels % 4 == 0 && aligned(dh_out, 16);
  const auto run = [&](auto kernel, auto* rows) {
    kernel<<<grid_for_warps(n), kHeadThreads, 0, s>>>(k, pos, rows, n, n_channels, d_alpha, d_color, dh_out);
  };
  const float* hf = static_cast<const float*>(h);
  const __nv_bfloat16* hb = static_cast<const __nv_bfloat16*>(h);
  if (h_dtype == INPC_F32) vec ? run(k_sh_head_bwd<float, true>, hf) : run(k_sh_head_bwd<float, false>, hf);
  else vec ? run(k_sh_head_bwd<__nv_bfloat16, true>, hb) : run(k_sh_head_bwd<__nv_bfloat16, false>, hb);
  return check_launch("k_sh_head_bwd");
}
