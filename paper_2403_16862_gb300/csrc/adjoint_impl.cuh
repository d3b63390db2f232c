// adjoint_impl.cuh -- the adjoint of the grid query (the table gradient),
// shared by the stand-alone adjoint (hashgrid.cu) and the fused rasterizer
// backward (raster_bwd.cu).
#pragma once

#include <algorithm>

#include "hashgrid_impl.cuh"

namespace inpc {
namespace {

// Levels per half of the adjoint's warp pairs for a grid of n_levels levels
// (the even warp of a pair takes the coarse half, the odd warp the fine one).
inline int adjoint_half(int n_levels) { return n_levels <= 8 ? 4 : n_levels <= 16 ? 8 : 16; }

// Whether the gradient rows of levels l_first .. n_levels - 1 stay within
// the L2 budget, so that reductions into all of them at once hit L2.
inline bool grad_levels_fit_l2(const GridParams& P, int l_first) {
  long long rows = 0;
  for (int l = l_first; l < P.n_levels; ++l) rows += level_rows(P, l);
  return rows * 16 <= kQueryL2Budget;
}

// One lane of the grid adjoint: one level, one x vertex of the cell (bx, the
// parity of that vertex).  Two adjacent lanes share a level, so a pair's
// reductions (x and x + 1 with the same y, z: rows differing in their low
// bits) usually fall in one 128-byte line and cost one L1 wavefront.
//
// add() of a fine lane: its four corner contributions straight to L2.
// add() of a coarse lane keeps one float4 accumulator per y-z corner in shared
// memory (acc[s kStride]) and sends a corner's sum to memory only when the
// next point needs a different vertex in that slot.  The slot of vertex
// (X, Y, Z) is given by the parities of X, Y and Z: every cell has exactly
// one corner of each parity class, and a step of one cell along an axis
// keeps the four shared vertices in their slots, so neighbouring cells
// share accumulators as well.  flush() sends what is left.
template <int kStride>
struct AdjointLane {
  static constexpr uint32_t kFar = 1u << 30;  // no cell held yet
  float* gl;
  uint32_t my, mz, rmask;  // a row is x + y my + z mz (dense) or (x ^ y my ^ z mz) & rmask (hashed)
  uint32_t bx;
  int N;
  bool dense;
  uint32_t hx, hy, hz;  // the cell whose corners the accumulators hold
  float4* acc;

  __device__ __forceinline__ AdjointLane(const GridParams& P, int l, bool active, float* grad_table, uint32_t bx_,
                                         float4* acc_)
      : bx(bx_), hx(kFar), hy(kFar), hz(kFar), acc(acc_) {
    gl = active ? grad_table + 4 * P.offset[l] : nullptr;
    dense = active && P.dense[active ? l : 0];
    const uint32_t side = active ? P.side[l] : 1u;
    my = dense ? side : 2654435761u;
    mz = dense ? side * side : 805459861u;
    rmask = dense ? 0xffffffffu : P.hash_mask;
    N = active ? P.res[l] : 1;
  }

  __device__ __forceinline__ uint32_t row(uint32_t X, uint32_t yb, uint32_t zb) const {
    return dense ? X + yb + zb : ((X ^ yb ^ zb) & rmask);
  }

  __device__ __forceinline__ void add(bool coarse, float x, float y, float z, const float (&dc)[4], uint64_t keep) {
    uint32_t cx, cy, cz;
    float gx[2], gy[2], gz[2];
    cell_frac(x, N, cx, gx[0], gx[1]);
    cell_frac(y, N, cy, gy[0], gy[1]);
    cell_frac(z, N, cz, gz[0], gz[1]);
    // slot s holds the corner whose offsets are s's bits xor the cell's
    // parities; swapping the weight pairs of odd cells makes gy[sy] that
    // corner's weight.  Along x this lane owns the vertex of parity bx.
    const uint32_t px = cx & 1u, py = cy & 1u, pz = cz & 1u;
    const uint32_t qx = hx & 1u, qy = hy & 1u, qz = hz & 1u;
    const uint32_t X = cx + (bx ^ px);
    const float wx = (bx ^ px) ? gx[1] : gx[0];
    if (py) swap_f(gy[0], gy[1]);
    if (pz) swap_f(gz[0], gz[1]);
    if (coarse) {
      // does the slot keep its vertex?
      const uint32_t HX = hx + (bx ^ qx);
      const bool kx = X == HX;
      const bool ky[2] = {cy + py == hy + qy, cy + (py ^ 1u) == hy + (qy ^ 1u)};
      const bool kz[2] = {cz + pz == hz + qz, cz + (pz ^ 1u) == hz + (qz ^ 1u)};
      const bool held = hx != kFar;
      // the y and z terms of the held cell's rows of slots sy, sz
      const uint32_t hyb[2] = {(hy + qy) * my, (hy + (qy ^ 1u)) * my};
      const uint32_t hzb[2] = {(hz + qz) * mz, (hz + (qz ^ 1u)) * mz};
#pragma unroll
      for (int s = 0; s < 4; ++s) {
        const uint32_t sy = s & 1, sz = s >> 1;
        const float w = wx * gy[sy] * gz[sz];
        const float4 a = acc[s * kStride];
        const bool same = kx && ky[sy] && kz[sz];
        // same vertex: add to the sum; otherwise start a new sum (fma onto 0)
        acc[s * kStride] = make_float4(__fmaf_rn(w, dc[0], same ? a.x : 0.f), __fmaf_rn(w, dc[1], same ? a.y : 0.f),
                                       __fmaf_rn(w, dc[2], same ? a.z : 0.f), __fmaf_rn(w, dc[3], same ? a.w : 0.f));
        // the slot moves to another vertex: send the old vertex its sum
        if (!same && held) red_add_v4(gl + 4ull * row(HX, hyb[sy], hzb[sz]), a, keep);
      }
      hx = cx;
      hy = cy;
      hz = cz;
    } else {
      // the y and z terms of this cell's rows of slots sy, sz
      const uint32_t yb[2] = {(cy + py) * my, (cy + (py ^ 1u)) * my};
      const uint32_t zb[2] = {(cz + pz) * mz, (cz + (pz ^ 1u)) * mz};
#pragma unroll
      for (int s = 0; s < 4; ++s) {
        const uint32_t sy = s & 1, sz = s >> 1;
        const float w = wx * gy[sy] * gz[sz];
        red_add_v4(gl + 4ull * row(X, yb[sy], zb[sz]), make_float4(w * dc[0], w * dc[1], w * dc[2], w * dc[3]), keep);
      }
    }
  }

  // A coarse lane's remaining sums.
  __device__ __forceinline__ void flush(uint64_t keep) const {
    if (hx == kFar) return;
    const uint32_t qx = hx & 1u, qy = hy & 1u, qz = hz & 1u;
    const uint32_t HX = hx + (bx ^ qx);
    const uint32_t hyb[2] = {(hy + qy) * my, (hy + (qy ^ 1u)) * my};
    const uint32_t hzb[2] = {(hz + qz) * mz, (hz + (qz ^ 1u)) * mz};
#pragma unroll
    for (int s = 0; s < 4; ++s) red_add_v4(gl + 4ull * row(HX, hyb[s & 1], hzb[s >> 1]), acc[s * kStride], keep);
  }
};

// Corner contributions of levels l_first .. n_levels - 1, level group after
// level group (grid y, plan_level_groups), so that the rows receiving
// reductions at a time are one group's and stay in L2: tables whose fine
// levels do not fit would otherwise miss L2 and go to DRAM twice per
// reduction (a read before the add, a write-back later).  d holds dL/dh in
// rows of 4 floats: level l of point p at d[(l - l_first) level_stride +
// p point_stride].  Two lanes per point, one per x vertex of the cell, 16
// consecutive points per warp; the contributions are AdjointLane's own,
// (w_x w_y) w_z times the row.
__global__ void __launch_bounds__(256) k_grad_levels(GridParams Gp, LevelGroups LG, int l_first,
                                                     const float* __restrict__ pos, const float4* __restrict__ d,
                                                     long long point_stride, long long level_stride, long long n,
                                                     float* __restrict__ grad_table) {
  const int lb = LG.begin[blockIdx.y], le = LG.begin[blockIdx.y + 1];
  const uint64_t keep = l2_evict_last(), stream = l2_evict_first();
  const uint32_t lane = threadIdx.x & 31u;
  const uint32_t bx = lane & 1u;
  // n < 2^31 (checked by the callers): point indices fit in 32 bits
  const uint32_t n_groups = (uint32_t)((n + 15) >> 4);
  const uint32_t n_warps = (gridDim.x * blockDim.x) >> 5;
  for (uint32_t g = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; g < n_groups; g += n_warps) {
    const uint32_t p = g * 16u + (lane >> 1);
    if (p >= (uint32_t)n) continue;  // nothing below is warp-collective
    const float* xyz = pos + 3ull * p;
    const float x = __ldg(xyz), y = __ldg(xyz + 1), z = __ldg(xyz + 2);
    for (int l = lb; l < le; ++l) {
      const uint4 r = ld_hint_u4(d + (l - l_first) * level_stride + p * point_stride, stream);
      const float4 v = make_float4(__uint_as_float(r.x), __uint_as_float(r.y), __uint_as_float(r.z),
                                   __uint_as_float(r.w));
      if (v.x == 0.f && v.y == 0.f && v.z == 0.f && v.w == 0.f) continue;
      uint32_t cx, cy, cz;
      float gx[2], gy[2], gz[2];
      const int N = Gp.res[l];
      cell_frac(x, N, cx, gx[0], gx[1]);
      cell_frac(y, N, cy, gy[0], gy[1]);
      cell_frac(z, N, cz, gz[0], gz[1]);
      float* gl = grad_table + 4 * Gp.offset[l];
      const float wx = gx[bx];
#pragma unroll
      for (int yz = 0; yz < 4; ++yz) {
        const int by = yz & 1, bz = yz >> 1;
        const float w = wx * gy[by] * gz[bz];
        const uint32_t row = vertex_row(Gp, l, cx + bx, cy + by, cz + bz);
        red_add_v4(gl + 4ull * row, make_float4(w * v.x, w * v.y, w * v.z, w * v.w), keep);
      }
    }
  }
}

inline inpc_status launch_grad_levels(const GridParams& Gp, int l_first, const float* pos, const float4* d,
                                      long long point_stride, long long level_stride, long long n, float* grad_table,
                                      cudaStream_t s) {
  const LevelGroups LG = plan_level_groups(Gp, 16, l_first);
  const long long cap = (long long)device_sm_count() * 16;
  const dim3 grid((unsigned)std::max<long long>(1, std::min<long long>((long long)ceil_div(2 * n, 256), cap)),
                  (unsigned)LG.n);
  INPC_TIMED("k_grad_levels", s,
             k_grad_levels<<<grid, 256, 0, s>>>(Gp, LG, l_first, pos, d, point_stride, level_stride, n, grad_table));
  return check_launch("k_grad_levels");
}

}  // namespace
}  // namespace inpc
