// raster_fwd.h -- the rasterizer forward's kernels by lane group and feature
// type, each set in a translation unit of its own (they compile in parallel).
#pragma once

#include "common.cuh"

namespace inpc {

struct RasterFwdCall {  // checked arguments of inpc_rasterize_fwd
  const inpc_camera* cam;
  const inpc_raster_opts* opts;
  const float* pos;
  const float* opacity;
  const void* feat;
  int64_t n;
  void* image;
  float* T_final;
  int32_t* n_contrib;
  void* workspace;
  cudaStream_t stream;
  bool together;  // the blending kernels may overlap
};

inpc_status raster_fwd_narrow4(const RasterFwdCall& c);   // FP32, at most 4 lanes per pixel
inpc_status raster_fwd_narrow16(const RasterFwdCall& c);  // FP32, 8 or 16 lanes
inpc_status raster_fwd_wide(const RasterFwdCall& c);      // FP32, whole warps
inpc_status raster_fwd_bf16(const RasterFwdCall& c);      // BF16, whole warps

// inpc_rasterize_fwd and inpc_rasterize_bwd_hashgrid with a choice of whether
// the blending kernels of the pass may overlap (launch_group).
inpc_status rasterize_fwd(const inpc_camera* cam, const inpc_raster_opts* opts, const float* pos, const float* opacity,
                          const void* feat, int64_t n, void* image, float* T_final, int32_t* n_contrib, void* workspace,
                          size_t workspace_bytes, inpc_stream_t stream, bool together);
inpc_status rasterize_bwd_hashgrid(const inpc_camera* cam, const inpc_raster_opts* opts, const inpc_hashgrid_desc* grid,
                                   const float* pos, const void* feat, int64_t n, const float* T_final,
                                   const int32_t* n_contrib, const float* d_image, float* grad_table, float* d_feat,
                                   void* workspace, size_t workspace_bytes, inpc_stream_t stream, bool together);

}  // namespace inpc
