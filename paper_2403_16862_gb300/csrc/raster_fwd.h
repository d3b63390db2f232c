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
};

inpc_status raster_fwd_narrow4(const RasterFwdCall& c);   // FP32, at most 4 lanes per pixel
inpc_status raster_fwd_narrow16(const RasterFwdCall& c);  // FP32, 8 or 16 lanes
inpc_status raster_fwd_wide(const RasterFwdCall& c);      // FP32, whole warps
inpc_status raster_fwd_bf16(const RasterFwdCall& c);      // BF16, whole warps

}  // namespace inpc
