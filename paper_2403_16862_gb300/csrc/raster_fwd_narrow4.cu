// raster_fwd_narrow4.cu -- rasterizer forward kernels: FP32, at most 4 lanes per pixel.
#include "raster_fwd.h"
#include "raster_impl.cuh"

namespace inpc {

inpc_status raster_fwd_narrow4(const RasterFwdCall& c) {
  RP P;
  INPC_TRY(make_rp(c.cam, c.opts, c.n, P, kMaxFwdPoints));
  P.together = c.together;
  const RasterWs ws = carve(c.workspace, P.n_pix, c.n);
  return dispatch(P.F, [&](auto Vc, auto Gc) -> inpc_status {
    constexpr int V = decltype(Vc)::value, GA = decltype(Gc)::value;
    if constexpr (GA <= 4)
      return launch_fwd<V, GA, float>(P, c.pos, c.opacity, static_cast<const float*>(c.feat), ws, static_cast<float*>(c.image),
                                   c.T_final, c.n_contrib, c.stream);
    return fail(INPC_ERR_UNSUPPORTED, "no raster_fwd_narrow4 kernel for n_channels = %d", P.F);
  });
}

}  // namespace inpc
