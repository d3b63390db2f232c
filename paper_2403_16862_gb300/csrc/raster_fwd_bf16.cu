// raster_fwd_bf16.cu -- rasterizer forward kernels: BF16 features and image, whole warps.
#include "raster_fwd.h"
#include "raster_impl.cuh"

namespace inpc {

inpc_status raster_fwd_bf16(const RasterFwdCall& c) {
  RP P;
  INPC_TRY(make_rp(c.cam, c.opts, c.n, P, kMaxFwdPoints));
  P.together = c.together;
  const RasterWs ws = carve(c.workspace, P.n_pix, c.n);
  return dispatch(P.F, [&](auto Vc, auto Gc) -> inpc_status {
    constexpr int V = decltype(Vc)::value, GA = decltype(Gc)::value;
    if constexpr (GA == 32)
      return launch_fwd<V, GA, __nv_bfloat16>(P, c.pos, c.opacity, static_cast<const __nv_bfloat16*>(c.feat), ws, static_cast<__nv_bfloat16*>(c.image),
                                   c.T_final, c.n_contrib, c.stream);
    return fail(INPC_ERR_UNSUPPORTED, "no raster_fwd_bf16 kernel for n_channels = %d", P.F);
  });
}

}  // namespace inpc
