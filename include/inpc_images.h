/* inpc_images.h -- accumulation of several feature images in one pass
 * (inference multisampling, Sec. 3.2), beside inpc_accumulate_image. */
#ifndef INPC_IMAGES_H
#define INPC_IMAGES_H

#include "inpc.h"

#define INPC_MAX_IMAGES 4

#ifdef __cplusplus
extern "C" {
#endif

/* acc[i] = (fresh ? 0 : acc[i]) + scale * images[0][i] + ... for i < n_elems,
 * the images in order, one rounding (FMA) each: the bits of a cleared acc and
 * one inpc_accumulate_image per image.  images: host array of n_images (1 to
 * INPC_MAX_IMAGES) device pointers; dtype INPC_F32 or INPC_BF16. */
inpc_status inpc_accumulate_images(const void* const* images, int32_t n_images, int32_t dtype, int64_t n_elems,
                                   float scale, int32_t fresh, float* acc, inpc_stream_t stream);

#ifdef __cplusplus
}
#endif

#endif
