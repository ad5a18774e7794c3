// lf_raster_bf16.cu - the raster kernels for BF16 textures (lf_raster_impl.h).
#define LF_RASTER_FORMAT LF_TEX_BF16
#include "lf_raster_impl.h"
