// lf_raster_fp8.cu - the raster kernels for FP8 E4M3 textures (lf_raster_impl.h).
#define LF_RASTER_FORMAT LF_TEX_FP8E4M3
#include "lf_raster_impl.h"
