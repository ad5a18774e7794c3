// lf_raster_f32.cu - the raster kernels for FP32 textures (lf_raster_impl.h).
#define LF_RASTER_FORMAT LF_TEX_F32
#include "lf_raster_impl.h"
