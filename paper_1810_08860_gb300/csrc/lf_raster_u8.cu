// lf_raster_u8.cu - the raster kernels for 8-bit textures (lf_raster_impl.h).
#define LF_RASTER_FORMAT LF_TEX_U8
#include "lf_raster_impl.h"
