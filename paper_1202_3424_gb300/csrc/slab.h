// The slab kernels' launchers, one translation unit per Ly (slab_y*.cu): the
// launcher for a z length, or null where the pass is not built.
#pragma once

#include "internal.h"

namespace dda {

#define DDA_SLAB_FN(LY)                                                                                             \
    cudaError_t (*slab_fn_##LY(int Lz))(const Geom&, int, float2*, const float4*, const Twiddles<float>&, const int*, \
                                        cudaStream_t)
DDA_SLAB_FN(16);
DDA_SLAB_FN(32);
DDA_SLAB_FN(48);
DDA_SLAB_FN(64);
DDA_SLAB_FN(96);
DDA_SLAB_FN(128);

}  // namespace dda
