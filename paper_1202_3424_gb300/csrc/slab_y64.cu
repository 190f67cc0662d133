// Slab passes (slab.cuh) with 64-point y transforms.
#include "slab.cuh"
#include "slab.h"

DDA_SLAB_DEFINE(64)
