// Slab passes (slab.cuh) with 32-point y transforms.
#include "slab.cuh"
#include "slab.h"

DDA_SLAB_DEFINE(32)
