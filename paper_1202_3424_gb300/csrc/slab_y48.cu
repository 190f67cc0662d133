// Slab passes (slab.cuh) with 48-point y transforms.
#include "slab.cuh"
#include "slab.h"

DDA_SLAB_DEFINE(48)
