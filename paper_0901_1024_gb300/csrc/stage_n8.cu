// Stage kernel instantiations for order N=8: register tiled, and tiles of shape 1.
#include "stage_kernel.cuh"
#include "stage_wide.cuh"
DG_INSTANTIATE_STAGE(8)
