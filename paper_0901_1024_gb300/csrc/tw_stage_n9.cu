// Streamed-operator tensor-core stage kernel instantiation for order N=9.
#include "tw_stage.cuh"
DG_INSTANTIATE_TW_STAGE(9)
