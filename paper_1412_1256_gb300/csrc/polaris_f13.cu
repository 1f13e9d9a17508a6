#include "polaris_fused.cuh"

POLARIS_INSTANTIATE_FUSED(13)
