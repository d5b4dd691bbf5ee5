// Per-tile implicit half instantiated for MH = 33.
#include "stage_kernels.cuh"

CH_STAGE_POST(33)
