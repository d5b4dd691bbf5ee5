// Per-tile implicit half instantiated for MH = 49.
#include "stage_kernels.cuh"

CH_STAGE_POST(49)
