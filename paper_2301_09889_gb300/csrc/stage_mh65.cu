// Per-tile implicit half instantiated for MH = 65.
#include "stage_kernels.cuh"

CH_STAGE_POST(65)
