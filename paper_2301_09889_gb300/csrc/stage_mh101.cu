// Per-tile implicit half instantiated for MH = 101.
#include "stage_kernels.cuh"

CH_STAGE_POST(101)
