// Per-tile implicit half instantiated for MH = 97.
#include "stage_kernels.cuh"

CH_STAGE_POST(97)
