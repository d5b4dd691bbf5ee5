// Per-tile implicit half instantiated for MH = 5, 9, 17.
#include "stage_kernels.cuh"

CH_STAGE_POST(5)
CH_STAGE_POST(9)
CH_STAGE_POST(17)
