// Register cosine transforms of a stage instantiated for orders 16, 24, 32, 48, 64, 96, float.
#include "stage_dct.cuh"

CH_DCT_INSTANTIATE(float, 16)
CH_DCT_INSTANTIATE(float, 24)
CH_DCT_INSTANTIATE(float, 32)
CH_DCT_INSTANTIATE(float, 48)
CH_DCT_INSTANTIATE(float, 64)
CH_DCT_INSTANTIATE(float, 96)
