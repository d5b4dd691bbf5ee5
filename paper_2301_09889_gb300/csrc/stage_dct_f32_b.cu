// Register cosine transforms of a stage instantiated for orders 128, 192, float.
#include "stage_dct.cuh"

CH_DCT_INSTANTIATE(float, 128)
CH_DCT_INSTANTIATE(float, 192)
