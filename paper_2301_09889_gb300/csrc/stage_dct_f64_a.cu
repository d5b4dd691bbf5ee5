// Register cosine transforms of a stage instantiated for orders 16, 24, 32, 48, 64, double.
#include "stage_dct.cuh"

CH_DCT_INSTANTIATE(double, 16)
CH_DCT_INSTANTIATE(double, 24)
CH_DCT_INSTANTIATE(double, 32)
CH_DCT_INSTANTIATE(double, 48)
CH_DCT_INSTANTIATE(double, 64)
