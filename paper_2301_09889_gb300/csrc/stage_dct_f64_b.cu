// Register cosine transforms of a stage instantiated for orders 96, 128, double.
#include "stage_dct.cuh"

CH_DCT_INSTANTIATE(double, 96)
CH_DCT_INSTANTIATE(double, 128)
