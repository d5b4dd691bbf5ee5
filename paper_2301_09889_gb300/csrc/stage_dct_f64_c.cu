// Register cosine transforms of a stage instantiated for orders 192, double.
#include "stage_dct.cuh"

CH_DCT_INSTANTIATE(double, 192)
