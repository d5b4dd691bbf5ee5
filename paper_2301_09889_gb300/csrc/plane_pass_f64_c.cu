// Three-pass nonlinear term instantiated for padded lengths 288, 384, double.
#include "plane_pass.cuh"

CH_PASS_INSTANTIATE(double, 288)
CH_PASS_INSTANTIATE(double, 384)
