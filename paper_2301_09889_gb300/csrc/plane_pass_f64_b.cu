// Three-pass nonlinear term instantiated for padded lengths 144, 192, double.
#include "plane_pass.cuh"

CH_PASS_INSTANTIATE(double, 144)
CH_PASS_INSTANTIATE(double, 192)
