// Three-pass nonlinear term instantiated for padded lengths 144, 192, 288, 384, float.
#include "plane_pass.cuh"

CH_PASS_INSTANTIATE(float, 144)
CH_PASS_INSTANTIATE(float, 192)
CH_PASS_INSTANTIATE(float, 288)
CH_PASS_INSTANTIATE(float, 384)
