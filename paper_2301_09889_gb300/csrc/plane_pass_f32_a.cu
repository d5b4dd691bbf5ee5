// Three-pass nonlinear term instantiated for padded lengths 12, 18, 24, 36, 48, 72, 96, float.
#include "plane_pass.cuh"

CH_PASS_INSTANTIATE(float, 12)
CH_PASS_INSTANTIATE(float, 18)
CH_PASS_INSTANTIATE(float, 24)
CH_PASS_INSTANTIATE(float, 36)
CH_PASS_INSTANTIATE(float, 48)
CH_PASS_INSTANTIATE(float, 72)
CH_PASS_INSTANTIATE(float, 96)
