// Three-pass nonlinear term instantiated for padded lengths 12, 18, 24, 36, 48, 72, 96, double.
#include "plane_pass.cuh"

CH_PASS_INSTANTIATE(double, 12)
CH_PASS_INSTANTIATE(double, 18)
CH_PASS_INSTANTIATE(double, 24)
CH_PASS_INSTANTIATE(double, 36)
CH_PASS_INSTANTIATE(double, 48)
CH_PASS_INSTANTIATE(double, 72)
CH_PASS_INSTANTIATE(double, 96)
