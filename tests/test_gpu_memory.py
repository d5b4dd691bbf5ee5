"""Device memory of single-environment handles, where the tables of the tau
solves outweigh the fields.

Per mode and environment a handle holds V, G and their previous right-hand
sides (4 ny complex values) and at most 9 ny node values; per mode and row of
one parity at most 38 table values under a free-slip top (3 x 2 stages and
parities of e, h, b, Q, 2 of the Poisson factors', 6 of the homogeneous v) and
92 with both walls (the folded rows beside them).  The rest: the Chebyshev
tables, some hundred values per mode, and small arrays.
"""

import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,nz", [(16, 65, 16), (8, 65, 8), (24, 50, 48), (32, 65, 32), (36, 65, 36), (48, 65, 48)])
@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("top_bc,rows", [(0, 92), (1, 38)])
def test_single_handles_stay_small(native_gpu, nx, ny, nz, precision, top_bc, rows):
    native = native_gpu
    env = native.env_create(native.params(nx=nx, ny=ny, nz=nz, lx=2.67, lz=0.8, precision=precision, top_bc=top_bc))
    try:
        held = native.env_info(env).device_bytes
    finally:
        native.env_destroy(env)
    P, Mh = nx // 2 * nz, (ny - 1) // 2 + 1
    assert held <= 13 * ny * P * 16 + rows * Mh * P * 8 + ny * ny * 12 + 100 * P * 8 + (32 << 10), held
