"""Device memory of single-environment handles, where the tables of the tau
solves outweigh the fields, and what the server reserves for a class.

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


# (nx, ny, nz, slots, precision, control, top_bc): sensing planes that add up
# beyond the allowance for rounding; direct sums; both sizes of a mixed handle's
# node array
@pytest.mark.parametrize("nx,ny,nz,slots,precision,control,top_bc", [
    (128, 17, 128, 64, 1, 0, 0), (128, 17, 128, 64, 0, 1, 1), (64, 17, 64, 24, 1, 1, 0), (16, 50, 16, 8, 1, 0, 1),
    (16, 201, 16, 1, 0, 1, 0), (36, 9, 36, 16, 1, 0, 0), (32, 33, 32, 1, 1, 0, 0)])
def test_admission_covers_what_a_class_holds(native_gpu, nx, ny, nz, slots, precision, control, top_bc):
    native = native_gpu
    kw = dict(nx=nx, ny=ny, nz=nz, lx=2.67, lz=0.8, precision=precision, control=control, top_bc=top_bc, autotune=0)
    env = native.env_create(native.params(**kw, batch=slots))
    try:
        held = native.env_info(env).device_bytes
    finally:
        native.env_destroy(env)
    srv = native.srv_create(64 << 30, slots)
    try:
        native.srv_admit(srv, native.params(**kw), seed=1)
        used = native.srv_stats(srv).hbm_used
    finally:
        native.srv_destroy(srv)
    assert held <= used <= held + (8 << 20), (held, used)
