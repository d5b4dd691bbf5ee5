"""The mean shear that the mixed-precision nonlinear term sees is the FP64
derivative of the mean flow, rounded once.

U has derivative coefficients b_m = (-1)^m (1 + k d), k steps below the top of
each parity's running sum b_m = b_{m+2} + 2 (m+1) a_{m+1}, with d = 4e-8 less
than half an ulp of 1 in FP32: a running sum in FP32 stays at 1 and loses up to
N d / 2 of every coefficient, a sum in FP64 rounds each by 6e-8 at most.  DU is
concentrated at the lower wall, so blowing and suction there (one spanwise mode,
kx = 0) carries it into omega_y, whose right-hand side is -i kz v DU.

Bar.  The FP32 path from DU to omega_y is four padded Fourier and two Chebyshev
line transforms and one product, some 40 roundings of 2.5e-8 rms each: 1.6e-7,
held to 5e-7.  An FP32 running sum is off by N d / (2 sqrt 3), 2.2e-6 at 193
nodes.
"""

import numpy as np
import pytest

from gpu_util import rel_l2

pytestmark = pytest.mark.gpu

NX, NZ = 8, 12


def _mean(ny):
    N, d = ny - 1, 4e-8
    a = np.zeros(ny)
    n = np.arange(3, ny)
    a[3:] = np.where(n % 2 == 1, 1.0, -1.0) * np.where(n >= N - 1, 1.0, d) / (2 * n)
    # no slip at both walls and the flow rate int U dy = 2
    a[1] = -a[3::2].sum()
    even = np.arange(4, ny, 2)
    w = 2.0 / (1.0 - even.astype(float) ** 2)
    a[0], a[2] = np.linalg.solve([[1.0, 1.0], [2.0, -2.0 / 3.0]], [-a[even].sum(), 2.0 - w @ a[even]])
    return a


# batch 1: the scans, batch 16 (768 modes): the per-thread solves of the implicit half
@pytest.mark.parametrize("ny", [193])
@pytest.mark.parametrize("batch", [1, 16])
def test_mean_shear_is_summed_in_fp64(native_gpu, ny, batch):
    native = native_gpu
    # viscous changes of U over a step stay far below d
    kw = dict(nx=NX, ny=ny, nz=NZ, lx=2 * np.pi, lz=2 * np.pi, re_tau=1e6, re_bulk=1e6, dt=1e-10)
    act = np.broadcast_to(0.5 * np.cos(2 * np.pi * np.arange(NZ) / NZ)[None, :, None], (batch, NZ, NX)).copy()
    envs = [native.env_create(native.params(**kw, batch=batch, precision=p)) for p in (0, 1)]
    try:
        st = native.unpack_state(native.env_get_state(envs[0], 0), NX, ny, NZ)
        for k in ("v", "g", "W", "vw"):
            st[k] = np.zeros_like(st[k])
        st["U"] = _mean(ny)
        for when in ("copies of the implicit half", "copies of a state from the host"):
            out = []
            for env in envs:
                for e in range(batch):
                    native.env_set_state(env, e, native.pack_state(st, NX, ny, NZ))
                obs, tau, rew = np.zeros((batch, 2, NZ, NX)), np.zeros(batch), np.zeros(batch)
                assert native.env_step(env, act, obs, tau, rew) == 0
                out.append([native.unpack_state(native.env_get_state(env, e), NX, ny, NZ) for e in (0, batch - 1)])
            for ref, got in zip(*out):
                # (the highest coefficients hold the wall values of omega_y)
                dg, dr = ((x["g"] - st["g"])[:ny - 4] for x in (got, ref))
                assert np.linalg.norm(dr) > 0
                assert rel_l2(dg, dr) < 5e-7, (when, rel_l2(dg, dr))
            # then: a state with wall velocity, its mean flow set anew
            st = dict(out[0][0], U=_mean(ny))
    finally:
        for env in envs:
            native.env_destroy(env)
