"""Rounding of the FP32 part of mixed handles against all-FP64 handles."""

import numpy as np
import pytest

import seeded_inputs as si

pytestmark = pytest.mark.gpu


def _errors(native, ny, dt=0.005, batch=16, steps=5):
    """rms over the slots of the relative errors of v and omega_y after `steps`."""
    nx, nz = 16, 16
    kw = dict(nx=nx, ny=ny, nz=nz, lx=2.67, lz=0.8, re_tau=180.0, re_bulk=2800.0, dt=dt, batch=batch)
    acts = np.stack([si.wall_action(nx, nz, 40 + e, 0.05 * 180 / 2800) for e in range(batch)])
    states = []
    for precision in (0, 1):
        env = native.env_create(native.params(**kw, precision=precision))
        try:
            for e in range(batch):
                native.env_set_state(env, e, native.pack_state(si.perturbed_poiseuille(nx, ny, nz, 100 + e, 0.2, 99),
                                                               nx, ny, nz))
            obs, tau, rew = np.zeros((batch, 2, nz, nx)), np.zeros(batch), np.zeros(batch)
            for _ in range(steps):
                assert native.env_step(env, acts, obs, tau, rew) == 0
            states.append([native.unpack_state(native.env_get_state(env, e), nx, ny, nz) for e in range(batch)])
        finally:
            native.env_destroy(env)
    return {k: np.sqrt(np.mean([np.linalg.norm(b[k] - a[k]) ** 2 / np.linalg.norm(a[k]) ** 2
                                for a, b in zip(*states)])) for k in ("v", "g")}


def test_direct_sums_round_like_transforms(native_gpu):
    """Chebyshev sums of 148 nodes (no register transform) leave omega_y no
    further off than the transforms of 129 nodes: the sums start at the highest,
    smallest coefficients.  Sixteen flows each; a sum of 74 terms that starts at
    the largest rounds each at the size of the whole."""
    sums, transforms = (_errors(native_gpu, ny)["g"] for ny in (148, 129))
    assert sums < 1.3 * transforms, (sums, transforms)


def test_time_steps_round_alike(native_gpu):
    """The error of v does not depend on how dt gamma_k and dt zeta_k round to
    FP32.  Their values are exact to 1e-10 at the first time step and, in all,
    5.4e-8 of dt too small and too large at the others: a rounding that every mode
    and step share, of the size of the whole error.  The rms over sixteen flows
    (each within some 20 %) scatters by 7 % between nearly equal time steps: held
    to 25 %."""
    exact, low, high = (_errors(native_gpu, 65, dt)["v"] for dt in (0.00502076, 0.00497612, 0.00498135))
    assert max(low, high) < 1.25 * exact, (exact, low, high)
