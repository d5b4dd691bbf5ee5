"""The forms that the sizes of a handle choose, at the edges of their ranges,
against the FP64 oracle: line lengths of the three-pass nonlinear term, register
cosine transforms and direct sums, the few-mode explicit half, the scans and
the per-thread solves, the action and observation transforms by lines, and the
columns of the stand-alone tau problems.

Bars.  Nonlinear term: four line transforms of at most 384 points and the
products between them, each within a few log2(384) roundings of 1.1e-16:
below 1e-14, held to 1e-13.  Steps: the relative L2 bars of the other step
tests, 1e-11 (all FP64) and 1e-4 (mixed), 1e-9 for the FP64 wall shear.  Tau
problems: 1e-12 per column, as in the unit test of the same entry point.
"""

import numpy as np
import pytest

import seeded_inputs as si
from gpu_util import oracle_params, rel_l2, run_batch_pair
from oracle import channel

pytestmark = pytest.mark.gpu

# padded lengths 12, 18, 24, 36, 48, 72, 96, 144, 192, 288, 384 in x and in z,
# and 54 and 6 (no passes); nine nodes, so that the last CTAs of the passes are partial
LINES = [(8, 12), (12, 8), (16, 24), (24, 16), (32, 48), (48, 32), (64, 96), (96, 64), (128, 192), (192, 128),
         (256, 8), (8, 256), (16, 16), (36, 8), (8, 36), (4, 12)]


@pytest.mark.parametrize("nx,nz", LINES)
@pytest.mark.parametrize("batch", [1, 3])
def test_nonlinear_lines(native_gpu, nx, nz, batch):
    import torch
    native, ny = native_gpu, 9
    ops = channel.Operators(oracle_params(nx=nx, ny=ny, nz=nz, lx=2 * np.pi, lz=np.pi))
    rng = np.random.default_rng(nx * 1000 + nz)
    q = np.fft.rfft2(rng.standard_normal((batch, 6, ny, nz, nx)))[..., :nx // 2] / (nx * nz)
    q[:, :, :, nz // 2] = 0.0
    ref = [channel.nonlinear_nodes(dict(zip(channel.NODE_FIELDS, q[b])), ops) for b in range(batch)]
    env = native.env_create(native.params(nx=nx, ny=ny, nz=nz, lx=2 * np.pi, lz=np.pi, batch=batch))
    try:
        d_q = torch.from_numpy(np.ascontiguousarray(q).view(np.float64)).cuda()
        d_h = torch.full((batch, 3, ny, nz, nx // 2, 2), float("nan"), dtype=torch.float64, device="cuda")
        native.ch_nonlinear(env, d_q.data_ptr(), d_h.data_ptr())
        torch.cuda.synchronize()
        h = d_h.cpu().numpy().view(np.complex128)[..., 0]
        assert torch.equal(d_q.cpu(), torch.from_numpy(np.ascontiguousarray(q).view(np.float64)))
    finally:
        native.env_destroy(env)
    for b in range(batch):
        for c, name in enumerate("xyz"):
            assert rel_l2(h[b, c], ref[b][name]) < 1e-13, (b, name)


# (ny, batch, top_bc) of an 8 x 12 plane (48 modes: three tiles of sixteen).
# Orders 16, 24, 32, 48, 64, 96, 128, 192 have register transforms, the others
# direct sums; batch 1: few-mode explicit half (FP64) and scans; 9: transforms or
# direct sums and scans; 16: 768 modes, the per-thread solves
STEPS = [(9, 1, 0), (10, 1, 0), (25, 1, 0), (50, 1, 0), (129, 1, 0), (130, 1, 0),
         (9, 9, 0), (17, 9, 0), (49, 9, 0), (50, 9, 0), (66, 9, 0),
         (9, 16, 0), (10, 16, 0), (17, 16, 0), (25, 16, 0), (33, 16, 0), (49, 16, 0), (51, 16, 0), (65, 16, 0),
         (97, 16, 0), (129, 16, 0), (148, 16, 0), (193, 16, 0), (201, 16, 0),
         (9, 1, 1), (34, 1, 1), (9, 16, 1), (17, 16, 1), (50, 16, 1), (64, 16, 1)]


@pytest.mark.parametrize("ny,batch,top_bc", STEPS)
@pytest.mark.parametrize("precision", [0, 1])
def test_step_orders_and_forms(native_gpu, ny, batch, top_bc, precision):
    kw = dict(nx=8, ny=ny, nz=12, lx=2.67, lz=0.8, re_tau=180.0, re_bulk=2800.0, dt=0.002, top_bc=top_bc,
              precision=precision)
    slots = sorted({0, batch - 1})
    info, res = run_batch_pair(native_gpu, kw, batch, slots, 1)
    assert info.post_batched == (1 if batch == 16 else 0)
    _check(res, kw)


# 24 x 32 planes of eleven environments: 8448 >= 8192 points, both transforms
# by lines; ten stay below; 36 has no lines
@pytest.mark.parametrize("nx,nz,batch", [(24, 32, 11), (24, 32, 10), (36, 24, 10)])
@pytest.mark.parametrize("precision", [0, 1])
def test_action_and_observation_lines(native_gpu, nx, nz, batch, precision):
    kw = dict(nx=nx, ny=17, nz=nz, lx=2.67, lz=0.8, re_tau=180.0, re_bulk=2800.0, dt=0.002, precision=precision)
    _, res = run_batch_pair(native_gpu, kw, batch, [0, batch - 1], 1)
    _check(res, kw)


def _check(res, kw):
    tol, tau_tol = ((1e-11, 1e-9), (1e-4, 1e-4))[kw["precision"]]
    for e, (lib, ora, ls, os_) in res.items():
        for k in ("v", "g", "U"):
            assert rel_l2(ls[k], os_[k]) <= tol, (e, k, rel_l2(ls[k], os_[k]))
        assert np.linalg.norm(ls["W"] - os_["W"]) <= tol * np.linalg.norm(os_["U"]), e
        assert rel_l2(lib[0][0], ora[0][0]) <= tol, (e, rel_l2(lib[0][0], ora[0][0]))
        assert abs(lib[0][1] - ora[0][1]) <= tau_tol * abs(ora[0][1]), e


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("batch", [2, 16])
@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
def test_non_finite_state_stays_in_its_slot(native_gpu, precision, batch, bad):
    """A non-finite coefficient of v reaches that environment's wall shear and
    no other environment."""
    native = native_gpu
    nx, ny, nz = 8, 33, 12
    kw = dict(nx=nx, ny=ny, nz=nz, lx=2.67, lz=0.8, re_tau=180.0, re_bulk=2800.0, dt=0.002, precision=precision)
    env = native.env_create(native.params(**kw, batch=batch))
    try:
        for e in range(batch):
            f = si.perturbed_poiseuille(nx, ny, nz, 40 + e, 0.1, 4)
            if e == 1:
                f["v"][3, 1, 1] = bad
            native.env_set_state(env, e, native.pack_state(f, nx, ny, nz))
        obs, tau, rew = np.zeros((batch, 2, nz, nx)), np.zeros(batch), np.zeros(batch)
        assert native.env_step(env, np.zeros((batch, nz, nx)), obs, tau, rew) == native.CH_ERR_DIVERGED
        finite = np.isfinite(tau) & np.isfinite(obs).all(axis=(1, 2, 3))
    finally:
        native.env_destroy(env)
    assert not finite[1] and finite[np.arange(batch) != 1].all()


# shortest and longest columns, even and odd orders, one problem and a partial block
@pytest.mark.parametrize("ny", [5, 6, 50, 130, 201])
@pytest.mark.parametrize("m", [1, 37])
def test_tau_columns(native_gpu, ny, m):
    import torch
    native = native_gpu
    ops = channel.Operators(oracle_params(nx=4, ny=ny, nz=4, lx=6.28, lz=3.14))
    rng = np.random.default_rng(ny)
    z = lambda *s: rng.standard_normal(s) + 1j * rng.standard_normal(s)
    lam = rng.uniform(0, 5e4, m)
    r, top, bot = z(m, ny) * 0.9 ** np.arange(ny), z(m), z(m)
    ref = channel.tau_dirichlet(ops, lam, r, top, bot)
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    d = [t(lam), t(r.view(np.float64)), t(top.view(np.float64)), t(bot.view(np.float64))]
    d_f = torch.zeros(m, ny, 2, dtype=torch.float64, device="cuda")
    native.ch_tau_helmholtz(ny, m, *(a.data_ptr() for a in d), d_f.data_ptr(), torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    f = d_f.cpu().numpy().view(np.complex128).reshape(m, ny)
    for i in range(m):
        assert rel_l2(f[i], ref[i]) < 1e-12, (i, lam[i])
