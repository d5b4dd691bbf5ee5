"""ch_nonlinear (FP64) in the forms its sizes choose: handles of both
precisions, clusters for small planes and passes above, the passes of a mixed
handle in one part and in two.  Bar: four line transforms of at most 192 points
and the products, a few log2(192) roundings of 1.1e-16 each, held to 1e-13.
"""

import numpy as np
import pytest

import seeded_inputs as si
from gpu_util import oracle_params, rel_l2
from oracle import channel

pytestmark = pytest.mark.gpu

# (nx, ny, nz, batch): clusters of one to four CTAs and their neighbours in
# passes; 64x33x64 x 2 and 64x34x64 x 2 take two parts in mixed handles, of 17
# and 16 and of 17 and 17 nodes; 36 has no passes
SIZES = [(8, 9, 8, 1), (8, 101, 8, 3), (8, 103, 8, 3), (8, 9, 16, 1), (8, 75, 16, 1), (8, 77, 16, 1), (8, 9, 24, 1),
         (24, 9, 8, 1), (12, 9, 8, 1), (8, 9, 64, 1), (32, 9, 32, 1), (24, 17, 48, 3), (64, 33, 64, 2), (64, 34, 64, 2),
         (128, 9, 128, 2), (36, 9, 24, 1), (16, 9, 16, 2)]


@pytest.mark.parametrize("nx,ny,nz,batch", SIZES)
@pytest.mark.parametrize("precision", [0, 1])
def test_nonlinear_forms(native_gpu, nx, ny, nz, batch, precision):
    import torch
    native = native_gpu
    kw = dict(nx=nx, ny=ny, nz=nz, lx=2 * np.pi, lz=np.pi, re_tau=180.0, re_bulk=2800.0, dt=0.002)
    ops = channel.Operators(oracle_params(**kw))
    rng = np.random.default_rng(nx * 1000 + nz + ny)
    q = np.fft.rfft2(rng.standard_normal((batch, 6, ny, nz, nx)))[..., :nx // 2] / (nx * nz)
    q[:, :, :, nz // 2] = 0.0
    d_q = torch.from_numpy(np.ascontiguousarray(q).view(np.float64)).cuda()
    d_h = torch.full((batch, 3, ny, nz, nx // 2, 2), float("nan"), dtype=torch.float64, device="cuda")
    fields = si.perturbed_poiseuille(nx, ny, nz, 3, 0.2, 4)
    act = np.stack([si.wall_action(nx, nz, 7 + e, 0.05 * 180 / 2800) for e in range(batch)])
    steps = []
    env = native.env_create(native.params(**kw, batch=batch, precision=precision))
    try:
        for call in (False, True):
            for e in range(batch):
                native.env_set_state(env, e, native.pack_state(fields, nx, ny, nz))
            if call:
                native.ch_nonlinear(env, d_q.data_ptr(), d_h.data_ptr())
            obs, tau, rew = np.zeros((batch, 2, nz, nx)), np.zeros(batch), np.zeros(batch)
            assert native.env_step(env, act, obs, tau, rew) == 0
            steps.append((obs.copy(), tau.copy(), native.env_get_state(env, batch - 1)))
        torch.cuda.synchronize()
    finally:
        native.env_destroy(env)
    h = d_h.cpu().numpy().view(np.complex128)[..., 0]
    for b in range(batch):
        ref = channel.nonlinear_nodes(dict(zip(channel.NODE_FIELDS, q[b])), ops)
        for c, name in enumerate("xyz"):
            assert rel_l2(h[b, c], ref[name]) < 1e-13, (b, name)
    assert all(np.array_equal(x, y) for x, y in zip(*steps))  # the call leaves nothing behind in the handle


def test_nonlinear_of_mixed_256_planes_stays_unsupported(native_gpu):
    import torch
    native = native_gpu
    env = native.env_create(native.params(nx=256, ny=9, nz=256, lx=6.28, lz=3.14, precision=1))
    try:
        d = torch.zeros(6, 9, 256, 128, 2, dtype=torch.float64, device="cuda")
        with pytest.raises(native.ChannelError) as exc:
            native.ch_nonlinear(env, d.data_ptr(), d.data_ptr())
        assert exc.value.code == native.CH_ERR_UNSUPPORTED
    finally:
        native.env_destroy(env)


@pytest.mark.parametrize("precision", [0, 1])
def test_single_16x16_planes_report_their_cluster(native_gpu, precision):
    """Planes of 16 x 16 modes run on two-CTA clusters until a batch has four
    planes per SM, then two to a CTA."""
    native = native_gpu
    for batch, cluster in ((1, 2), (80, 1)):
        env = native.env_create(native.params(nx=16, ny=65, nz=16, batch=batch, precision=precision, autotune=0))
        try:
            info = native.env_info(env)
        finally:
            native.env_destroy(env)
        assert info.plane_cluster == cluster and info.plane_team == (1 if batch == 80 else 0)
