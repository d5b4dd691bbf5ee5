"""The work that a user of the channel-flow environment has it do.

A *step* case advances one handle through ``env_step`` (host arrays, as an
actor process calls it), ``env_step_device`` (device tensors, as a learner on
the same GPU calls it) or ``env_set_state`` / ``env_step`` /
``env_get_state`` (an episode's interval from a stored initial condition to a
stored checkpoint).  A *served* case puts one request of every admitted
environment through the batching server.  *nonlinear* and *tau* cases are the
two stand-alone stages, ``ch_nonlinear`` and ``ch_tau_helmholtz``.

Mixed-precision results are taken in FP32, as the agents' networks take them;
all-FP64 results stay in FP64.

``exact`` restates the discretisation densely in 64 bits with torch: Fourier
transforms by ``torch.fft``, wall-normal operators as dense Chebyshev
matrices, and one LU of the coupled (phi, v) system per mode and stage.
"""

from __future__ import annotations

import math

import numpy as np
import torch

DEV = "cuda" if torch.cuda.is_available() else "cpu"

# Low-storage RK3 / Crank-Nicolson coefficients and stage end times.
GAMMA = (8 / 15, 5 / 12, 3 / 4)
ZETA = (0.0, -17 / 60, -5 / 12)
C_END = (8 / 15, 2 / 3, 1.0)

WINDOW, HIDDEN = 3, 64  # the shared policy: 3 x 3 window of u and v, two hidden layers of 64


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------

def _step(name, nx, ny, nz, batch=1, precision=0, top_bc=0, control=0, steps=1, io="host"):
    return {"name": name, "kind": "step", "nx": nx, "ny": ny, "nz": nz, "batch": batch, "precision": precision,
            "top_bc": top_bc, "control": control, "steps": steps, "io": io}


def listed():
    return [
        # one minimal channel in FP64, an action from the host every step: the
        # smallest call, an interactive actor or a debugging run
        _step("minimal_fp64", 16, 65, 16),
        # the training batch: 256 minimal channels in mixed precision, actions
        # and observations on the device
        _step("minimal_batch256_mixed", 16, 65, 16, batch=256, precision=1, io="device"),
        # the paper's open channel with the learnt policy evaluated on the
        # device: deployment of a trained agent on a batch of channels
        _step("open_batch128_policy_mixed", 16, 65, 16, batch=128, precision=1, top_bc=1, control=2, io="device"),
        # the drag-reduction validation of the open channel: 16 FP64 channels
        # under opposition control, over one actuation interval (dt+ = 0.6: ten
        # steps) from stored states to checkpoints
        _step("open_batch16_interval_fp64", 16, 65, 16, batch=16, top_bc=1, control=1, steps=10, io="checkpoint"),
        # mixed-size serving: one request from each of 44 environments
        {"name": "served_mixed_sizes", "kind": "served", "minimal": 24, "mid": 12, "larger": 8},
        # the larger channel under opposition control, the same interval
        _step("larger_fp64_interval", 64, 65, 64, control=1, steps=10, io="checkpoint"),
        # the same channel as a production run: two branches in one handle, mixed precision
        _step("larger_batch2_interval_mixed", 64, 65, 64, batch=2, precision=1, control=1, steps=10, io="checkpoint"),
        # a ragged grid (sizes that no kernel is specialised for, odd N)
        _step("ragged_batch8_mixed", 24, 50, 48, batch=8, precision=1),
        # Re_tau 395, one channel, mixed precision
        _step("re395_mixed", 128, 129, 128, precision=1),
        # Re_tau 550, the largest grid in use
        _step("re550_mixed", 256, 193, 256, precision=1, io="device"),
        # the dealiased nonlinear term alone, FP64, four channels of a ragged grid
        {"name": "nonlinear_ragged_fp64", "kind": "nonlinear", "nx": 24, "ny": 49, "nz": 32, "batch": 4},
        # stand-alone tau problems: both unknowns of the modes of a 64 x 64 channel
        {"name": "tau_ny65", "kind": "tau", "ny": 65, "m": 4031},
    ]


def draw(rng):
    u = rng.random()
    if u > 0.93:
        return {"kind": "served", "minimal": rng.randint(2, 24), "mid": rng.randint(1, 12), "larger": rng.randint(1, 8)}
    sizes = (8, 12, 16, 24, 32, 48, 64, 96, 128)
    if u < 0.15:
        ny = int(round(math.exp(rng.uniform(math.log(25), math.log(193)))))
        return {"kind": "tau", "ny": ny, "m": int(round(math.exp(rng.uniform(math.log(200), math.log(20000)))))}
    ny = rng.choice((33, 65, 97, 129)) if rng.random() < 0.35 else int(round(math.exp(rng.uniform(math.log(25), math.log(161)))))
    nx, nz = rng.choice(sizes), rng.choice(sizes)
    if u < 0.3:
        most = max(1, 2_000_000 // (nx * ny * nz))
        return {"kind": "nonlinear", "nx": nx, "ny": ny, "nz": nz, "batch": int(math.exp(rng.uniform(0, math.log(min(64, most)))))}
    precision = rng.choice((0, 1, 1))
    top_bc = rng.choice((0, 0, 1)) if ny <= 65 else 0
    steps = rng.choice((1, 1, 1, 3, 10))
    most = max(1, 4_000_000 // (nx * ny * nz * steps * (1 if precision else 4)))
    c = _step("", nx, ny, nz, int(math.exp(rng.uniform(0, math.log(min(300, most))))), precision, top_bc,
              rng.choice((0, 1, 2)), steps, rng.choice(("host", "device", "checkpoint")))
    del c["name"]
    return c


def _physics(c):
    """Box, Reynolds numbers and time step of a grid (the channels in use)."""
    n = c["nx"] * c["nz"]
    if n >= 256 * 256:
        re_tau, re_bulk, dt = 550.0, 10030.0, 0.002
    elif n >= 128 * 128:
        re_tau, re_bulk, dt = 395.0, 6875.0, 0.0025
    else:
        re_tau, re_bulk, dt = 180.0, 2800.0, 0.005
    return {"lx": min(2 * math.pi, 2.67 * c["nx"] / 16), "lz": min(math.pi, 0.8 * c["nz"] / 16), "re_tau": re_tau,
            "re_bulk": re_bulk, "dt": dt}


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _rng(seed, salt):
    g = torch.Generator()
    g.manual_seed(1_000_003 * (int(seed) + 1) + salt)
    return g


def _cos_table(N):
    """cos(pi j n / N), arguments reduced exactly."""
    i = torch.arange(N + 1, dtype=torch.int64, device=DEV)
    return torch.cos(math.pi * ((i[:, None] * i[None, :]) % (2 * N)).double() / N)


def _analysis(N):
    """Node values -> Chebyshev coefficients."""
    w = torch.ones(N + 1, dtype=torch.float64, device=DEV)
    w[0] = w[-1] = 0.5
    return 2.0 / N * w[:, None] * _cos_table(N) * w[None, :]


def _flows(c, seed, salt=0):
    """Developed-looking flows: plug-like mean, fluctuations in every kept mode
    with decaying spectra in all directions, all wall conditions met."""
    nx, ny, nz, B, top = c["nx"], c["ny"], c["nz"], c["batch"], c["top_bc"]
    nxh, N = nx // 2, ny - 1
    gen = _rng(seed, salt)
    K = max(1, min(12, (N - 7) // 2))  # polynomial content above the wall shapes
    ck = torch.randn(2, B, nz, nxh, K, 2, generator=gen, dtype=torch.float64).to(DEV)
    y = _cos_table(N)[:, 1]
    m = torch.arange(nz, device=DEV)
    m = torch.where(m < nz // 2, m, m - nz).double()
    i = torch.arange(nxh, device=DEV).double()
    amp = (1.0 + i[None, :] ** 2 + m[:, None] ** 2) ** -0.9
    amp[nz // 2] = 0.0
    amp[0, 0] = 0.0
    amp *= 0.06 / amp.square().sum().sqrt()
    decay = torch.arange(1, K + 1, device=DEV).double() ** -1.5
    co = torch.view_as_complex(ck * (amp[None, None, :, :, None] * decay)[..., None])
    for r in range(1, nz // 2):  # a real field: Hermitian in kz at kx = 0
        co[:, :, nz - r, 0] = co[:, :, r, 0].conj()
    if top:
        t = (1 - y) / 2
        q = 2 * t * t - 1
        wall_v, wall_g = t * (1 - t * t) ** 2 * 4, 1 - t * t
        U, W = 1.125 * (1 - t ** 8), 0.02 * (1 - t * t)
        poly = torch.cos(torch.arange(K, device=DEV).double()[:, None] * torch.arccos(q.clamp(-1, 1)))
    else:
        wall_v, wall_g = (1 - y * y) ** 2, 1 - y * y
        U, W = 1.125 * (1 - y ** 8), 0.02 * (1 - y * y)
        poly = _cos_table(N)[:K, :]
    A = _analysis(N)
    cv, cg = ((poly * w) @ A.T for w in (wall_v, wall_g))
    v = torch.einsum("bzxk,kn->bnzx", co[0], cv.to(torch.complex128))
    g = torch.einsum("bzxk,kn->bnzx", 3.0 * co[1], cg.to(torch.complex128))
    mean = torch.stack([A @ U, A @ W])
    return v, g, mean


def _states(c, seed, salt=0):
    """One serialised state per environment (the layout of env_get_state)."""
    v, g, mean = _flows(c, seed, salt)
    B, n = c["batch"], c["nz"] * (c["nx"] // 2)
    real = lambda a: torch.view_as_real(a.contiguous()).reshape(B, -1)  # noqa: E731
    tail = torch.zeros(B, 2 * n + 2, dtype=torch.float64, device=DEV)
    return torch.cat([real(v), real(g), mean.reshape(1, -1).expand(B, -1), tail], 1).cpu().numpy()


def _actions(c, seed, salt=0):
    """Zero-mean Gaussian wall velocities; about one in a hundred reaches the clip."""
    p = _physics(c)
    a = torch.randn(c["batch"], c["nz"], c["nx"], generator=_rng(seed, 7 + salt), dtype=torch.float64)
    return 0.4 * p["re_tau"] / p["re_bulk"] * (a - a.mean((1, 2), keepdim=True))


def _policy_layers(seed):
    gen = _rng(seed, 11)
    sizes = (2 * WINDOW * WINDOW, HIDDEN, HIDDEN, 1)
    return [(torch.randn(o, i, generator=gen, dtype=torch.float64) / math.sqrt(i),
             0.1 * torch.randn(o, generator=gen, dtype=torch.float64)) for i, o in zip(sizes, sizes[1:])]


def _nonlinear_input(c, seed):
    """Node values of six fields, [B][6][ny][nz][nx/2] complex, decaying spectra."""
    nz, nxh = c["nz"], c["nx"] // 2
    g = torch.Generator(DEV)
    g.manual_seed(1_000_003 * (int(seed) + 1) + 3)
    a = torch.view_as_complex(torch.randn(c["batch"], 6, c["ny"], nz, nxh, 2, generator=g, dtype=torch.float64, device=DEV))
    m = torch.arange(nz, device=DEV)
    m = torch.where(m < nz // 2, m, m - nz).double()
    i = torch.arange(nxh, device=DEV).double()
    a = a * (1.0 + i[None, :] ** 2 + m[:, None] ** 2) ** -0.75
    a[..., nz // 2, :] = 0
    a[..., 0, 0] = a[..., 0, 0].real.to(torch.complex128)
    for r in range(1, nz // 2):
        a[..., nz - r, 0] = a[..., r, 0].conj()
    return a


def _tau_input(c, seed):
    """lam of the stage operators (k^2 + 1 / (beta dt nu)) and of the Poisson problems, decaying right-hand sides."""
    g = torch.Generator(DEV)
    g.manual_seed(1_000_003 * (int(seed) + 1) + 5)
    M, ny = c["m"], c["ny"]
    lam = torch.exp(torch.rand(M, generator=g, dtype=torch.float64, device=DEV) * math.log(1e6))
    lam[::97] = 0.0
    r = torch.randn(M, ny, 2, generator=g, dtype=torch.float64, device=DEV)
    r = torch.view_as_complex(r * (1.0 + torch.arange(ny, device=DEV).double())[None, :, None] ** -1.0)
    w = torch.view_as_complex(torch.randn(2, M, 2, generator=g, dtype=torch.float64, device=DEV))
    return lam, r, w[0].contiguous(), w[1].contiguous()


# ---------------------------------------------------------------------------
# prepare and run
# ---------------------------------------------------------------------------

class _Handle:
    """An environment handle, destroyed with its owner."""

    def __init__(self, prm):
        from paper_2301_09889_gb300 import native
        self.native = native
        self.h = None
        self.h = native.env_create(prm)

    def __del__(self):
        if self.h is not None:
            self.native.env_destroy(self.h)


def _params(c):
    from paper_2301_09889_gb300 import native
    return native.params(nx=c["nx"], ny=c["ny"], nz=c["nz"], batch=c["batch"], precision=c["precision"], top_bc=c["top_bc"],
                         control=c["control"], steps_per_action=c["steps"], **_physics(c))


class _Server:
    """A batching server, stopped with its owner."""

    def __init__(self):
        from paper_2301_09889_gb300 import native
        self.native = native
        self.h = native.srv_create(16 << 30, 24)

    def __del__(self):
        self.native.srv_destroy(self.h)


def _groups(c):
    """The served classes as step cases, one batch entry per environment."""
    return [_step("", n, 65, n, batch=c[k], precision=1) for k, n in (("minimal", 16), ("mid", 32), ("larger", 64))]


def prepare(case, seed):
    c = case
    if c["kind"] == "served":
        srv, ids, acts = _Server(), [], []
        for k, g in enumerate(_groups(c)):
            states = _states(g, seed, 100 * k)
            for e in range(g["batch"]):
                ids.append(srv.native.srv_admit(srv.h, _params(dict(g, batch=1)), e))
                srv.native.srv_set_state(srv.h, ids[-1], states[e])
            acts.append(_actions(g, seed, 100 * k).numpy().reshape(-1))
        acts = np.concatenate(acts)
        return {"c": c, "srv": srv, "ids": ids, "acts": acts, "obs": np.zeros(2 * acts.size)}
    if c["kind"] == "tau":
        lam, r, top, bot = _tau_input(c, seed)
        return {"c": c, "lam": lam, "r": r, "top": top, "bot": bot, "f": torch.empty_like(r)}
    if c["kind"] == "nonlinear":
        q = _nonlinear_input(c, seed)
        env = _Handle(_params(dict(c, precision=0, top_bc=0, control=0, steps=1)))
        stream = torch.cuda.Stream()
        env.native.env_set_stream(env.h, stream.cuda_stream)
        h = torch.empty(c["batch"], 3, c["ny"], c["nz"], c["nx"] // 2, dtype=torch.complex128, device=DEV)
        torch.cuda.synchronize()
        return {"c": c, "env": env, "stream": stream, "q": q, "h": h}
    env = _Handle(_params(c))
    B, nz, nx = c["batch"], c["nz"], c["nx"]
    states = _states(c, seed)
    for e in range(B):
        env.native.env_set_state(env.h, e, states[e])
    s = {"c": c, "env": env}
    if c["control"] == 2:
        pol = env.native.policy(WINDOW, WINDOW, (HIDDEN, HIDDEN), True)
        env.native.env_set_policy(env.h, pol, torch.cat([t.reshape(-1) for wb in _policy_layers(seed) for t in wb]).numpy())
    act = _actions(c, seed) if c["control"] == 0 else None
    if c["io"] == "device":
        s["stream"] = torch.cuda.Stream()
        env.native.env_set_stream(env.h, s["stream"].cuda_stream)
        s["act"] = act.to(DEV) if act is not None else None
        s["out"] = torch.empty(B, 2 * nz * nx + 2, dtype=torch.float64, device=DEV)
        torch.cuda.synchronize()
    else:
        pin = lambda *shape: torch.zeros(*shape, dtype=torch.float64, pin_memory=True).numpy()  # noqa: E731
        s["obs"], s["tau"], s["rew"] = pin(B, 2, nz, nx), pin(B), pin(B)
        s["act"] = None
        if act is not None:
            s["act"] = pin(B, nz, nx)
            s["act"][:] = act.numpy()
        if c["io"] == "checkpoint":
            s["states"] = states
    return s


def run(state):
    s = state
    c = s["c"]
    if c["kind"] == "tau":
        from paper_2301_09889_gb300 import native
        native.ch_tau_helmholtz(c["ny"], c["m"], s["lam"].data_ptr(), s["r"].data_ptr(), s["top"].data_ptr(), s["bot"].data_ptr(),
                                s["f"].data_ptr(), torch.cuda.current_stream().cuda_stream)
        return s["f"]
    if c["kind"] == "served":
        srv = s["srv"]
        rc, tau, rew, status = srv.native.srv_wait_many(srv.h, srv.native.srv_submit_many(srv.h, s["ids"], s["acts"]), 60000, s["obs"])
        assert rc == 0 and not status.any()
        return {"obs": s["obs"].astype(np.float32), "wall_shear": tau.astype(np.float32), "reward": rew.astype(np.float32)}
    native, h = s["env"].native, s["env"].h
    if c["kind"] == "nonlinear":
        native.ch_nonlinear(h, s["q"].data_ptr(), s["h"].data_ptr())
        return s["h"]
    B, nz, nx = c["batch"], c["nz"], c["nx"]
    if c["io"] == "device":
        with torch.cuda.stream(s["stream"]):
            native.env_step_device(h, s["act"].data_ptr() if s["act"] is not None else None, s["out"].data_ptr())
            out = s["out"].float() if c["precision"] else s["out"]
        return {"obs": out[:, :-2].view(B, 2, nz, nx), "wall_shear": out[:, -2], "reward": out[:, -1]}
    if c["io"] == "checkpoint":
        for e in range(B):
            native.env_set_state(h, e, s["states"][e])
    native.env_step(h, s["act"], s["obs"], s["tau"], s["rew"])
    out = {"obs": s["obs"], "wall_shear": s["tau"], "reward": s["rew"]}
    if c["io"] == "checkpoint":
        # v, omega_y, U, W, the wall spectrum, time and step count of every environment
        out["state"] = np.stack([native.env_get_state(h, e) for e in range(B)])
    return {k: a.astype(np.float32) for k, a in out.items()} if c["precision"] else out


# ---------------------------------------------------------------------------
# what one pass cannot do without
# ---------------------------------------------------------------------------

def _plane_flops(nx, nz):
    """Nonlinear term of one plane: 6 inverse and 3 forward real 2D transforms on the 3/2 grid, the products."""
    mx, mz = 1.5 * nx, 1.5 * nz
    return 9 * (nx / 2) * 5 * mz * math.log2(mz) + 9 * mz * 2.5 * mx * math.log2(mx) + 9 * mx * mz


def work(case):
    c = case
    if c["kind"] == "tau":
        return {"bytes": c["m"] * (8 + 32 * c["ny"] + 32), "flops": c["m"] * c["ny"] * (2 * 13 + 12)}
    if c["kind"] == "served":
        parts = [work(g) for g in _groups(c)]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    nx, ny, nz, B = c["nx"], c["ny"], c["nz"], c["batch"]
    P, N = nz * nx // 2, ny - 1
    if c["kind"] == "nonlinear":
        return {"bytes": 9 * 16 * B * ny * P, "flops": B * ny * _plane_flops(nx, nz)}
    # the state (v, omega_y) read and written once, actions and observations;
    # per stage the plane transforms, nine complex Chebyshev transforms per mode
    # and the implicit half (about 170 operations per mode and node)
    stage = ny * _plane_flops(nx, nz) + P * (9 * 5 * N * math.log2(N) + 170 * ny)
    return {"bytes": B * (4 * 16 * ny * P + 8 * 3 * nx * nz), "flops": 3 * c["steps"] * B * stage}


# ---------------------------------------------------------------------------
# the same results in 64 bits
# ---------------------------------------------------------------------------

class _Dense:
    """Dense Chebyshev-tau / Fourier operators of one grid; pencils [B, P, ny]."""

    def __init__(self, c):
        ph = _physics(c)
        self.c, self.nx, self.ny, self.nz = c, c["nx"], c["ny"], c["nz"]
        nx, ny, nz = self.nx, self.ny, self.nz
        self.nxh, self.N = nx // 2, ny - 1
        N = self.N
        height = 2.0 if c["top_bc"] else 1.0
        self.nu, self.u_tau, self.dt = height / ph["re_bulk"], ph["re_tau"] / ph["re_bulk"], ph["dt"]
        f8 = {"dtype": torch.float64, "device": DEV}
        n = torch.arange(ny, **f8)
        self.S, self.A = _cos_table(N), _analysis(N)
        up = ((n[None, :] > n[:, None]) & ((n[None, :] + n[:, None]) % 2 == 1)).double()
        self.D = 2.0 * n[None, :] * up
        self.D[0] *= 0.5
        self.D2 = self.D @ self.D
        sign = 1.0 - 2.0 * (n % 2)
        one = torch.ones(ny, **f8)
        self.rows = {"top": one, "bot": sign, "dtop": n * n, "dbot": -sign * n * n, "d2top": n * n * (n * n - 1) / 3}
        self.flux = torch.where(n % 2 == 0, 2.0 / (1.0 - n * n + (n % 2)), torch.zeros_like(n))
        m = torch.arange(nz, device=DEV)
        m = torch.where(m < nz // 2, m, m - nz)
        m[nz // 2] = 0
        kx = 2 * math.pi / ph["lx"] * torch.arange(self.nxh, **f8)
        kz = 2 * math.pi / ph["lz"] * m.double()
        self.kx = kx[None, :].expand(nz, -1).reshape(-1, 1)
        self.kz = kz[:, None].expand(-1, self.nxh).reshape(-1, 1)
        self.k2 = self.kx ** 2 + self.kz ** 2
        keep = torch.ones(nz, self.nxh, dtype=torch.bool, device=DEV)
        keep[nz // 2] = False
        self.keep = keep.reshape(-1)
        live = self.keep.clone()
        live[0] = False
        self.live = live.nonzero()[:, 0]
        self.js = next((j for j in range(N, -1, -1) if (1 + math.cos(math.pi * j / N)) * ph["re_tau"] / height >= 15.0), 0)
        self.lu = [self._factor(k) for k in range(3)]

    def _factor(self, k):
        """LU of the omega_y, (phi, v), U and W systems of stage k."""
        N, ny, free = self.N, self.ny, self.c["top_bc"] == 1
        R, beta = self.rows, 0.5 * (GAMMA[k] + ZETA[k])
        s = 1.0 / (beta * self.dt * self.nu)
        k2 = self.k2[self.live, 0]
        eye = torch.eye(ny, dtype=torch.float64, device=DEV)[: N - 1]
        G = self.D2[: N - 1] - (k2 + s)[:, None, None] * eye
        wall = torch.stack([R["dtop"] if free else R["top"], R["bot"]])
        G = torch.cat([G, wall.repeat(len(k2), 1, 1)], 1)
        V = torch.zeros(len(k2), 2 * ny, 2 * ny, dtype=torch.float64, device=DEV)
        V[:, : N - 1, :ny] = G[:, : N - 1]
        V[:, N - 1: 2 * N - 2, :ny] = -eye
        V[:, N - 1: 2 * N - 2, ny:] = self.D2[: N - 1] - k2[:, None, None] * eye
        V[:, 2 * N - 2:, ny:] = torch.stack([R["top"], R["bot"], R["d2top"] if free else R["dtop"], R["dbot"]])
        W = torch.cat([self.D2[: N - 1] - s * eye, wall])
        U = torch.zeros(ny + 1, ny + 1, dtype=torch.float64, device=DEV)
        U[:ny, :ny] = W
        U[0, ny] = 2.0 / self.nu  # the forcing, with weight (alpha + beta) / beta
        U[ny, :ny] = self.flux
        return {"s": s, "ab": beta, "G": torch.linalg.lu_factor(G), "V": torch.linalg.lu_factor(V), "U": U, "W": W}

    def _solve(self, lu, rhs):
        """Complex right-hand sides [B, P, n] against the real systems [P, n, n]."""
        b = torch.view_as_real(rhs).permute(1, 2, 0, 3)
        x = torch.linalg.lu_solve(*lu, b.reshape(b.shape[0], b.shape[1], -1))
        return torch.view_as_complex(x.reshape(b.shape).permute(2, 0, 1, 3).contiguous())

    def _d(self, a):
        return a @ self.D.T.to(a.dtype)

    def _physical(self, f, mz, mx):
        """Kept spectra [..., nz, nxh] -> real values [..., mz, mx]."""
        h = self.nz // 2
        full = torch.zeros(*f.shape[:-2], mz, mx // 2 + 1, dtype=f.dtype, device=f.device)
        full[..., :h, : self.nxh] = f[..., :h, :]
        full[..., mz - h + 1:, : self.nxh] = f[..., h + 1:, :]
        return torch.fft.irfft2(full, s=(mz, mx), norm="forward")

    def _spectral(self, f):
        mz, h = f.shape[-2], self.nz // 2
        F = torch.fft.rfft2(f, norm="forward")[..., : self.nxh]
        out = torch.zeros(*f.shape[:-2], self.nz, self.nxh, dtype=F.dtype, device=f.device)
        out[..., :h, :] = F[..., :h, :]
        out[..., h + 1:, :] = F[..., mz - h + 1:, :]
        return out

    def cross(self, q):
        """Node spectra [B, 6, ..., nz, nxh] of velocity and vorticity -> dealiased u x omega."""
        u, v, w, ox, oy, oz = self._physical(q, 3 * self.nz // 2, 3 * self.nx // 2).unbind(1)
        return torch.stack([self._spectral(h) for h in (v * oz - w * oy, w * ox - u * oz, u * oy - v * ox)], 1)

    def _fields(self, st):
        v, g = st["v"], st["g"]
        ikx, ikz = 1j * self.kx, 1j * self.kz
        k2 = torch.where(self.k2 == 0, torch.ones_like(self.k2), self.k2)
        dv = self._d(v)
        u, w = (ikx * dv - ikz * g) / k2, (ikz * dv + ikx * g) / k2
        u[:, 0], w[:, 0] = st["U"].to(u.dtype), st["W"].to(u.dtype)
        ox, oz = self._d(w) - ikz * v, ikx * v - self._d(u)
        f = torch.stack([u, v, w, ox, g, oz], 1)
        return f * self.keep[:, None]

    def _stage(self, st, k, vw, prev):
        nz, nxh, ny = self.nz, self.nxh, self.ny
        f = self._fields(st)
        B = f.shape[0]
        nodes = (f @ self.S.T.to(f.dtype)).reshape(B, 6, nz, nxh, ny).permute(0, 1, 4, 2, 3)
        H = self.cross(nodes).permute(0, 1, 3, 4, 2).reshape(B, 3, nz * nxh, ny) @ self.A.T.to(f.dtype)
        hx, hy, hz = H.unbind(1)
        now = {"v": -self.k2 * hy - self._d(1j * self.kx * hx + 1j * self.kz * hz), "g": 1j * self.kz * hx - 1j * self.kx * hz,
               "U": hx[:, 0].real, "W": hz[:, 0].real}
        lu = self.lu[k]
        L, nul = self.live, lu["ab"] * self.dt * self.nu
        d2 = self.D2.T

        def rhs(a, name, k2):
            lap = a @ d2.to(a.dtype) - k2 * a
            h = GAMMA[k] * now[name] + (ZETA[k] * prev[name] if prev else 0)
            return -(a + nul * lap + self.dt * h) * lu["s"]

        v, g = st["v"], st["g"]
        rg = rhs(g, "g", self.k2)[:, L].clone()
        rg[..., ny - 2:] = 0
        rv = rhs(v @ d2.to(v.dtype) - self.k2 * v, "v", self.k2)[:, L]
        both = torch.zeros(B, len(L), 2 * ny, dtype=v.dtype, device=v.device)
        both[..., : ny - 2] = rv[..., : ny - 2]
        both[..., 2 * ny - 3] = vw[:, L]
        new = {"v": torch.zeros_like(v), "g": torch.zeros_like(g)}
        new["g"][:, L] = self._solve(lu["G"], rg)
        new["v"][:, L] = self._solve(lu["V"], both)[..., ny:]
        ru, rw = rhs(st["U"], "U", 0.0), rhs(st["W"], "W", 0.0)
        ru[:, ny - 2:], rw[:, ny - 2:] = 0, 0
        ru = torch.cat([ru, torch.full((B, 1), 2.0, dtype=torch.float64, device=DEV)], 1)
        new["U"] = torch.linalg.solve(lu["U"], ru.T).T[:, :ny]
        new["W"] = torch.linalg.solve(lu["W"], rw.T).T
        return new, now

    def observe(self, st):
        f = self._fields(st)[:, :2] @ self.S[self.js].to(torch.complex128)
        return self._physical(f.reshape(-1, 2, self.nz, self.nxh), self.nz, self.nx)

    def env_step(self, st, act, layers):
        """One environment step of every environment: (state, obs, wall shear, reward)."""
        c = self.c
        if c["control"] == 1:
            new = -(st["v"] @ self.S[self.js].to(torch.complex128)) * self.keep
        else:
            if c["control"] == 2:
                o, h = self.observe(st), WINDOW // 2
                x = torch.stack([torch.roll(o[:, ch], (h - dz, h - dx), (1, 2)) for ch in range(2) for dz in range(WINDOW)
                                 for dx in range(WINDOW)], -1)
                for w, b in layers[:-1]:
                    x = torch.relu(x @ w.to(DEV).T + b.to(DEV))
                act = self.u_tau * torch.tanh((x @ layers[-1][0].to(DEV).T + layers[-1][1].to(DEV))[..., 0])
            new = self._spectral(act.to(DEV).clamp(-self.u_tau, self.u_tau)).reshape(len(act), -1)
        new[:, 0] = 0
        old, shear = st["vw"], 0.0
        for s in range(c["steps"]):
            prev = None
            for k in range(3):
                vw = old + (s + C_END[k]) / c["steps"] * (new - old)
                st, prev = self._stage(st, k, vw, prev)
            shear = shear + self.nu * (st["U"] @ self.rows["dbot"])
        tau = shear / c["steps"]
        st["vw"] = new
        return st, self.observe(st), tau, 1.0 - tau / self.u_tau ** 2


def exact(case, seed):
    c = case
    if c["kind"] == "tau":
        lam, r, top, bot = _tau_input(c, seed)
        ny, N = c["ny"], c["ny"] - 1
        n = torch.arange(ny, dtype=torch.float64, device=DEV)
        D = 2.0 * n[None, :] * ((n[None, :] > n[:, None]) & ((n[None, :] + n[:, None]) % 2 == 1)).double()
        D[0] *= 0.5
        D2 = D @ D
        out = torch.empty_like(r)
        for a in range(0, c["m"], 4096):
            s = slice(a, min(a + 4096, c["m"]))
            M = (D2 - lam[s, None, None] * torch.eye(ny, dtype=torch.float64, device=DEV)).contiguous()
            M[:, N - 1], M[:, N] = 1.0, 1.0 - 2.0 * (n % 2)
            b = r[s].clone()
            b[:, N - 1], b[:, N] = top[s], bot[s]
            out[s] = torch.view_as_complex(torch.linalg.solve(M, torch.view_as_real(b)).contiguous())
        return out
    if c["kind"] == "served":
        parts = [_exact_step(g, seed, 100 * k) for k, g in enumerate(_groups(c))]
        return {k: torch.cat([p[k].reshape(-1) for p in parts]) for k in ("obs", "wall_shear", "reward")}
    nx, ny, nz = c["nx"], c["ny"], c["nz"]
    if c["kind"] == "nonlinear":
        d = _Dense.__new__(_Dense)
        d.nx, d.nz, d.nxh = nx, nz, nx // 2
        return d.cross(_nonlinear_input(c, seed))
    P = nz * nx // 2
    if 2 * P * (2 * ny) ** 3 > 5e11 or 24 * P * (2 * ny) ** 2 > 4e10:
        return None  # the dense systems take too long or too much memory
    return _exact_step(c, seed)


def _exact_step(c, seed, salt=0):
    ny, B, P = c["ny"], c["batch"], c["nz"] * c["nx"] // 2
    v, g, mean = _flows(c, seed, salt)
    pencils = lambda a: a.permute(0, 2, 3, 1).reshape(B, P, ny).contiguous()  # noqa: E731
    st = {"v": pencils(v), "g": pencils(g), "U": mean[0].expand(B, -1).clone(), "W": mean[1].expand(B, -1).clone(),
          "vw": torch.zeros(B, P, dtype=torch.complex128, device=DEV)}
    st, obs, tau, rew = _Dense(c).env_step(st, _actions(c, seed, salt) if c["control"] == 0 else None,
                                           _policy_layers(seed) if c["control"] == 2 else None)
    out = {"obs": obs, "wall_shear": tau, "reward": rew}
    if c["io"] == "checkpoint":
        real = lambda a: torch.view_as_real(a.permute(0, 2, 1).contiguous()).reshape(B, -1)  # noqa: E731
        clock = torch.tensor([_physics(c)["dt"] * c["steps"], float(c["steps"])], dtype=torch.float64, device=DEV).expand(B, -1)
        out["state"] = torch.cat([real(st["v"]), real(st["g"]), st["U"], st["W"], torch.view_as_real(st["vw"]).reshape(B, -1), clock], 1)
    return out
