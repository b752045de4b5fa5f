"""The register-resident float lines at the lengths where their blocking can go
wrong: two nodes, lengths around a warp's, around the switches from one number
of nodes per thread to the next, and the longest.

Vacuum and plasma lines: bit for bit against a float32 loop of the same
separately rounded operations.  Split line: against the FP64 split line on the
same inputs, every envelope (orders with and without a kernel of their own).
Tolerance of the split line: the carrier phase and the special functions are
good to about 5e-7 of the field, J1 of amplitude omega_p^2 a0 = 1e-3 a0 enters E2
through dt, so 200 steps keep E2 within 200 dt 1e-3 5e-7 < 5e-8 a0 of the FP64
line; 1e-6 a0 is held."""
import math

import numpy as np
import pytest

F = np.float32


def _float_line(E, B, J, wp2, r, hr, dt, n):
    q = F(dt) * wp2
    for _ in range(n):
        B[:-1] = B[:-1] - F(hr) * (E[1:] - E[:-1])
        J[:] = J + q * E
        E[1:] = (E[1:] - F(r) * (B[1:] - B[:-1])) - F(dt) * J[1:]
        B[:-1] = B[:-1] - F(hr) * (E[1:] - E[:-1])


@pytest.mark.gpu
@pytest.mark.parametrize("nz", [2, 3, 63, 64, 65, 129, 2047, 2048, 2049, 3071, 3073, 4097, 8191, 8192])
@pytest.mark.parametrize("n_lines", [1, 160])
def test_float_lines_bit_exact_at_blocking_edges(nz, n_lines):
    import torch
    from paper_2307_04843_gb300 import _lib
    rng = np.random.default_rng(nz)
    a = [rng.standard_normal(nz).astype(F) for _ in range(3)]
    wp2 = (0.01 * rng.random(nz)).astype(F)
    dz, dt, n = 0.1, 0.09, 13
    dev = [torch.as_tensor(np.tile(v, (n_lines, 1))).cuda() for v in a]
    _lib.ap_plasma1d_run(dev[0], dev[1], dev[2], dz, dt, n, wp2=torch.as_tensor(np.tile(wp2, (n_lines, 1))).cuda())
    ref = [v.copy() for v in a]
    _float_line(*ref, wp2, dt / dz, 0.5 * dt / dz, dt, n)
    for d, v in zip(dev, ref):
        assert np.array_equal(d.cpu().numpy(), np.tile(v, (n_lines, 1)))
    # without plasma: the vacuum line
    E, B = (torch.as_tensor(np.tile(v, (n_lines, 1))).cuda() for v in a[:2])
    _lib.ap_yee1d_run(E, B, dz, dt, n)
    e, b = a[0].copy(), a[1].copy()
    _float_line(e, b, np.zeros(nz, F), np.zeros(nz, F), dt / dz, 0.5 * dt / dz, 0.0, n)
    assert np.array_equal(E.cpu().numpy(), np.tile(e, (n_lines, 1)))
    assert np.array_equal(B.cpu().numpy(), np.tile(b, (n_lines, 1)))


ENVS = [dict(env="gauss", env_len=25.0), dict(env="sgauss", sg_order=1, env_len=20.0),
        dict(env="sgauss", sg_order=3, env_len=25.0), dict(env="sgauss", sg_order=4, env_len=30.0), dict(env="cw"),
        dict(env="sin2", env_len=6.0, vacuum=True)]


@pytest.mark.gpu
@pytest.mark.parametrize("nz", [2, 65, 512, 513, 1536, 1537, 4097])
@pytest.mark.parametrize("env", ENVS, ids=lambda e: e["env"] + str(e.get("sg_order", "")))
def test_split_line_float_matches_fp64(nz, env):
    import torch
    from paper_2307_04843_gb300 import _lib
    env = dict(env)
    dz = 2 * math.pi / 20
    dt = 0.9 * dz
    wp = math.sqrt(1e-3)
    pulse = dict(kind="plane", pol="x", a0=0.8, omega=1.0, phase0=0.3, z_focus=0.4, t_focus=-0.2)
    if not env.pop("vacuum", False):
        pulse.update(omega_p=wp, yee=True, yee_dx=dz, yee_dt=dt)
    pulse.update(env)
    rng = np.random.default_rng(nz)
    init = [1e-3 * rng.standard_normal((2, nz)) for _ in range(3)]
    out = {}
    with _lib.Handle(pulse) as h:
        for dtype in (torch.float64, torch.float32):
            E, B, J = (torch.as_tensor(v).cuda().float().to(dtype).contiguous() for v in init)
            h.apt1d(E, B, J, -0.5 * nz * dz, dz, -1.5, dt, 200, omega_p=wp)
            out[dtype] = [v.double().cpu().numpy() for v in (E, B, J)]
    for a, b in zip(out[torch.float32], out[torch.float64]):
        assert np.max(np.abs(a - b)) <= 1e-6, np.max(np.abs(a - b))
