"""Super-Gaussian envelopes of high order far from the pulse, where the
logarithmic derivatives of the envelope (u^(2g - 1) and its square) overflow
while the envelope is zero: lines, nodes, pushes and gradients there are those of
no pulse at all."""
import math

import numpy as np
import pytest

import oracle
from paper_2307_04843_gb300 import workloads
from support import THREADS, gpu_push, rel_u_err

L = 2 * math.pi


@pytest.mark.gpu
@pytest.mark.parametrize("order", [4, 8, 16])
@pytest.mark.parametrize("plasma", [True, False])
def test_split_line_longer_than_the_pulse(order, plasma):
    """Float against FP64.  Tolerance as for the split line at other orders:
    the envelope's exponent u^(2g) is good to 2g 2^-24 (3e-6 at order 16), J1 of
    amplitude 1e-3 enters E2 through dt, 100 steps of 0.28: below 1e-7 in all,
    1e-6 is held."""
    import torch
    from paper_2307_04843_gb300 import _lib
    nz, dz = 6144, L / 20
    dt = 0.9 * dz
    pulse = dict(kind="plane", pol="x", a0=0.8, omega=1.0, env="sgauss", sg_order=order, env_len=12.0)
    if plasma:
        pulse.update(omega_p=math.sqrt(1e-3), yee=True, yee_dx=dz, yee_dt=dt)
    out = []
    with _lib.Handle(pulse) as h:
        for dtype in (torch.float64, torch.float32):
            E, B, J = (torch.zeros((2, nz), dtype=dtype, device="cuda") for _ in range(3))
            h.apt1d(E, B, J, -0.5 * nz * dz, dz, -1.5, dt, 100, omega_p=math.sqrt(1e-3))
            out.append([v.double().cpu().numpy() for v in (E, B, J)])
    for a, b in zip(*out):
        assert np.all(np.isfinite(a)) and np.max(np.abs(a - b)) <= 1e-6


PLASMA = dict(kind="plane", pol="cp", env="sgauss", sg_order=16, env_len=10.0, a0=0.8, omega_p=0.3)


@pytest.mark.gpu
@pytest.mark.parametrize("precision,launch", [("fp32", dict(block=32)), ("fp32", dict(block=32, pairs=1)),
                                              ("fp32_phase64", None), ("fp64", None)])
def test_push_far_from_a_plasma_pulse(precision, launch):
    far = 2e7 if precision == "fp64" else 2000.0
    rng = np.random.default_rng(4)
    n = 70
    parts = dict(x=rng.uniform(-1, 1, n), y=rng.uniform(-1, 1, n), z=rng.uniform(-15.0, 15.0, n),
                 ux=np.zeros(n), uy=np.zeros(n), uz=np.zeros(n))
    parts["z"][1::2] += far
    out, _, st = gpu_push(PLASMA, parts, -5.0, 0.05, 200, precision, launch=launch)
    assert st == 0
    for k in ("ux", "uy", "uz"):
        assert np.all(out[k][1::2] == 0.0)
    near = {k: v[::2] for k, v in parts.items()}
    ref = oracle.push(PLASMA, near, -5.0, 0.05, 200, threads=THREADS)
    e = rel_u_err({k: v[::2] for k, v in out.items()}, ref)
    if precision == "fp64":
        assert np.max(e) <= 1e-10
    else:
        assert np.median(e) <= 1e-4 and np.max(e) <= 1e-3
    assert np.max(np.abs(ref["ux"])) > 0.3


@pytest.mark.gpu
@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_nodes_and_current_far_from_a_plasma_pulse(precision):
    import torch
    from paper_2307_04843_gb300 import _lib
    nz = 4001
    f = torch.full((6, nz, 1, 4), 9.0, dtype=torch.float64, device="cuda")
    j = torch.full((3, nz, 1, 4), 9.0, dtype=torch.float64, device="cuda")
    d = 2e5 if precision == "fp64" else 1.0
    with _lib.Handle(PLASMA) as h:
        h.eval_nodes(list(f), [0.0, 0.0, 15.0], [0.5, 0.5, d], 0.0, precision=precision)
        h.eval_current(list(j), [0.0, 0.0, 15.0], [0.5, 0.5, d], 0.0, precision=precision)
    assert torch.all(f == 0.0) and torch.all(j == 0.0)


@pytest.mark.gpu
@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("kind", ["plane", "gauss", "lg"])
def test_adjoint_with_particles_far_from_the_pulse(kind, precision):
    """Far particles add gamma = 1 each and nothing to the gradient."""
    import torch
    from paper_2307_04843_gb300 import _lib, autograd
    pulse = dict(kind=kind, pol="x", a0=1.5, omega=1.0, w0=2.5 * L, z_focus=0.0, env="sgauss", sg_order=16, env_len=10.0,
                 lg_p=1, lg_l=1)
    n = 256
    near = workloads.particles_uniform(((-2 * L, 2 * L),) * 2 + ((-L, L),), n, 5)
    both = {k: np.concatenate([v, v]) for k, v in near.items()}
    both["z"][n:] += 2e12 if precision == "fp64" else 2e5
    res = []
    for parts in (near, both):
        dev = _lib.to_device(parts, precision)
        off = torch.tensor([0, parts["x"].size], dtype=torch.int64, device="cuda")
        J, dJ = autograd.adjoint([pulse], dev, off, -2.0, 0.02, 60, 20, precision)
        res.append((J.cpu().numpy(), dJ.cpu().numpy()))
    np.testing.assert_allclose(res[1][0], 0.5 * (res[0][0] + 1.0), rtol=1e-6)
    np.testing.assert_allclose(res[1][1], 0.5 * res[0][1], rtol=1e-5, atol=1e-9)
    assert np.abs(res[0][1][0, 0]) > 1e-3
