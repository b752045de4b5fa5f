"""Gaussian beams on the grid nodes (float-float, rows of 32 nodes and more)
at the shapes where the slab kernel can go wrong: rows that end inside a
column block or a lane's four columns, rows aligned to 16 bytes and not, more
rows than a slab's 32, runs that cross z indices; both beam kinds, every
polarisation, stores and sums, float and double arrays, three components.

Tolerance as for the other FP32 node values: 4e-6 a0 against the oracle (plus one
float rounding of what is added to)."""
import math

import numpy as np
import pytest

import oracle

L = 2 * math.pi
KINDS = {"gauss": {}, "flying_cf": dict(beta_f=-1.0)}


def _case(kind, pol, shape, dtype, accumulate, offset=0, comps=range(6), **over):
    import torch
    from paper_2307_04843_gb300 import _lib
    pulse = dict(kind=kind, pol=pol, env="gauss", env_len=30.0, a0=1.5, w0=1.7 * L, z_focus=0.3, t_focus=0.2,
                 longitudinal=True, **KINDS[kind])
    pulse.update(over)
    nz, ny, nx = shape
    d = (4.0 * L / nx, 4.0 * L / ny, 1.1 * L / nz)
    lo = (-2.03 * L, -1.95 * L, -0.5 * L)
    ref = oracle.yee_nodes(pulse, shape, lo, d, 0.7)
    n = nz * ny * nx
    rng = np.random.default_rng(nx)
    base = rng.standard_normal((6, n)).astype(np.float32) if accumulate else np.zeros((6, n), np.float32)
    raw = [torch.zeros(n + 4, dtype=dtype, device="cuda") for _ in range(6)]
    f = [r[offset:offset + n].view(shape) if c in comps else None for c, r in enumerate(raw)]
    for c in comps:
        f[c].copy_(torch.as_tensor(base[c]).view(shape))
    with _lib.Handle(pulse) as h:
        h.eval_nodes(f, lo, d, 0.7, accumulate=accumulate, precision="fp32")
        assert h.status() == 0
    for c in comps:
        got = f[c].double().cpu().numpy()
        want = ref[c] + base[c].reshape(shape)
        assert np.all(np.abs(got - want) <= 4e-6 * pulse["a0"] + 6e-8 * np.abs(want)), (c, np.max(np.abs(got - want)))
        edge = raw[c].clone()
        edge[offset:offset + n] = 0
        assert not edge.any()  # nothing outside the arrays


@pytest.mark.gpu
@pytest.mark.parametrize("shape", [(2, 3, 32), (1, 33, 128), (3, 70, 129), (2, 32, 132), (5, 9, 260), (40, 1, 64)])
@pytest.mark.parametrize("kind", sorted(KINDS))
def test_slab_shapes(kind, shape):
    import torch
    _case(kind, "x", shape, torch.float32, False)
    _case(kind, "cp", shape, torch.float64, True)


@pytest.mark.gpu
@pytest.mark.parametrize("pol", ["x", "y", "cp", "cm"])
@pytest.mark.parametrize("accumulate", [False, True])
def test_slab_polarisations_and_unaligned_arrays(pol, accumulate):
    import torch
    for offset in (0, 1):  # 16-byte accesses, and rows that do not allow them
        _case("gauss", pol, (3, 37, 64), torch.float32, accumulate, offset)
    _case("gauss", pol, (3, 5, 64), torch.float32, accumulate, comps=(0, 2, 5))
    _case("gauss", pol, (3, 5, 64), torch.float32, accumulate, longitudinal=False, env="sin2", env_len=5.0)
