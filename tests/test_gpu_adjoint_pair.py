"""The two-particle float-float adjoint over its frames, envelopes and segment
lengths: both kinds, all polarisations, every envelope, checkpoint intervals
from 1 to the largest (the kernel picks its own segments within the
workspace that they buy), a zero amplitude, and tiles with a padding partner.

Reference: the FP64 adjoint (one particle per thread, generic Boris reverse) on
the same inputs.  Tolerance: 1e-3 of the row or of a thousandth of the largest,
as the method's gradients are held to."""
import math

import numpy as np
import pytest

from paper_2307_04843_gb300 import workloads

L = 2 * math.pi
KINDS = {"gauss": {}, "flying_cf": dict(beta_f=-0.6)}
ENVS = {"gauss": dict(env="gauss", env_len=25.0), "sin2": dict(env="sin2", env_len=4.0),
        "sgauss": dict(env="sgauss", sg_order=2, env_len=20.0), "cw": dict(env="cw")}


def _run(pulses, parts, off, n_steps, K, precision):
    import torch
    from paper_2307_04843_gb300 import _lib, autograd
    dev = _lib.to_device(parts, precision)
    J, dJ = autograd.adjoint(pulses, dev, torch.as_tensor(off).cuda(), -2.0, 0.02, n_steps, K, precision)
    return J.cpu().numpy(), dJ.cpu().numpy()


def _check(pulses, n_per, n_steps, K):
    off = (np.arange(len(pulses) + 1) * n_per).astype(np.int64)
    parts = workloads.particles_uniform(((-4 * L, 4 * L),) * 2 + ((-5 * L, 5 * L),), int(off[-1]), 31)
    rng = np.random.default_rng(8)
    for k in ("ux", "uy", "uz"):
        parts[k] = np.float32(rng.normal(0.0, 0.3, off[-1])).astype(np.float64)
    J64, d64 = _run(pulses, parts, off, n_steps, max(K, 16), "fp64")
    J32, d32 = _run(pulses, parts, off, n_steps, K, "fp32")
    np.testing.assert_allclose(J32, J64, rtol=1e-5)
    for c in range(4):
        scale = np.maximum(np.abs(d64[:, c]), 1e-3 * np.max(np.abs(d64)))
        assert np.all(np.abs(d32[:, c] - d64[:, c]) <= 1e-3 * scale), (c, d32[:, c], d64[:, c])


@pytest.mark.gpu
@pytest.mark.parametrize("lon", [True, False])
@pytest.mark.parametrize("env", sorted(ENVS))
@pytest.mark.parametrize("kind", sorted(KINDS))
def test_pair_adjoint_matches_fp64(kind, env, lon):
    pulses = [dict(kind=kind, pol=pol, a0=a0, omega=1.0, w0=2.5 * L, z_focus=0.5, t_focus=0.1, phase0=0.3,
                   longitudinal=lon, **KINDS[kind], **ENVS[env])
              for pol, a0 in (("x", 2.0), ("y", -1.5), ("cp", 2.5), ("cm", 1.0), ("x", 0.0))]
    _check(pulses, 129, 90, 20)


@pytest.mark.gpu
@pytest.mark.parametrize("n_steps,K", [(1, 1), (17, 1), (33, 256), (200, 1), (200, 7), (200, 200), (301, 256)])
def test_pair_adjoint_segment_lengths(n_steps, K):
    pulses = [dict(kind="gauss", pol="x", a0=2.0, omega=1.0, w0=2.5 * L, z_focus=0.5, longitudinal=True, **ENVS["gauss"])]
    _check(pulses, 257, n_steps, K)
