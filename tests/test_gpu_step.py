"""The float-float step over its polarisation frames, kinds and envelopes:
every polarisation of every kind (y-polarised and left-handed pulses run in a
turned or mirrored frame without a grid, and are turned into the grid's frame
with one), Laguerre orders at the loop edges of the step (p, |l| = 0, 1, 2,
both signs of l), an odd and the smallest number of flying-focus components,
and every envelope, one and two particles per thread.

Tolerances as for the other float-float pushes (median relative |du| <= 1e-4,
max <= 1e-3 against the oracle); the one- and two-particle kernels round alike,
so they agree bit for bit, with and without the light-front diagnostic."""
import math

import numpy as np
import pytest

import oracle
from paper_2307_04843_gb300 import workloads
from support import THREADS, gpu_push, rel_u_err

L = 2 * math.pi
BASE = dict(a0=3.0, omega=1.0, w0=2.5 * L, z_focus=0.7, t_focus=0.2, phase0=0.4, longitudinal=True, env="gauss", env_len=25.0)
KINDS = {
    "plane": dict(kind="plane"),
    "gauss": dict(kind="gauss"),
    "flying_cf": dict(kind="flying_cf", beta_f=-0.6),
    "lg00": dict(kind="lg", lg_p=0, lg_l=0),
    "lg01": dict(kind="lg", lg_p=0, lg_l=1),
    "lg0m2": dict(kind="lg", lg_p=0, lg_l=-2),
    "lg10": dict(kind="lg", lg_p=1, lg_l=0),
    "lg12": dict(kind="lg", lg_p=1, lg_l=2),
    "lg2m1": dict(kind="lg", lg_p=2, lg_l=-1),
    "flying2": dict(kind="flying", env="cw", n_comp=2, bw_frac=0.05, beta_f=0.99, ff_length=20 * L),
    "flying5": dict(kind="flying", env="cw", n_comp=5, bw_frac=0.04, beta_f=-0.8, ff_length=15 * L, a0=-2.0),
}


def _parts(n):
    parts = workloads.particles_uniform(((-4 * L, 4 * L),) * 2 + ((-5 * L, 5 * L),), n, 99)
    rng = np.random.default_rng(5)
    for k in ("ux", "uy", "uz"):  # float-representable momenta
        parts[k] = np.float32(rng.normal(0.0, 0.5, n)).astype(np.float64)
    return parts


def _check(out, ref):
    e = rel_u_err(out, ref)
    assert np.median(e) <= 1e-4 and np.max(e) <= 1e-3, (np.median(e), np.max(e))


def _same(a, b):
    for k in a:
        np.testing.assert_array_equal(a[k], b[k], err_msg=k)


@pytest.mark.gpu
@pytest.mark.parametrize("pol", ["x", "y", "cp", "cm"])
@pytest.mark.parametrize("name", sorted(KINDS))
def test_step_frames_and_kinds_match_oracle(name, pol):
    pulse = dict(BASE, pol=pol, **KINDS[name])
    parts = _parts(37)  # one warp and a ragged one; with pairs a padding partner
    args = (pulse, parts, -3.0, 0.02, 150, "fp32")
    ref = oracle.push(pulse, parts, -3.0, 0.02, 150, threads=THREADS)
    one, _, st1 = gpu_push(*args, launch=dict(block=32))
    two, _, st2 = gpu_push(*args, launch=dict(block=32, pairs=1))
    assert st1 == 0 and st2 == 0
    _check(one, ref)
    _same(one, two)
    lf, _, _ = gpu_push(*args, diag_keys=("lightfront",), launch=dict(block=32, pairs=1))
    _same(one, lf)


@pytest.mark.gpu
@pytest.mark.parametrize("pol", ["x", "y", "cp", "cm"])
@pytest.mark.parametrize("name", ["plane", "gauss", "lg12", "flying5"])
def test_step_frames_with_grid_match_oracle(name, pol):
    import torch
    from paper_2307_04843_gb300 import _lib
    pulse = dict(BASE, pol=pol, **KINDS[name])
    parts = _parts(37)
    box = ((-4 * L, 4 * L),) * 2 + ((-5 * L, 5 * L),)
    lo, hi = tuple(b[0] for b in box), tuple(b[1] for b in box)
    g = workloads.grid_field(box, 20, amplitude=0.2)
    ref = oracle.push(pulse, parts, -3.0, 0.02, 150, grid=(g, lo, hi), threads=THREADS)
    cells = _lib.pack_grid((torch.as_tensor(g).cuda(), lo, hi), layout="cells")
    args = (pulse, parts, -3.0, 0.02, 150, "fp32")
    base, _, _ = gpu_push(*args, grid=cells, launch=dict(block=64))
    _check(base, ref)
    for launch in (dict(block=64, grid_cache=1), dict(block=64, pairs=1), dict(block=64, pairs=1, grid_cache=1),
                   dict(block=64, pairs=1, grid_cache=2)):
        out, _, st = gpu_push(*args, grid=cells, launch=launch)
        assert st == 0
        _same(base, out)
    arrays, _, _ = gpu_push(*args, grid=(g, lo, hi))
    _check(arrays, ref)


@pytest.mark.gpu
@pytest.mark.parametrize("env", [dict(env="sin2", env_len=3.0), dict(env="sgauss", sg_order=1, env_len=9.0),
                                 dict(env="sgauss", sg_order=4, env_len=12.0), dict(env="cw")])
@pytest.mark.parametrize("name", ["plane", "gauss", "flying_cf", "lg12"])
def test_step_envelopes_match_oracle(name, env):
    pulse = dict(BASE, pol="x", **KINDS[name])
    pulse.update(env)
    parts = _parts(37)
    ref = oracle.push(pulse, parts, -3.0, 0.02, 150, threads=THREADS)
    one, _, _ = gpu_push(pulse, parts, -3.0, 0.02, 150, "fp32", launch=dict(block=32))
    two, _, _ = gpu_push(pulse, parts, -3.0, 0.02, 150, "fp32", launch=dict(block=32, pairs=1))
    _check(one, ref)
    _same(one, two)


def _default_and_one(pulse, parts, **kw):
    args = (pulse, parts, -3.0, 0.02, 12, "fp32")
    out, dg, st = gpu_push(*args, **kw)
    one, dg1, _ = gpu_push(*args, launch=dict(block=128), **kw)
    assert st == 0
    _same(out, one)
    return dg, dg1


@pytest.mark.gpu
@pytest.mark.parametrize("grid,per_sm", [(False, 640), (True, 1536)])
def test_default_shape_gives_the_same_bits_on_both_sides_of_its_lines(grid, per_sm):
    """The library's own launch shape (no ap_set_launch) just below and just
    above the sizes where it changes, against one particle per thread."""
    import torch
    from paper_2307_04843_gb300 import _lib
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    pulse = dict(BASE, pol="x", **KINDS["gauss"])
    g = None
    if grid:
        box = ((-4 * L, 4 * L),) * 2 + ((-5 * L, 5 * L),)
        f = torch.as_tensor(workloads.grid_field(box, 20, amplitude=0.2)).cuda()
        g = _lib.pack_grid((f, tuple(b[0] for b in box), tuple(b[1] for b in box)), layout="cells")
    for n in (per_sm * sms - 1, per_sm * sms + 1):
        dg, dg1 = _default_and_one(pulse, _parts(n), grid=g, hist=(4096, 0.0, 20.0))
        np.testing.assert_array_equal(dg["hist"], dg1["hist"])


@pytest.mark.gpu
def test_default_shape_batched():
    import torch
    from paper_2307_04843_gb300 import _lib
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    pulses = [dict(BASE, pol=p, **KINDS["gauss"]) for p in ("x", "cm", "y")]
    for n in (2048 * sms - 1, 2048 * sms + 1):
        parts = _parts(n)
        off = torch.tensor([0, n // 5, n // 5, n], dtype=torch.int64, device="cuda")
        res = []
        for launch in (None, dict(block=128)):
            with _lib.Handle(pulses) as h:
                if launch:
                    h.set_launch(**launch)
                dev = _lib.to_device(parts, "fp32")
                ws = torch.zeros(64, dtype=torch.int32, device="cuda")
                _lib.ap_gather_push_batched(h.h, dev, off, None, -3.0, 0.02, 12, "fp32", None, ws)
                assert h.status() == 0
                res.append(_lib.to_host(dev))
        _same(*res)


@pytest.mark.gpu
@pytest.mark.parametrize("z_focus", [2 * math.pi * 1e3, -2 * math.pi * 1e4])
def test_grid_gather_with_the_focus_far_from_the_grid(z_focus):
    """The grid unit along z is good to 2^-24 of itself wherever the pulse's
    focus (the origin of the step's longitudinal coordinate) lies.

    Node values of size A = 0.5 without any smoothness: a weight error of e
    cells in each of three directions moves the field by up to 6 A e.  With 33
    nodes e <= 3 * 2^-24 * 32, so over a time of 3 the momentum moves by
    5e-5, about 1e-4 with what the trajectory feeds back.  An error of 2^-24 of
    the focus distance in cells would move it by 1e-3 and 1e-2."""
    import torch
    from paper_2307_04843_gb300 import _lib
    rng = np.random.default_rng(7)
    box = ((-16.0, 16.0),) * 3
    lo, hi = (-16.0,) * 3, (16.0,) * 3
    g = np.float32(rng.uniform(-0.5, 0.5, (6, 33, 33, 33)))
    parts = workloads.particles_uniform(box, 257, 3)
    pulse = dict(kind="gauss", pol="x", env="gauss", env_len=25.0, a0=0.0, omega=1.0, w0=10.0, z_focus=z_focus)
    args = (pulse, parts, 0.3, 0.05, 60, "fp32")
    ref = oracle.push(pulse, parts, 0.3, 0.05, 60, grid=(g, lo, hi), threads=THREADS)
    dev = torch.as_tensor(g).cuda()
    cells = _lib.pack_grid((dev, lo, hi), layout="cells")
    outs = [gpu_push(*args, grid=cells, launch=kw)[0]
            for kw in (dict(block=64), dict(block=64, grid_cache=1), dict(block=64, pairs=1),
                       dict(block=64, pairs=1, grid_cache=1), dict(block=64, pairs=1, grid_cache=2))]
    arrays = gpu_push(*args, grid=(dev, lo, hi), launch=dict(block=64))[0]
    for out in outs[:1] + [arrays]:
        d = max(np.max(np.abs(out[k] - ref[k])) for k in ("ux", "uy", "uz"))
        assert d <= 1e-4, d
    for out in outs[1:]:
        _same(outs[0], out)


@pytest.mark.gpu
def test_envelope_argument_far_from_the_focus():
    """eta = (t - t_f) - (z - z_f)/v_g of an electron that meets the pulse at a
    large distance D = 1.04e6 from the focus is good to the rounding of t - t_f
    and of z - z_f.  The first is the same for all particles of a step, at most
    2^-25 2^20 = 0.031 here; the second averages out over 4000 particles (0.03 /
    sqrt(4000)), so the mean error stays within 0.035.  A mismatch between the
    factors of the two terms would add up to 2^-24 D = 0.06 to it, and 0.099 for
    this envelope if each factor is rounded to float for itself."""
    D, T = 1.04e6, 22.5
    rng = np.random.default_rng(11)
    n = 4000
    eta = rng.uniform(8.0, 14.0, n)
    eta = eta[np.cos(eta) > 0.5]
    n = eta.size
    zero = np.zeros(n)
    parts = dict(x=zero.copy(), y=zero.copy(), z=D - eta, ux=zero.copy(), uy=zero.copy(), uz=zero.copy())
    pulse = dict(kind="plane", pol="x", env="gauss", env_len=T, a0=1.0, omega=1.0)
    ref = oracle.push(pulse, parts, D, 1e-3, 1, threads=THREADS)
    for launch in (dict(block=32), dict(block=32, pairs=1)):
        out, _, st = gpu_push(pulse, parts, D, 1e-3, 1, "fp32", launch=launch)
        assert st == 0
        # d ln Gamma = -4 ln2 eta / T^2 d eta
        d = -np.log(out["ux"] / ref["ux"]) * T * T / (4 * math.log(2.0) * eta)
        assert abs(np.mean(d)) <= 0.035, np.mean(d)


@pytest.mark.gpu
@pytest.mark.parametrize("pol", ["x", "y", "cp", "cm"])
@pytest.mark.parametrize("env", [dict(env="gauss", env_len=15.0), dict(env="sgauss", sg_order=1, env_len=9.0),
                                 dict(env="sgauss", sg_order=5, env_len=12.0), dict(env="cw")])
def test_plasma_pulse_gives_the_same_bits_in_every_shape(env, pol):
    """The finite-duration terms of a pulse in a plasma round alike with one and
    two particles per thread, without a grid and with every cell cache."""
    import torch
    from paper_2307_04843_gb300 import _lib
    pulse = dict(kind="plane", pol=pol, a0=2.0, omega=1.0, omega_p=0.4, phase0=0.3, z_focus=0.7, **env)
    parts = _parts(199)
    box = ((-4 * L, 4 * L),) * 2 + ((-5 * L, 5 * L),)
    lo, hi = tuple(b[0] for b in box), tuple(b[1] for b in box)
    g = workloads.grid_field(box, 20, amplitude=0.2)
    cells = _lib.pack_grid((torch.as_tensor(g).cuda(), lo, hi), layout="cells")
    args = (pulse, parts, -3.0, 0.02, 150, "fp32")
    one, _, st = gpu_push(*args, launch=dict(block=32))
    assert st == 0
    _check(one, oracle.push(pulse, parts, -3.0, 0.02, 150, threads=THREADS))
    _same(one, gpu_push(*args, launch=dict(block=32, pairs=1))[0])
    base, _, _ = gpu_push(*args, grid=cells, launch=dict(block=64))
    for launch in (dict(block=64, grid_cache=1), dict(block=64, pairs=1), dict(block=64, pairs=1, grid_cache=1),
                   dict(block=64, pairs=1, grid_cache=2)):
        _same(base, gpu_push(*args, grid=cells, launch=launch)[0])


@pytest.mark.gpu
@pytest.mark.parametrize("per_set", [60, 257])
def test_default_shape_batched_with_a_grid(per_set):
    """Many small sets on a per-cell grid: the default pads a set to tiles of 64
    (a tile counter's final value shows the tiles: their number and one more pop
    for each block), and the states are those of an explicit shape."""
    import torch
    from paper_2307_04843_gb300 import _lib
    n_sets = 4096
    n = n_sets * per_set
    pulses = [dict(BASE, pol=p, **KINDS["gauss"]) for p in ("x", "cm")] * (n_sets // 2)
    parts = _parts(n)
    box = ((-4 * L, 4 * L),) * 2 + ((-5 * L, 5 * L),)
    f = torch.as_tensor(workloads.grid_field(box, 20, amplitude=0.2)).cuda()
    g = _lib.pack_grid((f, tuple(b[0] for b in box), tuple(b[1] for b in box)), layout="cells")
    off = torch.arange(n_sets + 1, dtype=torch.int64, device="cuda") * per_set
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    res = []
    for launch in (None, dict(block=128)):
        with _lib.Handle(pulses) as h:
            if launch:
                h.set_launch(**launch)
            dev = _lib.to_device(parts, "fp32")
            ws = torch.zeros(64, dtype=torch.int32, device="cuda")
            _lib.ap_gather_push_batched(h.h, dev, off, g, -3.0, 0.02, 4, "fp32", None, ws)
            assert h.status() == 0
            res.append(_lib.to_host(dev))
        if launch is None:
            pops = int(ws[0]) - n_sets * (-(-per_set // 64))
            assert 0 < pops <= 64 * sms, int(ws[0])
    _same(*res)


@pytest.mark.gpu
def test_set_launch_without_a_shape_gives_the_default_back():
    """Handle.set_launch() after an explicit shape: the tiles of the next batched
    call (see the tile counter) are those of a fresh handle."""
    import torch
    from paper_2307_04843_gb300 import _lib
    n_sets, per_set = 4096, 257
    parts = _parts(n_sets * per_set)
    box = ((-4 * L, 4 * L),) * 2 + ((-5 * L, 5 * L),)
    f = torch.as_tensor(workloads.grid_field(box, 20, amplitude=0.2)).cuda()
    g = _lib.pack_grid((f, tuple(b[0] for b in box), tuple(b[1] for b in box)), layout="cells")
    off = torch.arange(n_sets + 1, dtype=torch.int64, device="cuda") * per_set
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    with _lib.Handle([dict(BASE, pol="x", **KINDS["gauss"])] * n_sets) as h:
        for launch, tile in ((dict(block=256), 256), (dict(), 64)):
            h.set_launch(**launch)
            dev = _lib.to_device(parts, "fp32")
            ws = torch.zeros(64, dtype=torch.int32, device="cuda")
            _lib.ap_gather_push_batched(h.h, dev, off, g, -3.0, 0.02, 1, "fp32", None, ws)
            assert h.status() == 0
            assert 0 < int(ws[0]) - n_sets * (-(-per_set // tile)) <= 64 * sms
