"""Grid nodes: the ways of giving rows to warps, on both sides of the lines
between them.

Gaussian beams: slabs or rows, by the row's length, ny, the node type, the
alignment and the accumulation; against the oracle to 4e-6 a0, as the slab tests
hold.

Plane waves: rows in runs or in turn, by the row's length, the node type and the
accumulation.  The field of a row depends on its z index alone, so every value
is the one of a short-row grid, bit for bit."""
import math

import pytest

from test_gpu_nodes_slab import _case

L = 2 * math.pi


@pytest.mark.gpu
@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("dtype", ["float32", "float64"])
@pytest.mark.parametrize("nx,ny", [(191, 3), (192, 3), (193, 30), (200, 60), (256, 30), (289, 60), (641, 3)])
def test_plane_rows_are_those_of_a_short_row(nx, ny, dtype, precision):
    import torch
    from paper_2307_04843_gb300 import _lib
    dt = getattr(torch, dtype)
    nz = 700
    lo, d = [0.1, -0.3, -8.0], [0.2, 0.3, 0.05]
    with _lib.Handle(dict(kind="plane", pol="cp", env="gauss", env_len=12.0, a0=1.3, phase0=0.4)) as h:
        ref = torch.empty((6, nz, 1, 32), dtype=dt, device="cuda")
        h.eval_nodes(list(ref), lo, d, 0.7, precision=precision)
        f = torch.full((6, nz, ny, nx), 7.0, dtype=dt, device="cuda")
        h.eval_nodes(list(f), lo, d, 0.7, precision=precision)
        assert torch.equal(f, ref[..., :1].expand_as(f))
        acc, ref_acc = torch.full_like(f, 0.25), torch.full_like(ref, 0.25)
        h.eval_nodes(list(acc), lo, d, 0.7, accumulate=True, precision=precision)
        h.eval_nodes(list(ref_acc), lo, d, 0.7, accumulate=True, precision=precision)
        assert torch.equal(acc, ref_acc[..., :1].expand_as(acc))


# (nz, ny, nx) on both sides of each line, full and ragged blocks of 128 columns
STORED = [(3, 5, 64), (3, 6, 64), (2, 70, 36), (3, 2, 128), (3, 3, 128), (2, 33, 100), (2, 37, 200), (2, 3, 160),
          (2, 4, 160), (2, 40, 264), (2, 40, 260), (2, 11, 33), (2, 12, 33), (2, 40, 127), (2, 40, 129)]


@pytest.mark.gpu
@pytest.mark.parametrize("shape", STORED)
@pytest.mark.parametrize("kind", ["gauss", "flying_cf"])
def test_gaussian_nodes_stored_in_float(kind, shape):
    import torch
    _case(kind, "cp", shape, torch.float32, False)
    _case(kind, "y", shape, torch.float32, False, offset=1)


@pytest.mark.gpu
@pytest.mark.parametrize("shape", [(3, 2, 64), (3, 3, 64), (2, 40, 36), (3, 1, 128), (2, 37, 260), (2, 5, 33)])
def test_gaussian_nodes_summed_in_float(shape):
    import torch
    for offset in (0, 1):
        _case("gauss", "cm", shape, torch.float32, True, offset)


@pytest.mark.gpu
@pytest.mark.parametrize("shape", [(3, 2, 128), (3, 3, 128), (2, 37, 120), (2, 40, 64), (2, 33, 250), (2, 40, 300)])
@pytest.mark.parametrize("accumulate", [False, True])
def test_gaussian_nodes_in_double(shape, accumulate):
    import torch
    _case("gauss", "cp", shape, torch.float64, accumulate)
