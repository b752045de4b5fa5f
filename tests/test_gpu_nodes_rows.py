"""Grid nodes: the ways of giving rows to warps, on both sides of the lines
between them.

Plane waves: rows in runs or in turn, by the row's length, the node type and the
accumulation.  The field of a row depends on its z index alone, so every value
is the one of a short-row grid, bit for bit."""
import math

import pytest

L = 2 * math.pi


@pytest.mark.gpu
@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("dtype", ["float32", "float64"])
@pytest.mark.parametrize("nx", [191, 192, 193, 200, 256])
def test_plane_rows_are_those_of_a_short_row(nx, dtype, precision):
    import torch
    from paper_2307_04843_gb300 import _lib
    dt = getattr(torch, dtype)
    ny, nz = 3, 700
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
