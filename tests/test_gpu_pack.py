"""The per-cell coefficient copy of a grid (AP_PACK_CELLS) at the sizes where
its kernel can go wrong (one cell, rows that end inside a group of 32 cells,
a last group of one cell, several groups per warp), against the same
differences in double.

Tolerance: each coefficient is rounded once from a sum good to 2^-45 of the
largest corner, so it lies within half a unit in the last place (2^-24 of the
coefficient) plus 2^-45 of the largest corner of the exact value."""
import numpy as np
import pytest


def _reference(f):
    d = f.astype(np.float64)
    c = {(i, j, k): d[:, k:d.shape[1] - 1 + k, j:d.shape[2] - 1 + j, i:d.shape[3] - 1 + i]
         for i in (0, 1) for j in (0, 1) for k in (0, 1)}
    with np.errstate(invalid="ignore", over="ignore"):
        a1, a2, a3 = c[1, 0, 0] - c[0, 0, 0], c[0, 1, 0] - c[0, 0, 0], c[0, 0, 1] - c[0, 0, 0]
        a4 = (c[1, 1, 0] - c[1, 0, 0]) - a2
        a5 = (c[0, 1, 1] - c[0, 1, 0]) - a3
        a6 = (c[1, 0, 1] - c[1, 0, 0]) - a3
        a7 = ((c[1, 1, 1] - c[1, 1, 0]) - (c[1, 0, 1] - c[1, 0, 0])) - a5
    return np.stack([c[0, 0, 0], a1, a2, a3, a4, a5, a6, a7], axis=-1)  # [6, z, y, x, 8]


def _packed(f):
    import torch
    from paper_2307_04843_gb300 import _lib
    g = _lib.pack_grid((torch.as_tensor(f).cuda(), (0, 0, 0), (1, 1, 1)), layout="cells")
    nz, ny, nx = (v - 1 for v in f.shape[1:])
    p = g[3].cpu().numpy().reshape(nz, ny, nx, 3, 8, 2)
    return np.moveaxis(p, (3, 5), (0, 1)).reshape(6, nz, ny, nx, 8)


@pytest.mark.gpu
@pytest.mark.parametrize("shape", [(2, 2, 2), (2, 2, 34), (3, 5, 33), (4, 12, 4), (9, 33, 34), (70, 65, 130)])
def test_cell_coefficients_match_double_differences(shape):
    rng = np.random.default_rng(sum(shape))
    # magnitudes over many decades, so that the differences cancel and spread
    f = (rng.standard_normal((6,) + shape) * 10.0 ** rng.uniform(-8, 8, (6,) + shape)).astype(np.float32)
    ref = _reference(f)
    big = np.max(np.abs(ref[..., :1]))
    err = np.abs(_packed(f).astype(np.float64) - ref)
    assert np.all(err <= 2.0 ** -24 * np.abs(ref) + 2.0 ** -45 * big)


@pytest.mark.gpu
def test_cell_coefficients_of_huge_and_nonfinite_corners():
    rng = np.random.default_rng(3)
    f = (rng.choice([-3.0e38, 3.0e38, 1.0], (6, 5, 6, 37))).astype(np.float32)
    f[0, 2, 3, 4], f[1, 1, 1, 1], f[2, 4, 5, 36] = np.inf, np.nan, -np.inf
    ref, out = _reference(f), _packed(f)
    with np.errstate(over="ignore"):
        ref32 = ref.astype(np.float32)
    fin = np.isfinite(ref32)
    # infinities and NaN as the double differences give them (a NaN equals a NaN)
    np.testing.assert_array_equal(out[~fin], ref32[~fin])
    # the double differences drop a corner of 1 beside one of 3e38; the tolerance above covers that
    err = np.abs(out[fin].astype(np.float64) - ref[fin])
    assert np.all(err <= 2.0 ** -24 * np.abs(ref[fin]) + 2.0 ** -45 * 3.0e38)


@pytest.mark.gpu
@pytest.mark.parametrize("shape", [(2, 2, 2), (3, 5, 33), (20, 33, 34)])
@pytest.mark.parametrize("form", ["wide", "near", "linear"])
def test_cell_coefficients_of_cancelling_corners(shape, form):
    """Differences that cancel to their last bits, each cell against exact
    rational differences, on its own scale: half a unit in the last place, a
    fiftieth of that, and 2^-60 of the cell's largest corner.  Wide: corners of 1 beside ones of 1e-8, so that first
    differences have low parts of 24 bits; near: corners that agree to 1e-4;
    linear: fields whose second differences are rounding alone."""
    from fractions import Fraction
    rng = np.random.default_rng(sum(shape))
    if form == "wide":
        f = np.where(np.arange(shape[2]) % 2 == 0, 1.0, 1e-8 * (1.0 + rng.random((6,) + shape)))
    elif form == "near":
        f = 1.0 + 1e-4 * rng.standard_normal((6,) + shape)
    else:
        z, y, x = np.meshgrid(*(np.arange(n) for n in shape), indexing="ij")
        f = np.stack([1.0 + 0.1 * (c + 1) * x - 0.37 * y + 1e-3 * z for c in range(6)])
    f = f.astype(np.float32)
    out = _packed(f)
    nz, ny, nx = (v - 1 for v in shape)
    for _ in range(400):
        c, k, j, i = (int(rng.integers(0, n)) for n in (6, nz, ny, nx))
        v = {(x, y, z): Fraction(float(f[c, k + z, j + y, i + x])) for x in (0, 1) for y in (0, 1) for z in (0, 1)}
        a = [v[0, 0, 0], v[1, 0, 0] - v[0, 0, 0], v[0, 1, 0] - v[0, 0, 0], v[0, 0, 1] - v[0, 0, 0]]
        a.append(v[1, 1, 0] - v[1, 0, 0] - a[2])
        a.append(v[0, 1, 1] - v[0, 1, 0] - a[3])
        a.append(v[1, 0, 1] - v[1, 0, 0] - a[3])
        a.append(v[1, 1, 1] - v[1, 1, 0] - v[1, 0, 1] + v[1, 0, 0] - a[5])
        big = max(abs(x) for x in v.values())
        for p, want in enumerate(a):
            got = Fraction(float(out[c, k, j, i, p]))
            assert abs(got - want) <= abs(want) * Fraction(51, 50) / 2 ** 24 + big / 2 ** 60, (c, k, j, i, p)
