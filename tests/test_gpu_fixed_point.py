"""FP64 transforms in fixed point (csrc/fixed_bfly.cuh): every axis length's
plan, values spread over the exponent range, and the lines the integers do
not take (near overflow or underflow, infinities, NaN, zeros).

Tolerance of the parity tests, 4e-15 relative L2: each of the six line
transforms and the projection's four operations round to 53 bits (2^-53 =
1.1e-16 each, so below 1.2e-15), and the oracle's own FFT and projection
carry as much again, twice."""

import numpy as np
import pytest

from gpu_helpers import gff, rel_l2, torch_cuda
from oracle import spectral as sp
from rve_inputs import standard_normal

pytestmark = pytest.mark.gpu

TOL = 4e-15
AXES = [4, 6, 8, 10, 12, 16, 18, 20, 24, 30, 32, 36, 40, 48, 50, 54, 60, 64, 72, 80, 90, 96, 100, 108, 120, 128]


def _project(shape, x, mask=None, kind=0):
    torch = torch_cuda()
    g = gff()
    nz, ny, nx = shape
    h = g.gff_create(g.make_grid(nx, ny, nz), g.make_options(projection=kind))
    try:
        X = torch.from_numpy(np.ascontiguousarray(x.reshape(9, -1))).cuda()
        Y = torch.full_like(X, 7.0)
        g.gff_project(h, g.GFF_PREC_FP64, mask, X, Y)
        g.gff_sync(h)
        return Y.cpu().numpy().reshape(3, 3, nz, ny, nx)
    finally:
        g.gff_destroy(h)


def _noise(seed, shape):
    nz, ny, nx = shape
    return standard_normal(seed, 9 * nz * ny * nx).reshape(3, 3, nz, ny, nx)


@pytest.mark.parametrize("n", AXES)
def test_every_axis_length(n):
    for shape in ((n, 6, 8), (6, n, 4), (4, 8, n)):
        x = _noise(n, shape)
        assert rel_l2(_project(shape, x), sp.G(x, (1.0, 1.0, 1.0), sp.KIND_CONTINUOUS, None)) <= TOL, shape


@pytest.mark.parametrize("kind", ["mean", "spike", "decades", "mode"])
@pytest.mark.parametrize("shape", [(16, 32, 64), (10, 36, 20)])
def test_uneven_values(kind, shape):
    x = _noise(3, shape)
    if kind == "mean":  # a large mean stress: the fluctuations are what is left after it
        x += 1e3
    elif kind == "spike":
        x *= 1e-9
        x[:, :, 1, 2, 3] = 1.0
    elif kind == "decades":
        x *= 10.0 ** (-12.0 * (np.arange(x.size) % 13) / 12.0).reshape(x.shape)
    else:
        x = np.cos(2 * np.pi * 3 * np.arange(shape[2]) / shape[2] + np.zeros(x.shape))
    ref = sp.G(x, (1.0, 1.0, 1.0), sp.KIND_CONTINUOUS, None)
    # the rounding of what the mean leaves behind is relative to x
    assert np.linalg.norm(_project(shape, x) - ref) <= TOL * np.linalg.norm(x)


@pytest.mark.parametrize("e", [-900, 900])
def test_powers_of_two_scale_exactly(e):
    """Alignment is relative to each line's largest exponent: within the integers' range a power of two
    passes through every rounding."""
    shape = (12, 16, 20)
    x = _noise(5, shape)
    assert np.array_equal(_project(shape, np.ldexp(x, e)), np.ldexp(_project(shape, x), e))


@pytest.mark.parametrize("e", [-1000, 1005])
def test_ends_of_the_range_run_in_fp64(e):
    shape = (8, 8, 8)
    x = _noise(6, shape)
    y = np.ldexp(_project(shape, np.ldexp(x, e)), -e)
    assert rel_l2(y, sp.G(x, (1.0, 1.0, 1.0), sp.KIND_CONTINUOUS, None)) <= 1e-12


@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
def test_non_finite_values_reach_their_tensor_row_and_no_other(bad):
    shape = (8, 16, 12)
    x = _noise(7, shape)
    y0 = _project(shape, x)
    x[1, 2, 3, 4, 5] = bad
    y = _project(shape, x)
    assert not np.isfinite(y[1]).any()
    assert np.array_equal(y[0], y0[0]) and np.array_equal(y[2], y0[2])


def test_zero_lines_and_rows_stay_zero():
    shape = (8, 16, 12)
    x = np.zeros((3, 3) + shape)
    x[0, 0] = np.cos(2 * np.pi * np.arange(12) / 12)  # one mode along x: q = (q_x, 0, 0)
    y = _project(shape, x)
    assert rel_l2(y[0, 0], x[0, 0]) <= TOL
    assert np.abs(y[0, 1:]).max() <= 1e-15 and not y[1:].any()
