"""Error of the FP64 transforms on 64-bit integers (csrc/fixed_bfly.cuh) against
extended precision, on fields with a mean of twice their fluctuation, for
plans of two to four stages.

The operator with K = identity runs them without another rounding (K:x is then
x, bit for bit).  Bound: a value passes twelve roundings to 53 bits on its way
(row split, y, column split, packing, z, two in the projection, z, unpacking,
y, x and the division by N), each 4.7e-17 rms of a value with a logarithmically
spread mantissa, together 1.63e-16.  The integers between them are to stay
below these: twice the sum bounds the whole."""

import numpy as np
import pytest
import scipy.fft

from gpu_helpers import gff, torch_cuda
from rve_inputs import polycrystal, standard_normal

pytestmark = pytest.mark.gpu

BOUND = 2 * np.sqrt(12.0) * 4.7e-17
# (nz, ny, nx)
SHAPES = [(16, 16, 16), (100, 6, 90), (50, 54, 20), (108, 10, 36), (30, 120, 8), (60, 18, 50), (64, 64, 32), (8, 96, 72)]


def field(shape):
    nz, ny, nx = shape
    x = standard_normal(31, 9 * nz * ny * nx).reshape(9, -1)
    return x + 2.0 * standard_normal(32, 9).reshape(9, 1)


def identity_handle(g, shape):
    """A handle of this grid whose tangent is the identity."""
    nz, ny, nx = shape
    ms = polycrystal(shape, 2, 3)
    h = g.create_rve(ms, {0: g.make_material(g.GFF_MAT_SVK_CUBIC)}, g.make_options())
    g.gff_set_field(h, g.GFF_FIELD_K, np.repeat(np.eye(9).reshape(81, 1), nz * ny * nx, axis=1))
    return h


def extended_projection(x, shape):
    """G(x) of a (9, N) field over the unit cube in extended precision."""
    nz, ny, nx = shape
    X = scipy.fft.fftn(x.astype(np.longdouble).reshape(3, 3, nz, ny, nx), axes=(2, 3, 4))
    kap = [np.array([k if 2 * k < n else k - n for k in range(n)], dtype=np.longdouble) for n in (nx, ny, nz)]
    Q = [kap[0].reshape(1, 1, nx), kap[1].reshape(1, ny, 1), kap[2].reshape(nz, 1, 1)]
    keep = (2 * Q[0] != -nx) & (2 * Q[1] != -ny) & (2 * Q[2] != -nz)
    keep[0, 0, 0] = False
    q2 = Q[0] ** 2 + Q[1] ** 2 + Q[2] ** 2
    q2[0, 0, 0] = 1
    Y = np.empty_like(X)
    for i in range(3):
        t = np.where(keep, sum(X[i, j] * Q[j] for j in range(3)) / q2, 0)
        for j in range(3):
            Y[i, j] = t * Q[j]
    return scipy.fft.ifftn(Y, axes=(2, 3, 4)).real.reshape(9, -1)


@pytest.mark.skipif(np.finfo(np.longdouble).eps > 1e-18, reason="needs an extended long double")
@pytest.mark.parametrize("shape", SHAPES)
def test_error_against_extended_precision(shape):
    torch = torch_cuda()
    g = gff()
    x = field(shape)
    h = identity_handle(g, shape)
    try:
        X = torch.from_numpy(x).cuda()
        Y = torch.empty_like(X)
        g.gff_apply_operator(h, g.GFF_PREC_FP64, None, X, Y)
        g.gff_sync(h)
        y = Y.cpu().numpy()
    finally:
        g.gff_destroy(h)
    ref = extended_projection(x, shape)
    d = y.astype(np.longdouble) - ref
    assert float(np.sqrt((d * d).sum() / (ref * ref).sum())) <= BOUND


@pytest.mark.parametrize("tuned", [False, True])
@pytest.mark.parametrize("shape", SHAPES + [(64, 8, 8), (16, 64, 64), (40, 36, 48)])
def test_projections_take_the_arithmetic_of_operators(shape, tuned):
    """One arithmetic at every size and with every launch shape: with K = identity
    the operator is the bare projection, bit for bit."""
    torch = torch_cuda()
    g = gff()
    h = identity_handle(g, shape)
    try:
        if tuned:
            g.gff_autotune(h)
        X = torch.from_numpy(field(shape)).cuda()
        Y, Z = torch.empty_like(X), torch.empty_like(X)
        for mask in (None, [0, 1, 1, 1, 1, 1, 1, 0, 1]):
            m = None if mask is None else np.array(mask, dtype=np.uint8)
            g.gff_apply_operator(h, g.GFF_PREC_FP64, m, X, Y)
            g.gff_project(h, g.GFF_PREC_FP64, m, X, Z)
            g.gff_sync(h)
            assert torch.equal(Y, Z)
    finally:
        torch.cuda.synchronize()
        g.gff_destroy(h)
