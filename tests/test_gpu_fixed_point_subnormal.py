"""Fields below 2^-1042, where the high word of an FP64 value is zero: such
lines are not taken for lines of zeros, which the transforms skip."""

import numpy as np
import pytest

from gpu_helpers import gff, rel_l2, torch_cuda
from oracle import spectral as sp
from rve_inputs import standard_normal

pytestmark = pytest.mark.gpu


def project(shape, x):
    torch = torch_cuda()
    g = gff()
    nz, ny, nx = shape
    h = g.gff_create(g.make_grid(nx, ny, nz), g.make_options())
    try:
        X = torch.from_numpy(np.ascontiguousarray(x.reshape(9, -1))).cuda()
        Y = torch.full_like(X, 7.0)
        g.gff_project(h, g.GFF_PREC_FP64, None, X, Y)
        g.gff_sync(h)
        return Y.cpu().numpy().reshape(3, 3, nz, ny, nx)
    finally:
        g.gff_destroy(h)


@pytest.mark.parametrize("shape", [(8, 8, 8), (6, 10, 36)])
def test_subnormal_fields_are_projected(shape):
    """2^-1052 times a normal field carries 22 bits above the last one, 2^-1074.  The spectrum over N passes a few
    roundings to that unit u: at most 8 sqrt(N) u rms per voxel after the inverse (sums of N values of half a
    unit), 8 sqrt(N) 2^-22 / 0.57 of the projection."""
    nz, ny, nx = shape
    x = standard_normal(9, 9 * nz * ny * nx).reshape(3, 3, nz, ny, nx)
    y = project(shape, np.ldexp(x, -1052))
    ref = sp.G(x, (1.0, 1.0, 1.0), sp.KIND_CONTINUOUS, None)
    assert rel_l2(np.ldexp(y, 1052), ref) <= 8 * np.sqrt(nz * ny * nx) * 2.0 ** -22 / 0.57


def test_subnormal_components_beside_zero_ones():
    """One tensor row of subnormals, the others zero: the zeros stay, the row is projected."""
    shape = (8, 8, 8)
    x = np.zeros((3, 3) + shape)
    x[1] = standard_normal(10, 3 * 512).reshape((3,) + shape)
    y = np.ldexp(project(shape, np.ldexp(x, -1052)), 1052)
    assert not y[0].any() and not y[2].any()
    assert rel_l2(y[1], sp.G(x, (1.0, 1.0, 1.0), sp.KIND_CONTINUOUS, None)[1]) <= 8 * np.sqrt(512) * 2.0 ** -22 / 0.57
