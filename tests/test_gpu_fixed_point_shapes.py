"""FP64 launch shapes whose kernels differ (one block per strip or the TMA z
pass, one block per plane or the streamed inverse pass, the columns and threads
of each): the same bits whichever is set, on axes of two to four stages."""

import numpy as np
import pytest

from gpu_helpers import gff, rel_l2, torch_cuda, voxel_K_oracle
from oracle import spectral as sp
from rve_inputs import polycrystal, standard_normal

pytestmark = pytest.mark.gpu

# fwd threads, z columns, z threads, inv threads, inv blocks (> 0: streamed), TMA z blocks; few blocks, so that each
# walks several planes or strips and the last ones are left over
TILES = [(512, 8, 256, 512, 0, 0), (256, 4, 128, 256, 0, 0), (256, 16, 128, 512, 7, 0), (512, 32, 256, 256, 5, 0),
         (512, 8, 192, 512, 0, 7), (256, 8, 512, 256, 9, 11), (512, 16, 256, 512, 0, 5), (512, 16, 384, 512, 3, 13)]


@pytest.mark.parametrize("shape", [(100, 54, 36), (36, 10, 108), (54, 90, 20)])
def test_shapes_give_the_same_bits(shape):
    torch = torch_cuda()
    g = gff()
    nz, ny, nx = shape
    ms = polycrystal(shape, 6, 21)
    h = g.create_rve(ms, {0: g.make_material(g.GFF_MAT_SVK_CUBIC)}, g.make_options())
    mask = np.array([0, 1, 1, 1, 1, 1, 1, 0, 1], dtype=np.uint8)
    x = standard_normal(17, 9 * nz * ny * nx).reshape(9, -1)
    try:
        g.gff_constitutive(h, 1.0)
        X = torch.from_numpy(x).cuda()
        first = None
        for t in TILES:
            g.gff_set_tiles(h, t, TILES[0])
            outs = []
            for m in (None, mask):
                for call in (g.gff_apply_operator, g.gff_project):
                    Y = torch.full_like(X, 7.0)
                    call(h, g.GFF_PREC_FP64, m, X, Y)
                    g.gff_sync(h)
                    outs.append(Y.cpu().numpy())
            first = first or outs
            assert all(np.array_equal(a, b) for a, b in zip(outs, first)), t
    finally:
        g.gff_destroy(h)
    _, K = voxel_K_oracle(ms, np.tile(np.eye(3).reshape(3, 3, 1, 1, 1), (1, 1) + shape))
    assert rel_l2(first[0], sp.GK(K, x.reshape(3, 3, nz, ny, nx), ms.L, sp.KIND_CONTINUOUS)) <= 1e-12
