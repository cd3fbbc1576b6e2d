"""What the launch-shape tuner works on: FP64 lines of zeros leave the integer
stages at once, so its inputs must not be zeros; and a tangent that is in
place must stay as it is."""

import numpy as np
import pytest

from gpu_helpers import gff, torch_cuda
from rve_inputs import polycrystal

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(4, 4, 4), (10, 36, 50), (48, 48, 48)])
def test_tuner_reads_no_zeros_and_keeps_a_valid_tangent(shape):
    torch = torch_cuda()
    g = gff()
    N = int(np.prod(shape))
    ms = polycrystal(shape, 3, 5)
    # a handle whose tangent is not set lends its place to the tuner
    h = g.create_rve(ms, {0: g.make_material(g.GFF_MAT_SVK_CUBIC)}, g.make_options())
    try:
        g.gff_set_field(h, g.GFF_FIELD_K, np.zeros((81, N)))
        g.gff_set_microstructure(h, ms.grain_id.reshape(-1), ms.ngrains, ms.quat, ms.phase)  # (the tangent is none now)
        g.gff_autotune(h)
        K = g.gff_get_field(h, g.GFF_FIELD_K, N)
        assert np.isfinite(K).all() and (np.abs(K) >= 1).all() and (np.abs(K) < 2).all()
        assert (K < 0).any() and (K > 0).any()
        with pytest.raises(g.GffError):  # and there is no tangent still
            X = torch.zeros(9, N, dtype=torch.float64, device="cuda")
            g.gff_apply_operator(h, g.GFF_PREC_FP64, None, X, torch.empty_like(X))
        # a valid one is read only
        g.gff_set_field(h, g.GFF_FIELD_F, np.repeat(np.eye(3).reshape(9, 1), N, axis=1))
        g.gff_constitutive(h, 1.0)
        K = g.gff_get_field(h, g.GFF_FIELD_K, N)
        g.gff_autotune(h)
        assert np.array_equal(K, g.gff_get_field(h, g.GFF_FIELD_K, N))
    finally:
        torch.cuda.synchronize()
        g.gff_destroy(h)
