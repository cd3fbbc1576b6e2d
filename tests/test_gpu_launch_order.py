"""The passes of one apply overlap their start with the end of the pass before
(programmatic dependent launch).  Applies queued back to back on one stream,
on the handle's one spectrum and with other kernels between them, give bit for
bit what they give with the GPU idle in between; so does a captured sequence,
which is launched in the plain order."""

import numpy as np
import pytest

from gpu_helpers import gff, torch_cuda
from rve_inputs import polycrystal

pytestmark = pytest.mark.gpu

# the forward pass starts early up to 2^17 voxels: below, at and above; odd plans; one block per SM and several waves
SHAPES = [(4, 4, 4), (16, 16, 16), (10, 36, 50), (32, 64, 64), (36, 64, 64), (64, 64, 64)]


@pytest.mark.parametrize("tuned", [False, True])
@pytest.mark.parametrize("f64", [True, False])
@pytest.mark.parametrize("shape", SHAPES)
def test_queued_applies_equal_separate_ones(shape, f64, tuned):
    torch = torch_cuda()
    g = gff()
    ms = polycrystal(shape, 5, 3)
    h = g.create_rve(ms, {0: g.make_material(g.GFF_MAT_SVK_CUBIC)}, g.make_options())
    try:
        g.gff_set_field(h, g.GFF_FIELD_F, np.repeat(np.eye(3).reshape(9, 1), ms.n_voxels, axis=1))
        g.gff_constitutive(h, 1.0)
        if tuned:
            g.gff_autotune(h)
        prec = g.GFF_PREC_FP64 if f64 else g.GFF_PREC_MIXED
        gen = torch.Generator(device="cuda").manual_seed(5)
        x0 = torch.randn((2, 9, ms.n_voxels), generator=gen, device="cuda", dtype=torch.float64 if f64 else torch.float32)

        def sequence(pause):
            x, out = x0.clone(), []
            for _ in range(4):
                y = torch.empty_like(x)
                for i in range(2):  # the second apply reuses the spectrum the first still reads
                    g.gff_apply_operator(h, prec, None, x[i], y[i])
                    pause()
                x.copy_(x0).add_(y, alpha=1e-11)
                pause()
                out.append(y)
            return out

        want = sequence(torch.cuda.synchronize)
        for _ in range(3):
            got = sequence(lambda: None)
            torch.cuda.synchronize()
            assert all(torch.equal(a, b) for a, b in zip(got, want))

        s = torch.cuda.Stream()
        graph = torch.cuda.CUDAGraph()
        y = torch.empty_like(x0)
        g.gff_set_stream(h, s)
        torch.cuda.synchronize()
        with torch.cuda.graph(graph, stream=s):
            for i in range(2):
                g.gff_apply_operator(h, prec, None, x0[i], y[i])
        for _ in range(2):
            y.zero_()
            graph.replay()
            torch.cuda.synchronize()
            assert torch.equal(y, want[0])
    finally:
        torch.cuda.synchronize()
        g.gff_destroy(h)
