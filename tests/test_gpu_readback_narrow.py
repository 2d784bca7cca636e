"""Device read-back of narrow three-dimensional lattices, whose rows share blocks of 128 threads: widths at and
beside the powers of two that set the block's shape, heights at and beside its rows, against the host read-back
bit for bit."""
import numpy as np
import pytest

import paper_1009_0254_gb300 as lbf

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("q", [19, 27])
@pytest.mark.parametrize("precision", [lbf.LB_FP32, lbf.LB_FP64])
def test_narrow_lattices(q, precision):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1009_0254_gb300 import build
    build.build()
    # (width, block's columns): the rows of a block are 8 * 128 / columns
    for nx, cols in [(2, 2), (3, 4), (4, 4), (5, 8), (17, 32), (32, 32), (64, 64), (65, 128), (129, 128)]:
        for ny in {8 * 128 // cols, 8 * 128 // cols + 1, 7}:
            g = lbf.Lattice3(nx, ny, 2, lattice=q, seed=3, precision=precision)
            g.set_params(1e-4, 0.01, 0.8, 1.1, 0.9, lbf.LB_NOISE_LW)
            g.step(2)
            f = torch.full((q, 2, ny, nx), float("nan"), dtype=torch.float64, device="cuda")
            torch.cuda.synchronize()
            lbf.lb3_get_populations(g.ctx, f, lbf.LB_DEVICE)
            assert np.array_equal(f.cpu().numpy(), g.populations()), (nx, ny)
            g.close()
