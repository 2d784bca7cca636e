"""The binned spectra of one sample add up to the variances of their fields (Parseval, k = 0 left out) for
both CTA sizes of the binning kernel and lattices at the line between them.  Tolerance: 2 x 24 FP32 butterfly
levels at half an ulp (6e-8) each, 3e-6, and the binning's FP32 runs of 128 terms as much again: 1e-5."""
import numpy as np
import pytest

import paper_1009_0254_gb300 as lbf

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,nbins", [(2, 2, 8), (64, 32, 16), (1024, 1024, 512), (2048, 1024, 4096),
                                         (4096, 256, 64), (2048, 2048, 1024)])
def test_bins_add_up_to_the_variance(nx, ny, nbins):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1009_0254_gb300 import build
    build.build()
    g = lbf.Lattice(nx, ny, seed=4)
    g.set_params(1e-4, 0.01, 0.8, 1.1, 0.9, lbf.LB_NOISE_LW)
    g.set_sampling(9, nbins)
    g.step(9)
    S, jl, jt, counts, nsamples = g.structure_factor()
    assert nsamples == 1 and counts.sum() == nx * ny - 1
    m, _ = g.moments()
    rho, jx, jy = m[0] - m[0].mean(), m[1] - m[1].mean(), m[2] - m[2].mean()
    assert np.isclose(np.nansum(S * counts), (rho * rho).sum(), rtol=1e-5, atol=0)
    assert np.isclose(np.nansum((jl + jt) * counts), (jx * jx + jy * jy).sum(), rtol=1e-5, atol=0)
