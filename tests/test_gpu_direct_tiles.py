"""Lattices whose last tile column is stored by the threads (rows that end inside a 16-byte unit of the store
box) and so high that a CTA takes several tiles of the step kernel, boxed ones before direct ones: every
launch of the TMA-staged kernel leaves its whole state to the next, against the plain kernel.

Tolerance: both kernels sum in FP32; the bound of the parity tests, 1e-5."""
import numpy as np
import pytest

import paper_1009_0254_gb300 as lbf
from paper_1009_0254_gb300 import synth

pytestmark = pytest.mark.gpu


# tiles a row: 3 of 64 columns, 5 of 32; thousands of tiles for some 600 CTAs
@pytest.mark.parametrize("nx,ny,mode", [(130, 16000, lbf.LB_NOISE_LW), (129, 16001, lbf.LB_NOISE_OFF),
                                        (131, 16000, lbf.LB_NOISE_FULL_RS), (190, 15999, lbf.LB_NOISE_LW_LOCAL)])
def test_several_tiles_a_cta(nx, ny, mode, monkeypatch):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1009_0254_gb300 import build
    build.build()
    f0, out = None, []
    for kernel in ("tma", "simple"):
        monkeypatch.setenv("LBFLUCT_STEP_KERNEL", kernel)
        g = lbf.Lattice(nx, ny, seed=21)
        g.set_params(1e-4, 0.02, 0.8, 1.1, 0.9, mode)
        if f0 is None:
            f0 = g.populations()
            f0 *= 1.0 + synth.uniform(-0.02, 0.02, f0.size, seed=6).reshape(f0.shape)
        g.set_populations(f0)
        g.step(6)
        out.append(g.populations())
        g.close()
    assert np.abs(out[0] - out[1]).max() <= 1e-5
    assert np.abs(out[0] - f0).max() > 1e-4
