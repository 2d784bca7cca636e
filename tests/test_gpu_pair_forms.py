"""The paired step kernels (lb_pair.cuh) at the edges of their tiles, in the forms that test_gpu_pair.py leaves
out: noise at the local density, the eigen factor (both off-diagonal entries of the (4,9) block in use) and
the double well, against the FP64 oracle.  Tolerance: the parity tests' 1e-5."""
import numpy as np
import pytest

import oracle
import paper_1009_0254_gb300 as lbf
from oracle import theory as th
from paper_1009_0254_gb300 import synth

pytestmark = pytest.mark.gpu
SIZES = [(63, 7), (64, 8), (65, 9), (66, 16), (70, 17), (33, 15), (31, 33), (127, 5), (130, 8), (9, 64), (5, 3), (2, 2)]
WELL = th.DoubleWell(0.04, 0.5, 1.0)
FORMS = {"local": (lbf.LB_NOISE_LW_LOCAL, False, None), "lw eigen": (lbf.LB_NOISE_LW, True, None),
         "rs eigen": (lbf.LB_NOISE_FULL_RS, True, None), "well off": (lbf.LB_NOISE_OFF, False, WELL),
         "well lw": (lbf.LB_NOISE_LW, False, WELL), "well local": (lbf.LB_NOISE_LW_LOCAL, False, WELL)}


@pytest.mark.parametrize("kernel", [None, "tma"])
@pytest.mark.parametrize("form", sorted(FORMS))
def test_form_at_tile_edges(form, kernel, monkeypatch):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1009_0254_gb300 import build
    build.build()
    mode, eigen, eos = FORMS[form]
    params = (1e-4, 0.03, 0.8, 1.1, 0.9)
    if kernel:
        monkeypatch.setenv("LBFLUCT_STEP_KERNEL", kernel)
    else:
        monkeypatch.delenv("LBFLUCT_STEP_KERNEL", raising=False)
    # without a fixed kernel the sizes that take many steps a launch, odd heights among them
    for k, (nx, ny) in enumerate(SIZES if kernel else [(32, 33), (66, 47), (128, 101)]):
        g = lbf.Lattice(nx, ny, seed=70 + k)
        o = oracle.Lattice(nx, ny, seed=70 + k, eos=eos)
        if eos:
            g.set_eos(lbf.LB_EOS_DOUBLE_WELL, eos.beta, eos.rhoV, eos.rhoL)
        if eigen:
            g.set_noise_factor(lbf.LB_FACTOR_EIGEN)
        g.set_params(*params, mode)
        o.set_params(*params, mode, factor="eigen" if eigen else None)
        o.f = o.f * (1.0 + synth.gaussian_field((9, ny, nx), seed=70 + k, scale=0.01))
        g.set_populations(o.f, t=0)
        g.step(10)
        o.step(10)
        assert np.abs(g.populations() - o.f).max() <= 1e-5, (nx, ny)
        g.close()
