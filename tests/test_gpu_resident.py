"""Many steps of a small lattice in one launch (lb_step_resident.cu) against a launch per step: the
arithmetic and its order are the same, so the populations are equal bit for bit, on the smallest and the
largest lattices that it takes, with rows that the 16 bands share unevenly and every variant."""
import numpy as np
import pytest

import paper_1009_0254_gb300 as lbf
from paper_1009_0254_gb300 import synth

pytestmark = pytest.mark.gpu
SIZES = [(32, 32), (34, 33), (64, 47), (66, 64), (96, 50), (126, 127), (128, 128)]
RUNS = [(lbf.LB_NOISE_OFF, lbf.LB_FP32, False), (lbf.LB_NOISE_LW, lbf.LB_FP32, False),
        (lbf.LB_NOISE_LW_LOCAL, lbf.LB_FP32, False), (lbf.LB_NOISE_LW, lbf.LB_FP32, True),
        (lbf.LB_NOISE_LW_LOCAL, lbf.LB_FP32, True), (lbf.LB_NOISE_OFF, lbf.LB_FP32, True),
        (lbf.LB_NOISE_OFF, lbf.LB_FP16DEV, False), (lbf.LB_NOISE_LW, lbf.LB_FP16DEV, False),
        (lbf.LB_NOISE_LW_LOCAL, lbf.LB_FP16DEV, False)]


@pytest.mark.parametrize("mode,precision,poly", RUNS)
@pytest.mark.parametrize("nx,ny", SIZES)
def test_one_launch_equals_a_launch_per_step(nx, ny, mode, precision, poly, monkeypatch):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1009_0254_gb300 import build
    build.build()
    f0 = None
    out = []
    for kernel in (None, "tma"):
        if kernel:
            monkeypatch.setenv("LBFLUCT_STEP_KERNEL", kernel)
        else:
            monkeypatch.delenv("LBFLUCT_STEP_KERNEL", raising=False)
        g = lbf.Lattice(nx, ny, seed=7, precision=precision)
        if poly:
            g.set_eos(lbf.LB_EOS_DOUBLE_WELL, 0.04, 0.5, 1.0)
        g.set_params(1e-4, 0.01, 0.8, 1.1, 0.9, mode)
        if f0 is None:
            f0 = g.populations() * (1.0 + synth.gaussian_field((9, ny, nx), seed=3, scale=0.01))
        g.set_populations(f0)
        got = []
        for n in (4, 1, 8, 30):
            g.step(n)
            got.append(g.populations())
        out.append(got)
        g.close()
    for a, b in zip(*out):
        assert np.array_equal(a, b)
