"""Small FP32 lattices do take many steps a launch (lb_step_resident.cu), and launches end at the samples: the
launch counter tells them from a launch a step, and the spectra sampled on the way are the same."""
import numpy as np
import pytest

import paper_1009_0254_gb300 as lbf

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def _built():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1009_0254_gb300 import build
    build.build()


def _lattice(nx, ny, kernel, monkeypatch):
    if kernel:
        monkeypatch.setenv("LBFLUCT_STEP_KERNEL", kernel)
    else:
        monkeypatch.delenv("LBFLUCT_STEP_KERNEL", raising=False)
    g = lbf.Lattice(nx, ny, seed=5)
    g.set_params(1e-4, 0.01, 0.8, 1.1, 0.9, lbf.LB_NOISE_LW)
    return g


def _added(g, steps):
    n = lbf.lb_launch_count(g.ctx)
    g.step(steps)
    return lbf.lb_launch_count(g.ctx) - n


# the shortest call that takes one launch: four steps up to 8,192 nodes, eight above; and the longest launch
@pytest.mark.parametrize("nx,ny,least", [(32, 32, 4), (64, 128, 4), (66, 125, 8), (128, 128, 8)])
def test_launches(nx, ny, least, monkeypatch):
    g = _lattice(nx, ny, None, monkeypatch)
    assert _added(g, 30) == 1
    assert _added(g, least) == 1
    assert _added(g, least - 1) == least - 1
    assert _added(g, 4096 + least) == 2
    lbf.lb_set_kernel_timing(g.ctx, 1)           # timed: a launch a step
    assert _added(g, 30) == 30 and lbf.lb_kernel_time(g.ctx)[1] == 30
    lbf.lb_set_kernel_timing(g.ctx, 0)
    assert _added(g, 30) == 1
    g.close()
    g = _lattice(nx, ny, "tma", monkeypatch)
    assert _added(g, 30) == 30
    g.close()


@pytest.mark.parametrize("every", [1, 3, 9, 25])
def test_launches_end_at_the_samples(every, monkeypatch):
    out = []
    for kernel in (None, "tma"):
        g = _lattice(64, 64, kernel, monkeypatch)
        g.step(2)                                # the first sample is cut from a call that starts between two
        g.set_sampling(every, 16)
        for n in (7, 40, 1, 30):
            g.step(n)
        out.append((g.populations(), g.structure_factor()))
        g.close()
    (fa, a), (fb, b) = out
    assert np.array_equal(fa, fb)
    assert a[4] == b[4] == 80 // every - 2 // every
    # equal states; the bins are sums of FP32 runs in an order of their own (test_gpu_spectra_sums.py)
    for u, v in zip(a[:3], b[:3]):
        assert np.allclose(u, v, rtol=1e-5, atol=0, equal_nan=True)
    assert np.array_equal(a[3], b[3])
