"""A state read into device memory (one launch for all populations) equals the one read to the host
(population by population): the same values bit for bit, on odd sizes, sizes below a block and a ghost
width, and every storage, engine and lattice."""
import numpy as np
import pytest

import paper_1009_0254_gb300 as lbf

pytestmark = pytest.mark.gpu
PARAMS = (1e-4, 0.01, 0.8, 1.1, 0.9)
SIZES = [(2, 2), (33, 5), (128, 3), (257, 130), (64, 300)]


def _device(read, shape):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    f = torch.full(shape, float("nan"), dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    read(f)
    return f.cpu().numpy()


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1009_0254_gb300 import build
    build.build()
    lbf.load()


@pytest.mark.parametrize("precision", [lbf.LB_FP32, lbf.LB_FP16DEV, lbf.LB_FP64])
def test_single_lattice(precision):
    for nx, ny in SIZES:
        g = lbf.Lattice(nx, ny, seed=3, precision=precision)
        g.set_params(*PARAMS, lbf.LB_NOISE_LW)
        g.step(5)
        d = _device(lambda f: lbf.lb_get_populations(g.ctx, f, lbf.LB_DEVICE), (9, ny, nx))
        assert np.array_equal(d, g.populations()), (nx, ny)
        g.close()


def test_ensemble():
    e = lbf.Ensemble(SIZES, list(range(len(SIZES))))
    e.set_params(-1, *PARAMS, lbf.LB_NOISE_LW)
    e.step(5)
    for k, (nx, ny) in enumerate(SIZES):
        d = _device(lambda f: lbf.lb_batch_get_populations(e.b, k, f, lbf.LB_DEVICE), (9, ny, nx))
        assert np.array_equal(d, e.populations(k)), (nx, ny)


@pytest.mark.parametrize("precision", [lbf.LB_FP32, lbf.LB_FP64])
@pytest.mark.parametrize("q", [19, 27])
def test_three_dimensions(q, precision):
    for nx, ny, nz in [(2, 2, 2), (33, 5, 3), (130, 17, 9)]:
        g = lbf.Lattice3(nx, ny, nz, lattice=q, seed=3, precision=precision)
        g.set_params(*PARAMS, lbf.LB_NOISE_LW)
        g.step(3)
        d = _device(lambda f: lbf.lb3_get_populations(g.ctx, f, lbf.LB_DEVICE), (q, nz, ny, nx))
        assert np.array_equal(d, g.populations()), (nx, ny, nz)
        g.close()
