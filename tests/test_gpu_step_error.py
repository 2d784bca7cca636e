"""One step in FP32 against the same step with FP64 storage, from equal states and the same draws: relative
error of the populations' deviations, every mode and lattice that takes the packed normals.

Bound.  The normals' hardware approximations are off by 2.1e-7 of a normal (2^31 draws), of which 1.2e-7 is a
common factor that the noise amplitudes give back; 1.7e-7 is left.  A step adds the rounding of a stored value,
2^-25 and less, and that of a mode's factors, in quadrature, while the noise is only a part of the deviations:
the whole stays below the normals' 1.7e-7 in two dimensions.  D3Q19 and D3Q27 round more sums: 2e-7."""
import numpy as np
import pytest

import paper_1009_0254_gb300 as lbf

pytestmark = pytest.mark.gpu
MODES = [lbf.LB_NOISE_LW, lbf.LB_NOISE_FULL_RS, lbf.LB_NOISE_LW_LOCAL]


def _error(make, mode):
    a, b = make(lbf.LB_FP32), make(lbf.LB_FP64)
    for g in (a, b):
        g.set_params(1e-4, 0.01, 0.8, 1.0, 1.0, mode)
    f = a.populations()
    rest = f.reshape(len(f), -1)[:, 0].reshape((-1,) + (1,) * (f.ndim - 1)).copy()
    a.set_populations(f * (1.0 + 0.01 * np.random.default_rng(1).standard_normal(f.shape)))
    a.step(10)
    b.set_populations(a.populations(), t=10)
    a.step(1)
    b.step(1)
    fa, fb = a.populations(), b.populations()
    return np.sqrt(((fa - fb) ** 2).sum() / ((fb - rest) ** 2).sum())


@pytest.fixture(autouse=True)
def _built():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1009_0254_gb300 import build
    build.build()


@pytest.mark.parametrize("mode", MODES)
def test_two_dimensions(mode):
    assert _error(lambda p: lbf.Lattice(512, 512, seed=1, precision=p), mode) <= 1.7e-7


@pytest.mark.parametrize("mode", MODES)
@pytest.mark.parametrize("q", [19, 27])
def test_three_dimensions(q, mode):
    assert _error(lambda p: lbf.Lattice3(64, 64, 64, seed=1, lattice=q, precision=p), mode) <= 2e-7
