"""The paired step kernels (lb_pair.cuh) at the edges of their tiles against the FP64 oracle:
lattices one node short of, equal to and past a tile in x and y, rows that end inside a 16-byte
unit of the store box, odd rows (a last pair of one node), lattices smaller than a tile and than
the ghost width, on every storage, noise mode and engine that runs them.

Tolerances as in the parity tests: 1e-5 for FP32; FP16 holds df / w to half a unit in the last
place of a value of at most 0.5 (2^-13) per step, so 10 steps stay within 10 * 2^-13 * 4/9."""
import numpy as np
import pytest

import oracle
import paper_1009_0254_gb300 as lbf
from paper_1009_0254_gb300 import synth

pytestmark = pytest.mark.gpu
PARAMS = (1e-4, 0.04, 0.8, 1.1, 0.9)
SIZES = [(63, 7), (64, 8), (65, 9), (66, 16), (70, 17), (33, 15), (31, 33), (127, 5), (130, 8), (9, 64), (5, 3), (2, 2)]
MODES = {lbf.LB_NOISE_OFF: oracle.NOISE_OFF, lbf.LB_NOISE_LW: oracle.NOISE_LW,
         lbf.LB_NOISE_FULL_RS: oracle.NOISE_FULL_RS}
TOL = {lbf.LB_FP32: 1e-5, lbf.LB_FP16DEV: 10 * 2.0 ** -13 * 4 / 9}


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1009_0254_gb300 import build
    build.build()
    lbf.load()


def _oracle(nx, ny, mode, seed):
    o = oracle.Lattice(nx, ny, seed=seed)
    o.set_params(*PARAMS, MODES[mode])
    o.f = o.f * (1.0 + synth.gaussian_field((9, ny, nx), seed=seed, scale=0.01))
    return o


@pytest.mark.parametrize("precision", [lbf.LB_FP32, lbf.LB_FP16DEV])
@pytest.mark.parametrize("mode", sorted(MODES))
def test_single_lattice_at_tile_edges(mode, precision):
    for k, (nx, ny) in enumerate(SIZES):
        o = _oracle(nx, ny, mode, 50 + k)
        g = lbf.Lattice(nx, ny, seed=50 + k, precision=precision)
        g.set_params(*PARAMS, mode)
        g.set_populations(o.f)
        g.step(10)
        o.step(10)
        assert np.abs(g.populations() - o.f).max() <= TOL[precision], (nx, ny)


@pytest.mark.parametrize("mode", sorted(MODES))
def test_engines_at_tile_edges(mode):
    os_ = [_oracle(nx, ny, mode, 50 + k) for k, (nx, ny) in enumerate(SIZES)]
    ens = lbf.Ensemble(SIZES, [50 + k for k in range(len(SIZES))])
    ens.set_params(-1, *PARAMS, mode)
    srv = lbf.Server(1 << 30, max_active=32, max_chunk_steps=4)
    ids = []
    for k, (nx, ny) in enumerate(SIZES):
        ens.set_populations(k, os_[k].f)
        ids.append(srv.submit(nx, ny, 10, *PARAMS, noise_mode=mode, seed=50 + k, keep_state=True, init=os_[k].f))
    ens.step(10)
    for k, (nx, ny) in enumerate(SIZES):
        os_[k].step(10)
        assert np.abs(ens.populations(k) - os_[k].f).max() <= TOL[lbf.LB_FP32], ("batched", nx, ny)
        srv.wait(ids[k])
        assert np.abs(srv.fetch(ids[k], nx, ny) - os_[k].f).max() <= TOL[lbf.LB_FP32], ("served", nx, ny)
    srv.close()
