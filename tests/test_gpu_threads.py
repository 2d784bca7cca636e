"""Objects of different sizes side by side: each asks for its own amount of shared memory of the same kernels,
and neither may take it from the other, whether they are used in turn or from two host threads at once."""
import threading

import numpy as np
import pytest

import paper_1009_0254_gb300 as lbf

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1009_0254_gb300 import build
    build.build()
    lbf.load()


def _lattice(nx, ny, mode, nbins):
    import torch
    g = lbf.Lattice(nx, ny, seed=nx + ny, stream=torch.cuda.Stream())
    g.set_params(1e-4, 0.02, 0.8, 1.1, 0.9, mode)
    if nbins:
        g.set_sampling(1, nbins)
    return g


# many steps a launch (64^2 and 128^2); the transforms of the noise; the spectra's transforms and bins
@pytest.mark.parametrize("small,large,mode,bins,calls,steps", [
    ((64, 64), (128, 128), lbf.LB_NOISE_LW, (0, 0), 600, 8),
    ((64, 4096), (64, 8192), lbf.LB_NOISE_FULL, (0, 0), 200, 2),
    ((32, 64), (64, 64), lbf.LB_NOISE_LW, (8, 4096), 200, 2)])
def test_two_threads_step_lattices_of_two_sizes(small, large, mode, bins, calls, steps):
    want = []
    for (nx, ny), nb in zip((small, large), bins):
        g = _lattice(nx, ny, mode, nb)
        g.step(calls * steps)
        want.append(g.populations())
        g.close()
    lats = [_lattice(*small, mode, bins[0]), _lattice(*large, mode, bins[1])]
    errors, start = [], threading.Barrier(2)

    def work(g):
        start.wait()
        try:
            for _ in range(calls):
                g.step(steps)
            lbf.lb_synchronize(g.ctx)
        except lbf.LBError as e:
            errors.append(str(e))

    threads = [threading.Thread(target=work, args=(g,)) for g in lats]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
    for g, w in zip(lats, want):
        assert np.array_equal(g.populations(), w)
        g.close()


def test_a_later_ensemble_leaves_an_earlier_one_its_bins():
    ens = []
    for nb in (1024, 8):
        e = lbf.Ensemble([(32, 32)] * 2, [1, 2])
        e.set_params(-1, 1e-4, 0.02, 0.8, 1.1, 0.9, lbf.LB_NOISE_LW)
        e.set_sampling(2, nb)
        ens.append(e)
    for e in ens:
        e.step(4)
        assert e.structure_factor(0)[4] == 2


def test_a_later_server_leaves_an_earlier_one_its_noise():
    srv = [lbf.Server(1 << 30, max_active=4, max_chunk_steps=4) for _ in range(2)]
    order = [(0, 4096), (1, 64), (0, 4096)]
    out = []
    for k, ny in order:
        i = srv[k].submit(32, ny, 4, 1e-4, 0.02, 0.8, 1.1, 0.9, noise_mode=lbf.LB_NOISE_FULL, seed=3, keep_state=True)
        srv[k].wait(i)
        out.append(srv[k].fetch(i, 32, ny))
    assert np.array_equal(out[0], out[2])
    for s in srv:
        s.close()
