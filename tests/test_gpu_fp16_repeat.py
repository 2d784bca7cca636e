"""FP16 lattices give the same state bit for bit whichever kernel of theirs steps them, and the one of
golden/fp16_states.txt: the CRC-32 of the FP64 populations after the listed steps, recorded from the kernel that
steps one node a lane (lb_step_half.cu).  A sum taken in another order agrees to FP32
rounding, but sends the values next to a rounding boundary of FP16 the other way; within some tens of steps
the state and its structure factor then differ by 2^-11 a value.

The structure factor is transformed and binned in FP32 from equal states, so it agrees to the bound of
test_gpu_spectra_sums.py, 1e-5."""
import os
import zlib

import numpy as np
import pytest

import paper_1009_0254_gb300 as lbf
from paper_1009_0254_gb300 import synth

PARAMS = (1e-4, 0.02, 0.8, 1.1, 0.9)
BINS = 8
W = np.array([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4)
GOLDEN = os.path.join(os.path.dirname(os.path.abspath(__file__)), "golden", "fp16_states.txt")


def recorded():
    """(nx, ny, noise mode, noise factor, steps) -> (CRC-32, S per bin; none unless sizes are powers of two)."""
    out = {}
    with open(GOLDEN) as f:
        for line in f:
            if not line.startswith("#"):
                w = line.split()
                out[tuple(int(v) for v in w[:5])] = (int(w[5], 16), np.array([float(v) for v in w[6:]]))
    return out


def run(nx, ny, mode, factor, steps):
    g = lbf.Lattice(nx, ny, seed=nx + 1000 * ny, precision=lbf.LB_FP16DEV)
    g.set_params(*PARAMS, mode)
    if factor:
        lbf.lb_set_noise_factor(g.ctx, factor)
    pow2 = not (nx & (nx - 1)) and not (ny & (ny - 1))
    if pow2:
        g.set_sampling(steps, BINS)
    noise = synth.uniform(-0.02, 0.02, 9 * ny * nx, seed=nx + ny).reshape(9, ny, nx)
    g.set_populations(W[:, None, None] * (1.0 + noise))
    g.step(steps)
    S = g.structure_factor()[0] if pow2 else np.zeros(0)
    crc = zlib.crc32(np.ascontiguousarray(g.populations()).tobytes())
    g.close()
    return crc, S


@pytest.mark.gpu
@pytest.mark.parametrize("kernel", ["default", "tma"])
@pytest.mark.parametrize("case", sorted(recorded()))
def test_state_is_the_recorded_one(case, kernel, monkeypatch):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1009_0254_gb300 import build
    build.build()
    monkeypatch.delenv("LBFLUCT_STEP_KERNEL", raising=False)
    if kernel != "default":
        monkeypatch.setenv("LBFLUCT_STEP_KERNEL", kernel)
    crc, S = run(*case)
    want, want_s = recorded()[case]
    assert np.allclose(S, want_s, rtol=1e-5, atol=0, equal_nan=True), (S, want_s)
    assert crc == want
