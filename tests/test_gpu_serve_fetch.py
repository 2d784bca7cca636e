"""Two threads fetch kept states while the server admits and steps other requests: every state is the one that
the request gives alone, and all memory comes back."""
import threading

import numpy as np
import pytest

import paper_1009_0254_gb300 as lbf

pytestmark = pytest.mark.gpu
REQUESTS = [(32, 300, 1), (64, 200, 2), (128, 120, 3), (256, 60, 4)]


def test_fetches_beside_stepping():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1009_0254_gb300 import build
    build.build()
    par = (1e-4, 0.02, 0.8, 1.1, 0.9)
    srv = lbf.Server(1 << 28, max_active=6, max_chunk_steps=20)
    alone = {}
    for n, steps, seed in REQUESTS:
        i = srv.submit(n, n, steps, *par, seed=seed, keep_state=True)
        srv.wait(i, 60.0)
        alone[n] = srv.fetch(i, n, n)
    errors = []

    def client(k):
        try:
            for r in range(12):
                batch = [REQUESTS[(k + r + j) % 4] for j in range(3)]
                ids = [srv.submit(n, n, steps, *par, seed=seed, keep_state=True) for n, steps, seed in batch]
                for i, (n, _, _) in zip(ids, batch):
                    srv.wait(i, 60.0)
                    if not np.array_equal(srv.fetch(i, n, n), alone[n]):
                        errors.append("state of %d^2 differs" % n)
        except Exception as e:
            errors.append(repr(e))

    threads = [threading.Thread(target=client, args=(k,)) for k in range(2)]
    for t in threads:
        t.start()
    long_run = srv.submit(512, 512, 2000, *par, seed=9)
    for t in threads:
        t.join()
    assert not errors, errors
    srv.wait(long_run, 60.0)
    assert srv.stats().bytes_in_use == 0 and srv.stats().completed == 4 + 72 + 1
    srv.close()
