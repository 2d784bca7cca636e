"""A server that runs out of device memory while it admits a request loses that request only: whichever of an
admission's allocations fails, the request ends with LB_ENOMEM, and those before and after it run.

The allocations are made to fail on the host: a preloaded function returns cudaErrorMemoryAllocation from the
n-th cudaMallocFromPoolAsync of the process and calls the library's for all others."""
import os
import subprocess
import sys
import textwrap

import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SHIM = r"""
#define _GNU_SOURCE
#include <dlfcn.h>
#include <stddef.h>
#include <stdlib.h>
int cudaMallocFromPoolAsync(void** p, size_t bytes, void* pool, void* stream) {
    static int calls = 0;
    static int (*real)(void**, size_t, void*, void*) = NULL;
    const char* n = getenv("FAIL_POOL_ALLOCATION");
    if (__sync_add_and_fetch(&calls, 1) == (n ? atoi(n) : 0)) return 2;    /* cudaErrorMemoryAllocation */
    if (!real) {
        void* rt = dlopen("libcudart.so.13", RTLD_LAZY | RTLD_NOLOAD);
        real = rt ? (int (*)(void**, size_t, void*, void*))dlsym(rt, "cudaMallocFromPoolAsync") : NULL;
    }
    return real ? real(p, bytes, pool, stream) : 999;
}
"""

# a small request that runs for long, a large one behind it, then another small one
CHILD = textwrap.dedent("""
    import numpy as np
    import paper_1009_0254_gb300 as lbf
    srv = lbf.Server(1 << 30, max_active=8, max_chunk_steps=50)
    ids = [srv.submit(64, 64, 20000, seed=1, keep_state=True)]
    ids.append(srv.submit(1 << 11, 1 << 11, 60, seed=2))
    status = [srv.wait(ids[1], 60.0).status]
    ids.append(srv.submit(64, 64, 200, seed=3))
    status += [srv.wait(ids[k], 60.0).status for k in (0, 2)]
    mass = srv.fetch(ids[0], 64, 64).sum() if status[1] == lbf.LB_OK else 64.0 * 64.0
    print("STATUS", *status, abs(mass / 4096 - 1) < 1e-6, srv.stats().bytes_in_use)
    srv.close()
""")


# allocations: the state and the first tile table of request 0, the state and a larger table of request 1
@pytest.mark.parametrize("fails,want", [(0, (0, 0, 0)), (1, (0, -3, 0)), (2, (0, -3, 0)), (3, (-3, 0, 0)), (4, (-3, 0, 0))])
def test_one_allocation_fails_one_request(fails, want, tmp_path):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1009_0254_gb300 as lbf
    from paper_1009_0254_gb300 import build
    build.build()
    assert lbf.LB_ENOMEM == -3 and lbf.LB_OK == 0
    (tmp_path / "shim.c").write_text(SHIM)
    so = str(tmp_path / "shim.so")
    subprocess.run(["gcc", "-O1", "-shared", "-fPIC", "-o", so, str(tmp_path / "shim.c"), "-ldl"], check=True)
    env = dict(os.environ, LD_PRELOAD=so, FAIL_POOL_ALLOCATION=str(fails))
    r = subprocess.run([sys.executable, "-c", CHILD], cwd=ROOT, env=env, capture_output=True, text=True, timeout=300)
    line = [v for v in r.stdout.splitlines() if v.startswith("STATUS")]
    assert r.returncode == 0 and line, r.stdout + r.stderr
    assert line[0].split()[1:] == [str(v) for v in want] + ["True", "0"], line[0]
