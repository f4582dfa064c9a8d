"""Contexts of different sizes used by several host threads at once: kernels ask for shared memory by the lattice's
size, and a launch must not meet the limit that another thread's smaller lattice has set meanwhile."""
import threading

import numpy as np
import pytest
import torch

from paper_1802_06177_gb300 import inputs
from tests.gpu_util import cuda, make_ctx

pytestmark = pytest.mark.gpu
J = np.array([0.0, 45.0, 0.6, 0.01, 0.1, 0.2])


# Sides, slices, chains and updates of either thread, the updates looping inside the library. One-launch sweeps of 8x8,
# L = 100 need 52 KB, more than a kernel has without asking; of 16x16 and 8x10 every kernel of a determinant differs.
@pytest.mark.parametrize("sizes,precision", [(((8, 8, 100, 2, 400), (4, 4, 8, 4, 8000)), "fp64"),
                                             (((16, 16, 8, 2, 400), (8, 10, 8, 2, 800)), "fp64"),
                                             (((16, 16, 8, 2, 400), (8, 10, 8, 2, 800)), "fp32"),
                                             (((16, 16, 8, 2, 400), (8, 10, 8, 2, 800)), "bf16x9")])
def test_updates_of_two_sizes_on_two_threads(sizes, precision):
    errors, out = [], {}

    def work(k, Lx, Ly, L, n, updates):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                ctx = make_ctx(Lx, L, 10, Ly=Ly, precision=precision, max_fields=n, sweep_delta=0.4, seed=k)
                ctx.set_wolff(1)
                x, Jt = cuda(inputs.gaussian_fields(n, Lx, Ly, L, seed=k)), cuda(J)
                lnw, _ = ctx.chain_init(x, want_cdw=False)
                ctx.cumulative_update(x, Jt, 1, updates, 0, lnw)
                ctx.get_error()
                out.setdefault(k, []).append(x.cpu())
        except Exception as e:  # reported by the test's own thread
            errors.append(e)

    for k, s in enumerate(sizes):  # each alone
        work(k, *s)
    threads = [threading.Thread(target=work, args=(k, *s)) for k, s in enumerate(sizes)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
    assert all(torch.equal(*out[k]) for k in range(len(sizes)))
