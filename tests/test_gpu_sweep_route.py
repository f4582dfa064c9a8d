"""Which E_eff sweeps run in one launch: by the size of a chain, the number of chains and whether there are Wolff
updates; the chains are bit for bit the same either way."""
import numpy as np
import pytest
import torch

from tests.gpu_util import cuda, make_ctx

pytestmark = pytest.mark.gpu
J = np.array([0.0, 45.0, 0.6, 0.01, 0.1, 0.2])


@pytest.mark.parametrize("Lx,Ly,L,n,nwolff,fused", [(4, 4, 40, 1, 0, True), (8, 8, 64, 1, 0, True), (8, 8, 66, 3, 0, False),
                                                    (8, 8, 80, 4, 0, True), (8, 8, 128, 1, 0, False),
                                                    (8, 8, 128, 31, 0, False), (8, 8, 128, 32, 0, True),
                                                    (8, 8, 128, 1, 1, True), (8, 8, 130, 32, 1, False)])
def test_launches_of_the_sweeps(Lx, Ly, L, n, nwolff, fused):
    nsweeps = 3
    ctx = make_ctx(Lx, L, 2, Ly=Ly, max_fields=32, sweep_delta=0.4, seed=8)
    ctx.set_wolff(nwolff)
    x = np.random.default_rng(7).standard_normal((32, Lx * Ly, L))
    xg, acc = cuda(x[:n].copy()), torch.zeros(n, dtype=torch.int64, device="cuda")
    n0 = ctx.launch_count()
    ctx.eff_sweep(xg, cuda(J), nsweeps, sweep0=3, first_colour=1, n_acc=acc)
    assert ctx.launch_count() - n0 == (1 if fused else nsweeps * (2 + nwolff))
    # the same chains beside 31 others, which may take the other route
    xa, acca = cuda(x.copy()), torch.zeros(32, dtype=torch.int64, device="cuda")
    ctx.eff_sweep(xa, cuda(J), nsweeps, sweep0=3, first_colour=1, n_acc=acca)
    assert torch.equal(xa[:n], xg) and torch.equal(acca[:n], acc)
