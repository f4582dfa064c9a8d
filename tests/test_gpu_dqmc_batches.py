"""DQMC sweeps where G lies in shared memory, against the oracle field for field: odd numbers of sites (a chain's
G is then 8- but not 16-byte aligned) and the batched rank-16 updates on the tensor instruction (N > 64: partial
row and column tiles, several batches and a partial one per slice; N = 160 is
the largest G in shared memory and leaves no room for them)."""
import numpy as np
import pytest
import torch

from oracle import HolsteinParams
from oracle.dqmc import dqmc_sweeps
from paper_1802_06177_gb300 import inputs
from tests.gpu_util import cuda, make_ctx

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("Lx,Ly,L,n_s,delta", [(3, 3, 6, 3, 0.5), (5, 3, 5, 2, 0.5), (7, 7, 4, 2, 0.5), (9, 8, 6, 3, 0.3),
                                               (11, 9, 3, 2, 0.8), (12, 12, 4, 2, 0.5), (16, 10, 2, 2, 0.2)])
def test_sweeps_match_oracle(Lx, Ly, L, n_s, delta):
    nf, seed = 3, 4242
    x = inputs.mixed_fields(nf, Lx, Ly, L, seed=Lx * Ly)
    ctx = make_ctx(Lx, L, n_s, Ly=Ly, max_fields=nf, sweep_delta=delta, seed=seed)
    xg, na = cuda(x.copy()), torch.zeros(nf, dtype=torch.int64, device="cuda")
    ctx.dqmc_sweep(xg, 1, sweep0=5, n_acc_local=na)
    ctx.get_error()
    p = HolsteinParams(Lx, Ly, L, n_s=n_s)
    for f in range(nf):
        xo = x[f].copy()
        nl, _ = dqmc_sweeps(p, xo, 1, 5, f, seed, delta)
        assert np.array_equal(xg[f].cpu().numpy(), xo) and na[f].item() == nl
        assert nl > 16 or Lx * Ly < 65
