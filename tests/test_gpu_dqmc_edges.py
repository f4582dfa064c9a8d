"""DQMC sweeps at the edges of what fits in shared memory, against the oracle field for field: 7x21 (N = 147) is the
largest lattice with G and a batch of moves there, 10x15 the first with G alone, 11x15 (N = 165) the largest with
G there (6x27: the same with the longest lines' instance), 12x14 and 13x13 the first with G in global memory."""
import numpy as np
import pytest
import torch

from oracle import HolsteinParams
from oracle.dqmc import dqmc_sweeps
from paper_1802_06177_gb300 import inputs
from tests.gpu_util import cuda, make_ctx

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("Lx,Ly", [(7, 21), (10, 15), (11, 15), (6, 27), (12, 14), (13, 13)])
def test_sweep_matches_oracle(Lx, Ly):
    nf, L, n_s, seed, delta = 3, 3, 2, 515, 0.4
    x = inputs.mixed_fields(nf, Lx, Ly, L, seed=Lx + Ly)
    ctx = make_ctx(Lx, L, n_s, Ly=Ly, max_fields=nf, sweep_delta=delta, seed=seed)
    xg, na = cuda(x.copy()), torch.zeros(nf, dtype=torch.int64, device="cuda")
    ctx.dqmc_sweep(xg, 1, sweep0=4, n_acc_local=na)
    ctx.get_error()
    for f in range(nf):
        xo = x[f].copy()
        nl, _ = dqmc_sweeps(HolsteinParams(Lx, Ly, L, n_s=n_s), xo, 1, 4, f, seed, delta)
        assert np.array_equal(xg[f].cpu().numpy(), xo) and na[f].item() == nl and nl > 32
