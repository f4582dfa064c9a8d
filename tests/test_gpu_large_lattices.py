"""FP64 determinants, Green's functions and DQMC sweeps of the largest lattices (sides up to 32, N up to 1024), whose
panels of folded line transforms no longer fit 32 columns in shared memory, against the oracle. 26 x 32 is the
largest with a side of 32 that still does."""
import numpy as np
import pytest
import torch

from oracle import HolsteinParams
from oracle.dqmc import dqmc_sweeps
from oracle.fermion import fermion_logdet
from paper_1802_06177_gb300 import inputs
from tests.gpu_util import cuda, make_ctx

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("Lx,Ly", [(26, 32), (27, 32), (32, 27), (28, 31), (31, 28), (29, 30), (30, 29), (28, 32), (32, 32)])
def test_greens_matches_oracle(Lx, Ly):
    L, n_s = 3, 2
    x = inputs.gaussian_fields(1, Lx, Ly, L, seed=Lx)
    ctx = make_ctx(Lx, L, n_s, Ly=Ly, max_fields=1)
    G, ld, sg = ctx.greens(cuda(x))
    ctx.get_error()
    l_ref, s_ref, G_ref = fermion_logdet(HolsteinParams(Lx, Ly, L, n_s=n_s), x[0])
    assert abs(ld[0].item() - l_ref) < 1e-8 and sg[0].item() == s_ref
    assert np.abs(G[0].cpu().numpy() - G_ref).max() < 1e-9


def test_dqmc_sweep_matches_oracle():
    Lx, Ly, L, n_s, seed, delta = 27, 32, 2, 1, 99, 0.3
    x = inputs.gaussian_fields(1, Lx, Ly, L, seed=4)
    ctx = make_ctx(Lx, L, n_s, Ly=Ly, max_fields=1, sweep_delta=delta, seed=seed)
    xg, na = cuda(x.copy()), torch.zeros(1, dtype=torch.int64, device="cuda")
    ctx.dqmc_sweep(xg, 1, sweep0=3, n_acc_local=na)
    ctx.get_error()
    xo = x[0].copy()
    nl, _ = dqmc_sweeps(HolsteinParams(Lx, Ly, L, n_s=n_s), xo, 1, 3, 0, seed, delta)
    assert np.array_equal(xg[0].cpu().numpy(), xo) and na[0].item() == nl
