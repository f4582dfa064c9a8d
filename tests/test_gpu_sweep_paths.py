"""The E_eff sweeps' FP32 decision with integer-formed operands against the oracle's FP64 rule: fields and
acceptance counts bit for bit where the operands leave the FP32 range (zero, subnormal, large), where the
proposal width is zero or too small for the scaled product, and for the shortest lines and slices."""
import numpy as np
import pytest
import torch

from oracle import HolsteinParams
from oracle.chain import eff_sweeps
from tests.gpu_util import cuda, make_ctx

pytestmark = pytest.mark.gpu
J = np.array([0.0, 45.0, 0.6, 0.01, 0.1, 0.2])


@pytest.mark.parametrize("Lx,Ly,L,scale,delta", [
    (4, 2, 2, 1.0, 0.5), (2, 6, 10, 1.0, 0.5), (4, 4, 12, 0.0, 0.4), (4, 4, 12, 1e-42, 0.0), (4, 4, 12, 1e-300, 1e-260),
    (4, 4, 12, 1.0, 1e-260), (4, 4, 12, 1e25, 0.5), (4, 4, 12, 1e45, 0.5)])
def test_decisions_at_the_edges_of_fp32(Lx, Ly, L, scale, delta):
    seed = 77
    ctx = make_ctx(Lx, L, 2, Ly=Ly, max_fields=3, sweep_delta=delta, seed=seed)
    x = scale * np.random.default_rng(5).standard_normal((3, Lx * Ly, L))
    xg, n_acc = cuda(x.copy()), torch.zeros(3, dtype=torch.int64, device="cuda")
    ctx.eff_sweep(xg, cuda(J), 4, sweep0=9, first_colour=1, n_acc=n_acc)
    p = HolsteinParams(Lx, Ly, L, n_s=2)
    for f in range(3):
        xo = x[f].copy()
        na = eff_sweeps(p, xo, J[1:], 4, 9, 1, f, seed, delta)
        assert np.array_equal(xg[f].cpu().numpy(), xo)
        assert n_acc[f].item() == na


@pytest.mark.parametrize("Lx,Ly,L,nwolff", [(2, 2, 2, 2), (8, 16, 64, 1), (8, 16, 66, 1), (32, 32, 8, 0), (4, 4, 40, 3)])
def test_sweeps_in_one_launch_and_per_half_sweep(Lx, Ly, L, nwolff):
    """Chains up to 8192 sites x slices run all sweeps in one launch, larger ones a launch per half-sweep
    (8 x 16 x 64 and 8 x 16 x 66 lie on either side): both bit for bit the oracle's."""
    seed = 31
    ctx = make_ctx(Lx, L, 2, Ly=Ly, max_fields=2, sweep_delta=0.4, seed=seed)
    ctx.set_wolff(nwolff)
    x = np.random.default_rng(6).standard_normal((2, Lx * Ly, L))
    xg, n_acc = cuda(x.copy()), torch.zeros(2, dtype=torch.int64, device="cuda")
    ctx.eff_sweep(xg, cuda(J), 2, sweep0=12345, first_colour=0, n_acc=n_acc)
    p, sizes = HolsteinParams(Lx, Ly, L, n_s=2), []
    for f in range(2):
        xo = x[f].copy()
        na = eff_sweeps(p, xo, J[1:], 2, 12345, 0, f, seed, 0.4, nwolff=nwolff, wolff_sizes=sizes)
        assert np.array_equal(xg[f].cpu().numpy(), xo)
        assert n_acc[f].item() == na
    assert ctx.wolff_sites() == sum(sizes)
