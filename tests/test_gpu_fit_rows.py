"""The regression at the edges of its threads: fewer rows than warps, one row per thread and just above, several rows
per thread with a ragged last pass. The log-weights are exactly linear in the features."""
import numpy as np
import pytest
import torch

from tests.gpu_util import cuda, make_ctx

pytestmark = pytest.mark.gpu
J_TEST = np.array([1.5, 50.0, 0.35, -0.02, 0.06, 0.4])


@pytest.mark.parametrize("n", [6, 7, 32, 33, 223, 224, 225, 511, 513, 1025, 2048, 2049, 4500])
def test_fit_recovers_the_couplings(n):
    Lx, L = 4, 8
    rng = np.random.default_rng(n)
    x = cuda(rng.standard_normal((n, Lx * Lx, L)) * rng.uniform(0.3, 1.5, (n, 1, 1)) + rng.uniform(-0.8, 0.8, (n, 1, 1)))
    ctx = make_ctx(Lx, L, 4, max_fields=n)
    lnw = ctx.eff_log_weight(x, cuda(J_TEST))
    J, resid = ctx.fit_eff(x, lnw)
    # six unknowns: exact up to rounding times the condition of the few-row cases
    assert np.allclose(J.cpu().numpy(), J_TEST, rtol=1e-7, atol=1e-8) and resid.item() < 1e-8
    # the rows' order (and with it their threads) does not matter
    p = torch.randperm(n, device="cuda")
    J2, _ = ctx.fit_eff(x[p].contiguous(), lnw[p].contiguous())
    assert np.allclose(J2.cpu().numpy(), J.cpu().numpy(), rtol=1e-7, atol=1e-8)
