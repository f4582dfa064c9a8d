"""The five feature sums of E_eff where the threads' walk over a field has its edges: rows shorter and longer than the
256 values between a thread's steps and next to them, one slice, fields of fewer values than threads, the largest
lattice, and sides of two (a site is its neighbour's neighbour twice)."""
import numpy as np
import pytest
import torch

from tests.gpu_util import cuda, make_ctx

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("Lx,Ly,L", [(2, 2, 1), (3, 2, 5), (4, 4, 40), (2, 7, 255), (3, 3, 256), (2, 3, 257), (2, 2, 1023),
                                     (5, 4, 300), (16, 2, 32), (12, 12, 120), (32, 32, 3), (7, 31, 33)])
def test_features_match_plain_sums(Lx, Ly, L):
    a2 = (1.0 / 0.7 ** 2) ** 2
    x = np.random.default_rng(Lx * L).standard_normal((3, Lx * Ly, L))
    ctx = make_ctx(Lx, L, 2, Ly=Ly, max_fields=3, omega0=0.7)
    got = ctx.eff_features(cuda(x)).cpu().numpy()
    y = x.reshape(3, Ly, Lx, L)
    t, nb = np.roll(y, -1, 3), np.roll(y, -1, 2) + np.roll(y, -1, 1)
    terms = [(t - y) ** 2, 0.25 * y ** 4 - 0.5 * a2 * y ** 2, y ** 6 / 6.0 - 0.25 * a2 * y ** 4, y * nb, y * t]
    for q, term in enumerate(terms):
        ref, mag = term.sum(axis=(1, 2, 3)), np.abs(term).sum(axis=(1, 2, 3))
        # every partial sum rounded once, a few roundings per term
        assert (np.abs(got[:, q] - ref) <= 2.0 ** -53 * (Lx * Ly * L + 8) * mag).all(), q
    J = torch.tensor([0.3, 45.0, 0.6, 0.01, 0.1, 0.2], dtype=torch.float64, device="cuda")
    lnw = ctx.eff_log_weight(cuda(x), J).cpu().numpy()
    assert np.allclose(lnw, -0.1 * (0.3 + got @ J[1:].cpu().numpy()), rtol=1e-12, atol=1e-12)
