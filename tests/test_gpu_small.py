"""The one-launch FP64 determinant of small lattices (N <= 64) against the oracle and the general kernels: the
edges of its size classes (N = 16, 32, 64 and their neighbours), lines longer than 8 sites, ragged and long slice
groups, one field and many, and what must still be refused or flagged."""
import numpy as np
import pytest
import torch

from oracle import HolsteinParams
from oracle.fermion import fermion_logdet
from paper_1802_06177_gb300 import inputs
from tests.gpu_util import cuda, make_ctx

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("Lx,Ly,L,n_s", [(2, 2, 1, 1), (3, 5, 7, 3), (4, 4, 40, 10), (17, 1 + 1, 9, 4), (4, 8, 12, 5),
                                         (3, 11, 10, 10), (5, 5, 23, 8), (7, 7, 30, 7), (9, 7, 20, 6), (8, 8, 64, 8),
                                         (32, 2, 16, 8)])
def test_small_matches_oracle_and_general(Lx, Ly, L, n_s):
    nf = 5
    x = inputs.mixed_fields(nf, Lx, Ly, L, seed=Lx * L)
    ctx = make_ctx(Lx, L, n_s, Ly=Ly, max_fields=3, mu=0.2)
    G, ld, sg = ctx.greens(cuda(x))
    ld2, sg2 = ctx.logdet(cuda(x))
    ctx.get_error()
    assert torch.equal(ld, ld2) and torch.equal(sg, sg2)
    ctx.set_qr_path(1)
    Gg, ldg, sgg = ctx.greens(cuda(x))
    assert (G - Gg).abs().max().item() < 1e-9 and (ld - ldg).abs().max().item() < 1e-8 and torch.equal(sg, sgg)
    p = HolsteinParams(Lx, Ly, L, n_s=n_s, mu=0.2)
    for f in range(nf):
        l_ref, s_ref, G_ref = fermion_logdet(p, x[f])
        assert abs(ld[f].item() - l_ref) < 1e-8 and sg[f].item() == s_ref
        assert np.abs(G[f].cpu().numpy() - G_ref).max() < 1e-9


def test_small_flags_a_nan_field_and_keeps_the_others():
    x = inputs.gaussian_fields(4, 6, 6, 12, seed=3)
    ctx = make_ctx(6, 12, 4, max_fields=4)
    want, _ = ctx.logdet(cuda(x))
    x[2, 7, 3] = np.nan
    got, sg = ctx.logdet(cuda(x))
    from paper_1802_06177_gb300.slmc import SlmcError
    with pytest.raises(SlmcError) as e:
        ctx.get_error()
    assert e.value.status == 2
    keep = [0, 1, 3]
    assert torch.equal(got[keep], want[keep]) and torch.isnan(got[2]) and sg[2].item() == 0
