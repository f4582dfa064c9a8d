"""FP64 slice products through the separable hopping exponential against the dense ones: line lengths on both sides
of the forms' boundaries (folded sums up to 8 and above 16, tensor-instruction transforms between), ragged
column panels, columns spread over many orders of magnitude, and a field that is not finite."""
import numpy as np
import pytest
import torch

from oracle import HolsteinParams
from oracle.fermion import fermion_logdet
from paper_1802_06177_gb300 import inputs
from tests.gpu_util import cuda, make_ctx

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("Lx,Ly,n_s", [(8, 9, 5), (9, 8, 4), (16, 5, 6), (5, 16, 12), (13, 11, 7), (15, 10, 24), (16, 16, 8),
                                       (17, 5, 6), (3, 32, 5), (8, 8, 6)])
def test_line_transforms_match_dense_and_oracle(Lx, Ly, n_s):
    L, nf = 24, 3
    x = inputs.mixed_fields(nf, Lx, Ly, L, seed=Lx + 100 * Ly)
    x[0] *= 2.5  # columns of one group then span about ten orders of magnitude
    ctx = make_ctx(Lx, L, n_s, Ly=Ly, max_fields=nf, mu=-0.15)
    ctx.set_sub_batches(1)  # the general kernels at N <= 64 too
    G, ld, sg = ctx.greens(cuda(x))
    ctx.set_dense_slices(1)
    Gd, ldd, sgd = ctx.greens(cuda(x))
    assert (G - Gd).abs().max().item() < 1e-9 and (ld - ldd).abs().max().item() < 1e-8 and torch.equal(sg, sgd)
    p = HolsteinParams(Lx, Ly, L, n_s=n_s, mu=-0.15)
    for f in range(nf):
        l_ref, s_ref, G_ref = fermion_logdet(p, x[f])
        assert abs(ld[f].item() - l_ref) < 1e-8 and sg[f].item() == s_ref
        assert np.abs(G[f].cpu().numpy() - G_ref).max() < 1e-9


def test_line_transforms_keep_a_nan_field_apart():
    from paper_1802_06177_gb300.slmc import SlmcError
    x = inputs.gaussian_fields(3, 12, 10, 10, seed=8)
    ctx = make_ctx(12, 10, 5, Ly=10, max_fields=3)
    want, _ = ctx.logdet(cuda(x))
    x[1, 50, 3] = np.inf
    x[1, 51, 3] = np.nan
    got, sg = ctx.logdet(cuda(x))
    with pytest.raises(SlmcError):
        ctx.get_error()
    assert torch.equal(got[[0, 2]], want[[0, 2]]) and torch.isnan(got[1]) and sg[1].item() == 0


@pytest.mark.parametrize("dtau", [0.001, 0.1, 0.4, 0.5])
def test_line_transforms_near_and_far_from_the_identity(dtau):
    """The factor's digits are cut less the identity while its off-diagonal entries stay below 1/2 (dtau = 0.5: whole)."""
    Lx, Ly, L, n_s, nf = 12, 10, 6, 2, 2
    x = inputs.mixed_fields(nf, Lx, Ly, L, seed=3)
    ctx = make_ctx(Lx, L, n_s, Ly=Ly, max_fields=nf, dtau=dtau)
    G, ld, sg = ctx.greens(cuda(x))
    p = HolsteinParams(Lx, Ly, L, n_s=n_s, dtau=dtau)
    for f in range(nf):
        l_ref, s_ref, G_ref = fermion_logdet(p, x[f])
        assert abs(ld[f].item() - l_ref) < 1e-8 and sg[f].item() == s_ref
        assert np.abs(G[f].cpu().numpy() - G_ref).max() < 1e-9
