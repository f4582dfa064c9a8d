"""Q of an FP64 determinant from eight digits per operand (56 bits): as near to FP64 arithmetic as Q formed with FMAs, so
that G errs only by the QR's 49-bit trailing updates."""
import pytest
import torch

from paper_1802_06177_gb300 import inputs
from tests.gpu_util import cuda, make_ctx

pytestmark = pytest.mark.gpu


# Sizes on both sides of an accumulator set's six K chunks (N = 384) with panels of 16 and 32 columns. The Frobenius
# error of G against FP64 FMAs throughout, with Q by FMAs or eight digits / with seven: 27x26 2.4e-13 / 3.3e-13,
# 18x18 8.3e-14 / 1.04e-13, 16x16 7.5e-14 / 9.1e-14; the bounds lie halfway.
@pytest.mark.parametrize("Lx,Ly,L,n_s,nf,bound", [(27, 26, 4, 2, 3, 2.8e-13), (18, 18, 1, 1, 8, 9.3e-14),
                                                  (16, 16, 1, 1, 8, 8.2e-14)])
def test_q_adds_no_error_to_g(Lx, Ly, L, n_s, nf, bound):
    x = cuda(0.01 * inputs.gaussian_fields(nf, Lx, Ly, L, seed=11))
    ctx = make_ctx(Lx, L, n_s, Ly=Ly, max_fields=nf)
    ctx.set_tupdate_path(1)
    G, _, _ = ctx.greens(x)
    ctx.set_qr_path(1)
    ref, _, _ = ctx.greens(x)
    ctx.get_error()
    assert ((G - ref).norm(dim=(1, 2)) / ref.norm(dim=(1, 2))).mean().item() < bound


@pytest.mark.parametrize("Lx,Ly,panel", [(10, 8, 32), (9, 9, 32), (12, 8, 16), (24, 16, 32), (24, 16, 16), (25, 16, 32), (28, 28, 16),
                                         (32, 28, 0)])
def test_q_paths_agree(Lx, Ly, panel):
    """Both sides of the path's smallest N (81), one to three accumulator sets with either panel width, the largest N (896)."""
    x = cuda(inputs.mixed_fields(2, Lx, Ly, 4, seed=Lx))
    ctx = make_ctx(Lx, 4, 2, Ly=Ly, max_fields=2)
    ctx.set_tuning(panel, 0)
    G, ld, sg = ctx.greens(x)
    ctx.set_qr_path(1)
    Gr, ldr, sgr = ctx.greens(x)
    ctx.get_error()
    assert (G - Gr).abs().max().item() < 1e-9 and (ld - ldr).abs().max().item() < 1e-8 and torch.equal(sg, sgr)
