"""slmc_logdet_noalloc at the edge of its 16 MiB array."""
import pytest
import torch

from paper_1802_06177_gb300 import inputs
from tests.gpu_util import cuda, make_ctx

pytestmark = pytest.mark.gpu


def test_largest_fp32_field_of_529_sites():
    """One FP32 field of 23x23 sites and 419 slices fills the array to within 2 KB; one slice more is refused."""
    from paper_1802_06177_gb300.slmc import SlmcError, logdet_noalloc
    Lx, L, n_s = 23, 419, 10
    x = cuda(inputs.gaussian_fields(1, Lx, Lx, L, seed=6))
    got, sg = logdet_noalloc(x, Lx, Lx, L, n_s=n_s, precision="fp32")
    ctx = make_ctx(Lx, L, n_s, precision="fp32", max_fields=1)
    ctx.set_tupdate_path(1)
    ctx.set_qr_path(1)
    want, sw = ctx.logdet(x)
    assert (got - want).abs().max().item() <= 1e-10 and torch.equal(sg, sw)
    x = cuda(inputs.gaussian_fields(1, Lx, Lx, L + 1, seed=6))
    with pytest.raises(SlmcError) as e:
        logdet_noalloc(x, Lx, Lx, L + 1, n_s=n_s, precision="fp32")
    assert e.value.status == 5


@pytest.mark.parametrize("Lx,Ly,L,n_s,qr_mode,general", [(4, 4, 40, 10, "prepivot", False), (8, 8, 20, 6, "prepivot", False),
                                                         (9, 8, 40, 10, "prepivot", True), (4, 4, 40, 10, "pivoted", True)])
def test_fp64_arithmetic_is_the_documented_one(Lx, Ly, L, n_s, qr_mode, general):
    """The one-launch determinant up to 64 sites, the general kernels with FP64 FMAs above and in the pivoted mode."""
    from paper_1802_06177_gb300.slmc import logdet_noalloc
    x = cuda(inputs.mixed_fields(5, Lx, Ly, L, seed=12))
    got, sg = logdet_noalloc(x, Lx, Ly, L, n_s=n_s, qr_mode=qr_mode)
    ctx = make_ctx(Lx, L, n_s, Ly=Ly, max_fields=5, qr_mode=qr_mode)
    if general:
        ctx.set_tupdate_path(1)
        ctx.set_qr_path(1)
    n0 = ctx.launch_count()
    want, sw = ctx.logdet(x)
    assert (ctx.launch_count() - n0 > 1) == general
    assert torch.equal(got, want) and torch.equal(sg, sw)
