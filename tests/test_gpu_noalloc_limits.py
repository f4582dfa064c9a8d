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
