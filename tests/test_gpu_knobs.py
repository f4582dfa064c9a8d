"""Which kernels a context runs follows the values of its knobs, not whether a setter was called: the one-launch
FP64 determinant of small lattices comes back with the defaults, and the sub-batch split of small lattices
follows slmc_set_sub_batches alone."""
import pytest
import torch

from paper_1802_06177_gb300 import inputs
from tests.gpu_util import cuda, make_ctx, require_gpu

pytestmark = pytest.mark.gpu


def _launches(ctx, x):
    n0 = ctx.launch_count()
    out = ctx.logdet(x)[0]
    return ctx.launch_count() - n0, out


@pytest.mark.parametrize("setter,value,default", [("set_tuning", (16, 0), (0, 0)), ("set_qr_cluster", (1,), (0,)),
                                                  ("set_dense_slices", (1,), (0,)), ("set_tupdate_path", (1,), (0,)),
                                                  ("set_qr_path", (1,), (0,))])
def test_default_values_restore_the_one_launch_determinant(setter, value, default):
    x = cuda(inputs.mixed_fields(5, 4, 4, 20, seed=2))
    ctx = make_ctx(4, 20, 5, max_fields=5)
    n, want = _launches(ctx, x)
    assert n == 1
    getattr(ctx, setter)(*value)
    n, got = _launches(ctx, x)
    assert n > 1 and (got - want).abs().max().item() < 1e-8
    getattr(ctx, setter)(*default)
    n, got = _launches(ctx, x)
    assert n == 1 and torch.equal(got, want)


def test_split_of_small_lattices_follows_set_sub_batches_only():
    x = cuda(inputs.mixed_fields(66, 8, 8, 8, seed=2))
    for precision in ("fp64", "fp32"):
        ctx = make_ctx(8, 8, 4, precision=precision, max_fields=66)
        n1, want = _launches(ctx, x)
        ctx.set_tuning(0, 0)
        ctx.set_qr_cluster(0)
        ctx.set_dense_slices(0)
        ctx.set_tupdate_path(0)
        ctx.set_qr_path(0)
        ctx.set_sub_batch_priorities(1)
        ctx.set_sub_batch_priorities(0)
        n, got = _launches(ctx, x)
        assert n == n1 and torch.equal(got, want)
        ctx.set_sub_batches(1)
        ns, _ = _launches(ctx, x)
        ctx.set_sub_batches(2)
        n, got = _launches(ctx, x)
        assert n == 2 * ns and (got - want).abs().max().item() < 1e-8


def test_autotune_times_the_one_launch_determinant():
    """At 4x4 it takes a fraction of the general kernels' time; applying the result keeps it."""
    from paper_1802_06177_gb300.slmc import autotune
    require_gpu()
    r = autotune(4, 4, 20, precision="fp64", ntune=8, tol=1e-7)
    assert r["qr_panel"] == 0
    ctx = make_ctx(4, 20, r["n_s"], max_fields=5)
    ctx.set_tuning(r["qr_panel"], r["slice_cols"])
    assert _launches(ctx, cuda(inputs.mixed_fields(5, 4, 4, 20, seed=2)))[0] == 1
