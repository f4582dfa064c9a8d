"""The QR panels of batches with more fields than multiprocessors run with 256 threads per field instead of 512:
determinants and G of such a batch against the oracle and, bit for bit, against the same fields in small batches,
with both panel widths, seven and eight digits (DQMC) and a ragged last panel."""
import numpy as np
import pytest
import torch

from oracle import HolsteinParams
from oracle.dqmc import dqmc_sweeps
from oracle.fermion import fermion_logdet
from paper_1802_06177_gb300 import inputs
from tests.gpu_util import cuda, make_ctx

pytestmark = pytest.mark.gpu


def _more_than_sms():
    return torch.cuda.get_device_properties(0).multi_processor_count + 8


@pytest.mark.parametrize("Lx,Ly,panel,precision", [(9, 8, 32, "fp64"), (9, 8, 16, "fp64"), (11, 9, 32, "bf16x9"),
                                                   (7, 11, 16, "fp32"), (6, 6, 32, "fp64")])
def test_large_batch_matches_oracle_and_small_batches(Lx, Ly, panel, precision):
    nf, L, n_s = _more_than_sms(), 8, 4
    x = inputs.mixed_fields(nf, Lx, Ly, L, seed=Lx)
    out = []
    for max_fields in (nf, 20):
        ctx = make_ctx(Lx, L, n_s, Ly=Ly, precision=precision, max_fields=max_fields)
        ctx.set_tuning(panel, 0)
        if max_fields == nf:
            ctx.set_sub_batches(1)
        out.append(ctx.greens(cuda(x)))
        ctx.get_error()
    for a, b in zip(*out):
        assert torch.equal(a, b)
    p = HolsteinParams(Lx, Ly, L, n_s=n_s)
    tol = (1e-8, 1e-9) if precision == "fp64" else (5e-5, 1e-6)
    for f in (0, 1, nf // 2, nf - 1):
        l_ref, s_ref, G_ref = fermion_logdet(p, x[f])
        G, ld, sg = (t[f].cpu().numpy() for t in out[0])
        assert abs(ld - l_ref) < tol[0] and sg == s_ref and np.abs(G - G_ref).max() < tol[1]


def test_dqmc_of_more_chains_than_sms_matches_oracle():
    Lx, Ly, L, n_s, seed = 9, 8, 4, 2, 17
    nf = _more_than_sms()
    x = inputs.mixed_fields(nf, Lx, Ly, L, seed=3)
    ctx = make_ctx(Lx, L, n_s, Ly=Ly, max_fields=nf, sweep_delta=0.4, seed=seed)
    xg = cuda(x.copy())
    ctx.dqmc_sweep(xg, 1, sweep0=1)
    ctx.get_error()
    for f in (0, nf // 2, nf - 1):
        xo = x[f].copy()
        dqmc_sweeps(HolsteinParams(Lx, Ly, L, n_s=n_s), xo, 1, 1, f, seed, 0.4)
        assert np.array_equal(xg[f].cpu().numpy(), xo)
