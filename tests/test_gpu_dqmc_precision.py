"""The Green's function that decides the local moves of DQMC is as accurate as FP64 FMAs leave it (N > 64: the chains'
QR and Q run through products of digits). For each chain the half-widths of the proposals are found, from the oracle's G,
at which the first move's log acceptance ratio lies 4e-15 above and below ln u: the GPU accepts the one and rejects the
other.

The log ratio moves by 2 dl / R, up to 0.08, times an error of G_00, and by a few units of rounding: FP64 FMAs leave G
within 5e-14 at these sizes, 4e-15 in the log ratio (up to 5e-16 is seen). 49-bit digits shift it by 1e-15 to 5e-15 at 9x8
and by 4e-15 to 7e-13 at 9x9 with groups of 20 slices. The field is zero around the first site, so that nothing
cancels in the phonon part."""
import numpy as np
import pytest
from scipy.optimize import brentq

from oracle import HolsteinParams
from oracle.dqmc import dqmc_sweeps, greens_at, local_move, wrap
from oracle.lattice import exp_hopping
from paper_1802_06177_gb300 import inputs
from tests.gpu_util import cuda, make_ctx

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("Lx,Ly,L,n_s", [(9, 8, 160, 10), (9, 9, 160, 20), (12, 12, 80, 10)])
def test_first_move_flips_where_the_oracle_says(Lx, Ly, L, n_s):
    nf, seed, sweep = 6, 7, 3
    p = HolsteinParams(Lx, Ly, L, n_s=n_s)
    E, Einv = exp_hopping(Lx, Ly, 1.0, 0.0, p.dtau), exp_hopping(Lx, Ly, 1.0, 0.0, -p.dtau)
    x = inputs.mixed_fields(nf, Lx, Ly, L, seed=5)
    x[:, 0, [L - 1, 0, 1]] = 0.0
    for f in range(nf):
        G = wrap(p, greens_at(p, x[f], 0, E), x[f][:, 0], E, Einv)

        def excess(delta):
            _, _, _, lnr, u = local_move(p, x[f], G, 0, 0, sweep, f, seed, delta)
            return lnr - np.log(u)

        grid = np.linspace(0.01, 20.0, 2000)
        at = next(k for k in range(1, len(grid)) if excess(grid[k]) < 0)
        for margin in (4e-15, -4e-15):
            delta = brentq(lambda d: excess(d) - margin, grid[at - 1], grid[at], xtol=1e-16, rtol=1e-15)
            ctx = make_ctx(Lx, L, n_s, Ly=Ly, max_fields=nf, sweep_delta=delta, seed=seed)
            xg = cuda(x.copy())
            ctx.dqmc_sweep(xg, 1, sweep0=sweep)
            ctx.get_error()
            assert (xg[f, 0, 0].item() != 0.0) == (margin > 0), f


def test_sweeps_under_every_knob_match_the_oracle():
    """The QR's path steers the chains of DQMC, the T update's does not (the same launches)."""
    Lx, Ly, L, n_s, nf, seed = 9, 8, 6, 3, 2, 31
    x = inputs.mixed_fields(nf, Lx, Ly, L, seed=9)
    want, count = [x[f].copy() for f in range(nf)], {}
    for f in range(nf):
        dqmc_sweeps(HolsteinParams(Lx, Ly, L, n_s=n_s), want[f], 1, 2, f, seed, 0.4)
    for qr_path in (0, 1):
        for tupdate_path in (0, 1, 2):
            ctx = make_ctx(Lx, L, n_s, Ly=Ly, max_fields=nf, sweep_delta=0.4, seed=seed)
            ctx.set_qr_path(qr_path)
            ctx.set_tupdate_path(tupdate_path)
            xg, n0 = cuda(x.copy()), ctx.launch_count()
            ctx.dqmc_sweep(xg, 1, sweep0=2)
            ctx.get_error()
            assert all(np.array_equal(xg[f].cpu().numpy(), want[f]) for f in range(nf))
            assert count.setdefault(qr_path, ctx.launch_count() - n0) == ctx.launch_count() - n0
    assert count[1] < count[0]
