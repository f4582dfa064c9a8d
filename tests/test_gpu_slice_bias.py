"""The rounding of the hopping factors must not add up over the slices: every slice multiplies by the same table, so
a diagonal of 1 + 2e-4 rounded to FP64 shifts ln det by (N / 2) L times its rounding error. ln det of long chains with a
small dtau against extended precision."""
import numpy as np
import pytest

from paper_1802_06177_gb300 import inputs
from tests.gpu_util import cuda, make_ctx

pytestmark = pytest.mark.gpu
LD = np.longdouble


def _line(n, a):
    """exp(a h) of a ring of n sites, h its adjacency matrix (both bonds of a ring of two)."""
    h = np.zeros((n, n), LD)
    for i in range(n):
        h[i, (i + 1) % n] += 1
        h[(i + 1) % n, i] += 1
    E, T = np.eye(n, dtype=LD), np.eye(n, dtype=LD)
    for k in range(1, 25):
        T = T.dot(h) * (a / k)
        E = E + T
    return E


def _logdet(x, Lx, Ly, n_s, dtau):
    """ln|det(I + B_L .. B_1)| (mu = 0, lambda = 1) in extended precision, stabilised every n_s slices."""
    N, L = x.shape
    x, dtau = x.astype(LD), LD(dtau)
    Ex, Ey = _line(Lx, dtau), _line(Ly, dtau)
    U, lnD, T = np.eye(N, dtype=LD), np.zeros(N, LD), np.eye(N, dtype=LD)
    for l0 in range(0, L, n_s):
        for l in range(l0, min(L, l0 + n_s)):
            U = Ey.dot(U.reshape(Ly, Lx * N)).reshape(Ly, Lx, N)
            U = np.stack([Ex.dot(row) for row in U]).reshape(N, N) * np.exp(-dtau * x[:, l])[:, None]
        P = np.argsort(-(np.log(np.sqrt((U * U).sum(0))) + lnD), kind="stable")
        R, Q = U[:, P].copy(), np.eye(N, dtype=LD)
        vs = []
        for k in range(N - 1):
            v = R[k:, k].copy()
            v[0] += np.copysign(np.sqrt((v * v).sum()), v[0])
            b = 2 / (v * v).sum()
            R[k:, k:] -= np.outer(b * v, v.dot(R[k:, k:]))
            vs.append((v, b))
        for k in range(N - 2, -1, -1):
            v, b = vs[k]
            Q[k:, k:] -= np.outer(b * v, v.dot(Q[k:, k:]))
        R, d = np.triu(R), np.abs(np.diag(R))
        T = ((R * np.exp(lnD[P] - lnD[P][:, None])) / d[:, None]).dot(T[P])
        U, lnD = Q, np.log(d) + lnD[P]
    M = U.T * np.exp(-np.maximum(lnD, 0))[:, None] + np.exp(np.minimum(lnD, 0))[:, None] * T
    s = np.maximum(lnD, 0).sum()
    for k in range(N):
        p = k + np.argmax(np.abs(M[k:, k]))
        M[[k, p]] = M[[p, k]]
        s += np.log(abs(M[k, k]))
        M[k + 1:, k:] -= np.outer(M[k + 1:, k] / M[k, k], M[k, k:])
    return float(s)


def diagonal_rounding(n, dtau):
    d = _line(n, LD(dtau))[0, 0]
    return float(LD(np.float64(d)) - d)


@pytest.mark.parametrize("Lx,Ly,L,dtau", [(4, 4, 2000, 0.017), (6, 6, 2000, 0.014), (17, 3, 1000, 0.012)])
def test_tables_do_not_shift_the_determinant(Lx, Ly, L, dtau):
    n_s, N = 10, Lx * Ly
    x = inputs.gaussian_fields(1, Lx, Ly, L, seed=21)
    ref = _logdet(x[0], Lx, Ly, n_s, dtau)
    # ten times the rms of 12 independent roundings of 2^-54 per site and slice
    tol = 10 * np.sqrt(12.0 * N * L) * 2.0 ** -54
    assert 0.5 * N * L * abs(diagonal_rounding(Lx, dtau) + diagonal_rounding(Ly, dtau)) > 5 * tol  # sensitive
    for general in (False, True):
        ctx = make_ctx(Lx, L, n_s, Ly=Ly, max_fields=1, dtau=dtau)
        if general:  # the per-group kernels, FP64 FMAs in QR and T
            ctx.set_qr_path(1)
            ctx.set_tupdate_path(1)
        ld, _ = ctx.logdet(cuda(x))
        assert abs(ld[0].item() - ref) < tol
