"""The work that users of this package have it do, as cases that can be timed and compared.

A case names one kind of call and its sizes. The kinds, and what each stands for in real use:

  greens      Context.greens, then Context.measure_cdw on the G it returns: the exact determinant, the
              equal-time Green's function and S(pi, pi) of given fields in FP64 (a measurement after a sweep,
              or the check of a configuration).
  log_weight  Context.log_weight in a reduced-precision mode: the scoring of proposed configurations, the
              bulk of every self-learning round. Large lattices, where these modes are used.
  update      Context.cumulative_update with S(pi, pi): one step of SLMC production, the chains' state
              carried from call to call.
  sweep       Context.eff_sweep: the effective model's Markov chain alone, which proposes training
              configurations.
  batch       Batch.launch: one replay of the captured round of chains of uneven size.
  dqmc        Context.dqmc_sweep: the conventional method (training data, and the baseline).
  fit         Context.fit_eff: the regression of the effective model on scored configurations.

Model parameters are t = 1, mu = 0, dtau = 0.1 and lambda = omega0 = 1 (omega0 = 0.5, the paper's critical
point, where a case says so). Fields are drawn on the GPU from the seed: the first half of a batch iid
N(0, 1), the second half the checkerboard pattern 0.8 (-1)^(ix+iy) plus N(0, 0.3^2) noise, the two kinds of
field that the benchmark workloads hold.
"""
import os
from concurrent.futures import ThreadPoolExecutor

import numpy as np
import torch

from paper_1802_06177_gb300.slmc import UPDATE_CONTINUE, Batch, Context

DTAU = 0.1
# Couplings {E0, J_k, J_p, J_p', J_nn, J_nn'} as learned on the 24x24 lattice at beta = 24.
COUPLINGS = [0.0, 50.54, -0.122, 0.021, 0.037, 0.316]
# The published fit at g = 1, Omega = 0.5 (Table S1 of the paper's supplement), without its sixth-order
# term, which is not bounded below.
COUPLINGS_CRITICAL = [0.0, 50.0, 0.0139, 0.0, 0.00717, 0.0767]


def listed():
    return [
        # One chain of the smallest lattice advanced by one update: all launches and latency.
        dict(name="update_4x4_one_chain", kind="update", Lx=4, Ly=4, L=40, n=1, n_s=10, precision="fp64",
             nsweeps=50, wolff=0, omega0=1.0),
        # The small workload: 64 fields of 4x4, beta = 4.
        dict(name="greens_4x4", kind="greens", Lx=4, Ly=4, L=40, n=64, n_s=10),
        # Odd sizes: a rectangle whose sides and slices no tile divides, a short last slice group.
        dict(name="greens_18x10_ragged", kind="greens", Lx=18, Ly=10, L=37, n=50, n_s=10),
        # The plain FP64 workload: 256 fields of 12x12, beta = 12.
        dict(name="greens_12x12", kind="greens", Lx=12, Ly=12, L=120, n=256, n_s=10),
        # The benchmark workload: 512 fields of 16x16, beta = 16, slice products on the tensor cores.
        dict(name="log_weight_16x16_bf16x9", kind="log_weight", Lx=16, Ly=16, L=160, n=512, n_s=8,
             precision="bf16x9"),
        # The large lattice of the whole-pipeline workload in its default precision: few, large fields.
        dict(name="log_weight_24x24_fp32", kind="log_weight", Lx=24, Ly=24, L=240, n=32, n_s=8,
             precision="fp32"),
        # A production step of the autocorrelation study: 8x8 at the critical point with Wolff updates.
        dict(name="update_8x8_wolff", kind="update", Lx=8, Ly=8, L=40, n=128, n_s=10, precision="fp32",
             nsweeps=10, wolff=1, omega0=0.5),
        # The effective model's sweeps of the benchmark step.
        dict(name="sweep_16x16", kind="sweep", Lx=16, Ly=16, L=160, n=512, nsweeps=20, wolff=0),
        # The uneven batch, a thermalisation round: one graph launch advances 256 chains of four sizes.
        dict(name="batch_uneven", kind="batch", sizes="8x80 10x100 12x120 16x160", n=64, n_s=10,
             precision="bf16x9", nsweeps=20),
        # A DQMC step of the autocorrelation study: local updates and four block updates.
        dict(name="dqmc_8x8_block", kind="dqmc", Lx=8, Ly=8, L=40, n=128, n_s=10, nblock=4, omega0=0.5),
        # The DQMC benchmark: one chain per multiprocessor, local updates.
        dict(name="dqmc_12x12", kind="dqmc", Lx=12, Ly=12, L=120, n=152, n_s=10, nblock=0, omega0=1.0),
        # The regression on 2000 configurations.
        dict(name="fit_12x12", kind="fit", Lx=12, Ly=12, L=120, n=2000),
    ]


def _log_int(rng, lo, hi):
    return int(round(lo * (hi / lo) ** rng.random()))


def _even(v):
    return 2 * ((v + 1) // 2)


def draw(rng):
    kind = rng.choice(["greens", "greens", "log_weight", "log_weight", "update", "sweep", "batch", "dqmc", "fit"])
    if kind == "greens":  # any rectangle and number of slices, from one field to a full batch
        Lx, Ly = rng.randint(3, 18), rng.randint(3, 18)
        L, n_s = rng.randint(17, 160), rng.randint(6, 12)
        most = 0.5e11 / ((Lx * Ly) ** 3 * (L / n_s + 2.0))
        return dict(kind=kind, Lx=Lx, Ly=Ly, L=L, n=max(1, min(_log_int(rng, 1, 256), int(most))), n_s=n_s)
    if kind == "log_weight":  # the large lattices of production, odd sides and odd batches among them
        Lx, Ly = rng.randint(12, 24), rng.randint(12, 24)
        L, n_s = rng.randint(140, 240), rng.randint(6, 10)
        most = 1.0e11 / ((Lx * Ly) ** 3 * (L / n_s))
        return dict(kind=kind, Lx=Lx, Ly=Ly, L=L, n=max(2, min(_log_int(rng, 16, 512), int(most))), n_s=n_s,
                    precision=rng.choice(["bf16x9", "fp32"]))
    if kind == "update":  # the studies' sizes, from one chain to 128
        critical = rng.random() < 0.5
        return dict(kind=kind, Lx=_even(rng.randint(3, 10)), Ly=_even(rng.randint(3, 10)), L=_even(rng.randint(20, 60)),
                    n=_log_int(rng, 1, 128), n_s=rng.randint(8, 10), precision=rng.choice(["fp64", "fp32"]),
                    nsweeps=_log_int(rng, 5, 50), wolff=1 if critical else 0, omega0=0.5 if critical else 1.0)
    if kind == "sweep":
        return dict(kind=kind, Lx=_even(rng.randint(3, 24)), Ly=_even(rng.randint(3, 24)), L=_even(rng.randint(40, 240)),
                    n=_log_int(rng, 1, 256), nsweeps=_log_int(rng, 5, 100), wolff=rng.randint(0, 1))
    if kind == "batch":
        sizes = sorted(rng.sample([4, 6, 8, 10, 12, 14], rng.randint(2, 4)))
        return dict(kind=kind, sizes=" ".join("%dx%d" % (s, 10 * s) for s in sizes), n=_log_int(rng, 8, 64),
                    n_s=rng.randint(8, 10), precision=rng.choice(["bf16x9", "fp32"]), nsweeps=_log_int(rng, 5, 40))
    if kind == "dqmc":
        Lx, Ly, L = rng.randint(3, 13), rng.randint(3, 13), rng.randint(10, 120)
        nblock = rng.choice([0, 2, 4])
        most = 0.4e8 / ((Lx * Ly) ** 2 * L / 10.0 * (1 + nblock))
        return dict(kind=kind, Lx=Lx, Ly=Ly, L=L, n=max(4, min(_log_int(rng, 16, 152), int(most))),
                    n_s=rng.randint(8, 10), nblock=nblock, omega0=rng.choice([0.5, 1.0]))
    Lx, L = rng.randint(4, 16), rng.randint(40, 160)
    return dict(kind="fit", Lx=Lx, Ly=Lx, L=L, n=_log_int(rng, 500, 3000))


def _sizes(case):
    """(side, slices) of each class of a batch."""
    return [tuple(int(v) for v in s.split("x")) for s in case["sizes"].split()]


def _fields(n, Lx, Ly, L, seed):
    """n fields [n, N, L]: the first half iid N(0, 1), the rest the checkerboard pattern with noise."""
    g = torch.Generator(device="cuda").manual_seed(int(seed) & 0x7fffffffffff)
    x = torch.randn((n, Lx * Ly, L), generator=g, dtype=torch.float64, device="cuda")
    i = torch.arange(Lx * Ly, device="cuda")
    stag = 1.0 - 2.0 * ((i % Lx + i // Lx) % 2).double()
    h = (n + 1) // 2
    x[h:] = 0.8 * stag[None, :, None] + 0.3 * x[h:]
    return x


def _context(case, seed, precision, **kw):
    return Context(case["Lx"], case["Ly"], case["L"], dtau=DTAU, n_s=case.get("n_s", 10), precision=precision,
                   max_fields=case["n"], seed=seed, **kw)


def _features(x, Lx, Ly, a2=1.0):
    """The five sums of E_eff of each field, in plain torch (FP64)."""
    n, N, L = x.shape
    y = x.view(n, Ly, Lx, L)
    t = torch.roll(y, -1, 3)
    y2 = y * y
    s = lambda v: v.sum(dim=(1, 2, 3))  # noqa: E731
    return torch.stack([s((t - y) ** 2), s(0.25 * y2 * y2 - 0.5 * a2 * y2), s(y2 ** 3 / 6.0 - 0.25 * a2 * y2 * y2),
                        s(y * (torch.roll(y, -1, 2) + torch.roll(y, -1, 1))), s(y * t)], dim=1)


def _scored(case, seed):
    """Configurations of varied amplitude and log-weights near a linear model of their features."""
    n, Lx, Ly = case["n"], case["Lx"], case["Ly"]
    x = _fields(n, Lx, Ly, case["L"], seed)
    g = torch.Generator(device="cuda").manual_seed((int(seed) + 1) & 0x7fffffffffff)
    x *= 0.5 + torch.rand((n, 1, 1), generator=g, dtype=torch.float64, device="cuda")
    J = torch.tensor(COUPLINGS, dtype=torch.float64, device="cuda")
    lnw = -DTAU * (_features(x, Lx, Ly) @ J[1:]) + 5.0 * torch.randn(n, generator=g, dtype=torch.float64, device="cuda")
    return x, lnw


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        sizes = _sizes(case)
        J = torch.tensor(COUPLINGS, dtype=torch.float64, device="cuda")
        b = Batch([dict(Lx=s, L=L, nchains=case["n"], n_s=case["n_s"], precision=case["precision"], dtau=DTAU,
                        sweep_delta=0.3, seed=seed + q) for q, (s, L) in enumerate(sizes)])
        out = []
        for q, (s, L) in enumerate(sizes):
            x = _fields(case["n"], s, s, L, seed + 1000 * q)
            lnw, _ = b.context(q).chain_init(x, want_cdw=False)
            n_acc = torch.zeros(case["n"], dtype=torch.int64, device="cuda")
            n_sw = torch.zeros(case["n"], dtype=torch.int64, device="cuda")
            b.bind(q, x, J, lnw, None, n_acc, n_sw)
            out.append([x, lnw, n_acc, n_sw])
        torch.cuda.synchronize()
        b.capture(case["nsweeps"], 1)
        return dict(case=case, batch=b, J=J, out=out)
    if kind == "fit":
        x, lnw = _scored(case, seed)
        return dict(case=case, ctx=_context(case, seed, "fp32"), x=x, lnw=lnw)
    x = _fields(case["n"], case["Lx"], case["Ly"], case["L"], seed)
    st = dict(case=case, x=x)
    if kind == "greens":
        st["ctx"] = _context(case, seed, "fp64")
        return st
    if kind == "log_weight":
        st["ctx"] = _context(case, seed, case["precision"])
        return st
    st["n_acc"] = torch.zeros(case["n"], dtype=torch.int64, device="cuda")
    st["n_more"] = torch.zeros(case["n"], dtype=torch.int64, device="cuda")
    st["step"] = 0
    if kind == "sweep":
        st["ctx"] = _context(case, seed, "fp32", sweep_delta=0.3)
        st["ctx"].set_wolff(case["wolff"])
        st["J"] = torch.tensor(COUPLINGS, dtype=torch.float64, device="cuda")
    elif kind == "update":
        st["ctx"] = _context(case, seed, case["precision"], sweep_delta=0.3, omega0=case["omega0"])
        st["ctx"].set_wolff(case["wolff"])
        st["J"] = torch.tensor(COUPLINGS if case["omega0"] == 1.0 else COUPLINGS_CRITICAL, dtype=torch.float64,
                               device="cuda")
        st["lnw"], st["s"] = st["ctx"].chain_init(x)
        st["ctx"].set_update_counter(0)
    else:
        st["ctx"] = _context(case, seed, "fp64", sweep_delta=0.5, omega0=case["omega0"])
    return st


def run(state):
    kind, ctx = state["case"]["kind"], state.get("ctx")
    if kind == "greens":
        G, lndet, sign = ctx.greens(state["x"])
        return dict(G=G, lndet=lndet, sign=sign, S=ctx.measure_cdw(G))
    if kind == "log_weight":
        lnw, lndet, sign = ctx.log_weight(state["x"])
        return dict(lnw=lnw, lndet=lndet, sign=sign)
    if kind == "update":
        obs = ctx.cumulative_update(state["x"], state["J"], state["case"]["nsweeps"], 1, UPDATE_CONTINUE, state["lnw"],
                                    state["s"], state["n_acc"], state["n_more"], want_obs=True)
        return dict(x=state["x"], lnw=state["lnw"], S=state["s"], obs=obs, n_acc=state["n_acc"], n_sweep=state["n_more"])
    if kind == "sweep":
        nsweeps = state["case"]["nsweeps"]
        ctx.eff_sweep(state["x"], state["J"], nsweeps, sweep0=state["step"] * nsweeps, first_colour=state["step"] & 1,
                      n_acc=state["n_acc"])
        state["step"] += 1
        return dict(x=state["x"], n_acc=state["n_acc"])
    if kind == "batch":
        b, now = state["batch"], torch.cuda.current_stream()
        b.stream.wait_stream(now)
        b.launch(1)
        now.wait_stream(b.stream)
        return state["out"]
    if kind == "dqmc":
        ctx.dqmc_sweep(state["x"], 1, sweep0=state["step"], nblock=state["case"]["nblock"], n_acc_local=state["n_acc"],
                       n_acc_block=state["n_more"])
        state["step"] += 1
        return dict(x=state["x"], n_local=state["n_acc"], n_block=state["n_more"])
    J, resid = ctx.fit_eff(state["x"], state["lnw"])
    return dict(J=J, resid=resid)


def _det_flops(N, Lx, Ly, L, n_s, green):
    """Stabilised determinant of one field: separable slice products, then per group QR, Q and T, then the
    final LU (and, for G, the solve)."""
    groups = -(-L // n_s)
    return 2.0 * N * N * (Lx + Ly) * L + groups * (4 / 3 + 4 / 3 + 1) * N ** 3 + (2 / 3 + (2 if green else 0)) * N ** 3


# operations of one Metropolis decision of E_eff, a random number, the energy difference and the test among them
_SITE_FLOPS = 60.0


def work(case):
    kind, n = case["kind"], case["n"]
    if kind == "batch":
        b = f = 0.0
        for s, L in _sizes(case):
            N = s * s
            b += n * 16.0 * N * L
            f += n * (_det_flops(N, s, s, L, case["n_s"], False) + case["nsweeps"] * N * L * _SITE_FLOPS)
        return {"bytes": b, "flops": f}
    Lx, Ly, L = case["Lx"], case["Ly"], case["L"]
    N = Lx * Ly
    if kind == "greens":
        return {"bytes": 8.0 * n * (N * L + N * N + 3), "flops": n * _det_flops(N, Lx, Ly, L, case["n_s"], True)}
    if kind == "log_weight":
        return {"bytes": 8.0 * n * (N * L + 3), "flops": n * _det_flops(N, Lx, Ly, L, case["n_s"], False)}
    if kind == "update":
        return {"bytes": n * (16.0 * N * L + 64),
                "flops": n * (_det_flops(N, Lx, Ly, L, case["n_s"], True) + case["nsweeps"] * N * L * _SITE_FLOPS)}
    if kind == "sweep":
        return {"bytes": n * (16.0 * N * L + 16), "flops": n * case["nsweeps"] * N * L * _SITE_FLOPS}
    if kind == "dqmc":  # per slice the wrap and the rank-1 updates of half the sites; two chains of products
        groups = -(-L // case["n_s"])
        f = L * (4.0 * N * N * (Lx + Ly) + N ** 3) + 2 * _det_flops(N, Lx, Ly, L, case["n_s"], False)
        f += groups * 20 / 3 * N ** 3 + (1 + case["nblock"]) * (case["nblock"] > 0) * _det_flops(N, Lx, Ly, L, case["n_s"], False)
        return {"bytes": n * (16.0 * N * L + 32), "flops": n * f}
    return {"bytes": 8.0 * n * (N * L + 1), "flops": n * N * L * 25.0}


def _line(Ld):
    """The one-dimensional factor exp(dtau h) of a periodic line of Ld sites, h its hopping matrix (t = 1)."""
    h = np.zeros((Ld, Ld))
    for i in range(Ld):
        h[i, (i + 1) % Ld] += 1.0
        h[(i + 1) % Ld, i] += 1.0
    w, v = np.linalg.eigh(h)
    return torch.from_numpy((v * np.exp(DTAU * w)) @ v.T)


def _exact_field(x, Lx, Ly, n_s, green):
    """ln|det(I + B_L ... B_1)|, its sign and G of one field [N, L] (lambda = 1), in plain torch FP64: the
    product kept as U D T, refactored every n_s slices with its columns ordered by norm."""
    N, L = x.shape
    ex, ey = _line(Lx), _line(Ly)
    s = torch.exp(-DTAU * x)
    U, T, D = torch.eye(N, dtype=torch.float64), torch.eye(N, dtype=torch.float64), torch.ones(N, dtype=torch.float64)
    for l0 in range(0, L, n_s):
        for l in range(l0, min(L, l0 + n_s)):
            Y = torch.matmul(ex, U.view(Ly, Lx, N))
            U = torch.matmul(ey, Y.reshape(Ly, Lx * N)).view(N, N) * s[:, l, None]
        M = U * D
        p = torch.argsort(M.norm(dim=0), descending=True)
        U, R = torch.linalg.qr(M[:, p])
        D = R.diagonal().abs().clone()
        T = (R / D[:, None]) @ T[p]
    b, d = torch.clamp(D, min=1.0), torch.clamp(D, max=1.0)
    M = U.T / b[:, None] + d[:, None] * T
    sU, sM = torch.linalg.slogdet(U), torch.linalg.slogdet(M)
    G = torch.linalg.solve(M, U.T / b[:, None]) if green else None
    return (b.log().sum() + sM[1]).item(), int(round((sU[0] * sM[0]).item())), G


def _exact_bose(x):
    """dtau (lambda sum x - S_Bose) of each field of a batch (lambda = omega0 = 1)."""
    d = torch.roll(x, -1, 2) - x
    return DTAU * (x - 0.5 * x * x - d * d / (2.0 * DTAU * DTAU)).sum(dim=(1, 2))


def _exact_det(case, x, green):
    def one(f):
        torch.set_num_threads(1)  # one field per thread, as many threads as cores
        return _exact_field(x[f], case["Lx"], case["Ly"], case["n_s"], green)

    threads = torch.get_num_threads()
    try:
        with ThreadPoolExecutor(os.cpu_count()) as pool:
            return list(pool.map(one, range(case["n"])))
    finally:
        torch.set_num_threads(threads)


def exact(case, seed):
    """What run() returns for these inputs, in plain torch FP64. The states of Markov chains (update, sweep,
    batch, dqmc) are decided draw by draw by the package's own random streams and have no such value."""
    kind = case["kind"]
    if kind == "fit":
        x, lnw = _scored(case, seed)
        F, y = _features(x, case["Lx"], case["Ly"]).cpu().numpy(), lnw.cpu().numpy()
        mean, std = F.mean(0), F.std(0)
        A = np.concatenate([np.ones((len(y), 1)), (F - mean) / std], axis=1)
        c = np.linalg.lstsq(A, y - y.mean(), rcond=None)[0]
        resid = np.sqrt(np.mean((A @ c - (y - y.mean())) ** 2))
        slope = c[1:] / std
        J = -np.concatenate([[c[0] + y.mean() - slope @ mean], slope]) / DTAU
        return dict(J=J, resid=np.array([resid]))
    if kind not in ("greens", "log_weight"):
        return None
    x = _fields(case["n"], case["Lx"], case["Ly"], case["L"], seed).cpu()
    green = kind == "greens"
    got = _exact_det(case, x, green)
    lndet, sign = torch.tensor([g[0] for g in got], dtype=torch.float64), torch.tensor([g[1] for g in got], dtype=torch.int32)
    if not green:
        return dict(lnw=2.0 * lndet + _exact_bose(x), lndet=lndet, sign=sign)
    G = torch.stack([g[2] for g in got])
    N, Lx = x.shape[1], case["Lx"]
    i = torch.arange(N)
    st = 1.0 - 2.0 * ((i % Lx + i // Lx) % 2).double()
    g = torch.diagonal(G, dim1=1, dim2=2)
    GG = torch.einsum("i,j,fij,fji->f", st, st, G, G)
    S = (4.0 * ((st * (1.0 - g)).sum(1)) ** 2 + 2.0 * g.sum(1) - 2.0 * GG) / N
    return dict(G=G, lndet=lndet, sign=sign, S=S)
