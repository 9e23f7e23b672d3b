"""The calls a user of this library makes, with the sizes they are made at.

Most cases are one impurity solve, the unit every DMFT loop repeats: the bath
is set on every grid (set_G0, which rebuilds each chain's G), the chains sweep,
and G(tau), D, their error bars and the counters are read back per grid.  Two
cases go through other entry points: a whole iteration of the batched
multigrid DMFT loop, and the Green function of one field without allocation.

Grids, chains, U and beta are those of the library's workloads
(paper_0801_1222_gb300/inputs.py) or lie between them; the number of sweeps
per pass is cut so that a pass takes from about a millisecond to a second.
"""
import math

import numpy as np
import torch

from paper_0801_1222_gb300 import dmft, hfqmc, inputs

# Philox4x32-10 (the library's documented generator): multipliers and Weyl constants
_M0, _M1, _W0, _W1 = 0xD2511F53, 0xCD9E8D57, 0x9E3779B9, 0xBB67AE85


def _solve(name, L, chains, beta, U, warm, meas, precision="f32_delayed", k=0, n_wrap=0,
           rule="metropolis", mu=0.0):
    return {"name": name, "kind": "solve", "L": L, "chains": chains, "beta": beta, "U": U, "warm": warm,
            "meas": meas, "precision": precision, "k": k, "n_wrap": n_wrap, "rule": rule, "mu": mu}


def listed():
    return [
        # the smallest call: one FP64 chain on a coarse grid (workload single_L16)
        _solve("single_L16_f64", "16", "1", 8.0, "4.0", 50, 500, precision="f64_rank1"),
        # one grid with G on chip, the conventional fixed-dtau solve (workload fixed_L100)
        _solve("fixed_L100", "100", "256", 20.0, "5.0", 50, 500, k=16),
        # the headline: all grids of a multigrid solve at once (workload multigrid_L100_240)
        _solve("multigrid_L100_240", "100,120,140,160,200,240", "64,64,64,64,64,64", 40.0, "5.0", 50, 500),
        # the same with the long recompute interval, G(tau) then within 1e-5 of FP64
        _solve("multigrid_long_wrap", "100,120,140,160,200,240", "64,64,64,64,64,64", 40.0, "5.0", 50, 500,
               n_wrap=16384),
        # low temperature, fine grid: the largest matrices (workload large_L500)
        _solve("large_L500", "500", "128", 50.0, "4.8", 4, 40, k=64, n_wrap=64),
        # the ten to twenty solutions per grid of a conventional run: fewer chains than SMs
        _solve("few_chains_L200", "200", "16", 40.0, "5.0", 20, 200),
        # a bath without particle-hole symmetry (doped): both spins are swept
        _solve("doped_L100_240", "100,160,240", "50,50,50", 20.0, "4.0", 20, 200, mu=0.5),
        # ragged grids (no multiple of four), few slices, heat bath, a short interval
        _solve("ragged_heat_bath", "37,90,133", "40,40,40", 16.0, "4.0", 50, 500, n_wrap=32, rule="heat_bath"),
        # the FP64 path over the multigrid range: the reference run a user checks FP32 against
        _solve("f64_L100_240", "100,160,240", "51,51,50", 40.0, "5.0", 1, 9, precision="f64_rank1"),
        # FP32 with plain rank-1 updates
        _solve("f32_rank1_L64_128", "64,128", "76,76", 20.0, "4.0", 20, 200, precision="f32_rank1"),
        # one whole DMFT iteration of four U values on six grids, 1024 chains (workload dmft_c5)
        {"name": "dmft_iteration", "kind": "dmft", "L": "80,120,160,200,240,320", "chains": "42,42,42,42,42,46",
         "beta": 40.0, "U": "4.6,4.8,5.0,5.2", "warm": 20, "meas": 200},
        # G of one field into the caller's buffers, nothing allocated
        {"name": "green_L100", "kind": "green", "L": "100", "beta": 20.0, "U": "5.0"},
    ]


def _ints(text):
    return [int(v) for v in text.split(",")]


def _loguniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _us_per_proposal(L, precision, n_wrap):
    """Rough time of one proposal of one chain on one SM, for choosing sweep counts."""
    if precision == "f64_rank1":
        return 2.0 + 0.8e-3 * L * L
    if precision == "f32_rank1":
        return 2.0 + 0.2e-3 * L * L
    every = 64.0 / max(n_wrap, 16) if n_wrap else 1.0
    return 1.1 + 1.2 * every * (L / 230.0) ** 3


def draw(rng):
    kind = rng.choice(["half", "half", "half", "half", "doped", "rank1", "rank1", "green"])
    if kind == "green":
        L = int(_loguniform(rng, 8, 256.99))
        return {"kind": "green", "L": str(L), "beta": round(L * rng.uniform(0.1, 0.4), 3),
                "U": "%.2f" % rng.uniform(3.0, 5.2)}
    precision = "f32_delayed"
    lo, hi = 16, 512
    if kind == "rank1":
        precision = rng.choice(["f64_rank1", "f64_rank1", "f32_rank1"])
        hi = 256
    n = rng.choice([1, 1, 2, 3, 6])
    Ls = sorted(int(_loguniform(rng, lo, hi + 0.99)) for _ in range(n))
    if rng.random() < 0.6:  # most grids in use are multiples of four
        Ls = [max(16, L // 4 * 4) for L in Ls]
    per = max(1, int(_loguniform(rng, 1, 300 if precision == "f32_delayed" else 150) / n))
    n_wrap = rng.choice([0, 0, 0, 16, 32, 64, 8192]) if precision == "f32_delayed" else 0
    target = _loguniform(rng, 5e3, 2e5)  # microseconds
    chain_us = sum(per * L * _us_per_proposal(L, precision, n_wrap) for L in Ls)
    one = max(chain_us / 152.0, max(L * _us_per_proposal(L, precision, n_wrap) for L in Ls))
    sweeps = int(min(400, max(4, target / one)))
    warm = sweeps // 10
    beta = round(max(Ls) * rng.uniform(0.1, 0.25), 2)
    beta = max(beta, round(min(Ls) * 0.1, 2))
    # no grid coarser than dtau = 0.5, as in the workloads
    beta = min(beta, 0.5 * min(Ls))
    return {"kind": "solve", "L": ",".join(map(str, Ls)), "chains": ",".join([str(per)] * n), "beta": beta,
            "U": "%.2f" % rng.uniform(3.0, 5.2), "warm": warm, "meas": sweeps - warm, "precision": precision,
            "k": rng.choice([0, 0, 0, 8, 16, 32, 64]) if precision == "f32_delayed" else 0, "n_wrap": n_wrap,
            "rule": rng.choice(["metropolis", "metropolis", "heat_bath"]),
            "mu": round(rng.uniform(0.2, 0.8), 2) if kind == "doped" else 0.0}


def _bath(beta, L, mu, seed):
    """G0(tau_k) of a semi-elliptic bath (half-width about 2, drawn from the
    seed) at chemical potential mu: Gauss-Chebyshev quadrature of
    -rho(e) e^{-(e - mu) tau} / (1 + e^{-beta (e - mu)})."""
    D = 1.9 + 0.2 * np.random.RandomState(seed % (1 << 31)).rand()
    n = 400
    th = np.arange(1, n + 1) * np.pi / (n + 1)
    e, w = D * np.cos(th) - mu, 2.0 / (n + 1) * np.sin(th) ** 2
    tau = (np.arange(L) * (beta / L))[:, None]
    a = np.where(e > 0, -e * tau, e * (beta - tau))
    return -(np.exp(a) / (1.0 + np.exp(-beta * np.abs(e)))) @ w


def _context(case, seed):
    Ls, ch = _ints(case["L"]), _ints(case["chains"])
    Us = [float(u) for u in case["U"].split(",")]
    return hfqmc.HFQMC(case["beta"], [u for u in Us for _ in Ls], [case["beta"] / L for L in Ls] * len(Us),
                       ch * len(Us), seed=seed, precision=case.get("precision", "f32_delayed"),
                       k=case.get("k", 0), n_wrap=case.get("n_wrap", 0),
                       accept_rule=case.get("rule", "metropolis"), drift_fail=1e30)


def _field(L, seed):
    return np.where(np.random.RandomState((seed + 1) % (1 << 31)).rand(L) < 0.5, 1, -1).astype(np.int8)


def prepare(case, seed):
    if case["kind"] == "green":
        L = int(case["L"])
        return {"case": case, "L": L, "G0": torch.from_numpy(_bath(case["beta"], L, 0.0, seed)).cuda(),
                "s": torch.from_numpy(_field(L, seed)).cuda(),
                "Gup": torch.empty(L, L, dtype=torch.float64, device="cuda"),
                "Gdn": torch.empty(L, L, dtype=torch.float64, device="cuda")}
    state = {"case": case, "ctx": _context(case, seed)}
    if case["kind"] == "solve":
        state["baths"] = [_bath(case["beta"], L, case["mu"], seed) for L in _ints(case["L"])]
    return state


def run(state):
    case = state["case"]
    if case["kind"] == "green":
        hfqmc.hfqmc_green_noalloc(state["G0"].data_ptr(), state["s"].data_ptr(), state["L"],
                                  case["beta"] / state["L"], float(case["U"]), state["Gup"].data_ptr(),
                                  state["Gdn"].data_ptr(), torch.cuda.current_stream().cuda_stream)
        return [state["Gup"], state["Gdn"]]
    ctx = state["ctx"]
    if case["kind"] == "dmft":
        Ls = _ints(case["L"])
        loop = dmft.BatchedMultigridDMFT(ctx, case["beta"], [float(u) for u in case["U"].split(",")],
                                         [case["beta"] / L for L in Ls], ph_symmetric=True)
        recs = loop.iterate(case["warm"], case["meas"])
        acc = [ctx.get_stats(g)["accepted"] for g in range(ctx.n_grids)]
        return {"U": [[r["G_fine"].astype(np.float32), r["G_err"].astype(np.float32),
                       r["G_iw"].astype(np.complex64), np.float32(r["D"]), np.float32(r["D_err"]),
                       np.asarray(r["D_grids"], dtype=np.float32)] for r in recs],
                "accepted": np.asarray(acc, dtype=np.int64)}
    for g, b in enumerate(state["baths"]):
        ctx.set_G0(g, b)
    ctx.sweep(case["warm"], case["meas"])
    # the estimates of an FP32 path in its own working precision
    f = np.float64 if case["precision"] == "f64_rank1" else np.float32
    out = []
    for g in range(ctx.n_grids):
        G, E = ctx.get_G(g)
        D, dD = ctx.get_D(g)
        st = ctx.get_stats(g)
        out.append([G.astype(f), E.astype(f), np.asarray([D, dD], dtype=f),
                    np.asarray([st["proposals"], st["accepted"], st["recomputes"], st["numeric_errors"]],
                               dtype=np.int64)])
    return out


def work(case):
    """What one pass cannot do without: the rank-1 update of every accepted
    flip (2 L^2 multiply-adds per spin; one spin when G_dn = 1 - G_up^T) with
    about 0.4 of the proposals accepted, a residual and an update product per
    recompute and spin, one inversion per chain and spin for the new bath;
    each chain's G read and written once, the baths in, the estimates out."""
    if case["kind"] == "green":
        L = int(case["L"])
        return {"bytes": 16.0 * L * L + 9.0 * L, "flops": 2 * 2.0 * L ** 3}
    precision, n_wrap = case.get("precision", "f32_delayed"), case.get("n_wrap", 0)
    sweeps = case["warm"] + case["meas"]
    spins = 1 if precision == "f32_delayed" and case.get("mu", 0.0) == 0.0 else 2
    every = n_wrap or (64 if precision == "f32_delayed" else 16384)
    size = 8 if precision == "f64_rank1" else 4
    flops = bytes_ = 0.0
    for L, c in zip(_ints(case["L"]), _ints(case["chains"])):
        flips = 0.4 * sweeps * L * c
        flops += spins * (flips * 2.0 * L * L + flips / every * 4.0 * L ** 3) + c * 2 * 2.0 * L ** 3
        bytes_ += c * 2 * 2.0 * L * L * size + 8.0 * L + 16.0 * (L + 1)
    m = len(case["U"].split(","))
    return {"bytes": m * bytes_, "flops": m * flops}


# ---------------------------------------------------------------------------
# The same outputs in 64 bits: every chain of a grid in lockstep, one rank-1
# update per proposal, G rebuilt from the field by a linear solve now and then.
# ---------------------------------------------------------------------------
def _philox(l, t, c, g, seed):
    x0, x1, x2, x3 = np.broadcast_arrays(*(np.asarray(v, dtype=np.uint64) for v in (l, t, c, g)))
    k0, k1 = seed & 0xffffffff, (seed >> 32) & 0xffffffff
    lo, s32 = np.uint64(0xffffffff), np.uint64(32)
    for r in range(10):
        if r:
            k0, k1 = (k0 + _W0) & 0xffffffff, (k1 + _W1) & 0xffffffff
        p0, p1 = np.uint64(_M0) * x0, np.uint64(_M1) * x2
        x0, x1, x2, x3 = (p1 >> s32) ^ x1 ^ np.uint64(k0), p1 & lo, (p0 >> s32) ^ x3 ^ np.uint64(k1), p0 & lo
    return x0, x1


def _bath_matrix(G0):
    L = G0.shape[0]
    d = np.arange(L)[:, None] - np.arange(L)[None, :]
    return np.where(d >= 0, -G0[d % L], G0[d % L])


def _green(M, lam, s):
    """[1 + (1 - M)(e^{sigma lambda s} - 1)]^{-1} M for both spins; s: chains x L."""
    out = []
    eye = torch.eye(M.shape[0], dtype=torch.float64, device=M.device)
    for sig in (1, -1):
        d = torch.exp(sig * lam * s) - 1.0
        out.append(torch.linalg.solve(eye + (eye - M) * d[:, None, :], M.expand(s.shape[0], -1, -1)))
    return torch.stack(out)


def _exact_grid(case, seed, g, L, C, U):
    dev = "cuda"
    warm, meas = case["warm"], case["meas"]
    lam = math.acosh(math.exp(0.5 * case["beta"] / L * U))
    M = torch.from_numpy(_bath_matrix(_bath(case["beta"], L, case["mu"], seed))).to(dev)
    l, c = np.arange(L)[None, :], np.arange(C)[:, None]
    x0, _ = _philox(l | (1 << 16), 0, c, g, seed)
    s = torch.from_numpy(np.where(x0 & np.uint64(1), 1.0, -1.0)).to(dev)
    G = _green(M, lam, s)
    r = (torch.arange(L, device=dev)[None, :] + torch.arange(L, device=dev)[:, None])
    flat = ((r % L) * L + torch.arange(L, device=dev)[None, :]).reshape(-1)
    sgn = torch.where(r >= L, -1.0, 1.0).double()
    sig = torch.tensor([[1.0], [-1.0]], dtype=torch.float64, device=dev)
    gk = torch.zeros(C, L, dtype=torch.float64, device=dev)
    dd = torch.zeros(C, dtype=torch.float64, device=dev)
    bins, bind, cnt = torch.zeros(32, L, dtype=torch.float64, device=dev), [0.0] * 32, [0] * 32
    for sw in range(warm + meas):
        x0, x1 = _philox(l, sw, c, g, seed)
        if case["precision"] == "f32_delayed":
            u = (x0 >> np.uint64(8)).astype(np.float64) / 16777216.0
        else:
            u = ((x0 >> np.uint64(5)).astype(np.float64) * 67108864.0 + (x1 >> np.uint64(6))) / 9007199254740992.0
        u = torch.from_numpy(u).to(dev)
        if sw and sw % 10 == 0:
            G = _green(M, lam, s)
        for i in range(L):
            dl = torch.expm1(-2.0 * lam * sig * s[:, i])
            R1 = 1.0 + (1.0 - G[:, :, i, i]) * dl
            R = R1[0] * R1[1]
            ok = (u[:, i] < R) if case["rule"] == "metropolis" else (u[:, i] * (1.0 + R) < R)
            f = torch.where(ok, dl / R1, 0.0)
            col = G[:, :, :, i].clone()
            col[:, :, i] -= 1.0
            row = G[:, :, i, :] * f[:, :, None]
            G.view(2 * C, L, L).baddbmm_(col.view(2 * C, L, 1), row.view(2 * C, 1, L))
            s[:, i] = torch.where(ok, -s[:, i], s[:, i])
        if sw >= warm:
            gs = (G.view(2, C, L * L)[:, :, flat].view(2, C, L, L) * sgn).sum(-1).mean(0) / L
            n = 1.0 - G.diagonal(dim1=2, dim2=3)
            d1 = (n[0] * n[1]).mean(-1)
            gk += gs
            dd += d1
            b = (32 * (sw - warm)) // meas
            bins[b] += gs[0]
            bind[b] += float(d1[0])
            cnt[b] += 1
    means = (-gk / meas).cpu().numpy()
    dmean = (dd / meas).cpu().numpy()
    if C == 1:
        used = [b for b in range(32) if cnt[b]]
        sm = np.stack([-bins[b].cpu().numpy() / cnt[b] for b in used])
        sd = np.array([bind[b] / cnt[b] for b in used])
    else:
        sm, sd = means, dmean
    Gt = means.mean(0)
    err = sm.std(0, ddof=1) / math.sqrt(len(sm)) if len(sm) > 1 else np.full(L, np.nan)
    derr = sd.std(ddof=1) / math.sqrt(len(sd)) if len(sd) > 1 else np.nan
    return [np.append(Gt, -1.0 - Gt[0]), np.append(err, err[0]), np.asarray([dmean.mean(), derr]), None]


def exact(case, seed):
    if case["kind"] == "green":
        L = int(case["L"])
        lam = math.acosh(math.exp(0.5 * case["beta"] / L * float(case["U"])))
        G = _green(torch.from_numpy(_bath_matrix(_bath(case["beta"], L, 0.0, seed))), lam,
                   torch.from_numpy(_field(L, seed).astype(np.float64))[None, :])
        return [G[0, 0], G[1, 0]]
    if case["kind"] == "dmft":
        return None  # 1024 chains: minutes in 64 bits
    Ls, ch = _ints(case["L"]), _ints(case["chains"])
    sweeps = case["warm"] + case["meas"]
    seconds = sum(sweeps * L * (2.5e-4 + c * 4.0 * L * L * 8 / 3e12) for L, c in zip(Ls, ch))
    if seconds > 14.0:
        return None
    return [_exact_grid(case, seed, g, L, c, float(case["U"])) for g, (L, c) in enumerate(zip(Ls, ch))]
