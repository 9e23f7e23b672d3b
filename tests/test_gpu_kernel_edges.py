"""The CUDA kernels at the sizes where their tiles, shares and batches end,
against the FP64 oracle, through the C ABI.

Tolerances are the ones of the kernels' other tests: FP64 decisions equal the
oracle's and G agrees to 1e-10 of its largest entry; a refined FP32 G lies
within four FP32 roundings of the oracle's G for the same field (+ 1e-9); an
initial FP32 G is the FP64 inverse rounded once, so it lies within one FP32
rounding (2^-24 of the largest entry) and 1e-10 of it."""
import numpy as np
import pytest

from gpu_common import compare_chains, lib, make_pair

pytestmark = pytest.mark.gpu


# rank-1 sweep: half-warp rows up to 16, chunks of 32 columns, the resident G's limit
@pytest.mark.parametrize("L", [15, 16, 17, 31, 32, 33, 64, 65, 96, 97, 128, 129, 160, 161, 193])
@pytest.mark.parametrize("rule", ["metropolis", "heat_bath"])
def test_rank1_f64_follows_the_oracle(orc, L, rule):
    ctx, q = make_pair(orc, 0.125 * L, [(4.0, 0.125)], [2], n_wrap=7, accept_rule=rule)
    ctx.sweep(1, 2)
    q.sweep(1, 2)
    compare_chains(ctx, q)


# the same kernel in FP32 takes u < R as t(u) <= R on floats
@pytest.mark.parametrize("L", [16, 17, 33, 64, 128, 193])
@pytest.mark.parametrize("rule", ["metropolis", "heat_bath"])
def test_rank1_f32_follows_the_oracle(orc, L, rule):
    ctx, q = make_pair(orc, 0.125 * L, [(4.0, 0.125)], [4], n_wrap=16, accept_rule=rule, precision="f32_rank1",
                       drift_fail=1.0)
    ctx.sweep(1, 0)
    q.sweep(1, 0)
    same = [c for c, och in enumerate(q.chains[0]) if ctx.get_chain(0, c)["hash"] == och.decision_hash]
    assert len(same) >= 3
    for c in same:
        ch, och = ctx.get_chain(0, c), q.chains[0][c]
        assert np.array_equal(ch["s"], och.s)
        assert np.abs(ch["Gup"] - och.Gup).max() < 1e-3 and np.abs(ch["Gdn"] - och.Gdn).max() < 1e-3


# refinement: core matrices of 8, tiles of 64 rows and 128 columns, K steps of 16 and 32
@pytest.mark.parametrize("L", [15, 16, 17, 33, 63, 64, 65, 127, 128, 129, 192, 193, 255, 256, 257, 511, 512])
def test_refined_G_at_tile_edges(orc, L):
    beta = 0.1 * L
    # a recompute after every flip: the G left behind is a refined one
    ctx, q = make_pair(orc, beta, [(4.5, beta / L)], [1], precision="f32_delayed", n_wrap=1, drift_fail=1.0,
                       recompute="refine", seed=5)
    ctx.sweep(0, 1)
    st = ctx.get_stats(0)
    assert st["recomputes"] == st["accepted"] > 0 and st["recompute_fallbacks"] == 0
    M, lam = q.chains[0][0].M, q.chains[0][0].lmbda
    ch = ctx.get_chain(0, 0)
    for sig, G in ((1, ch["Gup"]), (-1, ch["Gdn"])):
        Gx, _ = orc.green(M, ch["s"], lam, sig)
        r = np.max(np.abs(Gx.astype(np.float32).astype(np.float64) - Gx))
        assert np.max(np.abs(G - Gx)) <= 4.0 * r + 1e-9, (L, sig)


# Green matrices of one field: 8 shares of each spin in shared memory, and beyond it
@pytest.mark.parametrize("L", [1, 2, 7, 8, 9, 31, 33, 64, 100, 156, 158, 159, 160, 200])
def test_noalloc_shares(orc, L):
    import torch

    from paper_0801_1222_gb300 import inputs
    h = lib()
    dtau, U = 0.2, 5.0
    g0 = inputs.bethe_G0_tau(dtau * L, L)
    s = np.where(np.random.default_rng(L).random(L) < 0.5, 1, -1).astype(np.int8)
    g0_d, s_d = torch.from_numpy(g0).cuda(), torch.from_numpy(s).cuda()
    out = [torch.full((L, L), np.nan, dtype=torch.float64, device="cuda") for _ in range(2)]
    assert h.hfqmc_green_noalloc(g0_d.data_ptr(), s_d.data_ptr(), L, dtau, U, out[0].data_ptr(),
                                 out[1].data_ptr(), 0) == 0
    torch.cuda.synchronize()
    M, lam = orc.bath_matrix(g0), orc.lam(dtau, U)
    for sig, G in ((1, out[0]), (-1, out[1])):
        Gx, _ = orc.green(M, s, lam, sig)
        assert np.max(np.abs(G.cpu().numpy() - Gx)) <= 1e-10 * np.abs(Gx).max()


# the initial G: clusters of 1, 2, 4 or 8 CTAs per matrix (by the number of
# chains and L), panels of 16 with a remainder, spin down mirrored or inverted
@pytest.mark.parametrize("mu", [0.0, 0.3])
@pytest.mark.parametrize("precision", ["f32_delayed", "f64_rank1"])
@pytest.mark.parametrize("L", [16, 63, 64, 127, 128, 193, 256, 257, 511])
def test_initial_G_by_clusters(orc, L, precision, mu):
    from paper_0801_1222_gb300 import inputs
    h = lib()
    beta, U = 0.1 * L, 4.5
    g0 = inputs.bethe_G0_tau(beta, L)
    if mu:
        g0 = g0 * np.exp(-mu * np.arange(L) / L)  # not symmetric under tau -> beta - tau
    got = []
    for chains in (1, 40, 200):
        if chains == 200 and L > 257:
            continue
        ctx = h.HFQMC(beta, U, [beta / L], [chains], seed=3, precision=precision)
        ctx.set_G0(0, g0)
        got.append([ctx.get_chain(0, c) for c in sorted({0, chains - 1})])
        ctx.close()
    M, lam = orc.bath_matrix(g0), orc.lam(beta / L, U)
    tol = 1e-10 if precision == "f64_rank1" else 2.0 ** -24 + 1e-10
    for chs in got:
        for ch in chs:
            for sig, G in ((1, ch["Gup"]), (-1, ch["Gdn"])):
                Gx, _ = orc.green(M, ch["s"], lam, sig)
                assert np.max(np.abs(G - Gx)) <= tol * np.abs(Gx).max(), (L, sig)
    # the same operations per entry however many CTAs share the matrix
    for chs in got[1:]:
        assert np.array_equal(chs[0]["s"], got[0][0]["s"])
        assert np.array_equal(chs[0]["Gup"], got[0][0]["Gup"]) and np.array_equal(chs[0]["Gdn"], got[0][0]["Gdn"])
