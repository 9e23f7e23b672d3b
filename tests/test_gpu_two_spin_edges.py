"""The refinement in the two-spin sweep (either spin with its own refinement, or
spin down mirrored, with G in shared memory or in HBM), and initial matrices
shared by clusters of every size, against the FP64 oracle.

Tolerances are those of the one-spin tests: a refined FP32 G lies within four
FP32 roundings of the oracle's G for the same field (+ 1e-9); an initial FP32 G
is the FP64 inverse rounded once (2^-24 of the largest entry, + 1e-10 of it)."""
import numpy as np
import pytest

from gpu_common import lib

pytestmark = pytest.mark.gpu


def _bath(beta, L, doped):
    from paper_0801_1222_gb300 import inputs
    g0 = inputs.bethe_G0_tau(beta, L)
    return g0 * np.exp(-0.3 * np.arange(L) / L) if doped else g0


def _check_refined(orc, ctx, g0, L, U, dtau):
    M, lam = orc.bath_matrix(g0), orc.lam(dtau, U)
    ch = ctx.get_chain(0, 0)
    for sig, G in ((1, ch["Gup"]), (-1, ch["Gdn"])):
        Gx, _ = orc.green(M, ch["s"], lam, sig)
        r = np.max(np.abs(Gx.astype(np.float32).astype(np.float64) - Gx))
        assert np.max(np.abs(G - Gx)) <= 4.0 * r + 1e-9, (L, sig)


# spin down: refined (doped, or the symmetry never used) or mirrored
@pytest.mark.parametrize("doped,ph", [(True, 0), (False, -1), (False, 1)])
@pytest.mark.parametrize("L", [17, 64, 100, 128, 129, 240, 257, 500])
def test_refined_G_of_both_spins(orc, L, doped, ph):
    U, dtau = 4.5, 0.1
    g0 = _bath(dtau * L, L, doped)

    # a recompute after every flip: the G left behind is a refined one
    ctx = lib().HFQMC(dtau * L, U, [dtau], [1], seed=5, n_wrap=1, drift_fail=1e30, recompute="refine", ph_symmetry=ph)
    ctx.set_G0(0, g0)
    ctx.sweep(0, 1)
    st = ctx.get_stats(0)
    assert st["recompute_fallbacks"] == 0 and st["ph_symmetric"] == (not doped and ph >= 0)
    assert st["recomputes"] == st["accepted"] > 0
    _check_refined(orc, ctx, g0, L, U, dtau)
    ctx.close()


# chain counts for clusters of 8 down to 1 CTA per matrix, uneven column shares
# among them; above 152 matrices the mirrored form with one CTA each
@pytest.mark.parametrize("doped", [False, True])
@pytest.mark.parametrize("L", [259, 300])
def test_initial_G_of_every_cluster_size(orc, L, doped):
    U, dtau = 4.5, 0.1
    g0 = _bath(dtau * L, L, doped)
    M, lam = orc.bath_matrix(g0), orc.lam(dtau, U)
    first = None
    for chains in (1, 9, 10, 12, 15, 17, 19, 21, 24, 30, 37, 50, 76, 160):
        ctx = lib().HFQMC(dtau * L, U, [dtau], [chains], seed=3)
        ctx.set_G0(0, g0)
        ch = ctx.get_chain(0, 0)
        ctx.close()
        if first is None:
            first = ch
            for sig, G in ((1, ch["Gup"]), (-1, ch["Gdn"])):
                Gx, _ = orc.green(M, ch["s"], lam, sig)
                assert np.max(np.abs(G - Gx)) <= (2.0 ** -24 + 1e-10) * np.abs(Gx).max(), sig
        # the same operations per entry however many CTAs share the matrix
        assert np.array_equal(ch["s"], first["s"]), chains
        assert np.array_equal(ch["Gup"], first["Gup"]) and np.array_equal(ch["Gdn"], first["Gdn"]), chains
