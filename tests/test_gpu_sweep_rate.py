"""Between two recomputes a sweep is the same work whatever the recompute is: a
context that refines must not sweep more slowly than one that recomputes by
Gauss-Jordan, whose kernel does not carry the refinement's code (registers
spilled for it cost the accept loop half its speed once).  Compared within one
run on one GPU, the same chains, the best of several calls each, neither
reaching a recompute."""
import numpy as np
import pytest

from gpu_common import lib

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L", [128, 240, 300])
def test_two_spin_sweep_between_recomputes(L):
    from paper_0801_1222_gb300 import inputs
    h = lib()
    beta = 0.2 * L
    g0 = inputs.bethe_G0_tau(beta, L) * np.exp(-0.3 * np.arange(L) / L)  # no particle-hole symmetry: both spins
    ms, left = {}, {}
    for recompute in ("gj", "refine"):
        ctx = h.HFQMC(beta, 4.0, [0.2], [40], seed=11, n_wrap=1 << 24, drift_fail=1e30, recompute=recompute)
        ctx.set_G0(0, g0)
        t = []
        for _ in range(6):
            ctx.sweep(1, 19)
            t.append(ctx.get_stats(0)["last_sweep_ms"])
        st = ctx.get_stats(0)
        assert st["recomputes"] == 0 and not st["ph_symmetric"]
        ms[recompute] = min(t[1:])
        left[recompute] = (st["k"], st["accepted"], ctx.get_chain(0, 39)["hash"])
        ctx.close()
    assert left["gj"] == left["refine"]  # the same delay depth, the same decisions
    assert ms["refine"] <= 1.2 * ms["gj"], ms
