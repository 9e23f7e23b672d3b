"""How long hfqmc_set_G0 takes against itself at another number of chains, within
one run on one GPU (the best of several calls each): where more matrices of the
same size only fill the SMs further, the time does not jump."""
import time

import numpy as np
import pytest

from gpu_common import lib

pytestmark = pytest.mark.gpu


def _set_ms(L, chains, precision, symmetric):
    from paper_0801_1222_gb300 import inputs
    beta = 0.2 * L
    g0 = inputs.bethe_G0_tau(beta, L)
    if not symmetric:
        g0 = g0 * np.exp(-0.3 * np.arange(L) / L)
    ctx = lib().HFQMC(beta, 4.0, [0.2], [chains], seed=11, precision=precision)
    t = []
    for _ in range(20):
        t0 = time.perf_counter()
        ctx.set_G0(0, g0)
        t.append((time.perf_counter() - t0) * 1e3)
    assert ctx.get_stats(0)["ph_symmetric"] == (symmetric and precision == "f32_delayed")
    ctx.close()
    return min(t[1:])


# two CTAs per chain on 152 SMs: 304 are two per SM, 400 three per SM, whose FP64
# pipe then has half as much again to do: 4/3 of the time on average, 3/2 on the
# fullest SM; in two waves twice
@pytest.mark.parametrize("L", [170, 256])
def test_three_initial_matrices_per_sm(L):
    two, three = (_set_ms(L, chains, "f64_rank1", False) for chains in (152, 200))
    assert three <= 1.65 * two, (two, three)


# a chain more has to take a smaller cluster (3 x 51 and 5 x 31 CTAs are more
# than 152); one less must not take longer because its clusters share SMs
@pytest.mark.parametrize("L,chains", [(100, 50), (200, 50), (256, 30)])
def test_clusters_do_not_share_sms(L, chains):
    here, more = (_set_ms(L, n, "f32_delayed", True) for n in (chains, chains + 1))
    assert here <= 1.12 * more, (here, more)
