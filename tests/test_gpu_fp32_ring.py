"""Rows of G that the FP32 Metropolis pass copies ahead into a ring in shared
memory: no copy may be under way when G is rewritten by a flush or its slot is
asked for again.

Few accepted flips (U = 8: runs of more than the ring's eight rejected sites)
and many (U = 1), flushes every 3 to 32 flips, one warp of columns to eight.
A row from before a flush would make a wrong G: the drift against the
recomputed G stays at FP32 rounding (1e-4, as in the FP32 test of the sweep),
and fields, accepted counts and G agree bit for bit between runs and splits.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("U", [1.0, 8.0])
@pytest.mark.parametrize("Lx,Ly,k", [(8, 4, 3), (8, 8, 16), (14, 10, 32), (16, 16, 4)])
def test_rows_ahead_survive_flushes_and_skips(Lx, Ly, k, U):
    import paper_1504_05090_gb300 as pkg
    g = pkg.Group(Lx=Lx, Ly=Ly, t=0.25, U=U, beta=2.0, dtau=0.125, n_chains=3, stab_interval=2,
                  delay_k=k, precision="fp32")
    first = None
    for cs in (1, 2, 4, 1):
        with pkg.DQMC([g], seed=19) as sim:
            sim.set_metropolis_split(cs)
            sim.sweep(2)
            got = (sim.field()[0], sim.stats()[1], sim.G(0, 0), sim.G(2, 0))
            assert np.all(sim.stats()[0] < 1e-4), sim.stats()[0]
        if first is None:
            first = got
        for a, b in zip(got, first):
            assert np.array_equal(a, b)
