"""Metropolis pass: which thread or CTA forms which entry of a flip's vectors
must not matter.

Sizes at the edges of the thread layout: one warp of columns (N = 16, 32), a
ragged last warp (N = 36, 100, 140, 196), the first size whose FP64
corrections are split over the cluster (N = 128) and the largest.  Every
element is formed by the same operations whatever the split, so fields,
accepted counts and G agree bit for bit; against the oracle 1e-10 relative.
"""
import numpy as np
import pytest

from oracle import dqmc as o

pytestmark = pytest.mark.gpu


def _grp(Lx, Ly, prec, k, C=2):
    import paper_1504_05090_gb300 as pkg
    return pkg.Group(Lx=Lx, Ly=Ly, t=0.25, U=3.0, beta=1.0, dtau=0.125, n_chains=C,
                     stab_interval=4, delay_k=k, precision=prec)


@pytest.mark.parametrize("prec", ["fp64", "df32", "fp32"])
@pytest.mark.parametrize("Lx,Ly,k", [(4, 4, 5), (8, 4, 8), (6, 6, 32), (10, 10, 7), (16, 8, 16), (14, 10, 32),
                                     (14, 14, 9), (16, 16, 32)])
def test_split_does_not_change_the_result(Lx, Ly, k, prec):
    import paper_1504_05090_gb300 as pkg
    first = None
    for cs in (1, 2, 4):
        with pkg.DQMC([_grp(Lx, Ly, prec, k)], seed=13) as sim:
            sim.set_metropolis_split(cs)
            sim.sweep(1)
            got = (sim.field()[0], sim.stats()[1], sim.G(1, 0))
        if first is None:
            first = got
        for a, b in zip(got, first):
            assert np.array_equal(a, b)


@pytest.mark.parametrize("Lx,Ly,k", [(4, 2, 3), (8, 4, 8), (16, 8, 16), (14, 10, 32)])
@pytest.mark.parametrize("prec", ["fp64", "df32"])
def test_sweep_matches_oracle(Lx, Ly, k, prec):
    import paper_1504_05090_gb300 as pkg
    g = _grp(Lx, Ly, prec, k)
    p = o.Params(Lx, Ly, 0.25, g.U, g.beta, g.dtau, n_s=g.stab_interval)
    with pkg.DQMC([g], seed=17) as sim:
        sim.sweep(1)
        ch = o.Chain(p, seed=17, chain=1)
        out = ch.sweep()
        assert np.array_equal(sim.field()[0][1], ch.field)
        assert sim.stats()[1][1] == out["accepted"]
        G = sim.G(1, 0)
        assert np.max(np.abs(G - out["G_up"])) < 1e-10 * np.max(np.abs(out["G_up"]))
