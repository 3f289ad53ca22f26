"""Slice wrap with the matrix in shared memory: the same numbers as the two
passes over memory, bit for bit, and the oracle's.

Sizes at the edges of its range (N = 4, 24 whatever the batch; N = 32 ... 64
where a group has a chain per SM), against a group too small for it; FP64
sweeps of the small lattices against the oracle, 1e-10 relative as everywhere
in these tests.
"""
import numpy as np
import pytest

from oracle import dqmc as o

pytestmark = pytest.mark.gpu


def _grp(Lx, Ly, prec, C):
    import paper_1504_05090_gb300 as pkg
    return pkg.Group(Lx=Lx, Ly=Ly, t=0.25, U=3.0, beta=1.0, dtau=0.125, n_chains=C,
                     stab_interval=4, delay_k=8, precision=prec)


@pytest.mark.parametrize("prec", ["df32", "fp32"])
@pytest.mark.parametrize("Lx,Ly", [(8, 4), (6, 6), (10, 6), (16, 4), (8, 8)])
def test_one_launch_equals_two_passes(Lx, Ly, prec):
    import paper_1504_05090_gb300 as pkg
    first = None
    for C in (3, 200):
        with pkg.DQMC([_grp(Lx, Ly, prec, C)], seed=29) as sim:
            sim.sweep(2)
            got = (sim.field()[0][:3], sim.stats()[1][:3], sim.G(0, 0), sim.G(2, 1))
        if first is None:
            first = got
        for a, b in zip(got, first):
            assert np.array_equal(a, b)


@pytest.mark.parametrize("Lx,Ly", [(2, 2), (4, 4), (6, 4)])
@pytest.mark.parametrize("prec", ["fp64", "df32"])
def test_small_lattices_match_oracle(Lx, Ly, prec):
    import paper_1504_05090_gb300 as pkg
    g = _grp(Lx, Ly, prec, 2)
    p = o.Params(Lx, Ly, 0.25, g.U, g.beta, g.dtau, n_s=g.stab_interval)
    with pkg.DQMC([g], seed=17) as sim:
        sim.sweep(1)
        ch = o.Chain(p, seed=17, chain=1)
        out = ch.sweep()
        assert np.array_equal(sim.field()[0][1], ch.field)
        G = sim.G(1, 0)
        assert np.max(np.abs(G - out["G_up"])) < 1e-10 * np.max(np.abs(out["G_up"]))
