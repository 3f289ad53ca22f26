"""Float-pair Kronecker transforms with packed sums: one or two vectors per
thread (chosen by the vectors per CTA) give the same numbers bit for bit, and
the oracle's.

Sides at the edges of the range (2 and 16, square and long), tiles of one to
sixteen vectors, ragged last tiles (N = 140, 4 x 4 = 16 with 16 vectors).
Tolerance: 1e-10 relative, as everywhere in these tests.
"""
import numpy as np
import pytest

from oracle import dqmc as o

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("Lx,Ly", [(16, 2), (2, 16), (6, 10), (14, 10), (16, 12), (16, 16)])
def test_vectors_per_thread_are_invisible_and_match_oracle(Lx, Ly):
    import paper_1504_05090_gb300 as pkg
    g = pkg.Group(Lx=Lx, Ly=Ly, t=0.25, U=3.0, beta=0.75, dtau=0.125, n_chains=2, stab_interval=3,
                  delay_k=8, precision="df32")
    p = o.Params(Lx, Ly, 0.25, g.U, g.beta, g.dtau, n_s=g.stab_interval)
    ch = o.Chain(p, seed=23, chain=1)
    out = ch.sweep()
    first = None
    for wrap in (1, 2, 4, 8, 16):
        with pkg.DQMC([g], seed=23) as sim:
            sim.set_tiles(0, 4, wrap, 0)
            sim.sweep(1)
            got = (sim.field()[0], sim.G(0, 0), sim.G(1, 0), sim.stats()[0])
        if first is None:
            first = got
            assert np.array_equal(got[0][1], ch.field)
            assert np.max(np.abs(got[2] - out["G_up"])) < 1e-10 * np.max(np.abs(out["G_up"]))
        for a, b in zip(got, first):
            assert np.array_equal(a, b)
