"""Column-pivoted QR in shared memory (N <= 144) through the stabilised Green
functions that it builds.

Sizes at its edges: the smallest matrix, sizes that are no multiple of the four
lanes per column or the eight columns per warp, the last size of every variant
(16, 36, 64, 104 -> 100, 144) and the first after it.  Tolerance: G of a UDV
chain agrees with the oracle's to 1e-10 relative, as everywhere in these tests.
"""
import numpy as np
import pytest

from oracle import dqmc as o

pytestmark = pytest.mark.gpu


def _grp(Lx, Ly, C, U=2.0, beta=4.0, dtau=0.125, ns=8, k=8, prec="fp64"):
    import paper_1504_05090_gb300 as pkg
    return pkg.Group(Lx=Lx, Ly=Ly, t=0.25, U=U, beta=beta, dtau=dtau, n_chains=C,
                     stab_interval=ns, delay_k=k, precision=prec)


@pytest.mark.parametrize("Lx,Ly", [(2, 2), (4, 2), (4, 4), (6, 4), (6, 6), (10, 4), (10, 6), (8, 8),
                                   (14, 6), (10, 10), (14, 8), (16, 8), (14, 10), (12, 12), (16, 10)])
def test_green_of_every_size_class_matches_oracle(Lx, Ly):
    import paper_1504_05090_gb300 as pkg
    g = _grp(Lx, Ly, C=2)
    p = o.Params(Lx, Ly, 0.25, g.U, g.beta, g.dtau, n_s=g.stab_interval)
    with pkg.DQMC([g], seed=21) as sim:
        ref = o.Chain(p, seed=21, chain=1).green(0, 1)
        G = sim.G(1, 0)
        assert np.max(np.abs(G - ref)) < 1e-10 * np.max(np.abs(ref))


@pytest.mark.parametrize("Lx,Ly,counts", [(8, 8, (1, 200)), (10, 8, (2, 60)), (12, 12, (2, 20, 60))])
def test_result_does_not_depend_on_the_ctas_per_matrix(Lx, Ly, counts):
    """1, 4 and 8 CTAs per matrix (chosen by the number of chains) give the same
    numbers bit for bit: the pivots are picked and every sum is formed in the
    same order."""
    import paper_1504_05090_gb300 as pkg
    first = None
    for C in counts:
        with pkg.DQMC([_grp(Lx, Ly, C=C, prec="df32")], seed=5) as sim:
            sim.sweep(1)
            got = (sim.field()[0][0], sim.G(0, 0))
        if first is None:
            first = got
        assert np.array_equal(got[0], first[0]) and np.array_equal(got[1], first[1])


def _layered(rng, count, L, Lx, Ly):
    """Staggered fields with a random sign per slice and fields of a random sign
    per row times one per column: many columns whose norms tie or nearly do."""
    x, y = np.meshgrid(np.arange(Lx), np.arange(Ly))
    out = np.empty((count, L, Ly, Lx), dtype=np.int8)
    for c in range(count):
        if c & 1:
            out[c] = rng.choice([-1, 1], size=(Ly, 1)) * rng.choice([-1, 1], size=(1, Lx))
        else:
            out[c] = rng.choice([-1, 1], size=(L, 1, 1)) * np.where((x + y) % 2, 1, -1)
    return out.reshape(count, L, Lx * Ly)


@pytest.mark.parametrize("Lx,Ly,counts", [(10, 8, (40,)), (10, 10, (40,)), (12, 12, (40, 10))])
def test_pivots_of_graded_symmetric_fields_do_not_depend_on_the_ctas(Lx, Ly, counts):
    """U = 8: columns lose most of their norm in a step, so that norms are summed
    afresh all the time; every chain, bit for bit, against one CTA per matrix."""
    import paper_1504_05090_gb300 as pkg

    def grp(C):
        return _grp(Lx, Ly, C=C, U=8.0, beta=10.0, dtau=0.25, ns=4)

    f = _layered(np.random.default_rng(0), 240, 40, Lx, Ly)
    for b0 in range(0, len(f), 80):
        with pkg.DQMC([grp(80)], seed=0) as sim:
            sim.set_field([f[b0:b0 + 80]])
            ref = [sim.G(c, 0) for c in range(80)]
        for C in counts:
            with pkg.DQMC([grp(C)], seed=0) as sim:
                for q in range(0, 80, C):
                    sim.set_field([f[b0 + q:b0 + q + C]])
                    for c in range(C):
                        assert np.array_equal(sim.G(c, 0), ref[q + c]), (b0, q, c, C)
