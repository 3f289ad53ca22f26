"""Gauss-Jordan inverse in shared memory through what is built from it: the
stabilised G, G(tau) (float-pair elimination in float-pair groups) and log W.

The variants (1, 4 or 8 CTAs per matrix, or the matrix in global memory) are
chosen by the matrices in flight, so they are compared by changing the number
of chains; every element is formed by the same operations, so G agrees bit for
bit and G(tau), whose bins are summed by atomics, to 1e-12 of its maximum.
Against the oracle: 1e-10 relative, as everywhere in these tests.
"""
import numpy as np
import pytest

from oracle import dqmc as o

pytestmark = pytest.mark.gpu


def _grp(Lx, Ly, C, prec="fp64", beta=2.0, dtau=0.125, ns=8):
    import paper_1504_05090_gb300 as pkg
    return pkg.Group(Lx=Lx, Ly=Ly, t=0.25, U=2.0, beta=beta, dtau=dtau, n_chains=C,
                     stab_interval=ns, delay_k=8, precision=prec)


@pytest.mark.parametrize("Lx,Ly,counts", [(8, 6, (1, 90)), (10, 8, (2, 80)), (14, 8, (1, 80)), (16, 8, (1, 80)),
                                          (12, 12, (2, 20, 80)), (14, 14, (2, 40)), (16, 14, (2, 20, 40))])
def test_variants_agree(Lx, Ly, counts):
    import paper_1504_05090_gb300 as pkg
    first = None
    for C in counts:
        with pkg.DQMC([_grp(Lx, Ly, C, prec="df32")], seed=9) as sim:
            got = (sim.G(0, 0), sim.gtau()[0][0], sim.grad()[2][0])
        if first is None:
            first = got
        assert np.array_equal(got[0], first[0])
        assert np.max(np.abs(got[1] - first[1])) < 1e-12 * np.max(np.abs(first[1]))
        assert got[2] == first[2]


@pytest.mark.parametrize("Lx,Ly", [(2, 2), (6, 2), (8, 6), (10, 8), (16, 8), (14, 14), (16, 14)])
@pytest.mark.parametrize("prec", ["fp64", "df32"])
def test_gtau_and_logw_match_oracle(Lx, Ly, prec):
    import paper_1504_05090_gb300 as pkg
    g = _grp(Lx, Ly, C=2, prec=prec)
    p = o.Params(Lx, Ly, 0.25, g.U, g.beta, g.dtau, n_s=g.stab_interval)
    with pkg.DQMC([g], seed=31) as sim:
        ch = o.Chain(p, seed=31, chain=1)
        ref = ch.gtau()
        tol = 1e-10 if prec == "fp64" else 1e-9
        assert np.max(np.abs(sim.gtau()[0][1] - ref)) < tol * np.max(np.abs(ref))
        assert sim.grad()[2][1] == pytest.approx(ch.logw(), rel=1e-10)


@pytest.mark.parametrize("Lx,Ly,counts", [(10, 6, (40, 80)), (8, 8, (40, 80)), (16, 8, (10, 40, 80)),
                                          (16, 14, (10, 30, 60))])
def test_every_chain_agrees_between_variants(Lx, Ly, counts):
    """4 CTAs against one (N <= 144), 8 against 4, 4 against the matrix in global
    memory (N = 224): every chain that the contexts share, U = 4, after a sweep."""
    import paper_1504_05090_gb300 as pkg
    ref = None
    for C in counts:
        g = pkg.Group(Lx=Lx, Ly=Ly, t=0.25, U=4.0, beta=5.0, dtau=0.25, n_chains=C, stab_interval=5,
                      delay_k=8, precision="df32")
        with pkg.DQMC([g], seed=9) as sim:
            sim.sweep(1)
            got = [sim.G(c, 0) for c in range(min(counts))]
            f = sim.field()[0][:min(counts)]
        if ref is None:
            ref, f0 = got, f
        assert np.array_equal(f, f0)
        for x, y in zip(got, ref):
            assert np.array_equal(x, y)
