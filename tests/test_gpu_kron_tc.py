"""Kronecker products with exp(-dtau K) on the tensor cores (UDV stack and G(tau)
propagation, N >= 64).

Sides at the edges of the 128 x 16 x 16 products: both at most 8 (half of the
inner dimension unused), one above 8, 16, and vector counts per CTA that leave
a remainder (10, 12, 14).  The same quantities on the FP64 pipe: G to 1e-11
relative, as the other comparisons of the two; G(tau) against the oracle to
1e-10 of its maximum in FP64 and 1e-9 in float pairs.
"""
import numpy as np
import pytest

from oracle import dqmc as o

pytestmark = pytest.mark.gpu

SIZES = [(8, 8), (16, 4), (4, 16), (10, 8), (12, 6), (14, 6), (10, 10), (16, 16)]


def _grp(Lx, Ly, prec="fp64", C=2):
    import paper_1504_05090_gb300 as pkg
    return pkg.Group(Lx=Lx, Ly=Ly, t=0.25, U=2.0, beta=2.0, dtau=0.125, n_chains=C,
                     stab_interval=7, delay_k=8, precision=prec)


@pytest.mark.parametrize("Lx,Ly", SIZES)
def test_stack_and_gtau_match_the_fp64_pipe(Lx, Ly):
    import paper_1504_05090_gb300 as pkg
    with pkg.DQMC([_grp(Lx, Ly)], seed=3) as a, pkg.DQMC([_grp(Lx, Ly)], seed=3) as b:
        b.set_gemm_mode("fp64")
        for sim in (a, b):
            sim.recompute_G()
        ga, gb = a.G(1, 0), b.G(1, 0)
        assert np.max(np.abs(ga - gb)) < 1e-11 * np.max(np.abs(gb))
        ta, tb = a.gtau()[0], b.gtau()[0]
        assert np.max(np.abs(ta - tb)) < 1e-11 * np.max(np.abs(tb))


@pytest.mark.parametrize("prec,tol", [("fp64", 1e-10), ("df32", 1e-9)])
@pytest.mark.parametrize("Lx,Ly", SIZES[:-1])
def test_gtau_matches_oracle(Lx, Ly, prec, tol):
    import paper_1504_05090_gb300 as pkg
    g = _grp(Lx, Ly, prec)
    with pkg.DQMC([g], seed=5) as sim:
        ref = o.Chain(o.Params(Lx, Ly, 0.25, g.U, g.beta, g.dtau, n_s=g.stab_interval), seed=5, chain=1).gtau()
        assert np.max(np.abs(sim.gtau()[0][1] - ref)) < tol * np.max(np.abs(ref))
