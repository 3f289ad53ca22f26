"""Panels of the blocked QR (N > 144) through the stabilised Green functions
that they build.

Sizes at the edges of the panels: last panels of 4, 8 and 32 columns, rows
that are and are not a multiple of a warp; a batch that fills the chip more
than once.  Tolerance: G of a UDV chain agrees with the oracle's to 1e-10
relative, as everywhere in these tests.
"""
import numpy as np
import pytest

from oracle import dqmc as o

pytestmark = pytest.mark.gpu


def _grp(Lx, Ly, C, U=2.0, beta=4.0, dtau=0.125, ns=8, k=8, prec="fp64"):
    import paper_1504_05090_gb300 as pkg
    return pkg.Group(Lx=Lx, Ly=Ly, t=0.25, U=U, beta=beta, dtau=dtau, n_chains=C,
                     stab_interval=ns, delay_k=k, precision=prec)


@pytest.mark.parametrize("Lx,Ly,C", [(16, 10, 2), (14, 12, 1), (16, 12, 1), (14, 14, 3), (16, 14, 1),
                                     (16, 16, 80)])
def test_green_of_every_panel_width_matches_oracle(Lx, Ly, C):
    import paper_1504_05090_gb300 as pkg
    g = _grp(Lx, Ly, C=C)
    p = o.Params(Lx, Ly, 0.25, g.U, g.beta, g.dtau, n_s=g.stab_interval)
    with pkg.DQMC([g], seed=21) as sim:
        for c in sorted({0, C - 1}):
            ref = o.Chain(p, seed=21, chain=c).green(0, 1)
            G = sim.G(c, 0)
            assert np.max(np.abs(G - ref)) < 1e-10 * np.max(np.abs(ref))


@pytest.mark.parametrize("Lx,Ly,beta,dtau,ns", [(16, 10, 10.0, 0.1, 8), (14, 12, 8.0, 0.2, 6)])
def test_blocked_qr_matches_pivoted_qr_above_144(Lx, Ly, beta, dtau, ns):
    """Partial last panels (N = 160: 32 columns, 168: 8), swept fields: G, the
    decisions of a sweep and G(tau) on the column-pivoted QR agree to 1e-10."""
    import paper_1504_05090_gb300 as pkg
    g = _grp(Lx, Ly, C=2, beta=beta, dtau=dtau, ns=ns, k=16)
    with pkg.DQMC([g], seed=7) as a, pkg.DQMC([g], seed=7) as b:
        b.set_qr_mode("pivoted")
        a.sweep(2)
        b.sweep(2)
        b.set_field(a.field())
        a.recompute_G()
        for step in range(2):
            for c in range(2):
                Ga, Gb = a.G(c, 0), b.G(c, 0)
                assert np.max(np.abs(Ga - Gb)) < 1e-10 * np.max(np.abs(Gb)), (step, c)
            if step == 0:
                a.sweep(1)
                b.sweep(1)
                assert np.array_equal(a.field()[0], b.field()[0])
        x, y = a.gtau()[0], b.gtau()[0]
        assert np.max(np.abs(x - y)) < 1e-10 * np.max(np.abs(y))
