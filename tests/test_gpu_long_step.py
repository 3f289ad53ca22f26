"""Stabilisation intervals over which a stack step stretches vectors far
(dtau = 0.4, n_s = 8: by up to e^21.7): G(tau) carries the rounding of every
step amplified, so it is reproduced only by the same operations.

golden/gtau_long_step.npz holds every fifth row of G(tau) of chain 1 after one
sweep (seed 41, U = 2, two chains) as formed by column-pivoted QR on global
memory (N < 64) or blocked QR with panels of two CTAs, Kronecker products of
eight digits and Gauss-Jordan elimination on global memory.  Another FP64-accurate
way differs by 4e-12 (6 x 6) to 2e-10 (12 x 12) of the maximum here.  Tolerance:
N 2^-52 of the maximum, the bins being sums of N numbers by atomics in any order.
"""
import os

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

GOLDEN = os.path.join(os.path.dirname(os.path.abspath(__file__)), "golden", "gtau_long_step.npz")


@pytest.mark.parametrize("Lx,Ly,prec,beta", [(6, 6, "df32", 20.0), (10, 6, "fp64", 20.0), (8, 8, "df32", 20.0),
                                             (12, 12, "fp64", 8.0), (14, 14, "df32", 8.0)])
def test_gtau_is_reproduced(Lx, Ly, prec, beta):
    import paper_1504_05090_gb300 as pkg
    g = pkg.Group(Lx=Lx, Ly=Ly, t=0.25, U=2.0, beta=beta, dtau=0.4, n_chains=2, stab_interval=8,
                  delay_k=16, precision=prec)
    ref = np.load(GOLDEN)["%dx%d_%s" % (Lx, Ly, prec)]
    with pkg.DQMC([g], seed=41) as sim:
        sim.sweep(1)
        got = sim.gtau()[0][1][::5]
    assert np.max(np.abs(got - ref)) < g.N * 2.0 ** -52 * np.max(np.abs(ref))
