"""Stack QR of columns whose squared norms approach the largest FP64 number.

A static staggered field at U = 12.1, beta = 40: the product of all B_l stretches
by e^{+-356}, and the last stack step has columns of 1e154 to 1.3e154, whose
squares are finite and twice their squares are not.  The field commutes with
itself along tau, so G(0) = 1 / (1 + B^L) in closed form; G agrees to 1e-10, for
every kernel of the QR (one, four and eight CTAs, panels).
"""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _exact(Lx, Ly, U, dtau, L):
    N = Lx * Ly
    i = np.arange(N)
    x, y = i % Lx, i // Lx
    A = np.zeros((N, N))
    for nb in ((x + 1) % Lx + Lx * y, (x - 1) % Lx + Lx * y, x + Lx * ((y + 1) % Ly), x + Lx * ((y - 1) % Ly)):
        np.add.at(A, (i, nb), 1.0)
    w, v = np.linalg.eigh(A)
    E = (v * np.exp(dtau * 0.25 * w)) @ v.T
    s = np.where((x + y) % 2, -1.0, 1.0)
    h = np.exp(0.5 * math.acosh(math.exp(0.5 * dtau * U)) * s)  # B = E h^2 = h^-1 (h E h) h
    w, v = np.linalg.eigh(h[:, None] * E * h)
    G = (v / (1.0 + np.exp(np.clip(L * np.log(w), -700.0, 700.0)))) @ v.T
    return s.astype(np.int8), G / h[:, None] * h


@pytest.mark.parametrize("Lx,Ly,C,U", [(4, 4, 1, 12.0954), (8, 8, 1, 12.1198), (10, 10, 1, 12.122), (10, 10, 80, 12.122),
                                       (12, 12, 1, 12.122), (14, 12, 1, 12.11), (16, 16, 1, 12.0954), (16, 16, 1, 12.12)])
def test_columns_near_the_end_of_the_range(Lx, Ly, C, U):
    import paper_1504_05090_gb300 as pkg
    g = pkg.Group(Lx=Lx, Ly=Ly, t=0.25, U=U, beta=40.0, dtau=0.25, n_chains=C, stab_interval=3,
                  delay_k=8, precision="fp64")
    s, ref = _exact(Lx, Ly, U, g.dtau, g.L)
    with pkg.DQMC([g], seed=1) as sim:
        sim.set_field([np.broadcast_to(s, (C, g.L, g.N))])
        assert np.max(np.abs(sim.G(C - 1, 0) - ref)) < 1e-10
