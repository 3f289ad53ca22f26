"""Tensor-core products of matrices of at most 64 x 64 through the stabilised
Green functions that they build.

Lattices whose products fill the 64 x 64 tile (N = 64), batches of one and of
more matrices than the chip holds at once, and the small trailing blocks of the
blocked QR (N = 168, 196: K = 32 with 8 and 4 rows).  Tolerance: G of a
UDV chain agrees with the oracle's to 1e-10 relative, as everywhere in these
tests; the products on the FP64 pipe give the same G to that tolerance.
"""
import numpy as np
import pytest

from oracle import dqmc as o

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("Lx,Ly,C,U", [(8, 8, 1, 2.0), (8, 8, 200, 4.0), (16, 4, 3, 0.0),
                                       (14, 12, 1, 2.0), (14, 14, 2, 2.0)])
def test_green_of_small_products_matches_oracle(Lx, Ly, C, U):
    import paper_1504_05090_gb300 as pkg
    g = pkg.Group(Lx=Lx, Ly=Ly, t=0.25, U=U, beta=4.0, dtau=0.125, n_chains=C, stab_interval=8,
                  delay_k=8, precision="fp64")
    p = o.Params(Lx, Ly, 0.25, U, 4.0, 0.125, n_s=8)
    with pkg.DQMC([g], seed=33) as a, pkg.DQMC([g], seed=33) as b:
        b.set_gemm_mode("fp64")
        for c in sorted({0, C - 1}):
            ref = o.Chain(p, seed=33, chain=c).green(0, 1)
            tol = 1e-10 * np.max(np.abs(ref))
            assert np.max(np.abs(a.G(c, 0) - ref)) < tol
            assert np.max(np.abs(b.G(c, 0) - ref)) < tol
