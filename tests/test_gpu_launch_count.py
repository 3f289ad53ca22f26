"""dqmc_launch_count with more matrices than one chunk of the tensor-core
products (256): what each product launches is counted, not a fixed number per
chunk.

16 x 10, one stabilisation point per sweep.  From 256 to 300 chains only the
chunked products launch more.  The five panels of a QR have 18 products; the six
whose sides are all at most 64 (trailing columns of the fourth panel, Q of the
last two) take the whole batch in one launch, so each of the two QRs adds 12.
The six square products of the stacks and of G add their 2 or 3 kernels: 16.
"""
import pytest

pytestmark = pytest.mark.gpu


def _launches(C):
    import paper_1504_05090_gb300 as pkg
    g = pkg.Group(Lx=16, Ly=10, t=0.25, U=2.0, beta=0.5, dtau=0.125, n_chains=C, stab_interval=4,
                  delay_k=8, precision="df32")
    with pkg.DQMC([g], seed=1) as sim:
        n0 = sim.launch_count()
        sim.sweep(1, measure=False)
        return sim.launch_count() - n0


def test_small_products_of_the_blocked_qr_count_once():
    assert _launches(300) - _launches(256) == 2 * 12 + 16
