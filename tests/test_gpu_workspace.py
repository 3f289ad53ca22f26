"""The workspace of the blocked QR is allocated only where a group can take that
QR: two N x N buffers and more per chain, nothing at N <= 144 unless the
stabilisation interval is long (exponent 21.7 against 10.8 here, with the same
number of stabilisation points)."""
import pytest

pytestmark = pytest.mark.gpu


def _used(Lx, Ly, C, ns):
    import torch

    import paper_1504_05090_gb300 as pkg
    g = pkg.Group(Lx=Lx, Ly=Ly, t=0.25, U=2.0, beta=0.4 * ns, dtau=0.4, n_chains=C, stab_interval=ns,
                  delay_k=8, precision="df32")
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    with pkg.DQMC([g], seed=1):
        return free - torch.cuda.mem_get_info()[0]


@pytest.mark.parametrize("Lx,Ly,C", [(8, 8, 1024), (12, 12, 256)])
def test_blocked_qr_workspace_only_where_it_is_used(Lx, Ly, C):
    _used(Lx, Ly, C, 4)  # modules and pools that stay
    short, long = _used(Lx, Ly, C, 4), _used(Lx, Ly, C, 8)
    N = Lx * Ly
    assert long - short > 0.9 * C * 2 * N * N * 8
