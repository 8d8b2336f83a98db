"""Device memory of a lattice and of a view, and what depends on the inverse
clover blocks being kept on the odd sites only: a singular block is refused on
either parity."""
import numpy as np
import pytest
import torch

from qxd_cases import Case

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__ as ge
    ge.build()
    if not torch.cuda.is_available():
        pytest.skip("no GPU")


def test_bytes_per_site():
    """1360 bytes of gauge field and 1872 of operator (FP64 hop links 576, clover
    576 + 288, their inverses on the odd sites 288 + 144) per site; allocations
    are rounded up to 2 MiB."""
    from paper_1710_08839_gb300 import qxd

    def used(make):
        torch.cuda.synchronize()
        before = torch.cuda.mem_get_info()[0]
        made = make()
        return made, before - torch.cuda.mem_get_info()[0]
    lat, own = used(lambda: qxd.Lattice(32, 16, 16, 16, 0b1110))
    view, extra = used(lat.view)
    slack = 3 * (2 << 20)
    assert own <= (1360 + 1872) * lat.V + slack
    assert extra <= 1872 * lat.V + slack
    view.close()
    lat.close()


@pytest.mark.parametrize("mask", [0, 0b0010, 0b1110])
@pytest.mark.parametrize("parity", [0, 1])
def test_singular_block_on_either_parity(parity, mask):
    """m0 at minus an eigenvalue of one site's clover term: that site's block is
    singular, all others are not (they are away from it by more than 1e-6)."""
    from paper_1710_08839_gb300 import qxd
    c = Case(4, 4, 2, 4, mask=mask, qhat=2, m0=-4.0, seed=parity)
    lex = parity  # (0, 0, 0, parity)
    op = c.oracle()
    block = np.empty((12, 12), dtype=np.complex128)
    for k in range(12):
        e = np.zeros((c.V, 12), dtype=np.complex128)
        e[lex, k] = 1.0
        block[:, k] = op.apply(e.reshape(c.V, 4, 3)).reshape(c.V, 12)[lex]
    ev = np.linalg.eigvalsh(block)
    lat = qxd.Lattice(c.T, c.L1, c.L2, c.L3, c.mask)
    lat.set_gauge(c.su3.cuda(), c.ang.cuda())
    lat.set_params(-4.0 - ev[3], c.csw, c.cswqed, c.qhat)
    with pytest.raises(qxd.QxdError) as e:
        lat.sw_build()
    assert e.value.code == qxd.QXD_ERR_SW_SINGULAR
    lat.set_params(-4.0 - ev[3] + 1e-6, c.csw, c.cswqed, c.qhat)
    lat.sw_build()
    lat.close()
