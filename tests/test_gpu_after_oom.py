"""A refused allocation is reported by the call that made it and by no other:
the next call on another lattice succeeds."""
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


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_next_call_is_not_refused(prec):
    from paper_1710_08839_gb300 import qxd
    c = Case(4, 4, 4, 6, qhat=2)
    lat = c.lattice()
    x = c.psi.to(torch.complex128 if prec == "fp64" else torch.complex64).cuda()
    y, z = torch.empty_like(x), torch.empty_like(x)
    lat.Dw(y, x)
    with pytest.raises(qxd.QxdError) as e:
        qxd.Lattice(256, 64, 128, 128, 0b1110)  # 537 million sites, 1.7 TB
    assert e.value.code == qxd.QXD_ERR_OOM
    lat.Dw(z, x)
    torch.cuda.synchronize()
    assert torch.equal(y, z)
    lat.close()
