"""The block-by-block copy of the operator that the FP32 Schwarz method works on
follows the operator: after new parameters, a new gauge field, a flow, and on
views, an application gives the bits of a fresh lattice with that operator."""
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


SIZE = dict(T=8, L1=8, L2=8, L3=16)


def _sap(lat, x):
    y = torch.empty_like(x)
    lat.sap(y, x, ncy=2, nmr=3)
    return y


def _fresh(c, m0, q, flow=0):
    from paper_1710_08839_gb300 import qxd
    lat = qxd.Lattice(c.T, c.L1, c.L2, c.L3, c.mask)
    lat.set_gauge(c.su3.cuda(), c.ang.cuda())
    if flow:
        lat.wflow(0.05, flow)
    lat.set_params(m0, 1.0, 1.0, q)
    lat.sw_build()
    return lat


def test_plan_follows_the_operator():
    a, b = Case(**SIZE, qhat=2, seed=3), Case(**SIZE, qhat=2, seed=4)
    x = a.psi.to(torch.complex64).cuda()
    lat = _fresh(a, 0.1, 2)
    view = lat.view()
    view.set_params(0.2, 1.0, 1.0, -1)
    view.sw_build()
    got = [_sap(lat, x), _sap(view, x)]
    lat.set_params(0.05, 1.0, 1.0, 0)
    lat.sw_build()
    got.append(_sap(lat, x))
    lat.wflow(0.05, 1)
    lat.sw_build()
    view.sw_build()
    got += [_sap(lat, x), _sap(view, x)]
    lat.set_gauge(b.su3.cuda(), b.ang.cuda())
    lat.sw_build()
    got.append(_sap(lat, x))
    torch.cuda.synchronize()
    view.close()
    lat.close()
    for y, args in zip(got, ((a, 0.1, 2), (a, 0.2, -1), (a, 0.05, 0), (a, 0.05, 0, 1), (a, 0.2, -1, 1), (b, 0.05, 0))):
        f = _fresh(*args)
        assert torch.equal(_sap(f, x), y)
        f.close()
