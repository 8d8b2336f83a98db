"""A gauge field that qxd_set_gauge refuses leaves neither the lattice nor its
views usable: the refused links have overwritten the old ones, so an operator
built from the old field would mix the two."""
import pytest
import torch

from qxd_cases import Case

pytestmark = pytest.mark.gpu

SIZE = dict(T=8, L1=8, L2=8, L3=16)


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__ as ge
    ge.build()
    if not torch.cuda.is_available():
        pytest.skip("no GPU")


def _refuse(qxd, lat, c, how):
    if how == "not SU(3)":
        u, a, flags, code = 1.5 * c.su3, c.ang, qxd.QXD_GAUGE_PHYSICAL_HALF, qxd.QXD_ERR_ARG
    else:  # the mirror half is no conjugate of the physical one
        u, a = torch.cat([c.su3, c.su3], 1), torch.cat([c.ang, c.ang], 1)
        flags, code = qxd.QXD_GAUGE_EXTENDED_CHECKED, qxd.QXD_ERR_NOT_ADMISSIBLE
    with pytest.raises(qxd.QxdError) as e:
        lat.set_gauge(u.contiguous().cuda(), a.contiguous().cuda(), flags)
    assert e.value.code == code


@pytest.mark.parametrize("how", ["not SU(3)", "not admissible"])
def test_views_are_stale_after_a_refused_field(how):
    from paper_1710_08839_gb300 import qxd
    c, d = Case(**SIZE, qhat=2, seed=3), Case(**SIZE, qhat=2, seed=4)
    x = c.psi.cuda()
    x32 = x.to(torch.complex64)
    lat = c.lattice()
    view = lat.view()
    view.set_params(0.15, 1.0, 1.0, -1)
    view.sw_build()
    y, y32 = torch.empty_like(x), torch.empty_like(x32)
    view.Dw(y, x)
    _refuse(qxd, lat, d, how)
    nat = torch.empty(2, lat.V * 24, dtype=torch.float32, device="cuda")
    calls = [lambda l: l.Dw(y, x), lambda l: l.Dw(y32, x32), lambda l: l.Dhat(y, x),
             lambda l: l.sap(y32, x32, ncy=1, nmr=1), lambda l: l.sw_logdet(qxd.QXD_SITES_ALL),
             lambda l: l.solve(y, x), lambda l: l.sw_build(),
             lambda l: qxd.qxd_Dw_batch([l.handle], [nat[0].data_ptr()], [nat[1].data_ptr()], qxd.QXD_FP32)]
    for l in (lat, view):
        for call in calls:
            with pytest.raises(qxd.QxdError) as e:
                call(l)
            assert e.value.code == qxd.QXD_ERR_STATE
    # a field that is accepted brings both back
    lat.set_gauge(d.su3.cuda(), d.ang.cuda())
    with pytest.raises(qxd.QxdError):
        view.Dw(y, x)
    view.sw_build()
    view.Dw(y, x)
    fresh = qxd.Lattice(d.T, d.L1, d.L2, d.L3, d.mask)
    fresh.set_gauge(d.su3.cuda(), d.ang.cuda())
    fresh.set_params(0.15, 1.0, 1.0, -1)
    fresh.sw_build()
    z = torch.empty_like(x)
    fresh.Dw(z, x)
    assert torch.equal(y, z)
    fresh.close()
    view.close()
    lat.close()
