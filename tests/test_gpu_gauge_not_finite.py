"""qxd_set_gauge refuses links and angles that are not finite, in each of its
input forms: one entry, a whole link (no finite deviation is left then), and
infinities; with one bad link among good ones at the first and the last site."""
import pytest
import torch

from qxd_cases import Case

pytestmark = pytest.mark.gpu

NAN, INF = float("nan"), float("inf")


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__ as ge
    ge.build()
    if not torch.cuda.is_available():
        pytest.skip("no GPU")


@pytest.mark.parametrize("site", [0, -1])
@pytest.mark.parametrize("what", ["entry nan", "entry imaginary nan", "link nan", "entry inf", "angle nan", "angle inf"])
@pytest.mark.parametrize("kind", ["half", "checked", "unchecked"])
def test_not_finite_is_refused(kind, what, site):
    from paper_1710_08839_gb300 import qxd
    c = Case(4, 2, 4, 6, mask=0b1110)
    u, a = c.su3.clone(), c.ang.clone()
    if kind != "half":
        u, a = torch.cat([u, u.conj().resolve_conj()], 1).contiguous(), torch.cat([a, -a], 1).contiguous()
    link = u.view(-1, 4, 3, 3)[site, 2]
    if what.startswith("angle"):
        a.view(-1, 4)[site, 2] = INF if "inf" in what else NAN
    elif what == "link nan":
        link[:] = complex(NAN, NAN)
    else:
        link[1, 2] = complex(0.1, NAN) if "imaginary" in what else complex(INF if "inf" in what else NAN, 0.1)
    flags = {"half": qxd.QXD_GAUGE_PHYSICAL_HALF, "checked": qxd.QXD_GAUGE_EXTENDED_CHECKED,
             "unchecked": qxd.QXD_GAUGE_EXTENDED_UNCHECKED}[kind]
    lat = qxd.Lattice(c.T, c.L1, c.L2, c.L3, c.mask)
    with pytest.raises(qxd.QxdError) as e:
        lat.set_gauge(u.cuda(), a.cuda(), flags)
    assert e.value.code == qxd.QXD_ERR_ARG and "not finite" in str(e.value)
    with pytest.raises(qxd.QxdError) as e:
        lat.gauge_observables(1 / 6)
    assert e.value.code == qxd.QXD_ERR_STATE
    lat.close()
