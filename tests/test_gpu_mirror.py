"""With C* boundaries and the gauge field given on the physical half, plaquettes,
clover blocks, their inverses and the hop links of the mirror half follow from
the physical ones by conjugation; the same field given on the whole lattice is
worked out on every site. Both give the same operator, observables and flow.
Tolerance: 1e-13 relative, the FP64 bound of the operator against the oracle
(both sides are within rounding of the same numbers)."""
import numpy as np
import pytest
import torch

from qxd_cases import Case, rel_max

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__ as ge
    ge.build()
    if not torch.cuda.is_available():
        pytest.skip("no GPU")


def _extended(c):
    return torch.cat([c.su3, c.su3.conj().resolve_conj()], 1).contiguous(), torch.cat([c.ang, -c.ang], 1).contiguous()


@pytest.mark.parametrize("mask", [0b1110, 0b0110, 0b1010, 0b0010])
@pytest.mark.parametrize("size", [(2, 2, 2, 2), (6, 4, 10, 6), (4, 6, 2, 14)])
def test_mirror_half_equals_whole_lattice(mask, size):
    from paper_1710_08839_gb300 import qxd
    c = Case(*size, mask=mask, qhat=2, m0=0.1, seed=mask)
    su3, ang = _extended(c)
    x = c.psi.cuda()
    got = []
    for flags, u, a in ((qxd.QXD_GAUGE_PHYSICAL_HALF, c.su3, c.ang), (qxd.QXD_GAUGE_EXTENDED_CHECKED, su3, ang),
                        (qxd.QXD_GAUGE_EXTENDED_UNCHECKED, su3, ang)):
        lat = qxd.Lattice(*size, mask)
        lat.set_gauge(u.cuda(), a.cuda(), flags)
        r = []
        for flowed in (False, True):
            if flowed:
                lat.wflow(0.05, 2)
            lat.set_params(c.m0, 1.0, 1.0, c.qhat)
            lat.sw_build()
            y, z = torch.empty_like(x), torch.empty_like(x)
            lat.Dw(y, x)
            lat.Dhat(z, x)
            r += [y.cpu().numpy(), z.cpu().numpy(), np.array([lat.sw_logdet(qxd.QXD_SITES_ALL)]),
                  np.array(lat.gauge_observables(1 / 6))[:2]]
        got.append(r)
        lat.close()
    for other in got[1:]:
        for a, b in zip(got[0], other):
            assert rel_max(a, b) < 1e-13


def test_flow_of_an_inadmissible_field():
    """A field that is no C* field, taken as it is: the first stage of the flow
    integrates the physical half in the given surroundings, then the mirror half
    is the conjugate."""
    from paper_1710_08839_gb300 import qxd
    size, mask = (4, 4, 4, 4), 0b1110
    c, d = Case(*size, mask=mask, seed=1), Case(*size, mask=mask, seed=2)
    su3 = torch.cat([c.su3, d.su3], 1).contiguous()
    ang = torch.cat([c.ang, d.ang], 1).contiguous()
    obs = []
    for u, a, flags in ((su3, ang, qxd.QXD_GAUGE_EXTENDED_UNCHECKED), (c.su3, c.ang, qxd.QXD_GAUGE_PHYSICAL_HALF)):
        lat = qxd.Lattice(*size, mask)
        lat.set_gauge(u.cuda(), a.cuda(), flags)
        lat.wflow(1e-7, 1)
        obs.append(np.array(lat.gauge_observables(1 / 6)))
        lat.close()
    # after the step the mirror half is the conjugate of the physical one on both
    # sides, and a step of 1e-7 moves the densities by about that much
    assert np.abs(obs[0] - obs[1]).max() < 1e-4 * np.abs(obs[1][:2]).max()
