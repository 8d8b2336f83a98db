"""The Wilson flow of a field whose mirror half is not the conjugate of the
physical one: the first stage integrates the physical links in the given
surroundings, and every stage then sets the mirror links to the conjugates.
Compared with the same in plain FP64 on the oracle's forces, over a step that is
large enough for the surroundings to show. Also what the comparison of the two
input forms leaves out: ln|Det| by parity and the topological charge."""
import numpy as np
import pytest
import torch

import oracle as O
from oracle import qxd_flow as F
from qxd_cases import Case, rel_max

pytestmark = pytest.mark.gpu

Q_EL = 1.0 / 6.0
EPS = 0.05


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__ as ge
    ge.build()
    if not torch.cuda.is_available():
        pytest.skip("no GPU")


def _mirrored(olat, U, A):
    """The mirror half set to the conjugate of the physical one."""
    U, A = U.reshape(*olat.N, 4, 3, 3).copy(), A.reshape(*olat.N, 4).copy()
    L1 = olat.L[1]
    U[:, L1:], A[:, L1:] = U[:, :L1].conj(), -A[:, :L1]
    return U.reshape(olat.V, 4, 3, 3), A.reshape(olat.V, 4)


def _step(olat, U, A):
    """Luscher's scheme, the mirror half renewed after every stage."""
    Z0, a0 = EPS * F.force_su3(olat, U), EPS * F.force_u1(olat, A)
    U, A = _mirrored(olat, F.expm_antihermitian(0.25 * Z0) @ U, A + 0.25 * a0)
    # the accumulated forces act on the physical links only
    Z1, a1 = EPS * F.force_su3(olat, U), EPS * F.force_u1(olat, A)
    X, x = 8.0 / 9.0 * Z1 - 17.0 / 36.0 * Z0, 8.0 / 9.0 * a1 - 17.0 / 36.0 * a0
    U, A = _mirrored(olat, F.expm_antihermitian(X) @ U, A + x)
    Z2, a2 = EPS * F.force_su3(olat, U), EPS * F.force_u1(olat, A)
    return _mirrored(olat, F.expm_antihermitian(0.75 * Z2 - X) @ U, A + 0.75 * a2 - x)


@pytest.mark.parametrize("mask", [0b1110, 0b0110, 0b0010])
@pytest.mark.parametrize("size,steps", [((4, 4, 4, 4), 1), ((6, 2, 4, 6), 2)])
def test_flow_in_the_given_surroundings(size, steps, mask):
    from paper_1710_08839_gb300 import qxd
    c, d = Case(*size, mask=mask, qhat=2, m0=0.2, seed=1), Case(*size, mask=mask, seed=2)
    su3 = torch.cat([c.su3, d.su3], 1).contiguous()
    ang = torch.cat([c.ang, d.ang], 1).contiguous()
    olat = O.Lattice(*size, mask)
    U, A = su3.numpy().reshape(olat.V, 4, 3, 3), ang.numpy().reshape(olat.V, 4)
    adm = _mirrored(olat, U, A)
    for _ in range(steps):
        U, A = _step(olat, U, A)
        adm = _step(olat, *adm)
    gf = O.GaugeField.from_extended(olat, U, A)
    ref = F.observables(olat, gf, Q_EL)
    other = F.observables(olat, O.GaugeField.from_extended(olat, *adm), Q_EL)
    # on the oracle alone: the surroundings of the first stage show, a million times above the bounds below
    assert abs(ref[0] - other[0]) > 1e-5 * ref[0] and abs(ref[1] - other[1]) > 1e-5 * ref[1]
    lat = qxd.Lattice(*size, mask)
    lat.set_gauge(su3.cuda(), ang.cuda(), qxd.QXD_GAUGE_EXTENDED_UNCHECKED)
    lat.wflow(EPS, steps)
    got = lat.gauge_observables(Q_EL)
    # the bounds of the flow's comparison with the oracle (tests/test_gpu_flow.py)
    assert abs(got[0] - ref[0]) <= 1e-11 * ref[0]
    assert abs(got[1] - ref[1]) <= 1e-11 * ref[1]
    assert abs(got[2] - ref[2]) <= 1e-11 * ref[0] * olat.V
    lat.set_params(c.m0, c.csw, c.cswqed, c.qhat)
    lat.sw_build()
    x = c.psi.cuda()
    y = torch.empty_like(x)
    lat.Dw(y, x)
    torch.cuda.synchronize()
    want = O.Dirac(olat, gf, c.m0, c.csw, c.cswqed, c.qhat).apply(c.psi.numpy())
    assert rel_max(y.cpu().numpy(), want) < 1e-12
    lat.close()


@pytest.mark.parametrize("mask", [0b1110, 0b1010, 0b0010])
def test_determinant_by_parity_and_charge(mask):
    """Both input forms of one field, against each other and the oracle. ln|Det|
    is a sum of V (or V/2) terms of order 1 to 10: 1e-13 of their size; Q_top of
    terms of either sign, bounded by E V."""
    from paper_1710_08839_gb300 import qxd
    size = (6, 4, 10, 6)
    c = Case(*size, mask=mask, qhat=2, m0=0.1, seed=mask)
    su3 = torch.cat([c.su3, c.su3.conj().resolve_conj()], 1).contiguous()
    ang = torch.cat([c.ang, -c.ang], 1).contiguous()
    olat = O.Lattice(*size, mask)
    gf = O.GaugeField.from_physical(olat, c.su3.numpy(), c.ang.numpy())
    ref = F.observables(olat, gf, Q_EL)
    op = O.Dirac(olat, gf, c.m0, c.csw, c.cswqed, c.qhat)
    e = np.zeros((12, olat.V, 12), dtype=np.complex128)
    for k in range(12):
        e[k, :, k] = 1.0
    blocks = np.empty((olat.V, 12, 12), dtype=np.complex128)
    for p in (0, 1):  # M acts within a site and hops change parity
        on = olat.parity(olat.all_sites()) == p
        for k in range(12):
            src = np.where(on[:, None], e[k], 0.0).reshape(olat.V, 4, 3)
            blocks[on, :, k] = op.apply(src).reshape(olat.V, 12)[on]
    par = olat.parity(olat.all_sites())
    for u, a, flags in ((c.su3, c.ang, qxd.QXD_GAUGE_PHYSICAL_HALF), (su3, ang, qxd.QXD_GAUGE_EXTENDED_CHECKED)):
        lat = qxd.Lattice(*size, mask)
        lat.set_gauge(u.cuda(), a.cuda(), flags)
        lat.set_params(c.m0, c.csw, c.cswqed, c.qhat)
        lat.sw_build()
        for sites, on in ((qxd.QXD_SITES_EVEN, par == 0), (qxd.QXD_SITES_ODD, par == 1), (qxd.QXD_SITES_ALL, par >= 0)):
            want = np.linalg.slogdet(blocks[on])[1].sum()
            assert abs(lat.sw_logdet(sites) - want) <= 1e-12 * abs(want)
        got = lat.gauge_observables(Q_EL)
        assert abs(got[2] - ref[2]) <= 1e-12 * ref[0] * olat.V
        lat.close()
