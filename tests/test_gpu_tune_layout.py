"""A launch shape timed on lexicographic fields does not decide for native ones:
the first native D times its own, and lexicographic calls keep that one. Inside a
stream capture, where nothing can be timed, the shape at hand is used."""
import pytest
import torch

from qxd_cases import Case

pytestmark = pytest.mark.gpu

LEX = "(tuned) on lexicographic fields"


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__ as ge
    ge.build()
    if not torch.cuda.is_available():
        pytest.skip("no GPU")


def _line(qxd, c, prec):
    key = f"Dw {prec} qhat!=0 {c.T}x{2 * c.L1}x{c.L2}x{c.L3} "
    return next(l for l in qxd.tune_report().splitlines() if l.startswith(key))


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
def test_native_fields_time_their_own_shape(prec):
    from paper_1710_08839_gb300 import qxd
    p, dt = (qxd.QXD_FP32, torch.complex64) if prec == "fp32" else (qxd.QXD_FP64, torch.complex128)
    c = Case(T=14, L1=6, L2=10, L3=6, qhat=2)  # a shape of its own
    lat = c.lattice()
    x = c.psi.to(dt).cuda()
    xn = torch.empty(lat.V * 24, dtype=torch.float32 if prec == "fp32" else torch.float64, device="cuda")
    yn, y, z = torch.zeros_like(xn), torch.empty_like(x), torch.empty_like(x)
    lat.pack(xn, x, p)
    lat.Dw(y, x)
    assert _line(qxd, c, prec).endswith(LEX)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        lat.Dw(yn, xn, prec=p, native=True)
    g.replay()
    lat.unpack(z, yn, p)
    assert torch.equal(y, z) and _line(qxd, c, prec).endswith(LEX)
    lat.Dw(yn, xn, prec=p, native=True)
    assert _line(qxd, c, prec).endswith("(tuned)")
    chosen = lat.dw_shape(p)
    lat.Dw(z, x)
    assert lat.dw_shape(p) == chosen and torch.equal(y, z)
    lat.set_dw_shape(p, 0, 64, 2)
    lat.Dw(yn, xn, prec=p, native=True)
    assert _line(qxd, c, prec).endswith("(set)")
    lat.close()
