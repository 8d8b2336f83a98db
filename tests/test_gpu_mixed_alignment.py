"""Lexicographic fields of which only one is 16-byte aligned: D takes a route of
its own for each combination (in FP32 the output alone decides whether it is
stored in place), the even-odd entry points go through layout conversions. The
same bits as with both aligned."""
import pytest
import torch

from qxd_cases import Case
from test_gpu_layouts import _offset_copy

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__ as ge
    ge.build()
    if not torch.cuda.is_available():
        pytest.skip("no GPU")


@pytest.mark.parametrize("which", ["in", "out"])
@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("size", [dict(T=2, L1=2, L2=2, L3=2, mask=0), dict(T=6, L1=4, L2=10, L3=6, mask=0b1110)])
def test_one_unaligned_field(size, prec, which):
    from paper_1710_08839_gb300 import qxd
    p, dt = (qxd.QXD_FP64, torch.complex128) if prec == "fp64" else (qxd.QXD_FP32, torch.complex64)
    c = Case(**size, qhat=2)
    lat = c.lattice()
    x = c.psi.to(dt).cuda()
    flat = torch.view_as_real(x).reshape(-1)
    for fn in (qxd.qxd_Dw, qxd.qxd_Dhat, qxd.qxd_eo_prepare, qxd.qxd_eo_reconstruct):
        # reconstruct reads the even sites of its output: the same start everywhere
        start = x.flip(0).contiguous()
        want = start.clone()
        fn(lat.handle, want.data_ptr(), x.data_ptr(), p)
        i = _offset_copy(x) if which == "in" else flat
        o = _offset_copy(start) if which == "out" else torch.view_as_real(start).reshape(-1)
        fn(lat.handle, o.data_ptr(), i.data_ptr(), p)
        torch.cuda.synchronize()
        assert torch.equal(torch.view_as_real(want).reshape(-1), o), fn.__name__
        assert torch.equal(i, flat)
    lat.close()
