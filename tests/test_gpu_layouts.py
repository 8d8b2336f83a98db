"""The operator's entry points give the same bits on native fields, on
lexicographic fields the kernels can read in place (16-byte aligned) and on
lexicographic fields at an 8-byte offset, which go through a layout
conversion, at sizes around the splits of the FP64 kernels' work (608
schedulers x 16 sites; 6 threads per site for what is left over)."""
import numpy as np
import pytest
import torch

from qxd_cases import Case, rel_max, rel_norm

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__ as ge
    ge.build()
    if not torch.cuda.is_available():
        pytest.skip("no GPU")


# simulated volumes 16, 2016, 4800, 4896, 9696, 9792, 12000: below one round of
# 4 sites per scheduler, at two, one round of 16, and beyond it with a rest
SIZES = [
    dict(T=2, L1=2, L2=2, L3=2, mask=0),
    dict(T=6, L1=6, L2=14, L3=2, mask=0b0110),
    dict(T=6, L1=10, L2=4, L3=10, mask=0b1010),
    dict(T=4, L1=6, L2=6, L3=34, mask=0),
    dict(T=6, L1=2, L2=4, L3=202, mask=0),
    dict(T=6, L1=6, L2=8, L3=34, mask=0),
    dict(T=10, L1=6, L2=10, L3=10, mask=0b1110),
]


def _offset_copy(x):
    """A copy of x whose data starts 8 bytes after a 16-byte boundary."""
    real = torch.view_as_real(x).reshape(-1)
    n = 8 // real.element_size()
    buf = torch.empty(real.numel() + n, dtype=real.dtype, device=x.device)
    v = buf[n:]
    v.copy_(real)
    assert v.data_ptr() % 16 == 8
    return v


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("size", range(len(SIZES)))
def test_layouts_agree(size, prec):
    from paper_1710_08839_gb300 import qxd
    p = qxd.QXD_FP64 if prec == "fp64" else qxd.QXD_FP32
    dt = torch.complex128 if prec == "fp64" else torch.complex64
    c = Case(**SIZES[size], qhat=2, seed=size)
    lat = c.lattice()
    x = c.psi.to(dt).cuda()
    real = torch.float64 if prec == "fp64" else torch.float32
    xn = torch.empty(lat.V * 24, dtype=real, device="cuda")
    lat.pack(xn, x, p)
    back = torch.full_like(x, float("nan"))
    lat.unpack(back, xn, p)
    assert torch.equal(back, x)
    xo = _offset_copy(x)
    ops = {
        "Dw": lambda o, i, flags: qxd.qxd_Dw(lat.handle, o.data_ptr(), i.data_ptr(), p | flags),
        "Dhat": lambda o, i, flags: qxd.qxd_Dhat(lat.handle, o.data_ptr(), i.data_ptr(), p | flags),
        "prepare": lambda o, i, flags: qxd.qxd_eo_prepare(lat.handle, o.data_ptr(), i.data_ptr(), p | flags),
        "reconstruct": lambda o, i, flags: qxd.qxd_eo_reconstruct(lat.handle, o.data_ptr(), i.data_ptr(), p | flags),
    }
    want = {}
    for name, op in ops.items():
        # reconstruct reads the even sites of its output: the same start everywhere
        lex, nat, off = x.flip(0).contiguous(), torch.empty_like(xn), _offset_copy(x.flip(0).contiguous())
        lat.pack(nat, lex, p)
        op(lex, x, 0)
        op(nat, xn, qxd.QXD_LAYOUT_NATIVE)
        op(off, xo, 0)
        lat.unpack(back, nat, p)
        torch.cuda.synchronize()
        want[name] = lex
        assert torch.equal(lex, back), name
        assert torch.equal(torch.view_as_real(lex).reshape(-1), off), name
    ref = c.oracle().apply(c.psi.numpy())
    got = want["Dw"].cpu().numpy().astype(np.complex128)
    assert (rel_max(got, ref) < 1e-13) if prec == "fp64" else (rel_norm(got, ref) < 1e-5)
    lat.close()
