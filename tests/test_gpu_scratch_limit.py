"""A call whose scratch fields do not all fit is refused, again on every later
call, and works once there is room: the three fields are allocated together."""
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


def test_scratch_is_all_or_nothing():
    from paper_1710_08839_gb300 import qxd
    c = Case(32, 24, 24, 24, mask=0b1110, qhat=2, device="cuda")  # 884736 sites: 170 MB per scratch field
    lat = c.lattice()
    x = c.psi.to(torch.complex64)
    y, want = torch.empty_like(x), torch.empty_like(x)
    nat = lat.pack(torch.empty(lat.V * 24, dtype=torch.float32, device="cuda"), x, qxd.QXD_FP32)
    out = torch.empty_like(nat)
    lat.Dw(out, nat, prec=qxd.QXD_FP32, native=True)
    lat.unpack(want, out, qxd.QXD_FP32)
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    field = lat.V * 24 * 8
    taken = torch.empty(torch.cuda.mem_get_info()[0] - 2 * field - field // 2, dtype=torch.uint8, device="cuda")
    try:
        for _ in range(3):
            for call in (lat.Dw, lat.Dhat, lat.eo_prepare):
                with pytest.raises(qxd.QxdError) as e:
                    call(y, x)
                assert e.value.code == qxd.QXD_ERR_OOM
    finally:
        del taken
        torch.cuda.empty_cache()
    lat.Dw(y, x)
    assert torch.equal(y, want)
    lat.close()
