"""The FP32 Schwarz kernel keeps its clover rows in tensor memory, which thread
blocks of an SM share: applications on two streams beside matrix products (whose
kernels allocate it too) give the bits of applications that run alone."""
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


@pytest.mark.parametrize("T,L,nmr", [(8, 8, 1), (16, 8, 4), (32, 16, 5)])
def test_streams_share_tensor_memory(T, L, nmr):
    from paper_1710_08839_gb300 import qxd
    c = Case(T=T, L1=L, L2=L, L3=L, qhat=2, seed=5)
    x = c.psi.to(torch.complex64).cuda()
    lats, alone = [], []
    for m0 in (0.1, 0.3):
        lat = qxd.Lattice(c.T, c.L1, c.L2, c.L3, c.mask)
        lat.set_gauge(c.su3.cuda(), c.ang.cuda())
        lat.set_params(m0, 1.0, 1.0, 2)
        lat.sw_build()
        y = torch.empty_like(x)
        lat.sap(y, x, ncy=2, nmr=nmr)
        lats.append(lat)
        alone.append(y)
    a = torch.randn(2048, 2048, device="cuda", dtype=torch.bfloat16)
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream() for _ in range(3)]
    outs = [[torch.empty_like(x) for _ in range(4)] for _ in lats]
    torch.cuda.synchronize()
    for k in range(4):
        with torch.cuda.stream(streams[2]):
            a @ a
        for lat, st, ys in zip(lats, streams, outs):
            lat.sap(ys[k], x, ncy=2, nmr=nmr, stream=st.cuda_stream)
    torch.cuda.synchronize()
    for ys, ref in zip(outs, alone):
        for y in ys:
            assert torch.equal(y, ref)
    for lat in lats:
        lat.close()
