"""The FP32 Schwarz method without the block-by-block copy of the operator (no
memory for it, or switched off) works on the native fields: the same bits from
every entry point, for lattices and views, alone and next to operators that have
their copy, and on streams of their own straight after the build."""
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


SIZES = [dict(T=8, L1=8, L2=8, L3=8, mask=0b1110), dict(T=16, L1=8, L2=24, L3=8, mask=0),
         dict(T=8, L1=4, L2=8, L3=16, mask=0b0010)]


def _pair(c):
    """The same operator with and without the copy."""
    from paper_1710_08839_gb300 import qxd
    out = []
    for copy in (1, 0):
        lat = qxd.Lattice(c.T, c.L1, c.L2, c.L3, c.mask)
        lat.set_sap_copy(copy)
        lat.set_gauge(c.su3.cuda(), c.ang.cuda())
        lat.set_params(c.m0, c.csw, c.cswqed, c.qhat)
        lat.sw_build()
        out.append(lat)
    return out


@pytest.mark.parametrize("qhat", [0, 2, -1])
@pytest.mark.parametrize("size", range(len(SIZES)))
def test_same_bits_without_the_copy(size, qhat):
    from paper_1710_08839_gb300 import qxd
    c = Case(**SIZES[size], qhat=qhat, seed=size)
    x = c.psi.cuda()
    x32 = x.to(torch.complex64)
    got = []
    for lat in _pair(c):
        r = []
        for ncy, nmr in ((1, 1), (3, 4)):
            y = torch.empty_like(x32)
            lat.sap(y, x32, ncy=ncy, nmr=nmr)
            r.append(y)
        nat = [lat.pack(torch.empty(lat.V * 24, dtype=torch.float32, device="cuda"), s * x32, qxd.QXD_FP32)
               for s in (1, -2, 0.5)]
        r += lat.sap_multi([torch.empty_like(n) for n in nat], nat, ncy=2, nmr=3)
        y = torch.empty_like(x)
        lat.solve(y, x, tol=1e-10, precond=qxd.QXD_PRECOND_SAP, inner_prec=qxd.QXD_FP32)
        r.append(y)
        got.append(r)
        torch.cuda.synchronize()
        lat.close()
    for a, b in zip(*got):
        assert torch.equal(a, b)


def test_follows_the_operator_and_views():
    c = Case(**SIZES[0], qhat=2)
    x = c.psi.to(torch.complex64).cuda()
    got = []
    for lat in _pair(c):
        view = lat.view()
        if not got:
            view.set_sap_copy(0)  # a view without beside a lattice with it, and the other way round
        ys = []
        for m0, q in ((0.1, -1), (0.3, 0)):
            for l in (lat, view):
                l.set_params(m0, 1.0, 1.0, q)
                l.sw_build()
                ys.append(torch.empty_like(x))
                l.sap(ys[-1], x, ncy=2, nmr=2)
        got.append(ys)
        torch.cuda.synchronize()
        view.close()
        lat.close()
    for a, b in zip(*got):
        assert torch.equal(a, b)


@pytest.mark.parametrize("first", [0, 1])
def test_streams_after_the_build(first):
    """Applications on two streams, the first ones after the build, each with
    its own operator object (a lattice's calls share its work fields)."""
    c = Case(**SIZES[1], qhat=2)
    lats = _pair(c)
    want = torch.empty_like(c.psi.to(torch.complex64).cuda())
    x = c.psi.to(torch.complex64).cuda()
    torch.cuda.synchronize()
    ys = []
    for k in (first, 1 - first):
        st = torch.cuda.Stream()
        y = torch.empty_like(x)
        torch.cuda.synchronize()
        lats[k].sap(y, x, ncy=3, nmr=4, stream=st)
        ys.append(y)
    torch.cuda.synchronize()
    lats[0].sap(want, x, ncy=3, nmr=4)
    torch.cuda.synchronize()
    assert torch.equal(ys[0], want) and torch.equal(ys[1], want)
    for lat in lats:
        lat.close()


@pytest.mark.parametrize("which", ["none has it", "one of two"])
def test_engine(which):
    """Requests of small lattices share one launch of the block solve."""
    from paper_1710_08839_gb300 import qxd
    cs = [Case(**SIZES[0], qhat=0, seed=5), Case(**SIZES[1], qhat=2, seed=6)]
    xs = [c.psi.cuda() for c in cs]
    got = []
    for drop in (False, True):
        pairs = [_pair(c) for c in cs]
        ops = [p[1 if drop and (which == "none has it" or i == 1) else 0] for i, p in enumerate(pairs)]
        e = qxd.Engine(1 << 30)
        ys = [torch.empty_like(x) for x in xs]
        ids = [e.submit(op, y, x, tol=1e-10) for op, y, x in zip(ops, ys, xs)]
        e.run()
        assert all(e.poll(i)[1]["status"] == qxd.QXD_OK for i in ids)
        e.close()
        got.append(ys)
        for p in pairs:
            for lat in p:
                lat.close()
    for a, b in zip(*got):
        assert torch.equal(a, b)


def test_the_switch_is_for_before_the_copy():
    from paper_1710_08839_gb300 import qxd
    a, b = _pair(Case(**SIZES[0]))
    with pytest.raises(qxd.QxdError) as e:
        a.set_sap_copy(0)
    assert e.value.code == qxd.QXD_ERR_STATE
    b.set_sap_copy(1)
    b.sw_build()
    with pytest.raises(qxd.QxdError) as e:
        b.set_sap_copy(1)
    assert e.value.code == qxd.QXD_ERR_STATE
    a.close()
    b.close()


def test_the_copy_leaves_half_of_the_memory():
    """With less than half of the device memory free qxd_sw_build makes no copy
    (the switch still answers then); once there is room the next build makes it."""
    from paper_1710_08839_gb300 import qxd
    c = Case(**SIZES[0], qhat=2)
    x = c.psi.to(torch.complex64).cuda()
    torch.cuda.empty_cache()
    free, total = torch.cuda.mem_get_info()
    taken = torch.empty(max(0, free - total // 2 + (64 << 20)), dtype=torch.uint8, device="cuda")
    try:
        lat = c.lattice()
        lat.set_sap_copy(1)
        y, z = torch.empty_like(x), torch.empty_like(x)
        lat.sap(y, x, ncy=2, nmr=2)
        torch.cuda.synchronize()
    finally:
        del taken
        torch.cuda.empty_cache()
    lat.sw_build()
    with pytest.raises(qxd.QxdError):
        lat.set_sap_copy(1)
    lat.sap(z, x, ncy=2, nmr=2)
    assert torch.equal(y, z)
    lat.close()
