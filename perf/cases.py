"""The work whose speed is followed: D and its even-odd forms, the Schwarz
preconditioner, a mixed-precision solve, the pseudofermion factor, the set-up
of an operator on a new gauge field, and the Wilson flow, each through the
public binding, from 1024 sites up to 64x64x32x32.

listed() gives the standing cases, draw(rng) further ones of the same ranges;
prepare() makes a case's inputs on the GPU from a seed, run() does one pass,
work() counts what a pass cannot do without, and exact() recomputes a pass in
64 bits with plain torch from the definitions of the operator.

Inputs are drawn on the GPU: SU(3) links near the identity (width ``eps``,
rows re-orthonormalised), photon angles of width 0.3 and Gaussian sources, on
the extended lattice of C* boundaries (x1 doubled).
"""
from __future__ import annotations

import math

import torch

from paper_1710_08839_gb300 import qxd

# zeros and poles of the factor P_1 of the paper's rational approximation (Table 2)
NU = (17.626, 5.9094, 2.7961, 1.4167, 0.73020, 0.37808, 0.19600)
MU = (12.383, 4.8370, 2.3515, 1.1994, 0.61927, 0.32079, 0.16632)
Q_EL = 1.0 / 6.0


def _case(name, op, T, L1, L2, L3, mask=0b1110, qhat=2, m0=0.05, prec="f64", native=False, **kw):
    c = {"name": name, "op": op, "T": T, "L1": L1, "L2": L2, "L3": L3, "mask": mask, "qhat": qhat, "m0": m0,
         "prec": prec, "native": native, "eps": 0.3}
    c.update(kw)
    return c


def listed():
    return [
        # one D on the smallest lattice of the parity workload: a call's latency
        _case("dw_f64_tiny", "dw", 8, 4, 4, 4, qhat=-1, m0=0.2),
        # D in double precision in the default layout, extents that fill no tile, periodic space, no charge
        _case("dw_f64_ragged", "dw", 20, 20, 14, 18, mask=0, qhat=0),
        # D in single precision on a caller's own (lexicographic) fields
        _case("dw_f32_lex", "dw", 32, 16, 16, 16, prec="f32"),
        # D inside a solver: native fields, the largest lattice
        _case("dw_f32_native", "dw", 64, 32, 32, 32, prec="f32", native=True),
        # even-odd source, D_hat and reconstruction, as a caller's own even-odd solver uses them
        _case("eo_f32_lex", "eo", 48, 24, 24, 24, prec="f32", qhat=-1),
        # D for many sources on two lattices at once (propagators of two ensembles)
        _case("batch_f32", "batch", 24, 12, 12, 12, prec="f32", native=True, rhs=6),
        # the Schwarz preconditioner as one solver step calls it
        _case("sap_f32", "sap", 64, 32, 32, 32, prec="f32", native=True, ncy=5, nmr=5),
        # the same for several sources of one operator
        _case("sap_multi_f32", "sap", 32, 16, 16, 16, prec="f32", native=True, ncy=5, nmr=5, rhs=6, qhat=-1),
        # a whole solve: SAP-preconditioned flexible GCR, single-precision inner, 1e-10
        _case("solve_mixed", "solve", 32, 16, 16, 16),
        # the pseudofermion factor P_1 by multi-shift CG in double precision
        _case("rational_f64", "rational", 24, 12, 12, 12, qhat=-1),
        # an operator on a new gauge field: ingest, clover term, ln|Det D_oo|, the first D
        _case("operator_setup", "setup", 48, 24, 24, 24),
        # observables along the Wilson flow of a configuration, and the operator on the flowed field
        _case("wilson_flow", "flow", 32, 16, 16, 16, steps=3),
    ]


_VMAX = {"dw": 64 * 64 * 32 * 32, "eo": 48 * 48 * 24 * 24, "batch": 24 * 24 * 12 * 12, "sap": 64 * 64 * 32 * 32,
         "solve": 32 * 32 * 16 * 16, "rational": 24 * 24 * 12 * 12, "setup": 48 * 48 * 24 * 24,
         "flow": 32 * 32 * 16 * 16}


def draw(rng):
    op = rng.choice(["dw", "dw", "eo", "batch", "sap", "sap", "solve", "rational", "setup", "flow"])
    mask = rng.choice([0b1110, 0b1110, 0b1110, 0b0110, 0b1010, 0b0010, 0])
    qhat = rng.choice([-1, 0, 2])
    m0 = round(rng.uniform(0.02, 0.2), 3)
    blocks = op in ("sap", "solve")  # 4^4 Schwarz blocks: extents in steps of 8
    vmax = _VMAX[op]
    v = math.exp(rng.uniform(math.log(4096 if blocks else 1024), math.log(vmax)))
    step = 8 if blocks else 2
    for _ in range(1000):
        T, L1, L2, L3 = (max(step, int(round(v ** 0.25 * rng.uniform(0.6, 1.7) / step)) * step) for _ in range(4))
        if not mask & 2:
            L1 *= 2
        if T * (2 * L1 if mask & 2 else L1) * L2 * L3 <= vmax:
            break
    else:
        T = L1 = L2 = L3 = step
    kw = {}
    prec = rng.choice(["f32", "f64"])
    native = rng.random() < 0.5
    if op == "batch":
        prec, native, kw = "f32", True, {"rhs": rng.randint(1, 6)}
    elif op == "sap":
        prec, native, kw = "f32", True, {"ncy": rng.randint(2, 5), "nmr": rng.randint(2, 5)}
        v = T * (2 * L1 if mask & 2 else L1) * L2 * L3
        if v * 4 <= vmax:
            kw["rhs"] = rng.randint(1, 3)
    elif op in ("solve", "setup", "flow"):
        prec, native = "f64", False
        if op == "flow":
            kw = {"steps": rng.randint(1, 3)}
    elif op == "rational":
        native = False
    c = _case("", op, T, L1, L2, L3, mask, qhat, m0, prec, native, **kw)
    del c["name"]
    return c


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _extent1(c):
    return 2 * c["L1"] if c["mask"] & 2 else c["L1"]


def _volume(c):
    return c["T"] * _extent1(c) * c["L2"] * c["L3"]


def _cross_conj(a, b):
    """conj(a x b) of rows of three."""
    return torch.stack([a[..., 1] * b[..., 2] - a[..., 2] * b[..., 1], a[..., 2] * b[..., 0] - a[..., 0] * b[..., 2],
                        a[..., 0] * b[..., 1] - a[..., 1] * b[..., 0]], dim=-1).conj()


def _gauge(c, g):
    """SU(3) links (T, L1, L2, L3, 4, 3, 3) and photon angles (..., 4) of the physical lattice."""
    shape = (c["T"], c["L1"], c["L2"], c["L3"], 4)

    def normals(*more):
        return torch.randn(*shape, *more, dtype=torch.float64, device="cuda", generator=g)

    r = c["eps"] * 0.5 * torch.complex(normals(2, 3), normals(2, 3))
    r[..., 0, 0] += 1.0
    r[..., 1, 1] += 1.0
    a = r[..., 0, :] / torch.linalg.vector_norm(r[..., 0, :], dim=-1, keepdim=True)
    b = r[..., 1, :]
    for _ in range(2):
        b = b - (a.conj() * b).sum(-1, keepdim=True) * a
        b = b / torch.linalg.vector_norm(b, dim=-1, keepdim=True)
    u = torch.stack([a, b, _cross_conj(a, b)], dim=-2)
    ang = torch.remainder(0.3 * normals() + math.pi, 2 * math.pi) - math.pi
    return u, ang


def _spinor(c, g):
    # the fields of the pseudofermion factor are in double precision whatever its operator's
    f64 = c["prec"] == "f64" or c["op"] == "rational"
    z = torch.randn(_volume(c), 4, 3, 2, dtype=torch.float64 if f64 else torch.float32, device="cuda", generator=g)
    return torch.view_as_complex(z)


def _batch_sizes(c):
    half = {k: max(2, c[k] // 4 * 2) for k in ("T", "L1", "L2", "L3")}
    return [c, dict(c, **half)]


def _inputs(c, seed):
    """The numbers of a case, the same for run() and exact()."""
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    if c["op"] == "batch":
        return [_gauge(s, g) + ([_spinor(s, g) for _ in range(c["rhs"])],) for s in _batch_sizes(c)]
    u, a = _gauge(c, g)
    return u, a, [_spinor(c, g) for _ in range(c.get("rhs", 1))]


def _operator(c, u, a):
    lat = qxd.Lattice(c["T"], c["L1"], c["L2"], c["L3"], c["mask"])
    lat.set_gauge(u, a)
    lat.set_params(c["m0"], 1.0, 1.0, c["qhat"])
    lat.sw_build()
    return lat


def _prec(c):
    return qxd.QXD_FP64 if c["prec"] == "f64" else qxd.QXD_FP32


def _native(c, lat, psi):
    """The source in the layout in which the case's program holds it."""
    if not c["native"]:
        return psi
    out = torch.empty(lat.V * 24, dtype=torch.float64 if c["prec"] == "f64" else torch.float32, device="cuda")
    return lat.pack(out, psi, _prec(c))


def prepare(case, seed):
    c = case
    if c["op"] == "batch":
        st = {"case": c, "lats": [], "src": [], "out": []}
        for s, (u, a, psis) in zip(_batch_sizes(c), _inputs(c, seed)):
            lat = _operator(s, u, a)
            st["src"] += [_native(c, lat, p) for p in psis]
            st["lats"] += [lat] * len(psis)
        st["out"] = [torch.empty_like(x) for x in st["src"]]
        return st
    u, a, psis = _inputs(c, seed)
    st = {"case": c}
    if c["op"] in ("setup", "flow"):
        st["lat"] = qxd.Lattice(c["T"], c["L1"], c["L2"], c["L3"], c["mask"])
        st["gauge"] = (u, a)
    else:
        st["lat"] = _operator(c, u, a)
    st["src"] = [_native(c, st["lat"], p) for p in psis]
    st["out"] = [torch.zeros_like(x) for x in st["src"]]
    if c["op"] == "eo":
        st["bhat"], st["dhat"] = torch.zeros_like(st["src"][0]), torch.zeros_like(st["src"][0])
    return st


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def run(state):
    c = state["case"]
    op = c["op"]
    src, out = state["src"], state["out"]
    if op == "batch":
        qxd.qxd_Dw_batch([l.handle for l in state["lats"]], [o.data_ptr() for o in out], [s.data_ptr() for s in src],
                         _prec(c), stream=torch.cuda.current_stream().cuda_stream)
        return out
    lat = state["lat"]
    if op == "dw":
        return lat.Dw(out[0], src[0], prec=_prec(c), native=c["native"])
    if op == "eo":
        lat.eo_prepare(state["bhat"], src[0], native=c["native"])
        lat.Dhat(state["dhat"], state["bhat"], native=c["native"])
        # reconstruction from the even sites of D_hat b_hat, in a copy as a solver's x would be
        out[0].copy_(state["dhat"])
        lat.eo_reconstruct(out[0], src[0], native=c["native"])
        return {"bhat": state["bhat"], "dhat": state["dhat"], "x": out[0]}
    if op == "sap":
        if len(src) == 1:
            return lat.sap(out[0], src[0], ncy=c["ncy"], nmr=c["nmr"], native=True, prec=qxd.QXD_FP32)
        return lat.sap_multi(out, src, ncy=c["ncy"], nmr=c["nmr"])
    if op == "solve":
        lat.solve(out[0], src[0], tol=1e-10, precond=qxd.QXD_PRECOND_SAP, inner_prec=qxd.QXD_FP32)
        return out[0]
    if op == "rational":
        _, info = lat.rational_apply(out[0], src[0], NU, MU, tol=1e-10, prec=_prec(c))
        return {"x": out[0], "action": info["action"]}
    u, a = state["gauge"]
    lat.set_gauge(u, a)
    obs = []
    if op == "flow":
        for _ in range(c["steps"]):
            lat.wflow(0.02, 1)
            obs.append(list(lat.gauge_observables(Q_EL)))
    lat.set_params(c["m0"], 1.0, 1.0, c["qhat"])
    lat.sw_build()
    logdet = lat.sw_logdet(qxd.QXD_SITES_ODD)
    return {"logdet": logdet, "obs": obs, "x": lat.Dw(out[0], src[0])}




# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
def work(case):
    c = case
    f64 = c["prec"] == "f64" or c["op"] in ("setup", "flow")
    q = c["qhat"] != 0
    w = 8 if f64 else 4
    spinor = 24 * w
    # operator data of a site: links (two rows in single precision), U(1) phases, one clover block pair
    links = 4 * (18 * w if f64 else 12 * w) + (4 * (2 * w if f64 else w) if q else 0)
    clover = 72 * w
    hop = 132 + 24 + 12 + (36 if q else 0)  # two SU(3) products, projection, accumulation, U(1) phase
    dw = 8 * hop + 504 + 24                 # flops of D at one site
    v = _volume(c)
    if c["op"] == "dw":
        return {"bytes": v * (2 * spinor + links + clover), "flops": v * dw}
    if c["op"] == "batch":
        b = f = 0
        for s in _batch_sizes(c):
            b += _volume(s) * (2 * spinor * c["rhs"] + links + clover)
            f += _volume(s) * dw * c["rhs"]
        return {"bytes": b, "flops": f}
    if c["op"] == "eo":
        # source (all), bhat and dhat (written whole), the even sites of bhat read again, x; both clover forms
        return {"bytes": v * (4.5 * spinor + links + 1.5 * clover), "flops": v * (8 * hop * 2 + 504 * 2 + 48)}
    n = c.get("rhs", 1)
    if c["op"] == "sap":
        # per visit of a block: a quarter of D's hops cross faces, then nmr + 1 even-odd steps of the block operator
        visit = 2 * hop + (c["nmr"] + 1) * (6 * hop + 504) + c["nmr"] * 72
        return {"bytes": v * (2 * spinor * n + links + clover), "flops": v * n * c["ncy"] * visit}
    if c["op"] == "solve":
        # four preconditioned steps and three double-precision residuals, the fewest seen
        visit = 2 * hop + 6 * (6 * hop + 504) + 5 * 72
        return {"bytes": v * (4 * (2 * 96 + 208 + 288) + 3 * (2 * 192 + links + clover)),
                "flops": v * (4 * (5 * visit + dw) + 3 * dw)}
    if c["op"] == "rational":
        # 50 steps of multi-shift CG, seven shifts: two applications of D_hat a step, x_j and p_j read and written
        return {"bytes": 50 * (v / 2) * (4 * (2 * links + clover + spinor) + 7 * 4 * spinor), "flops": 50 * 2 * v * dw}
    mm = 198  # one 3x3 complex product
    # ingest: links and angles once in, kept in both precisions; six field tensors; clover term and its inverse
    set_up = v * (4 * (144 + 8) / 2 + 4 * (144 + 48 + 8 + 16) + 480 + 2 * 72 * 12)
    fl = v * (6 * 5 * mm + 2 * 2500)
    if c["op"] == "flow":
        set_up += c["steps"] * 3 * (v / 2) * 4 * (2 * 152 + 2 * 80)
        fl += c["steps"] * 3 * (v / 2) * 4 * (9 * mm + 1000)
    return {"bytes": set_up + v * (2 * spinor + links + clover), "flops": fl + v * dw}


# ---------------------------------------------------------------------------
# the same in 64 bits from the definitions, with plain torch
# ---------------------------------------------------------------------------
_PAULI = ([[0, 1], [1, 0]], [[0, -1j], [1j, 0]], [[1, 0], [0, -1]])


def _gammas(dev):
    z, one = torch.zeros(2, 2, dtype=torch.complex128), torch.eye(2, dtype=torch.complex128)
    g = [torch.cat([torch.cat([z, -one], 1), torch.cat([-one, z], 1)], 0)]
    for s in _PAULI:
        s = torch.tensor(s, dtype=torch.complex128)
        g.append(torch.cat([torch.cat([z, -1j * s], 1), torch.cat([1j * s, z], 1)], 0))
    return [x.to(dev) for x in g]


def _mm(a, b):
    return (a[..., :, 0:1] * b[..., 0:1, :] + a[..., :, 1:2] * b[..., 1:2, :] + a[..., :, 2:3] * b[..., 2:3, :])


def _dag(a):
    return a.conj().transpose(-1, -2)


class _Exact:
    """D and what is built on it, on fields (N0, N1, N2, N3, spin, colour)."""

    def __init__(self, c, u, ang):
        self.c = c
        self.N = (c["T"], _extent1(c), c["L2"], c["L3"])
        if c["mask"] & 2:
            u, ang = torch.cat([u, u.conj()], 1), torch.cat([ang, -ang], 1)
        self.U = [u[..., m, :, :].resolve_conj().clone() for m in range(4)]
        self.A = [ang[..., m].clone() for m in range(4)]
        self.gam = _gammas(u.device)
        self.perm, self.phase = [], []
        for g in self.gam:
            p = g.abs().argmax(1)
            self.perm.append(p)
            self.phase.append(g.gather(1, p[:, None]).reshape(4, 1))
        x = torch.meshgrid(*[torch.arange(n, device=u.device) for n in self.N], indexing="ij")
        self.par = (x[0] + x[1] + x[2] + x[3]) % 2
        self.x = x

    def shift(self, f, mu, d):
        """f(x + d mu), with the shifted boundary in C* directions."""
        f = torch.roll(f, -d, mu)
        if mu >= 2 and self.c["mask"] & (1 << mu):
            e = f.select(mu, self.N[mu] - 1 if d > 0 else 0)
            e.copy_(torch.roll(e, self.c["L1"], 1))
        return f

    # -- operator -------------------------------------------------------
    def tensors(self):
        """Field tensors of the six planes: SU(3) F and the U(1) sum of four sines."""
        U, A, sh = self.U, self.A, self.shift
        self.F, self.G = {}, {}
        for m in range(4):
            for n in range(m + 1, 4):
                # plaquette at x, its corner at x + m, and so on: every leaf from one product of links
                a, b = U[m], U[n]
                bp, ap = sh(b, m, 1), sh(a, n, 1)
                q = _mm(_mm(a, bp), _mm(_dag(ap), _dag(b)))
                t = _mm(_mm(bp, _dag(ap)), _mm(_dag(b), a))
                q = q + sh(t, m, -1)
                t = _mm(_mm(_dag(ap), _dag(b)), _mm(a, bp))
                q = q + sh(sh(t, m, -1), n, -1)
                t = _mm(_mm(_dag(b), a), _mm(bp, _dag(ap)))
                q = q + sh(t, n, -1)
                self.F[m, n] = (q - _dag(q)) / 8
                s = torch.sin(A[m] + sh(A[n], m, 1) - sh(A[m], n, 1) - A[n])
                s = s + sh(s, m, -1)
                self.G[m, n] = s + sh(s, n, -1)

    def build(self):
        c = self.c
        self.tensors()
        e3 = torch.eye(3, dtype=torch.complex128, device=self.par.device)
        self.M = torch.zeros(*self.N, 2, 6, 6, dtype=torch.complex128, device=self.par.device)
        for i in range(6):
            self.M[..., i, i] = 4.0 + c["m0"]
        for (m, n), F in self.F.items():
            sig = 0.5j * (self.gam[m] @ self.gam[n] - self.gam[n] @ self.gam[m])
            X = F + (0.25j * c["qhat"]) * self.G[m, n][..., None, None] * e3
            for b in range(2):
                for i in range(2):
                    for j in range(2):
                        z = complex(sig[2 * b + i, 2 * b + j])
                        if z:
                            self.M[..., b, 3 * i:3 * i + 3, 3 * j:3 * j + 3] += 0.5j * z * X
        self.W = [torch.exp(1j * c["qhat"] * a)[..., None, None] * u for u, a in zip(self.U, self.A)]
        return self

    def invert(self):
        """M^-1 of every block by elimination (its diagonal dominates), and ln|det M| of every site."""
        a = self.M.clone()
        self.ln = torch.zeros(self.N, dtype=torch.float64, device=a.device)
        for k in range(6):
            p = a[..., k, k].clone()
            self.ln += torch.log(p.abs()).sum(-1)
            col = a[..., :, k].clone()
            col[..., k] = 0
            row = a[..., k, :] / p[..., None]
            row[..., k] = 1 / p
            a[..., :, k] = 0
            a[..., k, :] = 0
            a -= col[..., :, None] * row[..., None, :]
            a[..., k, :] = row
        self.Mi = a
        return self

    def site(self, M, v):
        w = v.reshape(*self.N, 2, 6)
        y = M[..., :, 0] * w[..., 0:1]
        for k in range(1, 6):
            y = y + M[..., :, k] * w[..., k:k + 1]
        return y.reshape(v.shape)

    def hops(self, v, W=None):
        """-1/2 sum of the eight hops."""
        out = torch.zeros_like(v)
        for m, w in enumerate(self.W if W is None else W):
            g = lambda z: self.phase[m] * z[..., self.perm[m], :]  # noqa: E731
            f = self.shift(v, m, 1)
            f = f - g(f)
            b = v + g(v)
            wd = _dag(w)
            f = (w[..., None, :, 0] * f[..., 0:1] + w[..., None, :, 1] * f[..., 1:2] + w[..., None, :, 2] * f[..., 2:3])
            b = (wd[..., None, :, 0] * b[..., 0:1] + wd[..., None, :, 1] * b[..., 1:2]
                 + wd[..., None, :, 2] * b[..., 2:3])
            out += f
            out += self.shift(b, m, -1)
        return -0.5 * out

    def D(self, v):
        return self.site(self.M, v) + self.hops(v)

    def on(self, parity, v):
        return v * (self.par == parity)[..., None, None]

    def dhat(self, v):
        v = self.on(0, v)
        return self.on(0, self.site(self.M, v) - self.hops(self.on(1, self.site(self.Mi, self.hops(v)))))

    def normal(self, v):
        s = torch.tensor([1.0, 1.0, -1.0, -1.0], dtype=torch.float64, device=v.device)[:, None]
        return s * self.dhat(s * self.dhat(v))

    # -- what is built on it ----------------------------------------------
    def sap(self, eta, ncy, nmr):
        blk = sum(x // 4 for x in self.x) % 2
        W = [w * (x % 4 < 3)[..., None, None] for w, x in zip(self.W, self.x)]
        n = [k // 4 for k in self.N]

        def sums(a):  # per block, back on the sites
            s = a.sum((-1, -2)).reshape(n[0], 4, n[1], 4, n[2], 4, n[3], 4).sum((1, 3, 5, 7), keepdim=True)
            return s.expand(n[0], 4, n[1], 4, n[2], 4, n[3], 4).reshape(self.N)[..., None, None]

        psi = torch.zeros_like(eta)
        for cy in range(ncy):
            for col in range(2):
                r = eta - self.D(psi) if cy or col else eta
                rho = self.on(0, r - self.hops(self.on(1, self.site(self.Mi, r)), W))
                de = torch.zeros_like(rho)
                for _ in range(nmr):
                    w = self.on(0, self.site(self.M, rho)
                                - self.hops(self.on(1, self.site(self.Mi, self.hops(rho, W))), W))
                    om = sums(w.conj() * rho) / sums((w.conj() * w).real)
                    de = de + om * rho
                    rho = rho - om * w
                d = de + self.on(1, self.site(self.Mi, r - self.hops(de, W)))
                psi = psi + d * (blk == col)[..., None, None]
        return psi

    def solve(self, b):
        """BiCGStab, started again on its true residual until that no longer falls."""
        x, r = torch.zeros_like(b), b.clone()
        dot = lambda u, v: (u.conj() * v).sum()  # noqa: E731
        bn = b.norm().item()
        for _ in range(6):
            r0, p, y, rho = r.clone(), r.clone(), torch.zeros_like(b), dot(r, r)
            start = r.norm().item()
            for _ in range(150):
                v = self.D(p)
                al = rho / dot(r0, v)
                s = r - al * v
                t = self.D(s)
                om = dot(t, s) / dot(t, t)
                y = y + al * p + om * s
                r = s - om * t
                if r.norm().item() < 1e-9 * start:
                    break
                new = dot(r0, r)
                p = r + (new / rho) * (al / om) * (p - om * v)
                rho = new
            x = x + y
            r = b - self.D(x)
            if r.norm().item() < 2e-15 * bn or r.norm().item() > 0.3 * start:
                break
        return x

    def rational(self, phi):
        """phi + sum_j rho_j (A + mu_j^2)^-1 phi, the systems by conjugate gradients with a shared Krylov space."""
        phi = self.on(0, phi)
        n2, m2 = [x * x for x in NU], [x * x for x in MU]
        out = phi.clone()
        sig = [s - min(m2) for s in m2]
        x = [torch.zeros_like(phi) for _ in m2]
        p = [phi.clone() for _ in m2]
        z, zp = [1.0] * len(m2), [1.0] * len(m2)
        base = m2.index(min(m2))
        r, rr, ap, bp = phi.clone(), phi.norm().item() ** 2, 1.0, 0.0
        stop = rr * 1e-28
        for _ in range(400):
            w = self.normal(p[base]) + m2[base] * p[base]
            al = rr / (p[base].conj() * w).sum().real.item()
            r = r - al * w
            new = r.norm().item() ** 2
            be = new / rr
            for j, s in enumerate(sig):
                zn = z[j] * zp[j] * ap / (ap * zp[j] * (1 + al * s) + al * bp * (zp[j] - z[j])) if z[j] else 0.0
                q = zn / z[j] if z[j] else 0.0
                x[j] = x[j] + (al * q) * p[j]
                p[j] = zn * r + (be * q * q) * p[j]
                zp[j], z[j] = z[j], zn
                if abs(zn) < 1e-60:
                    z[j] = 0.0
            rr, ap, bp = new, al, be
            if rr < stop:
                break
        for j, m in enumerate(m2):
            rho = math.prod(n - m for n in n2) / math.prod(o - m for k, o in enumerate(m2) if k != j)
            out = out + rho * x[j]
        return out, (phi.conj() * out).sum().real.item()

    def observables(self):
        self.tensors()
        v = math.prod(self.N)
        tr = lambda a, b: (a * b.transpose(-1, -2)).sum().real.item()  # noqa: E731
        F, G = self.F, self.G
        e = -sum(tr(f, f) for f in F.values()) / v
        e1 = sum((g / (4 * Q_EL)).square().sum().item() for g in G.values()) / v
        q = tr(F[0, 1], F[2, 3]) - tr(F[0, 2], F[1, 3]) + tr(F[0, 3], F[1, 2])
        return [e, e1, q * (0.5 if self.c["mask"] & 2 else 1.0) / (4 * math.pi ** 2)]

    def flow(self, eps):
        """One step of the third-order Runge-Kutta scheme of the Wilson flow."""
        sh = self.shift
        X, Xa = [0.0] * 4, [0.0] * 4
        for a, b in ((0.25, 0.0), (8 / 9, -17 / 9), (0.75, -1.0)):
            U, A = self.U, self.A
            for m in range(4):
                S, za = 0.0, 0.0
                for n in range(4):
                    if n == m:
                        continue
                    up = _mm(_mm(sh(U[n], m, 1), _dag(sh(U[m], n, 1))), _dag(U[n]))
                    dn = sh(_mm(_mm(_dag(sh(U[n], m, 1)), _dag(U[m])), U[n]), n, -1)
                    S = S + up + dn
                    th = A[m] + sh(A[n], m, 1) - sh(A[m], n, 1) - A[n]
                    za = za - (torch.sin(th) - sh(torch.sin(th), n, -1))
                W = _mm(U[m], S)
                P = W - _dag(W)
                tr = P.diagonal(dim1=-2, dim2=-1).sum(-1)
                Z = -0.5 * P + (tr / 6)[..., None, None] * torch.eye(3, dtype=P.dtype, device=P.device)
                X[m] = a * eps * Z + b * X[m]
                Xa[m] = a * eps * za + b * Xa[m]
            new, ang = [], []
            for m in range(4):
                t = X[m] / 16
                E = torch.eye(3, dtype=t.dtype, device=t.device) + torch.zeros_like(t)
                for k in range(16, 0, -1):
                    E = torch.eye(3, dtype=t.dtype, device=t.device) + _mm(t, E) / k
                for _ in range(4):
                    E = _mm(E, E)
                new.append(_mm(E, U[m]))
                ang.append(torch.remainder(A[m] + Xa[m] + math.pi, 2 * math.pi) - math.pi)
            self.U, self.A = new, ang


def exact(case, seed):
    c = case
    if c["op"] == "batch":
        out = []
        for s, (u, a, psis) in zip(_batch_sizes(c), _inputs(c, seed)):
            e = _Exact(s, u, a).build()
            out += [_laid_out(c, e, e.D(_field(e, p))) for p in psis]
        return out
    u, a, psis = _inputs(c, seed)
    e = _Exact(c, u, a)
    v = _field(e, psis[0])
    if c["op"] in ("setup", "flow"):
        obs = []
        if c["op"] == "flow":
            for _ in range(c["steps"]):
                e.flow(0.02)
                obs.append(e.observables())
        e.build().invert()
        return {"logdet": e.ln[e.par == 1].sum().item(), "obs": obs, "x": _laid_out(c, e, e.D(v))}
    e.build()
    if c["op"] == "dw":
        return _laid_out(c, e, e.D(v))
    if c["op"] == "solve":
        return _laid_out(c, e, e.solve(v))
    e.invert()
    if c["op"] == "rational":
        x, action = e.rational(v)
        return {"x": _laid_out(dict(c, native=False), e, x), "action": action}
    if c["op"] == "sap":
        r = [_laid_out(c, e, e.sap(_field(e, p), c["ncy"], c["nmr"])) for p in psis]
        return r if len(r) > 1 else r[0]
    bhat = e.on(0, v - e.hops(e.on(1, e.site(e.Mi, v))))
    dhat = e.dhat(bhat)
    x = dhat + e.on(1, e.site(e.Mi, v - e.hops(dhat)))
    return {"bhat": _laid_out(c, e, bhat), "dhat": _laid_out(c, e, dhat), "x": _laid_out(c, e, x)}


def _field(e, psi):
    return psi.to(torch.complex128).reshape(*e.N, 4, 3)


def _laid_out(c, e, v):
    """A field as run() returns it: lexicographic, or the native order (even sites first, components outermost)."""
    v = v.reshape(-1, 4, 3)
    if not c["native"]:
        return v
    order = torch.argsort(e.par.reshape(-1), stable=True)
    width = 2 if c["prec"] == "f64" else 4  # reals side by side: double2, float4
    r = torch.view_as_real(v[order]).reshape(v.shape[0], 24 // width, width)
    return r.permute(1, 0, 2).reshape(-1)
