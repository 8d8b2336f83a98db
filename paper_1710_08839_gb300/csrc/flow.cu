// Gauge observables and the Wilson flow (App. A; Luscher's flow, Sec. 3).
//
// * qxd_gauge_observables reduces the clover field tensors of the gauge
//   field (kept by qxd_set_gauge, one anti-Hermitian F per plane and site plus
//   the U(1) four-plaquette Im sum) to
//     E_SU(3) = 1/V sum_x sum_{mu<nu} |F_munu(x)|^2 = -1/(2V) sum tr{F F},
//     E_U(1)  = 1/V sum_x sum_{mu<nu} (Im sum / (4 q_el))^2,
//     Q_top   = 1/(4 pi^2) sum_x [tr F01 F23 - tr F02 F13 + tr F03 F12]
//   (the 24 terms of the epsilon sum, grouped), with the C* sum halved to
//   the physical lattice (the mirror half carries the conjugate field).
// * qxd_wflow integrates dV/dt = Z(V) V, Z = -1/2 (W - W^dag) +
//   1/6 tr(W - W^dag), W = U(x,mu) (sum of the six staples), with Luscher's
//   third-order Runge-Kutta scheme in its one-accumulator form
//     X <- a eps Z(W_i) + b X,  W_{i+1} = exp(X) W_i,
//     (a, b) = (1/4, 0), (8/9, -17/9), (3/4, -1),
//   and the compact U(1) field by the same scheme with
//     dA(x,mu)/dt = -sum_{nu != mu} [sin theta_munu(x) - sin theta_munu(x - nu)].
//   With C* boundaries only the physical links (x1 < L1) are integrated; each
//   update is written to the mirror link as its complex conjugate (-A for
//   the angle), which keeps the orbifold constraint exact. A stage is two
//   kernels bound by the FP64 units: the leaves of every plaquette, each
//   computed once (k_flow_leaves), and the links, updated in place from sums of
//   leaves (k_flow_link). On 32x32x16x16 sites a stage takes 0.83 + 0.43 ms,
//   both within a tenth of the FP64 issue rate; with six staples and W by
//   products at every link it took 3.1 ms.
#include <cmath>
#include <string>

#include "blas.cuh"
#include "su3.cuh"

namespace qxd {

int launch_field_tensor(qxd_lattice* lat);

namespace {

// ---------------------------------------------------------------------------
// observables
// ---------------------------------------------------------------------------

struct Anti {
    double d[3];  // F_ii = i d_i
    C64 o[3];     // F_01, F_02, F_12
};

__device__ __forceinline__ Anti load_plane(const double* __restrict__ F, size_t V, int plane, int s) {
    const double* f = F + (size_t)plane * 10 * V + s;
    Anti a;
    a.d[0] = f[0];
    a.d[1] = f[V];
    a.d[2] = f[2 * V];
    a.o[0] = mk(f[3 * V], f[4 * V]);
    a.o[1] = mk(f[5 * V], f[6 * V]);
    a.o[2] = mk(f[7 * V], f[8 * V]);
    return a;
}

// tr(A B) for anti-Hermitian A, B: -(sum a_i b_i + 2 Re sum_{i<j} A_ij conj(B_ij))
__device__ __forceinline__ double tr_ab(const Anti& a, const Anti& b) {
    double s = a.d[0] * b.d[0] + a.d[1] * b.d[1] + a.d[2] * b.d[2];
#pragma unroll
    for (int k = 0; k < 3; ++k) s += 2.0 * (a.o[k].re * b.o[k].re + a.o[k].im * b.o[k].im);
    return -s;
}

// planes in the order of the field tensor: 01 02 03 12 13 23
__global__ void __launch_bounds__(RED_THREADS) k_gauge_obs(int V, const double* __restrict__ F, double u1_norm,
                                                          double* __restrict__ partials) {
    double acc[3] = {0.0, 0.0, 0.0};
    for (int s = blockIdx.x * blockDim.x + threadIdx.x; s < V; s += gridDim.x * blockDim.x) {
        Anti f[6];
#pragma unroll
        for (int p = 0; p < 6; ++p) {
            f[p] = load_plane(F, (size_t)V, p, s);
            acc[0] -= tr_ab(f[p], f[p]);
            const double im = F[((size_t)p * 10 + 9) * V + s];
            acc[1] += im * im * u1_norm;
        }
        acc[2] += tr_ab(f[0], f[5]) - tr_ab(f[1], f[4]) + tr_ab(f[2], f[3]);
    }
    block_reduce_store<3>(acc, 3, partials);
}

// ---------------------------------------------------------------------------
// Wilson flow
// ---------------------------------------------------------------------------

// exp(X) for anti-Hermitian traceless X = i H (X: Im X_ii in d, upper entries
// in o). H is Hermitian and traceless, so H^3 = p H + q with p = tr(H^2)/2 and
// q = det H real, and every power is H^n = a_n + b_n H + c_n H^2 with
//   a_{n+1} = c_n q,  b_{n+1} = a_n + c_n p,  c_{n+1} = b_n
// (real), and exp(i H) = A + B H + C H^2 with A, B, C the sums of i^n a_n/n!
// and so on (the Taylor series, summed on these scalars). H is first scaled by
// 2^-k to |H|_F <= 1/2, where the terms up to n = 15 leave a remainder below
// 1e-18, and the result squared k times.
__device__ __forceinline__ M3 expi3(const AH& X0) {
    double n2 = 0.0;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        n2 = fma(X0.d[i], X0.d[i], n2);
        n2 = fma(2.0 * X0.o[i].re, X0.o[i].re, fma(2.0 * X0.o[i].im, X0.o[i].im, n2));
    }
    int k = 0;
    double sc = 1.0;
    while (n2 > 0.25 && k < 40) {
        n2 *= 0.25;
        sc *= 0.5;
        ++k;
    }
    // H = -i X: H_ii = Im X_ii, H_ij = -i X_ij
    double h[3];
    C64 o[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        h[i] = sc * X0.d[i];
        o[i] = sc * times_mi(X0.o[i]);
    }
    // H^2 (Hermitian): diagonal and the entries 01, 02, 12
    const double m01 = o[0].re * o[0].re + o[0].im * o[0].im, m02 = o[1].re * o[1].re + o[1].im * o[1].im,
                 m12 = o[2].re * o[2].re + o[2].im * o[2].im;
    const double s[3] = {fma(h[0], h[0], m01 + m02), fma(h[1], h[1], m01 + m12), fma(h[2], h[2], m02 + m12)};
    const C64 t[3] = {mulc(o[1], o[2]) + (h[0] + h[1]) * o[0], o[0] * o[2] + (h[0] + h[2]) * o[1],
                      cmul(o[0], o[1]) + (h[1] + h[2]) * o[2]};
    const double p = 0.5 * (s[0] + s[1] + s[2]);
    // det H = h0 h1 h2 + 2 Re(o01 o12 conj(o02)) - h0 m12 - h1 m02 - h2 m01
    const C64 oo = o[0] * o[2];
    const double q = h[0] * h[1] * h[2] + 2.0 * (oo.re * o[1].re + oo.im * o[1].im) - h[0] * m12 - h[1] * m02 - h[2] * m01;
    double a = 1.0, b = 0.0, c = 0.0;  // (a, b, c) / n!
    C64 A = mk(1.0, 0.0), B = mk(0.0, 0.0), Cc = mk(0.0, 0.0);
#pragma unroll
    for (int n = 1; n <= 15; ++n) {
        const double r = 1.0 / n;
        const double an = r * (c * q), bn = r * fma(c, p, a), cn = r * b;
        a = an;
        b = bn;
        c = cn;
        // i^n = 1, i, -1, -i
        if (n % 2) {
            A.im += n % 4 == 1 ? a : -a;
            B.im += n % 4 == 1 ? b : -b;
            Cc.im += n % 4 == 1 ? c : -c;
        } else {
            A.re += n % 4 == 0 ? a : -a;
            B.re += n % 4 == 0 ? b : -b;
            Cc.re += n % 4 == 0 ? c : -c;
        }
    }
    M3 E;
#pragma unroll
    for (int i = 0; i < 3; ++i) E.a[i][i] = rmad(s[i], Cc, rmad(h[i], B, A));
    const int oi[3] = {0, 0, 1}, oj[3] = {1, 2, 2};
#pragma unroll
    for (int e = 0; e < 3; ++e) {
        E.a[oi[e]][oj[e]] = mad(Cc, t[e], B * o[e]);
        E.a[oj[e]][oi[e]] = cmad(t[e], Cc, cmul(o[e], B));
    }
    for (int i = 0; i < k; ++i) E = mul(E, E);
    return E;
}

struct FlowStage {
    GaugeSet q;     // links integrated
    GaugeSet ql;    // plaquettes in buf (more than q only while the mirror half is not the exact conjugate)
    LeafBuf buf;
    double2* __restrict__ U;
    double* __restrict__ A;
    double* __restrict__ X;     // SU(3) accumulator, [4][9][n] (anti-Hermitian: 3 Im diag + 3 complex)
    double* __restrict__ Xa;    // U(1) accumulator, [4][n]
    double a, b;                // X <- a Z + b X (a includes eps)
};

__device__ __forceinline__ void store_link(double2* __restrict__ U, size_t V, int mu, int s, const M3& m, bool cj) {
#pragma unroll
    for (int e = 0; e < 9; ++e) {
        const C64 v = m.a[e / 3][e % 3];
        U[((size_t)mu * 9 + e) * V + s] = make_double2(v.re, cj ? -v.im : v.im);
    }
}

__device__ __forceinline__ double wrap_angle(double a) {
    const double pi = 3.14159265358979323846264338327950, two_pi = 6.283185307179586476925286766559;
    a += pi;
    if (!(a >= 0.0 && a < two_pi)) {  // fmod returns such a itself
        a = fmod(a, two_pi);
        if (a < 0.0) a += two_pi;
    }
    return a - pi;
}

// leaves of the plaquettes that the stage needs: three per plaquette
__global__ void __launch_bounds__(128) k_flow_leaves(GaugeSet q, const double2* __restrict__ U64,
                                                     const double* __restrict__ A64, LeafBuf buf) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t < q.n) plaquette_leaves<3>(q, U64, A64, blockIdx.y, t, buf);
}

// One thread per link. U(x,mu) times its staples is a sum of leaves through x:
// in plane (mu, nu), mu < nu, the link mu has the leaf from x and the adjoint
// of the one that plaquette x - nu shows to its corner y + nu; the link nu has
// the adjoint of the leaf from x and the one that plaquette x - mu shows to y +
// mu. So W = U S needs no product here: Z = -1/2 (W - W^+) + 1/6 tr(W - W^+) is
// a sum of six stored anti-Hermitian parts.
__global__ void __launch_bounds__(128) k_flow_link(FlowStage f) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= f.q.n) return;
    const int mu = blockIdx.y;
    const Geom& g = f.q.g;
    const size_t V = (size_t)g.V, n = f.q.n;
    int x[4];
    set_coords(f.q, t, x);
    bool never;
    const int own = set_index(f.ql, x, never);
    AH w{};  // Im W_ii and W_ij - conj(W_ji)
    double zu1 = 0.0;
    for (int nu = 0; nu < 4; ++nu) {
        if (nu == mu) continue;
        const bool first = mu < nu;
        const int plane = first ? plane_of(mu, nu) : plane_of(nu, mu);
        int c[4] = {x[0], x[1], x[2], x[3]};
        shift_coords(g, c, nu, -1);
        bool flip;
        const int y = set_index(f.ql, c, flip);
        const AH up = load_ah(f.buf.leaf<3>(plane, 0) + own, f.buf.n);
        const AH dn = load_ah(f.buf.leaf<3>(plane, first ? 2 : 1) + y, f.buf.n);
        const double sg = first ? 1.0 : -1.0, sf = flip ? -sg : sg;  // flip: conjugate dn
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            w.d[i] = fma(-sf, dn.d[i], fma(sg, up.d[i], w.d[i]));
            w.o[i].re = fma(-sg, dn.o[i].re, fma(sg, up.o[i].re, w.o[i].re));
            w.o[i].im = fma(-sf, dn.o[i].im, fma(sg, up.o[i].im, w.o[i].im));
        }
        // theta_munu(x) and theta_munu(x - nu)
        const double sx = f.buf.sines(plane)[own], sy = f.buf.sines(plane)[y];
        zu1 -= sg * (sx - (flip ? -sy : sy));
    }
    const double trim = (w.d[0] + w.d[1] + w.d[2]) * (1.0 / 3.0);
    double* X = f.X + (size_t)mu * 9 * n + t;
    AH xn;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        // Z_ii = -i Im W_ii + i (1/3) Im tr W, Z_ij = -1/2 (W_ij - conj(W_ji))
        xn.d[i] = f.a * (trim - w.d[i]);
        xn.o[i] = (-0.5 * f.a) * w.o[i];
    }
    if (f.b != 0.0) {
        const AH old = load_ah(X, n);
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            xn.d[i] = fma(f.b, old.d[i], xn.d[i]);
            xn.o[i] = rmad(f.b, old.o[i], xn.o[i]);
        }
    }
    store_ah(X, n, xn);
    const int s = native_of(g, x);
    const M3 Unew = mul(expi3(xn), load_link64(f.U, V, mu, s));
    double xa = f.a * zu1;
    if (f.b != 0.0) xa += f.b * f.Xa[mu * n + t];
    f.Xa[mu * n + t] = xa;
    const double anew = wrap_angle(f.A[mu * V + s] + xa);
    store_link(f.U, V, mu, s, Unew, false);
    f.A[mu * V + s] = anew;
    if (f.q.mirror) {
        x[1] += g.L1;
        const int sm = native_of(g, x);
        store_link(f.U, V, mu, sm, Unew, true);
        f.A[mu * V + sm] = -anew;
    }
}

// FP32 two-row links, FP32 angles and z = exp(iA) from the FP64 field
__global__ void k_gauge_derive(Geom g, const double2* __restrict__ U64, const double* __restrict__ A64,
                               float4* __restrict__ U32, double2* __restrict__ Z64, float4* __restrict__ A32) {
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= g.V) return;
    const size_t V = (size_t)g.V;
    float a32[4];
    for (int mu = 0; mu < 4; ++mu) {
        double2 u[6];
#pragma unroll
        for (int e = 0; e < 6; ++e) u[e] = U64[((size_t)mu * 9 + e) * V + s];
        U32[((size_t)mu * 3 + 0) * V + s] = make_float4((float)u[0].x, (float)u[0].y, (float)u[1].x, (float)u[1].y);
        U32[((size_t)mu * 3 + 1) * V + s] = make_float4((float)u[2].x, (float)u[2].y, (float)u[3].x, (float)u[3].y);
        U32[((size_t)mu * 3 + 2) * V + s] = make_float4((float)u[4].x, (float)u[4].y, (float)u[5].x, (float)u[5].y);
        const double a = A64[(size_t)mu * V + s];
        double sa, ca;
        sincos(a, &sa, &ca);
        Z64[(size_t)mu * V + s] = make_double2(ca, sa);
        a32[mu] = (float)a;
    }
    A32[s] = make_float4(a32[0], a32[1], a32[2], a32[3]);
}

}  // namespace

}  // namespace qxd

using namespace qxd;

extern "C" {

int qxd_gauge_observables(qxd_lattice* lat, double q_el, double* out) {
    if (!lat || !out) return fail(QXD_ERR_ARG, "qxd_gauge_observables: NULL argument");
    if (!(q_el > 0.0) || !std::isfinite(q_el)) return fail(QXD_ERR_ARG, "qxd_gauge_observables: q_el > 0 required");
    const qxd_lattice* own = gauge_owner(lat);
    if (!own->has_gauge) return fail(QXD_ERR_STATE, "qxd_gauge_observables: needs qxd_set_gauge first");
    Reducer red;
    int rc = red.init();
    if (rc) return rc;
    const Geom& g = lat->g;
    const double u1_norm = 1.0 / (16.0 * q_el * q_el);
    k_gauge_obs<<<RED_BLOCKS, RED_THREADS, 0, lat->stream>>>(g.V, own->ftens, u1_norm, red.partials);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) {
        red.release();
        return cuda_fail(e, "k_gauge_obs");
    }
    rc = reduce_finish(red, 3, lat->stream);
    if (!rc) {
        const double V = (double)g.V;
        const double w = (lat->cstar_mask & 2u) ? 0.5 : 1.0;
        const double pi = 3.14159265358979323846264338327950;
        out[0] = red.h_res[0] / V;
        out[1] = red.h_res[1] / V;
        out[2] = w * red.h_res[2] / (4.0 * pi * pi);
    }
    red.release();
    return rc;
}

int qxd_wflow(qxd_lattice* lat, double eps, int nsteps) {
    if (!lat) return fail(QXD_ERR_ARG, "qxd_wflow: lat is NULL");
    if (lat->parent) return fail(QXD_ERR_STATE, "qxd_wflow: a view shares its parent's gauge field; flow the parent");
    if (!lat->has_gauge) return fail(QXD_ERR_STATE, "qxd_wflow: needs qxd_set_gauge first");
    if (!std::isfinite(eps) || nsteps < 0) return fail(QXD_ERR_ARG, "qxd_wflow: finite eps and nsteps >= 0 required");
    if (nsteps == 0) return QXD_OK;
    const Geom& g = lat->g;
    const size_t V = (size_t)g.V;
    const bool cstar1 = lat->cstar_mask & 2u;
    // Work space: the operator's arrays, stale after the flow. The three leaves
    // of the six planes take 162 V doubles of leaf_buf's 216 V; the accumulators
    // (36 V and 4 V) lie behind them.
    const GaugeSet q = gauge_set(g, cstar1);
    double* X = leaf_buf(lat, q.n).b + (size_t)6 * 3 * 9 * V;
    double* Xa = X + 4 * 9 * V;
    static_assert(6 * 3 * 9 + 4 * 9 + 4 <= LEAF_REALS, "accumulators before the sines");
    const double coef[3][2] = {{0.25, 0.0}, {8.0 / 9.0, -17.0 / 9.0}, {0.75, -1.0}};
    bool exact = mirror_exact(lat);
    lat->has_clover = false;
    int rc;
    cudaError_t e = cudaSuccess;
    for (int step = 0; step < nsteps && e == cudaSuccess; ++step)
        for (int k = 0; k < 3 && e == cudaSuccess; ++k) {
            // every update sets the mirror links to the conjugates of the physical ones
            const GaugeSet ql = gauge_set(g, cstar1 && (exact || step || k));
            const FlowStage f{q, ql, leaf_buf(lat, ql.n), lat->U64, lat->A64, X, Xa, coef[k][0] * eps, coef[k][1]};
            k_flow_leaves<<<dim3((ql.n + 127) / 128, 6), 128, 0, lat->stream>>>(ql, lat->U64, lat->A64, f.buf);
            k_flow_link<<<dim3((q.n + 127) / 128, 4), 128, 0, lat->stream>>>(f);
            e = cudaGetLastError();
        }
    lat->mirror_built = cstar1;
    if (e == cudaSuccess) {
        k_gauge_derive<<<(g.V + 127) / 128, 128, 0, lat->stream>>>(g, lat->U64, lat->A64, lat->U32, lat->Z64,
                                                                   lat->A32);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaStreamSynchronize(lat->stream);
    // the clover terms of this lattice and its views are now stale
    ++lat->gauge_version;
    if (e != cudaSuccess) {
        // the field may be part-way through a step: unusable until set again
        lat->has_gauge = false;
        return cuda_fail(e, "qxd_wflow");
    }
    if ((rc = launch_field_tensor(lat))) {
        lat->has_gauge = false;
        return rc;
    }
    e = cudaStreamSynchronize(lat->stream);
    if (e != cudaSuccess) {
        lat->has_gauge = false;
        return cuda_fail(e, "qxd_wflow: field tensor");
    }
    return QXD_OK;
}

}  // extern "C"
