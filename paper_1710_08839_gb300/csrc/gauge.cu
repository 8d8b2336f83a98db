// Gauge-field ingest (orbifold mirror, Eq. (4a); SU(3) check; FP64 and FP32
// 2-row layouts) and the clover field tensors of the SW term (Eqs. (21)-(23)).
#include "su3.cuh"

namespace qxd {

namespace {

// One thread per link; a physical-half input is read and checked once and
// written to both halves (Eq. (4a): U^* and -A on the mirror site). Bound by
// the FP64 units (unitarity and determinant, sincos) and the 880 bytes a site
// takes in both precisions.
__global__ void __launch_bounds__(256) k_gauge_ingest(GaugeSet q, const double* __restrict__ su3,
                                                      const double* __restrict__ ang, double2* __restrict__ U64,
                                                      float4* __restrict__ U32, double* __restrict__ A64,
                                                      double2* __restrict__ Z64, float4* __restrict__ A32,
                                                      int* __restrict__ bad) {
    const size_t i4 = (size_t)blockIdx.x * blockDim.x + threadIdx.x;  // the four links of a site side by side
    const int t = (int)(i4 >> 2), mu = (int)(i4 & 3);
    if (t >= q.n) return;
    const Geom& g = q.g;
    const size_t V = (size_t)g.V;
    int x[4];
    set_coords(q, t, x);
    const size_t src = (((size_t)x[0] * q.n1 + x[1]) * g.N2 + x[2]) * g.N3 + x[3];
    const double* p = su3 + (src * 4 + mu) * 18;
    C64 u[3][3];
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j) u[i][j] = mk(p[(i * 3 + j) * 2], p[(i * 3 + j) * 2 + 1]);
    const double a = ang[src * 4 + mu];
    // SU(3) check: |U U^+ - 1| (Hermitian: the entries on and above the diagonal) and |det U - 1|, each entry compared
    // by itself (a maximum of them would drop a NaN)
    bool ok = isfinite(a);
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = i; j < 3; ++j) {
            const C64 s2 = cmad(u[j][2], u[i][2], cmad(u[j][1], u[i][1], mulc(u[i][0], u[j][0])));
            ok = ok && fabs(s2.re - (i == j ? 1.0 : 0.0)) <= 1e-10 && fabs(s2.im) <= 1e-10;
        }
    const C64 m0 = u[1][1] * u[2][2] - u[1][2] * u[2][1], m1 = u[1][2] * u[2][0] - u[1][0] * u[2][2],
              m2 = u[1][0] * u[2][1] - u[1][1] * u[2][0];
    const C64 det = mad(u[0][2], m2, mad(u[0][1], m1, u[0][0] * m0));
    ok = ok && fabs(det.re - 1.0) <= 1e-10 && fabs(det.im) <= 1e-10;
    if (!ok) atomicAdd(&bad[0], q.mirror ? 2 : 1);
    double sa, ca;
    sincos(a, &sa, &ca);
    for (int m = 0; m <= q.mirror; ++m) {
        const int s = native_of(g, x);
        const double sg = m ? -1.0 : 1.0;
#pragma unroll
        for (int e = 0; e < 9; ++e) U64[((size_t)mu * 9 + e) * V + s] = make_double2(u[e / 3][e % 3].re, sg * u[e / 3][e % 3].im);
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const C64 v = u[2 * k / 3][2 * k % 3], w = u[(2 * k + 1) / 3][(2 * k + 1) % 3];
            U32[((size_t)mu * 3 + k) * V + s] = make_float4((float)v.re, (float)(sg * v.im), (float)w.re, (float)(sg * w.im));
        }
        A64[(size_t)mu * V + s] = sg * a;
        Z64[(size_t)mu * V + s] = make_double2(ca, sg * sa);
        reinterpret_cast<float*>(A32 + s)[mu] = (float)(sg * a);
        x[1] += g.L1;
    }
}

// Extended input with the CHECKED flag: mirror site x (x1 >= L1) must hold
// U(x - L1 e1)^* and -A(x - L1 e1) (Eq. (4a)), compared on z = exp(iA).
__global__ void k_check_admissible(Geom g, const double* __restrict__ su3, const double* __restrict__ ang,
                                   int* __restrict__ bad) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= g.V) return;
    int x3 = i % g.N3, r = i / g.N3;
    int x2 = r % g.N2;
    r /= g.N2;
    int x1 = r % g.N1, x0 = r / g.N1;
    if (x1 < g.L1) return;
    size_t m = (size_t)i, p = (size_t)lex_index(g, x0, x1 - g.L1, x2, x3);
    int nbad = 0;
    for (int mu = 0; mu < 4; ++mu) {
        bool ok = true;
        for (int e = 0; e < 9; ++e) {
            double mre = su3[(m * 4 + mu) * 18 + 2 * e], mim = su3[(m * 4 + mu) * 18 + 2 * e + 1];
            double pre = su3[(p * 4 + mu) * 18 + 2 * e], pim = su3[(p * 4 + mu) * 18 + 2 * e + 1];
            ok = ok && fabs(mre - pre) <= 1e-12 && fabs(mim + pim) <= 1e-12;
        }
        double am = ang[m * 4 + mu], ap = ang[p * 4 + mu];
        double sm, cm, sp, cp;
        sincos(am, &sm, &cm);
        sincos(ap, &sp, &cp);
        ok = ok && fabs(cm - cp) <= 1e-12 && fabs(sm + sp) <= 1e-12;
        if (!ok) ++nbad;
    }
    if (nbad) atomicAdd(&bad[1], nbad);
}

// Clover field tensors (FP64): per plane mu < nu the SU(3) F_hat = (Q_munu -
// Q_munu^+)/8 with Q the four leaves through x (Q_numu = Q_munu^+), and the
// imaginary part of the sum of the four U(1) plaquettes z_munu(x) +
// z_munu(x-mu) + z_munu(x-nu) + z_munu(x-mu-nu) (Eqs. (22)-(23)). Bound by the
// FP64 units: first the leaves of every plaquette (plaquette_leaves), then
// their sums, for one or (exact mirror) half of the sites. 48x48x24x24 sites:
// 5.45 + 0.39 ms, 0.98 of the FP64 issue rate for 852 instructions per
// plaquette; 25.7 ms with the leaves of every site taken one by one.
__global__ void __launch_bounds__(128) k_leaves(GaugeSet q, const double2* __restrict__ U64,
                                                const double* __restrict__ A64, LeafBuf buf) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t < q.n) plaquette_leaves<4>(q, U64, A64, blockIdx.y, t, buf);
}

__global__ void __launch_bounds__(256) k_tensor_sum(GaugeSet q, LeafBuf buf, double* __restrict__ F) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= q.n) return;
    const Geom& g = q.g;
    const size_t V = (size_t)g.V;
    const int plane = blockIdx.y;
    int mu, nu, x[4], c[4];
    plane_dirs(plane, mu, nu);
    set_coords(q, t, x);
    AH f = load_ah(buf.leaf<4>(plane, 0) + t, q.n);
    double im = buf.sines(plane)[t];
    auto add = [&](int leaf, bool bm, bool bn) {
        c[0] = x[0]; c[1] = x[1]; c[2] = x[2]; c[3] = x[3];
        if (bm) shift_coords(g, c, mu, -1);
        if (bn) shift_coords(g, c, nu, -1);
        bool flip;
        const int y = set_index(q, c, flip);
        const AH l = load_ah(buf.leaf<4>(plane, leaf) + y, q.n);
        const double sf = flip ? -1.0 : 1.0;  // conjugate: Im P_ii and the imaginary parts change sign
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            f.d[i] = fma(sf, l.d[i], f.d[i]);
            f.o[i] = mk(f.o[i].re + l.o[i].re, fma(sf, l.o[i].im, f.o[i].im));
        }
        const double sn = buf.sines(plane)[y];
        im += flip ? -sn : sn;
    };
    add(1, true, false);
    add(2, false, true);
    add(3, true, true);
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        f.d[i] *= 0.25;
        f.o[i] = 0.125 * f.o[i];
    }
    double* out = F + (size_t)plane * 10 * V;
    const int s = native_of(g, x);
    store_ah(out + s, V, f);
    out[9 * V + s] = im;
    if (q.mirror) {  // the mirror site holds the conjugate
        x[1] += g.L1;
        const int sm = native_of(g, x);
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            f.d[i] = -f.d[i];
            f.o[i] = conj(f.o[i]);
        }
        store_ah(out + sm, V, f);
        out[9 * V + sm] = -im;
    }
}

}  // namespace

int launch_gauge_ingest(qxd_lattice* lat, const double* su3, const double* ang, int kind, int* d_bad) {
    const Geom& g = lat->g;
    QXD_CUDA(cudaMemsetAsync(d_bad, 0, 16, lat->stream));
    const int cstar1 = (lat->cstar_mask & 2u) ? 1 : 0;
    lat->mirror_built = cstar1 && kind == QXD_GAUGE_PHYSICAL_HALF;
    const GaugeSet q = gauge_set(g, mirror_exact(lat));
    const int blocks = (g.V + 127) / 128;
    k_gauge_ingest<<<(int)(((size_t)q.n * 4 + 255) / 256), 256, 0, lat->stream>>>(q, su3, ang, lat->U64, lat->U32, lat->A64,
                                                                                lat->Z64, lat->A32, d_bad);
    QXD_LAUNCHED("k_gauge_ingest");
    if (kind == QXD_GAUGE_EXTENDED_CHECKED && cstar1) {
        k_check_admissible<<<blocks, 128, 0, lat->stream>>>(g, su3, ang, d_bad);
        QXD_LAUNCHED("k_check_admissible");
    }
    return QXD_OK;
}

int launch_field_tensor(qxd_lattice* lat) {
    const GaugeSet q = gauge_set(lat->g, mirror_exact(lat));
    const LeafBuf buf = leaf_buf(lat, q.n);
    k_leaves<<<dim3((q.n + 127) / 128, 6), 128, 0, lat->stream>>>(q, lat->U64, lat->A64, buf);
    QXD_LAUNCHED("k_leaves");
    k_tensor_sum<<<dim3((q.n + 255) / 256, 6), 256, 0, lat->stream>>>(q, buf, lat->ftens);
    QXD_LAUNCHED("k_tensor_sum");
    return QXD_OK;
}

}  // namespace qxd
