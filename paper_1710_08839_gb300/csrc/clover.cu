// Site-diagonal part of D: M(x) = (4 + m0) + dDsw(x) (Eqs. (16), (21)) as two
// Hermitian 6x6 blocks per site, and their inverses (Doo^-1 of Sec. 2.4).
//
// In the chiral basis sigma_0k = diag(s_k, -s_k) and sigma_ij =
// -eps_ijk diag(s_k, s_k), so with X_munu = csw F_hat_munu + cswqed qhat
// (i/4) Im{4 plaquettes} (anti-Hermitian 3x3) the sum over mu, nu of
// (i/4) sigma_munu X_munu is block diagonal:
//   block +/- = (i/2) sum_k s_k (x) Y_k,  Y_k = +/- X_0k - E_k,
//   E_1 = X_23, E_2 = X_31, E_3 = X_12,
// i.e. (1/2) [[ i Y3, i Y1 + Y2 ], [ i Y1 - Y2, -i Y3 ]] on (spin a, colour).
#include "herm6.cuh"
#include "su3.cuh"

namespace qxd {

namespace {

struct AH3 {  // anti-Hermitian 3x3
    C64 a[3][3];
};

__device__ __forceinline__ AH3 load_plane(const double* __restrict__ F, size_t V, int s, int plane,
                                          double csw, double u1) {
    const double* f = F + (size_t)plane * 10 * V + s;
    AH3 X;
    double im_u1 = u1 * f[9 * V];
    X.a[0][0] = mk(0.0, csw * f[0] + im_u1);
    X.a[1][1] = mk(0.0, csw * f[1 * V] + im_u1);
    X.a[2][2] = mk(0.0, csw * f[2 * V] + im_u1);
    X.a[0][1] = mk(csw * f[3 * V], csw * f[4 * V]);
    X.a[0][2] = mk(csw * f[5 * V], csw * f[6 * V]);
    X.a[1][2] = mk(csw * f[7 * V], csw * f[8 * V]);
    X.a[1][0] = -conj(X.a[0][1]);
    X.a[2][0] = -conj(X.a[0][2]);
    X.a[2][1] = -conj(X.a[1][2]);
    return X;
}

__device__ __forceinline__ double cabs2(C64 a) { return a.re * a.re + a.im * a.im; }

// Gauss-Jordan inverse with partial pivoting; false if singular/non-finite.
__device__ bool invert6(const C64 H[6][6], C64 B[6][6]) {
    C64 A[6][6];
    double nrm = 0.0;
    for (int i = 0; i < 6; ++i) {
        double rs = 0.0;
        for (int j = 0; j < 6; ++j) {
            A[i][j] = H[i][j];
            B[i][j] = mk(i == j ? 1.0 : 0.0, 0.0);
            rs += sqrt(cabs2(H[i][j]));
        }
        nrm = fmax(nrm, rs);
    }
    if (!isfinite(nrm) || nrm == 0.0) return false;
    for (int k = 0; k < 6; ++k) {
        int piv = k;
        double best = cabs2(A[k][k]);
        for (int i = k + 1; i < 6; ++i) {
            double v = cabs2(A[i][k]);
            if (v > best) {
                best = v;
                piv = i;
            }
        }
        if (!(sqrt(best) >= 1e-12 * nrm)) return false;
        if (piv != k)
            for (int j = 0; j < 6; ++j) {
                C64 t = A[k][j];
                A[k][j] = A[piv][j];
                A[piv][j] = t;
                t = B[k][j];
                B[k][j] = B[piv][j];
                B[piv][j] = t;
            }
        C64 d = A[k][k];
        double id = 1.0 / cabs2(d);
        C64 inv = mk(d.re * id, -d.im * id);
        for (int j = 0; j < 6; ++j) {
            A[k][j] = A[k][j] * inv;
            B[k][j] = B[k][j] * inv;
        }
        for (int i = 0; i < 6; ++i) {
            if (i == k) continue;
            C64 f = A[i][k];
            for (int j = 0; j < 6; ++j) {
                A[i][j] = A[i][j] - f * A[k][j];
                B[i][j] = B[i][j] - f * B[k][j];
            }
        }
    }
    for (int i = 0; i < 6; ++i)
        for (int j = 0; j < 6; ++j)
            if (!isfinite(B[i][j].re) || !isfinite(B[i][j].im)) return false;
    return true;
}

// Inverse of a packed Hermitian 6x6 block, all in registers: A = L D L^H,
// A^-1 = M^H D^-1 M with M = L^-1. Returns false when a pivot falls below
// 1e-12 of the block norm (the caller then uses Gauss-Jordan with pivoting,
// which decides singularity).
__device__ __forceinline__ bool ldl_inverse6(const double a_d[6], const C64 a_l[15], double nrm, double i_d[6],
                                             C64 i_l[15]) {
    double D[6], iD[6];
    C64 L[15];
    if (!ldl6(a_d, a_l, 1e-12 * nrm, D, iD, L)) return false;
    // M = L^-1 (unit lower triangular)
    C64 M[15];
#pragma unroll
    for (int j = 0; j < 6; ++j)
#pragma unroll
        for (int i = j + 1; i < 6; ++i) {
            C64 v = -L[lidx6(i, j)];
#pragma unroll
            for (int k = j + 1; k < i; ++k) v = mad(-L[lidx6(i, k)], M[lidx6(k, j)], v);
            M[lidx6(i, j)] = v;
        }
    // (A^-1)_ij = sum_{k >= i} conj(M_ki) M_kj / D_k for i >= j (M_kk = 1)
#pragma unroll
    for (int i = 0; i < 6; ++i) {
        double v = iD[i];
        C64 s[6];  // M_ki / D_k
#pragma unroll
        for (int k = i + 1; k < 6; ++k) {
            const C64 m = M[lidx6(k, i)];
            s[k] = iD[k] * m;
            v = fma(s[k].re, m.re, fma(s[k].im, m.im, v));
        }
        i_d[i] = v;
#pragma unroll
        for (int j = 0; j < i; ++j) {
            C64 w = iD[i] * M[lidx6(i, j)];
#pragma unroll
            for (int k = i + 1; k < 6; ++k) w = cmad(s[k], M[lidx6(k, j)], w);
            i_l[lidx6(i, j)] = w;
        }
    }
    for (int i = 0; i < 6; ++i)
        if (!isfinite(i_d[i])) return false;
    return true;
}

// Block of the mirror site: with F -> F^* and the U(1) term reversed, the block
// H = (1/2) [[i Y3, i Y1 + Y2], [i Y1 - Y2, -i Y3]] + 4 + m0 becomes e H^* e^T
// with the spin flip e = [[0, 1], [-1, 0]], and so does its inverse.
__device__ __forceinline__ void spin_flip_conj(double d[6], C64 l[15]) {
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const double t = d[a];
        d[a] = d[3 + a];
        d[3 + a] = t;
    }
    // diagonal colour blocks trade places, conjugated
#pragma unroll
    for (int a = 1; a < 3; ++a)
#pragma unroll
        for (int b = 0; b < a; ++b) {
            const C64 t = conj(l[lidx6(a, b)]);
            l[lidx6(a, b)] = conj(l[lidx6(3 + a, 3 + b)]);
            l[lidx6(3 + a, 3 + b)] = t;
        }
    // lower-left colour block B -> -(B^+)^* = -B^T
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int b = a; b < 3; ++b) {
            const C64 t = -l[lidx6(3 + a, b)];
            l[lidx6(3 + a, b)] = -l[lidx6(3 + b, a)];
            l[lidx6(3 + b, a)] = t;
        }
}

// V: entries of the array per real, s: the site's
__device__ __forceinline__ void store_packed(const double d[6], const C64 l[15], int blk, double* __restrict__ C64p,
                                             float4* __restrict__ C32p, size_t V, int s) {
    double v[36];
#pragma unroll
    for (int i = 0; i < 6; ++i) v[i] = d[i];
#pragma unroll
    for (int k = 0; k < 15; ++k) {
        v[6 + 2 * k] = l[k].re;
        v[7 + 2 * k] = l[k].im;
    }
#pragma unroll
    for (int r = 0; r < 36; ++r) C64p[(size_t)(36 * blk + r) * V + s] = v[r];
#pragma unroll
    for (int q = 0; q < 9; ++q)
        C32p[(size_t)(9 * blk + q) * V + s] =
            make_float4((float)v[4 * q], (float)v[4 * q + 1], (float)v[4 * q + 2], (float)v[4 * q + 3]);
}

// One thread per (site, block): assemble the block from the field tensors,
// store it, invert it (LDL^H, Gauss-Jordan with pivoting as the fallback; on the
// even sites this only tells whether it is singular); with an exact mirror half
// both blocks of the mirror site follow. Bound by the FP64
// units. 48x48x24x24 sites: 1.96 ms; 5.24 ms for every site by itself, with 20
// square roots and 40 divisions a block.
__global__ void __launch_bounds__(128) k_clover_build(GaugeSet q, const double* __restrict__ F, double m0,
                                                      double csw, double u1coef, double* __restrict__ C64p,
                                                      float4* __restrict__ C32p, double* __restrict__ Ci64,
                                                      float4* __restrict__ Ci32, int* __restrict__ bad) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= q.n) return;
    const int blk = blockIdx.y;
    const Geom& g = q.g;
    const size_t V = (size_t)g.V;
    int x[4];
    set_coords(q, t, x);
    const int s = native_of(g, x);
    const double sg = blk == 0 ? 1.0 : -1.0;
    // planes: 0:(0,1) 1:(0,2) 2:(0,3) 3:(1,2) 4:(1,3) 5:(2,3)
    AH3 Y1, Y2, Y3;
    {
        AH3 X0 = load_plane(F, V, s, 0, csw, u1coef), X5 = load_plane(F, V, s, 5, csw, u1coef);
#pragma unroll
        for (int a = 0; a < 3; ++a)
#pragma unroll
            for (int b = 0; b < 3; ++b) Y1.a[a][b] = sg * X0.a[a][b] - X5.a[a][b];  // E1 = X23
    }
    {
        AH3 X1 = load_plane(F, V, s, 1, csw, u1coef), X4 = load_plane(F, V, s, 4, csw, u1coef);
#pragma unroll
        for (int a = 0; a < 3; ++a)
#pragma unroll
            for (int b = 0; b < 3; ++b) Y2.a[a][b] = sg * X1.a[a][b] + X4.a[a][b];  // E2 = X31 = -X13
    }
    {
        AH3 X2 = load_plane(F, V, s, 2, csw, u1coef), X3 = load_plane(F, V, s, 3, csw, u1coef);
#pragma unroll
        for (int a = 0; a < 3; ++a)
#pragma unroll
            for (int b = 0; b < 3; ++b) Y3.a[a][b] = sg * X2.a[a][b] - X3.a[a][b];  // E3 = X12
    }
    // packed Hermitian block (1/2) [[ i Y3, i Y1 + Y2 ], [ i Y1 - Y2, -i Y3 ]] + (4 + m0)
    double d[6];
    C64 l[15];
#pragma unroll
    for (int i = 0; i < 6; ++i) {
        const int a = i % 3, sa = i / 3;
        const C64 yy = sa == 0 ? 0.5 * times_i(Y3.a[a][a]) : 0.5 * times_mi(Y3.a[a][a]);
        d[i] = 4.0 + m0 + yy.re;
#pragma unroll
        for (int j = 0; j < i; ++j) {
            const int b = j % 3, sb = j / 3;
            C64 h;
            if (sa == sb) h = sa == 0 ? 0.5 * times_i(Y3.a[a][b]) : 0.5 * times_mi(Y3.a[a][b]);
            else h = 0.5 * (times_i(Y1.a[a][b]) - Y2.a[a][b]);  // lower-left block (sa = 1, sb = 0)
            l[lidx6(i, j)] = h;
        }
    }
    store_packed(d, l, blk, C64p, C32p, V, s);
    const double nrm = herm6_bound(d, l);
    double id[6];
    C64 il[15];
    // (sizes whose squares could overflow go to the pivoted form)
    bool ok = nrm <= 1e150 && nrm > 0.0 && ldl_inverse6(d, l, nrm, id, il);
    if (!ok) {
        C64 H[6][6], Hi[6][6];
        for (int i = 0; i < 6; ++i) {
            H[i][i] = mk(d[i], 0.0);
            for (int j = 0; j < i; ++j) {
                H[i][j] = l[lidx6(i, j)];
                H[j][i] = conj(l[lidx6(i, j)]);
            }
        }
        ok = invert6(H, Hi);
        for (int i = 0; i < 6; ++i) {
            id[i] = ok ? Hi[i][i].re : 0.0;
            for (int j = 0; j < i; ++j) il[lidx6(i, j)] = ok ? Hi[i][j] : mk(0.0, 0.0);
        }
        if (!ok) atomicAdd(&bad[0], q.mirror ? 2 : 1);
    }
    const bool odd = s >= g.Vh;  // and the mirror site with it: L1 is even
    if (odd) store_packed(id, il, blk, Ci64, Ci32, g.Vh, s - g.Vh);
    if (q.mirror) {
        x[1] += g.L1;
        const int sm = native_of(g, x);
        spin_flip_conj(d, l);
        store_packed(d, l, blk, C64p, C32p, V, sm);
        if (odd) {
            spin_flip_conj(id, il);
            store_packed(id, il, blk, Ci64, Ci32, g.Vh, sm - g.Vh);
        }
    }
}

// W = -1/2 z^qhat U per link, the link of the FP64 hops: z^qhat from z =
// exp(i A) by binary powering (|z| = 1, so z^-n = conj(z^n)). With an exact
// mirror half the mirror link is the conjugate.
__global__ void k_hop_links(GaugeSet q, const double2* __restrict__ Z, const double2* __restrict__ U, int qhat,
                            double2* __restrict__ W) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= q.n) return;
    const int mu = blockIdx.y;
    const Geom& g = q.g;
    const size_t V = (size_t)g.V;
    int x[4];
    set_coords(q, t, x);
    const int s = native_of(g, x);
    const double2 z = Z[mu * V + s];
    C64 b = mk(z.x, z.y), r = mk(1.0, 0.0);
    int m = qhat < 0 ? -qhat : qhat;
    while (m) {
        if (m & 1) r = r * b;
        b = b * b;
        m >>= 1;
    }
    if (qhat < 0) r = conj(r);
    r = -0.5 * r;
    x[1] += g.L1;
    const int sm = q.mirror ? native_of(g, x) : 0;
#pragma unroll
    for (int e = 0; e < 9; ++e) {
        const size_t k = ((size_t)mu * 9 + e) * V;
        const C64 w = r * mk(U[k + s].x, U[k + s].y);
        W[k + s] = make_double2(w.re, w.im);
        if (q.mirror) W[k + sm] = make_double2(w.re, -w.im);
    }
}

}  // namespace

int launch_clover_build(qxd_lattice* lat, int* d_bad) {
    const Geom& g = lat->g;
    QXD_CUDA(cudaMemsetAsync(d_bad, 0, 16, lat->stream));
    // U(1) part of X: cswqed * qhat * (i/4) Im{sum of 4 plaquettes}
    const double u1coef = lat->cswqed * (double)lat->qhat * 0.25;
    const GaugeSet q = gauge_set(g, mirror_exact(gauge_owner(lat)));
    k_clover_build<<<dim3((q.n + 127) / 128, 2), 128, 0, lat->stream>>>(q, lat->ftens, lat->m0, lat->csw, u1coef, lat->C64,
                                                                        lat->C32, lat->Cinv64, lat->Cinv32, d_bad);
    QXD_LAUNCHED("k_clover_build");
    k_hop_links<<<dim3((q.n + 255) / 256, 4), 256, 0, lat->stream>>>(q, lat->Z64, lat->U64, lat->qhat, lat->W64);
    QXD_LAUNCHED("k_hop_links");
    return QXD_OK;
}

}  // namespace qxd
