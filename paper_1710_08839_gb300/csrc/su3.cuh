// FP64 3x3 complex matrices and link/neighbour access of the gauge field
// (links in the native layout U64[mu][9][V], site coordinates on the
// simulated lattice with the shifted C* boundaries).
#pragma once

#include "qxd_internal.cuh"

namespace qxd {

namespace {

using C64 = cplx<double>;

struct M3 {
    C64 a[3][3];
};

__device__ __forceinline__ M3 mul(const M3& x, const M3& y) {
    M3 r;
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j)
            r.a[i][j] = mad(x.a[i][2], y.a[2][j], mad(x.a[i][1], y.a[1][j], x.a[i][0] * y.a[0][j]));
    return r;
}

// x * y^+
__device__ __forceinline__ M3 mul_nd(const M3& x, const M3& y) {
    M3 r;
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j)
            r.a[i][j] = cmad(y.a[j][2], x.a[i][2], cmad(y.a[j][1], x.a[i][1], mulc(x.a[i][0], y.a[j][0])));
    return r;
}

// x^+ * y
__device__ __forceinline__ M3 mul_dn(const M3& x, const M3& y) {
    M3 r;
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j)
            r.a[i][j] = cmad(x.a[2][i], y.a[2][j], cmad(x.a[1][i], y.a[1][j], cmul(x.a[0][i], y.a[0][j])));
    return r;
}

// Anti-Hermitian part of a product, the nine reals kept of every leaf: Im P_ii
// and P_ij - conj(P_ji) for (i, j) = (0,1), (0,2), (1,2). P_ij = sum_k x(i,k)
// y(k,j); XD, YD: that factor daggered. 90 instructions instead of 108 and 9
// for the difference.
struct AH {
    double d[3];
    C64 o[3];
};

template <bool XD, bool YD>
__device__ __forceinline__ AH ah_mul(const M3& x, const M3& y) {
    auto X = [&](int i, int k) { return XD ? conj(x.a[k][i]) : x.a[i][k]; };
    auto Y = [&](int k, int j) { return YD ? conj(y.a[j][k]) : y.a[k][j]; };
    AH r;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        double s = 0.0;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const C64 a = X(i, k), b = Y(k, i);
            s = k == 0 ? fma(a.re, b.im, a.im * b.re) : fma(a.re, b.im, fma(a.im, b.re, s));
        }
        r.d[i] = s;
    }
    const int oi[3] = {0, 0, 1}, oj[3] = {1, 2, 2};
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        const int i = oi[q], j = oj[q];
        C64 p = X(i, 0) * Y(0, j);
#pragma unroll
        for (int k = 1; k < 3; ++k) p = mad(X(i, k), Y(k, j), p);
        p = mk(p.re, -p.im);  // chain on with conj(p) - P_ji, conjugated back at the end
#pragma unroll
        for (int k = 0; k < 3; ++k) p = mad(-X(j, k), Y(k, i), p);
        r.o[q] = conj(p);
    }
    return r;
}

__device__ __forceinline__ M3 load_link64(const double2* __restrict__ U64, size_t V, int mu, int s) {
    M3 m;
#pragma unroll
    for (int e = 0; e < 9; ++e) {
        double2 v = U64[((size_t)mu * 9 + e) * V + s];
        m.a[e / 3][e % 3] = mk(v.x, v.y);
    }
    return m;
}

__device__ __forceinline__ void shift_coords(const Geom& g, int c[4], int mu, int dir) {
    const int N[4] = {g.N0, g.N1, g.N2, g.N3};
    int v = c[mu] + dir;
    bool crossed = (v == N[mu]) || (v < 0);
    c[mu] = crossed ? (dir > 0 ? 0 : N[mu] - 1) : v;
    if (crossed && ((mu == 2 && g.cs2) || (mu == 3 && g.cs3))) {
        c[1] += g.L1;
        if (c[1] >= g.N1) c[1] -= g.N1;
    }
}

__device__ __forceinline__ int native_of(const Geom& g, const int c[4]) {
    int lex = lex_index(g, c[0], c[1], c[2], c[3]);
    return native_index(g, lex, (c[0] + c[1] + c[2] + c[3]) & 1);
}

// Sites that carry the plaquettes of the gauge field: all of them, or, when
// the mirror half is the exact complex conjugate of the physical one, x1 < L1
// only (n1 = L1): the plaquettes of the mirror half are then the conjugates.
// Numbered like the native order, even sites first.
struct GaugeSet {
    Geom g;
    int n1;  // x1 extent of the set
    int n;   // sites
    int mirror;
};

inline GaugeSet gauge_set(const Geom& g, bool mirror) {
    GaugeSet q{g, mirror ? g.L1 : g.N1, 0, mirror ? 1 : 0};
    q.n = g.N0 * q.n1 * g.N2 * g.N3;
    return q;
}

// coordinates of site t of the set
__device__ __forceinline__ void set_coords(const GaugeSet& q, int t, int x[4]) {
    const int nh = q.n >> 1;
    const int p = t >= nh;
    int r = 2 * (t - p * nh);
    const int x3e = r % q.g.N3;
    r /= q.g.N3;
    x[2] = r % q.g.N2;
    r /= q.g.N2;
    x[1] = r % q.n1;
    x[0] = r / q.n1;
    x[3] = x3e + ((x[0] + x[1] + x[2] + x3e + p) & 1);
}

// number in the set of the site at coordinates c; flip: it is the mirror image
// of that site (conjugate the plaquette, change the sign of the U(1) sine)
__device__ __forceinline__ int set_index(const GaugeSet& q, const int c[4], bool& flip) {
    flip = c[1] >= q.n1;
    const int c1 = flip ? c[1] - q.n1 : c[1];
    const int lex = ((c[0] * q.n1 + c1) * q.g.N2 + c[2]) * q.g.N3 + c[3];
    return ((c[0] + c1 + c[2] + c[3]) & 1) * (q.n >> 1) + (lex >> 1);
}

__device__ __forceinline__ AH load_ah(const double* __restrict__ p, size_t stride) {
    AH r;
#pragma unroll
    for (int i = 0; i < 3; ++i) r.d[i] = p[i * stride];
#pragma unroll
    for (int k = 0; k < 3; ++k) r.o[k] = mk(p[(3 + 2 * k) * stride], p[(4 + 2 * k) * stride]);
    return r;
}

__device__ __forceinline__ void store_ah(double* __restrict__ p, size_t stride, const AH& a) {
#pragma unroll
    for (int i = 0; i < 3; ++i) p[i * stride] = a.d[i];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        p[(3 + 2 * k) * stride] = a.o[k].re;
        p[(4 + 2 * k) * stride] = a.o[k].im;
    }
}

// planes in the order of the field tensor: 01 02 03 12 13 23
__host__ __device__ __forceinline__ void plane_dirs(int plane, int& mu, int& nu) {
    mu = plane < 3 ? 0 : plane < 5 ? 1 : 2;
    nu = plane < 3 ? plane + 1 : plane < 5 ? plane - 1 : 3;
}
__host__ __device__ __forceinline__ int plane_of(int mu, int nu) { return mu == 0 ? nu - 1 : mu == 1 ? nu + 1 : 5; }

// Leaf buffers, in arrays of the lattice that a new gauge field makes stale: the
// hop links, the clover terms and their inverses, 234 V doubles side by side.
// First the leaves of the six planes, nine reals each (at most 6 x 4 x 9 = 216),
// then the sines of the U(1) plaquette angles, one per plane.
constexpr int LEAF_REALS = 216;
struct LeafBuf {
    double* b;
    double* sine;
    size_t n;  // sites of the set, at most V
    template <int LEAVES>
    __device__ __forceinline__ double* leaf(int plane, int l) const {
        return b + (size_t)(plane * LEAVES + l) * 9 * n;
    }
    __device__ __forceinline__ double* sines(int plane) const { return sine + (size_t)plane * n; }
};

// The leaves of plaquette (mu, nu) at site y of the set. With a = U(y,mu),
// b = U(y,nu), c = U(y+mu,nu), d = U(y+nu,mu) the four cyclic orders are
//   from y:            a c d^+ b^+ = (a c)(b d)^+
//   from y + mu:       c d^+ b^+ a = M N,    M = c d^+, N = b^+ a
//   from y + nu:       b^+ a c d^+ = N M
//   from y + mu + nu:  d^+ b^+ a c = (b d)^+ (a c)
// so each plaquette takes 4 products and 4 anti-Hermitian parts of products
// (792 FP64 instructions; 594 without the last, with (a M) b^+ as the first)
// where the four leaves of every site, taken one by one, take 12 products.
// LEAVES: 4, or 3 (without the last).
template <int LEAVES>
__device__ __forceinline__ void plaquette_leaves(const GaugeSet& q, const double2* __restrict__ U64,
                                                 const double* __restrict__ A64, int plane, int t, const LeafBuf& buf) {
    const Geom& g = q.g;
    const size_t V = (size_t)g.V;
    int mu, nu, x[4], c[4];
    plane_dirs(plane, mu, nu);
    set_coords(q, t, x);
    const int sx = native_of(g, x);
    c[0] = x[0]; c[1] = x[1]; c[2] = x[2]; c[3] = x[3];
    shift_coords(g, c, mu, 1);
    const int spm = native_of(g, c);
    c[0] = x[0]; c[1] = x[1]; c[2] = x[2]; c[3] = x[3];
    shift_coords(g, c, nu, 1);
    const int spn = native_of(g, c);
    const M3 a = load_link64(U64, V, mu, sx), b = load_link64(U64, V, nu, sx);
    const M3 cc = load_link64(U64, V, nu, spm), d = load_link64(U64, V, mu, spn);
    {
        const M3 M = mul_nd(cc, d), N = mul_dn(b, a);
        store_ah(buf.leaf<LEAVES>(plane, 1) + t, q.n, ah_mul<false, false>(M, N));
        store_ah(buf.leaf<LEAVES>(plane, 2) + t, q.n, ah_mul<false, false>(N, M));
        if (LEAVES == 3) store_ah(buf.leaf<LEAVES>(plane, 0) + t, q.n, ah_mul<false, true>(mul(a, M), b));
    }
    if (LEAVES == 4) {
        const M3 ac = mul(a, cc), bd = mul(b, d);
        store_ah(buf.leaf<LEAVES>(plane, 0) + t, q.n, ah_mul<false, true>(ac, bd));
        store_ah(buf.leaf<LEAVES>(plane, 3) + t, q.n, ah_mul<true, false>(bd, ac));
    }
    // U(1): z_munu(y) = exp(i (A(y,mu) + A(y+mu,nu) - A(y+nu,mu) - A(y,nu)))
    buf.sines(plane)[t] = sin(A64[(size_t)mu * V + sx] + A64[(size_t)nu * V + spm] - A64[(size_t)mu * V + spn] -
                              A64[(size_t)nu * V + sx]);
}

}  // namespace

// whether the mirror half of lat's gauge field is the exact conjugate of the
// physical half (built or flowed as such), so that x1 < L1 carries everything
inline bool mirror_exact(const qxd_lattice* lat) { return (lat->cstar_mask & 2u) && lat->mirror_built; }
inline LeafBuf leaf_buf(const qxd_lattice* lat, int n) {
    double* b = (double*)lat->W64;
    return LeafBuf{b, b + (size_t)LEAF_REALS * lat->g.V, (size_t)n};
}

}  // namespace qxd
