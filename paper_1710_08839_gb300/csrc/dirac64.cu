// FP64 stencils: D on the full lattice and its even-odd parts on one parity,
// with the work of a site split over several threads.
//
// GB300 issues two FP64 lanes per clock and SM, half a lane per scheduler: a
// warp's FP64 instruction occupies its scheduler for 64 clocks. A site's 1104
// FP64 instructions (8 hops x 84, 7 accumulations x 24, 264 for the two clover
// blocks) are what bounds these kernels, not its 1568 bytes, and a launch
// takes as long as the scheduler with the most of them. Hence the work of a
// site is split over 2 threads (by spin, 552 instructions each) and the warps
// are dealt out so that each of the 608 schedulers gets the same number; what
// is left over, up to 4864 sites, is split further, over 6 threads (spin and
// colour, 216 instructions: 8 hops x 18, 7 accumulations x 4, 44 for the clover
// rows; 8 lanes with two idle). Measured: 262144 sites 515 us (0.90 of the FP64
// issue rate; one thread per site 800 before the compound links and multiply-add
// chains), 41472 sites of D_hat's first half 91 us (four rounds of 552 and two of
// 216; one thread per site 120 us), D on 1024 lexicographic sites 12.3 us for the
// call (one thread per site, with the two layout conversions, 55 us). 128
// registers (4 blocks of 128 threads): 96 with spills took 3-5 % longer on 41472
// sites.
// In the chiral basis (1 -+ g_mu) psi is fixed by the half spinor (h_0, h_1):
// the thread of spin s forms h_s from two spin components of the neighbour
// (spin s, and spin 2 + s for mu = 0, 3 or 3 - s for mu = 1, 2), takes W h_s,
// and adds it to its upper spin s and, with a factor +-1 or +-i, to the lower
// spin of the same number. The threads of a pair exchange the lower sums
// before direction 1 and after direction 2, so every sum is taken in the order
// of dirac_hops and herm6_mul: the results are the same bits whatever the
// split.
#include "dirac64.cuh"

namespace qxd {

namespace {

// threads of a site and components of each: NC colours of spins s and 2 + s
template <int NC>
struct Split {
    static constexpr int LANES = NC == 3 ? 2 : 8;
    int s, c0;      // spin of the upper pair member, first colour
    double sgn;     // +1 for s = 0, -1 for s = 1
    bool live;      // NC = 1: lanes 6 and 7 of a site repeat the work of 4 and 5 and store nothing
    __device__ __forceinline__ Split() {
        const int l = threadIdx.x & (LANES - 1);
        s = l & 1;
        c0 = NC == 3 ? 0 : (l >> 1) < 2 ? (l >> 1) : 2;
        sgn = s ? -1.0 : 1.0;
        live = NC == 3 || l < 6;
    }
};

// Distribution of n sites over blocks of `warps` warps (see above): blocks
// [0, full) take 16 sites per warp in order, an equal number of warps for every
// scheduler; `rest` more blocks take the others, warp w of block b the chunk
// b + w * rest, so that they too spread over the SMs: 16 sites per warp, or 4
// (6 threads per site) if that takes less time.
constexpr int SCHEDULERS = 4 * NUM_SMS;
struct Deal {
    int n, full, rest, fine;
};
Deal deal(int n, int threads) {
    Deal d{n, 0, 0, 0};
    const int warps = threads / 32;
    d.full = (n / 16) / SCHEDULERS * SCHEDULERS / warps;
    const int left = n - d.full * warps * 16;
    // 6 threads per site: two rounds of 216 instructions at most, against one of
    // 552 (next to full blocks too: 41472 sites 97 -> 91 us)
    d.fine = left <= SCHEDULERS * 8;
    const int chunks = d.fine ? (left + 3) / 4 : (left + 15) / 16;
    d.rest = chunks <= NUM_SMS ? chunks : (chunks + SCHEDULERS - 1) / SCHEDULERS * (SCHEDULERS / warps);
    return d;
}
// site of this lane, -1 for a warp without sites; a lane beyond the last site
// repeats it (live = false)
template <int NC>
__device__ __forceinline__ int dealt_site(const Deal& d, bool& live) {
    constexpr int PER = 32 / Split<NC>::LANES;
    const int warps = blockDim.x >> 5, w = threadIdx.x >> 5, b = blockIdx.x;
    const int first = b < d.full ? (b * warps + w) * 16 : d.full * warps * 16 + (w * d.rest + (b - d.full)) * PER;
    if (first >= d.n) return -1;
    const int i = first + (threadIdx.x & 31) / Split<NC>::LANES;
    live = i < d.n;
    return live ? i : d.n - 1;
}

__device__ __forceinline__ C64 ld(const double2* __restrict__ p) {
    const double2 t = *p;
    return mk(t.x, t.y);
}

// One hop (1 -+ g_mu) W psi added to the sums: au the upper spin s, al the
// lower spin that direction MU feeds from this thread. n: where the
// neighbour's components start; link: component (0, 0) of W at the link's site.
template <int NC, int MU, int DIR, bool FIRST = false>
__device__ __forceinline__ void hop64(const double2* __restrict__ n, size_t kst, const double2* __restrict__ link,
                                      size_t V, const Split<NC>& sp, C64 au[NC], C64 al[NC]) {
    constexpr double D = DIR;
    const int lspin = (MU == 0 || MU == 3) ? 2 + sp.s : 3 - sp.s;
    C64 h[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const C64 a = ld(n + (3 * sp.s + c) * kst), b = ld(n + (3 * lspin + c) * kst);
        if (MU == 0) h[c] = DIR > 0 ? a + b : a - b;
        else if (MU == 1) h[c] = DIR > 0 ? a + times_i(b) : a - times_i(b);
        else if (MU == 2) h[c] = rmad(D * sp.sgn, b, a);
        else h[c] = mk(fma(-D * sp.sgn, b.im, a.re), fma(D * sp.sgn, b.re, a.im));
    }
#pragma unroll
    for (int k = 0; k < NC; ++k) {
        const int c = sp.c0 + k;
        C64 g;
        if (DIR > 0)  // row c of W
            g = mad(ld(link + (3 * c + 2) * V), h[2], mad(ld(link + (3 * c + 1) * V), h[1], ld(link + (3 * c) * V) * h[0]));
        else  // row c of W^+
            g = cmad(ld(link + (6 + c) * V), h[2], cmad(ld(link + (3 + c) * V), h[1], cmul(ld(link + c * V), h[0])));
        if (FIRST) {
            au[k] = al[k] = g;
            continue;
        }
        au[k] = au[k] + g;
        if (MU == 0) al[k] = DIR > 0 ? al[k] + g : al[k] - g;
        else if (MU == 1) al[k] = DIR > 0 ? al[k] + times_mi(g) : al[k] + times_i(g);
        else if (MU == 2) al[k] = rmad(D * sp.sgn, g, al[k]);
        else al[k] = mk(fma(D * sp.sgn, g.im, al[k].re), fma(-D * sp.sgn, g.re, al[k].im));
    }
}

template <int NC>
__device__ __forceinline__ void swap_pair(C64 a[NC]) {
#pragma unroll
    for (int k = 0; k < NC; ++k)
        a[k] = mk(__shfl_xor_sync(0xffffffffu, a[k].re, 1), __shfl_xor_sync(0xffffffffu, a[k].im, 1));
}

template <int NC, int MU, bool FIRST = false>
__device__ __forceinline__ void dir64(const Geom& g, const double2* __restrict__ W, const SpRef<double>& in,
                                      const Split<NC>& sp, int x0, int x1, int x2, int x3, int s, int po, C64 au[NC],
                                      C64 al[NC]) {
    const size_t V = g.V;
    const double2* Wm = W + (size_t)MU * 9 * V;
    const int lf = neighbour_lex<MU, +1>(g, x0, x1, x2, x3);
    hop64<NC, MU, +1, FIRST>(in.p + in.at(lf, native_index(g, lf, po)), in.stride, Wm + s, V, sp, au, al);
    const int lb = neighbour_lex<MU, -1>(g, x0, x1, x2, x3);
    const int sb = native_index(g, lb, po);
    hop64<NC, MU, -1>(in.p + in.at(lb, sb), in.stride, Wm + sb, V, sp, au, al);
}

// H psi at site x (native index s, neighbours of parity po): au spin s, al spin 2 + s
template <int NC>
__device__ __forceinline__ void hops64(const Geom& g, const double2* __restrict__ W, const SpRef<double>& in,
                                       const Split<NC>& sp, int x0, int x1, int x2, int x3, int s, int po, C64 au[NC],
                                       C64 al[NC]) {
    dir64<NC, 0, true>(g, W, in, sp, x0, x1, x2, x3, s, po, au, al);
    swap_pair<NC>(al);
    dir64<NC, 1>(g, W, in, sp, x0, x1, x2, x3, s, po, au, al);
    dir64<NC, 2>(g, W, in, sp, x0, x1, x2, x3, s, po, au, al);
    swap_pair<NC>(al);
    dir64<NC, 3>(g, W, in, sp, x0, x1, x2, x3, s, po, au, al);
}

// y += (or =) row r of a packed Hermitian 6x6 block (C its first real at the
// site) times the six components v(0..5), columns in ascending order and the
// diagonal last (the order of herm6_mul)
template <bool ADD, typename F>
__device__ __forceinline__ void herm6_row(const double* __restrict__ C, size_t V, int r, F v, C64& y) {
#pragma unroll
    for (int t = 0; t < 5; ++t) {
        const bool below = t < r;  // column j < r: L(r, j), else conj L(j, r)
        const int j = below ? t : t + 1;
        const int i = below ? r : j, l = below ? j : r;
        const double* e = C + (size_t)(6 + i * (i - 1) + 2 * l) * V;
        const double im = e[V];
        const C64 m = mk(e[0], below ? im : -im);
        y = !ADD && t == 0 ? m * v(j) : mad(m, v(j), y);
    }
    y = rmad(C[(size_t)r * V], v(r), y);
}

// acc (+)= M v at site s, v a spinor in memory: element k at v[k * kst]
template <int NC, bool ADD>
__device__ __forceinline__ void clover64(const double* __restrict__ C, size_t V, int s, const double2* __restrict__ v,
                                         size_t kst, const Split<NC>& sp, C64 au[NC], C64 al[NC]) {
#pragma unroll
    for (int blk = 0; blk < 2; ++blk)
#pragma unroll
        for (int k = 0; k < NC; ++k)
            herm6_row<ADD>(C + (size_t)36 * blk * V + s, V, 3 * sp.s + sp.c0 + k,
                           [&](int j) { return ld(v + (6 * blk + j) * kst); }, blk ? al[k] : au[k]);
}

// acc = M v, v spread over the threads of the site as acc is
template <int NC>
__device__ __forceinline__ void clover64_reg(const double* __restrict__ C, size_t V, int s, const Split<NC>& sp,
                                             const C64 vu[NC], const C64 vl[NC], C64 au[NC], C64 al[NC]) {
#pragma unroll
    for (int blk = 0; blk < 2; ++blk) {
        const C64* own = blk ? vl : vu;
        C64* y = blk ? al : au;
        if constexpr (NC == 3) {
            C64 w[6];  // the block's components in order
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                const C64 o = mk(__shfl_xor_sync(0xffffffffu, own[c].re, 1), __shfl_xor_sync(0xffffffffu, own[c].im, 1));
                w[c] = sp.s ? o : own[c];
                w[3 + c] = sp.s ? own[c] : o;
            }
#pragma unroll
            for (int k = 0; k < 3; ++k)
                herm6_row<false>(C + (size_t)36 * blk * V + s, V, 3 * sp.s + k, [&](int j) {
                    // j is t or t + 1 of an unrolled loop, chosen by the thread's spin
                    C64 x = w[0];
#pragma unroll
                    for (int q = 1; q < 6; ++q)
                        if (q == j) x = w[q];
                    return x;
                }, y[k]);
        } else {
            const int site = threadIdx.x & 24;  // first lane of the site
            C64 r = mk(0.0, 0.0);
            herm6_row<false>(C + (size_t)36 * blk * V + s, V, 3 * sp.s + sp.c0, [&](int j) {
                const int lane = site + (j >= 3 ? 1 + 2 * (j - 3) : 2 * j);
                return mk(__shfl_sync(0xffffffffu, own[0].re, lane), __shfl_sync(0xffffffffu, own[0].im, lane));
            }, r);
            y[0] = r;
        }
    }
}

template <int NC>
__device__ __forceinline__ void load_split(const SpRef<double>& f, size_t at, const Split<NC>& sp, C64 u[NC], C64 l[NC]) {
#pragma unroll
    for (int k = 0; k < NC; ++k) {
        u[k] = ld(f.p + at + (size_t)(3 * sp.s + sp.c0 + k) * f.stride);
        l[k] = ld(f.p + at + (size_t)(6 + 3 * sp.s + sp.c0 + k) * f.stride);
    }
}

template <int NC>
__device__ __forceinline__ void store_split(const SpRefOut<double>& f, size_t at, const Split<NC>& sp, const C64 u[NC],
                                            const C64 l[NC]) {
#pragma unroll
    for (int k = 0; k < NC; ++k) {
        f.p[at + (size_t)(3 * sp.s + sp.c0 + k) * f.stride] = make_double2(u[k].re, u[k].im);
        f.p[at + (size_t)(6 + 3 * sp.s + sp.c0 + k) * f.stride] = make_double2(l[k].re, l[k].im);
    }
}

template <int NC>
__device__ __forceinline__ void zero_split(const SpRefOut<double>& f, size_t at, const Split<NC>& sp) {
    C64 z[NC];
#pragma unroll
    for (int k = 0; k < NC; ++k) z[k] = mk(0.0, 0.0);
    store_split<NC>(f, at, sp, z, z);
}

// out = D in on the x0 planes [x0b, x0b + nx0)
template <int NC>
__device__ __forceinline__ void dirac64_site(const Geom& g, const Fields<double>& f, const SpRef<double>& in,
                                             const SpRefOut<double>& out, int x0b, int nx0, const Deal& d) {
    const Split<NC> sp;
    bool live;
    const int tau = dealt_site<NC>(d, live);
    if (tau < 0) return;
    int x0, x1, x2, x3;
    sweep_coords_slab(g, x0b, nx0, tau, x0, x1, x2, x3);
    const int p = (x0 + x1 + x2 + x3) & 1;
    const int lex = lex_index(g, x0, x1, x2, x3);
    const int s = native_index(g, lex, p);
    C64 au[NC], al[NC];
    hops64<NC>(g, f.U, in, sp, x0, x1, x2, x3, s, 1 - p, au, al);
    clover64<NC, true>(f.C, g.V, s, in.p + in.at(lex, s), in.stride, sp, au, al);
    if (live && sp.live) store_split<NC>(out, out.at(lex, s), sp, au, al);
}
__global__ void __launch_bounds__(DW_THREADS, 4)
    k_dirac64(Geom g, Fields<double> f, SpRef<double> in, SpRefOut<double> out, int x0b, int nx0, Deal d) {
    if (d.fine && blockIdx.x >= d.full) dirac64_site<1>(g, f, in, out, x0b, nx0, d);
    else dirac64_site<3>(g, f, in, out, x0b, nx0, d);
}

// the even-odd parts (modes of eo.cuh) on the sites of parity p (the inverse
// clover blocks of the odd sites, V/2 of each real)
template <int NC, int MODE>
__device__ __forceinline__ void dslash64_site(const Geom& g, int p, const Fields<double>& f, const SpRef<double>& in,
                                              const SpRef<double>& aux, const SpRefOut<double>& out,
                                              const double* __restrict__ Cl, const Deal& d) {
    const Split<NC> sp;
    bool live;
    const int tau = dealt_site<NC>(d, live);
    if (tau < 0) return;
    int x0, x1, x2, x3;
    sweep_coords_parity(g, p, tau, x0, x1, x2, x3);
    const int lex = lex_index(g, x0, x1, x2, x3);
    const int s = native_index(g, lex, p);
    C64 hu[NC], hl[NC], u[NC], l[NC];
    hops64<NC>(g, f.U, in, sp, x0, x1, x2, x3, s, 1 - p, hu, hl);
    if (MODE == EO_INV_HOP) {
        clover64_reg<NC>(Cl, g.Vh, s - g.Vh, sp, hu, hl, u, l);
    } else if (MODE == EO_CLOVER_AUX_MHOP || MODE == EO_G5_CLOVER_AUX_MHOP) {
#pragma unroll
        for (int k = 0; k < NC; ++k) {
            u[k] = -hu[k];
            l[k] = -hl[k];
        }
        clover64<NC, true>(Cl, g.V, s, aux.p + aux.at(lex, s), aux.stride, sp, u, l);
        if (MODE == EO_G5_CLOVER_AUX_MHOP) {  // gamma5 = diag(1, 1, -1, -1)
#pragma unroll
            for (int k = 0; k < NC; ++k) l[k] = -l[k];
        }
    } else {  // AUX_MHOP, INV_AUX_MHOP
        load_split<NC>(aux, aux.at(lex, s), sp, u, l);
#pragma unroll
        for (int k = 0; k < NC; ++k) {
            u[k] = u[k] - hu[k];
            l[k] = l[k] - hl[k];
        }
        if (MODE == EO_INV_AUX_MHOP) {
            clover64_reg<NC>(Cl, g.Vh, s - g.Vh, sp, u, l, hu, hl);
#pragma unroll
            for (int k = 0; k < NC; ++k) {
                u[k] = hu[k];
                l[k] = hl[k];
            }
        }
    }
    if (!live || !sp.live) return;
    store_split<NC>(out, out.at(lex, s), sp, u, l);
    if (out.zero_other) zero_split<NC>(out, out.at(lex ^ 1, p ? s - g.Vh : s + g.Vh), sp);
}
template <int MODE>
__global__ void __launch_bounds__(DW_THREADS, 4)
    k_dslash64(Geom g, int p, Fields<double> f, SpRef<double> in, SpRef<double> aux, SpRefOut<double> out,
               const double* __restrict__ Cl, Deal d) {
    if (d.fine && blockIdx.x >= d.full) dslash64_site<1, MODE>(g, p, f, in, aux, out, Cl, d);
    else dslash64_site<3, MODE>(g, p, f, in, aux, out, Cl, d);
}

}  // namespace

int launch_dirac64(qxd_lattice* lat, const SpRefOut<double>& out, const SpRef<double>& in, int threads, int rows,
                   int x0b, int nx0, cudaStream_t st) {
    Geom g = lat->g;
    g.R = rows;
    const Fields<double> f{nullptr, lat->W64, lat->C64};
    const Deal d = deal(nx0 * g.N1 * g.N2 * g.N3, threads);
    k_dirac64<<<d.full + d.rest, threads, 0, st>>>(g, f, in, out, x0b, nx0, d);
    QXD_LAUNCHED("k_dirac64");
    return QXD_OK;
}

int launch_eo64(qxd_lattice* lat, int mode, int p, const SpRef<double>& in, const SpRef<double>& aux,
                const SpRefOut<double>& out, cudaStream_t st) {
    const Geom& g = lat->g;
    const double* Cl = eo_inverse(mode) ? lat->Cinv64 : lat->C64;
    const Fields<double> f{nullptr, lat->W64, nullptr};
    const Deal d = deal(g.Vh, DW_THREADS);
    const int grid = d.full + d.rest;
    switch (mode) {
        case EO_INV_HOP: k_dslash64<EO_INV_HOP><<<grid, DW_THREADS, 0, st>>>(g, p, f, in, aux, out, Cl, d); break;
        case EO_CLOVER_AUX_MHOP: k_dslash64<EO_CLOVER_AUX_MHOP><<<grid, DW_THREADS, 0, st>>>(g, p, f, in, aux, out, Cl, d); break;
        case EO_AUX_MHOP: k_dslash64<EO_AUX_MHOP><<<grid, DW_THREADS, 0, st>>>(g, p, f, in, aux, out, Cl, d); break;
        case EO_G5_CLOVER_AUX_MHOP: k_dslash64<EO_G5_CLOVER_AUX_MHOP><<<grid, DW_THREADS, 0, st>>>(g, p, f, in, aux, out, Cl, d); break;
        default: k_dslash64<EO_INV_AUX_MHOP><<<grid, DW_THREADS, 0, st>>>(g, p, f, in, aux, out, Cl, d); break;
    }
    QXD_LAUNCHED("k_dslash64");
    return QXD_OK;
}

}  // namespace qxd
