// Schwarz alternating procedure (SAP) preconditioner on 4^4 blocks.
//
// The paper names the SAP-preconditioned GCR solver (Sec. 1-2) without
// giving it; this is the standard multiplicative Schwarz method. The lattice
// is cut into 4^4 blocks, coloured by the parity of their block coordinates
// so that blocks of one colour never touch. One cycle visits the blocks of
// colour 0, then of colour 1; for each block B (all blocks of a colour in
// parallel, one thread block each):
//   r_B   = eta_B - (D psi)_B                 (D over the whole lattice)
//   solve D_B delta = r_B approximately, D_B = D restricted to B with
//         the hops leaving B dropped, by nmr minimal-residual steps on the
//         even-odd form D_hat_B = M_ee - H_eo M_oo^-1 H_oe of the block
//   psi_B += delta
// Starting from psi = 0, ncy cycles give psi = SAP(eta).
// FP32, single lattice (k_sap_split): two threads per site pair, the block's
// interior compound links W' = -1/2 z^qhat U (all three rows) and two block
// fields in shared memory, the clover rows of each thread in tensor memory,
// both from a block-by-block copy of the operator (or from the native fields
// where there is none). The residual of a block is not recomputed from eta - D psi: the even-odd block solve
// leaves the block residual r_B - D_B delta equal to the MR residual rho on
// the even sites and to zero on the odd sites (delta_o = M_oo^-1 (r_o - H_oe
// delta_e) solves the odd rows exactly), and between two visits of a block
// psi changes only on the blocks of the other colour, by their last
// corrections delta. So a visit starts from
//   r_B = rho_B (even sites), 0 (odd sites)  -  D_cross delta,
// where D_cross keeps the hops of D that cross the faces of B (all other
// terms of D delta vanish on B), and r_B = eta_B on the first visit. The
// kernel keeps rho on the even sites and delta of every site in two work
// fields. FP32, batched (k_sap_block_batch): the same block solve over the
// blocks of several lattices in one launch, each job with its own work
// fields. FP64 (k_sap_block): one thread per site pair, the block fields in
// shared memory, links and clover blocks from the global fields.
#include <algorithm>
#include <vector>

#include "dirac_common.cuh"
#include "solver.cuh"

namespace qxd {

namespace {

using C64 = cplx<double>;

constexpr int SAP_BS = 4;          // block extent in every direction
constexpr int SAP_HALF = 128;      // sites of one parity per block
constexpr int SAP_THREADS = 128;   // one thread per (even, odd) site pair

// shared-memory half-spinor field of one block: double[24][128], conflict-free
struct SmemField {
    double* a;
    __device__ __forceinline__ void load(int slot, C64 v[12]) const {
#pragma unroll
        for (int i = 0; i < 12; ++i) v[i] = mk(a[(2 * i) * SAP_HALF + slot], a[(2 * i + 1) * SAP_HALF + slot]);
    }
    __device__ __forceinline__ void store(int slot, const C64 v[12]) const {
#pragma unroll
        for (int i = 0; i < 12; ++i) {
            a[(2 * i) * SAP_HALF + slot] = v[i].re;
            a[(2 * i + 1) * SAP_HALF + slot] = v[i].im;
        }
    }
};

struct Site {
    int l[4];   // coordinates inside the block
    int x[4];   // global coordinates
    int s;      // native index
    int lidx;   // local lexicographic index (0..255)
};

__device__ __forceinline__ Site make_site(const Geom& g, const int org[4], int lidx) {
    Site t;
    t.lidx = lidx;
    t.l[3] = lidx & 3;
    t.l[2] = (lidx >> 2) & 3;
    t.l[1] = (lidx >> 4) & 3;
    t.l[0] = (lidx >> 6) & 3;
#pragma unroll
    for (int m = 0; m < 4; ++m) t.x[m] = org[m] + t.l[m];
    const int p = (t.x[0] + t.x[1] + t.x[2] + t.x[3]) & 1;
    t.s = native_index(g, lex_index(g, t.x[0], t.x[1], t.x[2], t.x[3]), p);
    return t;
}

// Block number bidx of the blocks of this colour: blocks (b0, b1, b2, b3e) and
// (.., b3e + 1), b3e even, are one of each colour. Sets its origin, returns its
// number among all blocks (lexicographic in block coordinates).
__device__ __forceinline__ int block_origin(const SapGeom& sg, int bidx, int colour, int org[4]) {
    const int bi2 = 2 * bidx;
    const int b3e = bi2 % sg.nb3;
    int rest = bi2 / sg.nb3;
    const int b2 = rest % sg.nb2;
    rest /= sg.nb2;
    const int b1 = rest % sg.nb1;
    const int b0 = rest / sg.nb1;
    const int b3 = b3e + ((b0 + b1 + b2 + b3e + colour) & 1);
    org[0] = SAP_BS * b0;
    org[1] = SAP_BS * b1;
    org[2] = SAP_BS * b2;
    org[3] = SAP_BS * b3;
    return bi2 - b3e + b3;
}

// asynchronous copy of 16 bytes from global to shared memory (past L1), and the
// wait for this thread's copies
__device__ __forceinline__ void copy_async16(void* smem, const void* gmem) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(gmem) : "memory");
}
__device__ __forceinline__ void copy_async_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// native index of the in-block site one step back in direction MU
template <int MU>
__device__ __forceinline__ int back_native(const Geom& g, const Site& t) {
    int y[4] = {t.x[0], t.x[1], t.x[2], t.x[3]};
    y[MU] -= 1;
    return native_index(g, lex_index(g, y[0], y[1], y[2], y[3]), (y[0] + y[1] + y[2] + y[3]) & 1);
}

// hops of direction MU that stay inside the block (Dirichlet block boundary);
// the neighbour spinor comes from shared memory (field of the other parity).
// The links are compound (the charge and the factor -1/2 are in).
template <int MU>
__device__ __forceinline__ void block_dir(const Geom& g, const Fields<double>& f, const SmemField& src, const Site& t,
                                          C64 acc[12]) {
    constexpr int stride = MU == 0 ? 64 : MU == 1 ? 16 : MU == 2 ? 4 : 1;
    C64 v[12], h0[3], h1[3], g0[3], g1[3], u[3][3];
    if (t.l[MU] < SAP_BS - 1) {
        src.load((t.lidx + stride) >> 1, v);
        project<double, MU, +1>(v, h0, h1);
        load_link(f.U, g.V, MU, t.s, u);
        su3_mul(u, h0, g0);
        su3_mul(u, h1, g1);
        accumulate<double, MU, +1>(acc, g0, g1);
    }
    if (t.l[MU] > 0) {
        src.load((t.lidx - stride) >> 1, v);
        project<double, MU, -1>(v, h0, h1);
        load_link(f.U, g.V, MU, back_native<MU>(g, t), u);
        su3_dag_mul(u, h0, g0);
        su3_dag_mul(u, h1, g1);
        accumulate<double, MU, -1>(acc, g0, g1);
    }
}

__device__ __forceinline__ void block_hops(const Geom& g, const Fields<double>& f, const SmemField src, const Site& t,
                                           C64 acc[12]) {
#pragma unroll
    for (int i = 0; i < 12; ++i) acc[i] = mk(0.0, 0.0);
    block_dir<0>(g, f, src, t, acc);
    block_dir<1>(g, f, src, t, acc);
    block_dir<2>(g, f, src, t, acc);
    block_dir<3>(g, f, src, t, acc);
}

// r = eta - (D psi)(x), D over the whole lattice, at one site; out of line,
// for the one-thread-per-pair kernel, which calls it twice
__device__ __noinline__ void residual_at(const Geom& g, const Fields<double>& f, const double2* eta,
                                         const Site& t, bool psi_zero, C64 r[12]) {
    load_spinor(eta, g.V, t.s, r);
    if (psi_zero) return;
    const int po = 1 - ((t.x[0] + t.x[1] + t.x[2] + t.x[3]) & 1);
    C64 acc[12], v[12];
    dirac_hops<double, false>(g, f, f.psi, g.V, 0, 0.0, t.x[0], t.x[1], t.x[2], t.x[3], t.s, po, acc);
    load_spinor(f.psi, g.V, t.s, v);
    clover_mul<false, true>(f.C, g.V, t.s, v, acc);
#pragma unroll
    for (int i = 0; i < 12; ++i) r[i] = r[i] - acc[i];
}

// sum over the NT threads of the block, result in every thread. TAIL_SYNC
// guards red against the next call; a caller that passes a barrier before it
// reuses red may drop it.
template <typename R, int NT = SAP_THREADS, bool TAIL_SYNC = true>
__device__ __forceinline__ void block_sum3(R a, R b, R c, R* red, R out[3]) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        a += __shfl_xor_sync(0xffffffffu, a, o);
        b += __shfl_xor_sync(0xffffffffu, b, o);
        c += __shfl_xor_sync(0xffffffffu, c, o);
    }
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (lane == 0) {
        red[3 * warp] = a;
        red[3 * warp + 1] = b;
        red[3 * warp + 2] = c;
    }
    __syncthreads();
    out[0] = out[1] = out[2] = R(0);
#pragma unroll
    for (int w = 0; w < NT / 32; ++w) {
        out[0] += red[3 * w];
        out[1] += red[3 * w + 1];
        out[2] += red[3 * w + 2];
    }
    if (TAIL_SYNC) __syncthreads();
}

// Each thread owns one even and one odd site of the block: the local pair
// (2t, 2t + 1). Phases in order (each block-hop phase is one call of
// block_hops from a single call site, which keeps the code small):
//   residual on both sites; t_o = M_oo^-1 r_o
//   step 0:            rho = r_e - H_eo t_o                       (even)
//   step 2k+1, 2k+2:   t_o = M_oo^-1 H_oe rho (odd); w = M_ee rho - H_eo t_o,
//                      omega = <w,rho>/<w,w>, delta_e += omega rho,
//                      rho -= omega w (even)             for k < nmr
//   last step:         delta_o = M_oo^-1 (r_o - H_oe delta_e)     (odd)
__device__ __forceinline__ void sap_block_body(const Geom& g, const SapGeom& sg, int bidx, int colour, int psi_zero,
                                               const Fields<double>& f, const double* __restrict__ Cinv,
                                               const double2* __restrict__ eta, int nmr) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    double* sm = reinterpret_cast<double*>(smem_raw);
    const SmemField s_ro{sm};                   // r on the odd sites
    const SmemField s_rho{sm + 24 * SAP_HALF};  // MR residual (even)
    const SmemField s_t{sm + 48 * SAP_HALF};    // odd temporary / delta_e at the end
    double* red = sm + 72 * SAP_HALF;           // 3 * warps reduction slots

    int org[4];
    block_origin(sg, bidx, colour, org);
    const int t = threadIdx.x;
    const int base = 2 * t;
    const int par0 = ((base >> 6) + ((base >> 4) & 3) + ((base >> 2) & 3) + (base & 3)) & 1;
    const Site se = make_site(g, org, base + par0);
    const Site so = make_site(g, org, base + 1 - par0);

    // residual r = eta - D psi on both sites (one call site)
    C64 re[12], v[12], w[12], acc[12];
#pragma unroll 1
    for (int k = 0; k < 2; ++k) {
        residual_at(g, f, eta, k ? so : se, psi_zero, k ? v : re);
    }
    s_ro.store(t, v);
    clover_mul(Cinv, g.Vh, so.s - g.Vh, v, w);  // t_o = M_oo^-1 r_o
    s_t.store(t, w);
    __syncthreads();

    C64 rho[12], de[12];
#pragma unroll
    for (int i = 0; i < 12; ++i) de[i] = mk(0.0, 0.0);
    const int nsteps = 2 * nmr + 2;
#pragma unroll 1
    for (int step = 0; step < nsteps; ++step) {
        const bool odd = (step & 1) != 0;   // steps 1, 3, ..., 2 nmr + 1 work on the odd sites
        const bool last = step == nsteps - 1;
        // odd steps read rho (or delta_e on the last step), even steps read t_o
        block_hops(g, f, odd ? (last ? s_t : s_rho) : s_t, odd ? so : se, acc);
        // acc = H psi on the sites of this step's parity
        if (step == 0) {
#pragma unroll
            for (int i = 0; i < 12; ++i) rho[i] = re[i] - acc[i];
            s_rho.store(t, rho);
        } else if (last) {
            s_ro.load(t, v);
#pragma unroll
            for (int i = 0; i < 12; ++i) v[i] = v[i] - acc[i];
            clover_mul(Cinv, g.Vh, so.s - g.Vh, v, w);  // delta_o
        } else if (odd) {
            clover_mul(Cinv, g.Vh, so.s - g.Vh, acc, w);
            s_t.store(t, w);
        } else {
#pragma unroll
            for (int i = 0; i < 12; ++i) w[i] = -acc[i];
            clover_mul<false, true>(f.C, g.V, se.s, rho, w);
            double a_re = 0, a_im = 0, b = 0;
#pragma unroll
            for (int i = 0; i < 12; ++i) {
                a_re += w[i].re * rho[i].re + w[i].im * rho[i].im;
                a_im += w[i].re * rho[i].im - w[i].im * rho[i].re;
                b += w[i].re * w[i].re + w[i].im * w[i].im;
            }
            double sums[3];
            block_sum3(a_re, a_im, b, red, sums);
            if (sums[2] > 0.0) {  // else rho = 0 on the whole block: nothing to add
                const C64 om = mk(sums[0] / sums[2], sums[1] / sums[2]);
#pragma unroll
                for (int i = 0; i < 12; ++i) {
                    de[i] = mad(om, rho[i], de[i]);
                    rho[i] = mad(-om, w[i], rho[i]);
                }
            }
            if (step == nsteps - 2) s_t.store(t, de);  // delta_e for the last step
            else s_rho.store(t, rho);
        }
        __syncthreads();
    }
    // psi_B += delta (w holds delta_o)
    double2* psi = const_cast<double2*>(f.psi);
    if (psi_zero) {
        store_spinor(psi, g.V, se.s, de);
        store_spinor(psi, g.V, so.s, w);
    } else {
        load_spinor(f.psi, g.V, se.s, v);
#pragma unroll
        for (int i = 0; i < 12; ++i) v[i] = v[i] + de[i];
        store_spinor(psi, g.V, se.s, v);
        load_spinor(f.psi, g.V, so.s, v);
#pragma unroll
        for (int i = 0; i < 12; ++i) v[i] = v[i] + w[i];
        store_spinor(psi, g.V, so.s, v);
    }
}

__global__ void __launch_bounds__(SAP_THREADS, 2) k_sap_block(Geom g, SapGeom sg, int colour, int psi_zero,
                                                              Fields<double> f, const double* __restrict__ Cinv,
                                                              const double2* __restrict__ eta, int nmr) {
    sap_block_body(g, sg, blockIdx.x, colour, psi_zero, f, Cinv, eta, nmr);
}

// ---------------------------------------------------------------------------
// FP32 block solve with two threads per site pair (spin split)
//
// Thread 2t + sg owns the spin-sg half of every block spinor of local pair t:
// components 3 sg + c (upper chirality) and 6 + 3 sg + c (lower chirality,
// spin 2 + sg), c = 0..2. In the chiral basis (1 -+ g_mu) psi is fixed by a
// half spinor (h_0, h_1): the upper spins are U h and the lower ones a fixed
// 2x2 spin matrix times U h. Thread sg forms h_sg from two spin components of
// the neighbour, multiplies it by the link, and adds U h_sg to its own upper
// spin and to one lower spin: its own (mu = 0, 3) or its partner's
// (mu = 1, 2). The partner's share is exchanged once per hop set with a warp
// shuffle. The clover term acts within a chirality, so each thread computes
// its three rows of both 6x6 blocks after one shuffle of the partner's half.
// The block's compound links W' = -1/2 z^qhat U are staged once per launch
// with all three rows, so a hop is a projection, one 3x3 complex product and
// the accumulation: no third-row rebuild, no U(1) phase, no factor -1/2.
//
// What belongs to the operator is laid out block by block when the operator is
// built (k_sap_plan): the compound interior links as they go into shared
// memory, and the clover blocks that the block solve uses, M_oo^-1 and M_ee, as
// float4 [2][18][128] with the block's pairs in order. In the native layout a
// block's sites come in runs of 32 bytes whose other halves belong to blocks of
// the other colour: half of every DRAM access and three quarters of every
// cache line were of no use (64x64x32x32 sites, 5 cycles, 5 MR steps: 16.1 ms
// without, 14.7 with it; DRAM bytes of a launch on 48x48x24x24 1.15 -> 0.82 GB).
// The bodies of the block hops and of the crossing hops start with
// __syncwarp(): left to itself the compiler lets the lanes that skipped a body
// run ahead through the next ones, and warps took them twice (28 % more
// shared-memory loads; 14.3 -> 13.1 ms).
// ---------------------------------------------------------------------------
constexpr int SPLIT_THREADS = 256;
constexpr unsigned FULL_MASK = 0xffffffffu;

// Shared-memory block fields of the split kernel: complex numbers as float2,
// colour c of spin s of pair slot t at SPIN_STRIDE s + 128 c + t. The stride is
// 3 x 128 + 8: the two threads of a pair read the same slot in spins of
// opposite parity, and the 8 puts the eight pairs of a half warp on disjoint
// halves of the 32 banks. Addresses are linear in the slot, so the hops of a
// thread are its own base plus constants (a rotation by 8 within rows of 128
// did the same for the banks at 14 % of all instructions for addresses).
constexpr int SPIN_STRIDE = 3 * SAP_HALF + 8;
constexpr int FIELD_F2 = 4 * SPIN_STRIDE;  // float2 of a block field
__device__ __forceinline__ void ld3(const float2* p, cplx<float> v[3]) {
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const float2 x = p[c * SAP_HALF];
        v[c] = mk(x.x, x.y);
    }
}
__device__ __forceinline__ void ld_spin(const float2* a, int spin, int slot, cplx<float> v[3]) {
    ld3(a + SPIN_STRIDE * spin + slot, v);
}
__device__ __forceinline__ void st_spin(float2* a, int spin, int slot, const cplx<float> v[3]) {
    float2* p = a + SPIN_STRIDE * spin + slot;
#pragma unroll
    for (int c = 0; c < 3; ++c) p[c * SAP_HALF] = make_float2(v[c].re, v[c].im);
}
// own half: v[0..2] spin sg, v[3..5] spin 2 + sg
__device__ __forceinline__ void ld_half(const float2* a, int sg, int slot, cplx<float> v[6]) {
    ld_spin(a, sg, slot, v);
    ld_spin(a, 2 + sg, slot, v + 3);
}
__device__ __forceinline__ void st_half(float2* a, int sg, int slot, const cplx<float> v[6]) {
    st_spin(a, sg, slot, v);
    st_spin(a, 2 + sg, slot, v + 3);
}
__device__ __forceinline__ void ld_full(const float2* a, int slot, cplx<float> v[12]) {
#pragma unroll
    for (int sp = 0; sp < 4; ++sp) ld_spin(a, sp, slot, v + 3 * sp);
}
__device__ __forceinline__ void st_full(float2* a, int slot, const cplx<float> v[12]) {
#pragma unroll
    for (int sp = 0; sp < 4; ++sp) st_spin(a, sp, slot, v + 3 * sp);
}

// Block links of the split kernel in shared memory. The block operator uses
// only the links that stay inside the block, those of sites with l[mu] < 3,
// 192 per direction. Entry of the site of parity p and local index lidx in
// direction mu (stride S = 64, 16, 4, 1 in lidx):
//   mu = 0, 1, 2: p * 96 + compact pair slot, with the pair slot lidx >> 1
//                 written as hi * 2S + l * S/2 + lo (l = l[mu]) and compacted to
//                 hi * 3S/2 + l * S/2 + lo, so that consecutive pairs read
//                 consecutive entries;
//   mu = 3:       3 (lidx >> 2) + (lidx & 3).
constexpr int SPLIT_LINKS = 192;  // interior links per direction

template <int MU>
__device__ __forceinline__ int link_entry(int p, int lidx) {
    if constexpr (MU == 3) {
        return 3 * (lidx >> 2) + (lidx & 3);
    } else {
        constexpr int H = MU == 0 ? 32 : MU == 1 ? 8 : 2;  // S / 2
        const int slot = lidx >> 1;
        return p * (SPLIT_LINKS / 2) + (slot / (4 * H)) * (3 * H) + ((slot / H) & 3) * H + (slot & (H - 1));
    }
}

// Compound block links of the split kernel, W'(x,mu) = -1/2 z(x,mu)^qhat
// U(x,mu), all three rows, staged once per launch so that the hops need
// neither the third-row reconstruction nor the U(1) phase nor the factor
// -1/2. Entry e of direction mu: float4 W4[mu][k][e], k = 0..3, holds the
// complex entries (00, 01), (02, 10), (11, 12), (20, 21); float2 W2[mu][e]
// holds (22).
struct SplitLinks {
    const float4* W4;  // [4][4][192]
    const float2* W2;  // [4][192]
    template <int MU>
    __device__ __forceinline__ void link(int e, cplx<float> u[3][3]) const {
        const float4* w = W4 + MU * 4 * SPLIT_LINKS + e;
        const float4 a = w[0], b = w[SPLIT_LINKS], c = w[2 * SPLIT_LINKS], d = w[3 * SPLIT_LINKS];
        const float2 z = W2[MU * SPLIT_LINKS + e];
        u[0][0] = mk(a.x, a.y);
        u[0][1] = mk(a.z, a.w);
        u[0][2] = mk(b.x, b.y);
        u[1][0] = mk(b.z, b.w);
        u[1][1] = mk(c.x, c.y);
        u[1][2] = mk(c.z, c.w);
        u[2][0] = mk(d.x, d.y);
        u[2][1] = mk(d.z, d.w);
        u[2][2] = mk(z.x, z.y);
    }
};

// What the hops of a thread need to know of its site pair t: the block
// coordinates l (l[0..2] are those of both sites), where its spins sit in a
// block field, and the link entries of its sites without parity
struct SplitPair {
    int l0, l1, l2;
    int par0;       // the even site has local index 2 t + par0
    int a, b;       // slot t in spin sg, and in spin 3 - sg
    int e0, e1, e2, e3;
    __device__ __forceinline__ SplitPair(int t, int sg) {
        const int base = 2 * t;
        l0 = base >> 6;
        l1 = (base >> 4) & 3;
        l2 = (base >> 2) & 3;
        par0 = (l0 + l1 + l2 + (base & 3)) & 1;
        a = SPIN_STRIDE * sg + t;
        b = SPIN_STRIDE * (3 - sg) + t;
        e0 = link_entry<0>(0, base);
        e1 = link_entry<1>(0, base);
        e2 = link_entry<2>(0, base);
        e3 = link_entry<3>(0, base);
    }
};

// The compound links of site me (parity sg) that stay inside its block, to
// their entries of the block's links at W4, W2 (SplitLinks)
template <bool QNZ>
__device__ __forceinline__ void block_links(const Geom& g, const Fields<float>& f, const Site& me, int sg, float q,
                                            float4* __restrict__ W4, float2* __restrict__ W2) {
#pragma unroll
    for (int mu = 0; mu < 4; ++mu) {
        if (me.l[mu] == SAP_BS - 1) continue;
        const int e = mu == 0   ? link_entry<0>(sg, me.lidx)
                      : mu == 1 ? link_entry<1>(sg, me.lidx)
                      : mu == 2 ? link_entry<2>(sg, me.lidx)
                                : link_entry<3>(sg, me.lidx);
        cplx<float> u[3][3];
        load_link(f.U, g.V, mu, me.s, u);
        cplx<float> z = QNZ ? link_phase(f.A, g.V, mu, me.s, q) : mk(1.f, 0.f);
        z = -0.5f * z;
#pragma unroll
        for (int a = 0; a < 3; ++a)
#pragma unroll
            for (int b = 0; b < 3; ++b) u[a][b] = z * u[a][b];
        W4[(mu * 4 + 0) * SPLIT_LINKS + e] = make_float4(u[0][0].re, u[0][0].im, u[0][1].re, u[0][1].im);
        W4[(mu * 4 + 1) * SPLIT_LINKS + e] = make_float4(u[0][2].re, u[0][2].im, u[1][0].re, u[1][0].im);
        W4[(mu * 4 + 2) * SPLIT_LINKS + e] = make_float4(u[1][1].re, u[1][1].im, u[1][2].re, u[1][2].im);
        W4[(mu * 4 + 3) * SPLIT_LINKS + e] = make_float4(u[2][0].re, u[2][0].im, u[2][1].re, u[2][1].im);
        W2[mu * SPLIT_LINKS + e] = make_float2(u[2][2].re, u[2][2].im);
    }
}

constexpr int PLAN_LINK_F4 = 16 * SPLIT_LINKS + 2 * SPLIT_LINKS;  // float4 of one block's links
constexpr int PLAN_CLOVER_F4 = 2 * CLOVER_F4 * SAP_HALF;          // of its clover blocks
constexpr size_t split_link_bytes() { return 16 * SPLIT_LINKS * sizeof(float4) + 4 * SPLIT_LINKS * sizeof(float2); }

// Hops of direction MU inside the block for thread sg (sgn = +1 for sg = 0,
// -1 for sg = 1) at the site of parity p. With a the neighbour's spin sg and b
// the lower spin named below, h_sg = a + DIR c_MU b with c_0 = 1, c_1 = i, c_2 =
// sgn, c_3 = sgn i; g = U h_sg (U^+ backwards) goes to au (upper spin sg) and,
// times DIR, 1 / -i / sgn / -sgn i for MU = 0..3, to al (lower spin 2 + sg, MU =
// 0, 3) or ax (lower spin 3 - sg, the partner's, MU = 1, 2). l: the site's
// coordinate; fa, fb: the pair's slot in spins sg and, for MU = 1, 2, 3 - sg of
// the field; ef, eb: entries of the links at the site and at the site behind it;
// hop: slots to the next site.
template <int MU>
__device__ __forceinline__ void split_dir(const SplitLinks& bl, int l, const float2* fa, const float2* fb, int hopf,
                                          int hopb, int ef, int eb, float sgn, cplx<float> au[3], cplx<float> al[3],
                                          cplx<float> ax[3]) {
    const float2* lower = (MU == 0 || MU == 3) ? fa + 2 * SPIN_STRIDE : fb;
    cplx<float> a[3], b[3], h[3], gv[3], u[3][3];
    __syncwarp();  // one copy of each body per warp
    if (l < SAP_BS - 1) {
        ld3(fa + hopf, a);
        ld3(lower + hopf, b);
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            if (MU == 0) h[c] = a[c] + b[c];
            else if (MU == 1) h[c] = a[c] + times_i(b[c]);
            else if (MU == 2) h[c] = a[c] + sgn * b[c];
            else h[c] = a[c] + sgn * times_i(b[c]);
        }
        bl.link<MU>(ef, u);
        su3_mul(u, h, gv);
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            au[c] = au[c] + gv[c];
            if (MU == 0) al[c] = al[c] + gv[c];
            else if (MU == 1) ax[c] = ax[c] + times_mi(gv[c]);
            else if (MU == 2) ax[c] = ax[c] + sgn * gv[c];
            else al[c] = al[c] - sgn * times_i(gv[c]);
        }
    }
    __syncwarp();
    if (l > 0) {
        ld3(fa + hopb, a);
        ld3(lower + hopb, b);
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            if (MU == 0) h[c] = a[c] - b[c];
            else if (MU == 1) h[c] = a[c] - times_i(b[c]);
            else if (MU == 2) h[c] = a[c] - sgn * b[c];
            else h[c] = a[c] - sgn * times_i(b[c]);
        }
        bl.link<MU>(eb, u);
        su3_dag_mul(u, h, gv);
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            au[c] = au[c] + gv[c];
            if (MU == 0) al[c] = al[c] - gv[c];
            else if (MU == 1) ax[c] = ax[c] + times_i(gv[c]);
            else if (MU == 2) ax[c] = ax[c] - sgn * gv[c];
            else al[c] = al[c] + sgn * times_i(gv[c]);
        }
    }
}

// raw block-hop sum at the pair's site of parity p (src: field of the other
// parity), own half (acc[0..2] spin sg, acc[3..5] spin 2 + sg); every thread of
// the warp must call it (one shuffle at the end)
__device__ __forceinline__ void split_hops(const SplitLinks& bl, const float2* src, const SplitPair& sp, int t, int p,
                                           float sgn, cplx<float> acc[6]) {
    cplx<float> au[3], al[3], ax[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) au[c] = al[c] = ax[c] = mk(0.f, 0.f);
    const float2 *fa = src + sp.a, *fb = src + sp.b;
    const int d = p ? 1 - sp.par0 : sp.par0;         // the site is 2 t + d
    const int ef = p * (SPLIT_LINKS / 2), eb = SPLIT_LINKS / 2 - ef;  // entries of this parity and the other
    split_dir<0>(bl, sp.l0, fa, fb, 32, -32, sp.e0 + ef, sp.e0 + eb - 32, sgn, au, al, ax);
    split_dir<1>(bl, sp.l1, fa, fb, 8, -8, sp.e1 + ef, sp.e1 + eb - 8, sgn, au, al, ax);
    split_dir<2>(bl, sp.l2, fa, fb, 2, -2, sp.e2 + ef, sp.e2 + eb - 2, sgn, au, al, ax);
    split_dir<3>(bl, 2 * (t & 1) + d, fa, fb, d, d - 1, sp.e3 + d, sp.e3 + d - 1, sgn, au, al, ax);
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const float xr = __shfl_xor_sync(FULL_MASK, ax[c].re, 1);
        const float xi = __shfl_xor_sync(FULL_MASK, ax[c].im, 1);
        acc[c] = au[c];
        acc[3 + c] = al[c] + mk(xr, xi);
    }
}

// Tensor memory of the split kernel. The rows of M_oo^-1 and M_ee that a thread
// applies, 27 floats for each of the two 6x6 blocks of a matrix, are its own and
// are used in every MR step: they are put into tensor memory, whose lanes belong
// to the threads of a warp, once per launch. A warp reaches the 32 lanes from
// 32 (warp % 4) on, so warps w and w + 4 take different columns: 2 x 4 x 32
// columns for a thread block, and with two of them all 512 of an SM.
// Loaded again for every step, 73 KB per block outgrew L1 and, with 304 blocks
// in flight, L2: DRAM bytes of a launch on 48x48x24x24 sites 929 -> 606 MB, waits
// for global memory per instruction 2.0 -> 0.8, and with rows chosen and
// conjugated once 9 % fewer instructions; one application on 64x64x32x32 sites
// 12.52 -> 11.08 ms, six right-hand sides on 32x32x16x16 4.73 -> 4.24 ms. Filling
// the rows costs one pass and pays from the second MR step on: with nmr = 1, 2,
// 3, 5, 8 an application takes 7.80, 7.91, 8.71, 11.08, 14.84 ms, and 6.82, 8.31,
// 9.66, 12.58, 17.08 with the blocks read from memory in every step. There is no
// second form for nmr = 1: the solvers take 5 steps (the deflation's smoothing 4).
constexpr int TM_BLOCK = 32;             // columns of one 6x6 block's rows (28 used)
constexpr int TM_COLS = 2 * 4 * TM_BLOCK;

// the whole of warp 0; the address arrives in shared memory
__device__ __forceinline__ void tm_alloc(uint32_t* s_addr) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     (uint32_t)__cvta_generic_to_shared(s_addr)),
                 "n"(TM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
}
__device__ __forceinline__ void tm_free(uint32_t addr) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(addr), "n"(TM_COLS));
}
__device__ __forceinline__ void tm_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tm_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tm_store_wait() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// 28 columns of this thread's lane; every thread of the warp takes part
__device__ __forceinline__ void tm_store28(uint32_t a, const float r[28]) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
        "%15, %16};" ::"r"(a),
        "f"(r[0]), "f"(r[1]), "f"(r[2]), "f"(r[3]), "f"(r[4]), "f"(r[5]), "f"(r[6]), "f"(r[7]), "f"(r[8]), "f"(r[9]),
        "f"(r[10]), "f"(r[11]), "f"(r[12]), "f"(r[13]), "f"(r[14]), "f"(r[15]));
    asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"r"(a + 16),
                 "f"(r[16]), "f"(r[17]), "f"(r[18]), "f"(r[19]), "f"(r[20]), "f"(r[21]), "f"(r[22]), "f"(r[23]));
    asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1, %2, %3, %4};" ::"r"(a + 24), "f"(r[24]),
                 "f"(r[25]), "f"(r[26]), "f"(r[27]));
}
__device__ __forceinline__ void tm_load28(uint32_t a, float r[28]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
        "%15}, [%28];\n"
        "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%16, %17, %18, %19, %20, %21, %22, %23}, [%29];\n"
        "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%24, %25, %26, %27}, [%30];\n"
        "tcgen05.wait::ld.sync.aligned;"
        : "=f"(r[0]), "=f"(r[1]), "=f"(r[2]), "=f"(r[3]), "=f"(r[4]), "=f"(r[5]), "=f"(r[6]), "=f"(r[7]), "=f"(r[8]),
          "=f"(r[9]), "=f"(r[10]), "=f"(r[11]), "=f"(r[12]), "=f"(r[13]), "=f"(r[14]), "=f"(r[15]), "=f"(r[16]),
          "=f"(r[17]), "=f"(r[18]), "=f"(r[19]), "=f"(r[20]), "=f"(r[21]), "=f"(r[22]), "=f"(r[23]), "=f"(r[24]),
          "=f"(r[25]), "=f"(r[26]), "=f"(r[27])
        : "r"(a), "r"(a + 16), "r"(a + 24));
}

// What the rows of thread sg of both packed Hermitian 6x6 blocks of a site need,
// eight of the nine float4 of each; C: the site's first float4, the others
// `stride` apart. All loads of a matrix are under way before the first
// is used (block by block, with the stores between: 11.16 against 11.08 ms on
// 64x64x32x32 sites, 8.28 against 7.91 with 2 MR steps).
__device__ __forceinline__ void clover_load(const float4* __restrict__ C, size_t stride, int sg, float4 q[16]) {
#pragma unroll
    for (int blk = 0; blk < 2; ++blk) {
        const float4* Cb = C + 9 * blk * stride;
        q[8 * blk] = Cb[0], q[8 * blk + 1] = Cb[stride];
        q[8 * blk + 2] = Cb[(sg ? 8 : 2) * stride];
#pragma unroll
        for (int n = 3; n < 8; ++n) q[8 * blk + n] = Cb[n * stride];
    }
}

// This thread's rows (3 sg + a, a = 0..2), from clover_load, to tensor memory at
// a: per block E[a][b] (18 floats), L(3 sg + 1, 3 sg), L(3 sg + 2, 3 sg), L(3 sg +
// 2, 3 sg + 1) (6) and the diagonal (3). In block order the rows of thread sg see
// a Hermitian 3x3 diagonal block (entries d[3 sg + a] and L(3 sg + a, 3 sg + b))
// and the off-diagonal 3x3 block E = B[a][b] = L(3 + a, b) for sg = 1, B^+ for
// sg = 0.
__device__ __forceinline__ void clover_rows(const float4 q[16], int sg, uint32_t a) {
#pragma unroll
    for (int blk = 0; blk < 2; ++blk) {
        const float4 q0 = q[8 * blk], q1 = q[8 * blk + 1], X = q[8 * blk + 2], q3 = q[8 * blk + 3];
        const float4 q4 = q[8 * blk + 4], q5 = q[8 * blk + 5], q6 = q[8 * blk + 6], q7 = q[8 * blk + 7];
        // packed floats: d_i at i, L_k at (6 + 2k, 7 + 2k); float4 n holds 4n..4n+3
        const cplx<float> B[3][3] = {{mk(q3.x, q3.y), mk(q3.z, q3.w), mk(q4.x, q4.y)},
                                     {mk(q4.z, q4.w), mk(q5.x, q5.y), mk(q5.z, q5.w)},
                                     {mk(q6.z, q6.w), mk(q7.x, q7.y), mk(q7.z, q7.w)}};
        float r[28];
#pragma unroll
        for (int x = 0; x < 3; ++x)
#pragma unroll
            for (int y = 0; y < 3; ++y) {
                r[6 * x + 2 * y] = sg ? B[x][y].re : B[y][x].re;
                r[6 * x + 2 * y + 1] = sg ? B[x][y].im : -B[y][x].im;
            }
        r[18] = sg ? q6.x : q1.z, r[19] = sg ? q6.y : q1.w;  // L(4,3) : L(1,0)
        r[20] = X.x, r[21] = X.y;                            // L(5,3) : L(2,0)
        r[22] = X.z, r[23] = X.w;                            // L(5,4) : L(2,1)
        r[24] = sg ? q0.w : q0.x, r[25] = sg ? q1.x : q0.y, r[26] = sg ? q1.y : q0.z;
        r[27] = 0.f;
        tm_store28(a + blk * TM_BLOCK, r);
    }
}

// Own rows of the matrix at a times v; v and y are own halves, the partner's
// half is shuffled in. Every thread of the warp must call it.
__device__ __forceinline__ void clover_half(uint32_t tm, const cplx<float> v[6], cplx<float> y[6]) {
#pragma unroll
    for (int blk = 0; blk < 2; ++blk) {
        const cplx<float>* w = v + 3 * blk;
        cplx<float> pp[3], z[3];
#pragma unroll
        for (int k = 0; k < 3; ++k)
            pp[k] = mk(__shfl_xor_sync(FULL_MASK, w[k].re, 1), __shfl_xor_sync(FULL_MASK, w[k].im, 1));
        float r[28];
        tm_load28(tm + blk * TM_BLOCK, r);
        const cplx<float> l10 = mk(r[18], r[19]), l20 = mk(r[20], r[21]), l21 = mk(r[22], r[23]);
        // the diagonal, the largest term, comes last
        z[0] = cmad(l20, w[2], cmul(l10, w[1]));
        z[1] = cmad(l21, w[2], l10 * w[0]);
        z[2] = mad(l21, w[1], l20 * w[0]);
#pragma unroll
        for (int a = 0; a < 3; ++a)
#pragma unroll
            for (int b = 0; b < 3; ++b) z[a] = mad(mk(r[6 * a + 2 * b], r[6 * a + 2 * b + 1]), pp[b], z[a]);
#pragma unroll
        for (int a = 0; a < 3; ++a) y[3 * blk + a] = rmad(r[24 + a], w[a], z[a]);
    }
}

// The hop of D in direction MU that leaves the block at a site t on one of its
// two faces in that direction: forwards from the upper face, backwards from the
// lower one. Both cases run as one body with the sign as a factor and the link
// transposed where needed, so a warp whose lanes sit on both faces takes 4 hops
// instead of 8 half-empty ones.
template <bool QNZ, int MU>
__device__ __forceinline__ void crossing_load(const Geom& g, const Fields<float>& f, const float4* __restrict__ d,
                                              const Site& t, int po, HopData& h) {
    const bool fwd = t.l[MU] == SAP_BS - 1;
    const int lf = neighbour_lex<MU, +1>(g, t.x[0], t.x[1], t.x[2], t.x[3]);
    const int lb = neighbour_lex<MU, -1>(g, t.x[0], t.x[1], t.x[2], t.x[3]);
    const int sn = native_index(g, fwd ? lf : lb, po);
    const int sl = fwd ? t.s : sn;  // the link of x forwards, of the neighbour backwards
#pragma unroll
    for (int c = 0; c < 6; ++c) h.sp[c] = d[(size_t)c * g.V + sn];
#pragma unroll
    for (int k = 0; k < 3; ++k) h.lk[k] = f.U[((size_t)MU * 3 + k) * g.V + sl];
    if (QNZ) h.ang = reinterpret_cast<const float*>(f.A + sl)[MU];
}

// acc += raw crossing hop (without the factor -1/2) from the loads h
template <bool QNZ, int MU>
__device__ __forceinline__ void crossing_add(const HopData& h, float q, const Site& t, cplx<float> acc[12]) {
    const bool fwd = t.l[MU] == SAP_BS - 1;
    const float D = fwd ? 1.f : -1.f;
    cplx<float> v[12], h0[3], h1[3], g0[3], g1[3], u[3][3], w[3][3];
#pragma unroll
    for (int c = 0; c < 6; ++c) {
        v[2 * c] = mk(h.sp[c].x, h.sp[c].y);
        v[2 * c + 1] = mk(h.sp[c].z, h.sp[c].w);
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) {  // project<MU, DIR> with DIR = D
        const cplx<float> a0 = v[c], a1 = v[3 + c], a2 = v[6 + c], a3 = v[9 + c];
        if (MU == 0) h0[c] = rmad(D, a2, a0), h1[c] = rmad(D, a3, a1);
        else if (MU == 1) h0[c] = rmad(D, times_i(a3), a0), h1[c] = rmad(D, times_i(a2), a1);
        else if (MU == 2) h0[c] = rmad(D, a3, a0), h1[c] = rmad(-D, a2, a1);
        else h0[c] = rmad(D, times_i(a2), a0), h1[c] = rmad(-D, times_i(a3), a1);
    }
    link_rows(h.lk, u);
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int b = 0; b < 3; ++b) w[a][b] = mk(fwd ? u[a][b].re : u[b][a].re, fwd ? u[a][b].im : -u[b][a].im);
    su3_mul(w, h0, g0);
    su3_mul(w, h1, g1);
    if (QNZ) {
        cplx<float> ph = angle_phase(h.ang, q);
        ph.im *= D;
        times3(ph, g0);
        times3(ph, g1);
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) {  // accumulate<MU, DIR>
        acc[c] = acc[c] + g0[c];
        acc[3 + c] = acc[3 + c] + g1[c];
        if (MU == 0) acc[6 + c] = rmad(D, g0[c], acc[6 + c]), acc[9 + c] = rmad(D, g1[c], acc[9 + c]);
        else if (MU == 1) acc[6 + c] = rmad(D, times_mi(g1[c]), acc[6 + c]), acc[9 + c] = rmad(D, times_mi(g0[c]), acc[9 + c]);
        else if (MU == 2) acc[6 + c] = rmad(-D, g1[c], acc[6 + c]), acc[9 + c] = rmad(D, g0[c], acc[9 + c]);
        else acc[6 + c] = rmad(D, times_mi(g0[c]), acc[6 + c]), acc[9 + c] = rmad(D, times_i(g1[c]), acc[9 + c]);
    }
}

// raw sum of the hops of D at site t that leave its block
template <bool QNZ>
__device__ __forceinline__ void crossing_hops(const Geom& g, const Fields<float>& f, const float4* __restrict__ d,
                                              float q, const Site& t, int po, cplx<float> acc[12]) {
    HopData h;
#pragma unroll
    for (int i = 0; i < 12; ++i) acc[i] = mk(0.f, 0.f);
    __syncwarp();
    if (t.l[0] == SAP_BS - 1 || t.l[0] == 0) {
        crossing_load<QNZ, 0>(g, f, d, t, po, h);
        crossing_add<QNZ, 0>(h, q, t, acc);
    }
    __syncwarp();
    if (t.l[1] == SAP_BS - 1 || t.l[1] == 0) {
        crossing_load<QNZ, 1>(g, f, d, t, po, h);
        crossing_add<QNZ, 1>(h, q, t, acc);
    }
    __syncwarp();
    if (t.l[2] == SAP_BS - 1 || t.l[2] == 0) {
        crossing_load<QNZ, 2>(g, f, d, t, po, h);
        crossing_add<QNZ, 2>(h, q, t, acc);
    }
    __syncwarp();
    if (t.l[3] == SAP_BS - 1 || t.l[3] == 0) {
        crossing_load<QNZ, 3>(g, f, d, t, po, h);
        crossing_add<QNZ, 3>(h, q, t, acc);
    }
}

// How k_sap_split forms the residual of its blocks and what it keeps
enum SplitFlags : int {
    SF_FIRST = 1,  // first visit of this colour: r = eta, psi = delta (psi is not read)
    SF_CROSS = 2,  // subtract D_cross of the other colour's last corrections
    SF_KEEP_RHO = 4,    // keep rho of the even sites for the next visit of this colour
    SF_KEEP_DELTA = 8,  // keep delta for the next visit of the other colour
};

// One right-hand side of the FP32 block solve: source eta, output psi and the
// work fields, delta of every site (6 float4 per site, stride V) and rho of
// the even sites (stride Vh)
struct SplitWork {
    const float4* eta;
    float4* psi;
    float4* delta;
    float4* rho;
};

// right-hand sides of one operator solved in one launch
constexpr int SPLIT_MAXR = 12;
struct SplitRhsList {
    SplitWork r[SPLIT_MAXR];
    int n;
};

// Same phases as sap_block_body, with the site-pair work split over the two
// threads of a pair, for one right-hand side; the residual comes from eta on
// the first visit of a colour, else from the kept rho and the crossing hops of
// the kept delta.
// COPY: operator data from the block-by-block copy; else from the native fields
// (f.U, f.A, f.C, plan.Cinv), the block's links made here from the same
// expressions as in the copy. The results are the same bits.
template <bool QNZ, bool COPY>
__device__ __forceinline__ void sap_split_body(const Geom& g, const SapGeom& sgm, int bidx, int colour,
                                               const Fields<float>& f, const SapPlan& plan,
                                               const SplitWork& wk, int flags, int nmr, float q) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float4* sW4 = reinterpret_cast<float4*>(smem_raw);
    float2* sW2 = reinterpret_cast<float2*>(smem_raw + 16 * SPLIT_LINKS * sizeof(float4));
    const SplitLinks bl{sW4, sW2};
    float2* sm = reinterpret_cast<float2*>(smem_raw + split_link_bytes());
    float2* s_rho = sm;                 // r on the even sites, the MR residual, delta_o at the end
    float2* s_t = sm + FIELD_F2;        // r on the odd sites, the odd temporary, delta_e at the end
    float* red = reinterpret_cast<float*>(sm + 2 * FIELD_F2);  // 3 * warps reduction slots
    uint32_t* s_tm = reinterpret_cast<uint32_t*>(red + 3 * (SPLIT_THREADS / 32));

    if (threadIdx.x < 32) tm_alloc(s_tm);
    int org[4];
    const int blk = block_origin(sgm, bidx, colour, org);
    const int t = threadIdx.x >> 1;
    const int sg = threadIdx.x & 1;
    const float sgn = sg ? -1.f : 1.f;
    const SplitPair sp(t, sg);
    // the site whose residual this thread forms: the even one for sg = 0
    const Site me = make_site(g, org, 2 * t + (sg ? 1 - sp.par0 : sp.par0));
    const int even_s = __shfl_sync(FULL_MASK, me.s, threadIdx.x & 30);  // native index of the even site

    if constexpr (!COPY) {
        block_links<QNZ>(g, f, me, sg, q, sW4, sW2);
    } else {  // the block's links, copied while the residual is formed
        const float4* src = plan.links + (size_t)blk * PLAN_LINK_F4;
        for (int k = threadIdx.x; k < PLAN_LINK_F4; k += SPLIT_THREADS) copy_async16(sW4 + k, src + k);
    }
    tm_fence_before();
    __syncthreads();
    tm_fence_after();
    const uint32_t tm = *s_tm;
    // M_oo^-1 and M_ee of this pair, this thread's rows
    const uint32_t Moi = tm + ((threadIdx.x & 96u) << 16) + (threadIdx.x >> 7) * (TM_COLS / 2);
    const uint32_t Mee = Moi + 2 * TM_BLOCK;
    {
        const int odd_s = COPY ? 0 : __shfl_sync(FULL_MASK, me.s, (threadIdx.x & 30) | 1);
        const float4* oi = COPY ? plan.clover + (size_t)blk * PLAN_CLOVER_F4 + t : plan.Cinv + (odd_s - g.Vh);
        const float4* ee = COPY ? oi + CLOVER_F4 * SAP_HALF : f.C + even_s;
        float4 c[16];
        clover_load(oi, COPY ? SAP_HALF : g.Vh, sg, c);
        clover_rows(c, sg, Moi);
        clover_load(ee, COPY ? SAP_HALF : g.V, sg, c);
        clover_rows(c, sg, Mee);
        tm_store_wait();
    }

    {
        cplx<float> r[12];
        if (flags & SF_FIRST) {
            load_spinor(wk.eta, g.V, me.s, r);
        } else if (sg == 0) {  // even site: the kept rho
            load_spinor(wk.rho, g.Vh, me.s, r);
        } else {  // odd site: the block solve left no residual
#pragma unroll
            for (int i = 0; i < 12; ++i) r[i] = mk(0.f, 0.f);
        }
        if (flags & SF_CROSS) {  // r -= D_cross delta = r + 1/2 (crossing hops of delta)
            cplx<float> acc[12];
            crossing_hops<QNZ>(g, f, wk.delta, q, me, 1 - sg, acc);  // neighbours of the other parity
#pragma unroll
            for (int i = 0; i < 12; ++i) r[i] = r[i] + 0.5f * acc[i];
        }
        st_full(sg ? s_t : s_rho, t, r);
    }
    __syncwarp();
    copy_async_wait();
    __syncthreads();

    // r_o (this thread's half) stays in registers until the last step; the
    // pair overwrites its own halves of s_t with t_o = M_oo^-1 r_o
    cplx<float> ro[6], v[6], w[6], acc[6], rho[6];
    ld_half(s_t, sg, t, ro);
    clover_half(Moi, ro, w);
    st_half(s_t, sg, t, w);
    __syncthreads();

    // this thread's half of rho stays in registers (read back from shared memory
    // for every step: 12.56 against 12.52 ms on 64x64x32x32)
    cplx<float> de[6];
#pragma unroll
    for (int i = 0; i < 6; ++i) de[i] = mk(0.f, 0.f);
    const int nsteps = 2 * nmr + 2;
#pragma unroll 1
    for (int step = 0; step < nsteps; ++step) {
        const bool odd = (step & 1) != 0;
        const bool last = step == nsteps - 1;
        split_hops(bl, odd ? (last ? s_t : s_rho) : s_t, sp, t, odd ? 1 : 0, sgn, acc);
        // acc = H psi on the sites of this step's parity (the links carry the -1/2)
        if (step == 0) {
            ld_half(s_rho, sg, t, rho);  // r_e
#pragma unroll
            for (int i = 0; i < 6; ++i) rho[i] = rho[i] - acc[i];
            st_half(s_rho, sg, t, rho);
        } else if (last) {
#pragma unroll
            for (int i = 0; i < 6; ++i) v[i] = ro[i] - acc[i];
            clover_half(Moi, v, w);  // delta_o (s_rho is no longer read)
            st_half(s_rho, sg, t, w);
        } else if (odd) {
            clover_half(Moi, acc, w);
            st_half(s_t, sg, t, w);
        } else {
            clover_half(Mee, rho, w);
#pragma unroll
            for (int i = 0; i < 6; ++i) w[i] = w[i] - acc[i];
            float a_re = 0.f, a_im = 0.f, b = 0.f;
#pragma unroll
            for (int i = 0; i < 6; ++i) {
                a_re = fmaf(w[i].im, rho[i].im, fmaf(w[i].re, rho[i].re, a_re));
                a_im = fmaf(-w[i].im, rho[i].re, fmaf(w[i].re, rho[i].im, a_im));
                b = fmaf(w[i].im, w[i].im, fmaf(w[i].re, w[i].re, b));
            }
            float sums[3];
            // red is next written two steps later, after the barriers that end each step
            block_sum3<float, SPLIT_THREADS, false>(a_re, a_im, b, red, sums);
            if (sums[2] > 0.f) {  // else rho = 0 on the whole block: nothing to add
                const cplx<float> om = mk(sums[0] / sums[2], sums[1] / sums[2]);
#pragma unroll
                for (int i = 0; i < 6; ++i) {
                    de[i] = mad(om, rho[i], de[i]);
                    rho[i] = mad(-om, w[i], rho[i]);
                }
            }
            if (step == nsteps - 2) {
                st_half(s_t, sg, t, de);  // delta_e for the last step
                if (flags & SF_KEEP_RHO) {
                    // this thread's half of rho at the even site: components 3 sg + c and 6 + 3 sg + c
                    float2* kr = reinterpret_cast<float2*>(wk.rho);
#pragma unroll
                    for (int h = 0; h < 2; ++h)
#pragma unroll
                        for (int c = 0; c < 3; ++c) {
                            const int i = 6 * h + 3 * sg + c;
                            kr[2 * ((size_t)(i >> 1) * g.Vh + even_s) + (i & 1)] = make_float2(rho[3 * h + c].re, rho[3 * h + c].im);
                        }
                }
            } else {
                st_half(s_rho, sg, t, rho);
            }
        }
        tm_fence_before();
        __syncthreads();
    }
    tm_fence_after();
    if (threadIdx.x < 32) tm_free(tm);
    // psi_B += delta on this thread's site: delta_e in s_t, delta_o in s_rho
    cplx<float> d[12];
    ld_full(sg ? s_rho : s_t, t, d);
    if (flags & SF_KEEP_DELTA) store_spinor(wk.delta, g.V, me.s, d);
    if (!(flags & SF_FIRST)) {
        cplx<float> o[12];
        load_spinor(wk.psi, g.V, me.s, o);
#pragma unroll
        for (int i = 0; i < 12; ++i) d[i] = d[i] + o[i];
    }
    store_spinor(wk.psi, g.V, me.s, d);
}

// Thread block b: right-hand side b % n of lattice block b / n, so that the
// right-hand sides of a block run side by side and share its operator data in
// L2. (One thread block for all right-hand sides of a block, its links staged
// once, was slower at every size: 6 right-hand sides on 32x32x16x16 946 us each
// against 818, 12 on 16x16x8x8 269 against 61, where it left SMs idle.)
template <bool QNZ, bool COPY>
__global__ void __launch_bounds__(SPLIT_THREADS, 2) k_sap_split(const __grid_constant__ Geom g,
                                                                const __grid_constant__ SapGeom sgm, int colour,
                                                                const __grid_constant__ Fields<float> f,
                                                                const __grid_constant__ SapPlan plan,
                                                                const __grid_constant__ SplitRhsList rl, int flags,
                                                                int nmr, float q) {
    const int b = blockIdx.x / rl.n;
    sap_split_body<QNZ, COPY>(g, sgm, b, colour, f, plan, rl.r[blockIdx.x - b * rl.n], flags, nmr, q);
}

// The block-by-block copy of the operator for the split kernel: one thread
// block per lattice block, thread 2t + sg takes the site of parity sg of pair
// t (parity 0: links and M_ee, parity 1: links and M_oo^-1).
template <bool QNZ>
__global__ void __launch_bounds__(SPLIT_THREADS) k_sap_plan(Geom g, SapGeom sgm, Fields<float> f,
                                                            const float4* __restrict__ Cinv, float4* __restrict__ links,
                                                            float4* __restrict__ clover, float q) {
    int org[4];
    const int blk = block_origin(sgm, blockIdx.x >> 1, blockIdx.x & 1, org);
    float4* W4 = links + (size_t)blk * PLAN_LINK_F4;
    float2* W2 = reinterpret_cast<float2*>(W4 + 16 * SPLIT_LINKS);
    const int t = threadIdx.x >> 1;
    const int sg = threadIdx.x & 1;
    const int base = 2 * t;
    const int par0 = ((base >> 6) + ((base >> 4) & 3) + ((base >> 2) & 3) + (base & 3)) & 1;
    const Site me = make_site(g, org, base + (sg ? 1 - par0 : par0));
    block_links<QNZ>(g, f, me, sg, q, W4, W2);
    float4* C = clover + (size_t)blk * PLAN_CLOVER_F4 + (sg ? 0 : CLOVER_F4 * SAP_HALF) + t;
    const float4* src = sg ? Cinv + (me.s - g.Vh) : f.C + me.s;
    const size_t stride = sg ? g.Vh : g.V;
#pragma unroll
    for (int n = 0; n < CLOVER_F4; ++n) C[n * SAP_HALF] = src[n * stride];
}

// batched form: thread block b works on block (b - cta_begin) of the job
// whose range holds b (one launch serves every job of a batch; without COPY all
// of them read the native fields)
template <bool COPY>
__global__ void __launch_bounds__(SPLIT_THREADS, 2) k_sap_block_batch(const SapJob* __restrict__ jobs, int njobs,
                                                                      int colour, int flags, int nmr) {
    int lo = 0, hi = njobs - 1;
    const int b = blockIdx.x;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (jobs[mid].cta_begin <= b) lo = mid;
        else hi = mid - 1;
    }
    const SapJob& J = jobs[lo];
    const SplitWork wk{J.eta, const_cast<float4*>(J.f.psi), J.delta, J.rho};
    sap_split_body<true, COPY>(J.g, J.sg, b - J.cta_begin, colour, J.f, J.plan, wk, flags, nmr, J.q);
}

template <typename R>
size_t sap_smem_bytes() {
    if (sizeof(R) == 4)  // split kernel: interior compound links, two block fields, reduction slots of 8 warps
        return split_link_bytes() + 2 * FIELD_F2 * sizeof(float2) + 3 * (SPLIT_THREADS / 32) * sizeof(float) +
               sizeof(uint32_t);
    return (72 * SAP_HALF + 3 * (SAP_THREADS / 32)) * sizeof(R);
}

// Dynamic shared memory of the split kernel, and an L1/shared carveout just
// large enough for two blocks per SM.
template <typename K>
int split_attrs(K kernel, size_t smem) {
    int dev = 0, per_sm = 0;
    QXD_CUDA(cudaGetDevice(&dev));
    QXD_CUDA(cudaDeviceGetAttribute(&per_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev));
    QXD_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    if (per_sm > 0) {
        const long need = 2L * ((long)smem + 1024);
        const int pct = (int)std::min(100L, (100 * need + per_sm - 1) / per_sm);
        QXD_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout, pct));
    }
    return QXD_OK;
}

// flags of visit `cy` of colour `colour` out of ncy cycles
int split_flags(int cy, int colour, int ncy) {
    int fl = 0;
    if (cy == 0) fl |= SF_FIRST;
    if (cy > 0 || colour == 1) fl |= SF_CROSS;  // the other colour has a correction
    if (cy + 1 < ncy) fl |= SF_KEEP_RHO;
    if (cy + 1 < ncy || colour == 0) fl |= SF_KEEP_DELTA;
    return fl;
}

// FP64 visit `cy` of colour `colour` out of ncy cycles
int launch_sap_block64(qxd_lattice* lat, const SapGeom& sg, int cy, int colour, Fields<double> f,
                       const double* Cinv, const double2* eta, int nmr, cudaStream_t st) {
    const size_t smem = sap_smem_bytes<double>();
    const int psi_zero = (cy == 0 && colour == 0) ? 1 : 0;
    QXD_CUDA(cudaFuncSetAttribute(k_sap_block, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    k_sap_block<<<sg.nhalf, SAP_THREADS, smem, st>>>(lat->g, sg, colour, psi_zero, f, Cinv, eta, nmr);
    QXD_LAUNCHED("k_sap_block");
    return QXD_OK;
}

// FP32: the ncy cycles for the right-hand sides of rl (one operator)
template <bool QNZ, bool COPY>
int split_cycles(qxd_lattice* lat, const SapGeom& sg, const SplitRhsList& rl, int ncy, int nmr, cudaStream_t st) {
    const size_t smem = sap_smem_bytes<float>();
    const int rc = split_attrs(k_sap_split<QNZ, COPY>, smem);
    if (rc) return rc;
    const SapPlan plan = sap_plan(lat);
    const Fields<float> f{nullptr, lat->U32, lat->A32, lat->C32};
    for (int cy = 0; cy < ncy; ++cy)
        for (int colour = 0; colour < 2; ++colour) {
            k_sap_split<QNZ, COPY><<<sg.nhalf * rl.n, SPLIT_THREADS, smem, st>>>(lat->g, sg, colour, f, plan, rl,
                                                                           split_flags(cy, colour, ncy), nmr,
                                                                           (float)lat->qhat);
            QXD_LAUNCHED("k_sap_split");
        }
    return QXD_OK;
}

}  // namespace

namespace {

// why the lattice does not admit the block colouring (nullptr: it does)
const char* sap_refusal(const Geom& g) {
    const int N[4] = {g.N0, g.N1, g.N2, g.N3};
    for (int m = 0; m < 4; ++m)
        if (N[m] % SAP_BS || (N[m] / SAP_BS) % 2)
            return "SAP: every simulated extent must be a multiple of 8 "
                   "(4^4 blocks, even number of blocks per direction)";
    if (g.cs2 || g.cs3) {
        if (g.L1 % SAP_BS) return "SAP: with C* boundaries L1 must be a multiple of 4";
        const int sh = g.L1 / SAP_BS;
        if ((g.cs2 && (N[2] / SAP_BS + sh) % 2) || (g.cs3 && (N[3] / SAP_BS + sh) % 2))
            return "SAP: the block colouring is not consistent across the shifted "
                   "C* boundary (L_k/4 + L1/4 must be even)";
    }
    return nullptr;
}

}  // namespace

int sap_check(qxd_lattice* lat) {
    const char* why = sap_refusal(lat->g);
    return why ? fail(QXD_ERR_ARG, why) : QXD_OK;
}

bool sap_admissible(const qxd_lattice* lat) { return !sap_refusal(lat->g); }

namespace {

// Whether the copy, which the Schwarz method can do without, may have its
// memory: half of the device stays free, for the program's other lattices,
// views and fields, and 16 times the copy (8 KB per site; a mixed GCR solve
// with 16 Krylov pairs takes 4), for the work on this operator itself.
bool copy_has_room(size_t bytes) {
    size_t free_bytes = 0, total = 0;
    if (cudaMemGetInfo(&free_bytes, &total) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return free_bytes > bytes && free_bytes - bytes >= std::max(total / 2, 16 * bytes);
}

}  // namespace

// Part of qxd_sw_build, which waits for it: the copy is complete before any
// application, on whatever stream, can follow, and no application allocates.
// Without memory for it the block solve reads the native fields (sap_split_body
// without COPY: one application on 64x64x32x32 sites 12.78 ms instead of 11.08).
int launch_sap_plan(qxd_lattice* lat, cudaStream_t st) {
    const SapGeom sg = sap_geom(lat->g);
    if (!lat->sap_plan && lat->sap_copy_wanted) {
        const size_t bytes = (size_t)sg.nblk * (PLAN_LINK_F4 + PLAN_CLOVER_F4) * sizeof(float4);
        const cudaError_t e = copy_has_room(bytes) ? cudaMalloc(&lat->sap_plan, bytes) : cudaErrorMemoryAllocation;
        if (e != cudaSuccess) {
            lat->sap_plan = nullptr;
            if (e != cudaErrorMemoryAllocation) return cuda_fail(e, "SAP: cudaMalloc(operator by blocks)");
            cudaGetLastError();
        }
    }
    if (!lat->sap_plan) return QXD_OK;
    const Fields<float> f{nullptr, lat->U32, lat->A32, lat->C32};
    float4* clover = lat->sap_plan + (size_t)sg.nblk * PLAN_LINK_F4;
    if (lat->qhat != 0)
        k_sap_plan<true><<<sg.nblk, SPLIT_THREADS, 0, st>>>(lat->g, sg, f, lat->Cinv32, lat->sap_plan, clover,
                                                            (float)lat->qhat);
    else
        k_sap_plan<false><<<sg.nblk, SPLIT_THREADS, 0, st>>>(lat->g, sg, f, lat->Cinv32, lat->sap_plan, clover, 0.f);
    QXD_LAUNCHED("k_sap_plan");
    return QXD_OK;
}

SapPlan sap_plan(const qxd_lattice* lat) {
    if (!lat->sap_plan) return SapPlan{nullptr, nullptr, lat->Cinv32};
    return SapPlan{lat->sap_plan, lat->sap_plan + (size_t)sap_geom(lat->g).nblk * PLAN_LINK_F4, lat->Cinv32};
}

int sap_apply_multi(qxd_lattice* lat, int nrhs, void* const* outs, const void* const* ins, float4* const* works,
                    int ncy, int nmr, cudaStream_t st) {
    const SapGeom sg = sap_geom(lat->g);
    const size_t V = (size_t)lat->g.V;
    for (int i0 = 0; i0 < nrhs; i0 += SPLIT_MAXR) {
        SplitRhsList rl{};
        rl.n = std::min(SPLIT_MAXR, nrhs - i0);
        for (int i = 0; i < rl.n; ++i)
            rl.r[i] = SplitWork{(const float4*)ins[i0 + i], (float4*)outs[i0 + i], works[i0 + i],
                                works[i0 + i] + (size_t)SPINOR_F4 * V};
        const bool copy = lat->sap_plan != nullptr;
        const int rc = lat->qhat != 0 ? (copy ? split_cycles<true, true>(lat, sg, rl, ncy, nmr, st)
                                              : split_cycles<true, false>(lat, sg, rl, ncy, nmr, st))
                                      : (copy ? split_cycles<false, true>(lat, sg, rl, ncy, nmr, st)
                                              : split_cycles<false, false>(lat, sg, rl, ncy, nmr, st));
        if (rc) return rc;
    }
    return QXD_OK;
}

template <typename R>
int sap_apply(qxd_lattice* lat, SapWork& w, void* out, const void* in, int ncy, int nmr, cudaStream_t st) {
    const Geom& g = lat->g;
    w.sg = sap_geom(g);
    if constexpr (sizeof(R) == 4) {
        // the first visit of each colour writes psi = delta; work fields: delta
        // (V sites) and rho (Vh even sites), kept with the lattice
        if (!lat->sap_r) {
            const cudaError_t e = cudaMalloc(&lat->sap_r, ((size_t)g.V + g.Vh) * SPINOR_F4 * sizeof(float4));
            if (e != cudaSuccess) {
                lat->sap_r = nullptr;
                return cuda_fail(e, "SAP: cudaMalloc(work fields)");
            }
        }
        float4* work = lat->sap_r;
        return sap_apply_multi(lat, 1, &out, &in, &work, ncy, nmr, st);
    } else {
        // psi starts at zero; the first half-cycle writes the blocks of colour 0
        // without reading psi, and the blocks of colour 1 must read zeros there
        QXD_CUDA(cudaMemsetAsync(out, 0, (size_t)g.V * 24 * sizeof(R), st));
        const Fields<double> f{(const double2*)out, lat->W64, lat->C64};
        for (int cy = 0; cy < ncy; ++cy)
            for (int colour = 0; colour < 2; ++colour) {
                const int rc = launch_sap_block64(lat, w.sg, cy, colour, f, lat->Cinv64, (const double2*)in, nmr, st);
                if (rc) return rc;
            }
        return QXD_OK;
    }
}

template int sap_apply<float>(qxd_lattice*, SapWork&, void*, const void*, int, int, cudaStream_t);

SapGeom sap_geom(const Geom& g) {
    SapGeom sg;
    sg.nb0 = g.N0 / SAP_BS;
    sg.nb1 = g.N1 / SAP_BS;
    sg.nb2 = g.N2 / SAP_BS;
    sg.nb3 = g.N3 / SAP_BS;
    sg.nblk = sg.nb0 * sg.nb1 * sg.nb2 * sg.nb3;
    sg.nhalf = sg.nblk / 2;
    return sg;
}

void SapGraphCache::clear() {
    for (auto& e : entries) cudaGraphExecDestroy(e.exec);
    entries.clear();
}

void SapGraphCache::release() {
    clear();
    if (cap) cudaStreamDestroy(cap);
    cap = nullptr;
}

namespace {

void launch_batch_set(const SapJob* d_jobs, int njobs, int ctas, bool copy, int ncy, int nmr, size_t smem,
                      cudaStream_t st) {
    for (int cy = 0; cy < ncy; ++cy)
        for (int colour = 0; colour < 2; ++colour) {
            const int fl = split_flags(cy, colour, ncy);
            if (copy) k_sap_block_batch<true><<<ctas, SPLIT_THREADS, smem, st>>>(d_jobs, njobs, colour, fl, nmr);
            else k_sap_block_batch<false><<<ctas, SPLIT_THREADS, smem, st>>>(d_jobs, njobs, colour, fl, nmr);
        }
}

// the executable graph of this launch set, captured on first use
int batch_graph(SapGraphCache& gc, const SapJob* d_jobs, int njobs, int ctas, bool copy, int ncy, int nmr, size_t smem,
                cudaGraphExec_t* out) {
    ++gc.tick;
    for (auto& e : gc.entries)
        if (e.table == d_jobs && e.njobs == njobs && e.ctas == ctas && e.copy == copy && e.ncy == ncy && e.nmr == nmr) {
            e.last = gc.tick;
            ++gc.replays;
            *out = e.exec;
            return QXD_OK;
        }
    if (!gc.cap) QXD_CUDA(cudaStreamCreateWithFlags(&gc.cap, cudaStreamNonBlocking));
    QXD_CUDA(cudaStreamBeginCapture(gc.cap, cudaStreamCaptureModeThreadLocal));
    launch_batch_set(d_jobs, njobs, ctas, copy, ncy, nmr, smem, gc.cap);
    const cudaError_t le = cudaGetLastError();
    cudaGraph_t graph = nullptr;
    const cudaError_t ce = cudaStreamEndCapture(gc.cap, &graph);  // always ends the capture
    if (le != cudaSuccess || ce != cudaSuccess) {
        if (graph) cudaGraphDestroy(graph);
        return cuda_fail(le != cudaSuccess ? le : ce, "k_sap_block_batch graph capture");
    }
    cudaGraphExec_t exec = nullptr;
    const cudaError_t ie = cudaGraphInstantiate(&exec, graph, 0);
    cudaGraphDestroy(graph);
    if (ie != cudaSuccess) return cuda_fail(ie, "cudaGraphInstantiate (SAP launch set)");
    if ((int)gc.entries.size() >= SapGraphCache::kMax) {
        auto lru = std::min_element(gc.entries.begin(), gc.entries.end(),
                                    [](const SapGraphCache::Entry& a, const SapGraphCache::Entry& b) { return a.last < b.last; });
        cudaGraphExecDestroy(lru->exec);
        gc.entries.erase(lru);
    }
    gc.entries.push_back(SapGraphCache::Entry{d_jobs, njobs, ctas, ncy, nmr, copy, exec, gc.tick});
    ++gc.captures;
    *out = exec;
    return QXD_OK;
}

}  // namespace

int sap_apply_batch(std::vector<SapJob>& jobs, SapJob* d_jobs, int ncy, int nmr, cudaStream_t st,
                    SapGraphCache* graphs) {
    if (jobs.empty()) return QXD_OK;
    int ctas = 0;
    bool copy = true;  // every operator has its block-by-block copy
    for (auto& J : jobs) {  // the first visit of each colour writes psi without reading it
        J.cta_begin = ctas;
        ctas += J.sg.nhalf;
        copy = copy && J.plan.links;
    }
    QXD_CUDA(cudaMemcpyAsync(d_jobs, jobs.data(), jobs.size() * sizeof(SapJob), cudaMemcpyHostToDevice, st));
    const size_t smem = sap_smem_bytes<float>();
    int rc = copy ? split_attrs(k_sap_block_batch<true>, smem) : split_attrs(k_sap_block_batch<false>, smem);
    if (rc) return rc;
    const int njobs = (int)jobs.size();
    if (graphs) {
        cudaGraphExec_t exec = nullptr;
        if ((rc = batch_graph(*graphs, d_jobs, njobs, ctas, copy, ncy, nmr, smem, &exec))) return rc;
        QXD_CUDA(cudaGraphLaunch(exec, st));
        return QXD_OK;
    }
    launch_batch_set(d_jobs, njobs, ctas, copy, ncy, nmr, smem, st);
    QXD_LAUNCHED("k_sap_block_batch");
    return QXD_OK;
}
template int sap_apply<double>(qxd_lattice*, SapWork&, void*, const void*, int, int, cudaStream_t);

}  // namespace qxd

using namespace qxd;

extern "C" int qxd_sap(qxd_lattice* lat, void* out, const void* in, int ncy, int nmr, int flags, void* stream) {
    if (!lat || !out || !in) return fail(QXD_ERR_ARG, "qxd_sap: NULL argument");
    if (flags & ~(0x1 | 0x100)) return fail(QXD_ERR_ARG, "qxd_sap: bad flags (device buffers only)");
    if (ncy < 1 || nmr < 1) return fail(QXD_ERR_ARG, "qxd_sap: ncy and nmr must be >= 1");
    if (out == in) return fail(QXD_ERR_ARG, "qxd_sap: in and out must not overlap");
    if (!qxd::clover_ready(lat)) return fail(QXD_ERR_STATE, "qxd_sap: needs qxd_sw_build first");
    int rc = sap_check(lat);
    if (rc) return rc;
    const int prec = flags & 0x1;
    cudaStream_t st = stream ? (cudaStream_t)stream : lat->stream;
    SapWork w;
    if (flags & QXD_LAYOUT_NATIVE)
        return prec == QXD_FP32 ? sap_apply<float>(lat, w, out, in, ncy, nmr, st)
                                : sap_apply<double>(lat, w, out, in, ncy, nmr, st);
    if ((rc = ensure_scratch(lat))) return rc;
    if ((rc = launch_pack(lat, lat->scratch_in, in, prec, st))) return rc;
    rc = prec == QXD_FP32 ? sap_apply<float>(lat, w, lat->scratch_out, lat->scratch_in, ncy, nmr, st)
                          : sap_apply<double>(lat, w, lat->scratch_out, lat->scratch_in, ncy, nmr, st);
    if (rc) return rc;
    return launch_unpack(lat, out, lat->scratch_out, prec, st);
}

extern "C" int qxd_sap_multi(qxd_lattice* lat, int nrhs, void* const* out, const void* const* in, int ncy, int nmr,
                             void* stream) {
    if (!lat || !out || !in || nrhs < 1) return fail(QXD_ERR_ARG, "qxd_sap_multi: NULL argument or nrhs < 1");
    if (ncy < 1 || nmr < 1) return fail(QXD_ERR_ARG, "qxd_sap_multi: ncy and nmr must be >= 1");
    for (int i = 0; i < nrhs; ++i) {
        if (!out[i] || !in[i]) return fail(QXD_ERR_ARG, "qxd_sap_multi: NULL field");
        for (int j = 0; j < nrhs; ++j)
            if (out[i] == in[j] || (j != i && out[i] == out[j]))
                return fail(QXD_ERR_ARG, "qxd_sap_multi: outputs must differ from each other and from the inputs");
    }
    if (!qxd::clover_ready(lat)) return fail(QXD_ERR_STATE, "qxd_sap_multi: needs qxd_sw_build first");
    int rc = sap_check(lat);
    if (rc) return rc;
    const size_t per = ((size_t)lat->g.V + lat->g.Vh) * SPINOR_F4;  // float4 of one right-hand side's work fields
    if (lat->sap_multi_n < nrhs) {
        if (lat->sap_multi) cudaFree(lat->sap_multi);
        lat->sap_multi = nullptr;
        lat->sap_multi_n = 0;
        const cudaError_t e = cudaMalloc(&lat->sap_multi, per * nrhs * sizeof(float4));
        if (e != cudaSuccess) {
            lat->sap_multi = nullptr;
            return cuda_fail(e, "qxd_sap_multi: cudaMalloc(work fields)");
        }
        lat->sap_multi_n = nrhs;
    }
    std::vector<float4*> works(nrhs);
    for (int i = 0; i < nrhs; ++i) works[i] = lat->sap_multi + per * i;
    cudaStream_t st = stream ? (cudaStream_t)stream : lat->stream;
    return sap_apply_multi(lat, nrhs, out, in, works.data(), ncy, nmr, st);
}

extern "C" int qxd_set_sap_copy(qxd_lattice* lat, int enable) {
    if (!lat) return fail(QXD_ERR_ARG, "qxd_set_sap_copy: lat is NULL");
    if (lat->sap_plan) return fail(QXD_ERR_STATE, "qxd_set_sap_copy: the lattice has its copy already");
    lat->sap_copy_wanted = enable != 0;
    return QXD_OK;
}
