// Spinor layout conversion: lexicographic [site][spin][colour][re, im] <->
// native structure of arrays (even sites, then odd). The two sites of
// lexicographic indices 2h and 2h + 1 are one of each parity and both have
// native index h within it, so a tile of consecutive pairs is one contiguous
// range of the lexicographic field and, per component and parity, one
// contiguous range of the native field: a thread block copies the tile through
// shared memory with 16-byte accesses that are contiguous on both sides. Bound
// by memory: reads and writes every field once. (One thread per site, with 4-
// or 8-byte accesses 96 or 192 bytes apart, took 68 us to pack and 176 us to
// unpack an FP32 field of 1.3M sites, 255 MB in all; the tiles take 39 us each way, 6.5 TB/s.)
#include "dirac_common.cuh"
#include "eo.cuh"

namespace qxd {

namespace {

constexpr int LAYOUT_THREADS = 256;
constexpr int TILE_ELEMS = 768;  // 16-byte elements per tile: 64 pairs of FP32 sites, 32 of FP64

// parity of the site of lexicographic index 2h
__device__ __forceinline__ int pair_parity(const Geom& g, int h) {
    int r = 2 * h;
    const int x3 = r % g.N3;
    r /= g.N3;
    const int x2 = r % g.N2;
    r /= g.N2;
    return (x3 + x2 + r % g.N1 + r / g.N1) & 1;
}

enum { UNPACK = 0, PACK_ALL = 1, PACK_EVEN = 2 };  // PACK_EVEN: the even sites only

// T: float4 (C = 6 per site) or double2 (C = 12); pairs [h0, h1). A pair takes
// 2 C + 1 elements of shared memory, which spreads the strided side over the
// banks.
template <typename T, int C, int MODE>
__global__ void __launch_bounds__(LAYOUT_THREADS) k_layout(Geom g, const T* __restrict__ in, T* __restrict__ out, int h0,
                                                           int h1) {
    constexpr int PAIRS = TILE_ELEMS / (2 * C);
    constexpr bool PACK = MODE != UNPACK;
    __shared__ T sm[PAIRS * (2 * C + 1)];
    __shared__ int par0[PAIRS];
    const size_t V = g.V;
    for (int hb = h0 + blockIdx.x * PAIRS; hb < h1; hb += gridDim.x * PAIRS) {
        const int np = min(PAIRS, h1 - hb);
        if (threadIdx.x < np) par0[threadIdx.x] = pair_parity(g, hb + threadIdx.x);
        if (MODE != PACK_ALL) __syncthreads();
#pragma unroll
        for (int i = 0; i < TILE_ELEMS / LAYOUT_THREADS; ++i) {
            const int e = threadIdx.x + i * LAYOUT_THREADS;
            if (PACK) {
                const int j = e / (2 * C), k = e - j * 2 * C;
                if (j < np && (MODE == PACK_ALL || (k >= C) == (par0[j] != 0)))
                    sm[j * (2 * C + 1) + k] = __ldcs(&in[(size_t)hb * 2 * C + e]);
            } else {
                const int j = e % PAIRS, q = e / PAIRS, k = q % C, p = q / C;  // component k of parity p
                if (j < np) sm[j * (2 * C + 1) + (p ^ par0[j]) * C + k] = __ldcs(&in[k * V + (size_t)p * g.Vh + hb + j]);
            }
        }
        __syncthreads();
#pragma unroll
        for (int i = 0; i < TILE_ELEMS / LAYOUT_THREADS; ++i) {
            const int e = threadIdx.x + i * LAYOUT_THREADS;
            if (PACK) {
                const int j = e % PAIRS, q = e / PAIRS, k = q % C, p = q / C;
                if (j < np && (MODE == PACK_ALL || p == 0)) out[k * V + (size_t)p * g.Vh + hb + j] = sm[j * (2 * C + 1) + (p ^ par0[j]) * C + k];
            } else {
                const int j = e / (2 * C), k = e - j * 2 * C;
                if (j < np) out[(size_t)hb * 2 * C + e] = sm[j * (2 * C + 1) + k];
            }
        }
        __syncthreads();
    }
}

// lexicographic fields that are not 16-byte aligned: one thread per site
template <typename R, bool PACK>
__global__ void k_layout_site(Geom g, R* __restrict__ lex, typename Fields<R>::vec* __restrict__ nat, int s0, int s1) {
    const int l = s0 + blockIdx.x * blockDim.x + threadIdx.x;
    if (l >= s1) return;
    const int s = native_index(g, l, pair_parity(g, l >> 1) ^ (l & 1));
    R* p = lex + (size_t)l * 24;
    cplx<R> v[12];
    if (PACK) {
#pragma unroll
        for (int i = 0; i < 12; ++i) v[i] = mk(p[2 * i], p[2 * i + 1]);
        store_spinor(nat, g.V, s, v);
    } else {
        load_spinor(nat, g.V, s, v);
#pragma unroll
        for (int i = 0; i < 12; ++i) {
            p[2 * i] = v[i].re;
            p[2 * i + 1] = v[i].im;
        }
    }
}

template <typename R, int MODE>
int convert(qxd_lattice* lat, void* nat, void* lex, size_t s0, size_t ns, unsigned max_blocks, cudaStream_t st) {
    using T = typename Fields<R>::vec;
    constexpr int C = sizeof(R) == 4 ? SPINOR_F4 : SPINOR_D2;
    constexpr bool PACK = MODE != UNPACK;
    const Geom& g = lat->g;
    if (!aligned16(lex)) {
        k_layout_site<R, PACK><<<(unsigned)((ns + 255) / 256), 256, 0, st>>>(g, (R*)lex, (T*)nat, (int)s0, (int)(s0 + ns));
        QXD_LAUNCHED("k_layout_site");
        return QXD_OK;
    }
    constexpr int PAIRS = TILE_ELEMS / (2 * C);
    const int h0 = (int)(s0 / 2), h1 = (int)((s0 + ns) / 2);
    unsigned blocks = (unsigned)((h1 - h0 + PAIRS - 1) / PAIRS);
    if (blocks > max_blocks) blocks = max_blocks;
    k_layout<T, C, MODE><<<blocks, LAYOUT_THREADS, 0, st>>>(g, (const T*)(PACK ? lex : nat), (T*)(PACK ? nat : lex), h0, h1);
    QXD_LAUNCHED("k_layout");
    return QXD_OK;
}

}  // namespace

int launch_pack_sites(qxd_lattice* lat, void* nat, const void* lex, int prec, size_t s0, size_t ns, unsigned max_blocks,
                      cudaStream_t st) {
    void* l = const_cast<void*>(lex);
    return prec == QXD_FP32 ? convert<float, PACK_ALL>(lat, nat, l, s0, ns, max_blocks, st)
                            : convert<double, PACK_ALL>(lat, nat, l, s0, ns, max_blocks, st);
}

int launch_unpack_sites(qxd_lattice* lat, void* lex, const void* nat, int prec, size_t s0, size_t ns,
                        unsigned max_blocks, cudaStream_t st) {
    void* n = const_cast<void*>(nat);
    return prec == QXD_FP32 ? convert<float, UNPACK>(lat, n, lex, s0, ns, max_blocks, st)
                            : convert<double, UNPACK>(lat, n, lex, s0, ns, max_blocks, st);
}

int launch_pack(qxd_lattice* lat, void* nat, const void* lex, int prec, cudaStream_t st) {
    return launch_pack_sites(lat, nat, lex, prec, 0, (size_t)lat->g.V, ~0u, st);
}

int launch_pack_even(qxd_lattice* lat, void* nat, const void* lex, int prec, cudaStream_t st) {
    void* l = const_cast<void*>(lex);
    return prec == QXD_FP32 ? convert<float, PACK_EVEN>(lat, nat, l, 0, (size_t)lat->g.V, ~0u, st)
                            : convert<double, PACK_EVEN>(lat, nat, l, 0, (size_t)lat->g.V, ~0u, st);
}

int launch_unpack(qxd_lattice* lat, void* lex, const void* nat, int prec, cudaStream_t st) {
    return launch_unpack_sites(lat, lex, nat, prec, 0, (size_t)lat->g.V, ~0u, st);
}

}  // namespace qxd
