// Full-lattice application of D (Sec. 2.3, Eqs. (16)-(21)):
//   (D psi)(x) = M(x) psi(x) - 1/2 sum_mu [ (1 - g_mu) W(x,mu) psi(x+mu)
//                                  + (1 + g_mu) W(x-mu,mu)^+ psi(x-mu) ],
//   W(x,mu) = U(x,mu) z(x,mu)^qhat,  M(x) = (4 + m0) + dDsw(x),
// which is Eqs. (18)-(20) expanded (the diagonal 4 of Dw moved into M).
// FP32: one thread per site; spin projection to half spinors before the colour
// multiplication (the projectors commute with W). FP32: links as two rows
// plus the U(1) angle, hops software-pipelined (k_dirac32); FP64: compound
// links, a site's work split over threads (dirac64.cu).
// Both parities in one sweep, in the tiled order of sweep_coords so
// neighbour data is reused from L2.
//
// Chiral basis, psi = (psi0, psi1 | psi2, psi3):
//   (1 -+ g0): h = (psi0 +- psi2, psi1 +- psi3),   lower = (+-h0, +-h1)
//   (1 -+ g1): h = (psi0 +- i psi3, psi1 +- i psi2), lower = (-+i h1, -+i h0)
//   (1 -+ g2): h = (psi0 +- psi3, psi1 -+ psi2),   lower = (-+h1, +-h0)
//   (1 -+ g3): h = (psi0 +- i psi2, psi1 -+ i psi3), lower = (-+i h0, +-i h1)
#include <map>
#include <mutex>
#include <string>
#include <tuple>
#include <vector>

#include "dirac64.cuh"
#include "dirac_common.cuh"
#include "tune.cuh"

namespace qxd {

namespace {

// Both kernels apply D on the x0 planes [x0b, x0b + nx0) (all of them for
// x0b = 0, nx0 = N0), nsites = nx0 N1 N2 N3 threads.
// FP32: the pipelined hop order of hops_pipelined (128 registers)
template <bool QNZ>
__global__ void __launch_bounds__(DW_THREADS, DW_PP_MIN_BLOCKS)
    k_dirac32(Geom g, Fields<float> f, SpRefOut<float> out, float q, int x0b, int nx0, int nsites) {
    const int tau = blockIdx.x * blockDim.x + threadIdx.x;
    if (tau >= nsites) return;
    int x0, x1, x2, x3;
    sweep_coords_slab(g, x0b, nx0, tau, x0, x1, x2, x3);
    const int p = (x0 + x1 + x2 + x3) & 1;
    const int lex = lex_index(g, x0, x1, x2, x3);
    const int s = native_index(g, lex, p);
    int nb[8];
    neighbours8(g, x0, x1, x2, x3, 1 - p, nb);
    cplx<float> acc[12], v[12];
    hops_pipelined<QNZ>(f, f.psi, g.V, 0, g.V, s, nb, q, acc);
#pragma unroll
    for (int i = 0; i < 12; ++i) acc[i] = HopScale<float>::value * acc[i];
    load_spinor(f.psi, g.V, s, v);
    clover_mul<true, true>(f.C, g.V, s, v, acc);
    store_spinor_cs(out.p + out.at(lex, s), out.stride, 0, acc);
}

// FP32, the plain hop order (80 registers, 6 blocks per SM)
template <bool QNZ>
__global__ void __launch_bounds__(DW_THREADS, DwMinBlocks<float>::value)
    k_dirac(Geom g, Fields<float> f, SpRefOut<float> out, float q, int x0b, int nx0, int nsites) {
    const int tau = blockIdx.x * blockDim.x + threadIdx.x;
    if (tau >= nsites) return;
    int x0, x1, x2, x3;
    sweep_coords_slab(g, x0b, nx0, tau, x0, x1, x2, x3);
    const int p = (x0 + x1 + x2 + x3) & 1;
    const int lex = lex_index(g, x0, x1, x2, x3);
    const int s = native_index(g, lex, p);
    cplx<float> acc[12], v[12];
    dirac_hops<float, QNZ>(g, f, f.psi, g.V, 0, q, x0, x1, x2, x3, s, 1 - p, acc);
#pragma unroll
    for (int i = 0; i < 12; ++i) acc[i] = HopScale<float>::value * acc[i];
    load_spinor(f.psi, g.V, s, v);
    clover_mul<true, true>(f.C, g.V, s, v, acc);
    store_spinor_cs(out.p + out.at(lex, s), out.stride, 0, acc);
}

// D with launch shape sh (hop order, threads per block, sweep window) on the
// x0 planes [x0b, x0b + nx0); lex: lexicographic output, and in FP64 input
int launch_dirac_shape(qxd_lattice* lat, void* out, const void* in, int prec, const DwShape& sh, cudaStream_t st,
                       int x0b = 0, int nx0 = -1, bool lex = false) {
    Geom g = lat->g;
    g.R = sh.rows;
    if (nx0 < 0) nx0 = g.N0;
    const int n = nx0 * g.N1 * g.N2 * g.N3;
    const int blocks = (n + sh.threads - 1) / sh.threads;
    const bool qnz = lat->qhat != 0;
    if (prec == QXD_FP32) {
        const Fields<float> f{(const float4*)in, lat->U32, lat->A32, lat->C32};
        const SpRefOut<float> o = lex ? lex_out<float>(out) : full_out<float>(out, g.V);
        if (sh.pipelined) {
            if (qnz) k_dirac32<true><<<blocks, sh.threads, 0, st>>>(g, f, o, (float)lat->qhat, x0b, nx0, n);
            else k_dirac32<false><<<blocks, sh.threads, 0, st>>>(g, f, o, 0.f, x0b, nx0, n);
        } else {
            if (qnz) k_dirac<true><<<blocks, sh.threads, 0, st>>>(g, f, o, (float)lat->qhat, x0b, nx0, n);
            else k_dirac<false><<<blocks, sh.threads, 0, st>>>(g, f, o, 0.f, x0b, nx0, n);
        }
    } else {
        return launch_dirac64(lat, lex ? lex_out<double>(out) : full_out<double>(out, g.V),
                              lex ? lex_ref<double>(in) : full_ref<double>(in, g.V), sh.threads, sh.rows, x0b, nx0, st);
    }
    QXD_LAUNCHED("k_dirac");
    return QXD_OK;
}

// candidate sweep windows: divisors R of N2 with a window of N1 R N3 sites
// between 16K and 256K, the default (largest window <= 64K) and its nearest
// neighbours among them
std::vector<int> window_candidates(const Geom& g) {
    std::vector<int> ok;
    for (int R = 1; R <= g.N2; ++R) {
        const long long w = (long long)g.N1 * R * g.N3;
        if (g.N2 % R == 0 && w >= 16384 && w <= 262144) ok.push_back(R);
    }
    std::vector<int> out;
    int at = -1;
    for (int i = 0; i < (int)ok.size(); ++i)
        if (ok[i] == g.R) at = i;
    if (at < 0) return {g.R};
    for (int i = std::max(0, at - 1); i <= std::min((int)ok.size() - 1, at + 1); ++i) out.push_back(ok[i]);
    return out;
}

// time every candidate shape on this call's input (3 launches each after
// one untimed launch) and return the fastest
int tune_dirac(qxd_lattice* lat, void* out, const void* in, int prec, bool lex, cudaStream_t st, DwShape* best) {
    std::vector<DwShape> cand;
    const std::vector<int> rows = window_candidates(lat->g);
    for (int pl = (prec == QXD_FP32 ? 1 : 0); pl >= 0; --pl)
        for (int th : {128, 64})
            for (int R : rows) cand.push_back(DwShape{pl, th, R, 0.f});
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    QXD_CUDA(cudaEventCreate(&e0));
    if (cudaEventCreate(&e1) != cudaSuccess) {
        cudaEventDestroy(e0);
        return fail(QXD_ERR_CUDA, "autotune: cudaEventCreate");
    }
    int rc = QXD_OK;
    best->ms = 0.f;
    for (DwShape& c : cand) {
        if ((rc = launch_dirac_shape(lat, out, in, prec, c, st, 0, -1, lex))) break;
        cudaEventRecord(e0, st);
        for (int rep = 0; rep < 3 && !rc; ++rep) rc = launch_dirac_shape(lat, out, in, prec, c, st, 0, -1, lex);
        if (rc) break;
        cudaEventRecord(e1, st);
        const cudaError_t e = cudaEventSynchronize(e1);
        if (e != cudaSuccess) {
            rc = cuda_fail(e, "autotune: cudaEventSynchronize");
            break;
        }
        float ms = 0.f;
        cudaEventElapsedTime(&ms, e0, e1);
        c.ms = ms / 3;
        if (best->ms == 0.f || c.ms < best->ms) *best = c;
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    return rc;
}

}  // namespace

namespace {

bool capturing(cudaStream_t st) {
    cudaStreamCaptureStatus s = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(st, &s) == cudaSuccess) return s != cudaStreamCaptureStatusNone;
    cudaGetLastError();  // the legacy stream beside a capture elsewhere: nothing can be timed there either
    return true;
}

int dirac_full(qxd_lattice* lat, void* out, const void* in, int prec, bool lex, cudaStream_t st) {
    const DwKey key = dw_key(lat, prec);
    const bool tune = autotune_enabled();
    DwShape sh;
    bool timed_lex = false;
    // a shape timed on lexicographic fields is not kept for native ones, which
    // the solvers apply D to, unless the call cannot be timed
    if (!dw_shape_get(key, &sh, &timed_lex) || (timed_lex && !lex && tune && !capturing(st))) {
        if (tune) {
            int rc = tune_dirac(lat, out, in, prec, lex, st, &sh);
            if (rc) return rc;
        } else {
            sh = dw_default_shape(lat, prec);
        }
        dw_shape_put(key, sh, tune ? "tuned" : "default", tune && lex);
    }
    return launch_dirac_shape(lat, out, in, prec, sh, st, 0, -1, lex);
}

}  // namespace

int launch_dirac(qxd_lattice* lat, void* out, const void* in, int prec, cudaStream_t st) {
    return dirac_full(lat, out, in, prec, false, st);
}

// FP64, bound by arithmetic, reads and writes the caller's layout. FP32 gathers
// each site nine times, which wants the native layout, but writes it once: the
// input is packed (39 us for 1.3M sites), the output stored in place.
int launch_dirac_lex(qxd_lattice* lat, void* out, const void* in, void* nat_in, void* nat_out, int prec,
                     cudaStream_t st) {
    if (prec == QXD_FP64 && aligned16(out) && aligned16(in)) return dirac_full(lat, out, in, prec, true, st);
    int rc = launch_pack(lat, nat_in, in, prec, st);
    if (rc) return rc;
    if (prec == QXD_FP32 && aligned16(out)) return dirac_full(lat, out, nat_in, prec, true, st);
    if ((rc = dirac_full(lat, nat_out, nat_in, prec, false, st))) return rc;
    return launch_unpack(lat, out, nat_out, prec, st);
}

bool dirac_lex_needs_scratch(const void* out, const void* in, int prec) {
    return !(prec == QXD_FP64 && aligned16(out) && aligned16(in));
}

int launch_dirac_planes(qxd_lattice* lat, void* out, const void* in, int prec, int x0b, int nx0, cudaStream_t st) {
    DwShape sh;
    if (!dw_shape_get(dw_key(lat, prec), &sh)) sh = dw_default_shape(lat, prec);
    return launch_dirac_shape(lat, out, in, prec, sh, st, x0b, nx0);
}

}  // namespace qxd
