// Even-odd form of D (Sec. 2.4, Eqs. (29)-(30)). D = M + H with M the
// site-diagonal part and H the hopping part, H psi(x) = -1/2 sum_mu [...];
// H connects only sites of opposite parity, so
//   D_ee = M_ee, D_oo = M_oo, D_eo = H_eo, D_oe = H_oe,
//   D_hat = M_ee - H_eo M_oo^-1 H_oe   (on the even sites).
// The kernels below evaluate, for all sites x of one parity p,
//   INV_HOP          out = M^-1 (H psi)
//   CLOVER_AUX_MHOP  out = M aux - H psi
//   AUX_MHOP         out = aux - H psi
//   INV_AUX_MHOP     out = M^-1 (aux - H psi)
//   G5_CLOVER_AUX_MHOP  out = gamma5 (M aux - H psi)
// where psi lives on the other parity; in FP32 here, one thread per site, in
// FP64 in dirac64.cu. Each field is addressed as
// (pointer, stride, offset): element k of the site with native index s is at
// p[k * stride + s - offset], so full-lattice arrays (stride V, offset 0)
// and half-lattice arrays (stride V/2, offset parity * V/2) both work. M^-1 is
// kept and applied on the odd sites only.
#include <string>

#include "dirac_common.cuh"
#include "dirac64.cuh"
#include "eo.cuh"

namespace qxd {

namespace {

template <bool QNZ, int MODE>
__global__ void __launch_bounds__(DW_THREADS, DW_PP_MIN_BLOCKS)
    k_dslash_half(Geom g, int p, Fields<float> f, SpRef<float> in, SpRef<float> aux, SpRefOut<float> out,
                  const float4* __restrict__ Cl, float q) {
    const int tau = blockIdx.x * blockDim.x + threadIdx.x;
    if (tau >= g.Vh) return;
    int x0, x1, x2, x3;
    sweep_coords_parity(g, p, tau, x0, x1, x2, x3);
    const int lex = lex_index(g, x0, x1, x2, x3);
    const int s = native_index(g, lex, p);
    int nb[8];
    neighbours8(g, x0, x1, x2, x3, 1 - p, nb);
    cplx<float> acc[12], w[12];
    hops_pipelined<QNZ>(f, in.p, in.stride, in.off, g.V, s, nb, q, acc);
    constexpr float HS = HopScale<float>::value;  // H psi = HS acc
    if (MODE == EO_INV_HOP) {
        cplx<float> t[12];
#pragma unroll
        for (int i = 0; i < 12; ++i) t[i] = HS * acc[i];
        clover_mul<true>(Cl, g.Vh, s - g.Vh, t, w);
    } else if (MODE == EO_CLOVER_AUX_MHOP || MODE == EO_G5_CLOVER_AUX_MHOP) {
        cplx<float> a[12];
        load_spinor(aux.p + aux.at(lex, s), aux.stride, 0, a);
#pragma unroll
        for (int i = 0; i < 12; ++i) w[i] = (-HS) * acc[i];
        clover_mul<true, true>(Cl, g.V, s, a, w);
        if (MODE == EO_G5_CLOVER_AUX_MHOP) {
            // gamma5 = diag(1, 1, -1, -1): spins 2 and 3 change sign
#pragma unroll
            for (int i = 6; i < 12; ++i) w[i] = -w[i];
        }
    } else if (MODE == EO_AUX_MHOP) {
        load_spinor(aux.p + aux.at(lex, s), aux.stride, 0, w);
#pragma unroll
        for (int i = 0; i < 12; ++i) w[i] = rmad(-HS, acc[i], w[i]);
    } else {  // EO_INV_AUX_MHOP
        cplx<float> a[12];
        load_spinor(aux.p + aux.at(lex, s), aux.stride, 0, a);
#pragma unroll
        for (int i = 0; i < 12; ++i) a[i] = rmad(-HS, acc[i], a[i]);
        clover_mul<true>(Cl, g.Vh, s - g.Vh, a, w);
    }
    store_spinor(out.p + out.at(lex, s), out.stride, 0, w);
    if (out.zero_other) {
#pragma unroll
        for (int i = 0; i < 12; ++i) w[i] = mk(0.f, 0.f);
        store_spinor(out.p + out.at(lex ^ 1, p ? s - g.Vh : s + g.Vh), out.stride, 0, w);
    }
}

// out = M_oo^-1 in on the odd sites
template <typename R>
__global__ void k_minv_odd(Geom g, SpRef<R> in, SpRefOut<R> out, const typename Fields<R>::cvec* __restrict__ Cinv) {
    const int h = blockIdx.x * blockDim.x + threadIdx.x;
    if (h >= g.Vh) return;
    const int s = g.Vh + h;
    int lex = 0;
    if (in.lex || out.lex) {
        int x0, x1, x2, x3;
        native_coords(g, s, x0, x1, x2, x3);
        lex = lex_index(g, x0, x1, x2, x3);
    }
    cplx<R> a[12], w[12];
    load_spinor(in.p + in.at(lex, s), in.stride, 0, a);
    clover_mul<true>(Cinv, g.Vh, h, a, w);
    store_spinor(out.p + out.at(lex, s), out.stride, 0, w);
}

template <bool QNZ>
int launch_mode(qxd_lattice* lat, int mode, int p, const Fields<float>& f, SpRef<float> in, SpRef<float> aux,
                SpRefOut<float> out, const float4* Cl, cudaStream_t st) {
    const Geom& g = lat->g;
    const int blocks = (g.Vh + DW_THREADS - 1) / DW_THREADS;
    const float q = (float)lat->qhat;
    switch (mode) {
        case EO_INV_HOP: k_dslash_half<QNZ, EO_INV_HOP><<<blocks, DW_THREADS, 0, st>>>(g, p, f, in, aux, out, Cl, q); break;
        case EO_CLOVER_AUX_MHOP: k_dslash_half<QNZ, EO_CLOVER_AUX_MHOP><<<blocks, DW_THREADS, 0, st>>>(g, p, f, in, aux, out, Cl, q); break;
        case EO_AUX_MHOP: k_dslash_half<QNZ, EO_AUX_MHOP><<<blocks, DW_THREADS, 0, st>>>(g, p, f, in, aux, out, Cl, q); break;
        case EO_G5_CLOVER_AUX_MHOP: k_dslash_half<QNZ, EO_G5_CLOVER_AUX_MHOP><<<blocks, DW_THREADS, 0, st>>>(g, p, f, in, aux, out, Cl, q); break;
        default: k_dslash_half<QNZ, EO_INV_AUX_MHOP><<<blocks, DW_THREADS, 0, st>>>(g, p, f, in, aux, out, Cl, q); break;
    }
    QXD_LAUNCHED("k_dslash_half");
    return QXD_OK;
}

}  // namespace

template <>
int launch_eo<float>(qxd_lattice* lat, int mode, int p, SpRef<float> in, SpRef<float> aux, SpRefOut<float> out,
                     cudaStream_t st) {
    if (eo_inverse(mode) && p != 1) return fail(QXD_ERR_ARG, "launch_eo: M^-1 is kept on the odd sites");
    const Fields<float> f = fields_of<float>(lat);
    const float4* Cl = clover_of<float>(lat, eo_inverse(mode));
    if (lat->qhat != 0) return launch_mode<true>(lat, mode, p, f, in, aux, out, Cl, st);
    return launch_mode<false>(lat, mode, p, f, in, aux, out, Cl, st);
}
template <>
int launch_eo<double>(qxd_lattice* lat, int mode, int p, SpRef<double> in, SpRef<double> aux, SpRefOut<double> out,
                      cudaStream_t st) {
    if (eo_inverse(mode) && p != 1) return fail(QXD_ERR_ARG, "launch_eo: M^-1 is kept on the odd sites");
    return launch_eo64(lat, mode, p, in, aux, out, st);
}

template <typename R>
int launch_minv_odd(qxd_lattice* lat, SpRef<R> in, SpRefOut<R> out, cudaStream_t st) {
    const Geom& g = lat->g;
    const int blocks = (g.Vh + 255) / 256;
    k_minv_odd<R><<<blocks, 256, 0, st>>>(g, in, out, clover_of<R>(lat, true));
    QXD_LAUNCHED("k_minv_odd");
    return QXD_OK;
}

template int launch_minv_odd<float>(qxd_lattice*, SpRef<float>, SpRefOut<float>, cudaStream_t);
template int launch_minv_odd<double>(qxd_lattice*, SpRef<double>, SpRefOut<double>, cudaStream_t);

// D_hat psi_e = M_ee psi_e - H_eo M_oo^-1 H_oe psi_e; tmp is an odd-parity field
template <typename R>
int apply_dhat(qxd_lattice* lat, SpRefOut<R> out_e, SpRef<R> in_e, SpRefOut<R> tmp_o, cudaStream_t st) {
    int rc = launch_eo<R>(lat, EO_INV_HOP, 1, in_e, SpRef<R>{}, tmp_o, st);
    if (rc) return rc;
    return launch_eo<R>(lat, EO_CLOVER_AUX_MHOP, 0, as_in(tmp_o), in_e, out_e, st);
}
template int apply_dhat<float>(qxd_lattice*, SpRefOut<float>, SpRef<float>, SpRefOut<float>, cudaStream_t);
template int apply_dhat<double>(qxd_lattice*, SpRefOut<double>, SpRef<double>, SpRefOut<double>, cudaStream_t);

template <typename R>
int apply_g5dhat(qxd_lattice* lat, SpRefOut<R> out_e, SpRef<R> in_e, SpRefOut<R> tmp_o, cudaStream_t st) {
    int rc = launch_eo<R>(lat, EO_INV_HOP, 1, in_e, SpRef<R>{}, tmp_o, st);
    if (rc) return rc;
    return launch_eo<R>(lat, EO_G5_CLOVER_AUX_MHOP, 0, as_in(tmp_o), in_e, out_e, st);
}
template int apply_g5dhat<float>(qxd_lattice*, SpRefOut<float>, SpRef<float>, SpRefOut<float>, cudaStream_t);
template int apply_g5dhat<double>(qxd_lattice*, SpRefOut<double>, SpRef<double>, SpRefOut<double>, cudaStream_t);

namespace {

enum { EOAPI_DHAT, EOAPI_PREPARE, EOAPI_RECONSTRUCT };

// in/out are full-lattice arrays, tmp a native one. gin: the field whose even
// sites the hops gather (in for D_hat, x for the reconstruction).
template <typename R>
int eo_parts(qxd_lattice* lat, int what, SpRefOut<R> out, SpRef<R> in, SpRef<R> gin, void* tmp, cudaStream_t st) {
    const int V = lat->g.V;
    int rc;
    if (what == EOAPI_RECONSTRUCT)  // out holds x (even part read); in holds b
        return launch_eo<R>(lat, EO_INV_AUX_MHOP, 1, gin, in, out, st);
    out.zero_other = 1;  // the odd sites of out
    if (what == EOAPI_DHAT) {  // tmp (odd half of a full array) holds M_oo^-1 H_oe in_e
        const SpRefOut<R> t = full_out<R>(tmp, V);
        if ((rc = launch_eo<R>(lat, EO_INV_HOP, 1, gin, SpRef<R>{}, t, st))) return rc;
        return launch_eo<R>(lat, EO_CLOVER_AUX_MHOP, 0, as_in(t), in, out, st);
    }
    if ((rc = launch_minv_odd<R>(lat, in, full_out<R>(tmp, V), st))) return rc;
    return launch_eo<R>(lat, EO_AUX_MHOP, 0, full_ref<R>(tmp, V), in, out, st);
}

template <typename R>
int eo_native(qxd_lattice* lat, int what, void* out, const void* in, void* tmp, cudaStream_t st) {
    const SpRefOut<R> o = full_out<R>(out, lat->g.V);
    const SpRef<R> i = full_ref<R>(in, lat->g.V);
    return eo_parts<R>(lat, what, o, i, what == EOAPI_RECONSTRUCT ? as_in(o) : i, tmp, st);
}

// caller's lexicographic layout read and written in place. FP32: the field
// that the hops gather is packed first (its even sites), each site of which is
// read eight times; everything else is read or written once.
template <typename R>
int eo_lex(qxd_lattice* lat, int what, void* out, const void* in, cudaStream_t st) {
    const SpRefOut<R> o = lex_out<R>(out);
    const SpRef<R> i = lex_ref<R>(in);
    SpRef<R> gin = what == EOAPI_RECONSTRUCT ? as_in(o) : i;
    if (sizeof(R) == 4 && what != EOAPI_PREPARE) {
        const int rc = launch_pack_even(lat, lat->scratch_in, gin.p, QXD_FP32, st);
        if (rc) return rc;
        gin = full_ref<R>(lat->scratch_in, lat->g.V);
    }
    return eo_parts<R>(lat, what, o, i, gin, lat->scratch_lex, st);
}

int eo_api(qxd_lattice* lat, int what, void* out, const void* in, int flags, void* stream, const char* name) {
    if (!lat || !out || !in) return fail(QXD_ERR_ARG, std::string(name) + ": NULL argument");
    if (flags & ~(0x1 | 0x100)) return fail(QXD_ERR_ARG, std::string(name) + ": bad flags (device buffers only)");
    if (what != EOAPI_RECONSTRUCT && out == in)
        return fail(QXD_ERR_ARG, std::string(name) + ": in and out must not overlap");
    if (!qxd::clover_ready(lat)) return fail(QXD_ERR_STATE, std::string(name) + ": needs qxd_sw_build first");
    const int prec = flags & 0x1;
    cudaStream_t st = stream ? (cudaStream_t)stream : lat->stream;
    int rc = ensure_scratch(lat);
    if (rc) return rc;
    if (flags & QXD_LAYOUT_NATIVE)
        return prec == QXD_FP32 ? eo_native<float>(lat, what, out, in, lat->scratch_lex, st)
                                : eo_native<double>(lat, what, out, in, lat->scratch_lex, st);
    if (aligned16(in) && aligned16(out))
        return prec == QXD_FP32 ? eo_lex<float>(lat, what, out, in, st) : eo_lex<double>(lat, what, out, in, st);
    if ((rc = launch_pack(lat, lat->scratch_in, in, prec, st))) return rc;
    if (what == EOAPI_RECONSTRUCT && (rc = launch_pack(lat, lat->scratch_out, out, prec, st))) return rc;
    rc = prec == QXD_FP32 ? eo_native<float>(lat, what, lat->scratch_out, lat->scratch_in, lat->scratch_lex, st)
                          : eo_native<double>(lat, what, lat->scratch_out, lat->scratch_in, lat->scratch_lex, st);
    if (rc) return rc;
    return launch_unpack(lat, out, lat->scratch_out, prec, st);
}

}  // namespace

}  // namespace qxd

extern "C" {

int qxd_Dhat(qxd_lattice* lat, void* out, const void* in, int flags, void* stream) {
    return qxd::eo_api(lat, qxd::EOAPI_DHAT, out, in, flags, stream, "qxd_Dhat");
}

int qxd_eo_prepare(qxd_lattice* lat, void* out, const void* b, int flags, void* stream) {
    return qxd::eo_api(lat, qxd::EOAPI_PREPARE, out, b, flags, stream, "qxd_eo_prepare");
}

int qxd_eo_reconstruct(qxd_lattice* lat, void* x, const void* b, int flags, void* stream) {
    return qxd::eo_api(lat, qxd::EOAPI_RECONSTRUCT, x, b, flags, stream, "qxd_eo_reconstruct");
}

}  // extern "C"
