// Even-odd operator launchers and strided spinor references.
#pragma once

#include "dirac_common.cuh"

namespace qxd {

enum { EO_INV_HOP = 1, EO_CLOVER_AUX_MHOP = 2, EO_AUX_MHOP = 3, EO_INV_AUX_MHOP = 4,
       EO_G5_CLOVER_AUX_MHOP = 5 };

// spinor field reference: element k of a site at p[at(lexicographic index,
// native index) + k * stride]: native fields at p[k * stride + s - off],
// lexicographic ones (lex = elements per site, stride 1) at p[l * lex + k]
template <typename R>
struct SpRef {
    const typename Fields<R>::vec* p = nullptr;
    int stride = 0;
    int off = 0;
    int lex = 0;
    __device__ __forceinline__ size_t at(int l, int s) const { return lex ? (size_t)l * lex : (size_t)(s - off); }
};
// zero_other: the even-odd kernels also set the other site of each pair
// (lexicographic indices 2h and 2h + 1: one of each parity) to zero
template <typename R>
struct SpRefOut {
    typename Fields<R>::vec* p = nullptr;
    int stride = 0;
    int off = 0;
    int lex = 0;
    int zero_other = 0;
    __device__ __forceinline__ size_t at(int l, int s) const { return lex ? (size_t)l * lex : (size_t)(s - off); }
};
template <typename R>
inline SpRef<R> as_in(SpRefOut<R> o) {
    return SpRef<R>{o.p, o.stride, o.off, o.lex};
}
// full-lattice native array
template <typename R>
inline SpRef<R> full_ref(const void* p, int V) {
    return SpRef<R>{(const typename Fields<R>::vec*)p, V, 0};
}
template <typename R>
inline SpRefOut<R> full_out(void* p, int V) {
    return SpRefOut<R>{(typename Fields<R>::vec*)p, V, 0};
}
// full-lattice lexicographic array
template <typename R>
inline SpRef<R> lex_ref(const void* p) {
    return SpRef<R>{(const typename Fields<R>::vec*)p, 1, 0, sizeof(R) == 4 ? SPINOR_F4 : SPINOR_D2};
}
template <typename R>
inline SpRefOut<R> lex_out(void* p) {
    return SpRefOut<R>{(typename Fields<R>::vec*)p, 1, 0, sizeof(R) == 4 ? SPINOR_F4 : SPINOR_D2};
}
// the vector loads and stores of lexicographic fields need 16-byte alignment
inline bool aligned16(const void* p) { return ((uintptr_t)p & 15) == 0; }
// half-lattice native array holding the sites of parity par
template <typename R>
inline SpRef<R> half_ref(const void* p, int Vh, int par) {
    return SpRef<R>{(const typename Fields<R>::vec*)p, Vh, par * Vh};
}
template <typename R>
inline SpRefOut<R> half_out(void* p, int Vh, int par) {
    return SpRefOut<R>{(typename Fields<R>::vec*)p, Vh, par * Vh};
}

template <typename R>
Fields<R> fields_of(qxd_lattice* lat);
template <>
inline Fields<float> fields_of<float>(qxd_lattice* lat) {
    return Fields<float>{nullptr, lat->U32, lat->A32, lat->C32};
}
template <>
inline Fields<double> fields_of<double>(qxd_lattice* lat) {
    return Fields<double>{nullptr, lat->W64, lat->C64};
}
template <typename R>
const typename Fields<R>::cvec* clover_of(qxd_lattice* lat, bool inverse);
template <>
inline const float4* clover_of<float>(qxd_lattice* lat, bool inverse) {
    return inverse ? lat->Cinv32 : lat->C32;
}
template <>
inline const double* clover_of<double>(qxd_lattice* lat, bool inverse) {
    return inverse ? lat->Cinv64 : lat->C64;
}

// the modes with M^-1 are for the odd sites, p = 1 (QXD_ERR_ARG otherwise)
inline bool eo_inverse(int mode) { return mode == EO_INV_HOP || mode == EO_INV_AUX_MHOP; }
template <typename R>
int launch_eo(qxd_lattice* lat, int mode, int p, SpRef<R> in, SpRef<R> aux, SpRefOut<R> out, cudaStream_t st);
template <typename R>
int launch_minv_odd(qxd_lattice* lat, SpRef<R> in, SpRefOut<R> out, cudaStream_t st);
template <typename R>
int apply_dhat(qxd_lattice* lat, SpRefOut<R> out_e, SpRef<R> in_e, SpRefOut<R> tmp_o, cudaStream_t st);
// gamma5 D_hat psi_e (Hermitian: D_hat^dag = gamma5 D_hat gamma5)
template <typename R>
int apply_g5dhat(qxd_lattice* lat, SpRefOut<R> out_e, SpRef<R> in_e, SpRefOut<R> tmp_o, cudaStream_t st);

}  // namespace qxd
