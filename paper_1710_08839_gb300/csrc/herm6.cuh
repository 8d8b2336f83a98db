// LDL^H factorisation of the packed Hermitian 6x6 clover blocks (real diagonal,
// strictly lower part row major), in registers, FP64.
#pragma once

#include "qxd_internal.cuh"

namespace qxd {

__device__ __forceinline__ int lidx6(int i, int j) { return i * (i - 1) / 2 + j; }  // i > j

// row sums of |re| + |im|, an upper bound of the block's row-sum norm (no square roots)
__device__ __forceinline__ double herm6_bound(const double d[6], const cplx<double> l[15]) {
    double nrm = 0.0;
#pragma unroll
    for (int i = 0; i < 6; ++i) {
        double rs = fabs(d[i]);
#pragma unroll
        for (int j = 0; j < 6; ++j)
            if (j != i) {
                const cplx<double> z = i > j ? l[lidx6(i, j)] : l[lidx6(j, i)];
                rs += fabs(z.re) + fabs(z.im);
            }
        nrm = fmax(nrm, rs);
    }
    return nrm;
}

// A = L D L^H (L unit lower triangular), iD = 1 / D; false when a pivot falls
// below `least` in size or is not a number
__device__ __forceinline__ bool ldl6(const double a_d[6], const cplx<double> a_l[15], double least, double D[6],
                                     double iD[6], cplx<double> L[15]) {
#pragma unroll
    for (int j = 0; j < 6; ++j) {
        double dj = a_d[j];
        cplx<double> DL[5];  // D_k conj(L_jk)
#pragma unroll
        for (int k = 0; k < j; ++k) {
            const cplx<double> l = L[lidx6(j, k)];
            DL[k] = mk(D[k] * l.re, -D[k] * l.im);
            dj = fma(-DL[k].re, l.re, fma(DL[k].im, l.im, dj));
        }
        if (!(fabs(dj) >= least)) return false;
        D[j] = dj;
        iD[j] = 1.0 / dj;
#pragma unroll
        for (int i = j + 1; i < 6; ++i) {
            cplx<double> v = a_l[lidx6(i, j)];
#pragma unroll
            for (int k = 0; k < j; ++k) v = mad(-L[lidx6(i, k)], DL[k], v);
            L[lidx6(i, j)] = iD[j] * v;
        }
    }
    return true;
}

}  // namespace qxd
