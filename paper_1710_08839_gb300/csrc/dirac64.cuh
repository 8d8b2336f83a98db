// FP64 stencil launchers (dirac64.cu).
#pragma once

#include "eo.cuh"

namespace qxd {

using C64 = cplx<double>;

// out = D in on the x0 planes [x0b, x0b + nx0): threads per block, x2 rows per sweep chunk
int launch_dirac64(qxd_lattice* lat, const SpRefOut<double>& out, const SpRef<double>& in, int threads, int rows,
                   int x0b, int nx0, cudaStream_t st);
// an even-odd part (mode as in eo.cuh) on the sites of parity p
int launch_eo64(qxd_lattice* lat, int mode, int p, const SpRef<double>& in, const SpRef<double>& aux,
                const SpRefOut<double>& out, cudaStream_t st);

}  // namespace qxd
