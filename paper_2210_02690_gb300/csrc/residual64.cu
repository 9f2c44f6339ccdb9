// The FP64 operator without a matrix: J x and b - J x in 3D.
#include "residual.cuh"

#include <cstddef>

namespace stg {

// GB300's FP64 pipe bounds both forms.  In 3D the assembled one takes ((k+1) d)^2 multiply-adds a node pair (and 16.8 GB
// for 48^3, k = 1), this one 1300 to 1800 per cell and component: step of 48^3, k = 1 250 -> 245 ms, of 24^3, k = 2
// 126 -> 120 ms.  In 2D it was the slower one (256^2 k = 3 43 -> 48 ms, 352 x 64 order 4 32 -> 35 ms).
bool operator_mf_preferred(const Geom& g) { return g.dim == 3; }

void operator_coef(const Geom& g, const TimeData& td, const AsmCoef& cf, void* dst, cudaStream_t st) {
  upload_coefficients<3, 3, double>(g, td, cf, dst, st);
}

void operator_set_newton(void* coef, bool newton, cudaStream_t st) {
  STG_CUDA_OK(cudaMemsetAsync((char*)coef + offsetof(MfCoef<double>, newton), newton ? 1 : 0, sizeof(int), st));
}

void operator_mf(const Geom& g, const void* coef, const double* w, const double* x, const double* b, double* scratch,
                 double* out, cudaStream_t st) {
  if (g.dim != 3) throw Error{STG_EINVAL, "no matrix-free FP64 operator in 2D"};
  switch (g.nt) {
    case 1: return run3d<1, double>(g, coef, w, x, b, scratch, out, st);
    case 2: return run3d<2, double>(g, coef, w, x, b, scratch, out, st);
    default: return run3d<3, double>(g, coef, w, x, b, scratch, out, st);
  }
}

}  // namespace stg
