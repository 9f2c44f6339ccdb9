// The FP64 operator without a matrix: J x and b - J x in 3D.
#include "residual.cuh"

#include <cstddef>

namespace stg {

// GB300's FP64 pipe bounds both forms.  The assembled one leaves out the structural zeros of a block (k + 3 of 3 (k + 1)
// multiply-adds a row and node pair); this one takes 1300 to 1800 per cell and component, in waves of one CTA of 32
// cells an SM (4864 cells), and 110 to 340 us however few they are.  J x, matrix-free / assembled, us:
//   k = 0       64 cells 140 / 43, 4096 132 / 94, 64000 1125 / 773
//   k = 1       64 228 / 54, 4096 214 / 208, 32768 1189 / 1025, 110592 3637 / 3266; Oseen 13824 471 / 490, 46656 1406 / 1413,
//               64000 1856 / 1910, 110592 3039 / 3268
//   k = 2       64 341 / 60, 5832 591 / 436, 8000 596 / 566, 13824 843 / 896, 32768 1820 / 1974; Oseen 5832 512 / 437,
//               13824 724 / 895, 32768 1545 / 1976
// A Newton iterate's operator is matrix-free at any size: there is nothing to assemble for it (48^3, k = 1: 23 ms).
// In 2D it was the slower one (256^2 k = 3 step 43 -> 48 ms, 352 x 64 order 4 32 -> 35 ms).
bool operator_mf_preferred(const Geom& g, bool newton) {
  if (g.dim != 3) return false;
  return g.nt == 3 ? g.n_cells >= 10000 : g.nt == 2 && !newton && g.n_cells >= 40000;
}

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
