// The FP32 V-cycle's residual without a matrix (3D, order 4).
#include "residual.cuh"

namespace stg {

// 2D order 2 stays with the assembled rows: matrix-free they are as accurate (sweeps and V-cycles against the FP64
// form) and took 2 of the 19.4 ms of a 704 x 128 step off, but their roundings differ, and any other rounding moves a
// channel's solution by up to 2e-9 (through a pressure mode that the residual hardly sees).
bool residual_mf_supported(const Geom& g) { return g.dim == 3 || g.r == 4; }

long long residual_scratch(const Geom& g) { return g.dim == 3 ? 27LL * g.NV * g.n_cells : 0; }
size_t residual_coef_bytes() { return sizeof(MfCoef<double>); }

void residual_coef(const Geom& g, const TimeData& td, const AsmCoef& cf, void* dst, cudaStream_t st) {
  upload_coefficients<float>(g, td, cf, dst, st);
}

void residual_mf(const Geom& g, const void* coef, const float* w, const float* x, const float* b, float* scratch,
                 float* out, cudaStream_t st) {
  const MfCoef<float>* m = (const MfCoef<float>*)coef;
  if (g.dim == 3)
    dispatch3d<float>(g, m, w, x, b, scratch, out, st);
  else if (g.r == 4)
    dispatch2d<5, float>(g, m, w, x, b, out, st);
  else
    throw Error{STG_EINVAL, "no matrix-free FP32 residual for 2D order 2"};
}

}  // namespace stg
