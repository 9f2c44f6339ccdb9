// The FP32 V-cycle's residual without a matrix (3D, order 4).
#include "residual.cuh"

namespace stg {

// Only where its rounding error (rms over the rows of |error| / (|J| |x|), against J in 64 bits) is no larger than that
// of the entries rounded once.  16 x 8 order 4 and 6 x 4 x 8, entries -> matrix-free in 1e-8, Oseen (Newton's entries round
// more): velocity rows k = 1 4.77 -> 4.72 and 6.03 -> 5.00, k = 2 5.33 -> 4.09 and 6.83 -> 4.84; pressure rows 2.7 -> 2.2 and 3.6 ->
// 2.8; 3D k = 0 with Newton's term 7.53 -> 5.31.  Order 4, k = 0 with Newton's term has 4.95 -> 5.82, and an FP32 emulation of
// k = 0 without it 3.8 -> 4.8 (order 4) and 4.2 -> 4.9 (3D): these stay assembled, Oseen from the diagonals of the blocks.
// Steps, without a matrix -> assembled: 48^3 k = 0 76 -> 82 ms, 352 x 64 order 4, k = 0 12.3 -> 15.3 (Newton), 11.8 -> 13.7 (Oseen).
// 2D order 2 stays with the assembled rows: matrix-free they are as accurate and took 2 of the 19.4 ms of a 704 x 128 step
// off, but their roundings differ, and any other rounding moves a channel's solution by up to 2e-9 (through a pressure
// mode that the residual hardly sees).
bool residual_mf_supported(const Geom& g, bool newton) { return g.dim == 3 ? newton || g.nt >= 2 : g.r == 4 && g.nt >= 2; }

long long residual_scratch(const Geom& g) { return g.dim == 3 ? 27LL * g.NV * g.n_cells : 0; }
size_t residual_coef_bytes(const Geom& g, size_t value) {
  return kTableOffset +
         value * (g.dim == 3 ? pressure_table_values<3, 3, double>(g.nt) : pressure_table_values<2, 5, double>(g.nt));
}

void residual_coef(const Geom& g, const TimeData& td, const AsmCoef& cf, void* dst, cudaStream_t st) {
  if (g.dim == 3)
    upload_coefficients<3, 3, float>(g, td, cf, dst, st);
  else
    upload_coefficients<2, 5, float>(g, td, cf, dst, st);
}

void residual_mf(const Geom& g, const void* coef, const float* w, const float* x, const float* b, float* scratch,
                 float* out, cudaStream_t st) {
  if (!residual_mf_supported(g, true)) throw Error{STG_EINVAL, "no matrix-free FP32 residual on this level"};
  if (g.dim == 3)
    switch (g.nt) {
      case 1: return run3d<1, float>(g, coef, w, x, b, scratch, out, st);
      case 2: return run3d<2, float>(g, coef, w, x, b, scratch, out, st);
      default: return run3d<3, float>(g, coef, w, x, b, scratch, out, st);
    }
  if (g.nt == 2) return run2d<2, float>(g, coef, w, x, b, out, st);
  run2d<3, float>(g, coef, w, x, b, out, st);
}

}  // namespace stg
