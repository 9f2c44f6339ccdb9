// Coarse-level direct solver: interior elimination per cell column plus block
// cyclic reduction over the vertex planes, in precision T.  See coarse.cu.
#pragma once

#include <vector>

#include "common.cuh"

namespace stg {

// Scratch of gj_invert for the matrices that go by panels (FP32 beyond the 256 rows of the on-chip form, FP64): device
// arrays of pointers to one m x m block and gj_panel_values(m) values per matrix, and per matrix m pivot rows (piv),
// m row positions (pos) and a failure flag.
template <typename T>
struct GjScratch {
  T* const* alt = nullptr;
  T** panel = nullptr;
  int *piv = nullptr, *pos = nullptr, *fail = nullptr;
};
template <typename T>
bool gj_by_panels(long long m) {
  return sizeof(T) == 8 || m > 256;
}
// The panel, and for FP32 up to 511 rows its multipliers, its pivot rows and 32 reciprocal pivots behind them.
template <typename T>
long long gj_panel_values(long long m) {
  return sizeof(T) == 8 ? 16 * m : (m < 512 ? 3 * 32 * m + 32 : 32 * m);
}
// 512 threads hold 19 (FP32) or 18 (FP64) rows of a panel each.
template <typename T>
constexpr int gj_max_rows() {
  return sizeof(T) == 4 ? 9728 : 9216;
}
// In-place inverses of `batch` m x m row-major matrices by Gauss-Jordan with partial pivoting;
// status gets 1 + the index of a singular matrix (coarse_gj.cu).
template <typename T>
void gj_invert(int m, T* const* A, int batch, int* status, const GjScratch<T>& s, cudaStream_t st);

template <typename T>
struct CoarseView {
  Geom g;
  int pin, nsi, nsv, mV, mI;
  T *AII, *AIV, *AVI, *D, *L, *U;
  int* status;  // [0]: 1 + first singular block, [1]: unexpected coupling
};

template <typename T>
struct CrLevel {
  long long stride;
  int n_odd, n_left, n_right;
  T** oD;
  // solve lists.  Forward, even planes with a neighbour: b_j -= PL_j b_{j-st} + PR_j b_{j+st}
  // with PL_j = L_j D_{j-st}^{-1}, PR_j = U_j D_{j+st}^{-1} (so t = D^{-1} b of the odd planes is
  // never formed); backward, odd planes: x_i = D_i^{-1} b_i - GL_i x_{i-st} - GU_i x_{i+st}.
  // Absent terms are null pointers.
  int n_even;
  T **fA0, **fx0, **fA1, **fx1, **ey;
  T **bx, **bGL, **bxl, **qA1, **qx1, **bb;
  // factorisation lists: [GL_i | GU_i] = D_i^{-1} [L_i | U_i] (2 n_odd items); D_j -= L_j GU_{j-st}
  // + U_j GL_{j+st} (n_even items, A = eA0 / eA1, B = dB0 / dB1); new L_j = -L_j GL_{j-st}, new
  // U_j = -U_j GU_{j+st} (n_left + n_right items, written to this level's own blocks); PL_j, PR_j
  // (n_left + n_right items: A = uA, B = pB, C = pC)
  T **eA0, **eA1;
  T **gA, **gB, **gC, **dB0, **dB1, **dC, **uA, **uB, **uC, **pB, **pC;
};

// One step of the coarse solve (its plan is built once, at init), one launch each:
//   kGather  b (FP64, level layout) -> vertex and interior right-hand sides bV, bI
//   kMV      y_i = alpha (A0_i x0_i + A1_i x1_i) + A2_i x2_i + c_i + beta y_i, i < batch, M rows
//            per item (Ak: M x Nk row-major); a null array, or a null entry of one, drops its
//            term
//   kScatter xV, xI -> x, or added into x (FP64, level layout)
enum CoarseStepKind : int { kGather = 1, kMV = 2, kScatter = 4 };

template <typename T>
struct CStep {
  int kind, M, N0, N1, N2, batch;
  T alpha, beta;
  const T* const* A0;
  const T* const* x0;
  const T* const* A1;
  const T* const* x1;
  const T* const* A2;
  const T* const* x2;
  const T* const* c;
  T* const* y;
};

template <typename T>
struct CoarseSolver {
  CoarseView<T> v{};
  T *W = nullptr, *C = nullptr, *GL = nullptr, *GU = nullptr;
  T *bV = nullptr, *xV = nullptr, *bI = nullptr, *gI = nullptr, *xI = nullptr;
  T **d_AII = nullptr, **d_AIV = nullptr, **d_AVI = nullptr, **d_W = nullptr, **d_C = nullptr;
  T **d_bI = nullptr, **d_gI = nullptr, **d_xVs = nullptr, **d_xI = nullptr;
  T **d_cA0 = nullptr, **d_cx0 = nullptr, **d_cA1 = nullptr, **d_cx1 = nullptr, **d_cy = nullptr;
  T **d_top = nullptr, **d_topb = nullptr, **d_topx = nullptr;
  T** d_alt = nullptr;  // the second blocks of the interiors' inversion; the planes take GL's
  T** d_top_alt = nullptr;
  GjScratch<T> gj;
  std::vector<CrLevel<T>> levels;
  std::vector<void*> owned;
  // the solve as a list of steps, one launch each
  std::vector<CStep<T>> plan;

  void init(const Geom& g, bool pure_dirichlet);
  void release();
  // factor J_0 given in the internal level layout (FP64 operator), factors stored in T
  void factor(const int* rowptr, const int* colidx, const double* vv, const double* vp, const double* pv,
              cudaStream_t st);
  // x = J_0^{-1} b (add: x += J_0^{-1} b), both FP64 in the internal level layout, arithmetic in T
  void solve(const double* b, double* x, bool add, cudaStream_t st);
  // 0 = ok, > 0: 1 + singular block, -1: coupling outside the block structure (synchronises)
  int read_status(cudaStream_t st);

};

}  // namespace stg
