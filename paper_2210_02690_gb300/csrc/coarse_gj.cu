// Batched Gauss-Jordan inverses of the coarse solver's dense blocks: on chip for FP32 blocks of up to
// 256 rows, by panels for the others.  A translation unit of its own: its unrolled variants compile
// beside coarse.cu.
#include <algorithm>

#include "coarse.cuh"
#include "kernels.cuh"

namespace stg {

namespace {

// Gauss-Jordan inverse of an FP32 matrix held on chip, one CTA of NW warps per matrix: lane l
// of warp w holds rows l + 32 q (q < R) and columns w + NW k (k < CR + CS), column slots k < CR
// in registers and the others in a per-thread shared-memory slice (slot-major, thread-minor:
// conflict-free).  Partial pivoting without row interchanges: the pivot row p_j of column j is
// the unused row of largest |a_rj| (first such row on ties), it is scaled, and column j is
// eliminated from every other row.  After the last column, row p_j holds row j of the inverse
// of the row-permuted matrix, whose column c is column p_c of A^{-1}; the write-out puts a_{p_j c}
// at (j, p_c).  Rows are scaled lazily: row r is stored divided by sigma_r (1 until it becomes
// a pivot row, then 1 / a_pj), so the pivot row keeps its stored values (with 1 in column j)
// and every other entry takes the same fused multiply-add, a_rk -= a_rj (a_pk / a_pj), with the
// stored a_rj: no per-entry select.  One barrier a pivot step.  The warp that holds column j + 1 updates that column
// first, searches it and publishes it (with 1 / pivot) in the other half of a double buffer,
// then finishes its update: the search overlaps the rest of the CTA's update.  Each warp takes
// the pivot row's slice of its columns from its own lane p mod 32 through a per-warp buffer.
// Same pivots and operations as the panel form below, up to the order of equal-magnitude candidates.
template <int R, int CR, int CS, int NW>
__global__ void __launch_bounds__(32 * NW, 1) rgj_kernel(int m, float* const* As, int* status) {
  constexpr int C = CR + CS, NT = 32 * NW;
  float* G = As[blockIdx.x];
  extern __shared__ __align__(16) unsigned char sh_raw[];
  float* sp = reinterpret_cast<float*>(sh_raw) + threadIdx.x;  // slot (k, q) at ((k - CR) R + q) NT
  __shared__ float s_col[2][32 * R];
  __shared__ float s_prow[NW][C];
  __shared__ int s_piv[2];
  __shared__ float s_inv[2];
  __shared__ int s_pc[32 * R], s_pr[32 * R];  // pivot row of column c; column pivoted on row r
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  float a[R][CR > 0 ? CR : 1];
#define RGJ_GET(q, k) ((k) < CR ? a[q][(k) < CR ? (k) : 0] : sp[((k) - CR) * R * NT + (q) * NT])
#define RGJ_SET(q, k, v)                          \
  do {                                            \
    if ((k) < CR)                                 \
      a[q][(k) < CR ? (k) : 0] = (v);             \
    else                                          \
      sp[((k) - CR) * R * NT + (q) * NT] = (v);   \
  } while (0)
  unsigned used = 0;  // bit q: row lane + 32 q is a pivot row already (or padding)
  float sig[R];       // row scales (see above)
#pragma unroll
  for (int q = 0; q < R; ++q) {
    const int r = lane + 32 * q;
    sig[q] = 1.f;
    if (r >= m) used |= 1u << q;
#pragma unroll
    for (int k = 0; k < C; ++k) {
      const int c = w + NW * k;
      RGJ_SET(q, k, (r < m && c < m) ? G[(long long)r * m + c] : 0.f);
    }
  }
  // pivot search in column slot k of this warp; the result goes to buffer b
  auto search = [&](int k, int b) {
    float best = -1.f, val = 0.f;
    int bi = 0x7fffffff;
#pragma unroll
    for (int q = 0; q < R; ++q) {
      const float v = RGJ_GET(q, k);
      s_col[b][lane + 32 * q] = v;
      // rows of a lane ascend with q: '>' keeps the first maximum
      if (!((used >> q) & 1u) && fabsf(v) > best) {
        best = fabsf(v);
        bi = lane + 32 * q;
        val = v;
      }
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
      const float ob = __shfl_xor_sync(0xffffffffu, best, off);
      const int oi = __shfl_xor_sync(0xffffffffu, bi, off);
      const float ov = __shfl_xor_sync(0xffffffffu, val, off);
      if (ob > best || (ob == best && oi < bi)) {
        best = ob;
        bi = oi;
        val = ov;
      }
    }
    if (lane == 0) {
      const bool ok = best > 0.f && !isinf(val);
      s_piv[b] = ok ? bi : -1;
      s_inv[b] = ok ? 1.f / val : 0.f;
    }
  };
  if (w == 0) search(0, 0);
  int buf = 0;
  bool fail = false;
#pragma unroll
  for (int kj = 0; kj < C; ++kj) {
    for (int jw = 0; jw < NW; ++jw) {
      const int j = kj * NW + jw;
      if (j >= m) break;
      __syncthreads();
      const int p = s_piv[buf];
      if (p < 0) {
        fail = true;
        break;
      }
      const float inv = s_inv[buf];
      const int pq = p >> 5, pl = p & 31;
      const bool piv_lane = lane == pl;
#pragma unroll
      for (int q = 0; q < R; ++q)
        if (q == pq && piv_lane) {
#pragma unroll
          for (int k = 0; k < C; ++k) s_prow[w][k] = (w == jw && k == kj) ? inv : RGJ_GET(q, k) * inv;
        }
      if (piv_lane) used |= 1u << pq;
      __syncwarp();
      float f[R];
#pragma unroll
      for (int q = 0; q < R; ++q) {
        const bool pr_here = q == pq && piv_lane;
        f[q] = pr_here ? 0.f : s_col[buf][lane + 32 * q];  // the pivot row is not updated
        if (pr_here) sig[q] = inv;
      }
      if (w == jw) {
        // column j becomes -a_rj / a_pj; the pivot row stores 1 (times sigma_p = 1 / a_pj)
#pragma unroll
        for (int q = 0; q < R; ++q) RGJ_SET(q, kj, (q == pq && piv_lane) ? 1.f : 0.f);
      }
      // the row update of column slot k: a_rk -= f_r pr_k
      auto update = [&](int k) {
        const float pk = s_prow[w][k];
#pragma unroll
        for (int q = 0; q < R; ++q) RGJ_SET(q, k, fmaf(-f[q], pk, RGJ_GET(q, k)));
      };
      // look-ahead: column j + 1 is slot kj of warp jw + 1, or slot kj + 1 of warp 0
      const bool next_here = jw + 1 < NW;
      const int la_w = next_here ? jw + 1 : 0;
      const bool la = w == la_w && j + 1 < m && (next_here || kj + 1 < C);
      if (la) {
        if (next_here) {
          update(kj);
          search(kj, buf ^ 1);
        } else if (kj + 1 < C) {
          update(kj + 1);
          search(kj + 1, buf ^ 1);
        }
      }
      const int la_k = next_here ? kj : kj + 1;
#pragma unroll
      for (int k = 0; k < CR; ++k)
        if (!(la && k == la_k)) update(k);
      if (CS > 0) {
        // shared-memory slots: all R loads of a slot are issued together, and those of the
        // next slot before the stores of this one (the stores could alias the loads otherwise)
        float cur[R], nxt[R];
#pragma unroll
        for (int q = 0; q < R; ++q) cur[q] = RGJ_GET(q, CR);
#pragma unroll
        for (int k = CR; k < C; ++k) {
          if (k + 1 < C) {
#pragma unroll
            for (int q = 0; q < R; ++q) nxt[q] = RGJ_GET(q, k + 1 < C ? k + 1 : k);
          }
          if (!(la && k == la_k)) {
            const float pk = s_prow[w][k];
#pragma unroll
            for (int q = 0; q < R; ++q) RGJ_SET(q, k, fmaf(-f[q], pk, cur[q]));
          }
#pragma unroll
          for (int q = 0; q < R; ++q) cur[q] = nxt[q];
        }
      }
      if (tid == 0) {
        s_pc[j] = p;
        s_pr[p] = j;
      }
      buf ^= 1;
    }
    if (fail) break;
  }
  if (fail) {
    if (tid == 0) atomicCAS(status, 0, 1 + (int)blockIdx.x);
    return;
  }
  __syncthreads();
#pragma unroll
  for (int q = 0; q < R; ++q) {
    const int r = lane + 32 * q;
    if (r < m) {
      const long long row = (long long)s_pr[r] * m;
#pragma unroll
      for (int k = 0; k < C; ++k) {
        const int c = w + NW * k;
        if (c < m) G[row + s_pc[c]] = RGJ_GET(q, k) * sig[q];
      }
    }
  }
#undef RGJ_GET
#undef RGJ_SET
}

// ---------------------------------------------------------------- by panels
// Gauss-Jordan with partial pivoting by panels of w columns, without row interchanges.  A panel
// kernel (one CTA per matrix, the m x w panel in registers, R rows a thread) runs the w pivot steps on
// the panel alone; an update kernel over all SMs then gives the other columns, reading X and writing Y
// (two buffers in turn), with p_j the row of pivot j:
//   Y[r][c] = (r a pivot row of the panel ? 0 : X[r][c]) + sum_j P[r][j] X[p_j][c]
// with P the panel after its steps, or (SEQ) step by step with the multipliers F[r][j] and the pivot rows as
// they stand at their step (gj_rows_kernel):
//   Y[r][c] = X[r][c] - sum_j F[r][j] Q_j[c], j ascending.
// After the last column row p_j holds row j of the inverse of the row-permuted matrix, whose column c is
// column p_c of A^{-1}: the last update writes a_{p_j c} to (j, p_c).
//
// A pivot step has one barrier: every warp posts its best candidate |a_rj| (unused rows; of equal ones the one
// that row interchanges would have brought first) with that row's panel values, and after the barrier every
// warp finds the best of the posted ones by itself.  The panel's columns rotate by one a step, so that the
// pivot column is column 0 and the loop stays rolled (unrolled, each step's code ran once and its fetch
// took 1 us).
//
// It replaces one CTA per matrix in global memory (FP32 257 to 511 rows, FP64 from 167 on), one in shared memory
// (FP64) and a panel kernel with six barriers a step (512 rows and more), with their operations in
// their order for FP32 up to 1024 rows: the same bits.  16 blocks of 452 rows: 9.5 ms before.

__device__ __forceinline__ unsigned gj_key_hi(float v) { return v == v ? __float_as_uint(fabsf(v)) + 1u : 0u; }
__device__ __forceinline__ unsigned gj_key_lo(float) { return 0u; }
__device__ __forceinline__ unsigned gj_key_hi(double v) {
  return v == v ? (unsigned)(__double_as_longlong(fabs(v)) >> 32) + 1u : 0u;
}
__device__ __forceinline__ unsigned gj_key_lo(double v) { return v == v ? (unsigned)__double_as_longlong(fabs(v)) : 0u; }

// Lane of the largest (hi, lo) of the warp, of equal ones the smallest pos; hi, lo become that key.
template <typename T>
__device__ __forceinline__ int gj_warp_best(unsigned& hi, unsigned& lo, unsigned pos) {
  const unsigned mh = __reduce_max_sync(0xffffffffu, hi);
  unsigned ml = 0u;
  if (sizeof(T) == 8) ml = __reduce_max_sync(0xffffffffu, hi == mh ? lo : 0u);
  const bool top = hi == mh && (sizeof(T) == 4 || lo == ml);
  const unsigned mp = __reduce_min_sync(0xffffffffu, top ? pos : 0xffffffffu);
  const unsigned who = __ballot_sync(0xffffffffu, top && pos == mp);
  hi = mh;
  lo = ml;
  return __ffs(who) - 1;
}

// The three panels of a matrix and its reciprocal pivots.
template <typename T>
struct GjPanels {
  T *P, *F, *Q, *iv;
};
template <typename T, int W>
__device__ __forceinline__ GjPanels<T> gj_panels(T* p, int m) {
  return GjPanels<T>{p, p + (long long)W * m, p + 2LL * W * m, p + 3LL * W * m};
}

// w <= W columns from c0 on; thread t holds rows t + q blockDim.x (q < R).  P: m x W, the panel in its last w
// columns.  piv[b][j]: pivot row of column j; pos[b][r]: the row's place under row interchanges (the column pivoted
// on it once it has been a pivot row).
template <typename T, int R, int W, bool SEQ>
__global__ void __launch_bounds__(512, 1) gj_panel_kernel(int m, int c0, int w, const T* const* Xs, T* const* Ps,
                                                          int* __restrict__ piv, int* __restrict__ pos,
                                                          int* __restrict__ fail, int* __restrict__ status) {
  const int b = blockIdx.x, tid = threadIdx.x, nth = blockDim.x, lane = tid & 31, wid = tid >> 5, nw = nth >> 5;
  if (c0 > 0 && fail[b]) return;
  const T* X = Xs[b];
  const GjPanels<T> pn = gj_panels<T, W>(Ps[b], m);
  __shared__ __align__(16) T s_row[2][16][W];
  __shared__ unsigned s_hi[2][16], s_lo[2][16];
  __shared__ int s_id[2][16], s_pos[2][16];
  T a[R][W];
  int place[R];
#pragma unroll
  for (int q = 0; q < R; ++q) {
    const int r = tid + q * nth;
    place[q] = r >= m ? -1 : (c0 == 0 ? r : pos[(long long)b * m + r]);
#pragma unroll
    for (int c = 0; c < W; ++c) a[q][c] = (r < m && c < w) ? X[(long long)r * m + c0 + c] : (T)0;
  }
  if (c0 == 0 && tid == 0) fail[b] = 0;
#pragma unroll 1
  for (int jj = 0; jj < w; ++jj) {
    const int buf = jj & 1, j = c0 + jj;
    // this thread's candidate, then the warp's; rows at places below j have been pivot rows
    unsigned hi = 0u, lo = 0u, at = 0xffffffffu;
    int bq = 0;
#pragma unroll
    for (int q = 0; q < R; ++q) {
      const bool free_row = place[q] >= j;
      const unsigned h = free_row ? gj_key_hi(a[q][0]) : 0u, l = free_row ? gj_key_lo(a[q][0]) : 0u;
      if (h > hi || (h == hi && (l > lo || (l == lo && (unsigned)place[q] < at)))) {
        hi = h;
        lo = l;
        at = (unsigned)place[q];
        bq = q;
      }
    }
    const int src = gj_warp_best<T>(hi, lo, at);
    if (lane == src) {
      s_hi[buf][wid] = hi;
      s_lo[buf][wid] = lo;
      s_id[buf][wid] = tid + bq * nth;
      s_pos[buf][wid] = (int)at;
#pragma unroll
      for (int q = 0; q < R; ++q)
        if (q == bq) {
#pragma unroll
          for (int c = 0; c < W; ++c) s_row[buf][wid][c] = a[q][c];
        }
    }
    __syncthreads();
    hi = lane < nw ? s_hi[buf][lane] : 0u;
    lo = lane < nw ? s_lo[buf][lane] : 0u;
    const int best = gj_warp_best<T>(hi, lo, lane < nw ? (unsigned)s_pos[buf][lane] : 0xffffffffu);
    const int p = s_id[buf][best], pp = s_pos[buf][best];
    const T* row = s_row[buf][best];
    const T pv = row[0];
    if (hi == 0u || !(fabs(pv) > (T)0) || isinf(pv)) {  // the same for every thread
      if (tid == 0) {
        fail[b] = 1;
        atomicCAS(status, 0, 1 + b);
      }
      return;
    }
    const T iv = (T)1 / pv;
    T f[R];
#pragma unroll
    for (int q = 0; q < R; ++q) {
      f[q] = a[q][0];
      if (SEQ && tid + q * nth < m) pn.F[(long long)jj * m + tid + q * nth] = f[q];
    }
    if (SEQ && tid == 0) pn.iv[jj] = iv;
#pragma unroll
    for (int c = 1; c < W; ++c) {
      const T rc = row[c] * iv;
#pragma unroll
      for (int q = 0; q < R; ++q) a[q][c - 1] = fma(-f[q], rc, a[q][c]);
    }
#pragma unroll
    for (int q = 0; q < R; ++q) {
      a[q][W - 1] = -f[q] * iv;
      if (place[q] == j) place[q] = pp;
    }
    // the pivot row itself
    if ((p & 31) == lane) {
#pragma unroll
      for (int q = 0; q < R; ++q)
        if (p == tid + q * nth) {
#pragma unroll
          for (int c = 1; c < W; ++c) a[q][c - 1] = row[c] * iv;
          a[q][W - 1] = iv;
          place[q] = j;
          piv[(long long)b * m + j] = p;
        }
    }
  }
#pragma unroll
  for (int q = 0; q < R; ++q) {
    const int r = tid + q * nth;
    if (r < m) {
      pos[(long long)b * m + r] = place[q];
#pragma unroll
      for (int c = 0; c < W; ++c) pn.P[(long long)r * W + c] = a[q][c];
    }
  }
}

// SEQ: the panel's pivot rows in the other columns, one thread a column: Q_j as it stands at step j, scaled (for the
// other rows' update), and Y's pivot rows after the remaining steps.
template <typename T, int W>
__global__ void __launch_bounds__(64) gj_rows_kernel(int m, int c0, int w, const T* const* Xs, T* const* Ys, T* const* Ps,
                                                     const int* __restrict__ piv, const int* __restrict__ fail,
                                                     int last) {
  const int b = blockIdx.y;
  if (fail[b]) return;
  const T* X = Xs[b];
  T* Y = Ys[b];
  const GjPanels<T> pn = gj_panels<T, W>(Ps[b], m);
  const int* pv = piv + (long long)b * m;
  __shared__ __align__(16) T s_f[W][W];  // [step][pivot row]
  __shared__ T s_iv[W];
  __shared__ int s_p[W];
  const int tid = threadIdx.x, c = blockIdx.x * 64 + tid;
  if (tid < W) {
    s_p[tid] = tid < w ? pv[c0 + tid] : 0;
    s_iv[tid] = tid < w ? pn.iv[tid] : (T)0;
  }
  __syncthreads();
  for (int t = tid; t < W * W; t += 64) {
    const int i = t / W, j = t % W;
    s_f[i][j] = (i < w && j < w) ? pn.F[(long long)i * m + s_p[j]] : (T)0;
  }
  __syncthreads();
  if (c >= m || (c >= c0 && c < c0 + w)) return;
  T x[W];
#pragma unroll
  for (int j = 0; j < W; ++j) x[j] = j < w ? X[(long long)s_p[j] * m + c] : (T)0;
  // step i scales row i and takes it from every other pivot row: rows after it (not yet pivots) and before it alike
#pragma unroll
  for (int i = 0; i < W; ++i) {
    if (i < w) {
      x[i] *= s_iv[i];
      pn.Q[(long long)i * m + c] = x[i];
#pragma unroll
      for (int j = 0; j < W; ++j)
        if (j != i) x[j] = fma(-s_f[i][j], x[i], x[j]);
    }
  }
  const int cc = last ? pv[c] : c;
#pragma unroll
  for (int j = 0; j < W; ++j)
    if (j < w) Y[(long long)(last ? c0 + j : s_p[j]) * m + cc] = x[j];
}

// Y from X and the panel (see above); 16 TM wide tiles, TM x TM entries a thread.  Bound by the pass over
// the matrix (2 m^2 values) for short panels, by the FMAs (w per entry) otherwise.
template <typename T, int W, int TM, bool SEQ>
__global__ void __launch_bounds__(256) gj_panel_update_kernel(int m, int c0, int w, const T* const* Xs, T* const* Ys,
                                                              T* const* Ps, const int* __restrict__ piv,
                                                              const int* __restrict__ pos,
                                                              const int* __restrict__ fail, int last) {
  const int b = blockIdx.z;
  if (fail[b]) return;
  constexpr int BM = 16 * TM, BN = BM, PAD = 16 / sizeof(T);
  __shared__ __align__(16) T sa[W][BM + PAD];
  __shared__ __align__(16) T sb[W][BN + PAD];
  __shared__ int s_p[W];
  __shared__ int s_isp[BM];
  const int tid = threadIdx.x, tx = tid % 16, ty = tid / 16, r0 = blockIdx.y * BM, q0 = blockIdx.x * BN;
  const T* X = Xs[b];
  const GjPanels<T> pn = gj_panels<T, W>(Ps[b], m);
  const int* pv = piv + (long long)b * m;
  T x[TM][TM];
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TM; ++j) {
      const int r = r0 + ty * TM + i, c = q0 + tx * TM + j;
      x[i][j] = (r < m && c < m) ? X[(long long)r * m + c] : (T)0;
    }
  if (tid < BM) s_isp[tid] = 0;
  if (tid < w) s_p[tid] = pv[c0 + tid];
  __syncthreads();
  if (tid < w) {
    const int d = s_p[tid] - r0;
    if (d >= 0 && d < BM) s_isp[d] = 1;
  }
  for (int t = tid; t < BM * w; t += 256) {
    if (SEQ) {
      const int k = t / BM, i = t % BM;
      sa[k][i] = r0 + i < m ? -pn.F[(long long)k * m + r0 + i] : (T)0;
    } else {
      const int i = t / w, k = t - i * w;
      sa[k][i] = r0 + i < m ? pn.P[(long long)(r0 + i) * W + W - w + k] : (T)0;
    }
  }
  for (int t = tid; t < w * BN; t += 256) {
    const int k = t / BN, j = t % BN, c = q0 + j;
    const bool on = c < m && (c < c0 || c >= c0 + w);
    sb[k][j] = on ? (SEQ ? pn.Q[(long long)k * m + c] : X[(long long)s_p[k] * m + c]) : (T)0;
  }
  __syncthreads();
  T acc[TM][TM];
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TM; ++j) {
      if (!SEQ && s_isp[ty * TM + i]) x[i][j] = (T)0;
      acc[i][j] = SEQ ? x[i][j] : (T)0;
    }
#pragma unroll 4
  for (int k = 0; k < w; ++k) {
    T av[TM], bv[TM];
#pragma unroll
    for (int i = 0; i < TM; ++i) av[i] = sa[k][ty * TM + i];
#pragma unroll
    for (int j = 0; j < TM; ++j) bv[j] = sb[k][tx * TM + j];
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
      for (int j = 0; j < TM; ++j) acc[i][j] = fma(av[i], bv[j], acc[i][j]);
  }
  T* Y = Ys[b];
  const int* ps = pos + (long long)b * m;
#pragma unroll
  for (int i = 0; i < TM; ++i) {
    const int r = r0 + ty * TM + i;
    if (r >= m) continue;
    T* y = Y + (long long)(last ? ps[r] : r) * m;
#pragma unroll
    for (int j = 0; j < TM; ++j) {
      const int c = q0 + tx * TM + j;
      if (c >= m) continue;
      if (c >= c0 && c < c0 + w)
        y[last ? pv[c] : c] = pn.P[(long long)r * W + W - w + c - c0];
      else if (!SEQ)
        y[last ? pv[c] : c] = acc[i][j] + x[i][j];
      else if (!s_isp[ty * TM + i])
        y[last ? pv[c] : c] = acc[i][j];
    }
  }
}

template <typename T>
__global__ void __launch_bounds__(256) gj_copy_kernel(long long n, const T* const* Xs, T* const* Ys) {
  const T* X = Xs[blockIdx.y];
  T* Y = Ys[blockIdx.y];
  for (long long t = (long long)blockIdx.x * 256 + threadIdx.x; t < n; t += (long long)gridDim.x * 256) Y[t] = X[t];
}

// wp: panel width, at most W; 0: widths that make the number of panels even.
template <typename T, int R, int W, bool SEQ>
void invert_by_panels(int m, T* const* A, int batch, int wp, int* status, const GjScratch<T>& s, cudaStream_t st) {
  if (wp == 0) {
    const int even = 2 * ((m + 2 * W - 1) / (2 * W));
    wp = (m + even - 1) / even;
  }
  const int np = std::max(1, (m + wp - 1) / wp);
  const int threads = ((m + R - 1) / R + 31) / 32 * 32;
  // tiles of 48 for FP64 and the smaller blocks (134 and 226 rows fill them), of 64 for the larger
  constexpr int TMS = 3, TML = sizeof(T) == 8 ? 3 : 4;
  const int tile = 16 * (m < 512 ? TMS : TML);
  const dim3 grid((m + tile - 1) / tile, (m + tile - 1) / tile, batch);
  // the buffers take turns and the last update has to land in A: an odd number of panels starts from a copy
  T* const* X = A;
  T* const* Y = s.alt;
  if (np % 2) {
    gj_copy_kernel<T><<<dim3(std::min(64, (m * m + 255) / 256), batch), 256, 0, st>>>((long long)m * m, A, s.alt);
    STG_LAUNCH_OK();
    std::swap(X, Y);
  }
  for (int t = 0; t < np; ++t) {
    const int c0 = t * wp, w = std::min(wp, m - c0), last = t == np - 1 ? 1 : 0;
    gj_panel_kernel<T, R, W, SEQ><<<batch, threads, 0, st>>>(m, c0, w, X, s.panel, s.piv, s.pos, s.fail, status);
    STG_LAUNCH_OK();
    if constexpr (SEQ) {
      gj_rows_kernel<T, W><<<dim3((m + 63) / 64, batch), 64, 0, st>>>(m, c0, w, X, Y, s.panel, s.piv, s.fail, last);
      STG_LAUNCH_OK();
    }
    if (m < 512)
      gj_panel_update_kernel<T, W, TMS, SEQ>
          <<<grid, 256, 0, st>>>(m, c0, w, X, Y, s.panel, s.piv, s.pos, s.fail, last);
    else
      gj_panel_update_kernel<T, W, TML, SEQ>
          <<<grid, 256, 0, st>>>(m, c0, w, X, Y, s.panel, s.piv, s.pos, s.fail, last);
    STG_LAUNCH_OK();
    std::swap(X, Y);
  }
}

}  // namespace

// FP32 matrices of up to 256 rows: on-chip Gauss-Jordan, 16 warps a matrix (column slots of
// a thread beyond its register budget in shared memory)
template <int R, int CR, int CS, int NW>
static void launch_rgj(int m, float* const* A, int batch, int* status, cudaStream_t st) {
  const size_t smem = sizeof(float) * (size_t)CS * R * 32 * NW;
  if (smem > 48 * 1024)
    STG_CUDA_OK(cudaFuncSetAttribute(rgj_kernel<R, CR, CS, NW>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)smem));
  rgj_kernel<R, CR, CS, NW><<<batch, 32 * NW, smem, st>>>(m, A, status);
  STG_LAUNCH_OK();
}

static bool rgj_invert(int m, float* const* A, int batch, int* status, cudaStream_t st) {
  switch ((m + 15) / 16) {
    case 1: launch_rgj<1, 1, 0, 16>(m, A, batch, status, st); return true;
    case 2: launch_rgj<1, 2, 0, 16>(m, A, batch, status, st); return true;
    case 3: launch_rgj<2, 3, 0, 16>(m, A, batch, status, st); return true;
    case 4: launch_rgj<2, 4, 0, 16>(m, A, batch, status, st); return true;
    case 5: launch_rgj<3, 5, 0, 16>(m, A, batch, status, st); return true;
    case 6: launch_rgj<3, 6, 0, 16>(m, A, batch, status, st); return true;
    case 7: launch_rgj<4, 7, 0, 16>(m, A, batch, status, st); return true;
    case 8: launch_rgj<4, 8, 0, 16>(m, A, batch, status, st); return true;
    case 9: launch_rgj<5, 9, 0, 16>(m, A, batch, status, st); return true;
    case 10: launch_rgj<5, 10, 0, 16>(m, A, batch, status, st); return true;
    case 11: launch_rgj<6, 11, 0, 16>(m, A, batch, status, st); return true;
    case 12: launch_rgj<6, 11, 1, 16>(m, A, batch, status, st); return true;
    case 13: launch_rgj<7, 8, 5, 16>(m, A, batch, status, st); return true;
    case 14: launch_rgj<7, 8, 6, 16>(m, A, batch, status, st); return true;
    case 15: launch_rgj<8, 7, 8, 16>(m, A, batch, status, st); return true;
    case 16: launch_rgj<8, 7, 9, 16>(m, A, batch, status, st); return true;
    default: return false;
  }
}

static bool rgj_invert(int, double* const*, int, int*, cudaStream_t) { return false; }

template <typename T>
void gj_invert(int m, T* const* A, int batch, int* status, const GjScratch<T>& s, cudaStream_t st) {
  if (batch <= 0 || m <= 0) return;
  if (m > gj_max_rows<T>()) throw Error{STG_EINVAL, "coarse block larger than its inversion takes"};
  if (rgj_invert(m, A, batch, status, st)) return;
  // the panel's R W values of a thread fit 72 registers (512 threads have 128 each); FP64 halves W.  FP32 up to
  // 1024 rows in the operations and order of the forms it replaces (coarse factors of 2D levels keep their bits).
  constexpr int D = sizeof(T) / 4;
  constexpr bool F32 = sizeof(T) == 4;
  if (m < 512 || (m == 512 && !F32))
    invert_by_panels<T, 1, 32 / D, F32>(m, A, batch, 0, status, s, st);
  else if (m <= 1024)
    invert_by_panels<T, 2, 32 / D, false>(m, A, batch, F32 ? 32 : 0, status, s, st);
  else if (m <= 2048)
    invert_by_panels<T, 4, 16 / D, false>(m, A, batch, 0, status, s, st);
  else if (m <= 4608)
    invert_by_panels<T, 9, 8 / D, false>(m, A, batch, 0, status, s, st);
  else if (m <= 9216)
    invert_by_panels<T, 18, 4 / D, false>(m, A, batch, 0, status, s, st);
  else if constexpr (F32)
    invert_by_panels<T, 19, 4, false>(m, A, batch, 0, status, s, st);
}

template void gj_invert<float>(int, float* const*, int, int*, const GjScratch<float>&, cudaStream_t);
template void gj_invert<double>(int, double* const*, int, int*, const GjScratch<double>&, cudaStream_t);

}  // namespace stg
