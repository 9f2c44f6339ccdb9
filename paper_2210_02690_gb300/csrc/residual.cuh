// J x and b - J x without a matrix: the FP32 V-cycle's residual in 3D and for order 4 from two Radau nodes on (residual.cu;
// the other levels use vanka.cu's rows) and the FP64 operator in 3D (residual64.cu).
//
// The slab operator (Eq. (3.3) with D_ab and B_ab of Eq. (2.1), (2.2)) applied cell by cell by sum
// factorisation: the nodal values of a cell are interpolated to its Gauss points one direction at a
// time, differentiated there by the 1D collocation derivative, combined with the linearisation
// velocity at the points, and taken back by the transposed steps.  One thread holds one component
// (Radau node a, direction c) of one cell; the components of a cell exchange their values at the
// Gauss points through shared memory (time coupling, convection, Newton's term).  The velocity-pressure
// coupling is a small table per Radau node, component and set of Dirichlet faces, integrated in FP64 and
// rounded once, as an assembled block is: summed over the Gauss points in FP32 the pressure rows of order 4
// had twice an assembled row's rounding error.  (It is the faster form too: 48^3, k = 1 in FP64 4.22 -> 3.17 ms a launch,
// in FP32 142 -> 127 us.)  Everything else is read from nodal vectors, so a residual
// moves a few vectors where the assembled operator moved 4 (1 + (k+1) d^2) bytes per node pair in 2D and
// 4 ((k+1) d)^2 in 3D.
#pragma once

#include <algorithm>
#include <cstring>

#include "common.cuh"
#include "kernels.cuh"

namespace stg {
namespace {

__host__ __device__ constexpr int ipow(int b, int e) { return e == 0 ? 1 : b * ipow(b, e - 1); }

// 1D reference element with M = r + 1 equidistant nodes and M Gauss points on [-1, 1].
template <int DIM, int M, typename T>
struct Ref {
  T x[M], w[M];        // Gauss points and weights
  T wt[ipow(M, DIM)];  // products of the weights at the tensor points
  T L[M][M];           // Lagrange function of node l at Gauss point q: [q][l]
  T G[M][M];           // derivative at Gauss point q of the Lagrange function of Gauss point p: [q][p]
  T DN[2][M];          // derivative at -1 and +1 of the Lagrange function of node l
  T MM[M][M];          // integral of the product of the Lagrange functions of nodes l and m
};

template <int DIM, int M, typename T>
constexpr Ref<DIM, M, T> make_ref() {
  Ref<DIM, M, double> r{};
  if (M == 3) {
    const double x[3] = {-0.774596669241483377, 0.0, 0.774596669241483377};
    const double w[3] = {5.0 / 9.0, 8.0 / 9.0, 5.0 / 9.0};
    for (int i = 0; i < 3; ++i) {
      r.x[i] = x[i];
      r.w[i] = w[i];
    }
  } else {
    const double x[5] = {-0.906179845938663993, -0.538469310105683091, 0.0, 0.538469310105683091,
                         0.906179845938663993};
    const double w[5] = {0.236926885056189088, 0.478628670499366468, 128.0 / 225.0, 0.478628670499366468,
                         0.236926885056189088};
    for (int i = 0; i < M; ++i) {
      r.x[i] = x[i];
      r.w[i] = w[i];
    }
  }
  double node[M] = {};
  for (int l = 0; l < M; ++l) node[l] = -1.0 + 2.0 * l / (M - 1);
  const double end[2] = {-1.0, 1.0};
  for (int q = 0; q < M; ++q)
    for (int l = 0; l < M; ++l) {
      double v = 1.0, d = 0.0;
      for (int m = 0; m < M; ++m)
        if (m != l) v *= (r.x[q] - node[m]) / (node[l] - node[m]);
      for (int m = 0; m < M; ++m) {
        if (m == l) continue;
        double t = 1.0 / (r.x[l] - r.x[m]);
        for (int n = 0; n < M; ++n)
          if (n != l && n != m) t *= (r.x[q] - r.x[n]) / (r.x[l] - r.x[n]);
        d += t;
      }
      r.L[q][l] = v;
      r.G[q][l] = d;
    }
  for (int s = 0; s < 2; ++s)
    for (int l = 0; l < M; ++l) {
      double d = 0.0;
      for (int m = 0; m < M; ++m) {
        if (m == l) continue;
        double t = 1.0 / (node[l] - node[m]);
        for (int n = 0; n < M; ++n)
          if (n != l && n != m) t *= (end[s] - node[n]) / (node[l] - node[n]);
        d += t;
      }
      r.DN[s][l] = d;
    }
  for (int l = 0; l < M; ++l)
    for (int m = 0; m < M; ++m)
      for (int q = 0; q < M; ++q) r.MM[l][m] += r.w[q] * r.L[q][l] * r.L[q][m];
  Ref<DIM, M, T> o{};
  for (int i = 0; i < M; ++i) {
    o.x[i] = (T)r.x[i];
    o.w[i] = (T)r.w[i];
    for (int j = 0; j < M; ++j) {
      o.L[i][j] = (T)r.L[i][j];
      o.G[i][j] = (T)r.G[i][j];
      o.MM[i][j] = (T)r.MM[i][j];
    }
    for (int k = 0; k < 2; ++k) o.DN[k][i] = (T)r.DN[k][i];
  }
  for (int i = 0; i < ipow(M, DIM); ++i)
    o.wt[i] = (T)(r.w[i % M] * r.w[(i / M) % M] * (DIM == 3 ? r.w[(i / (M * M)) % M] : 1.0));
  return o;
}

// constant memory: after unrolling every entry is an operand of its multiply-add
template <int DIM, int M, typename T>
__constant__ Ref<DIM, M, T> c_ref = make_ref<DIM, M, T>();

// Pressure function m of P_{r-1}^disc at reference coordinates c.
template <int M>
__device__ __forceinline__ double pressure_fn(int m, const double* c) {
  if (m == 0) return 1.0;
  if (M == 3 || m <= 2) return c[m - 1];
  const double x = c[0], y = c[1];
  return m == 3 ? x * x : m == 4 ? x * y : m == 5 ? y * y : m == 6 ? x * x * x : m == 7 ? x * x * y : m == 8 ? x * y * y
                                                                                                        : y * y * y;
}

// Coefficients of the operator, cell volume / 2^d folded into the time factors.  They sit in device memory:
// a captured V-cycle sees a new slab length.
template <typename T>
struct MfCoef {
  T time[5][5];   // T_ab |det|
  T sa[5];        // tau w_a |det|
  T sc[3];        // 2 / h_e
  T nu, g1[3], g2[3];  // viscosity; gamma1 nu / h_e, gamma2 / h_e
  int newton;  // not 0: with Newton's term
};

// Pressure coefficients of a cell and Radau node, and the same padded to whole 16-byte loads of the table.
template <int M>
constexpr int kNP = M == 3 ? 4 : 10;  // M == 3: 3D
template <int M>
constexpr int kNPP = M == 3 ? 4 : 12;

// Entry (a, faces, c, i, m): pressure row m of Radau node a against component c at node i of a cell with these
// Dirichlet faces (bit 2 e + side).  The velocity rows take the negative transpose.
template <int DIM, int M, typename T>
__global__ void __launch_bounds__(128) pressure_table(int count, MfCoef<double> cf, T* __restrict__ table) {
  const Ref<DIM, M, double>& R = c_ref<DIM, M, double>;
  constexpr int N = ipow(M, DIM), NCLS = 1 << (2 * DIM);
  const int t = blockIdx.x * 128 + threadIdx.x;
  if (t >= count) return;
  const int m = t % kNPP<M>, i = t / kNPP<M> % N, c = t / (kNPP<M> * N) % DIM;
  const int faces = t / (kNPP<M> * N * DIM) % NCLS, a = t / (kNPP<M> * N * DIM * NCLS);
  if (m >= kNP<M>) {
    table[t] = (T)0;
    return;
  }
  const int in[3] = {i % M, i / M % M, i / (M * M)};
  double sum = 0.0;
  for (int q = 0; q < N; ++q) {
    const int qn[3] = {q % M, q / M % M, q / (M * M)};
    double v = 0.0, x[3];
    for (int p = 0; p < M; ++p) v += R.G[qn[c]][p] * R.L[p][in[c]];
    for (int e = 0; e < DIM; ++e) {
      x[e] = R.x[qn[e]];
      v *= e == c ? R.w[qn[e]] : R.w[qn[e]] * R.L[qn[e]][in[e]];
    }
    sum += v * pressure_fn<M>(m, x);
  }
  for (int side = 0; side < 2; ++side) {
    if (!(faces >> (2 * c + side) & 1) || in[c] != (side ? M - 1 : 0)) continue;
    const int e1 = c == 0 ? 1 : 0, e2 = c == 2 ? 1 : 2;
    for (int q = 0; q < N / M; ++q) {
      const int q1 = q % M, q2 = q / M;
      double x[3], v = R.w[q1] * R.L[q1][in[e1]];
      x[c] = side ? 1.0 : -1.0;
      x[e1] = R.x[q1];
      if (DIM == 3) {
        x[e2] = R.x[q2];
        v *= R.w[q2] * R.L[q2][in[e2]];
      }
      sum -= (side ? 1.0 : -1.0) * v * pressure_fn<M>(m, x);
    }
  }
  table[t] = (T)(cf.sa[a] * cf.sc[c] * sum);
}

template <int M, typename T>
__device__ __forceinline__ void load_table_row(const T* __restrict__ p, T (&t)[kNPP<M>]) {
  constexpr int V = 16 / sizeof(T);
#pragma unroll
  for (int j = 0; j < kNPP<M> / V; ++j) {
    const int4 u = __ldg(reinterpret_cast<const int4*>(p) + j);
    memcpy(&t[V * j], &u, 16);
  }
}

// A component's part of a cell's pressure rows from its nodal values V; table: the component's rows.
template <int M, int N, typename T>
__device__ __forceinline__ void pressure_rows(const T* __restrict__ table, const T (&V)[N], T (&pp)[kNP<M>]) {
#pragma unroll
  for (int m = 0; m < kNP<M>; ++m) pp[m] = (T)0;
#pragma unroll
  for (int i = 0; i < N; ++i) {
    T t[kNPP<M>];
    load_table_row<M, T>(table + i * kNPP<M>, t);
#pragma unroll
    for (int m = 0; m < kNP<M>; ++m) pp[m] += t[m] * V[i];
  }
}

// The pressure's part of the component's nodal rows, added to V.
template <int M, int N, typename T>
__device__ __forceinline__ void add_pressure(const T* __restrict__ table, const T (&p)[kNP<M>], T (&V)[N]) {
#pragma unroll
  for (int i = 0; i < N; ++i) {
    T t[kNPP<M>];
    load_table_row<M, T>(table + i * kNPP<M>, t);
#pragma unroll
    for (int m = 0; m < kNP<M>; ++m) V[i] -= t[m] * p[m];
  }
}

// One cell, component (a, c): on entry V = nodal values of x, W of the linearisation velocity; on
// return V holds the cell's contribution to the nodal rows, without the pressure's.  sv, sw: Gauss-point
// values of all components, [a DIM + c][point][lane].  on: the lane has a cell; faces: its Dirichlet faces;
// nodal(i, b): the value of x at node i and Radau node b once more.  Contains one barrier of the CTA.
//
// The time coupling of order 4 goes from nodes to nodes by the 1D mass matrices: through the Gauss points, with
// four factors of L, its velocity rows had up to 1.2 times the rounding error of assembled ones (k = 1, Oseen; the
// mass term is the largest there).  It costs 50 -> 66 us a launch on 352 x 64.  For order 2 the Gauss points round less
// (FP32 emulation in 3D, k = 0: 4.6e-8 against 6.5e-8).
template <int DIM, int M, int NT, typename T, typename Nodal>
__device__ __forceinline__ void cell_operator(const MfCoef<T>& cf, int a, int c, unsigned faces, T (&V)[ipow(M, DIM)],
                                              T (&W)[ipow(M, DIM)], T* sv, T* sw, int lane, bool on, Nodal nodal) {
  const Ref<DIM, M, T>& R = c_ref<DIM, M, T>;
  constexpr int N = ipow(M, DIM);
  constexpr bool kNodalMass = M == 5;
  auto interp = [&](T(&u)[N]) {
#pragma unroll
    for (int e = 0; e < DIM; ++e) {
      const int st = e == 0 ? 1 : e == 1 ? M : M * M;
#pragma unroll
      for (int ln = 0; ln < N / M; ++ln) {
        const int o = (ln / st) * st * M + ln % st;
        T t[M];
#pragma unroll
        for (int q = 0; q < M; ++q) {
          t[q] = R.L[q][0] * u[o];
#pragma unroll
          for (int l = 1; l < M; ++l) t[q] += R.L[q][l] * u[o + l * st];
        }
#pragma unroll
        for (int q = 0; q < M; ++q) u[o + q * st] = t[q];
      }
    }
  };
  interp(V);
  interp(W);
  const int v0 = a * DIM + c;
#pragma unroll
  for (int q = 0; q < N; ++q) {
    sv[(v0 * N + q) * 32 + lane] = V[q];
    sw[(v0 * N + q) * 32 + lane] = W[q];
  }
  __syncthreads();
  T val[N], res[N];
  const T sa = cf.sa[a];
#pragma unroll
  for (int q = 0; q < N; ++q) {
    T t = (T)0;
    if constexpr (!kNodalMass) {
      t = cf.time[a][0] * sv[(c * N + q) * 32 + lane];
#pragma unroll
      for (int b = 1; b < NT; ++b) t += cf.time[a][b] * sv[((b * DIM + c) * N + q) * 32 + lane];
    }
    val[q] = t;
    res[q] = (T)0;
  }
#pragma unroll
  for (int e = 0; e < DIM; ++e) {
    const int st = e == 0 ? 1 : e == 1 ? M : M * M;
    const T sce = cf.sc[e];
#pragma unroll
    for (int ln = 0; ln < N / M; ++ln) {
      const int o = (ln / st) * st * M + ln % st;
      T F[M];
#pragma unroll
      for (int q = 0; q < M; ++q) {
        const int id = o + q * st;
        T dv = R.G[q][0] * V[o];
#pragma unroll
        for (int l = 1; l < M; ++l) dv += R.G[q][l] * V[o + l * st];
        dv *= sce * sa;
        T add = sw[((a * DIM + e) * N + id) * 32 + lane] * dv;
        if (cf.newton) {
          T dw = R.G[q][0] * W[o];
#pragma unroll
          for (int l = 1; l < M; ++l) dw += R.G[q][l] * W[o + l * st];
          add += sv[((a * DIM + e) * N + id) * 32 + lane] * (dw * (sce * sa));
        }
        val[id] += add;
        F[q] = R.wt[id] * sce * (cf.nu * dv);
      }
#pragma unroll
      for (int q = 0; q < M; ++q)
#pragma unroll
        for (int l = 0; l < M; ++l) res[o + l * st] += R.G[q][l] * F[q];
    }
  }
#pragma unroll
  for (int id = 0; id < N; ++id) {
    const T wt = R.wt[id];
    res[id] += wt * val[id];
  }
  // transposed interpolation
#pragma unroll
  for (int e = 0; e < DIM; ++e) {
    const int st = e == 0 ? 1 : e == 1 ? M : M * M;
#pragma unroll
    for (int ln = 0; ln < N / M; ++ln) {
      const int o = (ln / st) * st * M + ln % st;
      T t[M];
#pragma unroll
      for (int l = 0; l < M; ++l) {
        t[l] = R.L[0][l] * res[o];
#pragma unroll
        for (int q = 1; q < M; ++q) t[l] += R.L[q][l] * res[o + q * st];
      }
#pragma unroll
      for (int l = 0; l < M; ++l) res[o + l * st] = t[l];
    }
  }
#pragma unroll
  for (int q = 0; q < N; ++q) V[q] = res[q];
  if constexpr (kNodalMass) {
    T t[N];
#pragma unroll
    for (int i = 0; i < N; ++i) {
      t[i] = (T)0;
#pragma unroll
      for (int b = 0; b < NT; ++b) t[i] += cf.time[a][b] * (on ? nodal(i, b) : (T)0);
    }
#pragma unroll
    for (int e = 0; e < DIM; ++e) {
      const int st = e == 0 ? 1 : e == 1 ? M : M * M;
#pragma unroll
      for (int ln = 0; ln < N / M; ++ln) {
        const int o = (ln / st) * st * M + ln % st;
        T u[M];
#pragma unroll
        for (int q = 0; q < M; ++q) {
          u[q] = R.MM[q][0] * t[o];
#pragma unroll
          for (int l = 1; l < M; ++l) u[q] += R.MM[q][l] * t[o + l * st];
        }
#pragma unroll
        for (int q = 0; q < M; ++q) t[o + q * st] = u[q];
      }
    }
#pragma unroll
    for (int i = 0; i < N; ++i) V[i] += t[i];
  }
  // Nitsche's terms of the Dirichlet faces, in nodal values: the penalty gamma2 / h is large against the other
  // terms, and only the face's own rows may carry its rounding
  if (faces) {
    constexpr int F = N / M;  // nodes, or Gauss points, of a face
    auto interp_face = [&](T(&u)[F], bool transposed) {
#pragma unroll
      for (int e = 0; e < DIM - 1; ++e) {
        const int st = e == 0 ? 1 : M;
#pragma unroll
        for (int ln = 0; ln < F / M; ++ln) {
          const int o = (ln / st) * st * M + ln % st;
          T t[M];
#pragma unroll
          for (int q = 0; q < M; ++q) {
            t[q] = (T)0;
#pragma unroll
            for (int l = 0; l < M; ++l) t[q] += (transposed ? R.L[l][q] : R.L[q][l]) * u[o + l * st];
          }
#pragma unroll
          for (int q = 0; q < M; ++q) u[o + q * st] = t[q];
        }
      }
    };
#pragma unroll
    for (int f = 0; f < 2 * DIM; ++f) {
      if (!(faces >> f & 1u)) continue;
      const int e0 = f >> 1, s0 = f & 1, st = e0 == 0 ? 1 : e0 == 1 ? M : M * M;
      const T ns = s0 ? (T)1 : (T)-1, sn = ns * cf.sc[e0];
      T tr[F], dn[F];
#pragma unroll
      for (int k = 0; k < F; ++k) {
        const int o = (k / st) * st * M + k % st;  // first node of the line along the normal
        dn[k] = (T)0;
#pragma unroll
        for (int l = 0; l < M; ++l) {
          const T u = nodal(o + l * st, a);
          dn[k] += R.DN[s0][l] * u;
          if (l == (s0 ? M - 1 : 0)) tr[k] = u;
        }
      }
      interp_face(tr, false);
      interp_face(dn, false);
#pragma unroll
      for (int k = 0; k < F; ++k) {
        const int t0 = k % M, t1 = DIM == 3 ? k / M : 0;  // tangential Gauss points, lower direction first
        T wt = sa * cf.sc[e0] * R.w[t0];
        if (DIM == 3) wt *= R.w[t1];
        T A = cf.g1[e0] * tr[k] - cf.nu * sn * dn[k];
        if (e0 == c) A += cf.g2[e0] * tr[k];
        dn[k] = -cf.nu * sn * tr[k] * wt;
        tr[k] = A * wt;
      }
      interp_face(tr, true);
      interp_face(dn, true);
#pragma unroll
      for (int k = 0; k < F; ++k) {
        const int o = (k / st) * st * M + k % st;
#pragma unroll
        for (int l = 0; l < M; ++l) {
          T add = R.DN[s0][l] * dn[k];
          if (l == (s0 ? M - 1 : 0)) add += tr[k];
          V[o + l * st] += add;
        }
      }
    }
  }
}

// Dirichlet faces of a cell (bit 2 e + side).
template <int DIM>
__device__ __forceinline__ unsigned cell_faces(const Geom& g, int cx, int cy, int cz) {
  unsigned f = 0;
  const int cc[3] = {cx, cy, cz};
#pragma unroll
  for (int e = 0; e < DIM; ++e) {
    if (cc[e] == 0) f |= g.dirichlet & (1u << (2 * e));
    if (cc[e] == g.n[e] - 1) f |= g.dirichlet & (1u << (2 * e + 1));
  }
  return f;
}

// 2D, order 4 (which has no obstacle): one launch.  A CTA owns 31 cell columns by ty cell rows and walks up the rows; warp v = (a, c), lane =
// cell column, lane 0 the column left of the owned ones.  A node's sum over its cells is formed in
// registers: the right edge of the left neighbour comes by a shuffle, the top edge of the row below is
// kept from the previous step (the row below the owned ones is computed for that alone).  Bound by FP32
// issue; the repeated column and row cost 32/31 and (ty + 1)/ty.
template <int NT, typename T>
__global__ void __launch_bounds__(64 * NT, NT == 2 ? 3 : 2) mf_residual2d(Geom g, const MfCoef<T>* __restrict__ cfp,
                                                        const T* __restrict__ table, const T* __restrict__ w,
                                                        const T* __restrict__ x, const T* __restrict__ b,
                                                        T* __restrict__ out, int ty) {
  pdl_wait();
  const MfCoef<T>& cf = *cfp;
  constexpr int M = 5, N = M * M, R = M - 1, NV = 2 * NT, NP = kNP<M>;
  extern __shared__ __align__(16) unsigned char mf_smem[];
  T* sv = reinterpret_cast<T*>(mf_smem);
  T* sw = sv + NV * N * 32;
  T* sp = sw + NV * N * 32;  // [component][m][lane]
  const int lane = threadIdx.x, v = threadIdx.y, a = v >> 1, c = v & 1;
  const int cx = (int)blockIdx.x * 31 - 1 + lane, y0 = (int)blockIdx.y * ty;
  const int y1 = min(y0 + ty, g.n[1]);
  const bool col = cx >= 0 && cx < g.n[0], owned = col && lane > 0;
  const bool last_col = cx == g.n[0] - 1;
  T carry[M];
#pragma unroll
  for (int i = 0; i < M; ++i) carry[i] = (T)0;
  for (int cy = y0 > 0 ? y0 - 1 : 0; cy < y1; ++cy) {
    T V[N], W[N], P[NP], pp[NP];
    const long long n0 = ((long long)R * cy * g.nn[0] + R * cx) * NV + v;
    if (!col) {
#pragma unroll
      for (int i = 0; i < N; ++i) V[i] = W[i] = (T)0;
#pragma unroll
      for (int m = 0; m < NP; ++m) P[m] = (T)0;
    } else {
#pragma unroll
      for (int i = 0; i < N; ++i) {
        const long long o = n0 + ((long long)(i / M) * g.nn[0] + i % M) * NV;
        V[i] = x[o];
        W[i] = w[o];
      }
      const T* pc = x + g.nvel + ((long long)cy * g.n[0] + cx) * (NT * NP) + a * NP;
#pragma unroll
      for (int m = 0; m < NP; ++m) P[m] = pc[m];
    }
    const unsigned faces = col ? cell_faces<2>(g, cx, cy, 0) : 0u;
    const T* rows_c = table + ((a * 16 + faces) * 2 + c) * (N * kNPP<M>);
    pressure_rows<M, N, T>(rows_c, V, pp);
    __syncthreads();  // the cell row below has been read from shared memory
#pragma unroll
    for (int m = 0; m < NP; ++m) sp[(v * NP + m) * 32 + lane] = pp[m];
    cell_operator<2, M, NT, T>(cf, a, c, faces, V, W, sv, sw, lane, col, [&](int i, int b_) {
      return x[n0 + ((long long)(i / M) * g.nn[0] + i % M) * NV + 2 * (b_ - a)];
    });
    add_pressure<M, N, T>(rows_c, P, V);
    const bool write = cy >= y0;
    if (write && owned) {
      const long long o0 = g.nvel + ((long long)cy * g.n[0] + cx) * (NT * NP) + a * NP;
      for (int m = c; m < NP; m += 2) {
        const T s = sp[(2 * a * NP + m) * 32 + lane] + sp[((2 * a + 1) * NP + m) * 32 + lane];
        out[o0 + m] = b ? b[o0 + m] - s : s;
      }
    }
    // node rows R cy + iy; the top one of the last cell row as well
    const int rows = cy == g.n[1] - 1 ? M : R;
#pragma unroll
    for (int iy = 0; iy < M; ++iy) {
      if (iy >= rows) break;  // uniform
      T e[M];
#pragma unroll
      for (int ix = 0; ix < M; ++ix) e[ix] = V[iy * M + ix] + (iy == 0 ? carry[ix] : (T)0);
      const T left = __shfl_up_sync(0xffffffffu, e[R], 1);
      e[0] += left;
      if (write && owned) {
#pragma unroll
        for (int ix = 0; ix < M; ++ix) {
          if (ix == R && !last_col) break;
          const long long o = ((long long)(R * cy + iy) * g.nn[0] + R * cx + ix) * NV + v;
          out[o] = b ? b[o] - e[ix] : e[ix];
        }
      }
    }
#pragma unroll
    for (int ix = 0; ix < M; ++ix) carry[ix] = V[R * M + ix];
  }
}

// 3D: the cells' contributions E[(v, node)][cell] and the pressure rows, one thread per (cell, component);
// then mf_nodes3d sums each node's cells.  E takes 27 sizeof(T) bytes per cell and component: at 48^3, k = 1 72 MB in
// FP32, which mostly stays in L2, and 143 MB in FP64, which does not.
template <int NT, typename T>
__global__ void __launch_bounds__(96 * NT) mf_cells3d(Geom g, const MfCoef<T>* __restrict__ cfp,
                                                     const T* __restrict__ table, const T* __restrict__ w,
                                                     const T* __restrict__ x, const T* __restrict__ b,
                                                     T* __restrict__ E, T* __restrict__ out) {
  pdl_wait();
  const MfCoef<T>& cf = *cfp;
  constexpr int N = 27, NV = 3 * NT, NP = kNP<3>;
  extern __shared__ __align__(16) unsigned char mf_smem[];
  T* sv = reinterpret_cast<T*>(mf_smem);
  T* sw = sv + NV * N * 32;
  T* sp = sw + NV * N * 32;
  const int lane = threadIdx.x, v = threadIdx.y, a = v / 3, c = v - 3 * a;
  const long long cell = (long long)blockIdx.x * 32 + lane;
  const bool on = cell < g.n_cells;
  const int cx = (int)(cell % g.n[0]), cy = (int)((cell / g.n[0]) % g.n[1]);
  const int cz = (int)(cell / ((long long)g.n[0] * g.n[1]));
  T V[N], W[N], P[NP], pp[NP];
  const long long n0 = node_id(g, 2 * cx, 2 * cy, 2 * cz) * NV + v;
  if (on) {
#pragma unroll
    for (int i = 0; i < N; ++i) {
      const long long o = n0 + (i % 3 + (long long)g.nn[0] * ((i / 3) % 3 + (long long)g.nn[1] * (i / 9))) * NV;
      V[i] = x[o];
      W[i] = w[o];
    }
    const T* pc = x + g.nvel + cell * (NT * NP) + a * NP;
#pragma unroll
    for (int m = 0; m < NP; ++m) P[m] = pc[m];
  } else {
#pragma unroll
    for (int i = 0; i < N; ++i) V[i] = W[i] = (T)0;
#pragma unroll
    for (int m = 0; m < NP; ++m) P[m] = (T)0;
  }
  auto node = [&](int i) {
    return n0 + (i % 3 + (long long)g.nn[0] * ((i / 3) % 3 + (long long)g.nn[1] * (i / 9))) * NV;
  };
  const unsigned faces = on ? cell_faces<3>(g, cx, cy, cz) : 0u;
  const T* rows_c = table + ((a * 64 + faces) * 3 + c) * (N * kNPP<3>);
  pressure_rows<3, N, T>(rows_c, V, pp);
#pragma unroll
  for (int m = 0; m < NP; ++m) sp[(v * NP + m) * 32 + lane] = pp[m];
  cell_operator<3, 3, NT, T>(cf, a, c, faces, V, W, sv, sw, lane, on, [&](int i, int) { return x[node(i)]; });
  add_pressure<3, N, T>(rows_c, P, V);
  if (on) {
#pragma unroll
    for (int i = 0; i < N; ++i) E[((long long)v * N + i) * g.n_cells + cell] = V[i];
    const long long o0 = g.nvel + cell * (NT * NP) + a * NP;
    for (int m = c; m < NP; m += 3) {
      T s = (T)0;
#pragma unroll
      for (int d = 0; d < 3; ++d) s += sp[((3 * a + d) * NP + m) * 32 + lane];
      out[o0 + m] = b ? b[o0 + m] - s : s;
    }
  }
}

// 32 nodes along x by the NV components.
template <typename T>
__global__ void mf_nodes3d(Geom g, const T* __restrict__ E, const T* __restrict__ b, T* __restrict__ out) {
  pdl_wait();
  const int ix = (int)blockIdx.x * 32 + threadIdx.x, iy = blockIdx.y, iz = blockIdx.z, v = threadIdx.y;
  if (ix >= g.nn[0]) return;
  int xl, xh, yl, yh, zl, zh;
  node_cells(ix, g.n[0], xl, xh);
  node_cells(iy, g.n[1], yl, yh);
  node_cells(iz, g.n[2], zl, zh);
  T s = (T)0;
  for (int cz = zl; cz <= zh; ++cz)
    for (int cy = yl; cy <= yh; ++cy)
      for (int cx = xl; cx <= xh; ++cx) {
        const int i = (ix - 2 * cx) + 3 * (iy - 2 * cy) + 9 * (iz - 2 * cz);
        s += E[((long long)v * 27 + i) * g.n_cells + cell_id(g, cx, cy, cz)];
      }
  const long long o = node_id(g, ix, iy, iz) * g.NV + v;
  out[o] = b ? b[o] - s : s;
}

template <typename T>
MfCoef<T> coefficients(const Geom& g, const TimeData& td, const AsmCoef& cf) {
  MfCoef<T> m{};
  double det = 1.0;
  for (int e = 0; e < g.dim; ++e) {
    det *= g.h[e] / 2.0;
    m.sc[e] = (T)(2.0 / g.h[e]);
    m.g1[e] = (T)(cf.gamma1 * cf.nu / g.h[e]);
    m.g2[e] = (T)(cf.gamma2 / g.h[e]);
  }
  for (int a = 0; a < g.nt; ++a) {
    m.sa[a] = (T)(cf.tau * td.w[a] * det);
    for (int b = 0; b < g.nt; ++b) m.time[a][b] = (T)(td.T[a][b] * det);
  }
  m.nu = (T)cf.nu;
  m.newton = cf.newton;
  return m;
}

// At least two CTAs per SM of the 152 where the mesh has them, at most 16 rows a CTA.
constexpr int kMinCtas = 304;

template <int DIM, int M, typename T>
constexpr int pressure_table_values(int nt) {
  return nt * (1 << (2 * DIM)) * DIM * ipow(M, DIM) * kNPP<M>;
}
// The coefficients, then the pressure table.
constexpr size_t kTableOffset = (sizeof(MfCoef<double>) + 15) / 16 * 16;
template <typename T>
const T* table_of(const void* coef) {
  return reinterpret_cast<const T*>(static_cast<const char*>(coef) + kTableOffset);
}

template <int NT, typename T>
void run2d(const Geom& g, const void* coef, const T* w, const T* x, const T* b, T* out, cudaStream_t st) {
  constexpr int NV = 2 * NT;
  constexpr size_t smem = sizeof(T) * 32 * NV * (2 * 25 + kNP<5>);
  if (smem > 48 * 1024)
    STG_CUDA_OK(cudaFuncSetAttribute(mf_residual2d<NT, T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  const int nbx = (g.n[0] + 30) / 31;
  const int ty = std::max(1, std::min(16, (int)((long long)nbx * g.n[1] / kMinCtas)));
  launch_k(mf_residual2d<NT, T>, dim3(nbx, (g.n[1] + ty - 1) / ty), dim3(32, NV), smem, st, g, (const MfCoef<T>*)coef,
           table_of<T>(coef), w, x, b, out, ty);
}

template <int NT, typename T>
void run3d(const Geom& g, const void* coef, const T* w, const T* x, const T* b, T* E, T* out, cudaStream_t st) {
  constexpr size_t smem = sizeof(T) * 32 * (3 * NT) * (2 * 27 + kNP<3>);
  if (smem > 48 * 1024)
    STG_CUDA_OK(cudaFuncSetAttribute(mf_cells3d<NT, T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  launch_k(mf_cells3d<NT, T>, grid_for(g.n_cells, 32), dim3(32, 3 * NT), smem, st, g, (const MfCoef<T>*)coef,
           table_of<T>(coef), w, x, b, E, out);
  launch_k(mf_nodes3d<T>, dim3((g.nn[0] + 31) / 32, g.nn[1], g.nn[2]), dim3(32, 3 * NT), 0, st, g, E, b, out);
}

template <int DIM, int M, typename T>
void upload_coefficients(const Geom& g, const TimeData& td, const AsmCoef& cf, void* dst, cudaStream_t st) {
  const MfCoef<T> m = coefficients<T>(g, td, cf);
  STG_CUDA_OK(cudaMemcpyAsync(dst, &m, sizeof(m), cudaMemcpyHostToDevice, st));
  const int count = pressure_table_values<DIM, M, T>(g.nt);
  pressure_table<DIM, M, T><<<(count + 127) / 128, 128, 0, st>>>(count, coefficients<double>(g, td, cf),
                                                                const_cast<T*>(table_of<T>(dst)));
  STG_LAUNCH_OK();
}

}  // namespace
}  // namespace stg
