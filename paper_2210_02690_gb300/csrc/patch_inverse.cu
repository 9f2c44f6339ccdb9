// FP32 inverses of the larger local matrices J_K (Eq. (3.4)): 2D k >= 2, order 4, 3D.
#include <cooperative_groups.h>

#include <type_traits>

#include "common.cuh"
#include "kernels.cuh"

namespace stg {
namespace {

constexpr int KB = 8;  // columns of a warp = pivots of an elimination block

// Gauss-Jordan without row interchanges on the equilibrated J_K, in blocks of KB = 8 pivots: one
// CTA (CL = 1) or a cluster of two CTAs (CL = 2, each CTA half of the columns) per patch, the
// matrix in registers.  Warp W holds the 8 columns of block W for all rows, lane l rows l + 32 q (q < RB).
// The warp of a block eliminates its columns among themselves (shuffles alone) and publishes the
// multipliers G[j][r] of the 8 steps (f_r / pivot; (pivot - 1) / pivot on the pivot row); after one
// barrier every other warp applies the steps to its columns, a[r][c] -= G[j][r] q_j[c], j ascending, with
// q_j the pivot row of step j as it stands at that step (the steps before it applied to the 8 pivot
// rows first, one lane a column).  These are the operations and the order of an elimination step by
// step, so the result does not depend on the blocking; what the blocking changes is one barrier per 8
// steps and 8 RB KB FMAs from 8 (RB + 2) shared-memory reads between barriers.  The warp of the next
// block goes on to eliminate it before the barrier (G is double-buffered).  Rolled loops keep the body
// in the instruction cache: with the pivot steps and the gather unrolled (310 KB of code) it ran no
// faster than one barrier per pivot.
//
// The pivots need no interchange because the velocity unknowns come before the pressure unknowns of
// the saddle-point matrix; a pivot below 1e-3 (entries are O(1) after equilibration) flags the
// patch, and the pivoting kernel redoes it.
//
// Bound: FP32 issue (2 n^3 flops a patch) and, where one patch fills an SM (n = 170, 255: 32% of the issue
// slots, the rest barriers and the gather), the elimination of the next block, whose 8 steps are a serial
// chain of shuffles, a division and RB x 8 FMAs.  Measured over a level, against one barrier per pivot with
// 8 x 8 tiles a thread: 256^2 n = 63 10.8 -> 2.8 ms, n = 84 14.5 -> 6.0 ms; 352 x 64 n = 120 16.1 -> 5.0 ms;
// 48^3 n = 170 123 -> 73 ms; 24^3 n = 255 46 -> 27 ms.  Two CTAs a patch for n = 170 (so that two patches
// share an SM) took 89 ms, the cluster barriers costing more than the overlap gave.
template <int RB, int NW, int CL>
struct PanelShared {
  float G[2][KB][32 * RB];        // [buffer][step][row]
  float rows[NW][KB][KB];         // a warp's columns of the block's pivot rows: as they are, then q_j
  float rmax[CL][32 * RB];        // row maxima of each CTA's columns
  float rs[32 * RB], cs[CL * NW * KB];
  int4 row[32 * RB];              // velocity row: first slot, wx, wx wy, value v; pressure row: -1, time node, m
  int bad;
};

// a0 += g q0, a1 += g q1 as one packed instruction (two IEEE fused multiply-adds): half the issue slots.
__device__ __forceinline__ void fma2(float& a0, float& a1, float g, float q0, float q1) {
  asm("{\n\t.reg .b64 x, y, z;\n\t"
      "mov.b64 x, {%0, %1};\n\t"
      "mov.b64 y, {%2, %2};\n\t"
      "mov.b64 z, {%3, %4};\n\t"
      "fma.rn.f32x2 x, y, z, x;\n\t"
      "mov.b64 {%0, %1}, x;\n\t}"
      : "+f"(a0), "+f"(a1)
      : "f"(g), "f"(q0), "f"(q1));
}

// f(integral_constant<qb>), qb < RB
template <int RB, int Q = 0, typename F>
__device__ __forceinline__ void with_slot(int qb, F& f) {
  if constexpr (Q + 1 == RB) {
    f(std::integral_constant<int, Q>{});
  } else {
    if (qb == Q)
      f(std::integral_constant<int, Q>{});
    else
      with_slot<RB, Q + 1>(qb, f);
  }
}

// Eliminates the 8 columns of a warp whose pivot rows are slot QB of lanes l0 .. l0 + 7; the columns rotate
// by one a step, so that the pivot column is column 0.  The slot of the pivot rows goes first and the
// next pivot row is fetched before the other slots take their FMAs.
template <int RB, int CL, int QB, typename Sh>
__device__ __forceinline__ void eliminate_block(float (&a)[RB][KB], Sh* const (&at)[CL], int l0, int buf, int lane) {
  bool bad = false;
  float r[KB];
#pragma unroll
  for (int c = 0; c < KB; ++c) r[c] = __shfl_sync(0xffffffffu, a[QB][c], l0);
#pragma unroll 1
  for (int jj = 0; jj < KB; ++jj) {
    if (!(fabsf(r[0]) > 1e-3f) || isinf(r[0])) bad = true;
    const float inv = 1.f / r[0];
    auto step = [&](int q, bool piv) {
      const float f = a[q][0], gj = (piv ? f - 1.f : f) * inv;
#pragma unroll
      for (int k = 0; k < CL; ++k) at[k]->G[buf][jj][lane + 32 * q] = gj;
#pragma unroll
      for (int c = 1; c < KB; ++c) a[q][c - 1] = fmaf(-gj, r[c], a[q][c]);
      a[q][KB - 1] = piv ? inv : -gj;
    };
    step(QB, lane == l0 + jj);
    float nx[KB];
#pragma unroll
    for (int c = 0; c < KB; ++c) nx[c] = __shfl_sync(0xffffffffu, a[QB][c], l0 + ((jj + 1) & 7));
#pragma unroll
    for (int q = 0; q < RB; ++q)
      if (q != QB) step(q, false);
#pragma unroll
    for (int c = 0; c < KB; ++c) r[c] = nx[c];
  }
  if (bad && lane == 0) {
#pragma unroll
    for (int k = 0; k < CL; ++k) at[k]->bad = 1;
  }
}

template <int RB, int NW, int CL, int MINB, typename FT>
__global__ void __launch_bounds__(32 * NW, MINB)
    invert_panels_kernel(Geom g, const int* __restrict__ rowptr, const double* __restrict__ vv,
                         const double* __restrict__ vp, const double* __restrict__ pv, FT* __restrict__ jinv,
                         long long stride, int* __restrict__ flags) {
  namespace cg = cooperative_groups;
  static_assert(NW * KB * CL <= 32 * RB, "one row per column");
  using Sh = PanelShared<RB, NW, CL>;
  __shared__ __align__(16) Sh sh;
  extern __shared__ __align__(16) float gathered[];  // [warp][row][column of the warp]
  const int n = g.npatch, NV = g.NV, dim = g.dim, npd = g.npd, nt = g.nt, nloc = g.nloc, vel = nloc * NV;
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  int rank = 0;
  Sh* at[CL];  // the shared memory of every CTA of the cluster
  at[0] = &sh;
  if constexpr (CL > 1) {
    cg::cluster_group cl = cg::this_cluster();
    rank = (int)cl.block_rank();
#pragma unroll
    for (int k = 0; k < CL; ++k) at[k] = cl.map_shared_rank(&sh, k);
  }
  auto barrier = [&]() {
    if constexpr (CL > 1)
      cg::this_cluster().sync();
    else
      __syncthreads();
  };
  const int W = rank * NW + w;  // warp and block index over the cluster
  const long long p = blockIdx.x / CL;
  int cx, cy, cz;
  patch_cell(g, p, cx, cy, cz);
  if (CL == 1 && dim == 2 && cell_masked(g, cx, cy)) {  // removed cell: block-uniform early return
    write_patch_projector(g, cx, cy, jinv + p * stride, tid, 32 * NW);
    return;
  }
  const long long cell = cell_id(g, cx, cy, cz);
  const int r1 = g.r + 1;
  for (int row = tid; row < 32 * RB; row += 32 * NW) {
    int4 v = make_int4(-1, 0, 0, 0);
    if (row < vel) {
      const int i = row / NV;
      const int ix = g.r * cx + i % r1, iy = g.r * cy + (i / r1) % r1, iz = g.r * cz + i / (r1 * r1);
      int xl, xh, yl, yh;
      stencil_range(ix, g.nn[0], xl, xh, g.r);
      stencil_range(iy, g.nn[1], yl, yh, g.r);
      v = make_int4((int)bcsr_slot(g, rowptr, ix, iy, iz, g.r * cx, g.r * cy, g.r * cz), xh - xl + 1,
                    (xh - xl + 1) * (yh - yl + 1), row - i * NV);
    } else if (row < n) {
      v.y = (row - vel) / npd;
      v.z = row - vel - v.y * npd;
    }
    sh.row[row] = v;
  }
  if (tid == 0) sh.bad = 0;
  __syncthreads();

  // gather, rounded to FP32; the identity beyond n.  A warp loads 4 rows by its 8 columns at a time (a block
  // row's values are contiguous) and turns them through shared memory.
  float* mine = gathered + w * (RB * KB * 32);
  {
    const int col = W * KB + (lane & 7);
    const bool cvel = col < vel;
    const int j = cvel ? col / NV : 0, s = col - j * NV;  // velocity column: node j = (jx, jy, jz), value s
    const int jx = j % r1, jy = (j / r1) % r1, jz = j / (r1 * r1);
    const int tb = cvel ? s / dim : (col - vel) / npd, m = col - vel - tb * npd;  // time node; coefficient
#pragma unroll 8
    for (int t = 0; t < RB * KB; ++t) {
      const int row = 4 * t + (lane >> 3);
      const int4 ri = sh.row[row];
      float x = row == col ? 1.f : 0.f;
      if (cvel) {
        if (row < vel)
          x = (float)vv[((long long)(ri.x + jz * ri.z + jy * ri.y + jx) * NV + ri.w) * NV + s];
        else if (row < n)
          x = tb == ri.y ? (float)pv[((cell * nt + tb) * npd + ri.z) * (long long)nloc * dim + j * dim + s - tb * dim]
                         : 0.f;
      } else if (col < n) {
        if (row < vel)
          x = ri.w / dim == tb ? (float)vp[(cell * vel + row) * npd + m] : 0.f;
        else if (row < n)
          x = 0.f;
      }
      mine[t * 32 + lane] = x;
    }
  }
  __syncwarp();
  float a[RB][KB];
#pragma unroll
  for (int q = 0; q < RB; ++q) {
    const float4 lo = *reinterpret_cast<const float4*>(mine + (lane + 32 * q) * KB);
    const float4 hi = *reinterpret_cast<const float4*>(mine + (lane + 32 * q) * KB + 4);
    a[q][0] = lo.x;
    a[q][1] = lo.y;
    a[q][2] = lo.z;
    a[q][3] = lo.w;
    a[q][4] = hi.x;
    a[q][5] = hi.y;
    a[q][6] = hi.z;
    a[q][7] = hi.w;
  }
  // equilibration: row scales over all columns, then column scales of the row-scaled matrix.  The
  // row maxima of the warps are combined in shared memory (as unsigned: non-negative floats order
  // like their bits)
  for (int i = tid; i < 32 * RB; i += 32 * NW)
    for (int k = 0; k < CL; ++k) sh.rmax[k][i] = 0.f;
  barrier();
#pragma unroll
  for (int q = 0; q < RB; ++q) {
    float mx = 0.f;
#pragma unroll
    for (int c = 0; c < KB; ++c) mx = fmaxf(mx, fabsf(a[q][c]));
    atomicMax(reinterpret_cast<unsigned*>(&sh.rmax[rank][lane + 32 * q]), __float_as_uint(mx));
  }
  if constexpr (CL > 1) {
    __syncthreads();
    for (int i = tid; i < 32 * RB; i += 32 * NW)
#pragma unroll
      for (int k = 0; k < CL; ++k)
        if (k != rank) at[k]->rmax[rank][i] = sh.rmax[rank][i];
  }
  barrier();
  for (int i = tid; i < 32 * RB; i += 32 * NW) {
    float mx = sh.rmax[0][i];
#pragma unroll
    for (int k = 1; k < CL; ++k) mx = fmaxf(mx, sh.rmax[k][i]);
    sh.rs[i] = mx > 0.f ? 1.f / mx : 1.f;
  }
  __syncthreads();
#pragma unroll
  for (int q = 0; q < RB; ++q) {
    const float rs = sh.rs[lane + 32 * q];
#pragma unroll
    for (int c = 0; c < KB; ++c) a[q][c] *= rs;
  }
#pragma unroll
  for (int c = 0; c < KB; ++c) {
    float mx = 0.f;
#pragma unroll
    for (int q = 0; q < RB; ++q) mx = fmaxf(mx, fabsf(a[q][c]));
    mx = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(mx)));
    const float cs = mx > 0.f ? 1.f / mx : 1.f;
#pragma unroll
    for (int q = 0; q < RB; ++q) a[q][c] *= cs;
    if (lane == 0) {
#pragma unroll
      for (int k = 0; k < CL; ++k) at[k]->cs[W * KB + c] = cs;
    }
  }
  // every CTA of a cluster is past the scales before G is written into its shared memory
  barrier();

  // block cb's pivot rows: slot cb / 4 of lanes 8 (cb % 4) .. + 7.  Step -1 only starts the chain.
  for (int cb = -1; cb * KB < n; ++cb) {
    const int buf = cb & 1, nb = cb + 1;
    if (cb >= 0) {
      barrier();
      if (W != cb) {
        // the steps before step j applied to its pivot row: lane = column
        float* rows = &sh.rows[w][0][0];
        if (lane < KB) {
          float q[KB];
#pragma unroll
          for (int j = 0; j < KB; ++j) q[j] = rows[j * KB + lane];
#pragma unroll
          for (int i = 0; i + 1 < KB; ++i) {
            const float4 lo = *reinterpret_cast<const float4*>(&sh.G[buf][i][cb * KB]);
            const float4 hi = *reinterpret_cast<const float4*>(&sh.G[buf][i][cb * KB + 4]);
            const float gi[KB] = {lo.x, lo.y, lo.z, lo.w, hi.x, hi.y, hi.z, hi.w};
#pragma unroll
            for (int j = i + 1; j < KB; ++j) q[j] = fmaf(-gi[j], q[i], q[j]);
          }
#pragma unroll
          for (int j = 1; j < KB; ++j) rows[j * KB + lane] = q[j];
        }
        __syncwarp();
#pragma unroll
        for (int j = 0; j < KB; ++j) {
          const float4 lo = *reinterpret_cast<const float4*>(rows + j * KB);
          const float4 hi = *reinterpret_cast<const float4*>(rows + j * KB + 4);
#pragma unroll
          for (int q = 0; q < RB; ++q) {
            const float gj = sh.G[buf][j][lane + 32 * q];
            fma2(a[q][0], a[q][1], -gj, lo.x, lo.y);
            fma2(a[q][2], a[q][3], -gj, lo.z, lo.w);
            fma2(a[q][4], a[q][5], -gj, hi.x, hi.y);
            fma2(a[q][6], a[q][7], -gj, hi.z, hi.w);
          }
        }
        __syncwarp();
      }
    }
    if (nb * KB >= n) break;  // uniform
    const int qb = nb >> 2, l0 = (nb & 3) * KB, nbuf = nb & 1;
    // one branch a block picks the slot of its pivot rows; inside, register indices are constants
    if (W == nb) {
      auto eliminate = [&](auto Q) { eliminate_block<RB, CL, decltype(Q)::value>(a, at, l0, nbuf, lane); };
      with_slot<RB>(qb, eliminate);
    } else if ((lane >> 3) == (nb & 3)) {
      float4* o = reinterpret_cast<float4*>(&sh.rows[w][lane & 7][0]);
      auto publish = [&](auto Q) {
        constexpr int q = decltype(Q)::value;
        o[0] = make_float4(a[q][0], a[q][1], a[q][2], a[q][3]);
        o[1] = make_float4(a[q][4], a[q][5], a[q][6], a[q][7]);
      };
      with_slot<RB>(qb, publish);
    }
    __syncwarp();
  }
  // sh.bad was last written before the last block's barrier; no CTA of a cluster may leave
  // while another can still address its shared memory
  barrier();
  if (sh.bad) {
    if (tid == 0 && rank == 0) flags[p] = 1;
    return;
  }
  // J_K^{-1} = Dc A'^{-1} Dr, column-major: element (row, col) at col * n + row
  FT* out = jinv + p * stride;
#pragma unroll
  for (int c = 0; c < KB; ++c) {
    const int col = W * KB + c;
    if (col >= n) continue;
    const float rc = sh.rs[col];
#pragma unroll
    for (int q = 0; q < RB; ++q) {
      const int row = lane + 32 * q;
      if (row < n) out[(long long)col * n + row] = cvt<FT>(a[q][c] * sh.cs[row] * rc);
    }
  }
}

template <int RB, int NW, int CL, int MINB, typename FT>
void launch(const Geom& g, const int* rowptr, const double* vv, const double* vp, const double* pv, FT* jinv,
            long long stride, int* flags, cudaStream_t st) {
  STG_CUDA_OK(cudaMemsetAsync(flags, 0, sizeof(int) * g.n_cells, st));
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)(CL * g.n_cells));
  cfg.blockDim = dim3(32 * NW);
  cfg.dynamicSmemBytes = sizeof(float) * NW * RB * KB * 32;
  const auto kern = invert_panels_kernel<RB, NW, CL, MINB, FT>;
  STG_CUDA_OK(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)cfg.dynamicSmemBytes));
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = CL;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = CL > 1 ? 1 : 0;
  STG_CUDA_OK(cudaLaunchKernelEx(&cfg, kern, g, rowptr, vv, vp, pv, jinv, stride, flags));
  STG_LAUNCH_OK();
}

}  // namespace

template <typename FT>
bool invert_panels(const Geom& g, const int* rowptr, const double* vv, const double* vp, const double* pv, FT* jinv,
                   long long stride, int* flags, cudaStream_t st) {
  switch (g.npatch) {
    case 60:   // order 4, k = 0
    case 63:   // 2D k = 2
      launch<2, 8, 1, 5, FT>(g, rowptr, vv, vp, pv, jinv, stride, flags, st);
      return true;
    case 84:   // 2D k = 3
    case 85:   // 3D k = 0
      launch<3, 11, 1, 3, FT>(g, rowptr, vv, vp, pv, jinv, stride, flags, st);
      return true;
    case 105:  // 2D k = 4
      launch<4, 14, 1, 2, FT>(g, rowptr, vv, vp, pv, jinv, stride, flags, st);
      return true;
    case 120:  // order 4, k = 1
      launch<4, 15, 1, 2, FT>(g, rowptr, vv, vp, pv, jinv, stride, flags, st);
      return true;
    case 170:  // 3D k = 1
      launch<6, 22, 1, 1, FT>(g, rowptr, vv, vp, pv, jinv, stride, flags, st);
      return true;
    case 180:  // order 4, k = 2
      launch<6, 23, 1, 1, FT>(g, rowptr, vv, vp, pv, jinv, stride, flags, st);
      return true;
    case 255:  // 3D k = 2: more registers than one CTA has (no 2D patch has this size, so no removed cells)
      launch<8, 16, 2, 1, FT>(g, rowptr, vv, vp, pv, jinv, stride, flags, st);
      return true;
    default: return false;
  }
}

template bool invert_panels<float>(const Geom&, const int*, const double*, const double*, const double*, float*,
                                   long long, int*, cudaStream_t);
template bool invert_panels<__nv_bfloat16>(const Geom&, const int*, const double*, const double*, const double*,
                                           __nv_bfloat16*, long long, int*, cudaStream_t);
template <>
bool invert_panels<double>(const Geom&, const int*, const double*, const double*, const double*, double*, long long,
                           int*, cudaStream_t) {
  return false;
}

}  // namespace stg
