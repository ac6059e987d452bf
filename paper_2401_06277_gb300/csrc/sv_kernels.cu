// sv_kernels.cu -- stencil kernels of the hot path on sm_103a, templated on
// the element type (double for the FP64 form and for FGMRES, float inside the
// mixed-precision preconditioner):
//   matrix-free Stokes operator / residual   (Section 2.2, Algorithm 1 residual)
//   FE restriction P^T and prolongation P    (Section 3, Algorithm 1)
//   precision conversions
// and, in FP64 only: right-hand side assembly and its transpose (Section 2.2)
// and the dense coarse solve (Algorithm 1, level 0).
#include <cuda_runtime.h>

#include "sv_internal.h"
#include "sv_level_ops.cuh"
#include "sv_stencil.cuh"

namespace sv {
namespace {

using ops::is_free;

template <typename T>
__global__ void k_apply(LevelDev L, const T* __restrict__ x, const T* __restrict__ b,
                        T* __restrict__ y, int residual) {
  pdl_begin();
  const int a = blockIdx.x * blockDim.x + threadIdx.x;
  const int bb = blockIdx.y * blockDim.y + threadIdx.y;
  if (a > L.n || bb > L.n) return;
  ops::apply_vertex<T>(L, x, b, y, residual, a, bb);
}

// ---------------------------------------------------------------------------
// Right-hand side b = [M f - L_{.,D} u_D ; u_D on D ; -B_{.,D} u_D].
// ---------------------------------------------------------------------------
// One vertex (a, bb): the four Q2 nodes (2a + PI, 2bb + PJ) of both components.
// b = (h/30)^2 (m (x) m) f on free rows, minus nu/90 (k (x) m + m (x) k) u_D over
// the Dirichlet columns (MASK: vertices within two of the boundary only), and
// b = u_D on Dirichlet rows.  The 6 x 6 f (and u_D) neighbourhood of each
// component is read once; coefficients are compile-time constants.
template <bool MASK>
__device__ __forceinline__ void rhs_vertex(const LevelDev& L, const double* __restrict__ f,
                                           const double* __restrict__ ud, double* __restrict__ b, int a,
                                           int bb) {
  const int nq = L.nq;
  const long long nv = L.nv;
  const int I0 = 2 * a, J0 = 2 * bb;
  const double cm = (L.h / 30.0) * (L.h / 30.0), cl = L.nu / 90.0;
#pragma unroll
  for (int c = 0; c < 2; ++c) {
    double F[6][6], U[6][6];
#pragma unroll
    for (int r = 0; r < 6; ++r)
#pragma unroll
      for (int q = 0; q < 6; ++q) {
        const int I = I0 - 2 + q, J = J0 - 2 + r;
        const bool in = !MASK || (I >= 0 && J >= 0 && I < nq && J < nq);
        const long long k = c * nv + static_cast<long long>(J) * nq + I;
        F[r][q] = in ? f[k] : 0.0;
        U[r][q] = (MASK && in && !is_free(I, J, nq)) ? ud[k] : 0.0;
      }
#pragma unroll
    for (int PJ = 0; PJ < 2; ++PJ) {
#pragma unroll
      for (int PI = 0; PI < 2; ++PI) {
        const int I = I0 + PI, J = J0 + PJ;
        if (MASK && (I >= nq || J >= nq)) continue;
        const long long k = c * nv + static_cast<long long>(J) * nq + I;
        if (MASK && !is_free(I, J, nq)) {
          b[k] = ud[k];
          continue;
        }
        double sm = 0.0, sl = 0.0;
#pragma unroll
        for (int dJ = -2; dJ <= 2; ++dJ)
#pragma unroll
          for (int dI = -2; dI <= 2; ++dI) {
            const double mm = m1(PI, dI) * m1(PJ, dJ);
            if (mm != 0.0) sm = fma(mm, F[PJ + dJ + 2][PI + dI + 2], sm);
            if (MASK) {
              const double cf = k1(PI, dI) * m1(PJ, dJ) + m1(PI, dI) * k1(PJ, dJ);
              if (cf != 0.0) sl = fma(cf, U[PJ + dJ + 2][PI + dI + 2], sl);
            }
          }
        b[k] = cm * sm - cl * sl;
      }
    }
  }
}

__global__ void k_rhs_vel(LevelDev L, const double* __restrict__ f, const double* __restrict__ ud,
                          double* __restrict__ b) {
  pdl_begin();
  const int a = blockIdx.x * blockDim.x + threadIdx.x;
  const int bb = blockIdx.y * blockDim.y + threadIdx.y;
  const int n = L.n;
  if (a > n || bb > n) return;
  if (a >= 2 && a <= n - 2 && bb >= 2 && bb <= n - 2)
    rhs_vertex<false>(L, f, ud, b, a, bb);
  else
    rhs_vertex<true>(L, f, ud, b, a, bb);
}

__global__ void k_rhs_p(LevelDev L, const double* __restrict__ ud, double* __restrict__ b) {
  pdl_begin();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const int j = blockIdx.y * blockDim.y + threadIdx.y;
  const int nq = L.nq, np = L.np, n = L.n;
  if (i >= np || j >= np) return;
  const long long nv = L.nv;
  // -B_{.,D} u_D with B = -(C (x) N) h for u_x, -(N (x) C) h for u_y
  double s = 0.0;
  for (int J = 2 * j - 2; J <= 2 * j + 2; ++J) {
    if (J < 0 || J >= nq) continue;
    for (int I = 2 * i - 2; I <= 2 * i + 2; ++I) {
      if (I < 0 || I >= nq || is_free(I, J, nq)) continue;
      const long long kk = static_cast<long long>(J) * nq + I;
      s += c1_full(i, I, n) * n1_full(j, J, n) * ud[kk];
      s += n1_full(i, I, n) * c1_full(j, J, n) * ud[nv + kk];
    }
  }
  b[2 * nv + static_cast<long long>(j) * np + i] = L.h * s;
}

// grad_f = R^T lambda: sum over free velocity rows k of (M)_{k,(I,J)} lambda_k.
__global__ void k_rhs_transpose(LevelDev L, const double* __restrict__ lam, double* __restrict__ g) {
  pdl_begin();
  const int I = blockIdx.x * blockDim.x + threadIdx.x;
  const int J = blockIdx.y * blockDim.y + threadIdx.y;
  const int nq = L.nq;
  if (I >= nq || J >= nq) return;
  const long long nv = L.nv;
  double sx = 0.0, sy = 0.0;
  for (int dJ = -2; dJ <= 2; ++dJ) {
    const int J2 = J + dJ;
    for (int dI = -2; dI <= 2; ++dI) {
      const int I2 = I + dI;
      if (!is_free(I2, J2, nq)) continue;
      // M is symmetric: M_{(I2,J2),(I,J)} = row of (I2,J2) at offset (-dI, -dJ)
      const double mm = m1(I2, -dI) * m1(J2, -dJ);
      const long long kk = static_cast<long long>(J2) * nq + I2;
      sx = fma(mm, lam[kk], sx);
      sy = fma(mm, lam[nv + kk], sy);
    }
  }
  const double cm = (L.h / 30.0) * (L.h / 30.0);
  const long long k = static_cast<long long>(J) * nq + I;
  g[k] = cm * sx;
  g[nv + k] = cm * sy;
}

// Restriction r_c = P^T r_f and prolongation x_f += P e_c (the weights: sv_level_ops.cuh).
// On the larger levels a thread walks up ROWS coarse rows, so that the row pass of a
// fine (coarse) node row is done once instead of by every output row that takes it, and
// symmetric taps are added before they are weighted.  Both kernels are bound by the FP64
// pipe in FP64: 90 operations per coarse element instead of 153 in the restriction.
// 2048^2 -> 1024^2 in FP64, against one thread per coarse element: restriction 287 -> 180
// us, prolongation 303 -> 210 us (0.38 and 0.68 GB moved: 56 and 101 us at the copy rate).
constexpr int MARCH_ROWS = 4;

// even node: v3 + 3/8 (v2 + v4) - 1/8 (v0 + v6); odd node: v5 + 3/4 (v4 + v6)
template <typename T>
__device__ __forceinline__ T rw_even(T v0, T v2, T v3, T v4, T v6) {
  return fma(T(-0.125), v0 + v6, fma(T(0.375), v2 + v4, v3));
}
template <typename T>
__device__ __forceinline__ T rw_odd(T v4, T v5, T v6) { return fma(T(0.75), v4 + v6, v5); }

// One thread per coarse element column ex (0..nc) and component c (2: the pressure).
template <typename T>
__global__ void __launch_bounds__(128) k_restrict_march(LevelDev F, LevelDev C, const T* __restrict__ rf,
                                                        T* __restrict__ rc) {
  pdl_begin();
  const int ex = blockIdx.x * blockDim.x + threadIdx.x, ey0 = blockIdx.y * MARCH_ROWS, c = blockIdx.z;
  if (ex > C.n) return;
  const int ey1 = min(ey0 + MARCH_ROWS, C.np), fq = F.nq, cq = C.nq;
  if (c == 2) {
    const T* pf = rf + 2 * F.nv;
    auto prow = [&](int fj) -> T {   // (1/2, 1, 1/2) along fine vertex row fj
      if (fj < 0 || fj >= F.np) return T(0);
      const T* p = pf + static_cast<long long>(fj) * F.np + 2 * ex;
      const T l = ex > 0 ? p[-1] : T(0), r = 2 * ex + 1 < F.np ? p[1] : T(0);
      return fma(T(0.5), l + r, p[0]);
    };
    T below = prow(2 * ey0 - 1);
    for (int ey = ey0; ey < ey1; ++ey) {
      const T at = prow(2 * ey), above = prow(2 * ey + 1);
      rc[2 * C.nv + static_cast<long long>(ey) * C.np + ex] = fma(T(0.5), below + above, at);
      below = above;
    }
    return;
  }
  const T* r = rf + c * F.nv;
  const int F0 = 4 * ex - 3;
  T H[7][2];   // fine rows 4 ey - 3 .. 4 ey + 3, coarse columns 2 ex, 2 ex + 1
  auto row = [&](int J, T (&h)[2]) {
    T v[7];
#pragma unroll
    for (int k = 0; k < 7; ++k)
      v[k] = (k != 1 && is_free(F0 + k, J, fq)) ? r[static_cast<long long>(J) * fq + F0 + k] : T(0);
    h[0] = rw_even(v[0], v[2], v[3], v[4], v[6]);
    h[1] = rw_odd(v[4], v[5], v[6]);
  };
#pragma unroll
  for (int k = 0; k < 3; ++k) row(4 * ey0 - 3 + k, H[k]);
  for (int ey = ey0; ey < ey1; ++ey) {
#pragma unroll
    for (int k = 3; k < 7; ++k) row(4 * ey - 3 + k, H[k]);
#pragma unroll
    for (int g = 0; g < 2; ++g) {
      const int I = 2 * ex + g;
      if (I >= cq) continue;
      T* o = rc + c * C.nv + static_cast<long long>(2 * ey) * cq + I;
      o[0] = is_free(I, 2 * ey, cq) ? rw_even(H[0][g], H[2][g], H[3][g], H[4][g], H[6][g]) : T(0);
      if (2 * ey + 1 < cq) o[cq] = is_free(I, 2 * ey + 1, cq) ? rw_odd(H[4][g], H[5][g], H[6][g]) : T(0);
#pragma unroll
      for (int k = 0; k < 3; ++k) H[k][g] = H[k + 4][g];
    }
  }
}

// One thread per pair of fine node columns (2 q, 2 q + 1), q in 0..2 nc, of component c (2:
// the fine vertex column q of the pressure): the even column is a coarse column, the odd
// one takes (3/8, 3/4, -1/8) or its mirror image.  Coarse rows per thread by size, since a
// smaller level is bound by the chain of read-modify-writes of a thread, a larger one by
// the FP64 pipe; FP64, 1 / 2 / 4 rows (us): to 2048^2 230 / 216 / 210, to 1024^2 60.6 / 56.9
// / 57.9, to 512^2 18.3 / 19.1 / 21.8, to 256^2 7.8 / 8.1 / 12.8.  The restriction only
// reads along its chain: 4 rows are the best (2 within 2%) from 512^2 on.
template <typename T>
__global__ void __launch_bounds__(128) k_prolong_march(LevelDev F, LevelDev C, const T* __restrict__ ec,
                                                       T* __restrict__ xf, int rows) {
  pdl_begin();
  const int q = blockIdx.x * blockDim.x + threadIdx.x, ey0 = blockIdx.y * rows, c = blockIdx.z;
  if (q > F.n) return;
  const int ey1 = min(ey0 + rows, C.np), fq = F.nq, cq = C.nq, ex = q >> 1;
  if (c == 2) {
    const T* e = ec + 2 * C.nv + ex;
    T* x = xf + 2 * F.nv + q;
    const bool odd = q & 1;
    auto at = [&](int j) -> T {   // fine vertex column q on coarse row j
      if (j > C.n) return T(0);
      const T* p = e + static_cast<long long>(j) * C.np;
      return odd ? T(0.5) * (p[0] + p[1]) : p[0];
    };
    T h0 = at(ey0);
    for (int ey = ey0; ey < ey1; ++ey) {
      const T h1 = at(ey + 1);
      x[static_cast<long long>(2 * ey) * F.np] += h0;
      if (ey < C.n) x[static_cast<long long>(2 * ey + 1) * F.np] += T(0.5) * (h0 + h1);
      h0 = h1;
    }
    return;
  }
  const T* e = ec + c * C.nv;
  T* x = xf + c * F.nv + 2 * q;
  const bool right = q & 1;   // fine columns 4 ex + 2, 4 ex + 3
  const T w0 = right ? T(-0.125) : T(0.375), w2 = right ? T(0.375) : T(-0.125);
  auto row = [&](int J, T (&h)[2]) {
    T v[3];
#pragma unroll
    for (int g = 0; g < 3; ++g)
      v[g] = is_free(2 * ex + g, J, cq) ? e[static_cast<long long>(J) * cq + 2 * ex + g] : T(0);
    h[0] = right ? v[1] : v[0];
    h[1] = fma(w2, v[2], fma(T(0.75), v[1], w0 * v[0]));
  };
  T H0[2], H1[2], H2[2];
  row(2 * ey0, H0);
  for (int ey = ey0; ey < ey1; ++ey) {
    row(2 * ey + 1, H1);
    row(2 * ey + 2, H2);
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const int I = 2 * q + k;
#pragma unroll
      for (int f = 0; f < 4; ++f) {
        const int J = 4 * ey + f;
        if (!is_free(I, J, fq)) continue;
        T* o = x + static_cast<long long>(J) * fq + k;
        const T v = *o;
        *o = f == 0 ? v + H0[k]
           : f == 2 ? v + H1[k]
           : f == 1 ? fma(T(-0.125), H2[k], fma(T(0.75), H1[k], fma(T(0.375), H0[k], v)))
                    : fma(T(0.375), H2[k], fma(T(0.75), H1[k], fma(T(-0.125), H0[k], v)));
      }
      H0[k] = H2[k];
    }
  }
}

// One output per thread (small levels; sv_level_ops.cuh): a warp takes one output kind
// of 32 consecutive cells, block.x = 32, output kind = blockIdx.y.
template <typename T>
__global__ void __launch_bounds__(32) k_apply_out(LevelDev L, const T* __restrict__ x, const T* __restrict__ b,
                                                  T* __restrict__ y, int residual) {
  pdl_begin();
  const int k = blockIdx.x * 32 + threadIdx.x;
  if (k >= L.np * L.np) return;
  const int bb = k / L.np, a = k - bb * L.np;
  switch (blockIdx.y) {
    case 0: ops::apply_out<T, 0, 0, 0>(L, x, b, y, residual, a, bb); break;
    case 1: ops::apply_out<T, 0, 0, 1>(L, x, b, y, residual, a, bb); break;
    case 2: ops::apply_out<T, 0, 1, 0>(L, x, b, y, residual, a, bb); break;
    case 3: ops::apply_out<T, 0, 1, 1>(L, x, b, y, residual, a, bb); break;
    case 4: ops::apply_out<T, 1, 0, 0>(L, x, b, y, residual, a, bb); break;
    case 5: ops::apply_out<T, 1, 0, 1>(L, x, b, y, residual, a, bb); break;
    case 6: ops::apply_out<T, 1, 1, 0>(L, x, b, y, residual, a, bb); break;
    case 7: ops::apply_out<T, 1, 1, 1>(L, x, b, y, residual, a, bb); break;
    default: ops::apply_out<T, 2, 0, 0>(L, x, b, y, residual, a, bb); break;
  }
}

template <typename T>
__global__ void __launch_bounds__(32) k_restrict_out(LevelDev F, LevelDev C, const T* __restrict__ rf,
                                                     T* __restrict__ rc) {
  pdl_begin();
  const int k = blockIdx.x * 32 + threadIdx.x;
  if (k >= C.np * C.np) return;
  const int ey = k / C.np, ex = k - ey * C.np;
  switch (blockIdx.y) {
    case 0: ops::restrict_out<T, 0, 0, 0>(F, C, rf, rc, ex, ey); break;
    case 1: ops::restrict_out<T, 0, 0, 1>(F, C, rf, rc, ex, ey); break;
    case 2: ops::restrict_out<T, 0, 1, 0>(F, C, rf, rc, ex, ey); break;
    case 3: ops::restrict_out<T, 0, 1, 1>(F, C, rf, rc, ex, ey); break;
    case 4: ops::restrict_out<T, 1, 0, 0>(F, C, rf, rc, ex, ey); break;
    case 5: ops::restrict_out<T, 1, 0, 1>(F, C, rf, rc, ex, ey); break;
    case 6: ops::restrict_out<T, 1, 1, 0>(F, C, rf, rc, ex, ey); break;
    case 7: ops::restrict_out<T, 1, 1, 1>(F, C, rf, rc, ex, ey); break;
    default: ops::restrict_out<T, 2, 0, 0>(F, C, rf, rc, ex, ey); break;
  }
}

// blockIdx.y: 0..31 = component * 16 + fy * 4 + fx, 32..35 = the fine vertices
template <typename T, int K>
__device__ __forceinline__ void prolong_case(const LevelDev& F, const LevelDev& C, const T* ec, T* xf, int ex, int ey,
                                             int kind) {
  if constexpr (K < 36) {
    if (kind == K) {
      if constexpr (K < 32) ops::prolong_out<T, (K >> 4), ((K >> 2) & 3), (K & 3)>(F, C, ec, xf, ex, ey);
      else ops::prolong_out<T, 2, (K >> 1) & 1, K & 1>(F, C, ec, xf, ex, ey);
    } else {
      prolong_case<T, K + 1>(F, C, ec, xf, ex, ey, kind);
    }
  }
}

template <typename T>
__global__ void __launch_bounds__(32) k_prolong_out(LevelDev F, LevelDev C, const T* __restrict__ ec,
                                                    T* __restrict__ xf) {
  pdl_begin();
  const int k = blockIdx.x * 32 + threadIdx.x;
  if (k >= C.np * C.np) return;
  const int ey = k / C.np, ex = k - ey * C.np;
  prolong_case<T, 0>(F, C, ec, xf, ex, ey, blockIdx.y);
}

template <typename TI, typename TO>
__global__ void k_convert(const TI* __restrict__ in, TO* __restrict__ out, long long N) {
  pdl_begin();
  for (long long i = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x; i < N;
       i += static_cast<long long>(gridDim.x) * blockDim.x)
    out[i] = static_cast<TO>(in[i]);
}

// e = G r, G dense N0 x N0: one warp per row, lanes along the row (coalesced),
// summed by a fixed shuffle tree (deterministic)
__global__ void k_coarse(const double* __restrict__ G, int N0, const double* __restrict__ r,
                         double* __restrict__ e) {
  pdl_begin();
  const int row = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (row >= N0) return;
  const double s = ops::coarse_row<double>(G, N0, r, row, lane);
  if (lane == 0) e[row] = s;
}

// Levels whose FP32 operator and transfers run one output per thread.  At np = 129 the operator
// has 4680 such warps for 608 sub-partitions; above, a thread per vertex fills them.  The
// prolongation's 36 outputs per coarse element fill them from half that size.
constexpr int OUT_MAX_NP = 129;
dim3 out_grid(int np, int kinds) { return dim3((np * np + 31) / 32, kinds); }

dim3 grid2(int nx, int ny, dim3 blk) {
  return dim3((nx + blk.x - 1) / blk.x, (ny + blk.y - 1) / blk.y);
}

}  // namespace

template <typename T>
void launch_apply(const LevelDev& L, const T* x, const T* b, T* y, int residual, cudaStream_t s) {
  const bool tc64 = sizeof(T) == 8 && L.op_digits != nullptr;
  if (!tc64) count_launches(1);
  if constexpr (sizeof(T) == 8) {   // FP64: up to the size from which on the contraction is faster (OP_TC64_MIN_N)
    if (tc64) launch_apply_tc64(L, x, residual ? b : nullptr, y, s);
    else launch_pdl(k_apply_out<T>, out_grid(L.np, 9), dim3(32), 0, s, L, x, b, y, residual);
  } else if (L.np <= OUT_MAX_NP) {
    launch_pdl(k_apply_out<T>, out_grid(L.np, 9), dim3(32), 0, s, L, x, b, y, residual);
  } else {
    dim3 blk(32, 8);
    launch_pdl(k_apply<T>, dim3(grid2(L.np, L.np, blk)), dim3(blk), 0, s, L, x, b, y, residual);
  }
}

void launch_rhs(const LevelDev& L, const double* f, const double* ud, double* b, cudaStream_t s) {
  count_launches(2);
  dim3 blk(32, 8);
  launch_pdl(k_rhs_vel, dim3(grid2(L.np, L.np, blk)), dim3(blk), 0, s, L, f, ud, b);
  launch_pdl(k_rhs_p, dim3(grid2(L.np, L.np, blk)), dim3(blk), 0, s, L, ud, b);
}

void launch_rhs_transpose(const LevelDev& L, const double* lam, double* g, cudaStream_t s) {
  count_launches(1);
  dim3 blk(32, 8);
  launch_pdl(k_rhs_transpose, dim3(grid2(L.nq, L.nq, blk)), dim3(blk), 0, s, L, lam, g);
}

template <typename T>
void launch_restrict(const LevelDev& F, const LevelDev& C, const T* rf, T* rc, cudaStream_t s) {
  count_launches(1);
  if (C.np <= OUT_MAX_NP) {
    launch_pdl(k_restrict_out<T>, out_grid(C.np, 9), dim3(32), 0, s, F, C, rf, rc);
    return;
  }
  launch_pdl(k_restrict_march<T>, dim3((C.np + 127) / 128, (C.np + MARCH_ROWS - 1) / MARCH_ROWS, 3), dim3(128), 0, s, F, C, rf, rc);
}

template <typename T>
void launch_prolong_add(const LevelDev& F, const LevelDev& C, const T* ec, T* xf, cudaStream_t s) {
  count_launches(1);
  if (C.np <= OUT_MAX_NP / 2 + 1) {
    launch_pdl(k_prolong_out<T>, out_grid(C.np, 36), dim3(32), 0, s, F, C, ec, xf);
    return;
  }
  const int rows = C.n <= 320 ? 1 : C.n <= 640 ? 2 : MARCH_ROWS;
  launch_pdl(k_prolong_march<T>, dim3((F.np + 127) / 128, (C.np + rows - 1) / rows, 3), dim3(128), 0, s, F, C, ec, xf, rows);
}

template <typename TI, typename TO>
void launch_convert(const TI* in, TO* out, long long N, cudaStream_t s) {
  count_launches(1);
  long long blocks = (N + 255) / 256;
  if (blocks > 152 * 16) blocks = 152 * 16;
  if (blocks < 1) blocks = 1;
  launch_pdl(k_convert<TI, TO>, dim3(static_cast<int>(blocks)), dim3(256), 0, s, in, out, N);
}

void launch_coarse(const double* G, int N0, const double* r, double* e, cudaStream_t s) {
  count_launches(1);
  launch_pdl(k_coarse, dim3((N0 + 7) / 8), dim3(256), 0, s, G, N0, r, e);
}

template void launch_apply<double>(const LevelDev&, const double*, const double*, double*, int, cudaStream_t);
template void launch_apply<float>(const LevelDev&, const float*, const float*, float*, int, cudaStream_t);
template void launch_restrict<double>(const LevelDev&, const LevelDev&, const double*, double*, cudaStream_t);
template void launch_restrict<float>(const LevelDev&, const LevelDev&, const float*, float*, cudaStream_t);
template void launch_prolong_add<double>(const LevelDev&, const LevelDev&, const double*, double*, cudaStream_t);
template void launch_prolong_add<float>(const LevelDev&, const LevelDev&, const float*, float*, cudaStream_t);
template void launch_convert<double, float>(const double*, float*, long long, cudaStream_t);
template void launch_convert<float, double>(const float*, double*, long long, cudaStream_t);

}  // namespace sv
