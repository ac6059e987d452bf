// sv_vanka_stencil.cu -- the additive Vanka correction as one stencil (Algorithm 3
// with the shared patch inverses of Section 6.3).
//
// On a uniform grid every patch of a class has the same inverse, so the sum over
// patches sum_i V_i^T diag(1/m) A_i^-1 V_i is itself a stencil: the nine
// corrections of a cell (Q2 nodes 2i, 2i+1 per axis of both components, and
// p(i, j)) are fixed linear combinations of the residual on the 9 x 9 nodes around
// node (2i, 2j) and the 3 x 3 vertices around (i, j).  The coefficients depend on
// the cell only through its distance to the boundary: seven positions per axis
// (0, 1, 2, interior, n-2, n-1, n), 49 cell types, the same on every level in the
// integer units of the stencils (below).  A sweep is then the residual kernel and
// one pass of dot products: no patch is solved, no correction is passed between
// patches, and every output is independent of the others.
//
// Units.  A patch matrix is D A_u D with A_u the integer-stencil matrix and D =
// diag(sqrt(cl) on velocities, cb / sqrt(cl) on the pressure).  With r_p scaled by
// cl / cb on input, the velocity corrections carry 1 / cl and the pressure
// correction 1 / cb.
#include <cuda_runtime.h>

#include <cmath>
#include <vector>

#include "sv_internal.h"
#include "sv_level_ops.cuh"
#include "sv_stencil.cuh"

namespace sv {
namespace {

using ops::is_free;

// Patch inverse of class (cx, cy) in integer units, 51 x 51 in slot order, zero rows
// and columns off the free slots (the identity rows of Dirichlet nodes are applied by
// the kernels directly).  Block elimination: z = K^-1 b^T, s = b z.
void unit_patch_inverse(int cx, int cy, std::vector<long double>& inv) {
  const int mx = axis_free_mask(cx), my = axis_free_mask(cy);
  int slot[25], m = 0;
  for (int w = 0; w < 25; ++w)
    if (((mx >> (w % 5)) & 1) && ((my >> (w / 5)) & 1)) slot[m++] = w;
  // parity of a window node is the parity of its offset from the (even) centre node
  auto kk = [](int a, int b) { return static_cast<long double>(k1(a & 1, b - a)); };
  auto mm = [](int a, int b) { return static_cast<long double>(m1(a & 1, b - a)); };
  std::vector<long double> A(m * 2 * m, 0.0L);   // [K | I] -> [I | K^-1]
  for (int r = 0; r < m; ++r) {
    for (int c = 0; c < m; ++c) {
      const int xi = slot[r] % 5, yi = slot[r] / 5, xj = slot[c] % 5, yj = slot[c] / 5;
      A[r * 2 * m + c] = kk(xi, xj) * mm(yi, yj) + mm(xi, xj) * kk(yi, yj);
    }
    A[r * 2 * m + m + r] = 1.0L;
  }
  for (int p = 0; p < m; ++p) {   // K is symmetric positive definite: no pivoting
    const long double d = 1.0L / A[p * 2 * m + p];
    for (int c = 0; c < 2 * m; ++c) A[p * 2 * m + c] *= d;
    for (int r = 0; r < m; ++r) {
      const long double f = A[r * 2 * m + p];
      if (r == p || f == 0.0L) continue;
      for (int c = 0; c < 2 * m; ++c) A[r * 2 * m + c] -= f * A[p * 2 * m + c];
    }
  }
  long double b[2][25], z[2][25], s = 0.0L;
  for (int r = 0; r < m; ++r) {
    const int dI = slot[r] % 5 - 2, dJ = slot[r] / 5 - 2;
    b[0][r] = crow(dI) * nrow(dJ);
    b[1][r] = nrow(dI) * crow(dJ);
  }
  for (int c = 0; c < 2; ++c)
    for (int r = 0; r < m; ++r) {
      z[c][r] = 0.0L;
      for (int k = 0; k < m; ++k) z[c][r] += A[r * 2 * m + m + k] * b[c][k];
      s += b[c][r] * z[c][r];
    }
  inv.assign(51 * 51, 0.0L);
  for (int c = 0; c < 2; ++c)
    for (int r = 0; r < m; ++r) {
      for (int c2 = 0; c2 < 2; ++c2)
        for (int k = 0; k < m; ++k)
          inv[(25 * c + slot[r]) * 51 + 25 * c2 + slot[k]] =
              (c == c2 ? A[r * 2 * m + m + k] : 0.0L) - z[c][r] * z[c2][k] / s;
      inv[(25 * c + slot[r]) * 51 + 50] = z[c][r] / s;
      inv[50 * 51 + 25 * c + slot[r]] = z[c][r] / s;
    }
  inv[50 * 51 + 50] = -1.0L / s;
}

std::vector<long double> build_stencil() {
  std::vector<long double> G(static_cast<size_t>(VS_TAB), 0.0L), inv[25];
  for (int cy = 0; cy < 5; ++cy)
    for (int cx = 0; cx < 5; ++cx) unit_patch_inverse(cx, cy, inv[cy * 5 + cx]);
  const int n = 16;                                   // a grid with every cell type
  const int rep[VS_POS] = {0, 1, 2, 8, n - 2, n - 1, n};
  for (int ty = 0; ty < VS_POS; ++ty)
    for (int tx = 0; tx < VS_POS; ++tx) {
      const int i = rep[tx], j = rep[ty];
      long double* g = G.data() + static_cast<size_t>(ty * VS_POS + tx) * VS_TYPE;
      for (int o = 0; o < 9; ++o, g += VS_OUT) {
        const int c = o >> 2, I = 2 * i + (o & 1), J = 2 * j + ((o >> 1) & 1);
        if (o < 8 && !(I > 0 && J > 0 && I < 2 * n && J < 2 * n)) continue;   // Dirichlet or outside
        const long double w = o < 8 ? 1.0L / (axis_mult(I, n) * axis_mult(J, n)) : 1.0L;
        for (int vj = j - 1; vj <= j + 1; ++vj)
          for (int vi = i - 1; vi <= i + 1; ++vi) {
            if (vi < 0 || vj < 0 || vi > n || vj > n) continue;
            int so = 50;
            if (o < 8) {
              const int wi = I - 2 * vi + 2, wj = J - 2 * vj + 2;
              if (wi < 0 || wj < 0 || wi > 4 || wj > 4) continue;
              so = 25 * c + wj * 5 + wi;
            } else if (vi != i || vj != j) {
              continue;
            }
            const long double* row = inv[axis_class(vj, n) * 5 + axis_class(vi, n)].data() + so * 51;
            for (int c2 = 0; c2 < 2; ++c2)
              for (int s = 0; s < 25; ++s) {
                const int wI = 2 * (vi - i) + 2 + s % 5, wJ = 2 * (vj - j) + 2 + s / 5;   // 0..8
                g[(wJ * 9 + wI) * 2 + c2] += w * row[25 * c2 + s];
              }
            g[162 + (vj - j + 1) * 3 + vi - i + 1] += w * row[50];
          }
      }
    }
  return G;
}

// ---------------------------------------------------------------------------
// One sweep from the residual r: x_out = x + omega (stencil r), Dirichlet rows
// x + omega r (their patch rows are identities and every patch holding the node
// adds r / m).  An output takes 81 x 2, 63 x 2 or 49 x 2 residuals and 9, 6 or 4
// pressures (the patches holding the node), the pressure 25 x 2 + 1.
//
// What bounds it is the FP64 pipe: a warp's FP64 instruction holds the unit of its
// SM sub-partition for 64 clocks, so on the small levels the time is the longest
// chain a warp runs, not the work.  Hence a warp takes one output kind of 4 x 2
// cells with four lanes per output, each lane every fourth coefficient (at most 42
// multiply-adds), summed by shuffles; three warps per CTA and three CTAs per tile
// spread the nine outputs of a cell over the SMs.  Zero guess, FP64: 9.0 us at n = 40,
// 17.6 at n = 64 (a solve at n = 32: 7.8 ms with patch solves, 3.6 with this sweep); FP32
// V-cycle of n = 128 with it up to n = 64: 260 -> 200 us.
// ---------------------------------------------------------------------------
constexpr int GX = 4, GY = 2, GW = GX + 4, GH = GY + 4, PARTS = 4;
static_assert(GX * GY * PARTS == 32, "a warp is one output kind of a tile");

template <typename T>
struct Pair;
template <>
struct Pair<double> { using type = double2; };
template <>
struct Pair<float> { using type = float2; };

template <typename T>
__global__ void __launch_bounds__(96) k_vanka_stencil(LevelDev L, const T* __restrict__ G, const T* __restrict__ x,
                                                      const T* __restrict__ r, T* __restrict__ xo, T su, T sp, T rps,
                                                      T omega) {
  using T2 = typename Pair<T>::type;
  pdl_begin();
  __shared__ T V[2][2 * GH][2 * GW];   // residual of the window's nodes, 0 off the free nodes
  __shared__ T P[GH][GW];              // (cl / cb) r_p
  const int nq = L.nq, np = L.np, n = L.n;
  const long long nv = L.nv;
  const int i0 = GX * blockIdx.x, j0 = GY * blockIdx.y;
  for (int t = threadIdx.x; t < 4 * GW * GH; t += 96) {
    const int c = t % (2 * GW), w = t / (2 * GW), I = 2 * (i0 - 2) + c, J = 2 * (j0 - 2) + w;
    const bool ok = is_free(I, J, nq);
    const long long k = static_cast<long long>(J) * nq + I;
    V[0][w][c] = ok ? r[k] : T(0);
    V[1][w][c] = ok ? r[nv + k] : T(0);
  }
  if (threadIdx.x < GW * GH) {
    const int c = threadIdx.x % GW, w = threadIdx.x / GW, gi = i0 - 2 + c, gj = j0 - 2 + w;
    const bool ok = gi >= 0 && gj >= 0 && gi <= n && gj <= n;
    P[w][c] = ok ? rps * r[2 * nv + static_cast<long long>(gj) * np + gi] : T(0);
  }
  __syncthreads();
  const int o = 3 * blockIdx.z + (threadIdx.x >> 5), part = (threadIdx.x & 31) / (GX * GY);
  const int lx = threadIdx.x % GX, ly = (threadIdx.x / GX) % GY, i = i0 + lx, j = j0 + ly;
  auto pos = [n](int a) { return a < 3 ? a : a <= n - 3 ? 3 : a >= n ? 6 : a - (n - 2) + 4; };
  const T* g = G + static_cast<size_t>(pos(j) * VS_POS + pos(i)) * VS_TYPE + o * VS_OUT;
  const T* v = &V[0][2 * ly][2 * lx];
  T a0 = T(0), a1 = T(0);
  auto node = [&](int J, int I) {
    const T2 w = __ldg(reinterpret_cast<const T2*>(g) + J * 9 + I);
    a0 = fma(w.x, v[J * 2 * GW + I], a0);
    a1 = fma(w.y, v[4 * GW * GH + J * 2 * GW + I], a1);
  };
  const int py = (o >> 1) & 1, px = o & 1;
  if (o == 8) {
#pragma unroll
    for (int e = part; e < 25; e += PARTS) node(2 + e / 5, 2 + e % 5);
    if (part == 0) a0 = fma(__ldg(g + 162 + 4), P[ly + 2][lx + 2], a0);
  } else {
    const int cnt = (9 - 2 * py) * (9 - 2 * px);   // node columns 2 px .. 8, rows 2 py .. 8
    if (px) {
#pragma unroll 8
      for (int e = part; e < cnt; e += PARTS) node(2 * py + e / 7, 2 + e % 7);
    } else {
#pragma unroll 8
      for (int e = part; e < cnt; e += PARTS) node(2 * py + e / 9, e % 9);
    }
#pragma unroll
    for (int k = part; k < 9; k += PARTS) {
      const int dj = k / 3, di = k % 3;
      if (dj >= py && di >= px) a1 = fma(__ldg(g + 162 + k), P[ly + 1 + dj][lx + 1 + di], a1);
    }
  }
  T d = a0 + a1;
  d += __shfl_xor_sync(0xffffffffu, d, 8);
  d += __shfl_xor_sync(0xffffffffu, d, 16);
  if (part != 0) return;
  if (o == 8) {
    if (i > n || j > n) return;
    const long long k = 2 * nv + static_cast<long long>(j) * np + i;
    xo[k] = fma(sp, d, x != nullptr ? x[k] : T(0));
  } else {
    const int I = 2 * i + px, J = 2 * j + py;
    if (I >= nq || J >= nq) return;
    const long long k = (o >> 2) * nv + static_cast<long long>(J) * nq + I;
    const T xv = x != nullptr ? x[k] : T(0);
    xo[k] = is_free(I, J, nq) ? fma(su, d, xv) : fma(omega, r[k], xv);
  }
}

}  // namespace

const std::vector<long double>& vanka_stencil() {
  static const std::vector<long double> G = build_stencil();
  return G;
}

std::vector<double> vanka_ring_table() {
  const std::vector<long double>& G = vanka_stencil();
  std::vector<double> R(RT_TAB, 0.0);
  for (int t = 0; t < VS_POS * VS_POS; ++t) {
    const long double* g = G.data() + static_cast<size_t>(t) * VS_TYPE;
    double* r = R.data() + static_cast<size_t>(t) * RT_TYPE;
    for (int k = 0; k < 171; ++k)
      for (int o = 0; o < 8; ++o) r[k * 8 + o] = static_cast<double>(g[o * VS_OUT + k]);
    const long double* gp = g + 8 * VS_OUT;
    for (int J = 2; J < 7; ++J)
      for (int I = 2; I < 7; ++I)
        for (int c = 0; c < 2; ++c)
          r[171 * 8 + ((J - 2) * 5 + I - 2) * 2 + c] = static_cast<double>(gp[(J * 9 + I) * 2 + c]);
    r[171 * 8 + 50] = static_cast<double>(gp[162 + 4]);
  }
  return R;
}

template <typename T>
void launch_vanka_stencil(const LevelDev& L, const T* G, const T* x, const T* b, T* xo, double omega, T* rscratch,
                          cudaStream_t s) {
  const T* r = b;
  if (x != nullptr) {
    launch_apply<T>(L, x, b, rscratch, 1, s);
    r = rscratch;
  }
  count_launches(1);
  launch_pdl(k_vanka_stencil<T>, dim3((L.np + GX - 1) / GX, (L.np + GY - 1) / GY, 3), dim3(96), 0, s, L, G, x, r, xo,
             T(omega / L.cl), T(omega / L.cb), T(L.cl / L.cb), T(omega));
}

template void launch_vanka_stencil<double>(const LevelDev&, const double*, const double*, const double*, double*,
                                           double, double*, cudaStream_t);
template void launch_vanka_stencil<float>(const LevelDev&, const float*, const float*, const float*, float*, double,
                                          float*, cudaStream_t);

}  // namespace sv
