// sv_vanka_stencil.cu -- the additive Vanka correction as one stencil (Algorithm 3
// with the shared patch inverses of Section 6.3), FP64.
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
#include <mutex>
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
// adds r / m).  A CTA takes 8 x 4 cells and three of the nine outputs per cell,
// one warp per output (so that loop bounds and coefficients are uniform in a warp
// of interior cells), one lane per cell.  An output takes 81 x 2, 63 x 2 or 49 x 2
// residuals and 9, 6 or 4 pressures (the patches holding the node), the pressure
// 25 x 2 + 1.  Bound: the FP64 pipe (one warp instruction in 16 clocks per SM), on
// the small levels by how evenly the outputs spread over the SMs, which is why
// three CTAs share the outputs of a tile.
// ---------------------------------------------------------------------------
constexpr int GX = 8, GY = 4, GW = GX + 4, GH = GY + 4;

__global__ void __launch_bounds__(96) k_vanka_stencil(LevelDev L, const double* __restrict__ G,
                                                      const double* __restrict__ x, const double* __restrict__ r,
                                                      double* __restrict__ xo, double su, double sp, double rps,
                                                      double omega) {
  pdl_begin();
  __shared__ double V[2][2][2][GH][GW];   // [component][J parity][I parity][cell row][cell column]
  __shared__ double P[GH][GW];            // (cl / cb) r_p
  const int nq = L.nq, np = L.np, n = L.n;
  const long long nv = L.nv;
  const int i0 = GX * blockIdx.x, j0 = GY * blockIdx.y;
  {
    const int cx = threadIdx.x % GW, cy = threadIdx.x / GW;   // 96 threads: 12 x 8 cells
    const int gi = i0 - 2 + cx, gj = j0 - 2 + cy;
#pragma unroll
    for (int PJ = 0; PJ < 2; ++PJ)
#pragma unroll
      for (int PI = 0; PI < 2; ++PI) {
        const int I = 2 * gi + PI, J = 2 * gj + PJ;
        const bool ok = is_free(I, J, nq);
        const double* p = r + static_cast<long long>(J) * nq + I;
        V[0][PJ][PI][cy][cx] = ok ? p[0] : 0.0;
        V[1][PJ][PI][cy][cx] = ok ? p[nv] : 0.0;
      }
    P[cy][cx] = (gi >= 0 && gj >= 0 && gi <= n && gj <= n) ? rps * r[2 * nv + static_cast<long long>(gj) * np + gi] : 0.0;
  }
  __syncthreads();
  const int o = 3 * blockIdx.z + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  const int lx = lane & (GX - 1), ly = lane / GX, i = i0 + lx, j = j0 + ly;
  auto pos = [n](int a) { return a < 3 ? a : a <= n - 3 ? 3 : a >= n ? 6 : a - (n - 2) + 4; };
  const double* g = G + static_cast<size_t>(pos(j) * VS_POS + pos(i)) * VS_TYPE + o * VS_OUT;
  double a0 = 0.0, a1 = 0.0, a2 = 0.0, a3 = 0.0;
  if (o < 8) {
    const int c = o >> 2, py = (o >> 1) & 1, px = o & 1;
    for (int J = 2 * py; J < 9; ++J) {
      const double* v = &V[0][J & 1][0][ly + (J >> 1)][lx];
      const double2* gj = reinterpret_cast<const double2*>(g + J * 18);
#pragma unroll
      for (int I = 0; I < 9; ++I) {
        if (I < 2 && px) continue;
        const double2 w = __ldg(gj + I);
        const double* vi = v + (I & 1) * (GH * GW) + (I >> 1);
        if (I & 1) {
          a2 = fma(w.x, vi[0], a2);
          a3 = fma(w.y, vi[4 * GH * GW], a3);
        } else {
          a0 = fma(w.x, vi[0], a0);
          a1 = fma(w.y, vi[4 * GH * GW], a1);
        }
      }
    }
#pragma unroll
    for (int k = 0; k < 9; ++k) {
      const int dj = k / 3, di = k % 3;
      if ((dj == 0 && py) || (di == 0 && px)) continue;   // the node's patches only
      a0 = fma(__ldg(g + 162 + k), P[ly + 1 + dj][lx + 1 + di], a0);
    }
    const int I = 2 * i + px, J = 2 * j + py;
    if (I >= nq || J >= nq) return;
    const long long k = c * nv + static_cast<long long>(J) * nq + I;
    const double xv = x != nullptr ? x[k] : 0.0;
    xo[k] = is_free(I, J, nq) ? fma(su, (a0 + a1) + (a2 + a3), xv) : fma(omega, r[k], xv);
  } else {
#pragma unroll
    for (int J = 2; J < 7; ++J) {
      const double* v = &V[0][J & 1][0][ly + (J >> 1)][lx];
      const double2* gj = reinterpret_cast<const double2*>(g + J * 18);
#pragma unroll
      for (int I = 2; I < 7; ++I) {
        const double2 w = __ldg(gj + I);
        const double* vi = v + (I & 1) * (GH * GW) + (I >> 1);
        if (I & 1) {
          a2 = fma(w.x, vi[0], a2);
          a3 = fma(w.y, vi[4 * GH * GW], a3);
        } else {
          a0 = fma(w.x, vi[0], a0);
          a1 = fma(w.y, vi[4 * GH * GW], a1);
        }
      }
    }
    a0 = fma(__ldg(g + 162 + 4), P[ly + 2][lx + 2], a0);
    if (i > n || j > n) return;
    const long long k = 2 * nv + static_cast<long long>(j) * np + i;
    xo[k] = fma(sp, (a0 + a1) + (a2 + a3), x != nullptr ? x[k] : 0.0);
  }
}

}  // namespace

const std::vector<long double>& vanka_stencil() {
  static const std::vector<long double> G = build_stencil();
  return G;
}

void launch_vanka_stencil(const LevelDev& L, const double* G, const double* x, const double* b, double* xo,
                          double omega, double* rscratch, cudaStream_t s) {
  const double* r = b;
  if (x != nullptr) {
    launch_apply<double>(L, x, b, rscratch, 1, s);
    r = rscratch;
  }
  count_launches(1);
  launch_pdl(k_vanka_stencil, dim3((L.np + GX - 1) / GX, (L.np + GY - 1) / GY, 3), dim3(96), 0, s, L, G, x, r, xo,
             omega / L.cl, omega / L.cb, L.cl / L.cb, omega);
}

}  // namespace sv
