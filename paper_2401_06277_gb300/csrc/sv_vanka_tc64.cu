// sv_vanka_tc64.cu -- the FP64 additive Vanka sweep on the 5th-generation tensor
// cores: the composite stencil of the interior (sv_vanka_stencil.cu) as an exact
// integer contraction.
//
// GB300 executes FP64 at 1/64 of its FP32 rate (2 fused multiply-adds per clock and
// SM), so 1125 multiply-adds per vertex cost 560 clocks of an SM; its tensor cores do
// 4096 FP16 multiply-adds per clock with FP32 accumulation.  Both operands are
// therefore split into small integers whose products and sums FP32 holds exactly
// (an error-free splitting, as in Ozaki, Ogita, Oishi and Rump, "Error-free
// transformations of matrix multiplication", Numerical Algorithms 59, 2012):
//   residual      r = 2^(E - 58) q, |r| < 2^E, q rounded to an integer, in
//                 6 balanced digits of 10 bits: q = sum_j d_j 1024^(5 - j), |d_j| <= 512
//   coefficients  G = 2^(e_o - 62) g (e_o per output kind), 7 balanced digits of 9 bits,
//                 |g_i| <= 256
// Each digit is exact in FP16.  A pair of digits (i, j) contributes an integer below
// 2^24 (171 products; the bound is computed from the digits when they are packed), so
// the FP32 accumulation is exact in any order.  The pairs with 9 i + 10 j <= 59 (27 of
// 42) are kept; those left out are below 2^-64 of the largest product.  The 27
// integers of an output are added in 64-bit integers (unit 2^16, the pressure's 2^14, of
// the last digit pair's) and rounded to FP64 at the end.  A residual loses what lies 58
// bits below the bound 2^E of the 6 x 132 cells in reach, at most 2^-55 of the largest of
// them; measured, a sweep's error against 64-bit mantissas is 2.6e-16 of the largest
// velocity (FP64 patch solves: 7e-16 to 1.4e-15) and 2.0e-16 for the pressure (2.6e-16).
//
// Outputs whose own patches hold only much smaller residuals would lose by that against
// FP64 patch solves, whose error follows their patches.  A single sweep therefore checks
// its cells: where nothing within 2^-8 of 2^E (2^-10 for the pressure, whose coefficients
// sum to less) lies in the patches of an output, that output is computed in FP64 by a
// second launch (k_vanka_fp64_cells).  What is lost elsewhere is below 2^-51 of the largest
// residual of the output's patches times the sum of its coefficients, less than the
// measured error of FP64 patch solves.  The sweeps of a cycle do without.
//
// Decomposition.  A CTA owns a strip of 128 cell columns and walks up it two cell rows
// at a time.  The digits of the cells lie in shared memory as planes [cell row][digit]
// [cell column] of 16 bytes (the 8 velocity residuals of a cell): the operand of the
// cells shifted by (dx, dy) is the same memory at another start address, so nothing is
// gathered (an implicit im2col with M = 128 consecutive cells).  One step computes two
// cell rows: K = 30 cell offsets x 8 + 3 x 4 pressures (17 MMAs of K = 16), N = 18
// columns per coefficient digit (9 outputs of each row).  Digit j of the residual is one
// chain of 17 MMAs with N = 18 (7 - j) into an accumulator of its own
// (chains j and j + 3 take turns); the coefficients (69 KB) stay in shared memory for the whole walk.
//
// Warps: 16 read the accumulators and update x (two groups, alternating steps), 9 load
// residuals and write digits, 3 issue the MMAs (an MMA takes a warp about as long to
// issue as the tensor cores to execute), and 4 compute the cells near the
// boundary, where the stencil differs, as FP64 dot products on the otherwise idle FP64
// units.  They meet only in mbarriers, per digit or pair of digits: a plane is overwritten
// for the next rows as soon as its chain has read it.
//
// The exponent E is shared by the cells in reach of a step.  It follows the residual:
// when the largest of the window leaves [2^(E-4), 2^E), the digits of the window are
// rewritten with a new E.  A residual that is not finite makes the cells of the step
// NaN, in a single sweep only the dofs of the patches that hold it.  Every wait is
// bounded; on expiry the kernel sets *err and returns.
//
// Bound: the tensor pipe and its operand reads.  An MMA of M = 128 takes N / 2 clocks
// from N = 128 on and about 38 + 0.22 N below, so the chains of a step take 25 clocks per
// vertex: 0.33 ms at 2048^2.  Measured 0.49 ms from a zero guess (the patch solves in
// FP64: 3.9 ms), 0.85 ms from an iterate, the residual included (5.5 ms).  The operand
// reads keep shared memory 97% busy, so the other warps' shared-memory accesses wait;
// hence the two epilogue groups (0.55 -> 0.50 ms) and one barrier for two digit planes
// (0.50 -> 0.49).  Small levels are bound by the prologue: 12.9 us at n = 64, 13.9 at 128.
// With the check 0.53 ms, and where it finds cells, of a random residual none, of a
// right-hand side with boundary data the strips along the walls: 2.5 ms; all cells 12.9 ms.
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <type_traits>

#include "sv_digits.cuh"
#include "sv_internal.h"
#include "sv_level_ops.cuh"
#include "sv_stencil.cuh"
#include "sv_tcgen05.cuh"

namespace sv {
namespace {

using namespace tc;
using namespace dig;
using ops::is_free;

constexpr int NG = 7;                            // digits of the coefficients
constexpr int NBLK = 18;                         // N columns per coefficient digit: 9 outputs of each cell row
constexpr int GROWS = NBLK * NG;                 // 126 rows of the coefficient operand
constexpr int KSTEPS = 17;
constexpr int CHUNK = GROWS * 16;                // 8 K-values of all coefficient rows
constexpr int GBYTES = 2 * KSTEPS * CHUNK + 32;  // + the two rows that N = 128 reads past the end
static_assert(GBYTES == TC64_BYTES, "size of the packed coefficients");
constexpr int RING_CTA_WARPS = 16, RING_PARTS_MAX_N = 256;
constexpr int MMA_WARPS = 3, RING_WARPS = 4;   // MMA warp w: chains w and w + 3, one accumulator
constexpr int NT = 32 * (EPI_WARPS + SLICE_WARPS + MMA_WARPS + RING_WARPS);

struct SM {
  static constexpr int RING = 0;                         // 6 cell rows
  static constexpr int P = RING + 6 * ROWB;              // pressures of the step: [digit][column] 16 B
  static constexpr int G = P + ROWB;
  static constexpr int CEXP = G + GBYTES;                // exponents of cells: 8 row pairs [row][column] of 16 bits
  static constexpr int PEXP = CEXP + 8 * 2 * WCOLS * 2;  // of pressures: 8 row pairs [row][column]
  static constexpr int BAR = (PEXP + 8 * 4 * WCOLS * 2 + 7) / 8 * 8;   // full[3] (plane pairs), done[2][6] (by step parity), free[3], gload
  static constexpr int MISC = BAR + 22 * 8;              // tmem slot, fail flag, 8 maxima, 8 minima, 4 exponents
  static constexpr int BYTES = MISC + 24 * 4;
  static_assert(G % 16 == 0 && BAR % 8 == 0 && BYTES <= 227 * 1024, "shared memory");
};

__host__ __device__ constexpr int chain_n(int j) { return (NBLK * (NG - j) + 15) / 16 * 16; }
// accumulator of the chains c and c + 3: its first tensor-memory column.  One more for
// each chain (five fit) let the MMAs run a step ahead and was slower (544 against 493 us
// at 2048^2): MMAs of N <= 128 read shared memory at 97% of its rate, and the other warps'
// accesses need the pauses.
__host__ __device__ constexpr int acc_col(int c) {
  int k = 0;
  for (int i = 0; i < c % MMA_WARPS; ++i) k += chain_n(i);
  return k;
}
static_assert(acc_col(2) + chain_n(2) <= 512, "tensor memory");
// instruction descriptor: D FP32, A and B FP16, both K-major, M = 128
__host__ __device__ constexpr uint32_t idesc(int n) {
  return (1u << 4) | (static_cast<uint32_t>(n >> 3) << 17) | ((128u >> 4) << 24);
}

struct Args {
  LevelDev L;
  const unsigned char* G;     // packed coefficient digits
  const double* Gd;           // the FP64 stencil table (cells near the boundary)
  const double* x;
  const double* r;
  double* xo;
  double su, sp;              // omega / cl, omega / cb
  double qu, qp;              // the same with the units of the digit sums
  double rps;                 // cl / cb
  double omega;
  int strips, ctas;           // CTAs past `ctas` compute cells near the boundary only
  int steps_per_seg;
  int* err;
  int wait_limit;
  const TC64Check check;      // flags null: every output is taken as it is
};

// FP64 dot products of the cells outside [3, n - 3]^2: three cell rows below and above,
// three columns left and right between them.  The MMAs take nearly all of the shared
// memory and L1 bandwidth, so a unit is laid out for few load wavefronts: four cells along
// the band x the eight velocity outputs, whose coefficients are adjacent in the table
// (a load of the residual serves eight lanes, one of the coefficients four); the pressure
// outputs take 32 cells.  Node rows and columns off the grid are left out.
struct Band {
  int i, j;          // this lane's cell
  bool in;
  int J0, J1, I0, I1;   // node rows and columns of the 9 x 9 window in use, uniform in the warp
};
__host__ __device__ constexpr int ring_units(int n, int cells) {
  return 6 * ((n + cells) / cells) + 6 * ((n - 5 + cells - 1) / cells);
}
__device__ __forceinline__ Band band_of(int n, int unit, int cells, int k) {
  const int w = (n + cells) / cells, h = (n - 5 + cells - 1) / cells;
  Band b;
  b.J0 = b.I0 = 0;
  b.J1 = b.I1 = 8;
  if (unit < 6 * w) {          // rows 0, 1, 2, n - 2, n - 1, n
    const int row = unit / w;
    b.j = row < 3 ? row : n - 2 + row - 3;
    b.i = cells * (unit - row * w) + k;
    b.in = b.i <= n;
    b.J0 = max(0, 5 - 2 * b.j);
    b.J1 = min(8, 2 * (n - b.j) + 3);
  } else {                     // columns, rows 3 .. n - 3
    const int v = unit - 6 * w, col = v / h;
    b.i = col < 3 ? col : n - 2 + col - 3;
    b.j = 3 + cells * (v - col * h) + k;
    b.in = b.j <= n - 3;
    b.I0 = max(0, 5 - 2 * b.i);
    b.I1 = min(8, 2 * (n - b.i) + 3);
  }
  return b;
}
__device__ __forceinline__ int cell_type(int n, const Band& b) {
  auto pos = [n](int a) { return a < 3 ? a : a <= n - 3 ? 3 : a >= n ? 6 : a - (n - 2) + 4; };
  return b.in ? pos(b.j) * VS_POS + pos(b.i) : 0;
}

// PARTS = 1: a unit is four cells, a lane one output of one of them (162 multiply-adds
// each: 10,000 clocks of a sub-partition's FP64 unit).  PARTS = 4: one cell, four lanes per
// output, for the grids on which the longest unit, not the work, sets the time.
template <int PARTS>
__device__ __forceinline__ void cell_velocity(const Args& A, const Band& b, int lane) {
  static_assert(PARTS == 1 || PARTS == 4, "lanes: 8 outputs x 4 cells or 4 parts");
  const LevelDev& L = A.L;
  const int n = L.n, nq = L.nq, np = L.np, o = lane & 7, part = PARTS == 4 ? lane >> 3 : 0;
  const long long nv = L.nv;
  const double* g = A.Gd + static_cast<size_t>(cell_type(n, b)) * RT_TYPE + o;
  const int px = o & 1, py = (o >> 1) & 1;   // the patches with an odd node lie to its right: from 2 px, 2 py on
  double a0 = 0.0, a1 = 0.0;
  auto node = [&](int rJ, int rI) {
    const int J = 2 * b.j - 4 + rJ;
    const double* rr = A.r + static_cast<long long>(J) * nq + 2 * b.i - 4 + rI;
    const double* gr = g + (rJ * 9 + rI) * 16;
    const bool ok = b.in && rI >= 2 * px && rJ >= 2 * py && is_free(2 * b.i - 4 + rI, J, nq);
    const double r0 = ok ? __ldg(rr) : 0.0, r1 = ok ? __ldg(rr + nv) : 0.0;
    a0 = fma(__ldg(gr), r0, a0);
    a1 = fma(__ldg(gr + 8), r1, a1);
  };
  if (PARTS == 1) {
    for (int rJ = b.J0; rJ <= b.J1; ++rJ) {
#pragma unroll 3
      for (int rI = b.I0; rI <= b.I1; ++rI) node(rJ, rI);
    }
  } else {   // every fourth node of the window (four wide at least)
    int rJ = b.J0, rI = b.I0 + part;
#pragma unroll 3
    for (int e = (b.J1 - b.J0 + 1) * (b.I1 - b.I0 + 1) - part; e > 0; e -= PARTS) {
      node(rJ, rI);
      rI += PARTS;
      if (rI > b.I1) {
        rI -= b.I1 - b.I0 + 1;
        ++rJ;
      }
    }
  }
  double ap = 0.0;
#pragma unroll
  for (int k = part; k < 9; k += PARTS) {
    const int pi = b.i + k % 3 - 1, pj = b.j + k / 3 - 1;
    const bool ok = b.in && k % 3 >= px && k / 3 >= py && pi >= 0 && pj >= 0 && pi <= n && pj <= n;
    const double r0 = ok ? __ldg(A.r + 2 * nv + static_cast<long long>(pj) * np + pi) : 0.0;
    ap = fma(__ldg(g + 162 * 8 + k * 8), r0, ap);
  }
  double d = fma(A.rps, ap, a0 + a1);
  if (PARTS == 4) {
    d += __shfl_xor_sync(0xffffffffu, d, 8);
    d += __shfl_xor_sync(0xffffffffu, d, 16);
  }
  const int I = 2 * b.i + px, J = 2 * b.j + py;
  if (part != 0 || !b.in || I >= nq || J >= nq) return;
  const long long k = (o >> 2) * nv + static_cast<long long>(J) * nq + I;
  const double xv = A.x != nullptr ? A.x[k] : 0.0;
  A.xo[k] = is_free(I, J, nq) ? fma(A.su, d, xv) : fma(A.omega, A.r[k], xv);
}

__device__ __forceinline__ void cell_pressure(const Args& A, const Band& b) {
  const LevelDev& L = A.L;
  const int n = L.n, nq = L.nq;
  const long long nv = L.nv;
  const double* g = A.Gd + static_cast<size_t>(cell_type(n, b)) * RT_TYPE + 171 * 8;
  double a0 = 0.0, a1 = 0.0;
  for (int rJ = max(2, b.J0); rJ <= min(6, b.J1); ++rJ) {
    const int J = 2 * b.j - 4 + rJ;
#pragma unroll
    for (int rI = 2; rI < 7; ++rI) {
      const int I = 2 * b.i - 4 + rI;
      const bool ok = b.in && is_free(I, J, nq);
      const double* rr = A.r + static_cast<long long>(J) * nq + I;
      const double* gr = g + ((rJ - 2) * 5 + rI - 2) * 2;
      a0 = fma(__ldg(gr), ok ? __ldg(rr) : 0.0, a0);
      a1 = fma(__ldg(gr + 1), ok ? __ldg(rr + nv) : 0.0, a1);
    }
  }
  if (!b.in) return;
  const long long k = 2 * nv + static_cast<long long>(b.j) * L.np + b.i;
  const double d = fma(A.rps * __ldg(g + 50), A.r[k], a0 + a1);
  A.xo[k] = fma(A.sp, d, A.x != nullptr ? A.x[k] : 0.0);
}

// All units, dealt to `slots` warps.
__device__ __forceinline__ void ring(const Args& A, int slot, int slots, int lane) {
  const int n = A.L.n, wide = n > RING_PARTS_MAX_N;
  const int uv = ring_units(n, wide ? 4 : 1), up = ring_units(n, 32);
  for (int u = slot; u < uv + up; u += slots) {
    if (u >= uv) cell_pressure(A, band_of(n, u - uv, 32, lane));
    else if (wide) cell_velocity<1>(A, band_of(n, u, 4, lane >> 3), lane);
    else cell_velocity<4>(A, band_of(n, u, 1, 0), lane);
  }
}

struct Shared {   // what the roles of a CTA share
  uint32_t full, done, free, tmem;
  volatile int* fail;
  volatile int* sexp;
  const unsigned short* cexp;
  const unsigned short* pexp;
  int i0, j0, rows, S;
};

// Outputs of a cell to which the contraction gives too little (bits: velocities, pressure):
// the patches that hold it have no residual within 2^-8 of 2^E (pressure: 2^-10).  Every
// velocity output lies in patches that hold the nodes of the 3 x 3 cells around and the
// pressures of the vertices i, i + 1 and j, j + 1; the pressure's patch the nodes of the
// cells i - 1, i and j - 1, j and its own pressure.  a: the cell's row in the step, col:
// its held column.
__device__ __forceinline__ unsigned too_small(const Shared& C, int s, int a, int col, int eb) {
  auto cell = [&](int r, int c) -> int { return C.cexp[(((r >> 1) & 7) * 2 + (r & 1)) * WCOLS + c]; };
  const int r = 2 * s + 2 + a;   // cell row of the walk, row r & 1 of pair r >> 1
  int mp = cell(r, col);
  if (mp >= eb - 7) return 0;
  const unsigned short* p = C.pexp + (((s + 2) & 7) * 4 + 1 + a) * WCOLS + col;
  mp = max(mp, static_cast<int>(p[0]));
  if (mp >= eb - 7) return 0;
  mp = max(max(mp, cell(r, col - 1)), max(cell(r - 1, col), cell(r - 1, col - 1)));
  int mu = max(mp, max(max(cell(r + 1, col - 1), cell(r + 1, col)), max(cell(r + 1, col + 1), cell(r, col + 1))));
  mu = max(max(mu, cell(r - 1, col + 1)), static_cast<int>(max(max(p[1], p[WCOLS]), p[WCOLS + 1])));
  return (mu < eb - 7 ? 1u : 0u) | (mp < eb - 9 ? 2u : 0u);
}
// Whether its reach holds anything but zeros
__device__ __forceinline__ bool any_residual(const Shared& C, int s, int a, int col) {
  unsigned m = 0;
#pragma unroll 1
  for (int r = 2 * s + a; r <= 2 * s + a + 4; ++r)
#pragma unroll 1
    for (int c = col - 2; c <= col + 2; ++c) m |= C.cexp[(((r >> 1) & 7) * 2 + (r & 1)) * WCOLS + c];
#pragma unroll 1
  for (int k = 0; k < 3; ++k)
#pragma unroll 1
    for (int c = col - 1; c <= col + 1; ++c) m |= C.pexp[(((s + 2) & 7) * 4 + a + k) * WCOLS + c];
  return m != 0;
}
// One chain's accumulators: T[o] += the digit sums (gi, c) with weight 2^(59 - 9 gi - 10 c),
// in units of 2^16 (velocities) and 2^14 (pressure): the sums of |G| / 2^e_o are below 5
// and 1.4, so |T| < 2^62.  Weights below the unit are rounded one by one (about a dozen).
constexpr int UNIT_U = 16, UNIT_P = 14;
template <int C, int GI>
__device__ __forceinline__ void add_chain(uint32_t taddr, long long (&T)[9]) {
  if constexpr (GI < NG - C) {
    constexpr int K = 59 - 9 * GI - 10 * C;
    constexpr bool two = GI + 1 < NG - C;
    uint32_t v[2][9];
    tmem_ld9(taddr + NBLK * GI, v[0]);
    if constexpr (two) tmem_ld9(taddr + NBLK * (GI + 1), v[1]);
    wait_ld();
#pragma unroll
    for (int o = 0; o < 8; ++o) {
      add_digit<K - UNIT_U>(T[o], v[0][o]);
      if constexpr (two) add_digit<K - 9 - UNIT_U>(T[o], v[1][o]);
    }
    add_digit<K - UNIT_P>(T[8], v[0][8]);
    if constexpr (two) add_digit<K - 9 - UNIT_P>(T[8], v[1][8]);
    add_chain<C, GI + 2>(taddr, T);
  }
}

// Accumulators to x, steps g, g + 2, ...: warp -> cell row a and lane quarter of the columns.
__device__ __forceinline__ void epilogue(const Args& A, const Shared& C, int g, int warp, int lane) {
  const LevelDev& L = A.L;
  const int n = L.n, nq = L.nq, np = L.np;
  const long long nv = L.nv;
  const int a = (warp >> 2) & 1, i = C.i0 + 32 * (warp & 3) + lane;
  const uint32_t tq = C.tmem + (static_cast<uint32_t>(32 * (warp & 3)) << 16) + 9 * a;
  for (int s = g; s < C.S; s += 2) {
    long long T[9];
#pragma unroll
    for (int o = 0; o < 9; ++o) T[o] = 0;
    auto chain = [&](auto c_) {
      constexpr int c = decltype(c_)::value;
      const bool ok = mbar_wait_or_fail(C.done + 8 * (ND * g + c), (s >> 1) & 1, A.wait_limit, C.fail);
      if (!__all_sync(0xffffffffu, ok)) return false;
      fence_after();
      add_chain<c, 0>(tq + acc_col(c), T);
      fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(C.free + 8 * (c % MMA_WARPS));
      return true;
    };
    if (!(chain(std::integral_constant<int, 0>{}) && chain(std::integral_constant<int, 1>{}) &&
          chain(std::integral_constant<int, 2>{}) && chain(std::integral_constant<int, 3>{}) &&
          chain(std::integral_constant<int, 4>{}) && chain(std::integral_constant<int, 5>{})))
      return;
    const int j = C.j0 + 2 * s + a;
    const bool mine = i <= n - 3 && 2 * s + a < C.rows;
    const int es = C.sexp[s & 3], eb = es & 0xffff;   // the sign: values were rounded
    if (A.check.flags != nullptr) {
      unsigned redo = 0;
      if (mine && es < 0) redo = too_small(C, s, a, i - C.i0 + 2, eb);
      if (redo != 0 && !any_residual(C, s, a, i - C.i0 + 2)) redo = 0;
      if (eb == 0x7ff) redo = 3;                      // values that are not finite
      if (mine) A.check.flags[static_cast<long long>(j) * np + i] = static_cast<unsigned char>(redo);
      if (mine && redo != 0) *A.check.any = A.check.call;
    }
    if (!mine) continue;
    const long long ku = static_cast<long long>(2 * j) * nq + 2 * i;
    const long long kp = 2 * nv + static_cast<long long>(j) * np + i;
    auto at = [&](int o) { return o == 8 ? kp : (o >> 2) * nv + ku + ((o >> 1) & 1) * nq + (o & 1); };
    double xv[9];
#pragma unroll
    for (int o = 0; o < 9; ++o) xv[o] = A.x != nullptr ? A.x[at(o)] : 0.0;
    const double qu = A.qu * exp_scale(eb, UNIT_U - 75), qp = A.qp * exp_scale(eb, UNIT_P - 75);
#pragma unroll
    for (int o = 0; o < 9; ++o) A.xo[at(o)] = fma(o == 8 ? qp : qu, to_double(T[o]), xv[o]);
  }
}

__global__ void __launch_bounds__(NT, 1) k_vanka_tc64(const Args A) {
  pdl_begin();
  extern __shared__ __align__(1024) unsigned char sm[];
  const LevelDev& L = A.L;
  const int n = L.n, nq = L.nq, np = L.np;
  const long long nv = L.nv;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const uint32_t s0 = su32(sm);
  const uint32_t bar_full = s0 + SM::BAR, bar_done = bar_full + 8 * ND, bar_free = bar_done + 16 * ND,
                 bar_g = bar_free + 8 * MMA_WARPS;
  uint32_t* tslot = reinterpret_cast<uint32_t*>(sm + SM::MISC);
  volatile int* fail = reinterpret_cast<volatile int*>(sm + SM::MISC + 4);
  unsigned* smax = reinterpret_cast<unsigned*>(sm + SM::MISC + 8);                    // 8 slots
  unsigned* smin = reinterpret_cast<unsigned*>(sm + SM::MISC + 40);                   // 8 slots
  volatile int* sexp = reinterpret_cast<volatile int*>(sm + SM::MISC + 72);   // 4 slots
  unsigned short* cexp = reinterpret_cast<unsigned short*>(sm + SM::CEXP);
  unsigned short* pexp = reinterpret_cast<unsigned short*>(sm + SM::PEXP);
  if (static_cast<int>(blockIdx.x) >= A.ctas) {
    if (warp < RING_CTA_WARPS)
      ring(A, RING_WARPS * A.ctas + (blockIdx.x - A.ctas) * RING_CTA_WARPS + warp,
           RING_WARPS * A.ctas + (gridDim.x - A.ctas) * RING_CTA_WARPS, lane);
    return;
  }
  const int i0 = 3 + COLS * (static_cast<int>(blockIdx.x) % A.strips);
  const int j0 = 3 + 2 * A.steps_per_seg * (static_cast<int>(blockIdx.x) / A.strips);
  const int rows = min(2 * A.steps_per_seg, n - 2 - j0);   // owned cell rows, up to n - 3
  const int S = (rows + 1) / 2;

  if (tid == 0) {
    for (int k = 0; k < ND; ++k) {
      if (k < ND / 2) mbar_init(bar_full + 8 * k, SLICE_WARPS);
      mbar_init(bar_done + 8 * k, 1);
      mbar_init(bar_done + 8 * (ND + k), 1);
    }
    for (int k = 0; k < MMA_WARPS; ++k) mbar_init(bar_free + 8 * k, EPI_GROUP);
    mbar_init(bar_g, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    *fail = 0;
    for (int k = 0; k < 8; ++k) {
      smax[k] = 0u;
      smin[k] = ~0u;
    }
  }
  for (int k = tid; k < ROWB / 16; k += NT)   // channels 4..7 of the pressures stay zero
    reinterpret_cast<uint4*>(sm + SM::P)[k] = make_uint4(0u, 0u, 0u, 0u);
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(su32(tslot)), "r"(512));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem = *tslot;
  if (tid == 0) {   // the coefficients, while the first window is loaded
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar_g), "r"(GBYTES) : "memory");
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(s0 + SM::G),
        "l"(A.G), "r"(GBYTES), "r"(bar_g)
        : "memory");
  }

  // ---- residuals to digits: a thread takes a cell (a, col) of a row pair q ----
  struct Cell {
    double v[8];
    double p[2];
  };
  auto load = [&](int q, int a, int col, bool act, Cell& c) {   // cell row j0 - 2 + 2 q + a; pressures j0 - 5 + 2 q + 2 a + {0, 1}
    const int gi = i0 - 2 + col, gj = j0 - 2 + 2 * q + a;
    const bool in = act && gi <= n && gj <= n;
#pragma unroll
    for (int o = 0; o < 8; ++o) {
      const int I = 2 * gi + (o & 1), J = 2 * gj + ((o >> 1) & 1);
      c.v[o] = (in && I < nq - 1 && J < nq - 1) ? A.r[(o >> 2) * nv + static_cast<long long>(J) * nq + I] : 0.0;
    }
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const int pj = j0 - 5 + 2 * q + 2 * a + k;
      c.p[k] = (act && q >= 2 && gi <= n && pj <= n) ? A.r[2 * nv + static_cast<long long>(pj) * np + gi] : 0.0;
    }
  };
  // pressures to their units; the pair's largest value (high word); with a check also the
  // smallest nonzero one, and the exponents of the cell and its pressures
  auto note = [&](int q, int a, int col, bool act, Cell& c) {
    c.p[0] *= A.rps;
    c.p[1] *= A.rps;
    auto high = [](double x) { return static_cast<unsigned>(__double2hiint(x)) & 0x7fffffffu; };
    unsigned m = 0u;
#pragma unroll
    for (int o = 0; o < 8; ++o) m = max(m, high(c.v[o]));
    const unsigned all = __reduce_max_sync(0xffffffffu, max(m, max(high(c.p[0]), high(c.p[1]))));
    if (lane == 0) atomicMax(smax + (q & 7), all);
    if (A.check.flags != nullptr) {
      auto mag = [&](double x) { return high(x) | min(static_cast<unsigned>(__double2loint(x)), 1u); };   // zero for zeros only
      auto ex = [](unsigned w) { return static_cast<unsigned short>(max(w >> 20, min(w, 1u))); };
      const unsigned p0 = mag(c.p[0]), p1 = mag(c.p[1]);
      unsigned l = min(p0 - 1u, p1 - 1u), v = 0u;
#pragma unroll
      for (int o = 0; o < 8; ++o) {
        v = max(v, mag(c.v[o]));
        l = min(l, mag(c.v[o]) - 1u);
      }
      if (act) {
        cexp[((q & 7) * 2 + a) * WCOLS + col] = ex(v);
        pexp[((q & 7) * 4 + 2 * a) * WCOLS + col] = ex(p0);
        pexp[((q & 7) * 4 + 2 * a + 1) * WCOLS + col] = ex(p1);
      }
      l = __reduce_min_sync(0xffffffffu, l);
      if (lane == 0) atomicMin(smin + (q & 7), l);
    }
  };
  auto words = [&](const Cell& c, int eb, unsigned long long (&w)[8]) {
#pragma unroll
    for (int o = 0; o < 8; ++o) w[o] = static_cast<unsigned long long>(to_fixed(c.v[o], eb)) + digit_bias();
  };
  auto words_p = [&](const Cell& c, int eb, unsigned long long (&w)[2]) {
#pragma unroll
    for (int k = 0; k < 2; ++k) w[k] = static_cast<unsigned long long>(to_fixed(c.p[k], eb)) + digit_bias();
  };
  auto put = [&](int q, int a, int col, int j, const unsigned long long (&w)[8]) {
    *reinterpret_cast<uint4*>(sm + SM::RING + (2 * (q % 3) + a) * ROWB + j * PLANE + col * 16) =
        make_uint4(digit2(w[0], w[1], j), digit2(w[2], w[3], j), digit2(w[4], w[5], j), digit2(w[6], w[7], j));
  };
  auto put_p = [&](int a, int col, int j, const unsigned long long (&w)[2]) {
    *reinterpret_cast<unsigned*>(sm + SM::P + j * PLANE + col * 16 + 4 * a) = digit2(w[0], w[1], j);
  };
  auto largest = [&](int q) {   // |x| < 2^(e - 1022) over the pairs q - 2 .. q
    const volatile unsigned* vm = smax;
    return static_cast<int>(max(vm[q & 7], max(vm[(q - 1) & 7], vm[(q - 2) & 7])) >> 20);
  };
  auto step_exp = [&](int q, int eb) {   // with the sign if a value of the pairs q - 2 .. q has bits below 2^(E - 58)
    if (A.check.flags == nullptr) return eb;
    const volatile unsigned* vm = smin;
    const unsigned l = min(vm[q & 7], min(vm[(q - 1) & 7], vm[(q - 2) & 7]));
    return eb | (l < (static_cast<unsigned>(eb - 5) << 20) - 1u ? static_cast<int>(0x80000000u) : 0);
  };

  // the first window (row pairs 0, 1, 2) by 27 warps at once
  int eb;
  {
    const int q = warp / SLICE_WARPS, t = tid - q * SLICE_T;
    const bool act = q < 3 && t < 2 * WCOLS;
    const int a = t >= WCOLS ? 1 : 0, col = t - a * WCOLS;
    Cell c;
    if (q < 3) {
      load(q, a, col, act, c);
      note(q, a, col, act, c);
    }
    __syncthreads();
    const int em = largest(2);
    eb = exp_for(em);
    if (act) {
      unsigned long long w[8], wp[2];
      words(c, eb, w);
      words_p(c, eb, wp);
#pragma unroll
      for (int j = 0; j < ND; ++j) {
        put(q, a, col, j, w);
        if (q == 2) put_p(a, col, j, wp);
      }
    }
    if (tid == 0) sexp[0] = step_exp(2, eb);
    fence_proxy();
    __syncthreads();
  }

  const Shared C{bar_full, bar_done, bar_free, tmem, fail, sexp, cexp, pexp, i0, j0, rows, S};
  if (warp < EPI_WARPS) {
    epilogue(A, C, warp / EPI_GROUP, warp, lane);
  } else if (warp < EPI_WARPS + SLICE_WARPS) {
    // ---- the row pairs after the first window ----
    const int t = tid - 32 * EPI_WARPS;
    const bool act = t < 2 * WCOLS;
    const int a = t >= WCOLS ? 1 : 0, col = t - a * WCOLS;
    Cell cur;
    if (S > 1) load(3, a, col, act, cur);
    for (int q = 3; q < S + 2; ++q) {
      note(q, a, col, act, cur);
      asm volatile("bar.sync 1, %0;" ::"n"(SLICE_T) : "memory");
      if (t == 0) {
        smax[(q + 3) & 7] = 0u;
        smin[(q + 3) & 7] = ~0u;
      }
      const int em = largest(q), s = q - 2;
      unsigned long long w[8], wp[2];
      const bool renew = !exp_fits(em, eb);
      if (renew) {   // uniform over the slicer warps: the window again, once the step before has read it
        eb = exp_for(em);
        for (int j = 0; j < ND; ++j)
          mbar_wait_or_fail(bar_done + 8 * (ND * ((s - 1) & 1) + j), ((s - 1) >> 1) & 1, A.wait_limit, fail);
        for (int qq = q - 2; qq < q; ++qq) {
          Cell c;
          load(qq, a, col, act, c);
          words(c, eb, w);
          if (act) {
#pragma unroll
            for (int j = 0; j < ND; ++j) put(qq, a, col, j, w);
          }
        }
      }
      if (t == 0) sexp[s & 3] = step_exp(q, eb);
      words(cur, eb, w);
      words_p(cur, eb, wp);
      if (q + 1 < S + 2) load(q + 1, a, col, act, cur);   // in flight while the planes are written
#pragma unroll
      for (int h = 0; h < ND / 2; ++h) {
        // two planes of the row pair are free once their chains of the step before have read
        // them (after a failed wait the results are void and only the arrivals matter)
        if (!renew) {
          mbar_wait_or_fail(bar_done + 8 * (ND * ((s - 1) & 1) + 2 * h), ((s - 1) >> 1) & 1, A.wait_limit, fail);
          mbar_wait_or_fail(bar_done + 8 * (ND * ((s - 1) & 1) + 2 * h + 1), ((s - 1) >> 1) & 1, A.wait_limit, fail);
        }
        if (act) {
#pragma unroll
          for (int j = 2 * h; j < 2 * h + 2; ++j) {
            put(q, a, col, j, w);
            put_p(a, col, j, wp);
          }
        }
        fence_proxy();
        __syncwarp();
        if (lane == 0) mbar_arrive(bar_full + 8 * h);
      }
    }
  } else if (warp < EPI_WARPS + SLICE_WARPS + MMA_WARPS) {
    // ---- the MMAs ----
    const uint32_t on = elect_one();
    auto wait = [&](uint32_t bar, uint32_t phase) {   // a vote, so that the loop stays uniform
      return __all_sync(0xffffffffu, mbar_wait_or_fail(bar, phase, A.wait_limit, fail)) != 0;
    };
    bool ok = wait(bar_g, 0);
    const int w = warp - (EPI_WARPS + SLICE_WARPS);
    int last = -1;   // the last chain committed, as s ND + c
    const uint32_t gl = desc_lo(s0 + SM::G, CHUNK), pl = desc_lo(s0 + SM::P + 16, 16);
    const uint32_t rl = desc_lo(s0 + SM::RING, 16), r2 = desc_lo(s0 + SM::RING + 64, ROWB);
    for (int s = 0; s < S && ok; ++s) {
      // the row pairs dy = (-2, -1), (0, 1), (2, 3) in units of 16 bytes
      const uint32_t us = s, row[3] = {us % 3 * (ROWB / 8), (us + 1) % 3 * (ROWB / 8), (us + 2) % 3 * (ROWB / 8)};
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int c = w + MMA_WARPS * h;
        if (ok && s > 0) ok = wait(bar_full + 8 * (c >> 1), (s - 1) & 1);   // step 0: the first window
        const int use = 2 * s + h;   // earlier chains of this accumulator
        if (ok && use > 0) ok = wait(bar_free + 8 * w, (use - 1) & 1);
        if (!ok) break;
        fence_after();
        const uint32_t d = tmem + acc_col(w), id = idesc(chain_n(c)), off = c * (PLANE / 16);
        int k = 0;
#pragma unroll
        for (int b = 0; b < 6; ++b)   // cell rows dy = -2 .. 3, offsets dx = (-2, -1) and (0, 1)
#pragma unroll
          for (int e = 0; e < 2; ++e, ++k)
            mma_f16(on, d, rl + off + row[b >> 1] + (b & 1) * (ROWB / 16) + 2 * e, gl + k * (CHUNK / 8), id, k > 0);
#pragma unroll
        for (int b = 0; b < 3; ++b, ++k)   // dx = 2 of both rows of a pair
          mma_f16(on, d, r2 + off + row[b], gl + k * (CHUNK / 8), id, 1);
#pragma unroll
        for (int e = 0; e < 2; ++e, ++k)   // pressures, dx = (-1, 0) and (1, none)
          mma_f16(on, d, pl + off + 2 * e, gl + k * (CHUNK / 8), id, 1);
        mma_commit(on, bar_done + 8 * (ND * (s & 1) + c));
        last = s * ND + c;
      }
    }
    // every chain that was issued has completed before the operands and tensor memory go
    if (last >= 0 && !mbar_wait(bar_done + 8 * (last % (2 * ND)), (last / (2 * ND)) & 1, TC_WAIT_LIMIT)) *fail = 1;
    mbar_wait(bar_g, 0, TC_WAIT_LIMIT);
    __syncwarp();
  } else {
    // ---- cells near the boundary ----
    ring(A, (warp - (EPI_WARPS + SLICE_WARPS + MMA_WARPS)) * A.ctas + blockIdx.x,
         RING_WARPS * A.ctas + (gridDim.x - A.ctas) * RING_CTA_WARPS, lane);
  }
  __syncwarp();
  fence_before();
  __syncthreads();
  fence_after();
  if (tid == 0 && *fail) atomicExch(A.err, 1);
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512));
}

// The pressure of one interior cell by a warp
__device__ __forceinline__ void warp_pressure(const Args& A, int i, int j, int lane) {
  const LevelDev& L = A.L;
  const double* g = A.Gd + static_cast<size_t>(3 * VS_POS + 3) * RT_TYPE + 171 * 8;
  const long long kp = 2 * L.nv + static_cast<long long>(j) * L.np + i;
  double d = 0.0;
  if (lane < 25) {   // all nodes are free
    const double* r = A.r + static_cast<long long>(2 * j - 2 + lane / 5) * L.nq + 2 * i - 2 + lane % 5;
    d = fma(__ldg(g + 2 * lane + 1), __ldg(r + L.nv), __ldg(g + 2 * lane) * __ldg(r));
  } else if (lane == 25) {
    d = A.rps * __ldg(g + 50) * __ldg(A.r + kp);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) d += __shfl_xor_sync(0xffffffffu, d, o);
  if (lane == 0) A.xo[kp] = fma(A.sp, d, A.x != nullptr ? A.x[kp] : 0.0);
}
// The outputs that the contraction leaves to FP64: a warp looks at 32 cells of a row and
// computes the flagged ones one at a time (many pressures by a lane each).  A cell costs
// about fifty times what it costs in the contraction, so they are spread over the whole GPU
// here, not done where they are found: residuals that are large along a wall flag all cells
// of the strips there.
__global__ void __launch_bounds__(128) k_vanka_fp64_cells(const Args A) {
  pdl_begin();
  if (*A.check.any != A.check.call) return;
  const int n = A.L.n, lane = threadIdx.x & 31, w = n - 5, per = (w + 31) / 32;
  Band b;
  b.I0 = b.J0 = 0;
  b.I1 = b.J1 = 8;
  for (int u = blockIdx.x * 4 + (threadIdx.x >> 5); u < w * per; u += gridDim.x * 4) {
    // columns shifted by a row each, or a warp would stay in the same ones
    const int i = 3 + 32 * ((u + u / per) % per) + lane, j = 3 + u / per;
    const unsigned redo = i <= n - 3 ? A.check.flags[static_cast<long long>(j) * A.L.np + i] : 0u;
    const unsigned vel = __ballot_sync(0xffffffffu, redo & 1u), pres = __ballot_sync(0xffffffffu, redo & 2u);
    b.j = j;
    b.in = true;
    for (unsigned m = vel; m != 0; m &= m - 1) {
      b.i = __shfl_sync(0xffffffffu, i, __ffs(m) - 1);
      cell_velocity<4>(A, b, lane);
    }
    if (__popc(pres) > 6) {
      b.i = i;
      if (redo & 2u) cell_pressure(A, b);
      __syncwarp();
    } else {
      for (unsigned m = pres; m != 0; m &= m - 1) warp_pressure(A, __shfl_sync(0xffffffffu, i, __ffs(m) - 1), j, lane);
    }
  }
}

}  // namespace

// Digits of the interior cell type in the K order of the kernel's MMAs.  Row 18 i + 9 a
// + o of the operand is digit i of output o of cell row j + a.  Returns the exponents of
// the velocity and pressure outputs and whether every digit pair sums below 2^24.
bool tc64_pack(std::vector<unsigned char>& out, int* eu, int* ep) {
  const std::vector<long double>& G = vanka_stencil();
  const long double* g0 = G.data() + static_cast<size_t>(3 * VS_POS + 3) * VS_TYPE;
  long double mu = 0.0L, mp = 0.0L;
  for (int o = 0; o < 9; ++o)
    for (int k = 0; k < VS_OUT; ++k) (o < 8 ? mu : mp) = std::max(o < 8 ? mu : mp, std::fabs(g0[o * VS_OUT + k]));
  std::frexp(static_cast<double>(mu) * 1.01, eu);   // max < 2^e / 1.01: the top digit stays within 256
  std::frexp(static_cast<double>(mp) * 1.01, ep);
  out.assign(GBYTES, 0);
  auto chunk_of = [](int dx, int dyi) {   // dyi = dy + 2 in 0..5
    return dx < 2 ? 4 * dyi + dx + 2 : 24 + dyi;
  };
  double sum[NG][18] = {};
  auto place = [&](int a, int o, int chunk, int ch, long double v) {
    long long X = llroundl(std::ldexp(v, 62 - (o < 8 ? *eu : *ep)));
    for (int i = NG - 1; i >= 0; --i) {
      long long d = i > 0 ? ((X + 256) & 511) - 256 : X;
      X = (X - d) >> 9;
      sum[i][9 * a + o] += std::fabs(static_cast<double>(d));
      const __half h = __float2half_rn(static_cast<float>(d));   // exact
      std::memcpy(out.data() + static_cast<size_t>(chunk) * CHUNK + (NBLK * i + 9 * a + o) * 16 + 2 * ch, &h, 2);
    }
  };
  for (int a = 0; a < 2; ++a)
    for (int o = 0; o < 9; ++o) {
      const long double* g = g0 + o * VS_OUT;
      for (int dy = -2; dy <= 3; ++dy)
        for (int dx = -2; dx <= 2; ++dx)
          for (int ch = 0; ch < 8; ++ch) {
            const int J = 2 * (dy - a) + ((ch >> 1) & 1) + 4, I = 2 * dx + (ch & 1) + 4;
            if (J < 0 || J > 8 || I > 8) continue;
            place(a, o, chunk_of(dx, dy + 2), ch, g[(J * 9 + I) * 2 + (ch >> 2)]);
          }
      for (int k = 0; k < 4; ++k)        // pressure row j - 1 + k
        for (int dx = -1; dx <= 1; ++dx) {
          const int dj = k - 1 - a;
          if (dj < -1 || dj > 1) continue;
          place(a, o, 30 + dx + 1, k, g[162 + (dj + 1) * 3 + dx + 1]);
        }
    }
  for (int i = 0; i < NG; ++i)
    for (int o = 0; o < 18; ++o)
      if (sum[i][o] * 512.0 > 16777216.0) return false;
  return true;
}

cudaError_t vanka_tc64_prepare() {
  return cudaFuncSetAttribute(k_vanka_tc64, cudaFuncAttributeMaxDynamicSharedMemorySize, SM::BYTES);
}

void launch_vanka_tc64(const LevelDev& L, const unsigned char* Gp, int eu, int ep, const double* Gd, const double* x,
                       const double* b, double* xo, double omega, double* rscratch, int* err, int wait_limit,
                       const TC64Check& check, cudaStream_t s) {
  const double* r = b;
  if (x != nullptr) {
    launch_apply<double>(L, x, b, rscratch, 1, s);
    r = rscratch;
  }
  int dev = 0, sms = 152;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const int cells = L.n - 5, strips = (cells + COLS - 1) / COLS, steps = (cells + 1) / 2;
  const int seg = segment_steps(strips, steps, sms, 4);
  // SMs left over compute cells near the boundary
  const int ctas = strips * ((steps + seg - 1) / seg), extra = ctas < sms ? sms - ctas : 0;
  Args A{L, Gp, Gd, x, r, xo, omega / L.cl, omega / L.cb, std::ldexp(omega / L.cl, eu), std::ldexp(omega / L.cb, ep),
         L.cl / L.cb, omega, strips, ctas, seg, err, wait_limit, check};
  count_launches(1);
  g_tc_launches.fetch_add(1, std::memory_order_relaxed);
  launch_pdl(k_vanka_tc64, dim3(ctas + extra), dim3(NT), SM::BYTES, s, A);
  if (check.flags != nullptr) {
    count_launches(1);
    launch_pdl(k_vanka_fp64_cells, dim3(4 * sms), dim3(128), 0, s, A);
  }
}

}  // namespace sv
