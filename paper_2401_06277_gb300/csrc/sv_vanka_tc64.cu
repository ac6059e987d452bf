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
//   residual      r = 2^(E - 58) q, |r| < 2^E, q rounded to an integer and written in
//                 6 balanced digits of 10 bits: q = sum_j d_j 1024^(5 - j), |d_j| <= 512
//   coefficients  G = 2^(e_o - 62) g (e_o per output kind), 7 balanced digits of 9 bits,
//                 |g_i| <= 256
// Each digit is exact in FP16.  A pair of digits (i, j) contributes an integer below
// 2^24 (171 products; the bound is computed from the digits when they are packed), so
// the FP32 accumulation is exact in any order.  The pairs with 9 i + 10 j <= 59 (27 of
// 42) are kept; those left out are below 2^-64 of the largest product.  The 27
// integers of an output are added in 64-bit integers and rounded once.  The error is
// that of rounding r to 58 bits below the largest residual of the 6 x 132 cells in
// reach: at most 2^-55 of it, where a sum of 171 FP64 products loses more.
//
// Decomposition.  A CTA owns a strip of 128 cell columns and walks up it two cell rows
// at a time.  The digits of the cells lie in shared memory as planes [cell row][digit]
// [cell column] of 16 bytes (the 8 velocity residuals of a cell): the operand of the
// cells shifted by (dx, dy) is the same memory at another start address, so nothing is
// gathered (an implicit im2col with M = 128 consecutive cells).  One step computes two
// cell rows: K = 30 cell offsets x 8 + 3 x 4 pressures (17 MMAs of K = 16), N = 24
// columns per coefficient digit (9 outputs of each row, padded to 12).  Digit j of the
// residual is one chain of 17 MMAs with N = 24 (7 - j) into an accumulator of its own
// (two alternate); the coefficients (91 KB) stay in shared memory for the whole walk.
//
// Warps: 8 read the accumulators and update x (one cell per thread and row), 9 load
// residuals and write digits, 1 issues the MMAs, and 4 compute the cells near the
// boundary, where the stencil differs, as FP64 dot products on the otherwise idle FP64
// units.  They meet only in mbarriers, per digit: plane j is overwritten for the next
// rows as soon as chain j has read it.
//
// The exponent E is shared by the cells in reach of a step.  It follows the residual:
// when the largest of the window leaves [2^(E-4), 2^E), the digits of the window are
// rewritten with a new E.  A residual that is not finite makes the cells of the step
// NaN.  Every wait is bounded; on expiry the kernel sets *err and returns.
//
// Bound: the tensor pipe and its operand reads.  A chain's MMA takes max(N / 2, 32 +
// N / 4) clocks, 376 for the six: 25 clocks per vertex, 0.33 ms at 2048^2.
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>

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
constexpr int NBLK = 24;                         // N columns per coefficient digit
constexpr int GROWS = NBLK * NG;                 // 168 rows of the coefficient operand
constexpr int KSTEPS = 17;
constexpr int CHUNK = GROWS * 16;                // 8 K-values of all coefficient rows
constexpr int GBYTES = 2 * KSTEPS * CHUNK + 128; // + the rows a padded N reads past the end
static_assert(GBYTES == TC64_BYTES, "size of the packed coefficients");
constexpr int RING_WARPS = 4;
constexpr int NT = 32 * (EPI_WARPS + SLICE_WARPS + 1 + RING_WARPS);

struct SM {
  static constexpr int RING = 0;                         // 6 cell rows
  static constexpr int P = RING + 6 * ROWB;              // pressures of the step: [digit][column] 16 B
  static constexpr int G = P + ROWB;
  static constexpr int BAR = G + GBYTES;                 // full[6], done[6], free[2], gload
  static constexpr int MISC = BAR + 16 * 8;              // tmem slot, fail flag, 8 maxima, 4 exponents
  static constexpr int BYTES = MISC + 4 * 16;
  static_assert(G % 128 == 0 && BAR % 8 == 0 && BYTES <= 227 * 1024, "shared memory");
};

__host__ __device__ constexpr int chain_n(int j) { return (NBLK * (NG - j) + 15) / 16 * 16; }
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
  int steps_per_seg;
  int* err;
  int wait_limit;
};

// FP64 dot products of the cells outside [3, n - 3]^2: three cell rows below and above,
// three columns left and right between them, in units of 8 cells and one output (a
// warp; four lanes per output).
__device__ __forceinline__ int ring_units(int n) {
  return 6 * ((n + 8) / 8) + 6 * ((n - 5 + 7) / 8);
}

__device__ void ring_unit(const Args& A, int unit, int o) {
  const LevelDev& L = A.L;
  const int n = L.n, nq = L.nq, np = L.np, lane = threadIdx.x & 31, part = lane >> 3, c8 = lane & 7;
  const long long nv = L.nv;
  const int w = (n + 8) / 8, h = (n - 5 + 7) / 8;
  int i, j;
  bool in;
  if (unit < 6 * w) {          // rows 0, 1, 2, n - 2, n - 1, n
    const int row = unit / w;
    j = row < 3 ? row : n - 2 + row - 3;
    i = 8 * (unit - row * w) + c8;
    in = i <= n && j <= n;
  } else {                     // columns, rows 3 .. n - 3
    const int v = unit - 6 * w, col = v / h;
    i = col < 3 ? col : n - 2 + col - 3;
    j = 3 + 8 * (v - col * h) + c8;
    in = i <= n && j <= n - 3;
  }
  auto pos = [n](int a) { return a < 3 ? a : a <= n - 3 ? 3 : a >= n ? 6 : a - (n - 2) + 4; };
  const double* g = A.Gd + static_cast<size_t>(pos(in ? j : 0) * VS_POS + pos(in ? i : 0)) * VS_TYPE + o * VS_OUT;
  double a0 = 0.0, a1 = 0.0;
  auto node = [&](int rJ, int rI) {
    const int I = 2 * i - 4 + rI, J = 2 * j - 4 + rJ;
    if (!in || !is_free(I, J, nq)) return;
    const double2 wgt = __ldg(reinterpret_cast<const double2*>(g) + rJ * 9 + rI);
    const double* p = A.r + static_cast<long long>(J) * nq + I;
    a0 = fma(wgt.x, __ldg(p), a0);
    a1 = fma(wgt.y, __ldg(p + nv), a1);
  };
  const int py = o == 8 ? 0 : (o >> 1) & 1, px = o == 8 ? 0 : o & 1;
  if (o == 8) {
#pragma unroll
    for (int e = part; e < 25; e += 4) node(2 + e / 5, 2 + e % 5);
  } else if (px) {
    const int cnt = (9 - 2 * py) * 7;
#pragma unroll 4
    for (int e = part; e < cnt; e += 4) node(2 * py + e / 7, 2 + e % 7);
  } else {
    const int cnt = (9 - 2 * py) * 9;
#pragma unroll 4
    for (int e = part; e < cnt; e += 4) node(2 * py + e / 9, e % 9);
  }
  double ap = 0.0;
  for (int k = part; k < 9; k += 4) {
    const int dj = k / 3 - 1, di = k % 3 - 1, pi = i + di, pj = j + dj;
    if (!in || pi < 0 || pj < 0 || pi > n || pj > n) continue;
    ap = fma(__ldg(g + 162 + k), A.rps * __ldg(A.r + 2 * nv + static_cast<long long>(pj) * np + pi), ap);
  }
  double d = (a0 + a1) + ap;
  d += __shfl_xor_sync(0xffffffffu, d, 8);
  d += __shfl_xor_sync(0xffffffffu, d, 16);
  if (part != 0 || !in) return;
  if (o == 8) {
    const long long k = 2 * nv + static_cast<long long>(j) * np + i;
    A.xo[k] = fma(A.sp, d, A.x != nullptr ? A.x[k] : 0.0);
  } else {
    const int I = 2 * i + px, J = 2 * j + py;
    if (I >= nq || J >= nq) return;
    const long long k = (o >> 2) * nv + static_cast<long long>(J) * nq + I;
    const double xv = A.x != nullptr ? A.x[k] : 0.0;
    A.xo[k] = is_free(I, J, nq) ? fma(A.su, d, xv) : fma(A.omega, A.r[k], xv);
  }
}

// T += D 2^k for the weights of the digit pairs; the compiler makes it one IMAD.WIDE
__device__ __forceinline__ void madw(long long& t, uint32_t f, int k) {
  t += static_cast<long long>(__float2int_rn(__uint_as_float(f))) * (1ll << k);
}

__global__ void __launch_bounds__(NT, 1) k_vanka_tc64(const Args A) {
  pdl_begin();
  extern __shared__ __align__(1024) unsigned char sm[];
  const LevelDev& L = A.L;
  const int n = L.n, nq = L.nq, np = L.np;
  const long long nv = L.nv;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const uint32_t s0 = su32(sm);
  const uint32_t bar_full = s0 + SM::BAR, bar_done = bar_full + 8 * ND, bar_free = bar_done + 8 * ND,
                 bar_g = bar_free + 16;
  uint32_t* tslot = reinterpret_cast<uint32_t*>(sm + SM::MISC);
  volatile int* fail = reinterpret_cast<volatile int*>(sm + SM::MISC + 4);
  int* smax = reinterpret_cast<int*>(sm + SM::MISC + 8);                    // 8 slots
  volatile int* sexp = reinterpret_cast<volatile int*>(sm + SM::MISC + 40);   // 4 slots
  const int i0 = 3 + COLS * static_cast<int>(blockIdx.x);
  const int j0 = 3 + 2 * A.steps_per_seg * static_cast<int>(blockIdx.y);
  const int rows = min(2 * A.steps_per_seg, n - 2 - j0);   // owned cell rows, up to n - 3
  const int S = (rows + 1) / 2;

  if (tid == 0) {
    for (int k = 0; k < ND; ++k) {
      mbar_init(bar_full + 8 * k, SLICE_WARPS);
      mbar_init(bar_done + 8 * k, 1);
    }
    mbar_init(bar_free, EPI_WARPS);
    mbar_init(bar_free + 8, EPI_WARPS);
    mbar_init(bar_g, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    *fail = 0;
    for (int k = 0; k < 8; ++k) smax[k] = 0;
  }
  for (int k = tid; k < ROWB / 16; k += NT)   // channels 4..7 of the pressures stay zero
    reinterpret_cast<uint4*>(sm + SM::P)[k] = make_uint4(0u, 0u, 0u, 0u);
  fence_proxy();
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(su32(tslot)), "r"(512));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem = *tslot;

  if (warp < EPI_WARPS) {
    // ---- accumulators to x: warp -> cell row a, lane quarter of the columns ----
    const int a = warp >> 2, col = 32 * (warp & 3) + lane, i = i0 + col;
    const uint32_t tq = tmem + (static_cast<uint32_t>(32 * (warp & 3)) << 16) + 12 * a;
    for (int s = 0; s < S; ++s) {
      const int j = j0 + 2 * s + a;
      const bool own = i <= n - 3 && 2 * s + a < rows;
      const long long ku = static_cast<long long>(2 * j) * nq + 2 * i;
      const long long kp = 2 * nv + static_cast<long long>(j) * np + i;
      double xv[9];
#pragma unroll
      for (int o = 0; o < 9; ++o) xv[o] = 0.0;
      if (own && A.x != nullptr) {
#pragma unroll
        for (int o = 0; o < 8; ++o) xv[o] = A.x[(o >> 2) * nv + ku + ((o >> 1) & 1) * nq + (o & 1)];
        xv[8] = A.x[kp];
      }
      long long hi[9], lo[9];
#pragma unroll
      for (int o = 0; o < 9; ++o) hi[o] = lo[o] = 0;
      bool ok = true;
#pragma unroll
      for (int c = 0; c < ND; ++c) {
        ok = ok && mbar_wait(bar_done + 8 * c, s & 1, A.wait_limit);
        ok = __all_sync(0xffffffffu, ok) && !*fail;
        if (!ok) break;
        fence_after();
#pragma unroll
        for (int i2 = 0; i2 < NG - c; i2 += 2) {
          uint32_t v[2][9];
          tmem_ld9(tq + 256 * (c & 1) + NBLK * i2, v[0]);
          if (i2 + 1 < NG - c) tmem_ld9(tq + 256 * (c & 1) + NBLK * (i2 + 1), v[1]);
          wait_ld();
#pragma unroll
          for (int u = 0; u < 2; ++u) {
            const int gi = i2 + u, k = 59 - 9 * gi - 10 * c;
            if (gi >= NG - c) continue;
#pragma unroll
            for (int o = 0; o < 9; ++o) {
              if (k >= 30) madw(hi[o], v[u][o], k - 30);
              else madw(lo[o], v[u][o], k);
            }
          }
        }
        fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(bar_free + 8 * (c & 1));
      }
      if (!ok) {
        if (lane == 0) *fail = 1;
        break;
      }
      const int eb = sexp[s & 3];
      const double sc = exp_scale(eb, -57);   // NaN where a residual of the window is not finite
      if (own) {
        const double qu = A.qu * sc, qp = A.qp * sc;
#pragma unroll
        for (int o = 0; o < 9; ++o) {
          const long long t = (hi[o] << 12) + ((lo[o] + (1ll << 17)) >> 18);
          const double d = static_cast<double>(t);
          if (o < 8) A.xo[(o >> 2) * nv + ku + ((o >> 1) & 1) * nq + (o & 1)] = fma(qu, d, xv[o]);
          else A.xo[kp] = fma(qp, d, xv[8]);
        }
      }
    }
  } else if (warp < EPI_WARPS + SLICE_WARPS) {
    // ---- residuals to digits: thread -> cell of the row pair ----
    const int t = tid - 32 * EPI_WARPS;
    const bool act = t < 2 * WCOLS;
    const int a = t >= WCOLS ? 1 : 0, col = act ? t - a * WCOLS : 0, gi = i0 - 2 + col;
    struct Cell {
      double v[8];
      double p[2];
    };
    auto load = [&](int q, Cell& c) {   // row pair q: cell rows j0 - 2 + 2 q + a; pressures j0 - 5 + 2 q + 2 a + {0, 1}
      const int gj = j0 - 2 + 2 * q + a;
      const bool in = act && gi <= n && gj <= n;
#pragma unroll
      for (int o = 0; o < 8; ++o) {
        const int I = 2 * gi + (o & 1), J = 2 * gj + ((o >> 1) & 1);
        c.v[o] = (in && I < nq - 1 && J < nq - 1) ? A.r[(o >> 2) * nv + static_cast<long long>(J) * nq + I] : 0.0;
      }
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        const int pj = j0 - 5 + 2 * q + 2 * a + k;
        c.p[k] = (act && q >= 2 && gi <= n && pj <= n)
                     ? A.rps * A.r[2 * nv + static_cast<long long>(pj) * np + gi] : 0.0;
      }
    };
    int eb = 0;
    auto words = [&](const Cell& c, unsigned long long (&w)[8]) {
#pragma unroll
      for (int o = 0; o < 8; ++o) w[o] = static_cast<unsigned long long>(to_fixed(c.v[o], eb)) + digit_bias();
    };
    auto put = [&](int q, int j, const unsigned long long (&w)[8]) {
      if (!act) return;
      const uint4 d = make_uint4(digit2(w[0], w[1], j), digit2(w[2], w[3], j), digit2(w[4], w[5], j), digit2(w[6], w[7], j));
      *reinterpret_cast<uint4*>(sm + SM::RING + (2 * (q % 3) + a) * ROWB + j * PLANE + col * 16) = d;
    };
    Cell cur, nxt;
    load(0, nxt);
    bool ok = true;
    for (int q = 0; q < S + 2 && ok; ++q) {
      cur = nxt;
      if (q + 1 < S + 2) load(q + 1, nxt);
      int m = 0;
#pragma unroll
      for (int o = 0; o < 8; ++o) m = max(m, __double2hiint(cur.v[o]) & 0x7fffffff);
      m = max(m, max(__double2hiint(cur.p[0]) & 0x7fffffff, __double2hiint(cur.p[1]) & 0x7fffffff));
      m = __reduce_max_sync(0xffffffffu, m);
      if (lane == 0) atomicMax(smax + (q & 7), m);
      asm volatile("bar.sync 1, %0;" ::"n"(SLICE_T) : "memory");
      if (t == 0) smax[(q + 3) & 7] = 0;
      if (q < 2) continue;
      const volatile int* vm = smax;
      const int em = max(vm[q & 7], max(vm[(q - 1) & 7], vm[(q - 2) & 7])) >> 20;   // |x| < 2^(em - 1022)
      const int s = q - 2;
      unsigned long long w[8];
      const bool renew = s == 0 || em > eb || (eb - em > 3 && eb > EB_MIN);
      if (renew) {   // uniform over the slicer warps
        eb = min(max(em + 1, EB_MIN), 0x7ff);
        if (s > 0) ok = mbar_wait(bar_done + 8 * (ND - 1), (s - 1) & 1, A.wait_limit);
        for (int qq = q - 2; qq < q; ++qq) {
          Cell c;
          load(qq, c);
          words(c, w);
#pragma unroll
          for (int j = 0; j < ND; ++j) put(qq, j, w);
        }
      }
      if (t == 0) sexp[s & 3] = em < 0x7ff ? eb : 0x7ff;
      words(cur, w);
      unsigned long long wp[2];
#pragma unroll
      for (int k = 0; k < 2; ++k) wp[k] = static_cast<unsigned long long>(to_fixed(cur.p[k], eb)) + digit_bias();
#pragma unroll
      for (int j = 0; j < ND; ++j) {
        if (!renew && ok) ok = mbar_wait(bar_done + 8 * j, (s - 1) & 1, A.wait_limit);
        if (ok) {
          put(q, j, w);
          if (act) *reinterpret_cast<unsigned*>(sm + SM::P + j * PLANE + col * 16 + 4 * a) = digit2(wp[0], wp[1], j);
        }
        fence_proxy();
        __syncwarp();
        if (lane == 0) mbar_arrive(bar_full + 8 * j);
      }
      if (!ok) *fail = 1;
      ok = !*fail;
      // every slicer warp leaves at the same row pair: the named barrier above counts them all
      asm volatile("bar.sync 1, %0;" ::"n"(SLICE_T) : "memory");
      ok = !*fail;
    }
  } else if (warp == EPI_WARPS + SLICE_WARPS) {
    if (lane == 0) {
      // ---- coefficients, then the MMAs ----
      asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar_g), "r"(GBYTES) : "memory");
      asm volatile(
          "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(s0 + SM::G),
          "l"(A.G), "r"(GBYTES), "r"(bar_g)
          : "memory");
      bool ok = mbar_wait(bar_g, 0, A.wait_limit);
      int issued = 0;   // chains committed
      for (int s = 0; s < S && ok; ++s) {
#pragma unroll 1
        for (int c = 0; c < ND && ok; ++c) {
          ok = mbar_wait(bar_full + 8 * c, s & 1, A.wait_limit);
          const int use = 3 * s + (c >> 1);   // earlier chains of this accumulator
          if (ok && use > 0) ok = mbar_wait(bar_free + 8 * (c & 1), (use - 1) & 1, A.wait_limit);
          if (!ok || *fail) {
            ok = false;
            break;
          }
          fence_after();
          const uint32_t d = tmem + 256 * (c & 1), id = idesc(chain_n(c));
          const uint32_t g0 = s0 + SM::G, pl = s0 + SM::RING + c * PLANE;
          const uint32_t row[3] = {pl + 2 * (s % 3) * ROWB, pl + 2 * ((s + 1) % 3) * ROWB, pl + 2 * ((s + 2) % 3) * ROWB};
          int k = 0;
#pragma unroll
          for (int b = 0; b < 6; ++b)   // cell rows dy = -2 .. 3, offsets dx = (-2, -1) and (0, 1)
#pragma unroll
            for (int h = 0; h < 2; ++h, ++k)
              mma_f16(d, umma_desc(row[b >> 1] + (b & 1) * ROWB + 32 * h, 16, 128),
                      umma_desc(g0 + 2 * k * CHUNK, CHUNK, 128), id, k > 0);
#pragma unroll
          for (int b = 0; b < 3; ++b, ++k)   // dx = 2 of both rows of a pair
            mma_f16(d, umma_desc(row[b] + 64, ROWB, 128), umma_desc(g0 + 2 * k * CHUNK, CHUNK, 128), id, 1);
          const uint32_t pp = s0 + SM::P + c * PLANE + 16;
#pragma unroll
          for (int h = 0; h < 2; ++h, ++k)   // pressures, dx = (-1, 0) and (1, none)
            mma_f16(d, umma_desc(pp + 32 * h, 16, 128), umma_desc(g0 + 2 * k * CHUNK, CHUNK, 128), id, 1);
          mma_commit(bar_done + 8 * c);
          ++issued;
        }
      }
      if (!ok) *fail = 1;
      // every chain that was issued has completed before the operands and tensor memory go
      if (issued > 0) {
        const int last = issued - 1;
        if (!mbar_wait(bar_done + 8 * (last % ND), (last / ND) & 1, TC_WAIT_LIMIT)) *fail = 1;
      }
      mbar_wait(bar_g, 0, TC_WAIT_LIMIT);
    }
    __syncwarp();
  } else {
    // ---- cells near the boundary: units dealt to the ring warps of all CTAs ----
    const int ctas = gridDim.x * gridDim.y, cta = blockIdx.y * gridDim.x + blockIdx.x;
    const int units = 9 * ring_units(n);
    for (int u = (warp - (EPI_WARPS + SLICE_WARPS + 1)) * ctas + cta; u < units; u += RING_WARPS * ctas)
      ring_unit(A, u / 9, u % 9);
  }
  __syncwarp();
  fence_before();
  __syncthreads();
  fence_after();
  if (tid == 0 && *fail) atomicExch(A.err, 1);
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512));
}

}  // namespace

// Digits of the interior cell type in the K order of the kernel's MMAs.  Row 24 i + 12 a
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
      std::memcpy(out.data() + static_cast<size_t>(chunk) * CHUNK + (NBLK * i + 12 * a + o) * 16 + 2 * ch, &h, 2);
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
                       cudaStream_t s) {
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
  Args A{L, Gp, Gd, x, r, xo, omega / L.cl, omega / L.cb, std::ldexp(omega / L.cl, eu), std::ldexp(omega / L.cb, ep),
         L.cl / L.cb, omega, seg, err, wait_limit};
  count_launches(1);
  g_tc_launches.fetch_add(1, std::memory_order_relaxed);
  launch_pdl(k_vanka_tc64, dim3(strips, (steps + seg - 1) / seg), dim3(NT), SM::BYTES, s, A);
}

}  // namespace sv
