// sv_apply_tc64.cu -- the FP64 operator and residual of the large levels as an exact
// integer contraction on the tensor cores.
//
// The coefficients of the stencils are integers up to 512 (sv_stencil.cuh), exact in
// FP16.  With x in 6 digits of 12 bits (sv_digits.cuh) a digit's products sum to less
// than 2^22, so FP32 holds every sum exactly; the six sums of an output are added
// exactly and rounded once, where the FP64 kernel rounds after each of up to 31
// multiply-adds.  The pressure enters the velocity rows scaled by cb / cl, so that one
// contraction gives (A x) / cl.
//
// The components keep exponents of their own: u and the pressures in reach share one,
// 2^EU, v and the pressures 2^EV, and the divergence rows sum their two parts apart, so
// that no row sees the size of a component that it does not contain.  The only other
// loss is that of x, truncated 71 bits below 2^EU or 2^EV: nothing of a value within
// 2^-19 of it.  An output whose reach holds smaller values is taken from the contraction
// only if a value of its own row is large enough: one with a coefficient of 32 or more at
// 2^-17 (a velocity node of the cell; 4 or more and 2^-19 in the divergence rows, whose
// coefficients sum to 60 and not 1300), or one with 1 or more at 2^-12 (a pressure).
// What is truncated is then at most 30 units of roundoff of sum |a| |x| over the row,
// less than the a-priori bound of the FP64 kernel (31).  The other outputs, and those
// with values in reach that are not finite, are computed in FP64, within a cycle (whose
// entries are not independent) only the latter.  Error against quadruple precision,
// random x at n = 512: 1.6e-16 of the largest velocity row (FP64 kernel 2.2e-16), 1.3e-16
// pressure (2.3e-16).
//
// Columns that the elimination drops (Dirichlet nodes, vertices outside the grid) read
// as zero and every remaining row is the interior one, so one coefficient set serves
// the whole grid; Dirichlet rows are the identity.
//
// One step is two cell rows of a strip of 128: K = 12 cell offsets (dx -1..1, dy -1..2)
// x 8 + 3 x (4 pressures, in units of 2^EU and of 2^EV), 8 MMAs (M = 128 cells, N = 2
// rows x 10 outputs padded to 32) per digit.  Bound: the latency of the instructions
// around the contraction (digits of 9 values, 60 sums per cell; the two epilogue groups
// and the digit warps are about equally long),
// no longer the FP64 pipe (334 operations a vertex at 2 per clock and SM).  2048^2 with b:
// 0.42 ms (the FP64 kernel: 1.52 ms; 6 digits of 10 bits under one exponent for all
// components, which lost the entries above: 0.355).  All outputs in FP64 (data falling by
// 2^-0.3 per column): 1.99 ms.  Two warps for the pressures alone took 0.44 ms, one
// epilogue group and two threads per cell for the digits 0.59.
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <cmath>
#include <cstdint>
#include <cstring>
#include <vector>

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

constexpr int NB = 32, KSTEPS = 8;               // operand rows (16 a + o), MMAs per digit
constexpr int CHUNK = NB * 16;
constexpr int GBYTES = 2 * KSTEPS * CHUNK;
constexpr int EDGE_WARPS = 2, EDGE_COLS = 8;     // FP64: columns past the last strip, if few
constexpr int NT = 32 * (EPI_WARPS + SLICE_WARPS + 1 + EDGE_WARPS);

struct SM {
  static constexpr int RING = 0;                 // 3 row pairs
  static constexpr int P = RING + 6 * ROWB;      // pressures of a step, two buffers
  static constexpr int G = P + 2 * ROWB;
  static constexpr int CEXP = G + GBYTES;        // exponents of cells: 8 row pairs [row][column] of uint2
  static constexpr int PEXP = CEXP + 8 * 2 * WCOLS * 8;   // of pressures: 8 steps [row][column] of 16 bits
  static constexpr int BAR = PEXP + 8 * 4 * WCOLS * 2;    // full[3], done[2], free[2], gload
  static constexpr int SMAX = BAR + 10 * 8;      // largest u, v, p of 8 row pairs, uint4
  static constexpr int LOST = SMAX + 8 * 16;     // what was truncated in 8 steps
  static constexpr int MISC = LOST + 8 * 4;      // tmem slot, fail flag, 4 exponents
  static constexpr int BYTES = MISC + 6 * 4;
  static_assert(G % 128 == 0 && BAR % 8 == 0 && SMAX % 16 == 0, "shared memory");
};

constexpr uint32_t IDESC = (1u << 4) | (static_cast<uint32_t>(NB >> 3) << 17) | ((128u >> 4) << 24);

struct Args {
  LevelDev L;
  const unsigned char* G;
  const double* x;
  const double* b;       // null: y = A x
  double* y;
  double ps;             // cb / cl
  int strips;
  int steps_per_seg;
  int* err;
  int wait_limit;
};

// Output o of cell (i, j) in FP64, out of line: the columns past the last strip and the
// outputs that the contraction leaves
__device__ __noinline__ void apply_cell(const Args& A, int i, int j, int o) {
  const int res = A.b != nullptr;
  switch (o) {
    case 0: ops::apply_out<double, 0, 0, 0>(A.L, A.x, A.b, A.y, res, i, j); break;
    case 1: ops::apply_out<double, 0, 0, 1>(A.L, A.x, A.b, A.y, res, i, j); break;
    case 2: ops::apply_out<double, 0, 1, 0>(A.L, A.x, A.b, A.y, res, i, j); break;
    case 3: ops::apply_out<double, 0, 1, 1>(A.L, A.x, A.b, A.y, res, i, j); break;
    case 4: ops::apply_out<double, 1, 0, 0>(A.L, A.x, A.b, A.y, res, i, j); break;
    case 5: ops::apply_out<double, 1, 0, 1>(A.L, A.x, A.b, A.y, res, i, j); break;
    case 6: ops::apply_out<double, 1, 1, 0>(A.L, A.x, A.b, A.y, res, i, j); break;
    case 7: ops::apply_out<double, 1, 1, 1>(A.L, A.x, A.b, A.y, res, i, j); break;
    default: ops::apply_out<double, 2, 0, 0>(A.L, A.x, A.b, A.y, res, i, j); break;
  }
}

// Those with their bit (u, v, divergence); out of line too, for the registers (424 -> 415 us)
__device__ __noinline__ void apply_cells(const Args& A, int i, int j, unsigned redo) {
  for (int o = 0; o < 9; ++o)
    if ((redo >> (o >> 2)) & 1) apply_cell(A, i, j, o);
}

// The exponents of a step (E + 1022 of u and v; 0x7ff: values that are not finite) and
// which components were truncated in it: u, v, the pressures in units of either
struct StepExp {
  int eu, ev;
  unsigned lost;
};
constexpr unsigned LOST_U = 1, LOST_V = 2, LOST_PU = 4, LOST_PV = 8;
// Exponents for maxima of mu and mv: kept while they fit within 2^4; one for both if the
// maxima are within 2^3 (the divergence rows then need one sum), until they are 2^6 apart.
__device__ __forceinline__ bool choose_exp(int mu, int mv, int& eu, int& ev) {
  const int m = max(mu, mv), apart = abs(mu - mv);
  if (eu == ev ? exp_fits(m, eu) && (apart <= 5 || eu == EB_MIN) : exp_fits(mu, eu) && exp_fits(mv, ev)) return false;
  eu = exp_for(apart <= 3 ? m : mu);
  ev = exp_for(apart <= 3 ? m : mv);
  return true;
}

// phase of full[s % 3] for step s >= 1 (step 0 needs no arrival)
__device__ __forceinline__ uint32_t full_phase(int s) { return (s % 3 == 0 ? s / 3 - 1 : s / 3) & 1; }

struct Shared {   // what the roles of a CTA share
  uint32_t full, done, free, tmem;
  volatile int* fail;
  volatile unsigned* sexp;
  const volatile unsigned* lost;
  const uint2* cexp;
  const unsigned short* pexp;
  int i0, j0, rows, S;
};

// 2^36 hi + lo as an FP64 number with a single rounding; both below 2^46 and offset by the
// bits of 1.5 2^52, so that they are FP64 numbers as they stand
constexpr long long OFFSET = 0x4338000000000000ll;
__device__ __forceinline__ double total(long long hi, long long lo) {
  constexpr double off = 6755399441055744.0, w = 68719476736.0;   // 1.5 2^52, 2^36
  return fma(__longlong_as_double(hi), w, -(off * w + off)) + __longlong_as_double(lo);
}

// Outputs of a cell that the contraction may not give (bits: u, v, divergence).  a: the
// cell's row in the step, col: its held column.
__device__ __forceinline__ unsigned lost_outputs(const Shared& C, int s, int a, int col, const StepExp& E) {
  const uint2 own = C.cexp[(((s + a) & 7) * 2 + 1 - a) * WCOLS + col];   // row 1 of pair s, row 0 of pair s + 1
  const unsigned short* pe = C.pexp + ((s + 1) & 7) * 4 * WCOLS;
  const int mu = own.x & 0xffffu, mv = own.x >> 16, md = own.y;
  unsigned out = 0;
  if ((E.lost & (LOST_U | LOST_PU)) && mu < E.eu - 16 && pe[(1 + a) * WCOLS + col + 1] < E.eu - 11) out |= 1;
  if ((E.lost & (LOST_V | LOST_PV)) && mv < E.ev - 16 && pe[(2 + a) * WCOLS + col] < E.ev - 11) out |= 2;
  if (md < max((E.lost & LOST_U) ? E.eu : 0, (E.lost & LOST_V) ? E.ev : 0) - 18) out |= 4;
  return out;
}
// Those of them that have anything but zeros in reach
__device__ __forceinline__ unsigned nonzero_reach(const uint2* cexp, const unsigned short* pexp, int s, int a, int col,
                                               unsigned out) {
  unsigned u = 0, v = 0, p = 0;
#pragma unroll 1
  for (int dy = -1; dy <= 1; ++dy)
#pragma unroll 1
    for (int dx = -1; dx <= 1; ++dx) {
      const int r = 2 * s + a + 1 + dy;   // cell row of the walk, row r & 1 of pair r >> 1
      const unsigned w = cexp[((r >> 1 & 7) * 2 + (r & 1)) * WCOLS + col + dx].x;
      u |= w & 0xffffu;
      v |= w >> 16;
      p |= pexp[(((s + 1) & 7) * 4 + 1 + a + dy) * WCOLS + col + dx];
    }
  if ((u | p) == 0) out &= ~1u;
  if ((v | p) == 0) out &= ~2u;
  if ((u | v) == 0) out &= ~4u;
  return out;
}

// Accumulators to y, steps g, g + 2, ...: warp -> cell row a and lane quarter of the columns.
__device__ __forceinline__ void epilogue(const Args& A, const Shared& C, int g, int warp, int lane) {
  const LevelDev& L = A.L;
  const int n = L.n, nq = L.nq, np = L.np;
  const long long nv = L.nv;
  const int a = (warp >> 2) & 1, i = C.i0 + 32 * (warp & 3) + lane;
  const uint32_t tq = C.tmem + (static_cast<uint32_t>(32 * (warp & 3)) << 16) + 16 * a + 256 * g;
  for (int s = g; s < C.S; s += 2) {
    const bool ok = mbar_wait_or_fail(C.done + 8 * g, (s >> 1) & 1, A.wait_limit, C.fail);
    if (!__all_sync(0xffffffffu, ok)) return;
    fence_after();
    double T[8], Tu, Tv = 0.0;   // the outputs' totals; the divergence as one or two
    // before the arrival: it lets step s + 2 run, after which the slot takes step s + 4's
    const unsigned w = C.sexp[s & 3];
    const StepExp E{static_cast<int>(w & 0xffffu), static_cast<int>(w >> 16), C.lost[s & 7]};
    {
      // six digit sums per output, weights 2^(60 - 12 c): three to a 64-bit integer, exact
      long long hi[10];
      uint32_t v[3][10];
#pragma unroll
      for (int c = 0; c < 3; ++c) tmem_ld10(tq + NB * c, v[c]);
      wait_ld();
      auto sum = [&](int o) {
        // an integer below 2^22 plus 1.5 2^23 has its bits at the end of the FP32 number
        auto bits = [](uint32_t f) { return static_cast<long long>(__float_as_int(__uint_as_float(f) + 12582912.0f)); };
        constexpr long long z = 0x4b400000ll;
        return OFFSET - z * ((1 << 24) + (1 << 12) + 1) + bits(v[0][o]) * (1 << 24) + bits(v[1][o]) * (1 << 12) + bits(v[2][o]);
      };
#pragma unroll
      for (int o = 0; o < 10; ++o) hi[o] = sum(o);
#pragma unroll
      for (int c = 0; c < 3; ++c) tmem_ld10(tq + NB * (3 + c), v[c]);
      wait_ld();
#pragma unroll
      for (int o = 0; o < 8; ++o) T[o] = total(hi[o], sum(o));
      if (E.eu == E.ev) {
        Tu = total(hi[8] + (hi[9] - OFFSET), sum(8) + (sum(9) - OFFSET));
      } else {
        Tu = total(hi[8], sum(8));
        Tv = total(hi[9], sum(9));
      }
    }
    const int j = C.j0 + 2 * s + a;
    const bool mine = i <= n && 2 * s + a < C.rows;
    unsigned redo = 0;
    if (mine && E.lost != 0 && L.every_entry) redo = lost_outputs(C, s, a, i - C.i0 + 2, E);
    if (redo != 0) redo = nonzero_reach(C.cexp, C.pexp, s, a, i - C.i0 + 2, redo);
    if (E.eu == 0x7ff) redo |= 5;
    if (E.ev == 0x7ff) redo |= 6;
    fence_before();
    __syncwarp();
    if (lane == 0) mbar_arrive(C.free + 8 * g);
    if (!mine) continue;
    const long long ku = static_cast<long long>(2 * j) * nq + 2 * i;
    const long long kp = 2 * nv + static_cast<long long>(j) * np + i;
    auto at = [&](int o) { return (o >> 2) * nv + ku + ((o >> 1) & 1) * nq + (o & 1); };
    const bool res = A.b != nullptr;
    const double tu = exp_scale(E.eu, -71), tv = exp_scale(E.ev, -71), cl = res ? -L.cl : L.cl, cb = res ? -L.cb : L.cb;
    const double su = cl * tu, sv = cl * tv, pu = cb * tu, pv = cb * tv;
    auto div = [&](double b0) { return E.eu == E.ev ? fma(pu, Tu, b0) : fma(pu, Tu, fma(pv, Tv, b0)); };
    if (i >= 1 && j >= 1 && i <= n - 1 && j <= n - 1 && redo == 0) {   // all four nodes exist and are free
      double bv[9];
#pragma unroll
      for (int o = 0; o < 8; ++o) bv[o] = res ? A.b[at(o)] : 0.0;
      bv[8] = res ? A.b[kp] : 0.0;
#pragma unroll
      for (int o = 0; o < 8; ++o) A.y[at(o)] = fma(o < 4 ? su : sv, T[o], bv[o]);
      A.y[kp] = div(bv[8]);
    } else {   // an output is written once: y may be b
#pragma unroll
      for (int o = 0; o < 8; ++o) {
        const int I = 2 * i + (o & 1), J = 2 * j + ((o >> 1) & 1);
        if (I >= nq || J >= nq || ((redo >> (o >> 2)) & 1)) continue;
        const long long k = at(o);
        const double b0 = res ? A.b[k] : 0.0;
        if (is_free(I, J, nq)) A.y[k] = fma(o < 4 ? su : sv, T[o], b0);
        else A.y[k] = res ? b0 - A.x[k] : A.x[k];   // Dirichlet row: identity
      }
      if (!(redo & 4)) A.y[kp] = div(res ? A.b[kp] : 0.0);
      if (redo != 0) apply_cells(A, i, j, redo);
    }
  }
}

__global__ void __launch_bounds__(NT, 1) k_apply_tc64(const Args A) {
  pdl_begin();
  extern __shared__ __align__(1024) unsigned char sm[];
  const LevelDev& L = A.L;
  const int n = L.n, nq = L.nq, np = L.np;
  const long long nv = L.nv;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const uint32_t s0 = su32(sm);
  const uint32_t bar_full = s0 + SM::BAR, bar_done = bar_full + 24, bar_free = bar_done + 24, bar_g = bar_free + 16;
  uint32_t* tslot = reinterpret_cast<uint32_t*>(sm + SM::MISC);
  volatile int* fail = reinterpret_cast<volatile int*>(sm + SM::MISC + 4);
  unsigned* smax = reinterpret_cast<unsigned*>(sm + SM::SMAX);
  unsigned* lost = reinterpret_cast<unsigned*>(sm + SM::LOST);
  volatile unsigned* sexp = reinterpret_cast<volatile unsigned*>(sm + SM::MISC + 8);   // 4 slots
  uint2* cexp = reinterpret_cast<uint2*>(sm + SM::CEXP);
  unsigned short* pexp = reinterpret_cast<unsigned short*>(sm + SM::PEXP);
  const int i0 = COLS * static_cast<int>(blockIdx.x);
  const int j0 = 2 * A.steps_per_seg * static_cast<int>(blockIdx.y);
  const int rows = min(2 * A.steps_per_seg, n + 1 - j0);
  const int S = (rows + 1) / 2;

  if (tid == 0) {
    for (int k = 0; k < 3; ++k) {
      mbar_init(bar_full + 8 * k, SLICE_WARPS);
      mbar_init(bar_done + 8 * k, 1);
    }
    mbar_init(bar_free, EPI_GROUP);
    mbar_init(bar_free + 8, EPI_GROUP);
    mbar_init(bar_g, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    *fail = 0;
    for (int k = 0; k < 40; ++k) smax[k] = 0u;   // and lost
  }
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

  // ---- values to digits: a thread takes a cell (a, col) of a row pair q ----
  struct Cell {
    double v[8];
    double p[2];
  };
  auto load = [&](int q, int a, int col, bool act, Cell& c) {   // cell row j0 - 1 + 2 q + a; pressures j0 - 3 + 2 q + 2 a + {0, 1}
    const int gi = i0 - 2 + col, gj = j0 - 1 + 2 * q + a;
#pragma unroll
    for (int o = 0; o < 8; ++o) {
      const int I = 2 * gi + (o & 1), J = 2 * gj + ((o >> 1) & 1);
      c.v[o] = (act && is_free(I, J, nq)) ? A.x[(o >> 2) * nv + static_cast<long long>(J) * nq + I] : 0.0;
    }
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const int pj = j0 - 3 + 2 * q + 2 * a + k;
      c.p[k] = (act && q >= 1 && gi >= 0 && gi <= n && pj >= 0 && pj <= n)
                   ? A.x[2 * nv + static_cast<long long>(pj) * np + gi] : 0.0;
    }
  };
  // sizes as high words, a set bit for what lies below them: zero for zeros only
  struct Small {
    unsigned u, v, p;   // the smallest nonzero ones, less one
  };
  auto mag = [](double x) {
    return (static_cast<unsigned>(__double2hiint(x)) & 0x7fffffffu) | min(static_cast<unsigned>(__double2loint(x)), 1u);
  };
  auto smallest = [&](const Cell& c) {
    Small r{~0u, ~0u, min(mag(c.p[0]) - 1u, mag(c.p[1]) - 1u)};
#pragma unroll
    for (int o = 0; o < 4; ++o) {
      r.u = min(r.u, mag(c.v[o]) - 1u);
      r.v = min(r.v, mag(c.v[4 + o]) - 1u);
    }
    return r;
  };
  // pressures to their units; the exponents of the cell; the row pair's largest values
  auto note = [&](int q, int a, int col, bool act, Cell& c) {
    c.p[0] *= A.ps;
    c.p[1] *= A.ps;
    unsigned v[8], m[3] = {0u, 0u, 0u};
#pragma unroll
    for (int o = 0; o < 8; ++o) {
      v[o] = mag(c.v[o]);
      m[o >> 2] = max(m[o >> 2], v[o]);
    }
    const unsigned p0 = mag(c.p[0]), p1 = mag(c.p[1]);
    m[2] = max(p0, p1);
    auto ex = [](unsigned w) { return max(w >> 20, min(w, 1u)); };   // nonzero for every value but zero
    if (act) {
      cexp[((q & 7) * 2 + a) * WCOLS + col] =
          make_uint2(ex(m[0]) | (ex(m[1]) << 16), ex(max(max(v[1], v[3]), max(v[6], v[7]))));
      pexp[((q & 7) * 4 + 2 * a) * WCOLS + col] = static_cast<unsigned short>(ex(p0));
      pexp[((q & 7) * 4 + 2 * a + 1) * WCOLS + col] = static_cast<unsigned short>(ex(p1));
    }
#pragma unroll
    for (int k = 0; k < 3; ++k) m[k] = __reduce_max_sync(0xffffffffu, m[k]);
    if (lane == 0) {
#pragma unroll
      for (int k = 0; k < 3; ++k) atomicMax(smax + 4 * (q & 7) + k, m[k]);
    }
    return smallest(c);
  };
  // exponents of the step with row pairs q - 1 and q; whether they changed
  auto choose = [&](int q, int& eu, int& ev) {
    const uint4 m0 = reinterpret_cast<const uint4*>(smax)[(q - 1) & 7], m1 = reinterpret_cast<const uint4*>(smax)[q & 7];
    // |x| < 2^(e - 1022); the step's pressures came with pair q
    return choose_exp(max(max(m0.x, m1.x), m1.z) >> 20, max(max(m0.y, m1.y), m1.z) >> 20, eu, ev);
  };
  auto truncated = [](const Small& c, int eu, int ev) {
    const unsigned lu = (static_cast<unsigned>(eu - 18) << 20) - 1u, lv = (static_cast<unsigned>(ev - 18) << 20) - 1u;
    return (c.u < lu ? LOST_U : 0u) | (c.v < lv ? LOST_V : 0u) | (c.p < lu ? LOST_PU : 0u) | (c.p < lv ? LOST_PV : 0u);
  };
  auto put = [&](int q, int a, int col, int eu, int ev, const Cell& c) {
    Wide w[8];
#pragma unroll
    for (int o = 0; o < 8; ++o) w[o] = to_wide(c.v[o], o < 4 ? eu : ev);
#pragma unroll
    for (int j = 0; j < ND; ++j)
      *reinterpret_cast<uint4*>(sm + SM::RING + (2 * (q % 3) + a) * ROWB + j * PLANE + col * 16) =
          make_uint4(wide_digit2(w[0], w[1], j), wide_digit2(w[2], w[3], j), wide_digit2(w[4], w[5], j),
                     wide_digit2(w[6], w[7], j));
  };
  auto put_p = [&](int s, int a, int col, int eu, int ev, const Cell& c) {   // in units of 2^EU, then of 2^EV
    unsigned char* p = sm + SM::P + (s & 1) * ROWB + col * 16 + 8 * a;
    const Wide w0 = to_wide(c.p[0], eu), w1 = to_wide(c.p[1], eu);
#pragma unroll
    for (int j = 0; j < ND; ++j) {
      const unsigned u = wide_digit2(w0, w1, j);
      *reinterpret_cast<uint2*>(p + j * PLANE) = make_uint2(u, u);
    }
    if (eu != ev) {
      const Wide z0 = to_wide(c.p[0], ev), z1 = to_wide(c.p[1], ev);
#pragma unroll
      for (int j = 0; j < ND; ++j) *reinterpret_cast<unsigned*>(p + j * PLANE + 4) = wide_digit2(z0, z1, j);
    }
  };

  // the first window (row pairs 0 and 1) by 18 warps at once
  int eu = -1, ev = -1;   // no exponents yet
  {
    const int q = warp / SLICE_WARPS, t = tid - q * SLICE_T;
    const bool act = q < 2 && t < 2 * WCOLS;
    const int a = t >= WCOLS ? 1 : 0, col = t - a * WCOLS;
    Cell c;
    Small small{~0u, ~0u, ~0u};
    if (q < 2) {
      load(q, a, col, act, c);
      small = note(q, a, col, act, c);
    }
    __syncthreads();
    choose(1, eu, ev);
    if (act) {
      put(q, a, col, eu, ev, c);
      if (q == 1) put_p(0, a, col, eu, ev, c);
      const unsigned l = truncated(small, eu, ev);
      if (l != 0) atomicOr(lost, l);
    }
    if (tid == 0) sexp[0] = eu | (ev << 16);
    fence_proxy();
    __syncthreads();
  }

  const Shared C{bar_full, bar_done, bar_free, tmem, fail, sexp, lost, cexp, pexp, i0, j0, rows, S};
  if (warp < EPI_WARPS) {
    epilogue(A, C, warp / EPI_GROUP, warp, lane);
  } else if (warp < EPI_WARPS + SLICE_WARPS) {
    // ---- the row pairs after the first window ----
    const int t = tid - 32 * EPI_WARPS;
    const bool act = t < 2 * WCOLS;
    const int a = t >= WCOLS ? 1 : 0, col = t - a * WCOLS;
    Cell cur;
    if (S > 1) load(2, a, col, act, cur);
    unsigned lost_before = lost[0];   // of this thread's cell of the row pair before; at first, of any
    for (int q = 2; q < S + 1; ++q) {
      const Small small = note(q, a, col, act, cur);
      asm volatile("bar.sync 1, %0;" ::"n"(SLICE_T) : "memory");
      if (t < 3) smax[4 * ((q + 3) & 7) + t] = 0u;
      const int s = q - 1;
      if (choose(q, eu, ev)) {   // uniform over the slicer warps: the other row pair again, with the new exponents
        mbar_wait_or_fail(bar_done + 8 * ((s - 1) & 1), ((s - 1) >> 1) & 1, A.wait_limit, fail);
        Cell c;
        load(q - 1, a, col, act, c);
        if (act) put(q - 1, a, col, eu, ev, c);
        lost_before = truncated(smallest(c), eu, ev);
      } else if (s >= 2) {
        // the row pair's slot and the pressure buffer are free once step s - 2 has read them
        // (after a failed wait the results are void and only the arrivals matter)
        mbar_wait_or_fail(bar_done + 8 * (s & 1), ((s - 2) >> 1) & 1, A.wait_limit, fail);
      }
      if (t == 0) {
        sexp[s & 3] = eu | (ev << 16);
        lost[(s + 1) & 7] = 0u;
      }
      const unsigned l = truncated(small, eu, ev);
      const unsigned lw = __reduce_or_sync(0xffffffffu, l | (lost_before & (LOST_U | LOST_V)));
      if (lw != 0 && lane == 0) atomicOr(lost + (s & 7), lw);
      lost_before = l;
      if (act) {
        put_p(s, a, col, eu, ev, cur);
        put(q, a, col, eu, ev, cur);
      }
      if (q + 1 < S + 1) load(q + 1, a, col, act, cur);   // in flight over the fence and the next barrier
      fence_proxy();
      __syncwarp();
      if (lane == 0) mbar_arrive(bar_full + 8 * (s % 3));
    }
  } else if (warp == EPI_WARPS + SLICE_WARPS) {
    // ---- the MMAs ----
    const uint32_t on = elect_one();
    auto wait = [&](uint32_t bar, uint32_t phase) {   // a vote, so that the loop stays uniform
      return __all_sync(0xffffffffu, mbar_wait_or_fail(bar, phase, A.wait_limit, fail)) != 0;
    };
    bool ok = wait(bar_g, 0);
    int issued = 0;
    for (int s = 0; s < S && ok; ++s) {
      if (s > 0) ok = wait(bar_full + 8 * (s % 3), full_phase(s));   // step 0: the first window
      const int use = s >> 1;
      if (ok && use > 0) ok = wait(bar_free + 8 * (s & 1), (use - 1) & 1);
      if (!ok) break;
      fence_after();
      const uint32_t gl = desc_lo(s0 + SM::G, CHUNK), pl = desc_lo(s0 + SM::P + (s & 1) * ROWB + 16, 16);
      const uint32_t rl = desc_lo(s0 + SM::RING + 16, 16), r2 = desc_lo(s0 + SM::RING + 48, ROWB);
      const uint32_t us = s, pair[2] = {us % 3 * (ROWB / 8), (us + 1) % 3 * (ROWB / 8)};   // units of 16 bytes
#pragma unroll 1
      for (int c = 0; c < ND; ++c) {
        const uint32_t d = tmem + 256 * (s & 1) + NB * c, off = c * (PLANE / 16);
        int k = 0;
#pragma unroll
        for (int b = 0; b < 4; ++b, ++k)   // cell rows dy = -1 .. 2, dx = (-1, 0)
          mma_f16(on, d, rl + off + pair[b >> 1] + (b & 1) * (ROWB / 16), gl + k * (CHUNK / 8), IDESC, k > 0);
#pragma unroll
        for (int b = 0; b < 2; ++b, ++k)   // dx = 1 of both rows of a pair
          mma_f16(on, d, r2 + off + pair[b], gl + k * (CHUNK / 8), IDESC, 1);
#pragma unroll
        for (int e = 0; e < 2; ++e, ++k)   // pressures, dx = (-1, 0) and (1, none)
          mma_f16(on, d, pl + off + 2 * e, gl + k * (CHUNK / 8), IDESC, 1);
      }
      mma_commit(on, bar_done + 8 * (s & 1));
      ++issued;
    }
    // every chain that was issued has completed before the operands and tensor memory go
    if (issued > 0 && !mbar_wait(bar_done + 8 * ((issued - 1) & 1), ((issued - 1) >> 1) & 1, TC_WAIT_LIMIT)) *fail = 1;
    mbar_wait(bar_g, 0, TC_WAIT_LIMIT);
    __syncwarp();
  } else {
    // ---- the columns past the last strip ----
    const int c0 = COLS * A.strips, w = n + 1 - c0;
    const int ctas = gridDim.x * gridDim.y, cta = blockIdx.y * gridDim.x + blockIdx.x;
    const int units = w > 0 ? 9 * ((w * (n + 1) + 31) / 32) : 0;   // 32 cells and one output
    for (int u = (warp - (EPI_WARPS + SLICE_WARPS + 1)) * ctas + cta; u < units; u += EDGE_WARPS * ctas) {
      const int e = (u / 9) * 32 + lane;
      if (e < w * (n + 1)) apply_cell(A, c0 + e % w, e / w, u % 9);
    }
  }
  __syncwarp();
  fence_before();
  __syncthreads();
  fence_after();
  if (tid == 0 && *fail) atomicExch(A.err, 1);
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512));
}

}  // namespace

// The integer coefficients in the K order of the kernel's MMAs: row 16 a + o of the
// operand is output o of cell row j + a.
void apply_tc64_pack(std::vector<unsigned char>& out) {
  out.assign(GBYTES, 0);
  auto place = [&](int a, int o, int chunk, int ch, double v) {
    const __half h = __float2half_rn(static_cast<float>(v));   // integers up to 512: exact
    std::memcpy(out.data() + static_cast<size_t>(chunk) * CHUNK + (16 * a + o) * 16 + 2 * ch, &h, 2);
  };
  for (int a = 0; a < 2; ++a)
    for (int o = 0; o < 10; ++o) {
      const int c = o >> 2, py = (o >> 1) & 1, px = o & 1;   // o = 8, 9: the divergence of u, of v
      for (int dyi = 0; dyi < 4; ++dyi)
        for (int dx = -1; dx <= 1; ++dx)
          for (int ch = 0; ch < 8; ++ch) {
            const int c2 = ch >> 2, I = 2 * dx + (ch & 1), J = 2 * (dyi - 1 - a) + ((ch >> 1) & 1);
            double v = 0.0;
            if (o >= 8) {
              if (c2 == o - 8) v = c2 == 0 ? crow(I) * nrow(J) : nrow(I) * crow(J);
            } else if (c2 == c) {
              const int dI = I - px, dJ = J - py;
              v = k1(px, dI) * m1(py, dJ) + m1(px, dI) * k1(py, dJ);
            }
            place(a, o, dx < 1 ? 2 * dyi + dx + 1 : 8 + dyi, ch, v);
          }
      if (o >= 8) continue;
      for (int k = 0; k < 4; ++k)        // pressure row j - 1 + k
        for (int dx = -1; dx <= 1; ++dx) {
          const int dj = k - 1 - a;
          place(a, o, 12 + dx + 1, 4 * (k >> 1) + 2 * c + (k & 1),   // the pressures in the unit of component c
                c == 0 ? ccol(px, dx) * ncol(py, dj) : ncol(px, dx) * ccol(py, dj));
        }
    }
}

cudaError_t apply_tc64_prepare() {
  return cudaFuncSetAttribute(k_apply_tc64, cudaFuncAttributeMaxDynamicSharedMemorySize, SM::BYTES);
}

void launch_apply_tc64(const LevelDev& L, const double* x, const double* b, double* y, cudaStream_t s) {
  int dev = 0, sms = 152;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  // strips of 128 columns (a remainder of up to EDGE_COLS goes to the FP64 warps: n + 1 is
  // one more than a multiple of 128 on most grids); each with its segments
  const int rem = L.np % COLS, strips = L.np / COLS + (rem > EDGE_COLS ? 1 : 0), steps = (L.np + 1) / 2;
  const int seg = segment_steps(strips, steps, sms, 3);
  Args A{L, L.op_digits, x, b, y, L.cb / L.cl, strips, seg, L.dev_err, L.wait_limit};
  count_launches(1);
  launch_pdl(k_apply_tc64, dim3(strips, (steps + seg - 1) / seg), dim3(NT), SM::BYTES, s, A);
}

}  // namespace sv
