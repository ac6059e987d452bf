// sv_apply_tc64.cu -- the FP64 operator and residual of the large levels as an exact
// integer contraction on the tensor cores.
//
// The coefficients of the stencils are integers up to 512 (sv_stencil.cuh), exact in
// FP16.  With x in 6 digits of 10 bits (sv_digits.cuh) a digit's products sum to less
// than 2^20, so FP32 holds every sum exactly; the six sums of an output are added in
// 64-bit integers and rounded once, where the FP64 kernel rounds after each of up to 31
// multiply-adds.  The pressure enters the velocity rows scaled by cb / cl, so that one
// contraction gives (A x) / cl.  The only other loss is that of x, truncated 58 bits below
// the bound of the 4 x 132 cells in reach.  Measured against 64-bit mantissas, random x:
// 2.0e-16 of the largest velocity row (FP64 kernel 2.2e-16), 1.6e-16 pressure (2.3e-16).
//
// Columns that the elimination drops (Dirichlet nodes, vertices outside the grid) read
// as zero and every remaining row is the interior one, so one coefficient set serves
// the whole grid; Dirichlet rows are the identity.  Cells with values that are not
// finite in reach are recomputed in FP64, so that they spread as before.
//
// One step is two cell rows of a strip of 128: K = 12 cell offsets (dx -1..1, dy -1..2)
// x 8 + 3 x 4 pressures, 8 MMAs (M = 128 cells, N = 2 rows x 9 outputs padded to 32) per
// digit.  Bound: the instructions around the contraction (digits of 9 values, 54 sums
// per cell: about 700 a vertex) and HBM, no longer the FP64 pipe (334 operations a
// vertex at 2 per clock and SM).  2048^2: 0.34 ms, 0.9 GB moved at 2.7 TB/s with b (the
// FP64 kernel: 1.52 ms); the two epilogue groups took it from 0.367 ms.
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
  static constexpr int BAR = G + GBYTES;         // full[3], done[2], free[2], gload
  static constexpr int MISC = BAR + 16 * 8;      // tmem slot, fail flag, 8 maxima, 4 exponents
  static constexpr int BYTES = MISC + 4 * 16;
  static_assert(G % 128 == 0 && BAR % 8 == 0, "shared memory");
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
// cells with non-finite values in reach
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

// phase of full[s % 3] for step s >= 1 (step 0 needs no arrival)
__device__ __forceinline__ uint32_t full_phase(int s) { return (s % 3 == 0 ? s / 3 - 1 : s / 3) & 1; }

struct Shared {   // what the roles of a CTA share
  uint32_t full, done, free, tmem;
  volatile int* fail;
  volatile int* sexp;
  int i0, j0, rows, S;
};

// Accumulators to y, steps g, g + 2, ...: warp -> cell row a and lane quarter of the
// columns.  The digit sums have weights 2^(50 - 10 c), taken in units of 2^7 (velocity
// rows: the coefficients sum to 1300 at most, |T| < 2^62) and 2^2 (pressure rows: 60).
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
    long long T[9];
    {
      uint32_t v[3][9];
#pragma unroll
      for (int c = 0; c < 3; ++c) tmem_ld9(tq + NB * c, v[c]);
      wait_ld();
#pragma unroll
      for (int o = 0; o < 9; ++o) T[o] = 0;
#pragma unroll
      for (int o = 0; o < 8; ++o) {
        add_digit<43>(T[o], v[0][o]);
        add_digit<33>(T[o], v[1][o]);
        add_digit<23>(T[o], v[2][o]);
      }
      add_digit<48>(T[8], v[0][8]);
      add_digit<38>(T[8], v[1][8]);
      add_digit<28>(T[8], v[2][8]);
#pragma unroll
      for (int c = 0; c < 3; ++c) tmem_ld9(tq + NB * (3 + c), v[c]);
      wait_ld();
#pragma unroll
      for (int o = 0; o < 8; ++o) {
        add_digit<13>(T[o], v[0][o]);
        add_digit<3>(T[o], v[1][o]);
        add_digit<-7>(T[o], v[2][o]);
      }
      add_digit<18>(T[8], v[0][8]);
      add_digit<8>(T[8], v[1][8]);
      add_digit<-2>(T[8], v[2][8]);
    }
    // before the arrival: it lets step s + 2 run, after which the slot takes step s + 4's
    const int eb = C.sexp[s & 3];
    fence_before();
    __syncwarp();
    if (lane == 0) mbar_arrive(C.free + 8 * g);
    const int j = C.j0 + 2 * s + a;
    if (i > n || 2 * s + a >= C.rows) continue;
    if (eb == 0x7ff) {
      for (int o = 0; o < 9; ++o) apply_cell(A, i, j, o);
      continue;
    }
    const long long ku = static_cast<long long>(2 * j) * nq + 2 * i;
    const long long kp = 2 * nv + static_cast<long long>(j) * np + i;
    auto at = [&](int o) { return (o >> 2) * nv + ku + ((o >> 1) & 1) * nq + (o & 1); };
    const bool res = A.b != nullptr;
    const double su = (res ? -L.cl : L.cl) * exp_scale(eb, -51), sp = (res ? -L.cb : L.cb) * exp_scale(eb, -56);
    if (i >= 1 && j >= 1 && i <= n - 1 && j <= n - 1) {   // all four nodes exist and are free
      double bv[9];
#pragma unroll
      for (int o = 0; o < 8; ++o) bv[o] = res ? A.b[at(o)] : 0.0;
      bv[8] = res ? A.b[kp] : 0.0;
#pragma unroll
      for (int o = 0; o < 8; ++o) A.y[at(o)] = fma(su, to_double(T[o]), bv[o]);
      A.y[kp] = fma(sp, to_double(T[8]), bv[8]);
    } else {
#pragma unroll
      for (int o = 0; o < 8; ++o) {
        const int I = 2 * i + (o & 1), J = 2 * j + ((o >> 1) & 1);
        if (I >= nq || J >= nq) continue;
        const long long k = at(o);
        const double b0 = res ? A.b[k] : 0.0;
        if (is_free(I, J, nq)) A.y[k] = fma(su, to_double(T[o]), b0);
        else A.y[k] = res ? b0 - A.x[k] : A.x[k];   // Dirichlet row: identity
      }
      A.y[kp] = fma(sp, to_double(T[8]), res ? A.b[kp] : 0.0);
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
  int* smax = reinterpret_cast<int*>(sm + SM::MISC + 8);                    // 8 slots
  volatile int* sexp = reinterpret_cast<volatile int*>(sm + SM::MISC + 40);   // 4 slots
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
    for (int k = 0; k < 8; ++k) smax[k] = 0;
  }
  for (int k = tid; k < 2 * ROWB / 16; k += NT)   // channels 4..7 of the pressures stay zero
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
  auto note_max = [&](int q, Cell& c) {   // pressures to their units; the pair's largest exponent
    c.p[0] *= A.ps;
    c.p[1] *= A.ps;
    int m = max(__double2hiint(c.p[0]) & 0x7fffffff, __double2hiint(c.p[1]) & 0x7fffffff);
#pragma unroll
    for (int o = 0; o < 8; ++o) m = max(m, __double2hiint(c.v[o]) & 0x7fffffff);
    m = __reduce_max_sync(0xffffffffu, m);
    if (lane == 0) atomicMax(smax + (q & 7), m);
  };
  auto put = [&](int q, int a, int col, int eb, const Cell& c) {
    unsigned long long w[8];
#pragma unroll
    for (int o = 0; o < 8; ++o) w[o] = static_cast<unsigned long long>(to_fixed(c.v[o], eb)) + digit_bias();
#pragma unroll
    for (int j = 0; j < ND; ++j)
      *reinterpret_cast<uint4*>(sm + SM::RING + (2 * (q % 3) + a) * ROWB + j * PLANE + col * 16) =
          make_uint4(digit2(w[0], w[1], j), digit2(w[2], w[3], j), digit2(w[4], w[5], j), digit2(w[6], w[7], j));
  };
  auto put_p = [&](int s, int a, int col, int eb, const Cell& c) {
    unsigned long long w[2];
#pragma unroll
    for (int k = 0; k < 2; ++k) w[k] = static_cast<unsigned long long>(to_fixed(c.p[k], eb)) + digit_bias();
#pragma unroll
    for (int j = 0; j < ND; ++j)
      *reinterpret_cast<unsigned*>(sm + SM::P + (s & 1) * ROWB + j * PLANE + col * 16 + 4 * a) = digit2(w[0], w[1], j);
  };
  auto largest = [&](int q) {   // |x| < 2^(e - 1022) over the pairs q - 1, q
    const volatile int* vm = smax;
    return max(vm[q & 7], vm[(q - 1) & 7]) >> 20;
  };

  // the first window (row pairs 0 and 1) by 18 warps at once
  int eb;
  {
    const int q = warp / SLICE_WARPS, t = tid - q * SLICE_T;
    const bool act = q < 2 && t < 2 * WCOLS;
    const int a = t >= WCOLS ? 1 : 0, col = t - a * WCOLS;
    Cell c;
    if (q < 2) {
      load(q, a, col, act, c);
      note_max(q, c);
    }
    __syncthreads();
    const int em = largest(1);
    eb = min(max(em + 1, EB_MIN), 0x7ff);
    if (act) {
      put(q, a, col, eb, c);
      if (q == 1) put_p(0, a, col, eb, c);
    }
    if (tid == 0) sexp[0] = em < 0x7ff ? eb : 0x7ff;
    fence_proxy();
    __syncthreads();
  }

  const Shared C{bar_full, bar_done, bar_free, tmem, fail, sexp, i0, j0, rows, S};
  if (warp < EPI_WARPS) {
    epilogue(A, C, warp / EPI_GROUP, warp, lane);
  } else if (warp < EPI_WARPS + SLICE_WARPS) {
    // ---- the row pairs after the first window ----
    const int t = tid - 32 * EPI_WARPS;
    const bool act = t < 2 * WCOLS;
    const int a = t >= WCOLS ? 1 : 0, col = t - a * WCOLS;
    Cell cur;
    if (S > 1) load(2, a, col, act, cur);
    for (int q = 2; q < S + 1; ++q) {
      note_max(q, cur);
      asm volatile("bar.sync 1, %0;" ::"n"(SLICE_T) : "memory");
      if (t == 0) smax[(q + 3) & 7] = 0;
      const int em = largest(q), s = q - 1;
      const bool renew = em > eb || (eb - em > 3 && eb > EB_MIN);
      if (renew) {   // uniform over the slicer warps: the other row pair again, with the new exponent
        eb = min(max(em + 1, EB_MIN), 0x7ff);
        mbar_wait_or_fail(bar_done + 8 * ((s - 1) & 1), ((s - 1) >> 1) & 1, A.wait_limit, fail);
        Cell c;
        load(q - 1, a, col, act, c);
        if (act) put(q - 1, a, col, eb, c);
      } else if (s >= 2) {
        // the row pair's slot and the pressure buffer are free once step s - 2 has read them
        // (after a failed wait the results are void and only the arrivals matter)
        mbar_wait_or_fail(bar_done + 8 * (s & 1), ((s - 2) >> 1) & 1, A.wait_limit, fail);
      }
      if (t == 0) sexp[s & 3] = em < 0x7ff ? eb : 0x7ff;
      if (act) {
        put(q, a, col, eb, cur);
        put_p(s, a, col, eb, cur);
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
    for (int o = 0; o < 9; ++o) {
      const int c = o >> 2, py = (o >> 1) & 1, px = o & 1;
      for (int dyi = 0; dyi < 4; ++dyi)
        for (int dx = -1; dx <= 1; ++dx)
          for (int ch = 0; ch < 8; ++ch) {
            const int c2 = ch >> 2, I = 2 * dx + (ch & 1), J = 2 * (dyi - 1 - a) + ((ch >> 1) & 1);
            double v = 0.0;
            if (o == 8) {
              v = c2 == 0 ? crow(I) * nrow(J) : nrow(I) * crow(J);
            } else if (c2 == c) {
              const int dI = I - px, dJ = J - py;
              v = k1(px, dI) * m1(py, dJ) + m1(px, dI) * k1(py, dJ);
            }
            place(a, o, dx < 1 ? 2 * dyi + dx + 1 : 8 + dyi, ch, v);
          }
      if (o == 8) continue;
      for (int k = 0; k < 4; ++k)        // pressure row j - 1 + k
        for (int dx = -1; dx <= 1; ++dx) {
          const int dj = k - 1 - a;
          place(a, o, 12 + dx + 1, k,
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
