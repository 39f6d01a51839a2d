// Register strips of the fixed-point kernels (mdagm_fx.cu, force_fx.cu): shapes, geometry
// and the checkerboard passes of Eq. (eq24) on them.
#pragma once

#include "fx.cuh"
#include "kernels.h"

#include <algorithm>
#include <cmath>

namespace hqmc {

// Fraction bits F of a slice's scale when a component below 2^E may grow by `growth` in
// magnitude and meets factors of modulus up to t: no value may pass 2^62.6, and the
// cross-term accumulator of a complex product, below sqrt(2) t 2^63 + |b|, not 0.95 2^63.
inline int fx_fraction_bits(double growth, double t) {
  const double lim = std::min(std::exp2(62.6), (0.95 - 1.4142135623730951 * t) * std::exp2(63.0));
  return (int)std::floor(std::log2(lim / growth));
}

// Strips of 2 rows (NBY = 1) up to L = 50; above, of 4 rows, where the last strip of a
// slice with L mod 4 = 2 has 2 (its upper rows idle).  Three warps per scheduler, which
// is what strips of 6 rows leave L = 66, ran at 39% issue, waiting on the multiply-add
// chains; 4 rows give it 18 warps instead of 12 in the same registers.
// Block sizes and the registers a thread then has: NBY = 1: 640 (96); NBY = 2: 512
// (128) or 608 (96: L = 66 and 68).
__host__ __device__ inline int fx_nby(int L) { return L <= 50 ? 1 : 2; }
__host__ __device__ inline int fx_threads(int L) { return L / 2 * ((L + 2 * fx_nby(L) - 1) / (2 * fx_nby(L))); }

// W <- P W on a slice in shared memory, FP64, links converted from the table.
static __device__ __noinline__ void slow_sweep(const Geo g, double2* W, const int4* __restrict__ U, const int nt) {
#pragma unroll 1
  for (int k = 0; k < 7; ++k) {
    const int fam = kApplyOrder[6 - k];
    for (int b = threadIdx.x; b < g.V / 2; b += nt) {
      int i, j, c;
      bond_of(g, fam, b, i, j, c);
      const double2 u = fx_link_to_double(U[fx_link_index(g.L, i % g.L, i / g.L, c)]);
      const double2 vi = W[i], vj = W[j];
      W[i] = cfma(vi, u, vj);
      W[j] = cfmac(vj, u, vi);
    }
    __syncthreads();
  }
}

__device__ __forceinline__ bool links_bad(const MdagmArgs<double>& a, int slice) {
  unsigned bad = 0;
  for (int k = 0; k < a.nsub; ++k) bad |= __ldg(a.ubad + slice * a.nsub + k);
  return bad != 0;
}

__device__ __forceinline__ void bond2(longlong2& vi, longlong2& vj, const int4 u) {
  const longlong2 a = vi, b = vj;
  vi = cfma(a, u, b);
  vj = cfmac(b, u, a);
}

// A thread's strip: strip.cuh's geometry, with the rows of the last strip of a slice
// cut to what is left (nr = H, or 2 in a cut strip).
struct FxStrip {
  int L, Lh, i, il, ir, hv;
  int x0, x1;       // own columns 2i + 1, (2i + 2) mod L
  int base, nr;     // first C row, rows
  int own, up;      // row hand-over entries of this strip and of the one above
};

template <int NBY>
__device__ __forceinline__ FxStrip fx_strip(int L, int tid) {
  constexpr int H = 2 * NBY;
  FxStrip s;
  s.L = L;
  s.Lh = L >> 1;
  const int jj = tid / s.Lh, strips = (L + H - 1) / H;
  s.i = tid - jj * s.Lh;
  s.x0 = 2 * s.i + 1;
  s.x1 = (2 * s.i + 2 == L) ? 0 : 2 * s.i + 2;
  s.il = (s.i == 0) ? s.Lh - 1 : s.i - 1;
  s.ir = (s.i == s.Lh - 1) ? 0 : s.i + 1;
  s.hv = L * s.Lh;
  s.base = jj * H;
  s.nr = min(H, L - s.base);
  s.own = jj * L + s.i;
  s.up = (jj + 1 == strips ? 0 : jj + 1) * L + s.i;
  return s;
}
// Row r of the strip in D alignment (base + 1 + r, the last one mod L).
__device__ __forceinline__ int fx_drow(const FxStrip& s, int r) {
  const int y = s.base + 1 + r;
  return y == s.L ? 0 : y;
}

// This thread's own entry of E for row r, column c (planar, as in family 1's exchange).
__device__ __forceinline__ int fx_slot(const FxStrip& s, int r, int c) { return (s.base + r) * s.Lh + s.i + (c ? s.hv : 0); }

template <int N> struct FxInt { static constexpr int v = N; };
struct FxTrue { static constexpr bool value = true; };
struct FxFalse { static constexpr bool value = false; };

// v <- P v on the strip (D alignment on entry and exit), the passes of strip_sweep
// (strip.cuh): F4 [D] | shift | F3 F2 [C] | F1 | F2 F3 [C] | shift | F4 [D].  Links are
// read where they are used (a slice's links do not fit the registers beside the strip;
// they come from L1 or L2), before the barrier where one precedes their use.  Row
// hand-overs go through R0 and R1, which the two barriers between their uses keep apart.
// AHEAD: links of the pass after a barrier are read before it, all at once; else (96
// registers for 4 rows) each where its bond is.
template <int NBY, bool AHEAD>
__device__ __forceinline__ void fx_sweep(longlong2 (&v)[2 * NBY][2], const int4* __restrict__ U, const FxStrip& s,
                                         longlong2* __restrict__ E, longlong2* __restrict__ R0,
                                         longlong2* __restrict__ R1) {
  constexpr int H = 2 * NBY;
  const int L = s.L, Lh = s.Lh;
  const bool full = NBY == 1 || s.nr == H;
  // the strip's links (fx_link_index): x-bonds of row base + r, r Lh entries on; y-bonds with
  // tails on rows base + 2b (even, family 3) and base + 1 + 2b (odd, family 4), b L entries on
  const int4* const U1l = U + s.base * Lh + s.i;         // 2i -> x0
  const int4* const U1r = U + s.base * Lh + s.ir;        // x1 -> 2i + 3
  const int4* const U2 = U1l + L * Lh;                   // x0 -> x1
  const int4* const U3 = U + 2 * L * Lh + (s.base >> 1) * L;
  const int x0 = Lh + s.i, x1 = s.ir;                    // columns x0 (odd) and x1 (even) of a y-bond row
  int4 u[AHEAD ? NBY : 1][2];
  auto load_y = [&](int row0) {
#pragma unroll
    for (int b = 0; b < (AHEAD ? NBY : 0); ++b)
      if (b == 0 || full) {
        u[b][0] = __ldg(U3 + (row0 * Lh + b) * L + x0);
        u[b][1] = __ldg(U3 + (row0 * Lh + b) * L + x1);
      }
  };
  auto pass_y = [&](int row0) {
#pragma unroll
    for (int b = 0; b < NBY; ++b)
      if (b == 0 || full) {
        bond2(v[2 * b][0], v[2 * b + 1][0], AHEAD ? u[AHEAD ? b : 0][0] : __ldg(U3 + (row0 * Lh + b) * L + x0));
        bond2(v[2 * b][1], v[2 * b + 1][1], AHEAD ? u[AHEAD ? b : 0][1] : __ldg(U3 + (row0 * Lh + b) * L + x1));
      }
  };
  auto pass_x = [&]() {
#pragma unroll
    for (int r = 0; r < H; ++r)
      if (r < 2 || full) bond2(v[r][0], v[r][1], __ldg(U2 + r * Lh));
  };
  load_y(1);
  pass_y(1);  // F4
  load_y(0);
  R0[s.up] = full ? v[H - 1][0] : v[1][0];
  R0[s.up + Lh] = full ? v[H - 1][1] : v[1][1];
  __syncthreads();
#pragma unroll
  for (int r = H - 1; r > 0; --r) {
    v[r][0] = v[r - 1][0];
    v[r][1] = v[r - 1][1];
  }
  v[0][0] = R0[s.own];
  v[0][1] = R0[s.own + Lh];
  pass_y(0);  // F3
  pass_x();   // F2
  {
    longlong2* const e0 = E + s.base * Lh + s.i;
    int4 wl[AHEAD ? H : 1], wr[AHEAD ? H : 1];
#pragma unroll
    for (int r = 0; r < H; ++r)
      if (r < 2 || full) {
        if (AHEAD) {
          wl[AHEAD ? r : 0] = __ldg(U1l + r * Lh);
          wr[AHEAD ? r : 0] = __ldg(U1r + r * Lh);
        }
        e0[r * Lh] = v[r][0];
        e0[r * Lh + s.hv] = v[r][1];
      }
    __syncthreads();
    const longlong2* const el = E + s.hv + s.base * Lh + s.il;
    const longlong2* const er = E + s.base * Lh + s.ir;
#pragma unroll
    for (int r = 0; r < H; ++r)
      if (r < 2 || full) {
        v[r][0] = cfmac(v[r][0], AHEAD ? wl[AHEAD ? r : 0] : __ldg(U1l + r * Lh), el[r * Lh]);
        v[r][1] = cfma(v[r][1], AHEAD ? wr[AHEAD ? r : 0] : __ldg(U1r + r * Lh), er[r * Lh]);
      }
  }
  pass_x();   // F2
  load_y(0);
  pass_y(0);  // F3
  load_y(1);
  R1[s.own] = v[0][0];
  R1[s.own + Lh] = v[0][1];
  __syncthreads();
#pragma unroll
  for (int r = 0; r < H - 1; ++r) {
    v[r][0] = v[r + 1][0];
    v[r][1] = v[r + 1][1];
  }
  const longlong2 t0 = R1[s.up], t1 = R1[s.up + Lh];
  if (full) {
    v[H - 1][0] = t0;
    v[H - 1][1] = t1;
  } else {
    v[1][0] = t0;
    v[1][1] = t1;
  }
  pass_y(1);  // F4
}

// The instantiation of a lattice: f(NBY, CAP).
template <class Fn>
inline cudaError_t fx_pick(int L, Fn f) {
  const int n = fx_threads(L);
  if (fx_nby(L) == 1) return f(FxInt<1>{}, FxInt<640>{});
  if (n <= 512) return f(FxInt<2>{}, FxInt<512>{});
  if (n <= 608) return f(FxInt<2>{}, FxInt<608>{});
  return cudaErrorInvalidValue;
}

}  // namespace hqmc
