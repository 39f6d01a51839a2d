// The separate FP64 tau-line preconditioner (operator and recursions: precond.cu), in fixed
// point (arithmetic: fx.cuh).
//
// A step of either recursion is two real products per component, with 1 - rho and
// rho^{W+1}: 6 integer multiply-adds against 2 FP64 multiply-adds, which take three times
// as long on this GPU.  A lane is one real component (16 sites a row, 256 contiguous
// bytes).  A tile's rows (its slices and the halo, W on either side) are read from global
// memory once, all requested together; their largest component sets the tile's scale, and
// both passes run over shared memory: u rows to x rows, x rows to z.
//
// Growth: x = F_W u and F_W^dagger x each grow a component by at most 1/(1 - rho).  Where
// a coefficient is out of the limbs' range (rho < 0.6), or a tile holds an infinity or a
// NaN, the same passes run in FP64.  So they do, in an application a program calls
// (hqmc_apply_precond), for a tile in which some eight rows of a site lie below 2^-4 of the
// largest component: the small elements of z would have fewer bits than a double there.
// (Gaussian input, L = 48: error of z 7.5e-17 of its 2-norm at one scale, 1.7e-16 in FP64; at
// 2^-4 the former is what FP64's rounding is on values so much smaller.)  CG is judged by
// the norm of its residual.
#include "fx_strip.cuh"
#include "line_pos.cuh"

namespace hqmc {

namespace {
constexpr int kSites = 16;   // per tile; two lanes each
constexpr int kWarps = 8;    // 33 us at L = 48 against 37 with 12 and 43 with 16: each restarts both windows
constexpr size_t kMaxSmem = 226 * 1024;
}  // namespace

size_t line64_smem_bytes(const LineCoef& lc, int tc) { return (size_t)(2 * tc + 3 * lc.W + 2) * 32 * sizeof(double); }

void line_fx_coef(LineCoef& lc) {
  const double om = 1 - lc.rho, sc = lc.scale - 1;
  lc.fx = 0;
  lc.rhoH = std::pow(lc.rho, (lc.W + 1) / 2);
  if (lc.rhoH > 0.4 || !(om > 0) || om > 0.4 || lc.rhoW1 > 0.4 || std::fabs(sc) > 0.4) return;
  // largest operand: x + acc of the backward recursion; cross terms of two real products
  lc.fxF = fx_fraction_bits((1 / om + 1) / om, (std::max(om + lc.rhoW1, std::fabs(sc))) / std::sqrt(2.0));
  if (lc.fxF < 54) return;
  auto limbs = [](double v, int* l) {
    const long long q = std::llrint(std::ldexp(v, 62)) << 2;
    l[0] = fx_hi(q);
    l[1] = fx_lo(q);
  };
  limbs(-om, lc.nom);
  limbs(-lc.rhoW1, lc.nrw);
  limbs(sc, lc.sc1);
  limbs(lc.rhoH, lc.rh);
  lc.fx = 1;
}

// Tiles: heights as line_chunk_candidates sets them (64, 96 at L = 48, 220 at L = 66).  One
// application inside a solve, us, events around each launch, heights 64 / 96 / 165 / 220:
// L = 24 14.3 / 15.8 / 18.4 / 20.4, L = 34 22.7 / 20.8 / 21.9 / 23.2, L = 48 45.0 / 36.8 / 35.0 /
// 45.1, L = 66 100 / 82 / 81 / 105 (a tile of 220 slices fills an SM).
LineLaunch line64_launch(const Geo& g, const LineCoef& lc, int num_sms, size_t smem_per_sm) {
  LineLaunch ll = line_launch(g, line_chunk_candidates(g, 8, lc.W, num_sms, smem_per_sm).front());
  while (ll.chunk > 16 && line64_smem_bytes(lc, ll.chunk) > std::min(smem_per_sm - 1024, kMaxSmem)) ll.chunk /= 2;
  ll = line_launch(g, ll.chunk);
  ll.block = 32 * kWarps;
  ll.gx = (g.V + kSites - 1) / kSites;
  return ll;
}

namespace {

// Conversions for the middle of the exponent range, where a denormal is far below a unit.
// In by integer steps, out by the FP64 pipe's conversion (with the unit's exponent added):
// the two then take about the same time on their pipes (both by integers 105 us at L = 66
// against 99, both by the FP64 pipe 51 against 45 at L = 48 with 16 warps).
__device__ __forceinline__ long long line_from_double(double x, int s0, int flip) {
  const int hi = __double2hiint(x), lo = __double2loint(x);
  const int s = min(s0 - 1 - ((hi >> 20) & 0x7ff), 63);
  const unsigned ah = (__funnelshift_l(lo, hi, 10) & 0x3fffffffu) | 0x40000000u;
  const unsigned long long a = ((unsigned long long)ah << 32) | ((unsigned)lo << 10);
  const long long r = (long long)((a >> s) + 1) >> 1;
  const long long sg = (hi >> 31) ^ flip;
  return (r ^ sg) - sg;
}
__device__ __forceinline__ double line_to_double(long long v, int k) {
  const double d = __ll2double_rn(v);
  const int hi = __double2hiint(d);
  return __hiloint2double(hi == 0 ? 0 : hi + k, __double2loint(d));
}

// The recursions' arithmetic: acc <- v + rho acc; the same with the slice that leaves the
// window; z from the backward sum.
struct LineF64 {
  using T = double;
  const LineCoef& lc;
  __device__ __forceinline__ double square(double sum, double x) const { return fma(x, x, sum); }
  __device__ __forceinline__ double total(double sum) const { return sum; }
  __device__ __forceinline__ double zero() const { return 0.0; }
  __device__ __forceinline__ double step(double v, double acc) const { return fma(lc.rho, acc, v); }
  // a + rho^half b, for the two halves of a window's first sum
  __device__ __forceinline__ double join(double a, double b) const { return fma(lc.rhoH, b, a); }
  __device__ __forceinline__ double slide(double in, double acc, double out) const {
    return fma(-lc.rhoW1, out, fma(lc.rho, acc, in));
  }
  __device__ __forceinline__ double z(double acc) const { return lc.scale * acc; }
};
struct LineFx {
  using T = long long;
  const LineCoef& lc;
  int k;  // exponent of a unit, in the place of a double's upper half
  __device__ __forceinline__ long long zero() const { return 0; }
  // v + rho acc = v + acc - (1 - rho) acc
  __device__ __forceinline__ long long step(long long v, long long acc) const {
    return fx_fma(v + acc, lc.nom[0], lc.nom[1], acc);
  }
  __device__ __forceinline__ long long slide(long long in, long long acc, long long out) const {
    // the terms of `out` first: only two multiply-adds wait for acc
    const int dh = fx_hi(out), dl = fx_lo(out);
    const long long h0 = fx_madw(lc.nrw[0], dh, in);
    const long long c0 = fx_madw(lc.nrw[1], dh, fx_madw(lc.nrw[0], dl, kFxRound));
    const int bh = fx_hi(acc), bl = fx_lo(acc);
    const long long h = fx_madw(lc.nom[0], bh, h0 + acc);
    const long long c = fx_madw(lc.nom[1], bh, fx_madw(lc.nom[0], bl, c0));
    return h + (long long)(int)(c >> 32);
  }
  __device__ __forceinline__ long long join(long long a, long long b) const {
    return fx_fma(a, lc.rh[0], lc.rh[1], b);
  }
  // Sum of x^2 in units of 2^64, each term rounded (x of a tile's largest entries is 2^52
  // and more, a term 2^40): below 2^57.6 each for x < 2^60.8, at most 41 of them per lane.
  __device__ __forceinline__ long long square(long long sum, long long x) const {
    const int h = fx_hi(x), l = fx_lo(x);
    return fx_madw(h, h, sum) + (fx_madw(h, l, 1ll << 30) >> 31);
  }
  __device__ __forceinline__ double total(long long sum) const { return __ll2double_rn(sum) * 0x1p64; }
  __device__ __forceinline__ double z(long long acc) const {
    return line_to_double(fx_fma(acc, lc.sc1[0], lc.sc1[1], acc), k);
  }
};

// Both passes over the staged rows U; zl = this lane's component of row t0 of z, rows V
// sites apart.  The warps split the rows of x, then those of z, into ranges and restart
// the window for each.  Returns the lane's sum of squares of x over the own rows.
template <class A>
__device__ __forceinline__ double line_passes(const A& ar, const typename A::T* __restrict__ U,
                                              typename A::T* __restrict__ X, double* __restrict__ zl, size_t rowlen,
                                              bool ok, bool want_xx, int nt, int W, int warp, int lane, int& za, int& zb) {
  using T = typename A::T;
  const int nx = nt + W + 1;  // rows of x: slices t0 .. t1 + W
  // sum_m rho^(W - m) v(m), m = 0 .. W, as two chains
  auto window = [&](auto v) {
    const int half = (W + 1) / 2;
    T old = ar.zero(), now = ar.zero();
#pragma unroll 2
    for (int m = 0; m < half; ++m) {
      old = ar.step(v(m), old);
      now = ar.step(v(m + W + 1 - half), now);
    }
    if (W + 1 > 2 * half) old = ar.step(v(half), old);  // W even: the middle row
    return ar.join(now, old);
  };
  T xx = ar.zero();
  {
    const int per = (nx + kWarps - 1) / kWarps;
    const int a = warp * per, b = min(nx, a + per);
    if (a < b) {
      T acc = window([&](int m) { return U[(a + m) * 32 + lane]; });
      for (int i = a;;) {
        X[i * 32 + lane] = acc;
        if (want_xx && i < nt) xx = ar.square(xx, acc);
        if (++i == b) break;
        acc = ar.slide(U[(i + W) * 32 + lane], acc, U[(i - 1) * 32 + lane]);
      }
    }
  }
  __syncthreads();
  const int per = (nt + kWarps - 1) / kWarps;
  za = warp * per;
  zb = min(nt, za + per);
  if (za < zb) {
    T acc = window([&](int m) { return X[(zb - 1 + W - m) * 32 + lane]; });
    double* zr = zl + (zb - 1) * rowlen;
    for (int i = zb - 1;; --i, zr -= rowlen) {
      if (ok) *zr = ar.z(acc);
      if (i == za) break;
      acc = ar.slide(X[(i - 1) * 32 + lane], acc, X[(i + W) * 32 + lane]);
    }
  }
  return ar.total(xx);
}

// One tile: 16 sites (column bx), slices [t0, t1).  local: a tile of uneven size in FP64.
__device__ __forceinline__ void line64_tile(const Geo& g, const LineCoef& lc, int t0, int t1,
                                            const double2* __restrict__ u, double2* __restrict__ z,
                                            double* __restrict__ part, int bx, int slot, bool local) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ double red[32];
  __shared__ uint32_t s_key;
  __shared__ int s_uneven;
  const int N = g.Ntau, V = g.V, W = lc.W;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int c = 2 * kSites * bx + lane;  // component of a slice
  const bool ok = c < 2 * V;
  const int cr = ok ? c : 2 * V - 1;  // lanes past the last site read a valid one and store nothing
  const int nt = t1 - t0, nu = nt + 2 * W + 1;  // rows of u: slices t0 - W .. t1 + W
  const size_t rowlen = 2 * (size_t)V;
  double* const U = reinterpret_cast<double*>(smem_raw);
  double* const X = U + (size_t)nu * 32;
  if (threadIdx.x == 0) {
    s_key = 0;
    s_uneven = 0;
  }
  __syncthreads();
  // 1. the rows; every warp copies and converts every eighth
  const LinePos first = line_pos(t0 - W + warp, N);
  {
    int m = first.m;
    const double* const ul = reinterpret_cast<const double*>(u) + cr;
    const uint32_t dst = (uint32_t)__cvta_generic_to_shared(U + lane);
    for (int row = warp; row < nu; row += kWarps) {
      asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(dst + row * 256), "l"(ul + m * rowlen) : "memory");
      for (m += kWarps; m >= N;) m -= N;
    }
    asm volatile("cp.async.wait_all;\n" ::: "memory");
  }
  uint32_t key = 0;
#pragma unroll 4
  for (int row = warp; row < nu; row += kWarps) key = max(key, fx_key(U[row * 32 + lane]));
  key = __reduce_max_sync(0xffffffffu, key);
  if (lane == 0) atomicMax(&s_key, key);
  __syncthreads();
  if (local) {  // uniform over the grid; each group of eight of this warp's rows (the last eight at the end)
    const int nr = nu > warp ? (nu - warp + kWarps - 1) / kWarps : 0;
    bool uneven = false;
    for (int k = 0; k < nr; k += 8) {
      const int k0 = max(0, min(k, nr - 8)), k1 = min(nr, k0 + 8);
      uint32_t big = 0;
      for (int m = k0; m < k1; ++m) big = max(big, fx_key(U[(warp + m * kWarps) * 32 + lane]));
      big = max(big, __shfl_xor_sync(0xffffffffu, big, 1));  // of both components of the site
      uneven |= fx_uneven(big, s_key, 4);
    }
    if (uneven) s_uneven = 1;
    __syncthreads();
  }
  int e = fx_exponent(s_key);
  const bool fixed = lc.fx && e < kFxBad && !(local && s_uneven);
  if (s_key == 0) e = 0;  // all zero: any scale
  // near the ends of the exponent range the rows are scaled on the way in and out
  const bool far = fixed && (e < -800 || e > 800);
  if (far) {
    const int by = e < 0 ? 960 : -960;
    for (int row = warp; row < nu; row += kWarps) U[row * 32 + lane] = scalbn(U[row * 32 + lane], by);
    e = max(e, -1100) + by;
  }
  const int F = lc.fxF;
  {
    const int sb = 1085 - F + e;
    int m = first.m, neg = first.sgn < 0.f ? -1 : 0;  // the sign of the antiperiodic extension
#pragma unroll 2
    for (int row = warp; row < nu; row += kWarps) {
      const double v = U[row * 32 + lane];
      if (fixed) {
        reinterpret_cast<long long*>(U)[row * 32 + lane] = line_from_double(v, sb, neg);
      } else if (neg) {
        U[row * 32 + lane] = -v;
      }
      for (m += kWarps; m >= N;) {
        m -= N;
        neg = ~neg;
      }
    }
  }
  __syncthreads();
  double* const zl = reinterpret_cast<double*>(z) + (size_t)t0 * rowlen + cr;
  int za, zb;
  double xx;
  if (fixed) {
    const LineFx ar{lc, (e - F) * (1 << 20)};
    xx = line_passes(ar, reinterpret_cast<const long long*>(U), reinterpret_cast<long long*>(X), zl, rowlen, ok,
                     part != nullptr, nt, W, warp, lane, za, zb);
  } else {
    xx = line_passes(LineF64{lc}, U, X, zl, rowlen, ok, part != nullptr, nt, W, warp, lane, za, zb);
  }
  if (far) {
    const int by = s_key < (1000u << 20) ? -960 : 960;
    for (int i = za; i < zb && ok; ++i) zl[i * rowlen] = scalbn(zl[i * rowlen], by);
    e += by;
  }
  if (part) {
    double tot = lc.scale * block_sum(ok ? xx : 0.0, red);
    if (fixed) tot = scalbn(scalbn(tot, e - F), e - F);
    if (threadIdx.x == 0) part[slot] = tot;
  }
}

__global__ void __launch_bounds__(32 * kWarps, 3) line_precond64_kernel(Geo g, const __grid_constant__ LineCoef lc, int tc,
                                                                        const double2* __restrict__ u,
                                                                        double2* __restrict__ z, double* __restrict__ part,
                                                                        const CgState* st) {
  pdl_begin();
  if (!line_gate(st)) return;  // uniform over the grid
  const int t0 = blockIdx.y * tc;
  line64_tile(g, lc, t0, min(g.Ntau, t0 + tc), u, z, part, blockIdx.x, blockIdx.y * gridDim.x + blockIdx.x,
              st == nullptr);
}

// Many chains in one launch: block b runs tile tiles[b] = (chain, bx, by) with that
// chain's descriptor, so each chain's tiles and partials are those of its own launch.
__global__ void __launch_bounds__(32 * kWarps, 3) line_precond64_batch_kernel(
    const LineBatchDesc<double>* __restrict__ descs, const int4* __restrict__ tiles) {
  pdl_begin();
  __shared__ LineBatchDesc<double> d;
  const int4 t = tiles[blockIdx.x];
  if (threadIdx.x == 0) d = descs[t.x];
  __syncthreads();
  if (!line_gate(d.st)) return;  // uniform over the block
  const int t0 = t.z * d.tc;
  line64_tile(d.g, d.lc, t0, min(d.g.Ntau, t0 + d.tc), d.u, d.z, d.part, t.y, t.z * d.gx + t.y, false);
}

}  // namespace

cudaError_t prepare_line_precond64(const LineCoef& lc, int tc) {
  return raise_smem_limit(line_precond64_kernel, line64_smem_bytes(lc, tc));
}

cudaError_t launch_line_precond64(const Geo& g, const LineCoef& lc, const LineLaunch& ll, const double2* r, double2* z,
                                  double* part_rz, const CgState* st, cudaStream_t s) {
  return launch_after(line_precond64_kernel, dim3(ll.gx, ll.gy), ll.block, line64_smem_bytes(lc, ll.chunk), s, g, lc, ll.chunk, r, z, part_rz, st);
}

cudaError_t prepare_line_precond64_batch(size_t smem) { return raise_smem_limit(line_precond64_batch_kernel, smem); }

cudaError_t launch_line_precond64_batch(const LineBatchDesc<double>* descs, const int4* tiles, int ntiles, size_t smem,
                                        cudaStream_t s) {
  return launch_after(line_precond64_batch_kernel, ntiles, 32 * kWarps, smem, s, descs, tiles);
}

}  // namespace hqmc
