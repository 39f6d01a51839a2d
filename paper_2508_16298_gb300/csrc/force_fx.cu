// Pseudofermion force in fixed point (Supplement SI, Eqs. (force&CG) and (fermion_force);
// the walk over the factors of B is force.cu's, the arithmetic fx.cuh's).
//
// One CTA per slice, u and w in register strips.  With u_k = P(k+1) ... P(7) X_tau and
// w_k = P(k-1) ... P(1) Y_{tau+1}, a bond (i, j) of position k adds
//   -2 cB Im[conj(w_i) U u_j - conj(w_j) conj(U) u_i].
// The step w' = P(k) w has w'_j - w_j = conj(U) w_i and w'_i - w_i = U w_j, so this is
//   -2 cB (Im[conj(w'_j - w_j) u_j] - Im[conj(w'_i - w_i) u_i]):
// one real product sum per site beside the steps of u and w.  The step back of u is
// left unnormalised, (1 - U T) = (1 - t_f^2) P(k)^{-1}: the constant goes into the
// position's coefficient.
//
// Scales: u at slice tau's own exponent with Fu fraction bits (it only grows by P's
// norm), w at the larger of the two slices' with Fw; the host derives both from dtau t
// (fx_force_scales).
//
// The FP64 kernel (force.cu) is bound by the FP64 rate: 21 passes over two slices.  Here,
// per bond and position, 60 integer multiply-adds; NBY = 1 spills about 400 bytes at 96
// registers, NBY = 2 keeps w in shared memory for that reason (444 us without at L = 66).
// Fermion part, fixed point and FP64: L = 24, Ntau = 240: 25 us, 53 us; L = 48, 480: 128,
// 389; L = 66, 660: 387, 905.  Error of dS_f against quad precision: 9e-17 (3.4e-16).
#include "force_slice.cuh"
#include "fx_strip.cuh"

#include <cmath>

namespace hqmc {

FxForceScales fx_force_scales(double a) {
  FxForceScales s{};
  const double t1 = std::tanh(std::fabs(a)), t2 = std::tanh(std::fabs(a) / 2);
  const double cB = std::cosh(a) * std::pow(std::cosh(a / 2), 6);
  const double g = (1 + t1) * std::pow(1 + t2, 6), r2 = std::sqrt(2.0);
  const double gu = r2 * g, gw = r2 * g * (1 + cB * g);  // growth of a component of u and of w
  s.Fu = fx_fraction_bits(gu, t1);
  s.Fw = fx_fraction_bits(gw, t1);
  // high-limb product sum of d = w' - w (|d| <= t |w|) and u: two terms of 2^(Fw + Fu - 64)
  const double hh = 2 * (t1 * gw) * gu * std::ldexp(1.0, s.Fw + s.Fu - 64) + 4;
  s.shift = std::min(20, 62 - (int)std::ceil(std::log2(hh)));
  s.inv1 = 1 / (1 - t1 * t1);
  s.inv2 = 1 / (1 - t2 * t2);
  // -2 cB / prod (1 - t_f^2), with 1 / (1 - tanh^2) = cosh^2; in extended precision, since an
  // error here is in every bond alike
  const long double c1 = std::cosh((long double)a), c2 = std::cosh((long double)a / 2);
  long double c = -2.0L * c1 * c2 * c2 * c2 * c2 * c2 * c2;
  for (int k = 0; k < 7; ++k) {
    c *= k == 3 ? c1 * c1 : c2 * c2;
    s.coef[k] = (double)c;
  }
  return s;
}

// (vi, vj) <- (1 - U T)(vi, vj)
__device__ __forceinline__ void bond2_back(longlong2& vi, longlong2& vj, const int4 u) {
  bond2(vi, vj, make_int4(-u.x, -u.y, -u.z, -u.w));
}

struct FxForceArgs {
  MdagmArgs<double> a;  // geometry, links, x = X
  FxForceScales s;
  double* dSf;
};

// One bond of a position: u back, then w forward; returns the bond's product sum.
__device__ __forceinline__ long long force_bond(longlong2& ui, longlong2& uj, longlong2& wi, longlong2& wj, const int4 k,
                                                int shift) {
  bond2_back(ui, uj, k);
  const longlong2 oi = wi, oj = wj;
  bond2(wi, wj, k);
  return fx_im(make_longlong2(wj.x - oj.x, wj.y - oj.y), uj, shift) -
         fx_im(make_longlong2(wi.x - oi.x, wi.y - oi.y), ui, shift);
}

// The slice in FP64, for non-finite data and for slices of uneven size (fx_uneven), whose small
// elements would have fewer bits than a double.
struct LimbLinks {
  const int4* __restrict__ U;
  int L;
  __device__ __forceinline__ double2 operator()(int i, int c) const {
    return fx_link_to_double(U[fx_link_index(L, i % L, i / L, c)]);
  }
};
static __device__ __noinline__ void slow_force(const MdagmArgs<double>& a, const FxForceScales& fs, double* dSf, int tau,
                                               unsigned char* smem, int nt) {
  force_slice(a.g, a.cB, fs.inv1, fs.inv2, LimbLinks{a.UF + (size_t)tau * a.g.V * 2, a.g.L}, a.x, dSf, tau, smem, nt);
}

template <int NBY>
__device__ __forceinline__ void force_fx_slice(const MdagmArgs<double>& a, const FxForceScales& fs, double* dSf, int tau,
                                               int nt) {
  constexpr int H = 2 * NBY;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ uint32_t s_key[2];
  __shared__ int s_uneven;
  const int V = a.g.V, N = a.g.Ntau, L = a.g.L, Lh = L >> 1;
  longlong2* const E = reinterpret_cast<longlong2*>(smem_raw);
  longlong2* const R0 = E + V;
  longlong2* const R1 = R0 + 2 * nt;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const unsigned wmask = nt - 32 * warp >= 32 ? 0xffffffffu : (1u << (nt - 32 * warp)) - 1u;
  const int taup = (tau == N - 1) ? 0 : tau + 1;
  const double sgn = (tau < N - 1) ? 1.0 : -1.0;
  const size_t bt = (size_t)tau * V, bp = (size_t)taup * V;
  const int4* const U = a.UF + bt * 2;
  const FxStrip s = fx_strip<NBY>(L, tid);
  const bool full = NBY == 1 || s.nr == H;
  if (tid < 2) s_key[tid] = 0;
  if (tid == 0) s_uneven = 0;
  __syncthreads();
  // NBY = 2: w in this thread's slots of shared memory and dS_f summed in place, which the
  // 96 registers of a 4-row strip have no room for
  constexpr bool WREG = NBY == 1;
  longlong2* const W = R1 + 2 * nt;
  longlong2 u[H][2], w[WREG ? H : 1][2];
  auto get_w = [&](int r, int c) -> longlong2 { return WREG ? w[WREG ? r : 0][c] : W[(2 * r + c) * nt + tid]; };
  auto put_w = [&](int r, int c, longlong2 x) {
    if (WREG) w[WREG ? r : 0][c] = x;
    else W[(2 * r + c) * nt + tid] = x;
  };
  uint32_t ku = 0, kw = 0;
#pragma unroll
  for (int r = 0; r < H; ++r)
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      if (r >= 2 && !full) break;
      const size_t i = fx_drow(s, r) * L + (c ? s.x1 : s.x0);
      const double2 x = a.x[bt + i], y = a.x[bp + i];
      u[r][c] = make_longlong2(__double_as_longlong(x.x), __double_as_longlong(x.y));
      put_w(r, c, make_longlong2(__double_as_longlong(y.x), __double_as_longlong(y.y)));
      ku = max(ku, max(fx_key(x.x), fx_key(x.y)));
      kw = max(kw, max(fx_key(y.x), fx_key(y.y)));
    }
  const uint32_t strip_u = ku, strip_w = kw;
  ku = __reduce_max_sync(wmask, ku);
  kw = __reduce_max_sync(wmask, kw);
  if (lane == 0) {
    atomicMax(&s_key[0], ku);
    atomicMax(&s_key[1], kw);
  }
  __syncthreads();
  const int eu = fx_exponent(s_key[0]), ew = max(eu, fx_exponent(s_key[1]));
  bool fp64 = ew >= kFxBad || links_bad(a, tau);
  if (!fp64) {
    if (fx_uneven(strip_u, s_key[0]) || fx_uneven(strip_w, s_key[1])) s_uneven = 1;
    const int s0 = fx_shift_base(eu, fs.Fu);
#pragma unroll
    for (int r = 0; r < H; ++r)
#pragma unroll
      for (int c = 0; c < 2; ++c)
        u[r][c] = make_longlong2(fx_from_double(__longlong_as_double(u[r][c].x), s0),
                                 fx_from_double(__longlong_as_double(u[r][c].y), s0));
    fx_sweep<NBY, NBY == 1>(u, U, s, E, R0, R1);  // P X_tau
    fp64 = s_uneven != 0;  // set before the sweep's barriers
  }
  if (fp64) {
    __syncthreads();  // the sweep's last reads of R1
    slow_force(a, fs, dSf, tau, smem_raw, nt);
    return;
  }
  {  // w = Y_{tau+1} = X_{tau+1} - s cB P X_tau
    const int s0 = fx_shift_base(ew, fs.Fw), n = ew - eu + fs.Fu - fs.Fw;
    const bool plus = taup == 0;  // the antiperiodic wrap
#pragma unroll
    for (int r = 0; r < H; ++r)
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        const longlong2 z = make_longlong2(fx_shr(fx_fma(u[r][c].x, a.cm1h, a.cm1l, u[r][c].x), n),
                                           fx_shr(fx_fma(u[r][c].y, a.cm1h, a.cm1l, u[r][c].y), n));
        const longlong2 y = get_w(r, c);
        const longlong2 x = make_longlong2(fx_from_double(__longlong_as_double(y.x), s0),
                                           fx_from_double(__longlong_as_double(y.y), s0));
        put_w(r, c, plus ? make_longlong2(x.x + z.x, x.y + z.y) : make_longlong2(x.x - z.x, x.y - z.y));
      }
  }
  const int es = ew - fs.Fw + eu - fs.Fu + 64 - fs.shift;  // a product sum counts 2^es
  const int4* const U1l = U + s.base * Lh + s.i;
  const int4* const U1r = U + s.base * Lh + s.ir;
  const int4* const U2 = U1l + L * Lh;
  const int4* const U3 = U + 2 * L * Lh + (s.base >> 1) * L;
  const int x0 = Lh + s.i, x1 = s.ir;
  // dS_f of C row r, column c, direction: own x-bonds (tails x0, x1) and y-bonds
  double d[WREG ? H : 1][2][2];
  double2* const out = reinterpret_cast<double2*>(dSf) + bt;
  auto add = [&](int r, int c, int dir, double coef, double v, bool again) {
    if (WREG) {
      double& o = d[WREG ? r : 0][c][dir];
      o = again ? fma(coef, v, o) : __dmul_rn(coef, v);
    } else {
      double* const o = reinterpret_cast<double*>(out + (s.base + r) * L + (c ? s.x1 : s.x0)) + dir;
      *o = again ? fma(coef, v, *o) : __dmul_rn(coef, v);
    }
  };
  // families 4 (D, row0 = 1) and 3 (C, row0 = 0): tails on C rows row0 + 2b
  auto pass_y = [&](auto row, double coef, bool again) {
    constexpr int row0 = decltype(row)::v;
#pragma unroll
    for (int b = 0; b < NBY; ++b)
      if (b == 0 || full)
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          const int4 k = __ldg(U3 + (row0 * Lh + b) * L + (c ? x1 : x0));
          longlong2 wi = get_w(2 * b, c), wj = get_w(2 * b + 1, c);
          const double v = fx_to_double(force_bond(u[2 * b][c], u[2 * b + 1][c], wi, wj, k, fs.shift), es);
          put_w(2 * b, c, wi);
          put_w(2 * b + 1, c, wj);
          add(2 * b + row0, c, 1, coef, v, again);
        }
  };
  auto pass_x = [&](double coef, bool again) {
#pragma unroll
    for (int r = 0; r < H; ++r)
      if (r < 2 || full) {
        longlong2 wi = get_w(r, 0), wj = get_w(r, 1);
        const double v = fx_to_double(force_bond(u[r][0], u[r][1], wi, wj, __ldg(U2 + r * Lh), fs.shift), es);
        put_w(r, 0, wi);
        put_w(r, 1, wj);
        add(r, 0, 0, coef, v, again);
      }
  };
  // one row to the strip above (D -> C) or below; u through R0, w through R1
  const int last = full ? H - 1 : 1;
  auto shift_up = [&]() {
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      R0[s.up + c * Lh] = full ? u[H - 1][c] : u[1][c];
      R1[s.up + c * Lh] = get_w(last, c);
    }
  };
  auto take_up = [&]() {
#pragma unroll
    for (int c = 0; c < 2; ++c) {
#pragma unroll
      for (int r = H - 1; r > 0; --r) {
        u[r][c] = u[r - 1][c];
        put_w(r, c, get_w(r - 1, c));
      }
      u[0][c] = R0[s.own + c * Lh];
      put_w(0, c, R1[s.own + c * Lh]);
    }
  };
  auto take_down = [&]() {
#pragma unroll
    for (int c = 0; c < 2; ++c) {
#pragma unroll
      for (int r = 0; r < H - 1; ++r) {
        u[r][c] = u[r + 1][c];
        put_w(r, c, get_w(r + 1, c));
      }
      const longlong2 t = R0[s.up + c * Lh];
      if (full) u[H - 1][c] = t;
      else u[1][c] = t;
      put_w(last, c, R1[s.up + c * Lh]);
    }
  };
  pass_y(FxInt<1>{}, sgn * fs.coef[0], false);  // position 1: family 4
  __syncthreads();                // the forward sweep's last reads of R1
  shift_up();
  __syncthreads();
  take_up();
  pass_y(FxInt<0>{}, sgn * fs.coef[1], false);  // 2: family 3
  pass_x(sgn * fs.coef[2], false);              // 3: family 2
  {                               // 4: family 1, u then w through E, then the heads' sums
    longlong2* const e0 = E + s.base * Lh + s.i;
    const longlong2* const el = E + s.hv + s.base * Lh + s.il;
    const longlong2* const er = E + s.base * Lh + s.ir;
#pragma unroll
    for (int r = 0; r < H; ++r)
      if (r < 2 || full) {
        e0[r * Lh] = u[r][0];
        e0[r * Lh + s.hv] = u[r][1];
      }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < H; ++r)
      if (r < 2 || full) {
        const int4 kl = __ldg(U1l + r * Lh), kr = __ldg(U1r + r * Lh);
        u[r][0] = cfmac(u[r][0], make_int4(-kl.x, -kl.y, -kl.z, -kl.w), el[r * Lh]);
        u[r][1] = cfma(u[r][1], make_int4(-kr.x, -kr.y, -kr.z, -kr.w), er[r * Lh]);
      }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < H; ++r)
      if (r < 2 || full) {
        e0[r * Lh] = get_w(r, 0);
        e0[r * Lh + s.hv] = get_w(r, 1);
      }
    __syncthreads();
    long long head[H], tail[H];
#pragma unroll
    for (int r = 0; r < H; ++r)
      if (r < 2 || full) {
        const int4 kl = __ldg(U1l + r * Lh), kr = __ldg(U1r + r * Lh);
        const longlong2 o0 = get_w(r, 0), o1 = get_w(r, 1);
        const longlong2 n0 = cfmac(o0, kl, el[r * Lh]), n1 = cfma(o1, kr, er[r * Lh]);
        put_w(r, 0, n0);
        put_w(r, 1, n1);
        head[r] = fx_im(make_longlong2(n0.x - o0.x, n0.y - o0.y), u[r][0], fs.shift);
        tail[r] = fx_im(make_longlong2(n1.x - o1.x, n1.y - o1.y), u[r][1], fs.shift);
      }
    __syncthreads();
    long long* const h0 = reinterpret_cast<long long*>(E);
#pragma unroll
    for (int r = 0; r < H; ++r)
      if (r < 2 || full) h0[(s.base + r) * Lh + s.i] = head[r];
    __syncthreads();
#pragma unroll
    for (int r = 0; r < H; ++r)
      if (r < 2 || full)
        add(r, 1, 0, sgn * fs.coef[3], fx_to_double(h0[(s.base + r) * Lh + s.ir] - tail[r], es), false);
  }
  pass_x(sgn * fs.coef[4], true);               // 5: family 2
  pass_y(FxInt<0>{}, sgn * fs.coef[5], true);   // 6: family 3
#pragma unroll
  for (int c = 0; c < 2; ++c) {
    R0[s.own + c * Lh] = u[0][c];
    R1[s.own + c * Lh] = get_w(0, c);
  }
  __syncthreads();
  take_down();
  pass_y(FxInt<1>{}, sgn * fs.coef[6], true);   // 7: family 4
  if (WREG) {
#pragma unroll
    for (int r = 0; r < H; ++r) {
      const int y = (s.base + r) * L;
      out[y + s.x0] = make_double2(d[WREG ? r : 0][0][0], d[WREG ? r : 0][0][1]);
      out[y + s.x1] = make_double2(d[WREG ? r : 0][1][0], d[WREG ? r : 0][1][1]);
    }
  }
}

template <int NBY, int CAP>
__global__ void __launch_bounds__(CAP, 1) force_fx_kernel(const __grid_constant__ FxForceArgs f) {
  pdl_begin();
  force_fx_slice<NBY>(f.a, f.s, f.dSf, blockIdx.x, (int)blockDim.x);
}

// The force of many chains: block b serves slice tile.y of chain tile.x (x of its
// descriptor: X).
template <int NBY, int CAP>
__global__ void __launch_bounds__(CAP, 1) force_fx_batch_kernel(const MdagmArgs<double>* __restrict__ descs,
                                                                const ChainDesc* __restrict__ chains,
                                                                const int4* __restrict__ tiles) {
  pdl_begin();
  __shared__ MdagmArgs<double> a;
  __shared__ FxForceScales fs;
  const int4 t = tiles[blockIdx.x];
  if (threadIdx.x == 0) {
    a = descs[t.x];
    a.x = chains[t.x].X;
    fs = chains[t.x].fs;
  }
  __syncthreads();
  const int H = 2 * NBY, nt = (a.g.L >> 1) * ((a.g.L + H - 1) / H);
  if ((int)threadIdx.x >= nt) return;
  force_fx_slice<NBY>(a, fs, chains[t.x].dSf, t.y, nt);
}

// Two slices of shared memory at least: what the FP64 walk of a non-finite slice needs.
static size_t force_smem(const Geo& g) {
  const size_t n = g.V + (fx_nby(g.L) == 1 ? 4 : 12) * (size_t)fx_threads(g.L);
  return (n > 2 * (size_t)g.V ? n : 2 * (size_t)g.V) * sizeof(longlong2);
}

cudaError_t prepare_force_fx(const Geo& g) {
  return fx_pick(g.L, [&](auto nby, auto cap) { return raise_smem_limit(force_fx_kernel<nby.v, cap.v>, force_smem(g)); });
}

cudaError_t launch_force_fx(const MdagmArgs<double>& a, const FxForceScales& fs, double* dSf, cudaStream_t s) {
  return fx_pick(a.g.L, [&](auto nby, auto cap) {
    return launch_after(force_fx_kernel<nby.v, cap.v>, a.g.Ntau, fx_threads(a.g.L), force_smem(a.g), s, FxForceArgs{a, fs, dSf});
  });
}

cudaError_t launch_force_fx_batch(const MdagmArgs<double>* descs, const ChainDesc* chains, const int4* tiles, int ntiles,
                                  int Lmax, cudaStream_t s) {
  const Geo g{Lmax, Lmax * Lmax, Lmax / 2, 1};
  return fx_pick(Lmax, [&](auto nby, auto cap) {
    const cudaError_t e = raise_smem_limit(force_fx_batch_kernel<nby.v, cap.v>, force_smem(g));
    if (e != cudaSuccess) return e;
    return launch_after(force_fx_batch_kernel<nby.v, cap.v>, ntiles, fx_threads(Lmax), force_smem(g), s, descs, chains, tiles);
  });
}

}  // namespace hqmc
