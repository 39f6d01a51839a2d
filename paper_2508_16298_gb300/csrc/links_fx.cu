// Link tables of a gauge field from integer arithmetic (fx.cuh): U = t_f e^{i theta} in
// limbs for the fixed-point operators, in FP64 and FP32, and theta as float.
//
// The FP64 sines, cosines and roundings of links_kernel (vec.cu) run at this GPU's FP64
// rate (about 40 operations per angle at 2 per clock and SM); here an angle is 15
// 64-bit integer products, and a wrap to float 10 integer operations.
#include "fx_gauss.cuh"
#include "kernels.h"

#include <cmath>

namespace hqmc {

constexpr int kLinkThreads = 256;
constexpr int kLinkSites = 4;  // sites per thread

int fx_link_blocks(const Geo& g) { return (g.V + kLinkThreads * kLinkSites - 1) / (kLinkThreads * kLinkSites); }

// Constants, computed once (256 logarithms in extended precision take 0.1 ms).
const longlong2* fx_sine_table() {
  struct Table {
    longlong2 v[kDrawTable];
    Table() {
      for (int k = 0; k < 256; ++k) v[k] = fx_table_angle(k, kFxEighth);
      fx_log_table(v + 256);
    }
  };
  static const Table t;
  return t.v;
}

// t (cos, sin)(2 pi k / 256) in units of 2^-64 for t = tanh a, then tanh a / 2 (|t| < 1/2; in
// extended precision, since an error here is in every link alike).
void fx_link_tables(double a, longlong2* tab) {
  for (int f = 0; f < 2; ++f) {
    const __int128 t = (__int128)std::llrint(std::ldexp(std::tanh((long double)a / (f ? 2 : 1)), 64));
    for (int k = 0; k < 256; ++k) {
      const longlong2 e = fx_table_angle(k, kFxEighth);
      const __int128 half = (__int128)1 << 61;
      tab[256 * f + k] = make_longlong2((long long)((t * e.x + half) >> 62), (long long)((t * e.y + half) >> 62));
    }
  }
}

// t e^{i theta} in units of 2^-64.
struct FxLink {
  longlong2 u;
  bool finite;
};
__device__ __forceinline__ FxLink fx_link(double theta, const longlong2* __restrict__ tab, double t) {
  const uint32_t a = fx_abs_hi(theta);
  if (a < kFxMaxAngle) return FxLink{fx_cossin(fx_turns(theta), tab), true};
  if (a < kFxNotFinite) {
    double sn, cs;
    sincos(theta, &sn, &cs);
    return FxLink{make_longlong2(__double2ll_rn(t * cs * 0x1p64), __double2ll_rn(t * sn * 0x1p64)), true};
  }
  return FxLink{make_longlong2(0, 0), false};
}

__device__ __forceinline__ int4 fx_limbs(const FxLink& k) {
  if (!k.finite) return make_int4(kFxBadLink, 0, 0, 0);
  return fx_link_limbs(k.u.x, k.u.y);
}
__device__ __forceinline__ float2 fx_link_float(const FxLink& k) {
  if (!k.finite) return make_float2(__int_as_float(0x7fc00000), __int_as_float(0x7fc00000));
  return make_float2(__ll2float_rn(k.u.x) * 0x1p-64f, __ll2float_rn(k.u.y) * 0x1p-64f);
}
__device__ __forceinline__ double2 fx_link_double(const FxLink& k) {
  const double nan = __longlong_as_double(0x7ff8000000000000ll);
  if (!k.finite) return make_double2(nan, nan);
  return make_double2(fx_to_double_normal(k.u.x, -64), fx_to_double_normal(k.u.y, -64));
}

// Part `sub` of slice tau's sites.
__device__ __forceinline__ void links_fx_part(const Geo& g, const double* __restrict__ theta,
                                              const longlong2* __restrict__ tab, const LinksFx& o, double t1, double t2,
                                              int tau, int sub) {
  const size_t base = (size_t)tau * g.V;
  bool bad = false;
  const int nsub = (g.V + kLinkThreads * kLinkSites - 1) / (kLinkThreads * kLinkSites);
  const int per = (g.V + nsub - 1) / nsub, end = min(g.V, (sub + 1) * per);
  for (int s = sub * per + threadIdx.x; s < end; s += blockDim.x) {
    const size_t i = base + s;
    const double2 th = reinterpret_cast<const double2*>(theta)[i];
    if (o.UF || o.U32 || o.U64) {
      const bool odd = s % g.L & 1;  // odd tail: family 2, else family 1
      const FxLink ux = fx_link(th.x, tab + (odd ? 256 : 0), odd ? t2 : t1);
      const FxLink uy = fx_link(th.y, tab + 256, t2);
      if (o.UF) {
        const int x = s % g.L, y = s / g.L;
        o.UF[2 * base + fx_link_index(g.L, x, y, 0)] = fx_limbs(ux);
        o.UF[2 * base + fx_link_index(g.L, x, y, 1)] = fx_limbs(uy);
        bad |= !ux.finite || !uy.finite;
      }
      if (o.U32) {
        o.U32[2 * i] = fx_link_float(ux);
        o.U32[2 * i + 1] = fx_link_float(uy);
      }
      if (o.U64) {
        o.U64[2 * i] = fx_link_double(ux);
        o.U64[2 * i + 1] = fx_link_double(uy);
      }
    }
    if (o.th32) o.th32[i] = make_float2(fx_wrap_float(th.x), fx_wrap_float(th.y));
  }
  if (o.UF) {
    const int any = __syncthreads_or(bad);
    if (threadIdx.x == 0) o.ubad[tau * nsub + sub] = any ? 1u : 0u;
  }
}

__global__ void __launch_bounds__(kLinkThreads) links_fx_kernel(Geo g, const double* __restrict__ theta,
                                                                const longlong2* __restrict__ tab, LinksFx o, double t1,
                                                                double t2, int nsub) {
  pdl_begin();
  const int tau = blockIdx.x / nsub;
  links_fx_part(g, theta, tab, o, t1, t2, tau, blockIdx.x - tau * nsub);
}

cudaError_t launch_links_fx(const Geo& g, const double* theta, const longlong2* tab, const LinksFx& o, double t1,
                            double t2, cudaStream_t s) {
  const int nsub = fx_link_blocks(g);
  const int threads = g.V >= kLinkThreads ? kLinkThreads : (g.V + 31) / 32 * 32;
  return launch_after(links_fx_kernel, g.Ntau * nsub, threads, 0, s, g, theta, tab, o, t1, t2, nsub);
}

__global__ void __launch_bounds__(kLinkThreads) batch_links_fx_kernel(const ChainDesc* __restrict__ descs,
                                                                      const int2* __restrict__ tiles) {
  pdl_begin();
  const int2 t = tiles[blockIdx.x];
  const ChainDesc& d = descs[t.x];
  const int nsub = (d.g.V + kLinkThreads * kLinkSites - 1) / (kLinkThreads * kLinkSites);
  const int tau = t.y / nsub;
  links_fx_part(d.g, d.theta, d.fxtab, LinksFx{d.UF, d.ubad, nullptr, nullptr, d.U64}, d.t1, d.t2, tau, t.y - tau * nsub);
}

cudaError_t launch_batch_links_fx(const ChainDesc* d, const int2* tiles, int ntiles, cudaStream_t s) {
  return launch_after(batch_links_fx_kernel, ntiles, kLinkThreads, 0, s, d, tiles);
}

}  // namespace hqmc
