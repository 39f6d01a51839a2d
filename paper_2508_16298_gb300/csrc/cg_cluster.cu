// Plain FP64 conjugate gradients of a small lattice, in one thread-block cluster.
//
// With a few thousand sites an iteration of the two-kernel loop is nothing but latency:
// two launches, and in each a head that sums the other's partials (19 us at L = 8, Ntau = 40
// for 0.3 MFLOP).  Here one cluster of up to 16 CTAs, which the hardware starts together,
// runs the iterations of a whole loop body: a CTA owns up to ceil(Ntau / 16) slices, a thread
// one bond of each checkerboard family of one slice (their links in registers) and two
// sites (x, r, p in registers).  Slices meet through distributed shared memory: an
// iteration has three cluster barriers, after z = P p is published and after each of the
// two dot products, whose warp sums every CTA adds in the same order.  The factor passes run
// in fixed point (fx.cuh) where the hopping allows it: 14 passes of FP64 products are 3.5 us
// of an iteration at 8^2 x 40.  What is left is the FP64 pipe (2 lanes a clock per SM on 16
// SMs) in the vector work, and the chains of the two sums and their divisions.
//   time of an iteration    L = 8, Ntau = 40    6, 40    10, 100    12, 120
//   two kernels [us]                    18.8     27.8       22.7       22.6
//   here, passes in FP64                10.2     13.7       19.4    (576 threads: not used)
//   here                                 9.4     13.3       14.8
// (a trajectory of 11 solves at 8^2 x 40: 59.7 -> 29.8 ms; short solves count their start
// here, so 6^2 is not below 8^2).  Up to 384 threads, one bond of each family for each, in 154
// to 162 registers; 576 threads, which 12^2 x 120 needs, would have 112 each (not measured).
#include "fx_strip.cuh"
#include "kernels.h"

#include <cooperative_groups.h>

namespace cg = cooperative_groups;

namespace hqmc {

namespace {

constexpr int kMaxCtas = 16, kMaxThreads = 384, kMaxWarps = kMaxThreads / 32;

__device__ __forceinline__ void cluster_sync_all() {
  __syncwarp();
  asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;\n" ::: "memory");
}

struct Shared {
  double part[2][kMaxCtas * kMaxWarps];  // warp sums of <p, q> and <r, r> of all CTAs
  double value;                          // step length, or beta of the next direction
  uint32_t key[2];                       // of the largest component before each sweep
  int stop;
};

// Sum over the cluster: every warp's sum goes to all CTAs, whose first warp adds them.
// The result is valid in the first warp.
__device__ __forceinline__ double cluster_sum(cg::cluster_group& cl, Shared& sh, int which, double v, int C, int nw) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  v = __shfl_sync(0xffffffffu, warp_sum(v), 0);
  if (lane < C) cl.map_shared_rank(&sh, lane)->part[which][warp * C + (int)cl.block_rank()] = v;
  cluster_sync_all();
  return warp == 0 ? warp_sum_partials(sh.part[which], C * nw) : 0.0;
}

// Slices [tb, te) of CTA `rank`.
__device__ __forceinline__ int slice_begin(int rank, int N, int per) { return min(N, rank * per); }

// FX: the sweeps in fixed point at the scale of the CTA's largest component (F fraction bits).
template <bool FX>
__global__ void __launch_bounds__(kMaxThreads, 1) cg_cluster_kernel(const MdagmArgs<double> a, double2* __restrict__ xg,
                                                                    double2* __restrict__ rg, int per, int max_its,
                                                                    int F) {
  pdl_begin();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ Shared sh;
  cg::cluster_group cl = cg::this_cluster();
  const int rank = (int)cl.block_rank(), C = (int)cl.num_blocks();
  const int V = a.g.V, N = a.g.Ntau, nb = V >> 1, T = per * nb, nw = blockDim.x >> 5;
  double2* const P = reinterpret_cast<double2*>(smem_raw);  // p, z and w of this CTA's slices
  double2* const Z = P + per * V;
  double2* const W = Z + per * V;
  longlong2* const Q = reinterpret_cast<longlong2*>(W);
  CgState* const st = a.st;
  const int tid = threadIdx.x;
  const int tb = slice_begin(rank, N, per), nt = slice_begin(rank + 1, N, per) - tb;
  int k = st->k;
  const int seg = st->seg_start, maxit = st->maxit;
  const double tol2bb = st->tol2bb;
  const bool run = *(volatile int*)&st->done == CG_RUNNING;
  double rr = k == seg ? st->rr[k & 1] : a.part_in[0], rr_old = st->rr[(k + 1) & 1];
  if (tid == 0) sh.key[0] = sh.key[1] = 0;
  cluster_sync_all();  // every CTA has read the state
  if (!run) return;

  // this thread's bonds: slice tid / nb of the CTA, bond tid % nb of each family
  int ij[4];
  double2 u[4];  // FP64
  int4 uf[4];    // FX: limbs
  {
    const int sl = tid / nb, b = tid - sl * nb;
    const bool ok = tid < T && sl < nt;
#pragma unroll
    for (int f = 0; f < 4; ++f) {
      int i = 0, j = 0, c = 0;
      bond_of(a.g, f + 1, ok ? b : 0, i, j, c);
      u[f] = ok ? __ldg(a.U + 2 * ((size_t)(tb + sl) * V + i) + c) : make_double2(0.0, 0.0);
      if (FX) uf[f] = fx_link_limbs(__double2ll_rn(u[f].x * 0x1p64), __double2ll_rn(u[f].y * 0x1p64));
      ij[f] = ok ? (sl * V + i) | ((sl * V + j) << 16) : -1;
    }
  }
  // its sites: two neighbours of the CTA's nt V
  const int e[2] = {2 * tid, 2 * tid + 1};
  bool own[2];
  double2 x[2], r[2], p[2];
  const double2* p0 = (k & 1) ? a.pbuf[1] : a.pbuf[0];
#pragma unroll
  for (int s = 0; s < 2; ++s) {
    own[s] = tid < T && e[s] < nt * V;
    const size_t gi = (size_t)tb * V + e[s];
    x[s] = r[s] = p[s] = make_double2(0.0, 0.0);
    if (own[s]) {
      x[s] = xg[gi];
      r[s] = rg[gi];
      if (k != seg) p[s] = p0[gi];
    }
  }
  auto sweep = [&](double2* v) {  // v <- P v on every slice (families 4 3 2 1 2 3 4)
#pragma unroll
    for (int m = 0; m < 7; ++m) {
      constexpr int fam[7] = {3, 2, 1, 0, 1, 2, 3};
      const int f = fam[m];
      if (ij[f] >= 0) {
        const int i = ij[f] & 0xffff, j = ij[f] >> 16;
        const double2 ul = FX ? __ldg(a.U + 2 * ((size_t)tb * V + i) + (f >= 2 ? 1 : 0)) : u[f];
        const double2 vi = v[i], vj = v[j];
        v[i] = cfma(vi, ul, vj);
        v[j] = cfmac(vj, ul, vi);
      }
      __syncthreads();
    }
  };
  auto sweep_fx = [&]() {
#pragma unroll
    for (int m = 0; m < 7; ++m) {
      constexpr int fam[7] = {3, 2, 1, 0, 1, 2, 3};
      const int f = fam[m];
      if (ij[f] >= 0) {
        const int i = ij[f] & 0xffff, j = ij[f] >> 16;
        const longlong2 vi = Q[i], vj = Q[j];
        Q[i] = cfma(vi, uf[f], vj);
        Q[j] = cfmac(vj, uf[f], vi);
      }
      __syncthreads();
    }
  };
  // v <- P v for this thread's sites (with a barrier before and after); buf: work in FP64.
  // Scales near the ends of the exponent range, zeros and non-finite values take FP64.
  auto apply = [&](double2 (&v)[2], double2* buf, int which) {
    if (FX) {
      uint32_t key = 0;
#pragma unroll
      for (int s = 0; s < 2; ++s)
        if (own[s]) key = max(key, max(fx_key(v[s].x), fx_key(v[s].y)));
      key = __reduce_max_sync(0xffffffffu, key);
      if ((tid & 31) == 0) atomicMax(&sh.key[which], key);
      __syncthreads();
      const int e10 = fx_exponent(sh.key[which]);
      if (tid == 0) sh.key[which ^ 1] = 0;  // of the next call: last read before this barrier
      if (e10 > -800 && e10 < 800) {
        const int sb = fx_shift_base(e10, F);
#pragma unroll
        for (int s = 0; s < 2; ++s)
          if (own[s]) Q[e[s]] = make_longlong2(fx_from_double(v[s].x, sb), fx_from_double(v[s].y, sb));
        __syncthreads();
        sweep_fx();
#pragma unroll
        for (int s = 0; s < 2; ++s)
          if (own[s])
            v[s] = make_double2(fx_to_double_normal(Q[e[s]].x, e10 - F), fx_to_double_normal(Q[e[s]].y, e10 - F));
        return;
      }
    }
#pragma unroll
    for (int s = 0; s < 2; ++s)
      if (own[s]) buf[e[s]] = v[s];
    __syncthreads();
    sweep(buf);
#pragma unroll
    for (int s = 0; s < 2; ++s)
      if (own[s]) v[s] = buf[e[s]];
  };
  const double cB = a.cB;
  // the slices before and after this CTA's (another CTA's, or its own other end)
  const int tl = tb == 0 ? N - 1 : tb - 1, tr = tb + nt == N ? 0 : tb + nt;
  const double2* const Zl = cl.map_shared_rank(Z, tl / per) + (tl % per) * V;
  const double2* const Pr = cl.map_shared_rank(P, tr / per) + (tr % per) * V;
  int done = CG_RUNNING;
  double pq_last = 0.0, alpha_last = 0.0;
  bool first = k == seg;
  for (int it = 0;; ++it) {
    // head: every CTA takes the same decisions from the same sums
    double beta = 0.0;
    if (k >= maxit) done = CG_MAXIT;
    else if (!first) {
      if (tid < 32) {
        int stop = CG_RUNNING;
        if (!isfinite(rr)) stop = CG_NONFINITE;
        else if (rr <= tol2bb) stop = CG_REC_CONVERGED;
        else if (!(rr > 0.0)) stop = CG_BREAKDOWN;
        else beta = rr / rr_old;
        if (tid == 0) {
          sh.stop = stop;
          sh.value = beta;
        }
      }
      __syncthreads();
      done = sh.stop;
      beta = sh.value;
    }
    if (done != CG_RUNNING || it == max_its) break;
    double2 z[2], w[2];
#pragma unroll
    for (int s = 0; s < 2; ++s)
      if (own[s]) {
        p[s] = first ? r[s] : caxpy(r[s], beta, p[s]);
        P[e[s]] = p[s];
        z[s] = p[s];
      }
    first = false;
    apply(z, Z, 0);
    if (FX) {
#pragma unroll
      for (int s = 0; s < 2; ++s)
        if (own[s]) Z[e[s]] = z[s];
    }
    cluster_sync_all();  // p and z = P p of all slices
    double2 t[2];
#pragma unroll
    for (int s = 0; s < 2; ++s)
      if (own[s]) {
        const int sl = e[s] >= V ? e[s] / V : 0, site = e[s] - sl * V, tau = tb + sl;
        const double sig = tau == 0 ? -1.0 : 1.0, sigp = tau == N - 1 ? -1.0 : 1.0;
        const double2 zl = sl == 0 ? Zl[site] : Z[e[s] - V];
        const double2 pr = sl == nt - 1 ? Pr[site] : P[e[s] + V];
        t[s] = caxpy(p[s], -sig * cB, zl);
        w[s] = caxpy(cscale(cB, z[s]), -sigp, pr);
      }
    apply(w, W, 1);
    double acc = 0.0;
    double2 q[2];
#pragma unroll
    for (int s = 0; s < 2; ++s)
      if (own[s]) {
        q[s] = caxpy(t[s], cB, w[s]);
        acc += cdot_re_own(p[s], q[s]);
      }
    double pq = cluster_sum(cl, sh, 0, acc, C, nw);
    if (tid < 32) {
      const bool bad = !isfinite(pq) || !(pq > 0.0);
      if (tid == 0) {
        sh.stop = bad ? (isfinite(pq) ? CG_BREAKDOWN : CG_NONFINITE) : CG_RUNNING;
        sh.value = bad ? 0.0 : rr / pq;
      }
    }
    __syncthreads();
    done = sh.stop;
    if (done != CG_RUNNING) break;
    const double alpha = sh.value;
    if (tid == 0) {
      pq_last = pq;
      alpha_last = alpha;
    }
    acc = 0.0;
#pragma unroll
    for (int s = 0; s < 2; ++s)
      if (own[s]) {
        r[s] = caxpy(r[s], -alpha, q[s]);
        x[s] = caxpy(x[s], alpha, p[s]);
        acc += cdot_re_own(r[s], r[s]);
      }
    const double rn = cluster_sum(cl, sh, 1, acc, C, nw);
    rr_old = rr;
    rr = rn;  // the first warp's; the others take decisions from it through sh
    ++k;
  }
  double2* pn = (k & 1) ? a.pbuf[1] : a.pbuf[0];
#pragma unroll
  for (int s = 0; s < 2; ++s)
    if (own[s]) {
      const size_t gi = (size_t)tb * V + e[s];
      xg[gi] = x[s];
      rg[gi] = r[s];
      pn[gi] = p[s];
    }
  if (rank == 0 && tid == 0) {
    st->k = st->k2 = k;
    st->rr[k & 1] = rr;
    if (k != seg) st->rr[(k + 1) & 1] = rr_old;
    const_cast<double*>(a.part_in)[0] = rr;
    if (pq_last != 0.0) {
      st->pq_last = pq_last;
      st->alpha_last = alpha_last;
    }
    st->done = done;
  }
}

size_t cluster_smem(const Geo& g, int per) { return (size_t)3 * per * g.V * sizeof(double2); }

}  // namespace

ClusterCg cg_cluster_shape(const Geo& g, double t1, double t2) {
  ClusterCg c{};
  c.fx = std::fabs(t1) <= kFxMaxLink;
  // growth of a component through P (fx_strip.cuh)
  c.F = fx_fraction_bits(std::sqrt(2.0) * (1 + std::fabs(t1)) * std::pow(1 + std::fabs(t2), 6), std::fabs(t1));
  if (g.Ntau < 2) return c;
  c.per = (g.Ntau + kMaxCtas - 1) / kMaxCtas;
  c.ctas = (g.Ntau + c.per - 1) / c.per;
  c.threads = (c.per * (g.V / 2) + 31) / 32 * 32;
  if (c.threads > kMaxThreads) c.ctas = 0;
  return c;
}

static cudaLaunchConfig_t cluster_config(const Geo& g, const ClusterCg& c, cudaLaunchAttribute* attr, cudaStream_t s) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(c.ctas);
  cfg.blockDim = dim3(c.threads);
  cfg.dynamicSmemBytes = cluster_smem(g, c.per);
  cfg.stream = s;
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = c.ctas;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cfg;
}

// Whether the device can hold the cluster (c.ctas = 0 otherwise).
cudaError_t prepare_cg_cluster(const Geo& g, ClusterCg* c) {
  if (!c->ctas) return cudaSuccess;
  cudaError_t e = raise_smem_limit(c->fx ? cg_cluster_kernel<true> : cg_cluster_kernel<false>, cluster_smem(g, c->per));
  if (e == cudaSuccess && c->ctas > 8)
    e = cudaFuncSetAttribute(c->fx ? cg_cluster_kernel<true> : cg_cluster_kernel<false>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  if (e != cudaSuccess) return e;
  cudaLaunchAttribute attr[1];
  const cudaLaunchConfig_t cfg = cluster_config(g, *c, attr, 0);
  int n = 0;
  if (cudaOccupancyMaxActiveClusters(&n, c->fx ? cg_cluster_kernel<true> : cg_cluster_kernel<false>, &cfg) != cudaSuccess || n < 1) {
    cudaGetLastError();
    c->ctas = 0;
  }
  return cudaSuccess;
}

cudaError_t launch_cg_cluster(const MdagmArgs<double>& a, const ClusterCg& c, double2* x, double2* r, int max_its,
                              cudaStream_t s) {
  cudaLaunchAttribute attr[2];
  cudaLaunchConfig_t cfg = cluster_config(a.g, c, attr, s);
  attr[1] = pdl_attribute();
  cfg.numAttrs = 2;
  return cudaLaunchKernelEx(&cfg, c.fx ? cg_cluster_kernel<true> : cg_cluster_kernel<false>, a, x, r, c.per, max_its, c.F);
}

}  // namespace hqmc
