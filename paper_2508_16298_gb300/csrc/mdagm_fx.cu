// FP64 M^dagger M and M in fixed point (Methods, "Matrix-free representation of
// M^dagger M v"; checkerboard of Eq. (eq24)); the arithmetic is that of fx.cuh.
//
// With B_tau = cB P_tau and z_tau = P_tau x_tau, row tau of M^dagger M is
//   y_tau = t_tau + cB P_tau w_tau,
//   t_tau = x_tau - s_tau cB z_{tau-1},   w_tau = cB z_tau - s'_tau x_{tau+1}.
// As the FP32 kernel of mdagm_walk.cu, each CTA walks a contiguous range of slices
// with the slice in register strips (strip.cuh), so a range of n slices costs 2 n + 1
// sweeps.
//
// The FP64 kernels of mdagm.cu and mdagm_block.cu are bound by the FP64 rate.  Here the
// integer multiply-adds (12 per site and factor) would take 16,000 clocks per sweep of
// an L = 66 slice; measured are 26,000 to 36,000 (35% issue: link reads from L2 and
// dependent chains on 18 warps), and a third of the time goes to the conversions at
// the rows' ends.  One apply, L2 not flushed, against the FP64 kernels: L = 24, Ntau =
// 240: 24.6 us (36.9), L = 34, 333: 47 us (94), L = 48, 480: 86 us (225), L = 66, 660:
// 230 us (538).  Relative error (2-norm) against 64-bit plain torch at every L tested:
// 2.2e-16 (2.7e-16).
//
// Scales.  z_tau is computed at the scale of slice tau's own largest component, row
// tau's second sweep at that of the largest of slices tau - 1, tau, tau + 1; t_{tau+1}
// is held at that of tau and tau + 1.  All are functions of the slices alone, so a row
// is the same bit for bit however the slices are split into ranges, and a slice's
// partial sums (one slot per slice) too.
//
// A row that an infinity, a NaN or a non-finite angle reaches is computed in FP64
// instead (slow_row), with the outcome FP64 arithmetic gives it.  So is a row of an apply
// that a slice of very uneven size enters (fx_uneven in fx.cuh): its small elements would
// have fewer bits than a double.  A solve, which is judged by the norm of its residual,
// has no such rows.
#include "fx_strip.cuh"

namespace hqmc {

// t_tau waits for the row's second sweep in registers for NBY = 1 (t_{tau+1} is then the
// only one in shared memory), else both wait in the CTA's part of the scratch (written
// and read back by the same thread, two slices, L2-resident).
bool fx_tmem(int L) { return fx_nby(L) == 1; }
size_t fx_scratch(int L) { return fx_tmem(L) ? 0 : (size_t)2 * 4 * fx_nby(L) * fx_threads(L); }

// Shared memory: family-1 exchange and x_{tau+1} (one slice each), two row exchanges
// (2 entries a thread each), and t_{tau+1} where t_tau is in registers.
size_t fx_smem_bytes(const Geo& g) {
  const size_t slot = (size_t)fx_threads(g.L) * 4 * fx_nby(g.L);  // entries of one value per strip site
  return (g.V + (fx_tmem(g.L) ? 2 : 1) * slot + 4 * fx_threads(g.L)) * sizeof(longlong2);
}

// ---- FP64 row for non-finite and uneven data ------------------------------------------------

template <int MODE>
__device__ __forceinline__ double2 fx_load(const MdagmArgs<double>& a, const double2* p_old, double beta, bool first,
                                           size_t i) {
  // past L1, which is left to the links
  if (MODE == MODE_CGDIR) {
    const double2 r = __ldcg(a.r + i);
    return first ? r : caxpy(r, beta, __ldcg(p_old + i));
  }
  return __ldcg(a.x + i);
}

// Writes one component of a result row and adds its terms to the partial sums.
template <int MODE>
__device__ __forceinline__ void fx_emit(const MdagmArgs<double>& a, const double2* p_new, size_t i, double2 q,
                                        double& acc0, double& acc1) {
  if (MODE == MODE_RESID) {  // r = b - O x
    const double2 b = a.b[i];
    const double2 r = make_double2(b.x - q.x, b.y - q.y);
    if (a.r_out_fp32) reinterpret_cast<float2*>(a.r_out)[i] = make_float2((float)r.x, (float)r.y);
    else reinterpret_cast<double2*>(a.r_out)[i] = r;
    acc0 += r.x * r.x + r.y * r.y;
    acc1 += b.x * b.x + b.y * b.y;
  } else {
    a.y[i] = q;
    if (MODE == MODE_CGDIR) acc0 += cdot_re(p_new[i], q);
  }
}

// Row j in FP64 from its three slices; W: one slice of shared memory.  The terms that
// wait for the second sweep are parked in the output array; a float residual has no
// room for them, and its row becomes NaN (its sum, which ends the solve, is NaN either way).
// Returns this thread's terms of the row's sums.
template <int MODE>
__device__ __noinline__ double2 slow_row(const MdagmArgs<double>& a, const double2* p_old, double2* p_new, double beta,
                                         bool first, int j, double2* W, int nt) {
  double acc0 = 0.0, acc1 = 0.0;
  const Geo g = a.g;
  const int V = g.V, N = g.Ntau, jm = j == 0 ? N - 1 : j - 1, jp = j == N - 1 ? 0 : j + 1;
  const double s = j == 0 ? -1.0 : 1.0, sp = j == N - 1 ? -1.0 : 1.0;
  const size_t bj = (size_t)j * V;
  const bool fp32 = MODE == MODE_RESID && a.r_out_fp32;
  double2* park = MODE == MODE_RESID ? reinterpret_cast<double2*>(a.r_out) : a.y;
  __syncthreads();
  for (int i = threadIdx.x; i < V; i += nt) W[i] = fx_load<MODE>(a, p_old, beta, first, (size_t)jm * V + i);
  __syncthreads();
  slow_sweep(g, W, a.UF + (size_t)jm * V * 2, nt);
  for (int i = threadIdx.x; i < V; i += nt) {
    const double2 x = fx_load<MODE>(a, p_old, beta, first, bj + i);
    if (!fp32) park[bj + i] = caxpy(x, -s * a.cB, W[i]);
    W[i] = x;
  }
  __syncthreads();
  slow_sweep(g, W, a.UF + bj * 2, nt);
  for (int i = threadIdx.x; i < V; i += nt)
    W[i] = caxpy(cscale(a.cB, W[i]), -sp, fx_load<MODE>(a, p_old, beta, first, (size_t)jp * V + i));
  __syncthreads();
  slow_sweep(g, W, a.UF + bj * 2, nt);
  const double nan = __longlong_as_double(0x7ff8000000000000ll);
  for (int i = threadIdx.x; i < V; i += nt) {
    double2 q = fp32 ? make_double2(nan, nan) : caxpy(park[bj + i], a.cB, W[i]);
    if (MODE == MODE_CGDIR) {  // the row's p in this thread's order of sites
      a.y[bj + i] = q;
      acc0 += cdot_re(fx_load<MODE>(a, p_old, beta, first, bj + i), q);
    } else {
      fx_emit<MODE>(a, p_new, bj + i, q, acc0, acc1);
    }
  }
  __syncthreads();
  return make_double2(acc0, acc1);
}

// ---- M^dagger M over the slices [tb, te) of one chain -------------------------------
template <int MODE, int NBY, bool AHEAD>
__device__ __forceinline__ void fx_range(const MdagmArgs<double>& a, const int tb, const int te, const bool writer,
                                         const int nt, const int cta) {
  constexpr int H = 2 * NBY;
  constexpr bool TREG = NBY == 1;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ int s_flags;
  __shared__ double s_beta;
  __shared__ int s_k;
  __shared__ uint32_t s_key[3];
  // APPLY: of slice j in place j mod 8; set after its fetch, read after the second sweeps of the
  // rows that use it, cleared four fetches ahead (a fetch's barrier lies between any two of these)
  __shared__ int s_uneven[8];
  __shared__ double s_red[2][2][32];
  const int V = a.g.V, N = a.g.Ntau, L = a.g.L;
  longlong2* const E = reinterpret_cast<longlong2*>(smem_raw);
  longlong2* const X1 = E + V;
  const int nslot = 2 * H * nt;  // entries of one value per strip site (the idle rows of a cut strip included)
  longlong2* const R0 = X1 + nslot;
  longlong2* const R1 = R0 + 2 * nt;
  longlong2* const T = TREG ? R1 + 2 * nt : a.tscr + (size_t)cta * 2 * nslot;
  auto park = [&](longlong2* p, longlong2 x) {
    if (TREG) *p = x;
    else __stcg(p, x);
  };
  auto unpark = [&](const longlong2* p) -> longlong2 { return TREG ? *p : __ldcg(p); };

  if (MODE == MODE_CGDIR) {
    cgdir_head<double>(a, writer, s_flags, s_beta, s_k);
    if (s_flags & 1) return;  // uniform over the chain's CTAs
  }
  if (MODE == MODE_RESID && a.gate != GATE_ALWAYS) {
    if (threadIdx.x == 0) s_flags = gate_open(a.gate, *(volatile int*)&a.st->done) ? 0 : 1;
    __syncthreads();
    if (s_flags & 1) return;
  }
  const bool first = MODE == MODE_CGDIR && (s_flags & 2);
  const double beta = MODE == MODE_CGDIR ? s_beta : 0.0;
  const double2* p_old = nullptr;
  double2* p_new = nullptr;
  if (MODE == MODE_CGDIR) {
    p_old = (s_k & 1) ? a.pbuf[1] : a.pbuf[0];
    p_new = (s_k & 1) ? a.pbuf[0] : a.pbuf[1];
  }
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = (nt + 31) >> 5;
  const unsigned wmask = nt - 32 * warp >= 32 ? 0xffffffffu : (1u << (nt - 32 * warp)) - 1u;
  const FxStrip sg = fx_strip<NBY>(L, tid);
  const bool full = NBY == 1 || sg.nr == H;
  const int F = a.F;
  auto wrap = [N](int j) { return j < 0 ? j + N : (j >= N ? j - N : j); };

  // Brings slice ju (mod N) into this thread's slots of X1 as doubles, writes p_new for
  // an own slice, and returns the slice's exponent (one barrier).
  auto fetch = [&](int ju, bool own, int slot) -> int {
    const size_t base = (size_t)wrap(ju) * V;
    uint32_t key = 0;
#pragma unroll
    for (int r = 0; r < H; ++r) {
      if (r >= 2 && !full) break;
      const int y = fx_drow(sg, r) * L;
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        const size_t i = base + y + (c ? sg.x1 : sg.x0);
        const double2 x = fx_load<MODE>(a, p_old, beta, first, i);
        if (MODE == MODE_CGDIR && own) p_new[i] = x;
        X1[(2 * r + c) * nt + tid] = make_longlong2(__double_as_longlong(x.x), __double_as_longlong(x.y));
        key = max(key, max(fx_key(x.x), fx_key(x.y)));
      }
    }
    const uint32_t strip = key;
    key = __reduce_max_sync(wmask, key);
    if (lane == 0) atomicMax(&s_key[slot], key);
    if (tid == 0) {  // of the next call: last read before the previous barriers
      s_key[slot == 2 ? 0 : slot + 1] = 0;
      if (MODE == MODE_APPLY) s_uneven[(ju + 4) & 7] = 0;
    }
    __syncthreads();
    if (MODE == MODE_APPLY && fx_uneven(strip, s_key[slot])) s_uneven[ju & 7] = 1;
    return fx_exponent(s_key[slot]);
  };
  // This thread's slots of X1 from doubles to fixed point.
  auto convert = [&](int e) {
    const int s0 = fx_shift_base(e, F);
    const int n = full ? 2 * H : 4;
#pragma unroll 2
    for (int m = 0; m < n; ++m) {
      const longlong2 x = X1[m * nt + tid];
      X1[m * nt + tid] = make_longlong2(fx_from_double(__longlong_as_double(x.x), s0),
                                        fx_from_double(__longlong_as_double(x.y), s0));
    }
  };

  // Warp 0: row j's sums over the warps, in a fixed order.
  auto row_sums = [&](int j) {
    const int par = j & 1;
    const double s0 = lane_sum(lane < nw ? s_red[par][0][lane] : 0.0, min(nt, 32));
    if (lane == 0) a.part_out[wrap(j)] = s0;
    if (MODE == MODE_RESID) {
      const double s1 = lane_sum(lane < nw ? s_red[par][1][lane] : 0.0, min(nt, 32));
      if (lane == 0) a.part_out[a.nslots + wrap(j)] = s1;
    }
  };

  if (tid < 3) s_key[tid] = 0;
  if (MODE == MODE_APPLY && tid < 8) s_uneven[tid] = 0;
  __syncthreads();
  longlong2 v[H][2], t[TREG ? H : 1][2];
  int e_prev = kFxZero;                                  // exponent of slice j - 1
  int e_cur = fetch(tb - 1, false, 0);                   // of slice j
  int e_t = kFxZero, e_next = kFxZero, e_w = kFxZero;    // of t_j, slice j + 1, row j
  bool z_bad = true, zp_bad = true, slow = false;        // z_j, z_{j-1}, row j are not finite
  bool u_bad = links_bad(a, wrap(tb - 1));               // links of slice j
  if (e_cur < kFxBad) convert(e_cur);
#pragma unroll
  for (int r = 0; r < H; ++r)
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      v[r][c] = X1[(2 * r + c) * nt + tid];
      if (TREG) t[r][c] = make_longlong2(0, 0);
    }

  int slot = 1;
  // Two sweeps per slice (one for the halo slice tb - 1), in a loop so that the sweep's
  // code is there once: with two copies the kernel stalled on instruction fetch.
#pragma unroll 1
  for (int q = 2 * (tb - 1); q < 2 * te; q += q == 2 * (tb - 1) ? 2 : 1) {
    const int j = q >> 1, js = wrap(j);
    const bool second = q & 1, own = j >= tb;
    if (!second) {
      zp_bad = z_bad;
      z_bad = e_cur >= kFxBad || u_bad;
      if (MODE == MODE_APPLY && j > tb) z_bad |= s_uneven[j & 7] != 0;  // barriers of row j - 1 lie between
    }
    if (second ? !slow : !z_bad) fx_sweep<NBY, AHEAD>(v, a.UF + (size_t)js * V * 2, sg, E, R0, R1);  // z_j, or P_j w_j
    if (!second) {
      const int jn = wrap(j + 1);
      u_bad = links_bad(a, jn);
      e_next = fetch(j + 1, j + 1 < te, slot);
      slot = slot == 2 ? 0 : slot + 1;
      if (j > tb && warp == 0 && MODE != MODE_APPLY) row_sums(j - 1);  // written before the barriers above
      const bool x_bad = e_next >= kFxBad;
      slow = z_bad || zp_bad || x_bad;
      const int e_m = max(e_cur, e_next);
      e_w = max(e_prev, e_m);
      if (!x_bad) convert(e_next);
      if (!z_bad && !x_bad) {
        // t_{j+1} = x_{j+1} - s_{j+1} cB z_j and w_j = cB z_j - s'_j x_{j+1}
        auto combine = [&](auto plain) {
          const int n_zm = e_m - e_cur, n_xm = e_m - e_next, n_zw = e_w - e_cur, n_xw = e_w - e_next;
          const bool neg_t = jn == 0, neg_w = js == N - 1;  // s_{j+1} = -1, s'_j = -1
#pragma unroll
          for (int r = 0; r < H; ++r)
#pragma unroll
            for (int c = 0; c < 2; ++c) {
              const int k = (2 * r + c) * nt + tid;
              const longlong2 x = X1[k];
              const longlong2 z = make_longlong2(fx_fma(v[r][c].x, a.cm1h, a.cm1l, v[r][c].x),
                                                 fx_fma(v[r][c].y, a.cm1h, a.cm1l, v[r][c].y));  // cB z_j
              longlong2* const tk = T + (TREG ? k : k + ((j + 1) & 1) * nslot);
              if constexpr (decltype(plain)::value) {
                park(tk, make_longlong2(x.x - z.x, x.y - z.y));
                v[r][c] = make_longlong2(z.x - x.x, z.y - x.y);
              } else {
                const longlong2 zm = make_longlong2(fx_shr(z.x, n_zm), fx_shr(z.y, n_zm));
                const longlong2 xm = make_longlong2(fx_shr(x.x, n_xm), fx_shr(x.y, n_xm));
                park(tk, neg_t ? make_longlong2(xm.x + zm.x, xm.y + zm.y) : make_longlong2(xm.x - zm.x, xm.y - zm.y));
                const longlong2 zw = make_longlong2(fx_shr(z.x, n_zw), fx_shr(z.y, n_zw));
                const longlong2 xw = make_longlong2(fx_shr(x.x, n_xw), fx_shr(x.y, n_xw));
                v[r][c] = neg_w ? make_longlong2(zw.x + xw.x, zw.y + xw.y) : make_longlong2(zw.x - xw.x, zw.y - xw.y);
              }
            }
        };
        // most rows: one scale and no sign (the halo row's w is not used)
        if (e_cur == e_w && e_next == e_w && jn != 0) combine(FxTrue{});
        else combine(FxFalse{});
      }
      if (own) continue;
    } else {
      double acc0 = 0.0, acc1 = 0.0;
      if (MODE == MODE_APPLY && (s_uneven[(j - 1) & 7] | s_uneven[j & 7] | s_uneven[(j + 1) & 7])) slow = true;
      if (!slow) {
        const int n_t = e_w - e_t;
        // the row in fixed point to this thread's slots of X1's neighbour E (free since the
        // sweep's last barrier), then out in a loop; an all-zero row gives zeros
#pragma unroll
        for (int r = 0; r < H; ++r) {
          if (r >= 2 && !full) break;
#pragma unroll
          for (int c = 0; c < 2; ++c) {
            const int k = (2 * r + c) * nt + tid;
            const longlong2 tv = TREG ? t[r][c] : unpark(T + k + (j & 1) * nslot);
            E[fx_slot(sg, r, c)] = make_longlong2(fx_shr(tv.x, n_t) + fx_fma(v[r][c].x, a.cm1h, a.cm1l, v[r][c].x),
                                                  fx_shr(tv.y, n_t) + fx_fma(v[r][c].y, a.cm1h, a.cm1l, v[r][c].y));
          }
        }
        const size_t bj = (size_t)js * V;
        const int n = full ? 2 * H : 4;
#pragma unroll 2
        for (int m = 0; m < n; ++m) {
          const longlong2 f = E[fx_slot(sg, m >> 1, m & 1)];
          fx_emit<MODE>(a, p_new, bj + fx_drow(sg, m >> 1) * L + (m & 1 ? sg.x1 : sg.x0),
                        make_double2(fx_to_double(f.x, e_w - F), fx_to_double(f.y, e_w - F)), acc0, acc1);
        }
      } else {
        const double2 acc = slow_row<MODE>(a, p_old, p_new, beta, first, js, reinterpret_cast<double2*>(E), nt);
        acc0 = acc.x;
        acc1 = acc.y;
      }
      if (MODE != MODE_APPLY) {
        acc0 = lane_sum(acc0, nt - 32 * warp);
        if (lane == 0) s_red[j & 1][0][warp] = acc0;
        if (MODE == MODE_RESID) {
          acc1 = lane_sum(acc1, nt - 32 * warp);
          if (lane == 0) s_red[j & 1][1][warp] = acc1;
        }
      }
    }
    // on to slice j + 1
    e_t = max(e_cur, e_next);
    e_prev = e_cur;
    e_cur = e_next;
#pragma unroll
    for (int r = 0; r < H; ++r)
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        const int k = (2 * r + c) * nt + tid;
        v[r][c] = X1[k];
        if (TREG) t[r][c] = T[k];
      }
  }
  if (MODE != MODE_APPLY) {
    __syncthreads();
    if (warp == 0) row_sums(te - 1);
  }
}

template <int MODE, int NBY, int CAP>
__global__ void __launch_bounds__(CAP, 1) mdagm_fx_kernel(const __grid_constant__ MdagmArgs<double> a) {
  pdl_begin();
  const int N = a.g.Ntau;
  const int tb = (int)((long long)blockIdx.x * N / gridDim.x), te = (int)((long long)(blockIdx.x + 1) * N / gridDim.x);
  fx_range<MODE, NBY, NBY == 1>(a, tb, te, blockIdx.x == 0, (int)blockDim.x, (int)blockIdx.x);
}

// Many lattices (the chains of a batch, the systems of an estimate) in one launch: block b
// serves the slices [tile.y, tile.z) of lattice tile.x as its range tile.w.  The block has
// the threads of the largest; the others' surplus threads leave at once.
template <int MODE, int NBY, int CAP>
__global__ void __launch_bounds__(CAP, 1) mdagm_fx_batch_kernel(const MdagmArgs<double>* __restrict__ descs,
                                                                const int4* __restrict__ tiles) {
  pdl_begin();
  __shared__ MdagmArgs<double> a;
  const int4 t = tiles[blockIdx.x];
  if (threadIdx.x == 0) a = descs[t.x];
  __syncthreads();
  const int H = 2 * NBY, nt = (a.g.L >> 1) * ((a.g.L + H - 1) / H);
  if ((int)threadIdx.x >= nt) return;
  fx_range<MODE, NBY, NBY == 1>(a, t.y, t.z, t.y == 0, nt, t.w);
}

template <int MODE>
cudaError_t launch_mdagm_fx(const SliceLaunch& sl, const MdagmArgs<double>& a, cudaStream_t s) {
  if (sl.grid < 1 || sl.grid > sl.g.Ntau) return cudaErrorInvalidValue;
  return fx_pick(sl.g.L, [&](auto nby, auto cap) {
    return launch_after(mdagm_fx_kernel<MODE, nby.v, cap.v>, sl.grid, fx_threads(sl.g.L), fx_smem_bytes(sl.g), s, a);
  });
}

template <int MODE>
cudaError_t prepare_mdagm_fx(const SliceLaunch& sl) {
  return fx_pick(sl.g.L, [&](auto nby, auto cap) {
    return raise_smem_limit(mdagm_fx_kernel<MODE, nby.v, cap.v>, fx_smem_bytes(sl.g));
  });
}
template cudaError_t launch_mdagm_fx<MODE_APPLY>(const SliceLaunch&, const MdagmArgs<double>&, cudaStream_t);
template cudaError_t launch_mdagm_fx<MODE_RESID>(const SliceLaunch&, const MdagmArgs<double>&, cudaStream_t);
template cudaError_t launch_mdagm_fx<MODE_CGDIR>(const SliceLaunch&, const MdagmArgs<double>&, cudaStream_t);
template cudaError_t prepare_mdagm_fx<MODE_APPLY>(const SliceLaunch&);
template cudaError_t prepare_mdagm_fx<MODE_RESID>(const SliceLaunch&);
template cudaError_t prepare_mdagm_fx<MODE_CGDIR>(const SliceLaunch&);

// Instantiation class of a lattice in a batched launch (lattices of one class share it).
int fx_class(int L) { return fx_nby(L) == 1 ? 0 : fx_threads(L) <= 512 ? 1 : 2; }

// Lmax: the largest lattice among the tiles, all of one class.
template <int MODE>
cudaError_t launch_mdagm_fx_batch(const MdagmArgs<double>* descs, const int4* tiles, int ntiles, int Lmax,
                                  cudaStream_t s) {
  const Geo g{Lmax, Lmax * Lmax, Lmax / 2, 1};
  return fx_pick(Lmax, [&](auto nby, auto cap) {
    const cudaError_t e = raise_smem_limit(mdagm_fx_batch_kernel<MODE, nby.v, cap.v>, fx_smem_bytes(g));
    if (e != cudaSuccess) return e;
    return launch_after(mdagm_fx_batch_kernel<MODE, nby.v, cap.v>, ntiles, fx_threads(Lmax), fx_smem_bytes(g), s, descs, tiles);
  });
}
template cudaError_t launch_mdagm_fx_batch<MODE_RESID>(const MdagmArgs<double>*, const int4*, int, int, cudaStream_t);
template cudaError_t launch_mdagm_fx_batch<MODE_CGDIR>(const MdagmArgs<double>*, const int4*, int, int, cudaStream_t);

// CTAs of this shape the device keeps resident per SM (0: none fit).
int mdagm_fx_blocks_per_sm(const SliceLaunch& sl) {
  int n = 0;
  const cudaError_t e = fx_pick(sl.g.L, [&](auto nby, auto cap) {
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, mdagm_fx_kernel<MODE_CGDIR, nby.v, cap.v>,
                                                         fx_threads(sl.g.L), fx_smem_bytes(sl.g));
  });
  if (e != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return n;
}

// ---------------------------------------------------------------------------
// y = M x:        y_tau = x_tau - s_tau  cB P_{tau-1} x_{tau-1}
// y = M^dagger x: y_tau = x_tau - s'_tau cB P_tau x_{tau+1}   (B Hermitian)
// One CTA per slice; the sweep at the scale of the slice it acts on.
template <int NBY>
__device__ __forceinline__ void fx_apply_M_slice(const MdagmArgs<double>& a, int dagger, int tau, int nt) {
  constexpr int H = 2 * NBY;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ uint32_t s_key;
  __shared__ int s_uneven;
  const int V = a.g.V, N = a.g.Ntau, L = a.g.L;
  longlong2* const E = reinterpret_cast<longlong2*>(smem_raw);
  longlong2* const R0 = E + V;
  longlong2* const R1 = R0 + 2 * nt;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const unsigned wmask = nt - 32 * warp >= 32 ? 0xffffffffu : (1u << (nt - 32 * warp)) - 1u;
  const int src = dagger ? (tau == N - 1 ? 0 : tau + 1) : (tau == 0 ? N - 1 : tau - 1);
  const int us = dagger ? tau : src;  // links of slice us
  const double f = ((dagger ? tau == N - 1 : tau == 0) ? 1.0 : -1.0) * a.cB;
  const size_t bs = (size_t)src * V, bt = (size_t)tau * V;
  const int4* const U = a.UF + (size_t)us * V * 2;
  const FxStrip sg = fx_strip<NBY>(L, tid);
  const bool full = NBY == 1 || sg.nr == H;
  if (tid == 0) {
    s_key = 0;
    s_uneven = 0;
  }
  __syncthreads();
  longlong2 v[H][2];
  uint32_t key = 0;
#pragma unroll
  for (int r = 0; r < H; ++r)
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      if (r >= 2 && !full) break;
      const double2 x = a.x[bs + fx_drow(sg, r) * L + (c ? sg.x1 : sg.x0)];
      v[r][c] = make_longlong2(__double_as_longlong(x.x), __double_as_longlong(x.y));
      key = max(key, max(fx_key(x.x), fx_key(x.y)));
    }
  const uint32_t strip = key;
  key = __reduce_max_sync(wmask, key);
  if (lane == 0) atomicMax(&s_key, key);
  __syncthreads();
  const int e = fx_exponent(s_key);
  bool fp64 = e >= kFxBad || links_bad(a, us);
  if (!fp64) {
    if (fx_uneven(strip, s_key)) s_uneven = 1;
    const int s0 = fx_shift_base(e, a.F);
#pragma unroll
    for (int r = 0; r < H; ++r)
#pragma unroll
      for (int c = 0; c < 2; ++c)
        v[r][c] = make_longlong2(fx_from_double(__longlong_as_double(v[r][c].x), s0),
                                 fx_from_double(__longlong_as_double(v[r][c].y), s0));
    fx_sweep<NBY, NBY == 1>(v, U, sg, E, R0, R1);
    fp64 = s_uneven != 0;  // set before the sweep's barriers
  }
  if (fp64) {
    double2* const W = reinterpret_cast<double2*>(E);
    for (int i = tid; i < V; i += nt) W[i] = a.x[bs + i];
    __syncthreads();
    slow_sweep(a.g, W, U, nt);
    for (int i = tid; i < V; i += nt) a.y[bt + i] = caxpy(a.x[bt + i], f, W[i]);
    return;
  }
#pragma unroll
  for (int r = 0; r < H; ++r)
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      if (r >= 2 && !full) break;
      const size_t i = bt + fx_drow(sg, r) * L + (c ? sg.x1 : sg.x0);
      a.y[i] = caxpy(a.x[i], f, make_double2(fx_to_double(v[r][c].x, e - a.F), fx_to_double(v[r][c].y, e - a.F)));
    }
}

template <int NBY, int CAP>
__global__ void __launch_bounds__(CAP, 1) apply_M_fx_kernel(const __grid_constant__ MdagmArgs<double> a, const int dagger) {
  pdl_begin();
  fx_apply_M_slice<NBY>(a, dagger, blockIdx.x, (int)blockDim.x);
}

static size_t fx_apply_smem_bytes(const Geo& g) { return (size_t)(g.V + 4 * fx_threads(g.L)) * sizeof(longlong2); }

cudaError_t launch_apply_M_fx(const SliceLaunch& sl, const MdagmArgs<double>& a, int dagger, cudaStream_t s) {
  return fx_pick(sl.g.L, [&](auto nby, auto cap) {
    return launch_after(apply_M_fx_kernel<nby.v, cap.v>, sl.g.Ntau, fx_threads(sl.g.L), fx_apply_smem_bytes(sl.g), s, a, dagger);
  });
}

// y = M^dagger x of many lattices: block b serves slice tile.y of lattice tile.x.
template <int NBY, int CAP>
__global__ void __launch_bounds__(CAP, 1) apply_Mdag_fx_batch_kernel(const MdagmArgs<double>* __restrict__ descs,
                                                                     const int4* __restrict__ tiles) {
  pdl_begin();
  __shared__ MdagmArgs<double> a;
  const int4 t = tiles[blockIdx.x];
  if (threadIdx.x == 0) a = descs[t.x];
  __syncthreads();
  const int H = 2 * NBY, nt = (a.g.L >> 1) * ((a.g.L + H - 1) / H);
  if ((int)threadIdx.x >= nt) return;
  fx_apply_M_slice<NBY>(a, 1, t.y, nt);
}

cudaError_t launch_apply_Mdag_fx_batch(const MdagmArgs<double>* descs, const int4* tiles, int ntiles, int Lmax,
                                       cudaStream_t s) {
  const Geo g{Lmax, Lmax * Lmax, Lmax / 2, 1};
  return fx_pick(Lmax, [&](auto nby, auto cap) {
    const cudaError_t e = raise_smem_limit(apply_Mdag_fx_batch_kernel<nby.v, cap.v>, fx_apply_smem_bytes(g));
    if (e != cudaSuccess) return e;
    return launch_after(apply_Mdag_fx_batch_kernel<nby.v, cap.v>, ntiles, fx_threads(Lmax), fx_apply_smem_bytes(g), s, descs, tiles);
  });
}

cudaError_t prepare_apply_M_fx(const SliceLaunch& sl) {
  return fx_pick(sl.g.L, [&](auto nby, auto cap) {
    return raise_smem_limit(apply_M_fx_kernel<nby.v, cap.v>, fx_apply_smem_bytes(sl.g));
  });
}

}  // namespace hqmc
