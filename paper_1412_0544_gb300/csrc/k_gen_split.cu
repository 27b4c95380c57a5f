// k_gen_split.cu -- the generic scheme (any explicit tableau of up to 7 stages, coupling range 1
// or 2) for FP64 in the split form of rk4_split.cuh: K1 = f(y) in FP64, the later slopes' negated
// differences n_m = K1 - k_m in float pairs,
//   d_j = c_j K1 - sum_m a_jm n_m      (u_j = y + dt d_j, c_j the row sum; Eq. (4))
//   y <- y + dt (B K1 - sum_m b_m n_m)  (B the sum of the weights; Eq. (5)),
// for whatever tableau the kernel is given at run time.
//
// What bounds it: Dormand-Prince 5 with second neighbours issued 123 DFMA per site-step, now 16
// (10 for the first slope, 6 for the update) beside some 1100 FP32 operations: FMA pipe 47 %,
// FP64 pipe 35 % busy, 16 warps per SM (128 registers), the rest latency.  Every thread holds two
// sites (one packed pair) whatever the tiling's sites per thread, so a tile of W sites runs on
// W / 2 threads; the differences lie in thread-private shared-memory records, which both frees
// their registers (five stages of three pairs, 60 registers) and lets the stage loops run over any
// tableau's nonzero entries without a kernel per tableau.  Measured at N = 2^20, us per step, best
// tiling: Dormand-Prince 5 + second neighbours 245 -> 78, RK4 + second neighbours 128 -> 54 (run-time
// tableaux 345 -> 78).  With the state and the first slope in registers too (164, one block of 256
// threads per SM) it took 89.
//
// Error against long double, in units of the FP64 form's: 1.00 from 10 .. 20 steps on, 1.05 after
// one Dormand-Prince step from a random state (z alone 1.15; its differences carry dt |x - c|, and
// pairs of their own roundings), 1.01 for RK4 with second neighbours.  The tails are normalised
// (pair_norm) where the rows multiply them by up to 11; without, 1.12.  The weights' sum is carried
// to a float beyond FP64: its own rounding, times dt K1 every step, was a drift of 1.2.
#include <algorithm>

#include "rk4_generic.cuh"

namespace rk4d {

constexpr int kGenSplitThreads = 512;

// 8-byte words of a thread's record: the pairs of up to s - 1 differences and, when parked (blocks
// of up to 256 threads), the state and the first slope in FP64; odd (see split_record_words).
__host__ __device__ constexpr int gen_record_words(int s, int D, bool park) {
  return ((s - 1 + (park ? 2 : 0)) * D * 2) | 1;
}

// A tile outside the split's range in the FP64 form (two sites per thread, run-time tableau).
template <int MODEL, int RANGE>
__device__ __noinline__ void gen_wide_tile(const BlockedJob &job, ChainDesc ch, int64_t t0, int H, Coef<double> cf,
                                           double kappa2, const Tableau<double> &tb, unsigned char *smem) {
  constexpr int D = Dim<MODEL>::D, V = 2;
  const int W = blockDim.x * V;
  double *edge = reinterpret_cast<double *>(smem);
  double *tl = edge + gen_edge_values(V);
  tile_load<double, D, false>(tl, static_cast<const double *>(job.in), ch.off, ch.n, ch.bc, t0, W, job.total, job.hdr);
  tile_load_wait();
  __syncthreads();
  double y[V][D], cmp[V][D];
  const int base = threadIdx.x * V;
  uint32_t ghost = 0;
#pragma unroll
  for (int v = 0; v < V; ++v) {
    const int64_t g = t0 + base + v;
    if (ch.bc == FIXED && (g < 0 || g >= ch.n)) ghost |= 1u << v;
#pragma unroll
    for (int d = 0; d < D; ++d) {
      y[v][d] = tl[(base + v) * D + d];
      cmp[v][d] = 0.0;
    }
  }
  gen_tile_advance<double, MODEL, V, RANGE, false, true, 0>(y, cmp, ghost, job.K, cf, kappa2, tb, edge);
  const int64_t g0 = t0 + H, rem = ch.n - g0;
  const int cnt = (int)(rem < job.G ? rem : job.G);
  bool bad = false;
#pragma unroll
  for (int v = 0; v < V; ++v)
#pragma unroll
    for (int d = 0; d < D; ++d) {
      tl[(base + v) * D + d] = y[v][d];
      bad |= base + v >= H && base + v < H + cnt && nonfinite(y[v][d]);
    }
  report_nonfinite(job.hdr, __syncthreads_or(bad));
  if (cnt > 0) tile_store<double, D>(static_cast<double *>(job.out), tl, ch.off, H, g0, cnt, job.total, W, job.hdr);
}

// K steps on the thread's two sites.  ex: two parities of 16 bytes per thread, a thread's two
// coupling coordinates (FP64, or their increments as a packed pair), read by its neighbours.
template <int MODEL, int RANGE, bool MASK, bool PARK>
__device__ __forceinline__ void gen_split_advance(double (&y)[2][Dim<MODEL>::D], uint32_t ghost, int K,
                                                  const Coef<double> &cf, double kappa2, const SplitCoef &sc,
                                                  const SplitTableau &tb, ulonglong2 *ex, f32x2 *rec) {
  constexpr int D = Dim<MODEL>::D;
  using T = f32x2;
  const int tid = threadIdx.x, bd = blockDim.x;
  const int lt = tid > 0 ? tid - 1 : tid, rt = tid < bd - 1 ? tid + 1 : tid;
  const StageCoef<T> c = stage_coef<T>(sc);
  double *py = reinterpret_cast<double *>(rec + (tb.s - 1) * D * 2), *pk = py + 2 * D;
  if constexpr (PARK) {
#pragma unroll
    for (int i = 0; i < 2 * D; ++i) py[i] = y[i / D][i % D];
  }
  int parity = 0;
  auto exchange = [&](ulonglong2 mine, ulonglong2 &l, ulonglong2 &r) {
    ulonglong2 *e = ex + parity * bd;
    parity ^= 1;
    e[tid] = mine;
    neighbour_warp_sync();
    l = e[lt];
    r = e[rt];
  };
#pragma unroll 1
  for (int s = 0; s < K; ++s) {
    double k1d[2][D];
    FPair<T> k1[D];
    SplitBase<T> base = {};
    {
      if constexpr (PARK) {
#pragma unroll
        for (int i = 0; i < 2 * D; ++i) y[i / D][i % D] = py[i];
      }
      double x[2];
#pragma unroll
      for (int v = 0; v < 2; ++v) x[v] = (MASK && ((ghost >> v) & 1u)) ? 0.0 : y[v][0];
      ulonglong2 l, r;
      exchange(make_ulonglong2(__double_as_longlong(x[0]), __double_as_longlong(x[1])), l, r);
      const double l2 = __longlong_as_double(l.x), l1 = __longlong_as_double(l.y);
      const double r1 = __longlong_as_double(r.x), r2 = __longlong_as_double(r.y);
      slope_gen<double, MODEL, RANGE>(y[0], l1, x[1], l2, r1, cf, kappa2, k1d[0]);
      slope_gen<double, MODEL, RANGE>(y[1], x[0], r1, l1, r2, cf, kappa2, k1d[1]);
#pragma unroll
      for (int i = 0; i < D; ++i) k1[i] = Lanes<T>::split(&k1d[0][i], D);
      if constexpr (MODEL == ROESSLER) {
        base.z = Lanes<T>::split(&y[0][2], D);
        base.t = x_minus_c<T>(Lanes<T>::split(&y[0][0], D), {vset<T>(sc.ch), vset<T>(sc.cl)});
      }
      if constexpr (PARK) {
#pragma unroll
        for (int i = 0; i < 2 * D; ++i) pk[i] = k1d[i / D][i % D];
      }
    }
#pragma unroll 1
    for (int j = 1; j < tb.s; ++j) {
      if (!((tb.need >> j) & 1u)) continue;
      FPair<T> d[D], n[D];
      {
        const FPair<T> cj = {vset<T>(tb.ch[j]), vset<T>(tb.cl[j])};
        const T nc = vset<T>(-tb.ch[j]);
#pragma unroll
        for (int i = 0; i < D; ++i) d[i] = pair_mul(cj, nc, k1[i]);
      }
#pragma unroll 2
      for (int q0 = 0; q0 < tb.na[j]; ++q0) {
        const int m = tb.ma[j][q0];
        const FPair<T> a = {vset<T>(tb.ah[j][m]), vset<T>(tb.al[j][m])};
        const T na = vset<T>(-tb.ah[j][m]);
        const f32x2 *q = rec + (m - 1) * D * 2;
#pragma unroll
        for (int i = 0; i < D; ++i) d[i] = pair_fnma<T>(a, na, {q[2 * i], q[2 * i + 1]}, d[i]);
      }
#pragma unroll
      for (int i = 0; i < D; ++i) d[i] = pair_norm(d[i]);
      FPair<T> X = d[0];
      if constexpr (MASK) {
        const bool g0 = ghost & 1u, g1 = ghost & 2u;
        X.h = pack2(g0 ? 0.f : lane0(X.h), g1 ? 0.f : lane1(X.h));
        X.l = pack2(g0 ? 0.f : lane0(X.l), g1 ? 0.f : lane1(X.l));
      }
      ulonglong2 l, r;
      exchange(make_ulonglong2(X.h, X.l), l, r);
      const FPair<T> xl = {pack2(lane1(l.x), lane0(X.h)), pack2(lane1(l.y), lane0(X.l))};
      const FPair<T> xr = {pack2(lane1(X.h), lane0(r.x)), pack2(lane1(X.l), lane0(r.y))};
      // second neighbours: the left thread's two sites, the right thread's two sites
      split_stage<MODEL, T, RANGE, true>(d, xl, xr, base, c, n, {l.x, l.y}, {r.x, r.y});
      f32x2 *o = rec + (j - 1) * D * 2;
#pragma unroll
      for (int i = 0; i < D; ++i) {
        n[i] = pair_norm(n[i]);
        o[2 * i] = n[i].h;
        o[2 * i + 1] = n[i].l;
      }
    }
    FPair<T> N[D];
#pragma unroll
    for (int i = 0; i < D; ++i) N[i] = {0ull, vmul(vset<T>(-tb.Bl), k1[i].h)};
#pragma unroll 2
    for (int q0 = 0; q0 < tb.nb; ++q0) {
      const int m = tb.mb[q0];
      const FPair<T> b = {vset<T>(tb.bh[m]), vset<T>(tb.bl[m])};
      const T nb = vset<T>(-tb.bh[m]);
      const f32x2 *q = rec + (m - 1) * D * 2;
#pragma unroll
      for (int i = 0; i < D; ++i) N[i] = pair_fma<T>(b, nb, {q[2 * i], q[2 * i + 1]}, N[i]);
    }
#pragma unroll
    for (int i = 0; i < D; ++i) {
      double nd[2];
      join(N[i], nd, 1);
      if constexpr (PARK) {
        py[i] = fma(sc.w, fma(tb.B, pk[i], -nd[0]), py[i]);
        py[D + i] = fma(sc.w, fma(tb.B, pk[D + i], -nd[1]), py[D + i]);
      } else {
        y[0][i] = fma(sc.w, fma(tb.B, k1d[0][i], -nd[0]), y[0][i]);
        y[1][i] = fma(sc.w, fma(tb.B, k1d[1][i], -nd[1]), y[1][i]);
      }
    }
  }
  if constexpr (PARK) {
#pragma unroll
    for (int i = 0; i < 2 * D; ++i) y[i / D][i % D] = py[i];
  }
}

template <int MODEL, int RANGE, int NT>
__global__ void __launch_bounds__(NT, NT <= 256 ? 2 : 1) k_gen_split(BlockedJob job, Coef<double> cf, double kappa2, SplitCoef sc,
                                                  SplitTableau st, Tableau<double> tb, int H) {
  constexpr int D = Dim<MODEL>::D;
  constexpr bool PARK = NT <= 256;
  extern __shared__ __align__(16) unsigned char smem[];
  ChainDesc ch;
  int64_t tile = blockIdx.x;
  if (job.nchains == 1) {
    ch = job.one;
  } else {
    const int ci = batch_chain(job.bt, job.nchains, tile, smem, tile);
    ch = job.chains[ci];
    cf.kappa = ch.kappa;
    split_set_kappa(sc, ch.kappa);
  }
  const int W = blockDim.x * 2;
  const int64_t t0 = tile * (int64_t)job.G - H;
  ulonglong2 *ex = reinterpret_cast<ulonglong2 *>(smem);
  double *tl = reinterpret_cast<double *>(ex + 2 * blockDim.x);  // the tile, then the records in its place
  f32x2 *rec = reinterpret_cast<f32x2 *>(tl) + threadIdx.x * gen_record_words(st.s, D, PARK);
  tile_load<double, D, false>(tl, static_cast<const double *>(job.in), ch.off, ch.n, ch.bc, t0, W, job.total, job.hdr);
  tile_load_wait();
  __syncthreads();
  double y[2][D];
  const int base = threadIdx.x * 2;
  const bool edge_tile = ch.bc == FIXED && (t0 < 0 || t0 + W > ch.n);
  uint32_t ghost = 0;
  bool wide = false, live = false;  // as in tile_item
#pragma unroll
  for (int v = 0; v < 2; ++v) {
    const int64_t g = t0 + base + v;
    if (edge_tile && (g < 0 || g >= ch.n)) ghost |= 1u << v;
#pragma unroll
    for (int d = 0; d < D; ++d) {
      y[v][d] = tl[(base + v) * D + d];
      wide |= !split_in_range<MODEL>(y[v][d], d, cf.c, sc);
      live |= !is_nan(y[v][d]) && !((ghost >> v) & 1u);
    }
  }
  const bool nan_tile = __syncthreads_or(wide);
  if (nan_tile && __syncthreads_or(live)) {
    gen_wide_tile<MODEL, RANGE>(job, ch, t0, H, cf, kappa2, tb, smem);
    return;
  }
  if (edge_tile) gen_split_advance<MODEL, RANGE, true, PARK>(y, ghost, job.K, cf, kappa2, sc, st, ex, rec);
  else gen_split_advance<MODEL, RANGE, false, PARK>(y, 0u, job.K, cf, kappa2, sc, st, ex, rec);
  __syncthreads();  // every record is read before the tile is written over them
  const int64_t g0 = t0 + H, rem = ch.n - g0;
  const int cnt = (int)(rem < job.G ? rem : job.G);
  wide = false;
#pragma unroll
  for (int v = 0; v < 2; ++v)
#pragma unroll
    for (int d = 0; d < D; ++d) {
      tl[(base + v) * D + d] = y[v][d];
      wide |= base + v >= H && base + v < H + cnt && !split_in_range<MODEL>(y[v][d], d, cf.c, sc);
    }
  if (__syncthreads_or(wide) && !nan_tile) {
    gen_wide_tile<MODEL, RANGE>(job, ch, t0, H, cf, kappa2, tb, smem);
    return;
  }
  report_nonfinite(job.hdr, nan_tile);
  if (cnt > 0) tile_store<double, D>(static_cast<double *>(job.out), tl, ch.off, H, g0, cnt, job.total, W, job.hdr);
}

template <int MODEL, int RANGE, int NT>
static cudaError_t launch_gen_split_k(int threads, const BlockedJob &job, const CoefD &cfd, const TableauD &td,
                                      double dt, int H, cudaStream_t st) {
  constexpr int D = Dim<MODEL>::D;
  static PerDevice attr;
  const cudaError_t e = set_smem_limit_once(k_gen_split<MODEL, RANGE, NT>, 200 * 1024, attr);
  if (e != cudaSuccess) return e;
  if (job.ntiles <= 0) return cudaSuccess;
  const size_t ours = (size_t)threads * (2 * sizeof(ulonglong2) +
                                         sizeof(double) * std::max(2 * D, gen_record_words(td.s, D, NT <= 256)));
  const size_t wide = sizeof(double) * ((size_t)gen_edge_values(2) + (size_t)threads * 2 * D);
  k_gen_split<MODEL, RANGE, NT><<<(unsigned)job.ntiles, threads, std::max(ours, wide), st>>>(
      job, to_coef<double>(cfd, cfd.kappa), cfd.kappa2, split_coef(MODEL, cfd, true), split_tableau(td),
      to_tableau<double>(td, dt), H);
  return cudaGetLastError();
}
template <int MODEL, int RANGE>
static cudaError_t launch_gen_split_m(int sites, const BlockedJob &job, const CoefD &cf, const TableauD &tb, double dt,
                                      int H, cudaStream_t st) {
  const int threads = sites / 2;
  return threads <= 256 ? launch_gen_split_k<MODEL, RANGE, 256>(threads, job, cf, tb, dt, H, st)
                        : launch_gen_split_k<MODEL, RANGE, kGenSplitThreads>(threads, job, cf, tb, dt, H, st);
}

cudaError_t launch_gen_split(int model, int range, int sites, const BlockedJob &job, const CoefD &cf,
                             const TableauD &tb, double dt, int H, cudaStream_t st) {
  if (sites / 2 > kGenSplitThreads) return cudaErrorInvalidValue;
  if (model == ROESSLER)
    return range == 1 ? launch_gen_split_m<ROESSLER, 1>(sites, job, cf, tb, dt, H, st)
                      : launch_gen_split_m<ROESSLER, 2>(sites, job, cf, tb, dt, H, st);
  return range == 1 ? launch_gen_split_m<HARMONIC, 1>(sites, job, cf, tb, dt, H, st)
                    : launch_gen_split_m<HARMONIC, 2>(sites, job, cf, tb, dt, H, st);
}

// ---- one stage per launch ---------------------------------------------------------------------

// Stage state j in the split form: the increments d_j of every site (float pairs, in job.u).
template <int MODEL>
__global__ void __launch_bounds__(256) k_gen_split_state(GenStagedJob job, SplitTableau st, Tableau<double> tb, int j) {
  constexpr int D = Dim<MODEL>::D;
  if (job.hdr->wide[job.parity]) {
    gen_state_sweep<double, D>(job, tb, j);
    return;
  }
  const double *K = static_cast<const double *>(job.k);
  float2 *U = static_cast<float2 *>(job.u);
  const size_t plane = (size_t)job.total * D;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < (int64_t)plane; i += stride) {
    FPair<float> d = pair_mul<float>({st.ch[j], st.cl[j]}, -st.ch[j], split1(K[i]));
    for (int m = 1; m < j; ++m) {
      if (!((st.anz[j] >> m) & 1u)) continue;
      const float2 n = reinterpret_cast<const float2 *>(K + m * plane)[i];
      d = pair_fnma<float>({st.ah[j][m], st.al[j][m]}, -st.ah[j][m], {n.x, n.y}, d);
    }
    d = pair_norm(d);
    U[i] = make_float2(d.h, d.l);
  }
}

// Slope j: the first slope in FP64, or the negated difference of a later one as pairs.
template <int MODEL, int RANGE>
__global__ void __launch_bounds__(256) k_gen_split_slope(GenStagedJob job, Coef<double> cf, double kappa2, SplitCoef sc,
                                                         int j) {
  constexpr int D = Dim<MODEL>::D;
  if (j == 0 || job.hdr->wide[job.parity]) {
    gen_slope_sweep<double, MODEL, RANGE>(job, cf, kappa2, j);
    return;
  }
  const double *Y = static_cast<const double *>(job.y);
  const float2 *U = static_cast<const float2 *>(job.u);
  float2 *N = reinterpret_cast<float2 *>(static_cast<double *>(job.k) + (size_t)j * job.total * D);
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < job.total; i += stride) {
    ChainDesc ch;
    SplitCoef s = sc;
    if (job.nchains == 1) {
      ch = job.one;
    } else {
      int lo = 0, hi = job.nchains - 1;
      while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (job.chains[mid].off <= i) lo = mid; else hi = mid - 1;
      }
      ch = job.chains[lo];
      split_set_kappa(s, ch.kappa);
    }
    const int64_t li = i - ch.off;
    auto xat = [&](int64_t q) -> FPair<float> {  // coupling increment of chain site q
      const int64_t g = (ch.bc == PERIODIC) ? ch.off + wrap(q, ch.n) : ((q < 0 || q >= ch.n) ? -1 : ch.off + q);
      if (g < 0 || !bounds_ok(job.hdr, in_range(g, 1, job.total))) return {0.f, 0.f};
      const float2 u = U[g * D];
      return {u.x, u.y};
    };
    FPair<float> d[D], n[D];
#pragma unroll
    for (int q = 0; q < D; ++q) {
      const float2 u = U[i * D + q];
      d[q] = {u.x, u.y};
    }
    SplitBase<float> base = {};
    if constexpr (MODEL == ROESSLER) {
      base.z = split1(Y[i * D + 2]);
      base.t = x_minus_c<float>(split1(Y[i * D]), {s.ch, s.cl});
    }
    const FPair<float> none = {0.f, 0.f};
    split_stage<MODEL, float, RANGE, true>(d, xat(li - 1), xat(li + 1), base, stage_coef<float>(s), n,
                                     RANGE == 2 ? xat(li - 2) : none, RANGE == 2 ? xat(li + 2) : none);
#pragma unroll
    for (int q = 0; q < D; ++q) {
      n[q] = pair_norm(n[q]);
      N[i * D + q] = make_float2(n[q].h, n[q].l);
    }
  }
}

template <int MODEL>
__global__ void __launch_bounds__(256) k_gen_split_combine(GenStagedJob job, SplitCoef sc, SplitTableau st,
                                                           Tableau<double> tb) {
  constexpr int D = Dim<MODEL>::D;
  if (job.hdr->wide[job.parity]) {
    gen_combine_sweep<double, D, false>(job, tb);
    if (blockIdx.x == 0 && threadIdx.x == 0) job.hdr->wide[job.parity ^ 1] = 1u;
    return;
  }
  double *Y = static_cast<double *>(job.y);
  const double *K = static_cast<const double *>(job.k);
  const size_t plane = (size_t)job.total * D;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  bool wide = false, bad = false;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < (int64_t)plane; i += stride) {
    FPair<float> N = {0.f, vmul(-st.Bl, split1(K[i]).h)};
    for (int m = 1; m < st.s; ++m) {
      if (!((st.bnz >> m) & 1u)) continue;
      const float2 n = reinterpret_cast<const float2 *>(K + m * plane)[i];
      N = pair_fma<float>({st.bh[m], st.bl[m]}, -st.bh[m], {n.x, n.y}, N);
    }
    double nd;
    join(N, &nd, 1);
    const double r = fma(sc.w, fma(st.B, K[i], -nd), Y[i]);
    Y[i] = r;
    wide |= !split_in_range<MODEL>(r, (int)(i % D), sc.c, sc);
    bad |= nonfinite(r);
  }
  if (wide) job.hdr->wide[job.parity ^ 1] = 1u;
  if (bad) atomicOr(&job.hdr->status, ST_NONFINITE);
}

template <int MODEL, int RANGE>
static cudaError_t gen_split_step(const GenStagedJob &job, const CoefD &cfd, const TableauD &td, double dt,
                                  cudaStream_t st) {
  if (job.total <= 0) return cudaSuccess;
  const Tableau<double> tb = to_tableau<double>(td, dt);
  const SplitTableau stb = split_tableau(td);
  const SplitCoef sc = split_coef(MODEL, cfd, true);
  const Coef<double> cf = to_coef<double>(cfd, cfd.kappa);
  const unsigned grid = (unsigned)staged_grid(job.total);
  for (int j = 0; j < td.s; ++j) {
    if (j > 0) k_gen_split_state<MODEL><<<grid, 256, 0, st>>>(job, stb, tb, j);
    k_gen_split_slope<MODEL, RANGE><<<grid, 256, 0, st>>>(job, cf, cfd.kappa2, sc, j);
  }
  k_gen_split_combine<MODEL><<<grid, 256, 0, st>>>(job, sc, stb, tb);
  return cudaGetLastError();
}

cudaError_t launch_gen_split_step(int model, int range, const GenStagedJob &job, const CoefD &cf, const TableauD &tb,
                                  double dt, cudaStream_t st) {
  if (model == ROESSLER)
    return range == 1 ? gen_split_step<ROESSLER, 1>(job, cf, tb, dt, st) : gen_split_step<ROESSLER, 2>(job, cf, tb, dt, st);
  return range == 1 ? gen_split_step<HARMONIC, 1>(job, cf, tb, dt, st) : gen_split_step<HARMONIC, 2>(job, cf, tb, dt, st);
}

}  // namespace rk4d
