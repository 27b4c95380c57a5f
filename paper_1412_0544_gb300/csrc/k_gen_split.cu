// k_gen_split.cu -- the generic scheme (any explicit tableau of up to 7 stages, coupling range 1
// or 2) for FP64 in the split form of rk4_split.cuh, taken one term further: K1 = f(y) and M = J(y) K1
// (the first-order term of every later slope) in FP64, and what is left of the later slopes, the
// remainders r_m = K1 + c_m dt M - k_m, in float pairs:
//   u_j = y + dt (c_j K1 + e_j),  e_j = (sum_m a_jm c_m) dt M - sum_m a_jm r_m    (c_j the row sum; Eq. (4))
//   -r_j = dt J(y) e_j + (0, 0, dt^2 (c_j K1 + e_j)_x (c_j K1 + e_j)_z)       (f's only product: Eq. (6))
//   y <- y + dt (B K1 + (sum_m b_m c_m) dt M - sum_m b_m r_m)             (B the sum of the weights; Eq. (5)),
// for whatever tableau the kernel is given at run time.  A first stage after K1 (no a_jm with m >= 1) has
// e_j = 0 and needs no exchange, so a step exchanges as often as the tableau has stages.
//
// Why the extra term: the differences K1 - k_m are c_m dt |J| times K1, and with rows up to 25 in sum of
// magnitudes (Dormand-Prince 5) their pairs' errors showed: 1.05 of the FP64 form's error after one step
// (z 1.15, 2.2 at |x|, |z| = 20; x 1.04 with kappa = 2, kappa2 = 0.7), because the FP64 form rounds its state
// only once a step.  The remainders are smaller again by dt |J|: 0.87 .. 1.002 in each component after
// one and two steps (Dormand-Prince 5 and RK4, dt = 0.01 .. 0.06, kappa up to 2, kappa2 up to 0.7, |x|, |z| up
// to 15).  e_z, which x - c multiplies, is normalised (z 1.004 -> 0.981 with Fehlberg's tableau, dt = 0.0138).
// M's rows in pairs left x at 1.03.
// The weights' sum is carried to a float beyond FP64: its own rounding, times dt K1 every step, was a
// drift of 1.2 after 20 steps.
//
// What bounds it: the FP64 pipe takes 30 instructions per site-step with second neighbours (10 for K1, 11 for
// M, 3 and 6 for the update; 123 in the FP64 form) beside about 1300 FP32
// operations, 16 warps per SM (128 registers).  Every thread holds two sites (one packed pair) whatever the
// tiling's sites per thread, so a tile of W sites runs on W / 2 threads; M and the remainders lie in
// thread-private shared-memory records, which both frees their registers and lets the stage loops run over
// any tableau's nonzero entries without a kernel per tableau.  Measured at N = 2^20, us per step, best
// tiling, FP64 form -> now: Dormand-Prince 5 + second neighbours 245 -> 101, RK4 + second neighbours 128 -> 83
// (78 and 54 with differences from K1 alone, 16 FP64 instructions).
#include <algorithm>

#include "rk4_generic.cuh"

namespace rk4d {

constexpr int kGenSplitThreads = 512;

// 8-byte words of a thread's record: -dt M and the remainders of `slots` stages as pairs and, when parked
// (blocks of up to 256 threads), the state and the FP64 part of the update; odd (see split_record_words).
__host__ __device__ constexpr int gen_record_words(int slots, int D, bool park) {
  return ((slots + 1 + (park ? 2 : 0)) * D * 2) | 1;
}

// r_z = -(z dt e_x + (x - c) dt e_z + (dt dx)(dt dz)), the first two only when there is an e (EX); nde, dfe:
// dt e_x = dfe - nde (split_linear); d: the increments c_j K1 + e of x and z.
template <typename T, bool EX>
__device__ __forceinline__ FPair<T> gen_remainder_z(const FPair<T> &dx, const FPair<T> &dz, const FPair<T> &ez, T nde, T dfe,
                                                    const SplitBase<T> &b, const FPair<T> &tau) {
  const T m1 = vset<T>(-1.f);
  const T ntau = vmul(m1, tau.h);
  FPair<T> u, v;
  T np3, e3;
  u = pair_mul(tau, ntau, dx);
  v = pair_mul(tau, ntau, dz);
  mul_coef(u, vmul(m1, u.h), v, np3, e3);
  if constexpr (!EX) return {np3, vmul(m1, e3)};
  T np1, e1, np2, e2, s, ne1, ne2;
  mul_coef(b.z, vmul(m1, b.z.h), FPair<T>{vmul(m1, nde), dfe}, np1, e1);
  mul_coef(b.t, vmul(m1, b.t.h), pair_mul(tau, ntau, ez), np2, e2);
  FPair<T> r;
  two_sum(np1, np2, s, ne1);
  two_sum(s, np3, r.h, ne2);
  r.l = vadd(vsub(ne1, vadd(e1, e2)), vsub(ne2, e3));
  return r;
}

// M = J(y) K1 of one site: slope_gen's rows are linear but for the Roessler chain's z.
template <int MODEL, int RANGE>
__device__ __forceinline__ void gen_second_slope(const double *y, const double *k1, double l1, double r1, double l2,
                                                 double r2, const Coef<double> &cf, double kappa2, double *M) {
  slope_gen<double, MODEL, RANGE>(k1, l1, r1, l2, r2, cf, kappa2, M);
  if constexpr (MODEL == ROESSLER) M[2] = fma(y[2], k1[0], mul(fma(y[0], cf.one, -cf.c), k1[2]));
}
// The FP64 part of the update, B K1 + (sum_m b_m c_m) dt M.
__device__ __forceinline__ double gen_update64(double k1, double M, const SplitTableau &tb) {
  return fma(tb.E, M, tb.unit ? k1 : mul(tb.B, k1));
}
// -dt M as a pair.
template <typename T> __device__ __forceinline__ FPair<T> gen_first_order(const FPair<T> &M, const FPair<T> &tau) {
  const T m1 = vset<T>(-1.f);
  return pair_mul(FPair<T>{vmul(m1, tau.h), vmul(m1, tau.l)}, tau.h, M);
}

// A tile outside the split's range in the FP64 form (two sites per thread).  SHAPE: the tableau's nonzero
// pattern where it is one of the compiled ones (Dormand-Prince 5 + second neighbours, 2^20 sites,
// 128 x 4 x 2, a state of 1e-25: 302 -> 251 us per step, 269 as the one form of a kernel of its own).
template <int MODEL, int RANGE, uint64_t SHAPE>
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
  gen_tile_advance<double, MODEL, V, RANGE, false, true, SHAPE>(y, cmp, ghost, job.K, cf, kappa2, tb, edge);
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
// coupling coordinates (FP64, or as a packed pair), read by its neighbours.
template <int MODEL, int RANGE, bool MASK, bool PARK>
__device__ __forceinline__ void gen_split_advance(double (&y)[2][Dim<MODEL>::D], uint32_t ghost, int K,
                                                  const Coef<double> &cf, double kappa2, const SplitCoef &sc,
                                                  const SplitTableau &tb, ulonglong2 *ex, f32x2 *rec) {
  constexpr int D = Dim<MODEL>::D;
  using T = f32x2;
  const int tid = threadIdx.x, bd = blockDim.x;
  const int lt = tid > 0 ? tid - 1 : tid, rt = tid < bd - 1 ? tid + 1 : tid;
  const StageCoef<T> c = stage_coef<T>(sc);
  f32x2 *rm = rec + 2 * D;  // the remainders, after -dt M
  double *py = reinterpret_cast<double *>(rm + tb.slots * 2 * D), *ps = py + 2 * D;
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
  auto exchange64 = [&](const double (&x)[2], double (&l)[2], double (&r)[2]) {
    ulonglong2 a, b;
    exchange(make_ulonglong2(__double_as_longlong(x[0]), __double_as_longlong(x[1])), a, b);
    l[1] = __longlong_as_double(a.x);
    l[0] = __longlong_as_double(a.y);
    r[0] = __longlong_as_double(b.x);
    r[1] = __longlong_as_double(b.y);
  };
#pragma unroll 1
  for (int s = 0; s < K; ++s) {
    double s64[2][D];
    FPair<T> k1x = {}, k1z = {};  // of the first slope only these two enter a product,
    T k1h[D];                     // and the heads B's rounding
    SplitBase<T> base = {};
    {
      if constexpr (PARK) {
#pragma unroll
        for (int i = 0; i < 2 * D; ++i) y[i / D][i % D] = py[i];
      }
      double x[2], l[2], r[2], k1[2][D], M[2][D];
#pragma unroll
      for (int v = 0; v < 2; ++v) x[v] = (MASK && ((ghost >> v) & 1u)) ? 0.0 : y[v][0];
      exchange64(x, l, r);
      slope_gen<double, MODEL, RANGE>(y[0], l[0], x[1], l[1], r[0], cf, kappa2, k1[0]);
      slope_gen<double, MODEL, RANGE>(y[1], x[0], r[0], l[0], r[1], cf, kappa2, k1[1]);
#pragma unroll
      for (int v = 0; v < 2; ++v) x[v] = (MASK && ((ghost >> v) & 1u)) ? 0.0 : k1[v][0];
      exchange64(x, l, r);
      gen_second_slope<MODEL, RANGE>(y[0], k1[0], l[0], x[1], l[1], r[0], cf, kappa2, M[0]);
      gen_second_slope<MODEL, RANGE>(y[1], k1[1], x[0], r[0], l[0], r[1], cf, kappa2, M[1]);
#pragma unroll
      for (int i = 0; i < D; ++i) {
#pragma unroll
        for (int v = 0; v < 2; ++v) s64[v][i] = gen_update64(k1[v][i], M[v][i], tb);
        const FPair<T> k = Lanes<T>::split(&k1[0][i], D);
        k1h[i] = k.h;
        if (i == 0) k1x = k;
        if (i == 2) k1z = k;
        const FPair<T> m = gen_first_order(Lanes<T>::split(&M[0][i], D), c.tau);
        rec[2 * i] = m.h;
        rec[2 * i + 1] = m.l;
      }
      if constexpr (MODEL == ROESSLER) {
        base.z = Lanes<T>::split(&y[0][2], D);
        base.t = x_minus_c<T>(Lanes<T>::split(&y[0][0], D), {vset<T>(sc.ch), vset<T>(sc.cl)});
      }
      if constexpr (PARK) {
#pragma unroll
        for (int i = 0; i < 2 * D; ++i) ps[i] = s64[i / D][i % D];
      }
    }
    FPair<T> n[D];
#pragma unroll 1
    for (int j = 1; j <= tb.last; ++j) {
      if (!((tb.need >> j) & 1u)) continue;
      FPair<T> e[D];
#pragma unroll
      for (int i = 0; i < D; ++i) n[i] = e[i] = {0ull, 0ull};
      T nde = 0ull, dfe = 0ull;
      const bool row = tb.na[j] > 0;
      if (row) {
        const FPair<T> g = {vset<T>(-tb.gh[j]), vset<T>(-tb.gl[j])};
        const T ng = vset<T>(tb.gh[j]);
#pragma unroll
        for (int i = 0; i < D; ++i) e[i] = pair_mul(g, ng, {rec[2 * i], rec[2 * i + 1]});
#pragma unroll 2
        for (int q0 = 0; q0 < tb.na[j]; ++q0) {
          const int m = tb.ma[j][q0];
          const FPair<T> a = {vset<T>(tb.ah[j][m]), vset<T>(tb.al[j][m])};
          const T na = vset<T>(-tb.ah[j][m]);
          const f32x2 *q = rm + tb.slot[m] * D * 2;
#pragma unroll
          for (int i = 0; i < D; ++i) e[i] = pair_fnma<T>(a, na, {q[2 * i], q[2 * i + 1]}, e[i]);
        }
        if constexpr (MODEL == ROESSLER) e[2] = pair_norm(e[2]);
        FPair<T> X = e[0];
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
        split_linear<MODEL, T, RANGE>(e, xl, xr, c, n, nde, dfe, {l.x, l.y}, {r.x, r.y});
      }
      if constexpr (MODEL == ROESSLER) {
        const FPair<T> cj = {vset<T>(tb.ch[j]), vset<T>(tb.cl[j])};
        const T nc = vset<T>(-tb.ch[j]);
        const FPair<T> dx = pair_fma(cj, nc, k1x, e[0]), dz = pair_fma(cj, nc, k1z, e[2]);
        n[2] = row ? gen_remainder_z<T, true>(dx, dz, e[2], nde, dfe, base, c.tau)
                   : gen_remainder_z<T, false>(dx, dz, e[2], nde, dfe, base, c.tau);
      }
      if (j != tb.last) {
        f32x2 *o = rm + tb.slot[j] * D * 2;
#pragma unroll
        for (int i = 0; i < D; ++i) {
          o[2 * i] = n[i].h;
          o[2 * i + 1] = n[i].l;
        }
      }
    }
    FPair<T> N[D];
#pragma unroll
    for (int i = 0; i < D; ++i) N[i] = {0ull, vmul(vset<T>(-tb.Bl), k1h[i])};
#pragma unroll 2
    for (int q0 = 0; q0 < tb.nb; ++q0) {
      const int m = tb.mb[q0];
      const FPair<T> b = {vset<T>(tb.bh[m]), vset<T>(tb.bl[m])};
      const T nb = vset<T>(-tb.bh[m]);
      const f32x2 *q = rm + tb.slot[m] * D * 2;
#pragma unroll
      for (int i = 0; i < D; ++i) N[i] = pair_fma<T>(b, nb, {q[2 * i], q[2 * i + 1]}, N[i]);
    }
    const FPair<T> bl = {vset<T>(tb.bh[tb.last]), vset<T>(tb.bl[tb.last])};
    const T nbl = vset<T>(-tb.bh[tb.last]);
#pragma unroll
    for (int i = 0; i < D; ++i) {
      double nd[2];
      join(pair_fma<T>(bl, nbl, n[i], N[i]), nd, 1);
#pragma unroll
      for (int v = 0; v < 2; ++v) {
        if constexpr (PARK) {
          py[v * D + i] = fma(sc.w, fma(ps[v * D + i], cf.one, -nd[v]), py[v * D + i]);
        } else {
          y[v][i] = fma(sc.w, fma(s64[v][i], cf.one, -nd[v]), y[v][i]);
        }
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
                                                  SplitTableau st, Tableau<double> tb, uint64_t shape, int H) {
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
  auto wide_tile = [&]() {
    if (shape == kShapeDopri5) gen_wide_tile<MODEL, RANGE, kShapeDopri5>(job, ch, t0, H, cf, kappa2, tb, smem);
    else if (shape == kShapeRK4) gen_wide_tile<MODEL, RANGE, kShapeRK4>(job, ch, t0, H, cf, kappa2, tb, smem);
    else gen_wide_tile<MODEL, RANGE, 0>(job, ch, t0, H, cf, kappa2, tb, smem);
  };
  ulonglong2 *ex = reinterpret_cast<ulonglong2 *>(smem);
  double *tl = reinterpret_cast<double *>(ex + 2 * blockDim.x);  // the tile, then the records in its place
  f32x2 *rec = reinterpret_cast<f32x2 *>(tl) + threadIdx.x * gen_record_words(st.slots, D, PARK);
  tile_load<double, D, false>(tl, static_cast<const double *>(job.in), ch.off, ch.n, ch.bc, t0, W, job.total, job.hdr);
  tile_load_wait();
  __syncthreads();
  double y[2][D];
  const int base = threadIdx.x * 2;
  const bool edge_tile = ch.bc == FIXED && (t0 < 0 || t0 + W > ch.n);
  uint32_t ghost = 0;
  auto own_c = [](int) -> const double * { return nullptr; };
  bool odd = false, nan_tile = false;  // as in tile_item
#pragma unroll
  for (int v = 0; v < 2; ++v) {
    const int64_t g = t0 + base + v;
    if (edge_tile && (g < 0 || g >= ch.n)) ghost |= 1u << v;
#pragma unroll
    for (int d = 0; d < D; ++d) {
      y[v][d] = tl[(base + v) * D + d];
      odd |= !((ghost >> v) & 1u) && !split_holds<MODEL>(y[v][d], d, nullptr, sc);
    }
  }
  if (__syncthreads_or(odd)) {
    const int last = base + 2;
    const bool next = last < W && (!edge_tile || (t0 + last >= 0 && t0 + last < ch.n));
    const int b = block_or(split_tile_bits<MODEL, 2>(y, ghost, sc, next ? tl + last * D : nullptr, own_c, [](int) { return true; }),
                           reinterpret_cast<int *>(smem));
    nan_tile = (b & kSplitWide) && !(b & kSplitLive);
    if (!nan_tile && ((b & kSplitWide) || ((b & kSplitGap) && (b & kSplitSome)))) {
      wide_tile();
      return;
    }
  }
  if (edge_tile) gen_split_advance<MODEL, RANGE, true, PARK>(y, ghost, job.K, cf, kappa2, sc, st, ex, rec);
  else gen_split_advance<MODEL, RANGE, false, PARK>(y, 0u, job.K, cf, kappa2, sc, st, ex, rec);
  __syncthreads();  // every record is read before the tile is written over them
  const int64_t g0 = t0 + H, rem = ch.n - g0;
  const int cnt = (int)(rem < job.G ? rem : job.G);
  auto stored_site = [&](int v) { return base + v >= H && base + v < H + cnt; };
  odd = false;
#pragma unroll
  for (int v = 0; v < 2; ++v)
#pragma unroll
    for (int d = 0; d < D; ++d) {
      tl[(base + v) * D + d] = y[v][d];
      odd |= stored_site(v) && !split_holds<MODEL>(y[v][d], d, nullptr, sc);
    }
  if (__syncthreads_or(odd) && !nan_tile) {
    const int b = block_or(split_tile_bits<MODEL, 2>(y, ghost, sc, nullptr, own_c, stored_site), reinterpret_cast<int *>(smem));
    if ((b & kSplitWide) || split_has_front(b)) {
      wide_tile();
      return;
    }
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
  const SplitTableau stb = split_tableau(td, dt);
  const size_t ours = (size_t)threads * (2 * sizeof(ulonglong2) +
                                         sizeof(double) * std::max(2 * D, gen_record_words(stb.slots, D, NT <= 256)));
  const size_t wide = sizeof(double) * ((size_t)gen_edge_values(2) + (size_t)threads * 2 * D);
  k_gen_split<MODEL, RANGE, NT><<<(unsigned)job.ntiles, threads, std::max(ours, wide), st>>>(
      job, to_coef<double>(cfd, cfd.kappa), cfd.kappa2, split_coef(MODEL, cfd, true), stb,
      to_tableau<double>(td, dt), tableau_shape(td), H);
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

// M of site i from the first slopes in job.k.
template <int MODEL, int RANGE>
__device__ __forceinline__ void gen_staged_second(const GenStagedJob &job, const ChainDesc &ch, int64_t i,
                                                  const Coef<double> &c, double kappa2, double *M) {
  constexpr int D = Dim<MODEL>::D;
  const double *Y = static_cast<const double *>(job.y), *K = static_cast<const double *>(job.k);
  const int64_t li = i - ch.off;
  auto xat = [&](int64_t q) {
    const int64_t g = gen_site(job, ch, q);
    return g < 0 ? 0.0 : K[g * D];
  };
  double y[D], k1[D];
#pragma unroll
  for (int q = 0; q < D; ++q) {
    y[q] = Y[i * D + q];
    k1[q] = K[i * D + q];
  }
  gen_second_slope<MODEL, RANGE>(y, k1, xat(li - 1), xat(li + 1), RANGE == 2 ? xat(li - 2) : 0.0,
                                 RANGE == 2 ? xat(li + 2) : 0.0, c, kappa2, M);
}

// Stage state j in the split form: e_j of every site (float pairs, in job.u).
template <int MODEL, int RANGE>
__global__ void __launch_bounds__(256) k_gen_split_state(GenStagedJob job, Coef<double> cf, double kappa2, SplitCoef sc,
                                                         SplitTableau st, Tableau<double> tb, int j) {
  constexpr int D = Dim<MODEL>::D;
  const double *K = static_cast<const double *>(job.k);
  float2 *U = static_cast<float2 *>(job.u);
  const size_t plane = (size_t)job.total * D;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < job.total; i += stride) {
    Coef<double> c = cf;
    int ci;
    const ChainDesc ch = gen_site_chain(job, i, c, ci);
    if (wide_chain(job.wide[2 * ci + job.parity])) {
      gen_state_site<double, D>(job, tb, i, j);
      continue;
    }
    if (st.na[j] == 0) continue;  // e_j = 0
    double M[D];
    gen_staged_second<MODEL, RANGE>(job, ch, i, c, kappa2, M);
#pragma unroll
    for (int d = 0; d < D; ++d) {
      const FPair<float> nm = gen_first_order<float>(split1(M[d]), {sc.tauh, sc.taul});
      FPair<float> e = pair_mul<float>({-st.gh[j], -st.gl[j]}, st.gh[j], nm);
      for (int q = 0; q < st.na[j]; ++q) {
        const int m = st.ma[j][q];
        const float2 n = reinterpret_cast<const float2 *>(K + m * plane)[i * D + d];
        e = pair_fnma<float>({st.ah[j][m], st.al[j][m]}, -st.ah[j][m], {n.x, n.y}, e);
      }
      if (MODEL == ROESSLER && d == 2) e = pair_norm(e);
      U[i * D + d] = make_float2(e.h, e.l);
    }
  }
}

// Slope j: the first slope in FP64, or the remainder of a later one as pairs.
template <int MODEL, int RANGE>
__global__ void __launch_bounds__(256) k_gen_split_slope(GenStagedJob job, Coef<double> cf, double kappa2, SplitCoef sc,
                                                         SplitTableau st, int j) {
  constexpr int D = Dim<MODEL>::D;
  const double *Y = static_cast<const double *>(job.y), *K = static_cast<const double *>(job.k);
  const float2 *U = static_cast<const float2 *>(job.u);
  float2 *N = reinterpret_cast<float2 *>(static_cast<double *>(job.k) + (size_t)j * job.total * D);
  const bool row = st.na[j] > 0;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < job.total; i += stride) {
    Coef<double> c = cf;
    int ci;
    const ChainDesc ch = gen_site_chain(job, i, c, ci);
    if (j == 0 || wide_chain(job.wide[2 * ci + job.parity])) {
      gen_slope_site<double, MODEL, RANGE>(job, ch, c, kappa2, i, j);
      continue;
    }
    SplitCoef s = sc;
    split_set_kappa(s, c.kappa);
    const int64_t li = i - ch.off;
    auto xat = [&](int64_t q) -> FPair<float> {
      const int64_t g = gen_site(job, ch, q);
      if (g < 0) return {0.f, 0.f};
      const float2 u = U[g * D];
      return {u.x, u.y};
    };
    const StageCoef<float> co = stage_coef<float>(s);
    FPair<float> e[D], n[D];
#pragma unroll
    for (int q = 0; q < D; ++q) n[q] = e[q] = {0.f, 0.f};
    float nde = 0.f, dfe = 0.f;
    if (row) {
#pragma unroll
      for (int q = 0; q < D; ++q) {
        const float2 u = U[i * D + q];
        e[q] = {u.x, u.y};
      }
      const FPair<float> none = {0.f, 0.f};
      split_linear<MODEL, float, RANGE>(e, xat(li - 1), xat(li + 1), co, n, nde, dfe, RANGE == 2 ? xat(li - 2) : none,
                                        RANGE == 2 ? xat(li + 2) : none);
    }
    if constexpr (MODEL == ROESSLER) {
      const FPair<float> cj = {st.ch[j], st.cl[j]};
      const FPair<float> dx = pair_fma(cj, -cj.h, split1(K[i * D]), e[0]), dz = pair_fma(cj, -cj.h, split1(K[i * D + 2]), e[2]);
      const SplitBase<float> base = {split1(Y[i * D + 2]), x_minus_c<float>(split1(Y[i * D]), {s.ch, s.cl})};
      n[2] = row ? gen_remainder_z<float, true>(dx, dz, e[2], nde, dfe, base, co.tau)
                 : gen_remainder_z<float, false>(dx, dz, e[2], nde, dfe, base, co.tau);
    }
#pragma unroll
    for (int q = 0; q < D; ++q) N[i * D + q] = make_float2(n[q].h, n[q].l);
  }
}

template <int MODEL, int RANGE>
__global__ void __launch_bounds__(256) k_gen_split_combine(GenStagedJob job, Coef<double> cf, double kappa2, SplitCoef sc,
                                                           SplitTableau st, Tableau<double> tb) {
  constexpr int D = Dim<MODEL>::D;
  double *Y = static_cast<double *>(job.y);
  const double *K = static_cast<const double *>(job.k);
  const size_t plane = (size_t)job.total * D;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < job.total; i += stride) {
    Coef<double> c = cf;
    int ci;
    const ChainDesc ch = gen_site_chain(job, i, c, ci);
    unsigned *next = job.wide + 2 * ci + (job.parity ^ 1);
    if (wide_chain(job.wide[2 * ci + job.parity])) {
      gen_combine_site<double, D, false>(job, tb, i);
      *next = kWideRange;
      continue;
    }
    bool wide = false, bad = false;
    double M[D];
    gen_staged_second<MODEL, RANGE>(job, ch, i, c, kappa2, M);
#pragma unroll
    for (int d = 0; d < D; ++d) {
      FPair<float> N = {0.f, vmul(-st.Bl, split1(K[i * D + d]).h)};
      for (int q = 0; q <= st.nb; ++q) {
        const int m = q < st.nb ? st.mb[q] : st.last;
        const float2 n = reinterpret_cast<const float2 *>(K + m * plane)[i * D + d];
        N = pair_fma<float>({st.bh[m], st.bl[m]}, -st.bh[m], {n.x, n.y}, N);
      }
      double nd;
      join(N, &nd, 1);
      const double r = fma(sc.w, fma(gen_update64(K[i * D + d], M[d], st), c.one, -nd), Y[i * D + d]);
      Y[i * D + d] = r;
      wide |= !split_in_range<MODEL>(r, d, nullptr, sc);
      bad |= nonfinite(r);
    }
    if (wide) *next = kWideRange;
    if (bad) atomicOr(&job.hdr->status, ST_NONFINITE);
  }
}

template <int MODEL, int RANGE>
static cudaError_t gen_split_step(const GenStagedJob &job, const CoefD &cfd, const TableauD &td, double dt,
                                  cudaStream_t st) {
  if (job.total <= 0) return cudaSuccess;
  const Tableau<double> tb = to_tableau<double>(td, dt);
  const SplitTableau stb = split_tableau(td, dt);
  const SplitCoef sc = split_coef(MODEL, cfd, true);
  const Coef<double> cf = to_coef<double>(cfd, cfd.kappa);
  const unsigned grid = (unsigned)staged_grid(job.total);
  for (int j = 0; j < td.s; ++j) {
    if (j > 0) k_gen_split_state<MODEL, RANGE><<<grid, 256, 0, st>>>(job, cf, cfd.kappa2, sc, stb, tb, j);
    k_gen_split_slope<MODEL, RANGE><<<grid, 256, 0, st>>>(job, cf, cfd.kappa2, sc, stb, j);
  }
  k_gen_split_combine<MODEL, RANGE><<<grid, 256, 0, st>>>(job, cf, cfd.kappa2, sc, stb, tb);
  return cudaGetLastError();
}

cudaError_t launch_gen_split_step(int model, int range, const GenStagedJob &job, const CoefD &cf, const TableauD &tb,
                                  double dt, cudaStream_t st) {
  if (model == ROESSLER)
    return range == 1 ? gen_split_step<ROESSLER, 1>(job, cf, tb, dt, st) : gen_split_step<ROESSLER, 2>(job, cf, tb, dt, st);
  return range == 1 ? gen_split_step<HARMONIC, 1>(job, cf, tb, dt, st) : gen_split_step<HARMONIC, 2>(job, cf, tb, dt, st);
}

}  // namespace rk4d
