// rk4_tile.cuh -- temporal blocking of one tile (Sec. 2.3 of the paper, on the GPU).
//
// A thread block owns a tile of W = blockDim.x * V consecutive sites of one chain: the G
// interior sites it will write back plus a halo of H = 4k sites on each side.  Thread t holds
// sites t*V .. t*V+V-1 in registers.  Every RK stage needs the coupling coordinate of both
// neighbours: inside a thread it is a register, across threads an exchange through shared
// memory (one __syncthreads per stage; see tile_advance).  Sites at the tile's
// ends read a stand-in value, so after m stages only sites [m, W - m) are exact -- the
// paper's observation that the error from the missing coupling moves one site inward per
// stage -- and after 4k stages exactly the interior [4k, W - 4k) is.
//
// Fixed ends: sites of the tile outside the chain are ghosts whose coupling coordinate is
// forced to zero at every stage (r_0 = r_{N+1} = 0).  Periodic ends: the tile is a window of
// the periodically extended chain (indices taken mod N), so no special case is needed.
#pragma once
#include <type_traits>

#include "rk4_device.cuh"
#include "rk4_internal.h"
#include "rk4_split.cuh"

namespace rk4d {

constexpr unsigned kFull = 0xffffffffu;

// Index checks of a debug build (-DRK4_DEBUG_BOUNDS): a range that would leave its buffer
// latches ST_BOUNDS in the status word and the access is skipped.  In a release build the
// check is the constant true and costs nothing.
__device__ __forceinline__ bool bounds_ok(WsHeader *hdr, bool ok) {
#ifdef RK4_DEBUG_BOUNDS
  if (!ok && hdr) atomicOr(&hdr->status, ST_BOUNDS);
  return ok;
#else
  (void)hdr;
  (void)ok;
  return true;
#endif
}

// Whether [first, first + count) lies inside [0, size).
__device__ __forceinline__ bool in_range(int64_t first, int64_t count, int64_t size) {
  return first >= 0 && count >= 0 && first + count <= size;
}

// NaN or infinity, tested on the exponent bits with integer instructions: a floating-point
// compare would take issue slots of the FP64 pipe, which bounds the FP64 kernels.
__device__ __forceinline__ bool nonfinite(double x) {
  return (__double2hiint(x) & 0x7ff00000) == 0x7ff00000;
}
__device__ __forceinline__ bool nonfinite(float x) {
  return (__float_as_uint(x) & 0x7f800000u) == 0x7f800000u;
}

// Latch ST_NONFINITE when any value of a result about to be stored is NaN or infinite (one
// thread per block reports; `any` is the block-wide vote).
__device__ __forceinline__ void report_nonfinite(WsHeader *hdr, int any) {
  if (any && threadIdx.x == 0 && hdr) atomicOr(&hdr->status, ST_NONFINITE);
}

// Largest block the tile kernels are compiled for, by sites per thread: the register budget
// (about 9 values per site plus temporaries) must fit 65536 registers per block.
__host__ __device__ constexpr int max_threads_for(int v) { return v <= 1 ? 1024 : (v <= 4 ? 512 : 256); }

// Neighbour exchange of the tile kernels, by sites per thread: with 4 or more, every thread
// publishes its end values in shared memory (fewer MIO instructions, measured +4-8 % in FP32
// and +2 % in heterogeneous FP64); with fewer, warp shuffles plus warp-edge slots (the
// per-thread slots' four address registers cost 6-12 more registers there, which drops a
// resident block: -12 to -18 %).
__host__ __device__ constexpr bool thread_exchange(int v) { return v >= 4; }
// Shared-memory values the exchange takes at the front of a tile kernel's dynamic shared memory.
__host__ __device__ constexpr int edge_values(int v) { return thread_exchange(v) ? 4 * max_threads_for(v) : 128; }

// Store v to shared memory only when p holds, as a predicated instruction (no divergent
// branch around it).
__device__ __forceinline__ void st_shared_if(bool p, float *a, float v) {
  const unsigned s = static_cast<unsigned>(__cvta_generic_to_shared(a));
  asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.b32 q, %2, 0;\n\t@q st.shared.f32 [%0], %1;\n\t}" ::"r"(s), "f"(v),
               "r"(static_cast<int>(p))
               : "memory");
}
__device__ __forceinline__ void st_shared_if(bool p, double *a, double v) {
  const unsigned s = static_cast<unsigned>(__cvta_generic_to_shared(a));
  asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.b32 q, %2, 0;\n\t@q st.shared.f64 [%0], %1;\n\t}" ::"r"(s), "d"(v),
               "r"(static_cast<int>(p))
               : "memory");
}

// Shared-memory accesses through 32-bit shared-window addresses (four such registers per
// thread carry the neighbour exchange below; generic pointers would take twice as many).
__device__ __forceinline__ unsigned smem_addr(const void *p) {
  return static_cast<unsigned>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ void st_shared(unsigned a, float v) {
  asm volatile("st.shared.f32 [%0], %1;" ::"r"(a), "f"(v) : "memory");
}
__device__ __forceinline__ void st_shared(unsigned a, double v) {
  asm volatile("st.shared.f64 [%0], %1;" ::"r"(a), "d"(v) : "memory");
}
__device__ __forceinline__ void ld_shared(unsigned a, float &v) {
  asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(a) : "memory");
}
__device__ __forceinline__ void ld_shared(unsigned a, double &v) {
  asm volatile("ld.shared.f64 %0, [%1];" : "=d"(v) : "r"(a) : "memory");
}

// Synchronise this warp with its two neighbouring warps only, for a neighbour exchange in
// which each thread reads the slots of the threads just before and after it: one named barrier
// per pair of adjacent warps (ids 1 .. 15, 64 threads each; id 0 is __syncthreads), so a warp
// waits for its neighbours rather than for the slowest warp of the block.  Warp w takes the
// barrier it shares with w - 1 and then the one it shares with w + 1; the chain starting at
// warp 0 (which has no left barrier) completes every pair, so no warp waits forever.  The
// barriers also order the shared-memory accesses of the threads of each warp.  Needs a block of
// at most 16 warps (512 threads), every thread of a warp taking part.
__device__ __forceinline__ void neighbour_warp_sync() {
  const int w = threadIdx.x >> 5, nw = blockDim.x >> 5;
  if (nw > 16) {  // more pairs than named barriers: the whole block instead (block-uniform)
    __syncthreads();
    return;
  }
  if (nw == 1) {
    __syncwarp();
    return;
  }
  if (w > 0) asm volatile("bar.sync %0, 64;" ::"r"(w) : "memory");
  if (w < nw - 1) asm volatile("bar.sync %0, 64;" ::"r"(w + 1) : "memory");
}

// The barrier of a tile kernel's neighbour exchange, where each thread (warp) reads only the
// slots of its neighbours: FP64 waits for the neighbouring warps only (neighbour_warp_sync,
// measured 7 % faster: the warps of a block no longer enter each stage's FP64 stream in lock
// step); FP32 keeps the one block-wide barrier per stage (the two named barriers measured 16-28 %
// slower there).
template <typename R> __device__ __forceinline__ void stage_sync() {
  if constexpr (sizeof(R) == 8) neighbour_warp_sync(); else __syncthreads();
}

// Advance the registers of one tile by K steps.  `edge` is edge_values(V) values of shared
// memory, two alternating slots by stage parity.  Per-thread exchange (thread_exchange(V)): a
// slot is [first x of each thread | last x of each thread], strided by the compile-time
// largest block so that the per-stage offsets are immediates; every thread stores its two
// coupling coordinates and, after the stage's one barrier, loads its neighbours'
// (conflict-free: consecutive threads, consecutive addresses), four shared-memory
// instructions per warp and stage.  Warp exchange: a slot is [first x of each warp | last x
// of each warp]; shuffles carry the values inside a warp and lanes 0 and 31 publish theirs by
// predicated stores, read back as uniform (broadcast) loads and selects.  Either way the two
// tile ends read a stand-in (their own value), which only ever reaches halo sites.  Stage 0
// of every step reads y directly (it is the stage state), so no register copies are needed
// between steps.
template <typename R, int MODEL, int V, bool KAHAN, bool MASK, bool HET = false>
__device__ __forceinline__ void tile_advance(R (&y)[V][Dim<MODEL>::D], R (&cmp)[V][Dim<MODEL>::D],
                                             uint32_t ghost, int K, const Coef<R> &cf, R *edge,
                                             const Coef<R> *cs = nullptr) {
  constexpr int D = Dim<MODEL>::D;
  constexpr bool kThread = thread_exchange(V);
  constexpr int NT = max_threads_for(V);
  const int tid = threadIdx.x;
  // per-thread exchange: this thread's slots (parity 0) and its neighbours' (unused and
  // never computed by the warp exchange)
  unsigned my_first = 0, my_last = 0, left_last = 0, right_first = 0;
  if constexpr (kThread) {
    my_first = smem_addr(edge + tid);
    my_last = smem_addr(edge + NT + tid);
    left_last = my_last - (tid > 0 ? (unsigned)sizeof(R) : 0u);
    right_first = my_first + (tid < (int)blockDim.x - 1 ? (unsigned)sizeof(R) : 0u);
  }
  // warp exchange
  const int lane = tid & 31;
  const int warp = tid >> 5;
  const int nw = blockDim.x >> 5;
  const bool is_first = lane == 0, is_last = lane == 31;
  const int prev = (warp > 0) ? warp - 1 : warp;
  const int next = (warp < nw - 1) ? warp + 1 : warp;
  R u[V][D], acc[V][D];
  // FP32-Kahan tiles with an even number of sites per thread run on packed instructions
  constexpr bool kPacked = std::is_same<R, float>::value && KAHAN && (V % 2 == 0);
  constexpr int P = V / 2;
  if constexpr (kPacked) {
#pragma unroll
    for (int v = 0; v < V; ++v)
#pragma unroll
      for (int d = 0; d < D; ++d) hold<MODEL>(d, y[v][d], cmp[v][d]);
  }

#pragma unroll 2  // halves the loop-carried register moves (measured +4 % in FP32)
  for (int s = 0; s < K; ++s) {
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      R xs[V];
#pragma unroll
      for (int v = 0; v < V; ++v) {
        const R x = (j == 0) ? y[v][0] : u[v][0];
        xs[v] = (MASK && ((ghost >> v) & 1u)) ? R(0) : x;
      }
      R left, right;
      if constexpr (kThread) {
        const unsigned po = (j & 1) * 2 * NT * (unsigned)sizeof(R);  // the stage's parity slot
        st_shared(my_first + po, xs[0]);
        st_shared(my_last + po, xs[V - 1]);
        stage_sync<R>();
        ld_shared(left_last + po, left);
        ld_shared(right_first + po, right);
      } else {
        left = __shfl_up_sync(kFull, xs[V - 1], 1);
        right = __shfl_down_sync(kFull, xs[0], 1);
        R *eb = edge + (j & 1) * 64;  // [0,32): first x of each warp, [32,64): last x
        st_shared_if(is_first, eb + warp, xs[0]);
        st_shared_if(is_last, eb + 32 + warp, xs[V - 1]);
        stage_sync<R>();
        const R from_prev = eb[32 + prev];
        const R from_next = eb[next];
        left = is_first ? from_prev : left;
        right = is_last ? from_next : right;
      }
      if constexpr (kPacked) {
        // sites p and p + V / 2 in the two halves of packed FP32 instructions: a pair's neighbours
        // are, except at the thread's ends, the adjacent pairs as they stand
        float2 X[P];
#pragma unroll
        for (int p = 0; p < P; ++p) X[p] = make_float2(xs[p], xs[p + P]);
        const float2 first = make_float2(left, xs[P - 1]), last = make_float2(xs[P], right);
#pragma unroll
        for (int p = 0; p < P; ++p) {
          float2 yy[D], uu[D], ac[D], cm[D], k[D];
#pragma unroll
          for (int d = 0; d < D; ++d) {
            yy[d] = make_float2(y[p][d], y[p + P][d]);
            uu[d] = (j == 0) ? yy[d] : make_float2(u[p][d], u[p + P][d]);
            ac[d] = make_float2(acc[p][d], acc[p + P][d]);
            cm[d] = make_float2(cmp[p][d], cmp[p + P][d]);
          }
          const Coef2 c2 = HET ? pair_coef(cs[p], cs[p + P]) : pair_coef(cf, cf);
          slope2<MODEL>(uu, p == 0 ? first : X[p - 1], p == P - 1 ? last : X[p + 1], c2, k);
          stage_update2<D>(j, k, yy, uu, ac, cm, c2);
#pragma unroll
          for (int d = 0; d < D; ++d) {
            y[p][d] = yy[d].x;
            y[p + P][d] = yy[d].y;
            u[p][d] = uu[d].x;
            u[p + P][d] = uu[d].y;
            acc[p][d] = ac[d].x;
            acc[p + P][d] = ac[d].y;
            cmp[p][d] = cm[d].x;
            cmp[p + P][d] = cm[d].y;
          }
        }
      } else {
#pragma unroll
        for (int v = 0; v < V; ++v) {
          const R xl = (v == 0) ? left : xs[v - 1];
          const R xr = (v == V - 1) ? right : xs[v + 1];
          R k[D];
          if constexpr (HET)
            slope<R, MODEL>((j == 0) ? y[v] : u[v], xl, xr, cs[v], k);  // site-dependent f_i, g_i (Eq. (1))
          else
            slope<R, MODEL>((j == 0) ? y[v] : u[v], xl, xr, cf, k);
          stage_update<R, D, KAHAN>(j, k, y[v], u[v], acc[v], cmp[v], cf);
        }
      }
    }
  }
  if constexpr (kPacked) {
#pragma unroll
    for (int v = 0; v < V; ++v)
#pragma unroll
      for (int d = 0; d < D; ++d) unhold<MODEL>(d, y[v][d], cmp[v][d]);
  }
}

// tile_advance for FP64 in the split form (rk4_split.cuh).  The same exchange and barriers; a
// stage's exchanged value is the coupling coordinate in FP64 for the first stage and its
// increment (head and tail, also 8 bytes) for the others.  The thread's V sites are paired
// (p, p + V / 2) for the packed instructions, so that a pair's neighbours are, except at the
// thread's ends, the adjacent pairs as they stand.
// spd, spf (heterogeneous chains): this thread's first private slots of the site parameters in
// FP64 (V x P, strided by the block) and of the pair coefficients (V / 2 packed kt, at and c).
// PARK: what a stage does not need every moment (the state and the first slope in FP64, the
// slope's pairs, the base values of z) lies in a record of the thread's own in shared memory,
// rec, of split_record_words() 8-byte words -- an odd number, so that the threads of a warp reach
// the same word of their records without bank conflicts.
// KREG: the coupling strength is a value of the thread's own (cf.kappa; packed tiles).
template <int MODEL, int V> __host__ __device__ constexpr int split_record_words() {
  return (3 * V * Dim<MODEL>::D + (MODEL == ROESSLER ? 2 * V : 0)) | 1;
}
// The FP64 constants of a split step, eight doubles for each warp in shared memory, which a step
// loads into registers: {1, -2, kappa, a | w2, c | -0, b, 6, tau / 3}.  A DFMA whose operands are
// three different registers was measured to issue every 16 cycles per SM and one with two (the third
// a constant or an immediate), or a DADD, every 19 (0.595 and 0.501 T/s, 4 to 32 warps per SM, any
// number of independent chains).  Left to itself the compiler feeds the constants from the
// constant bank, and 11 of the step's 13 instructions are of the slow kind.  Not with one site per
// thread, the form of short chains, which waits for latencies and not for the pipe (1000 sites,
// 128 x 1 x 8: 1.57 us per step without, 1.64 with).  N = 2^24, site-steps/s,
// before -> after: 256 x 4 x 8 3.41e10 -> 3.57e10, 256 x 4 x 4 3.42e10 -> 3.64e10, harmonic 128 x 4 x 4
// 5.74e10 -> 6.43e10.
__device__ __forceinline__ double *fp64_const_slot() {
  __shared__ __align__(16) double s[32][8];
  return s[threadIdx.x >> 5];
}
template <int MODEL>
__device__ __forceinline__ void fp64_const_store(const Coef<double> &cf, double w) {
  double *s = fp64_const_slot();
  if ((threadIdx.x & 31) == 0) {
    s[0] = 1.0;
    s[1] = -2.0;
    s[2] = cf.kappa;
    s[3] = MODEL == ROESSLER ? cf.a : cf.w2;
    s[4] = MODEL == ROESSLER ? cf.c : -0.0;
    s[5] = cf.b;
    s[6] = 6.0;
    s[7] = w;
  }
  __syncwarp();
}
__device__ __forceinline__ void ld_shared2(unsigned a, double &u, double &v) {
  asm volatile("ld.shared.v2.f64 {%0, %1}, [%2];" : "=d"(u), "=d"(v) : "r"(a) : "memory");
}

template <int MODEL, int V, bool MASK, bool HET, bool PARK = false, bool KREG = false>
__device__ __forceinline__ void split_advance(double (&y)[V][Dim<MODEL>::D], uint32_t ghost, int K,
                                              const Coef<double> &cf, const SplitCoef &sc, double *edge,
                                              const double *spd = nullptr, const f32x2 *spf = nullptr,
                                              double *rec = nullptr) {
  constexpr int D = Dim<MODEL>::D;
  constexpr int P = V < 2 ? 1 : V / 2;
  using T = std::conditional_t<V == 1, float, f32x2>;
  constexpr bool kThread = thread_exchange(V);
  constexpr int NT = max_threads_for(V);
  const int tid = threadIdx.x;
  unsigned my_first = 0, my_last = 0, left_last = 0, right_first = 0;
  if constexpr (kThread) {
    my_first = smem_addr(edge + tid);
    my_last = smem_addr(edge + NT + tid);
    left_last = my_last - (tid > 0 ? 8u : 0u);
    right_first = my_first + (tid < (int)blockDim.x - 1 ? 8u : 0u);
  }
  const int lane = tid & 31;
  const int warp = tid >> 5;
  const int nw = blockDim.x >> 5;
  const bool is_first = lane == 0, is_last = lane == 31;
  const int prev = (warp > 0) ? warp - 1 : warp;
  const int next = (warp < nw - 1) ? warp + 1 : warp;
  auto exchange = [&](int j, double first, double last, double &left, double &right) {
    if constexpr (kThread) {
      const unsigned po = (j & 1) * 2 * NT * 8u;
      st_shared(my_first + po, first);
      st_shared(my_last + po, last);
      neighbour_warp_sync();
      ld_shared(left_last + po, left);
      ld_shared(right_first + po, right);
    } else {
      left = __shfl_up_sync(kFull, last, 1);
      right = __shfl_down_sync(kFull, first, 1);
      double *eb = edge + (j & 1) * 64;
      st_shared_if(is_first, eb + warp, first);
      st_shared_if(is_last, eb + 32 + warp, last);
      neighbour_warp_sync();
      const double from_prev = eb[32 + prev];
      const double from_next = eb[next];
      left = is_first ? from_prev : left;
      right = is_last ? from_next : right;
    }
  };
  const StageCoef<T> sc0 = stage_coef<T>(sc);
  constexpr bool kConst = V > 1;
  unsigned fc = 0;
  if constexpr (kConst) {
    fp64_const_store<MODEL>(cf, sc.w);
    fc = smem_addr(fp64_const_slot());
  }
  static_assert(!PARK || V >= 2, "records hold packed pairs");
  double *rk = rec + V * D;                                      // first slope, FP64
  f32x2 *rp = reinterpret_cast<f32x2 *>(rec + 2 * V * D);        // its pairs: h, l of each (p, component)
  f32x2 *rb = reinterpret_cast<f32x2 *>(rec + 3 * V * D);        // z.h, z.l, t.h, t.l of each p
  if constexpr (PARK) {
#pragma unroll
    for (int v = 0; v < V; ++v)
#pragma unroll
      for (int i = 0; i < D; ++i) rec[v * D + i] = y[v][i];
  }

#pragma unroll 1
  for (int s = 0; s < K; ++s) {
    double k1d[V][D];
    FPair<T> k1[P][D], d[P][D], N[P][D];
    SplitBase<T> base[P];
    {
      if constexpr (PARK) {
#pragma unroll
        for (int v = 0; v < V; ++v)
#pragma unroll
          for (int i = 0; i < D; ++i) y[v][i] = rec[v * D + i];
      }
      double xs[V], left, right;
#pragma unroll
      for (int v = 0; v < V; ++v) xs[v] = (MASK && ((ghost >> v) & 1u)) ? 0.0 : y[v][0];
      exchange(0, xs[0], xs[V - 1], left, right);
      double one = cf.one, m2 = -2.0, kap = cf.kappa, p0 = MODEL == ROESSLER ? cf.a : cf.w2;
      double p1 = MODEL == ROESSLER ? cf.c : -0.0, p2 = cf.b;
      if constexpr (kConst) {
        ld_shared2(fc, one, m2);
        ld_shared2(fc + 16, kap, p0);
        ld_shared2(fc + 32, p1, p2);
        if constexpr (KREG) kap = cf.kappa;
      }
#pragma unroll
      for (int v = 0; v < V; ++v) {
        const double xl = (v == 0) ? left : xs[v - 1];
        const double xr = (v == V - 1) ? right : xs[v + 1];
        if constexpr (HET) {
          const double *q = spd + v * Dim<MODEL>::P * blockDim.x;
          p0 = q[0];
          if constexpr (MODEL == ROESSLER) {
            p2 = q[blockDim.x];
            p1 = q[2 * blockDim.x];
          }
          kap = q[(Dim<MODEL>::P - 1) * blockDim.x];
        }
        const double lap = fma(m2, y[v][0], fma(xl, one, xr));  // as slope() computes it
        if constexpr (MODEL == ROESSLER) {
          k1d[v][0] = fma(kap, lap, -fma(y[v][1], one, y[v][2]));
          k1d[v][1] = fma(p0, y[v][1], y[v][0]);
          k1d[v][2] = fma(y[v][2], y[v][0], fma(-p1, y[v][2], p2));
        } else {
          k1d[v][0] = y[v][1];
          k1d[v][1] = fma(kap, lap, -fma(p0, y[v][0], p1));  // p1 = -0: the rounded product
        }
      }
#pragma unroll
      for (int p = 0; p < P; ++p) {
#pragma unroll
        for (int i = 0; i < D; ++i) d[p][i] = k1[p][i] = Lanes<T>::split(&k1d[p][i], P * D);
        if constexpr (MODEL == ROESSLER) {
          FPair<T> c = {vset<T>(sc.ch), vset<T>(sc.cl)};
          if constexpr (HET) c = {spf[(p * 6 + 4) * blockDim.x], spf[(p * 6 + 5) * blockDim.x]};
          base[p].z = Lanes<T>::split(&y[p][2], P * D);
          base[p].t = x_minus_c(Lanes<T>::split(&y[p][0], P * D), c);
        }
      }
      if constexpr (PARK) {
#pragma unroll
        for (int v = 0; v < V; ++v)
#pragma unroll
          for (int i = 0; i < D; ++i) rk[v * D + i] = k1d[v][i];
#pragma unroll
        for (int p = 0; p < P; ++p) {
#pragma unroll
          for (int i = 0; i < D; ++i) {
            rp[(p * D + i) * 2] = k1[p][i].h;
            rp[(p * D + i) * 2 + 1] = k1[p][i].l;
          }
          if constexpr (MODEL == ROESSLER) {
            rb[p * 4] = base[p].z.h;
            rb[p * 4 + 1] = base[p].z.l;
            rb[p * 4 + 2] = base[p].t.h;
            rb[p * 4 + 3] = base[p].t.l;
          }
        }
      }
    }
#pragma unroll
    for (int j = 1; j < 4; ++j) {
      FPair<T> X[P];  // the increments' coupling coordinate, zero at ghost sites
#pragma unroll
      for (int p = 0; p < P; ++p) {
        X[p] = d[p][0];
        if constexpr (MASK) {
          if constexpr (V == 1) {
            if (ghost & 1u) X[p] = {0.f, 0.f};
          } else {
            const bool g0 = (ghost >> p) & 1u, g1 = (ghost >> (p + P)) & 1u;
            X[p].h = pack2(g0 ? 0.f : lane0(X[p].h), g1 ? 0.f : lane1(X[p].h));
            X[p].l = pack2(g0 ? 0.f : lane0(X[p].l), g1 ? 0.f : lane1(X[p].l));
          }
        }
      }
      FPair<T> first, last;  // left neighbours of the first pair, right neighbours of the last
      double left, right;
      if constexpr (V == 1) {
        const double mine = __longlong_as_double((long long)pack2(X[0].h, X[0].l));
        exchange(j, mine, mine, left, right);
        const f32x2 l = (f32x2)__double_as_longlong(left), r = (f32x2)__double_as_longlong(right);
        first = {lane0(l), lane1(l)};
        last = {lane0(r), lane1(r)};
      } else {
        exchange(j, __longlong_as_double((long long)pack2(lane0(X[0].h), lane0(X[0].l))),
                 __longlong_as_double((long long)pack2(lane1(X[P - 1].h), lane1(X[P - 1].l))), left, right);
        const f32x2 l = (f32x2)__double_as_longlong(left), r = (f32x2)__double_as_longlong(right);
        first = {pack2(lane0(l), lane0(X[P - 1].h)), pack2(lane1(l), lane0(X[P - 1].l))};
        last = {pack2(lane1(X[0].h), lane0(r)), pack2(lane1(X[0].l), lane1(r))};
      }
#pragma unroll
      for (int p = 0; p < P; ++p) {
        FPair<T> n[D];
        StageCoef<T> c = sc0;
        if constexpr (HET) {
          constexpr int S = MODEL == ROESSLER ? 6 : 4;
          c.kt = {spf[(p * S + 0) * blockDim.x], spf[(p * S + 1) * blockDim.x]};
          c.at = {spf[(p * S + 2) * blockDim.x], spf[(p * S + 3) * blockDim.x]};
        }
        if constexpr (PARK && MODEL == ROESSLER)
          base[p] = {{rb[p * 4], rb[p * 4 + 1]}, {rb[p * 4 + 2], rb[p * 4 + 3]}};
        split_stage<MODEL, T>(d[p], p == 0 ? first : X[p - 1], p == P - 1 ? last : X[p + 1], base[p], c, n);
#pragma unroll
        for (int i = 0; i < D; ++i) {
          if constexpr (PARK) {
            if (j < 3) k1[p][i] = {rp[(p * D + i) * 2], rp[(p * D + i) * 2 + 1]};
          }
          split_update<T>(j, k1[p][i], n[i], d[p][i], N[p][i]);
        }
      }
    }
    double six = 6.0, w = sc.w;
    if constexpr (kConst) ld_shared2(fc + 48, six, w);
#pragma unroll
    for (int p = 0; p < P; ++p)
#pragma unroll
      for (int i = 0; i < D; ++i) {
        double nd[2];
        join(N[p][i], nd, 1);
        if constexpr (PARK) {
          rec[p * D + i] = split_final(rec[p * D + i], rk[p * D + i], nd[0], six, w);
          rec[(p + P) * D + i] = split_final(rec[(p + P) * D + i], rk[(p + P) * D + i], nd[1], six, w);
        } else {
          y[p][i] = split_final(y[p][i], k1d[p][i], nd[0], six, w);
          if constexpr (V > 1) y[p + P][i] = split_final(y[p + P][i], k1d[p + P][i], nd[1], six, w);
        }
      }
  }
  if constexpr (PARK) {
#pragma unroll
    for (int v = 0; v < V; ++v)
#pragma unroll
      for (int i = 0; i < D; ++i) y[v][i] = rec[v * D + i];
  }
}

// Block-cooperative copies of `count` values between global and shared memory.
//
// copy_in_vec / copy_out_vec access global memory by 16-byte vectors wherever whole vectors
// lie inside the range, whatever the range's alignment: when the shared-memory side sits at the
// same 16-byte offset it is accessed by vectors too, otherwise each vector's values move to or
// from shared memory singly.  A vector that would reach past either end of the range is
// replaced by single accesses, so nothing outside the range is read or written.  The persistent
// kernel uses this form: its blocks load tiles in lock step after every grid barrier, and batch
// chains start anywhere, so single loads of misaligned windows sat on its critical path
// (measured 8 % faster with vectors).
//
// copy_out moves whole 16-byte vectors when both sides are aligned and the size is a
// multiple of 16 bytes (every tile of a single chain), single values otherwise.
template <typename R>
__device__ __forceinline__ void copy_out(R *__restrict__ dst, const R *src, int count) {
  if ((reinterpret_cast<uintptr_t>(dst) & 15u) == 0 && (reinterpret_cast<uintptr_t>(src) & 15u) == 0 &&
      ((count * (int)sizeof(R)) & 15) == 0) {
    const int nv = count * (int)sizeof(R) / 16;
    int4 *d4 = reinterpret_cast<int4 *>(dst);
    const int4 *s4 = reinterpret_cast<const int4 *>(src);
    for (int e = threadIdx.x; e < nv; e += blockDim.x) d4[e] = s4[e];
  } else {
    for (int e = threadIdx.x; e < count; e += blockDim.x) dst[e] = src[e];
  }
}
// copy_out for a range whose shared-memory side sits at the same 16-byte offset as its global
// side (the interior of a batch tile whose window starts on a 16-byte boundary): the values
// before the first and after the last whole vector singly, the rest by 16-byte vectors on both
// sides.  Any other range is copied singly.
template <typename R>
__device__ __forceinline__ void copy_out_matched(R *__restrict__ dst, const R *src, int count) {
  constexpr int kPer = 16 / (int)sizeof(R);
  const unsigned md = (unsigned)(reinterpret_cast<uintptr_t>(dst) & 15u);
  if (md != (unsigned)(reinterpret_cast<uintptr_t>(src) & 15u)) {
    for (int e = threadIdx.x; e < count; e += blockDim.x) dst[e] = src[e];
    return;
  }
  int head = (int)(((16u - md) & 15u) / sizeof(R));
  if (head > count) head = count;
  const int nv = (count - head) / kPer;
  for (int e = threadIdx.x; e < head; e += blockDim.x) dst[e] = src[e];
  int4 *d4 = reinterpret_cast<int4 *>(dst + head);
  const int4 *s4 = reinterpret_cast<const int4 *>(src + head);
  for (int e = threadIdx.x; e < nv; e += blockDim.x) d4[e] = s4[e];
  for (int e = head + nv * kPer + threadIdx.x; e < count; e += blockDim.x) dst[e] = src[e];
}

template <typename R>
__device__ __forceinline__ void copy_in_vec(R *dst, const R *__restrict__ src, int count) {
  constexpr int kPer = 16 / (int)sizeof(R);
  const unsigned ms = (unsigned)(reinterpret_cast<uintptr_t>(src) & 15u);
  int head = (int)(((16u - ms) & 15u) / sizeof(R));  // values before the first whole vector
  if (head > count) head = count;
  const int nv = (count - head) / kPer;
  for (int e = threadIdx.x; e < head; e += blockDim.x) dst[e] = __ldcg(src + e);
  const int4 *s4 = reinterpret_cast<const int4 *>(src + head);
  if (ms == (unsigned)(reinterpret_cast<uintptr_t>(dst) & 15u)) {
    int4 *d4 = reinterpret_cast<int4 *>(dst + head);
    for (int e = threadIdx.x; e < nv; e += blockDim.x) d4[e] = __ldcg(s4 + e);
  } else {
    for (int e = threadIdx.x; e < nv; e += blockDim.x) {
      const int4 w = __ldcg(s4 + e);
      const R *p = reinterpret_cast<const R *>(&w);
      R *d = dst + head + e * kPer;
#pragma unroll
      for (int q = 0; q < kPer; ++q) d[q] = p[q];
    }
  }
  for (int e = head + nv * kPer + threadIdx.x; e < count; e += blockDim.x) dst[e] = __ldcg(src + e);
}
template <typename R>
__device__ __forceinline__ void copy_out_vec(R *__restrict__ dst, const R *src, int count) {
  constexpr int kPer = 16 / (int)sizeof(R);
  const unsigned md = (unsigned)(reinterpret_cast<uintptr_t>(dst) & 15u);
  int head = (int)(((16u - md) & 15u) / sizeof(R));
  if (head > count) head = count;
  const int nv = (count - head) / kPer;
  for (int e = threadIdx.x; e < head; e += blockDim.x) dst[e] = src[e];
  int4 *d4 = reinterpret_cast<int4 *>(dst + head);
  if (md == (unsigned)(reinterpret_cast<uintptr_t>(src) & 15u)) {
    const int4 *s4 = reinterpret_cast<const int4 *>(src + head);
    for (int e = threadIdx.x; e < nv; e += blockDim.x) d4[e] = s4[e];
  } else {
    for (int e = threadIdx.x; e < nv; e += blockDim.x) {
      int4 w;
      R *p = reinterpret_cast<R *>(&w);
      const R *sp = src + head + e * kPer;
#pragma unroll
      for (int q = 0; q < kPer; ++q) p[q] = sp[q];
      d4[e] = w;
    }
  }
  for (int e = head + nv * kPer + threadIdx.x; e < count; e += blockDim.x) dst[e] = src[e];
}

// Asynchronous global-to-shared copies (cp.async): the data lands in shared memory while the
// issuing threads go on computing; cp_async_wait<N>() waits until at most the N most recently
// committed groups are still in flight (a hardware wait that always ends).
__device__ __forceinline__ void cp_async(void *smem, const void *g, int bytes) {
  const unsigned s = smem_addr(smem);
  const size_t ga = __cvta_generic_to_global(g);
  if (bytes == 16)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(s), "l"(ga) : "memory");
  else if (bytes == 8)
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(s), "l"(ga) : "memory");
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(s), "l"(ga) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// Copy into shared memory without waiting (tile_load_wait): 16-byte copies where both sides share
// their offset within a 16-byte line, single values otherwise; nothing outside the range is read.
// COH: nothing may come from L1, which copies of less than 16 bytes go through, so those values are
// loaded (and waited for) here.
template <bool COH, typename R>
__device__ __forceinline__ void copy_in_async(R *dst, const R *__restrict__ src, int count) {
  constexpr int kPer = 16 / (int)sizeof(R);
  const unsigned ms = (unsigned)(reinterpret_cast<uintptr_t>(src) & 15u);
  if (ms != (unsigned)(reinterpret_cast<uintptr_t>(dst) & 15u)) {
    if constexpr (COH) {
      copy_in_vec(dst, src, count);
    } else {
      for (int e = threadIdx.x; e < count; e += blockDim.x) cp_async(dst + e, src + e, (int)sizeof(R));
    }
    return;
  }
  auto one = [&](int e) {
    if constexpr (COH) dst[e] = __ldcg(src + e); else cp_async(dst + e, src + e, (int)sizeof(R));
  };
  int head = (int)(((16u - ms) & 15u) / sizeof(R));
  if (head > count) head = count;
  const int nv = (count - head) / kPer;
  for (int e = threadIdx.x; e < nv; e += blockDim.x) cp_async(dst + head + e * kPer, src + head + e * kPer, 16);
  if (head > 0)
    for (int e = threadIdx.x; e < head; e += blockDim.x) one(e);
  if (head + nv * kPer < count)
    for (int e = head + nv * kPer + threadIdx.x; e < count; e += blockDim.x) one(e);
}

// Copy the W sites starting at chain index t0 (may be negative or run past the end) of the
// chain at `off` into shared memory, coalesced.  Periodic: wrapped; fixed: zero outside the
// chain.  A tile that crosses a chain end is copied as a few contiguous segments (one index
// wrap per segment, not per element): at most 2 for chains longer than the tile, N / W + 2
// for shorter periodic chains.
// The copies are asynchronous: tile_load_wait (or a commit and a later wait) before the barrier that
// precedes their use.  Loads into registers and on to shared memory, three 16-byte vectors per
// thread and array one after the other, took a block 9700 cycles a tile beside 5000 of arithmetic
// (FP32, 256 x 4 x 4, four resident blocks), with these 5100; N = 2^24, site-steps/s before -> after:
// FP32 256 x 4 x 4 2.77e11 -> 3.56e11, x 8 4.04e11 -> 4.31e11, x 16 4.53e11 -> 4.55e11, persistent x 8
// 3.65e11 -> 3.94e11; FP64 256 x 4 x 1 2.71e10 -> 3.07e10, x 2 3.27e10 -> 3.43e10.
template <typename R, int D, bool COH>
__device__ __forceinline__ void tile_load(R *tile, const R *__restrict__ src, int64_t off, int64_t n, int bc,
                                          int64_t t0, int W, int64_t sites, WsHeader *hdr) {
  const int total = W * D;
  if (t0 >= 0 && t0 + W <= n) {
    if (!bounds_ok(hdr, in_range(off + t0, W, sites))) return;
    copy_in_async<COH>(tile, src + (off + t0) * D, total);
    return;
  }
  int covered = 0;  // block-uniform loop over contiguous segments
  while (covered < W) {
    const int64_t g = t0 + covered;
    const int64_t rest = W - covered;
    int len;
    const R *seg = nullptr;  // NULL: a run of fixed-end ghosts (zeros)
    if (bc == PERIODIC) {
      const int64_t gw = wrap(g, n);
      len = (int)(rest < n - gw ? rest : n - gw);
      seg = src + (off + gw) * D;
    } else if (g < 0) {
      len = (int)(rest < -g ? rest : -g);
    } else if (g >= n) {
      len = (int)rest;
    } else {
      len = (int)(rest < n - g ? rest : n - g);
      seg = src + (off + g) * D;
    }
    R *dst = tile + covered * D;
    const int cnt = len * D;
    if (seg && !bounds_ok(hdr, in_range(seg - src, cnt, sites * D))) seg = nullptr;
    if (seg) {
      copy_in_async<COH>(dst, seg, cnt);
    } else {
      for (int e = threadIdx.x; e < cnt; e += blockDim.x) dst[e] = R(0);
    }
    covered += len;
  }
}

__device__ __forceinline__ void tile_load_wait() {
  cp_async_commit();
  cp_async_wait<0>();
}

// Store `cnt` sites of the tile starting at tile-local site `first` to chain index g0 (VEC:
// copy_out_vec, for the persistent kernel; MATCHED: copy_out_matched, for tiles whose window
// starts on a 16-byte boundary).
template <typename R, int D, bool VEC = false, bool MATCHED = false>
__device__ __forceinline__ void tile_store(R *__restrict__ dst, const R *tile, int64_t off, int first, int64_t g0,
                                           int cnt, int64_t sites, int W, WsHeader *hdr) {
  if (!bounds_ok(hdr, in_range(off + g0, cnt, sites) && in_range(first, cnt, W))) return;
  if constexpr (MATCHED) copy_out_matched(dst + (off + g0) * D, tile + first * D, cnt * D);
  else if constexpr (VEC) copy_out_vec(dst + (off + g0) * D, tile + first * D, cnt * D);
  else copy_out(dst + (off + g0) * D, tile + first * D, cnt * D);
}

// Sites per 16 bytes of a [sites][D] array of R, in whole sites (16 / gcd(16, D sizeof(R))).
template <typename R, int D> __host__ __device__ constexpr int align_sites() {
  int a = D * (int)sizeof(R), b = 16;
  while (b) {
    const int t = a % b;
    a = b;
    b = t;
  }
  return 16 / a;
}

// What a tile (or a packed tile's segment) holds, as far as the split form asks, in the bits of a thread's
// sites OR-ed over it.
enum : int {
  kSplitWide = 1,    // a stored value that is not zero and out of range
  kSplitLive = 2,    // a value that is not NaN
  kSplitGap = 4,     // two neighbouring sites that are all zero
  kSplitSome = 8,    // a value that is not zero
  kSplitZero = 16,   // (<< d) a stored value of component d that is zero
  kSplitValue = 128  // (<< d) one anywhere that is not
};
__device__ __forceinline__ bool split_has_front(int b) {  // zeros and nonzero values, of one component
  return ((b / kSplitZero) & (b / kSplitValue) & 7) != 0;
}
// The bits of the thread's sites that are not ghosts.  c(v): the site's own c or NULL; stored(v): whether it is
// stored (of the loaded tile, all are); next: the state of the site after the thread's last one, or NULL.
template <int MODEL, int V, typename C, typename S>
__device__ __forceinline__ int split_tile_bits(const double (&y)[V][Dim<MODEL>::D], uint32_t ghost, const SplitCoef &sc,
                                               const double *next, C &&c, S &&stored) {
  constexpr int D = Dim<MODEL>::D;
  int b = 0;
  bool before = false;  // the site before is all zero
#pragma unroll
  for (int v = 0; v < V; ++v) {
    const bool real = !((ghost >> v) & 1u);
    bool rest = real;
#pragma unroll
    for (int d = 0; d < D; ++d) {
      if (is_zero(y[v][d])) {
        if (real && stored(v)) b |= kSplitZero << d;
      } else {
        rest = false;
        if (real) b |= kSplitSome | (kSplitValue << d);
        if (real && stored(v) && !split_holds<MODEL>(y[v][d], d, c(v), sc)) b |= kSplitWide;
      }
      if (real && !is_nan(y[v][d])) b |= kSplitLive;
    }
    if (rest && before) b |= kSplitGap;
    before = rest;
  }
  if (before && next) {
    bool rest = true;
#pragma unroll
    for (int d = 0; d < D; ++d) rest = rest && is_zero(next[d]);
    if (rest) b |= kSplitGap;
  }
  return b;
}
// The bits of all threads of the block; word: shared memory that nothing else uses meanwhile.
__device__ __forceinline__ int block_or(int b, int *word) {
  if (threadIdx.x == 0) *word = 0;
  __syncthreads();
  b = __reduce_or_sync(kFull, b);
  if (b && (threadIdx.x & 31) == 0) atomicOr(word, b);
  __syncthreads();
  b = *word;
  __syncthreads();
  return b;
}

// OR b into the word of the thread's segment (NULL: none); one access a warp where its threads share it.
__device__ __forceinline__ void segment_or(int b, int *word) {
  const unsigned long long w = (unsigned long long)word;
  if (__all_sync(kFull, w == __shfl_sync(kFull, w, 0))) {
    b = __reduce_or_sync(kFull, b);
    if (threadIdx.x & 31) return;
  }
  if (word && b) atomicOr(word, b);
}

// Process one (chain, tile) item end to end: load, advance K steps, store the interior.
// ALN (batch tiles): the window starts at the last multiple of align_sites() at or before
// tile G - H in the state array, so it moves by whole 16-byte vectors wherever the chain
// starts; the left halo is then H .. H + A - 1 sites, and the host shrinks G by A - 1 so that
// the right halo keeps at least H.
// Shared memory: edge[edge_values(V)] | tile[W*D] | ctile[W*D] (Kahan) | ptile[W*P]
// (heterogeneous).
// `sites` is the number of sites in the state buffers (for the debug bounds checks); hdr the
// status word, where a non-finite stored value is reported.
// SPLIT (FP64): the split form of the step.  Returns false, with nothing stored, when a value the
// tile loads or would store (or a site's own parameter) is outside the split's range: the caller
// then runs the item again in the FP64 form.  True otherwise; the same for every thread.  PARK: the
// threads' records (split_advance) take the tile's place in shared memory while it is advanced.
template <typename R, int MODEL, int V, bool KAHAN, bool COH, bool HET = false, bool ALN = false, bool SPLIT = false,
          bool PARK = false>
__device__ __forceinline__ bool tile_item(const R *__restrict__ in, R *__restrict__ out, const R *__restrict__ cin,
                                          R *__restrict__ cout, const ChainDesc &ch, int64_t tile, int K, int G,
                                          const Coef<R> &cf, unsigned char *smem, int64_t sites, WsHeader *hdr,
                                          const R *__restrict__ sp = nullptr, const SplitCoef *sc = nullptr) {
  constexpr int D = Dim<MODEL>::D;
  constexpr int P = Dim<MODEL>::P;
  R *edge = reinterpret_cast<R *>(smem);
  const int W = blockDim.x * V;
  const int H = 4 * K;
  const int64_t g0 = tile * (int64_t)G;  // first interior site
  int64_t t0 = g0 - H;
  if constexpr (ALN) {
    constexpr int A = align_sites<R, D>();
    const int64_t a = ch.off + t0;  // rounded down (toward minus infinity) to a multiple of A
    t0 = (a >= 0 ? a / A : -((-a + A - 1) / A)) * A - ch.off;
  }
  const int hl = (int)(g0 - t0);  // left halo: H, or up to A - 1 sites more with ALN
  R *tl = edge + edge_values(V);
  R *ctl = tl + W * D;
  R *ptl = ctl + (KAHAN ? W * D : 0);

  tile_load<R, D, COH>(tl, in, ch.off, ch.n, ch.bc, t0, W, sites, hdr);
  if constexpr (KAHAN) tile_load<R, D, COH>(ctl, cin, ch.off, ch.n, ch.bc, t0, W, sites, hdr);
  if constexpr (HET) tile_load<R, P, COH>(ptl, sp, ch.off, ch.n, ch.bc, t0, W, sites, hdr);
  tile_load_wait();
  __syncthreads();

  R y[V][D], cmp[V][D];
  const int base = threadIdx.x * V;
#pragma unroll
  for (int v = 0; v < V; ++v)
#pragma unroll
    for (int d = 0; d < D; ++d) {
      y[v][d] = tl[(base + v) * D + d];
      if constexpr (KAHAN) cmp[v][d] = ctl[(base + v) * D + d]; else cmp[v][d] = R(0);
    }

  // fixed ends: the thread's sites outside the chain (ghosts)
  const bool edge_tile = (ch.bc == FIXED) && (t0 < 0 || t0 + W > ch.n);
  uint32_t ghost = 0;
  if (edge_tile) {
#pragma unroll
    for (int v = 0; v < V; ++v) {
      const int64_t g = t0 + base + v;
      if (g < 0 || g >= ch.n) ghost |= 1u << v;
    }
  }
  bool nan_tile = false;  // SPLIT: every value is NaN already (a chain that has blown up), and stays so
  if constexpr (SPLIT) {
    double *spd = nullptr;
    f32x2 *spf = nullptr;
    auto own_c = [&](int v) -> const double * { return HET && MODEL == ROESSLER ? &ptl[(base + v) * P + 2] : nullptr; };
    bool odd = false, out = false;  // a value that is zero or out of range; a parameter out of range
#pragma unroll
    for (int v = 0; v < V; ++v)
#pragma unroll
      for (int d = 0; d < D; ++d) odd |= !((ghost >> v) & 1u) && !split_holds<MODEL>(y[v][d], d, own_c(v), *sc);
    if constexpr (HET) {
#pragma unroll
      for (int v = 0; v < V; ++v)
#pragma unroll
        for (int i = 0; i < P; ++i) out |= !split_param_in_range(ptl[(base + v) * P + i], sc->most[i]);
    }
    if (__syncthreads_or(odd | out)) {
      const int last = base + V;  // the next thread's first site, if it is the chain's
      const bool next = last < W && (!edge_tile || (t0 + last >= 0 && t0 + last < ch.n));
      int b = split_tile_bits<MODEL, V>(y, ghost, *sc, next ? tl + last * D : nullptr, own_c, [](int) { return true; });
      if (out) b |= kSplitWide | kSplitLive;
      b = block_or(b, reinterpret_cast<int *>(smem));
      nan_tile = (b & kSplitWide) && !(b & kSplitLive);
      if (!nan_tile && ((b & kSplitWide) || ((b & kSplitGap) && (b & kSplitSome)))) return false;
    }
    if constexpr (HET) {
      // the parameters move to thread-private slots (consecutive threads, consecutive addresses),
      // beside the pair coefficients of each pair of sites
      constexpr int S = MODEL == ROESSLER ? 6 : 4;
      double p[V][P];
#pragma unroll
      for (int v = 0; v < V; ++v)
#pragma unroll
        for (int i = 0; i < P; ++i) p[v][i] = ptl[(base + v) * P + i];
      __syncthreads();
      spd = ptl + threadIdx.x;
      spf = reinterpret_cast<f32x2 *>(ptl + W * P) + threadIdx.x;
#pragma unroll
      for (int v = 0; v < V; ++v)
#pragma unroll
        for (int i = 0; i < P; ++i) spd[(v * P + i) * blockDim.x] = p[v][i];
#pragma unroll
      for (int q = 0; q < V / 2; ++q) {
        const FPair<float> k0 = times_tau(p[q][P - 1], *sc), k1 = times_tau(p[q + V / 2][P - 1], *sc);
        const FPair<float> a0 = times_tau(p[q][0], *sc), a1 = times_tau(p[q + V / 2][0], *sc);
        f32x2 *o = spf + q * S * blockDim.x;
        o[0] = pack2(k0.h, k1.h);
        o[blockDim.x] = pack2(k0.l, k1.l);
        o[2 * blockDim.x] = pack2(a0.h, a1.h);
        o[3 * blockDim.x] = pack2(a0.l, a1.l);
        if constexpr (MODEL == ROESSLER) {
          const FPair<float> c0 = split1(p[q][2]), c1 = split1(p[q + V / 2][2]);
          o[4 * blockDim.x] = pack2(c0.h, c1.h);
          o[5 * blockDim.x] = pack2(c0.l, c1.l);
        }
      }
    }
    double *rec = nullptr;
    if constexpr (PARK) rec = tl + threadIdx.x * split_record_words<MODEL, V>();
    if (edge_tile) split_advance<MODEL, V, true, HET, PARK>(y, ghost, K, cf, *sc, edge, spd, spf, rec);
    else split_advance<MODEL, V, false, HET, PARK>(y, 0u, K, cf, *sc, edge, spd, spf, rec);
    if constexpr (PARK) __syncthreads();  // every record is read before the tile is written over them
  } else {
    Coef<R> cs[HET ? V : 1];
    if constexpr (HET) {
#pragma unroll
      for (int v = 0; v < V; ++v) cs[v] = site_coef<R, MODEL>(cf, ptl + (base + v) * P);
    }
    if (edge_tile) tile_advance<R, MODEL, V, KAHAN, true, HET>(y, cmp, ghost, K, cf, edge, cs);
    else tile_advance<R, MODEL, V, KAHAN, false, HET>(y, cmp, 0u, K, cf, edge, cs);
  }

  const int64_t rem = ch.n - g0;
  const int cnt = (int)(rem < G ? rem : G);
  bool bad = false;  // a stored (interior) value is NaN or infinite (SPLIT: zero or out of range)
  auto own_c = [&](int v) -> const R * { return HET && MODEL == ROESSLER ? &ptl[(v * P + 2) * blockDim.x + threadIdx.x] : nullptr; };
  auto stored_site = [&](int v) { return base + v >= hl && base + v < hl + cnt; };
#pragma unroll
  for (int v = 0; v < V; ++v) {
    const bool stored = stored_site(v);
#pragma unroll
    for (int d = 0; d < D; ++d) {
      tl[(base + v) * D + d] = y[v][d];
      if constexpr (KAHAN) ctl[(base + v) * D + d] = cmp[v][d];
      if constexpr (SPLIT) {
        bad |= stored && !split_holds<MODEL>(y[v][d], d, own_c(v), *sc);
      } else {
        bad |= stored && nonfinite(y[v][d]);
      }
    }
  }
  const int any_bad = __syncthreads_or(bad);
  if constexpr (SPLIT) {
    if (any_bad && !nan_tile) {
      const int b = block_or(split_tile_bits<MODEL, V>(y, ghost, *sc, nullptr, own_c, stored_site), reinterpret_cast<int *>(smem));
      if ((b & kSplitWide) || split_has_front(b)) return false;
    }
    report_nonfinite(hdr, nan_tile);
  } else {
    report_nonfinite(hdr, any_bad);
  }
  if (cnt > 0) {
    tile_store<R, D, COH, ALN>(out, tl, ch.off, hl, g0, cnt, sites, W, hdr);
    if constexpr (KAHAN) tile_store<R, D, COH, ALN>(cout, ctl, ch.off, hl, g0, cnt, sites, W, hdr);
  }
  __syncthreads();  // shared memory is reused by the next item
  return true;
}

// Process one packed tile: segments s0 .. s1 - 1 of `segs`, side by side in slot order, each a
// window [g0 - H, g0 + cnt + H + pad) of its own chain (wrapped or zero outside the chain like a
// plain tile).  The neighbour exchange runs across segment borders as if the tile were one
// chain: a wrong neighbour at a border, like a missing one at a tile end, spoils one more site
// per stage, so after K steps only each segment's H-site halos are spoilt and its cnt interior
// sites are exact.  Every thread's sites lie in one segment (o and L are multiples of V), so a
// thread takes its chain's coupling strength and, for fixed ends, its ghost mask; threads past
// the last segment advance zeros that are never stored.
// SPLIT, PARK: as tile_item, but each segment leaves the split form by itself, so that a chain's result does
// not depend on the chains it shares a tile with: the segments that do are not stored but marked in the
// exchange's memory (a word each: a tile has at most 2048 / 10 segments with two sites per thread, 1024 / 9
// with one, and the exchange 256 words or more), and the result is false when there are any.  FLAGGED (the
// FP64 form after that): only the marked segments are stored.
template <typename R, int MODEL, int V, bool KAHAN, bool COH, bool SPLIT = false, bool PARK = false, bool FLAGGED = false>
__device__ __forceinline__ bool packed_tile_item(const R *__restrict__ in, R *__restrict__ out,
                                                 const R *__restrict__ cin, R *__restrict__ cout,
                                                 const ChainDesc *chains, const SegDesc *segs, int s0, int s1,
                                                 int K, const Coef<R> &cf, unsigned char *smem, int64_t sites,
                                                 WsHeader *hdr, const SplitCoef *scp = nullptr) {
  constexpr int D = Dim<MODEL>::D;
  R *edge = reinterpret_cast<R *>(smem);
  R *tl = edge + edge_values(V);
  const int W = blockDim.x * V;
  R *ctl = tl + W * D;
  const int H = 4 * K;
  int *flag = reinterpret_cast<int *>(smem);

  int used = 0;  // slots covered by the segments (they are in slot order)
  for (int s = s0; s < s1; ++s) {
    const SegDesc sd = segs[s];
    if (!bounds_ok(hdr, sd.o >= used && sd.L >= 0 && sd.o + sd.L <= W)) continue;
    const ChainDesc ch = chains[sd.chain];
    tile_load<R, D, COH>(tl + sd.o * D, in, ch.off, ch.n, ch.bc, sd.g0 - H, sd.L, sites, hdr);
    if constexpr (KAHAN) tile_load<R, D, COH>(ctl + sd.o * D, cin, ch.off, ch.n, ch.bc, sd.g0 - H, sd.L, sites, hdr);
    used = sd.o + sd.L;
  }
  for (int e = used * D + threadIdx.x; e < W * D; e += blockDim.x) {
    tl[e] = R(0);
    if constexpr (KAHAN) ctl[e] = R(0);
  }
  tile_load_wait();
  __syncthreads();

  // this thread's segment: the last one starting at or before its first slot
  const int base = threadIdx.x * V;
  int my = -1;
  if (s1 > s0) {
    int lo = s0, hi = s1 - 1;
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (segs[mid].o <= base) lo = mid; else hi = mid - 1;
    }
    if (segs[lo].o <= base && base < segs[lo].o + segs[lo].L) my = lo;
  }
  Coef<R> c = cf;
  uint32_t ghost = 0;
  int rel = 0, cnt = 0;  // first site's position in the segment's window; the segment's interior sites
  if (my >= 0) {
    const SegDesc sd = segs[my];
    const ChainDesc ch = chains[sd.chain];
    c.kappa = (R)ch.kappa;
    rel = base - sd.o;
    cnt = sd.cnt;
    if (ch.bc == FIXED) {
#pragma unroll
      for (int v = 0; v < V; ++v) {
        const int64_t g = sd.g0 - H + rel + v;
        if (g < 0 || g >= ch.n) ghost |= 1u << v;
      }
    }
  }

  R y[V][D], cmp[V][D];
#pragma unroll
  for (int v = 0; v < V; ++v)
#pragma unroll
    for (int d = 0; d < D; ++d) {
      y[v][d] = tl[(base + v) * D + d];
      if constexpr (KAHAN) cmp[v][d] = ctl[(base + v) * D + d]; else cmp[v][d] = R(0);
    }
  bool wide = false, all_nan = false;  // SPLIT: this thread's segment leaves the form; is NaN and nothing else
  auto own_c = [](int) -> const double * { return nullptr; };
  auto stored_site = [&](int v) { return my >= 0 && rel + v >= H && rel + v < H + cnt; };
  bool mine = true;                    // FLAGGED: the segment is stored
  if constexpr (FLAGGED) {
    mine = my >= 0 && flag[my - s0] != 0;
    __syncthreads();  // before the exchange writes there
  }
  if constexpr (SPLIT) {
    bool odd = false;  // a value that is zero or out of range
#pragma unroll
    for (int v = 0; v < V; ++v)
#pragma unroll
      for (int d = 0; d < D; ++d)
        odd |= my >= 0 && !((ghost >> v) & 1u) && !split_holds<MODEL>(y[v][d], d, nullptr, *scp);
    if (__syncthreads_or(odd)) {
      for (int s = threadIdx.x; s < s1 - s0; s += blockDim.x) flag[s] = 0;
      __syncthreads();
      int b = 0;
      if (my >= 0) {
        const int last = base + V;  // the next thread's first site, if it is the segment's and the chain's
        bool next = last < segs[my].o + segs[my].L;
        if (next && chains[segs[my].chain].bc == FIXED) {
          const int64_t g = segs[my].g0 - H + rel + V;
          next = g >= 0 && g < chains[segs[my].chain].n;
        }
        b = split_tile_bits<MODEL, V>(y, ghost, *scp, next ? tl + last * D : nullptr, own_c, [](int) { return true; });
      }
      segment_or(b, my >= 0 ? &flag[my - s0] : nullptr);
      __syncthreads();
      if (my >= 0) {
        b = flag[my - s0];
        all_nan = (b & kSplitWide) && !(b & kSplitLive);
        wide = !all_nan && ((b & kSplitWide) || ((b & kSplitGap) && (b & kSplitSome)));
      }
      if (!__syncthreads_or(my >= 0 && !wide)) return false;  // every segment is marked
    }
    SplitCoef sc = *scp;
    split_set_kappa(sc, c.kappa);
    double *rec = nullptr;
    if constexpr (PARK) rec = tl + threadIdx.x * split_record_words<MODEL, V>();
    split_advance<MODEL, V, true, false, PARK, true>(y, ghost, K, c, sc, edge, nullptr, nullptr, rec);
    if constexpr (PARK) __syncthreads();
  } else {
    tile_advance<R, MODEL, V, KAHAN, true>(y, cmp, ghost, K, c, edge);
  }

  bool bad = false;  // a stored (interior) value is NaN or infinite (SPLIT: zero or out of range)
#pragma unroll
  for (int v = 0; v < V; ++v) {
    const bool stored = stored_site(v);
#pragma unroll
    for (int d = 0; d < D; ++d) {
      tl[(base + v) * D + d] = y[v][d];
      if constexpr (KAHAN) ctl[(base + v) * D + d] = cmp[v][d];
      if constexpr (SPLIT) bad |= stored && !split_holds<MODEL>(y[v][d], d, nullptr, *scp);
      else bad |= stored && mine && nonfinite(y[v][d]);
    }
  }
  int any = __syncthreads_or(bad | wide);
  bool marked = FLAGGED;  // the words say which segments to leave out (SPLIT) or to store (FLAGGED)
  if constexpr (SPLIT) {
    if (any) {
      for (int s = threadIdx.x; s < s1 - s0; s += blockDim.x) flag[s] = 0;
      __syncthreads();
      segment_or(my >= 0 ? split_tile_bits<MODEL, V>(y, ghost, *scp, nullptr, own_c, stored_site) : 0,
                 my >= 0 ? &flag[my - s0] : nullptr);
      __syncthreads();
      if (my >= 0 && !all_nan) wide |= (flag[my - s0] & kSplitWide) || split_has_front(flag[my - s0]);
      report_nonfinite(hdr, __syncthreads_or(all_nan));
      any = __syncthreads_or(wide);
    }
    if (any) {
      marked = true;
      for (int s = threadIdx.x; s < s1 - s0; s += blockDim.x) flag[s] = 0;
      __syncthreads();
      if (wide) flag[my - s0] = 1;
      __syncthreads();
    }
  } else {
    report_nonfinite(hdr, any);
    if constexpr (FLAGGED) {
      if (my >= 0 && base == segs[my].o) flag[my - s0] = mine;
      __syncthreads();
    }
  }
  for (int s = s0; s < s1; ++s) {
    const SegDesc sd = segs[s];
    if (sd.cnt <= 0 || !bounds_ok(hdr, sd.o >= 0 && sd.o + sd.L <= W && sd.cnt + 2 * H <= sd.L)) continue;
    if (marked && (flag[s - s0] != 0) != FLAGGED) continue;
    const ChainDesc ch = chains[sd.chain];
    tile_store<R, D, COH>(out, tl, ch.off, sd.o + H, sd.g0, sd.cnt, sites, W, hdr);
    if constexpr (KAHAN) tile_store<R, D, COH>(cout, ctl, ch.off, sd.o + H, sd.g0, sd.cnt, sites, W, hdr);
  }
  __syncthreads();  // shared memory is reused by the next item
  return !SPLIT || !any;
}

// The chain of site i of the state (the last one that starts at or before it).
__device__ __forceinline__ int site_chain(const ChainDesc *chains, int nchains, int64_t i) {
  int lo = 0, hi = nchains - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (chains[mid].off <= i) lo = mid; else hi = mid - 1;
  }
  return lo;
}

// Locate the chain of a tile index through the prefix array (first tile of each chain).
__device__ __forceinline__ int find_chain(const int32_t *prefix, int nchains, int64_t tile) {
  int lo = 0, hi = nchains - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (prefix[mid] <= tile) lo = mid; else hi = mid - 1;
  }
  return lo;
}

// find_chain by one warp: each round the 32 lanes test 32 evenly spaced candidates at once and
// the range shrinks 32-fold, so 4096 chains take three rounds of loads instead of twelve
// dependent ones.  Call with all 32 lanes of a warp; every lane returns the answer.
__device__ __forceinline__ int find_chain_warp(const int32_t *prefix, int nchains, int64_t tile) {
  const int lane = threadIdx.x & 31;
  int lo = 0, hi = nchains - 1;  // the answer (largest c with prefix[c] <= tile) lies in [lo, hi]
  while (hi > lo) {
    const int step = (hi - lo + 32) / 32;  // ceil((hi - lo + 1) / 32)
    const int c = lo + lane * step;
    const unsigned ok = __ballot_sync(kFull, c <= hi && prefix[c] <= tile);
    const int last = 31 - __clz(ok);  // lane 0's candidate, lo, always qualifies
    lo += last * step;
    hi = min(hi, lo + step - 1);
  }
  return lo;
}

// The chain of a batch tile, found once per block: the first warp searches (find_chain_warp)
// and passes the answer to the others through the first word of the block's shared memory (the
// neighbour-exchange area, which the tile kernels first write after the barrier that ends
// their tile load, when every thread has read the answer).
__device__ __forceinline__ int find_chain_block(const int32_t *prefix, int nchains, int64_t tile,
                                                unsigned char *smem) {
  int *slot = reinterpret_cast<int *>(smem);
  if (threadIdx.x < 32) {
    const int c = find_chain_warp(prefix, nchains, tile);
    if (threadIdx.x == 0) *slot = c;
  }
  __syncthreads();
  return *slot;
}

// Chain and chain-local tile index of full tile f of a batch launch: one load from the tile
// table when the launch has one, else the block's search of the first-tile prefix.  Every
// thread of the block calls it and gets the same answer.
__device__ __forceinline__ int batch_chain(const BatchTiles &bt, int nchains, int64_t f, unsigned char *smem,
                                           int64_t &local) {
  if (bt.tile_chain) {
    const int2 tc = __ldg(&bt.tile_chain[f]);
    local = tc.y;
    return tc.x;
  }
  const int ci = find_chain_block(bt.full_prefix, nchains, f, smem);
  local = f - bt.full_prefix[ci];
  return ci;
}

template <typename R> __host__ __device__ inline Coef<R> to_coef(const CoefD &c, double kappa) {
  Coef<R> r;
  r.a = (R)c.a; r.b = (R)c.b; r.c = (R)c.c; r.kappa = (R)kappa; r.w2 = (R)c.w2;
  r.h2 = (R)c.h2; r.h1 = (R)c.h1; r.dt6 = (R)c.dt6; r.dt3 = (R)c.dt3; r.one = R(1);
  return r;
}

}  // namespace rk4d
