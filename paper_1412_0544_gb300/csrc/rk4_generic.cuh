// rk4_generic.cuh -- per-site arithmetic of the generic explicit Runge-Kutta scheme (any
// tableau of up to kMaxStages stages, coupling range 1 or 2).  Shared by the staged and the
// blocked generic kernels so that both perform the same operations in the same order.
#pragma once
#include "rk4_tile.cuh"

namespace rk4d {

// Largest block of the generic tile kernel (it keeps every stage slope of every site in
// registers, so the register budget of a block decides): 512 threads for FP32 with two sites
// per thread or a compiled tableau shape (at most 128 registers per thread), 256 otherwise.
template <typename R, int V, uint64_t SHAPE> struct GenBounds {
  static constexpr int threads = (sizeof(R) == 4 && (SHAPE != 0 || V == 2)) ? 512 : 256;
};
// Shared-memory values of the generic tile kernel's neighbour exchange: 2 parities x 2 pairs
// of coupling coordinates per thread of the largest block any instantiation allows.
constexpr int kGenEdgeThreads = 512;
__host__ __device__ constexpr int gen_edge_values(int v) { return (void)v, 2 * 4 * kGenEdgeThreads; }

// The tableau in the working precision: a_jm dt and b_m dt rounded once on the host, plus
// bit masks of the nonzero entries (zero entries are skipped, in every kernel alike).
template <typename R> struct Tableau {
  int s;
  R adt[kMaxStages][kMaxStages];
  R bdt[kMaxStages];
  uint32_t anz[kMaxStages];
  uint32_t bnz;
};

// The nonzero pattern of a tableau ("shape") packed into one word, for kernels compiled for a
// fixed tableau: the stage count in bits 0-2, a_jm (m < j) at bit 3 + j (j - 1) / 2 + m, b_m
// at bit 24 + m.  SHAPE = 0 reads the pattern from the tableau at run time.  Either way the
// same zero entries are skipped, so both forms perform the same operations.
__host__ __device__ constexpr uint64_t shape_a_bit(int j, int m) { return 1ull << (3 + j * (j - 1) / 2 + m); }
__host__ __device__ constexpr uint64_t shape_b_bit(int m) { return 1ull << (24 + m); }
// Stages of a compiled shape that the result needs (bit m set): nonzero weight, or used by a
// needed later stage.  The others are skipped outright, exchange included.
__host__ __device__ constexpr uint32_t shape_needed(uint64_t shape) {
  const int s = (int)(shape & 7u);
  uint32_t need = 0;
  for (int m = 0; m < s; ++m)
    if (shape & shape_b_bit(m)) need |= 1u << m;
  for (int j = s - 1; j >= 0; --j)
    if ((need >> j) & 1u)
      for (int m = 0; m < j; ++m)
        if (shape & shape_a_bit(j, m)) need |= 1u << m;
  return need;
}
template <uint64_t SHAPE> __device__ __forceinline__ constexpr bool gen_stage_needed(int j) {
  if constexpr (SHAPE != 0) return (shape_needed(SHAPE) >> j) & 1u; else return true;
}
template <uint64_t SHAPE, typename R> __device__ __forceinline__ int gen_stages(const Tableau<R> &tb) {
  if constexpr (SHAPE != 0) return (int)(SHAPE & 7u); else return tb.s;
}
template <uint64_t SHAPE, typename R> __device__ __forceinline__ bool gen_a_nonzero(const Tableau<R> &tb, int j, int m) {
  if constexpr (SHAPE != 0) return (SHAPE & shape_a_bit(j, m)) != 0; else return (tb.anz[j] >> m) & 1u;
}
template <uint64_t SHAPE, typename R> __device__ __forceinline__ bool gen_b_nonzero(const Tableau<R> &tb, int m) {
  if constexpr (SHAPE != 0) return (SHAPE & shape_b_bit(m)) != 0; else return (tb.bnz >> m) & 1u;
}

// The nonzero pattern of a tableau (see shape_a_bit): the key of the compiled shapes.
inline uint64_t tableau_shape(const TableauD &t) {
  uint64_t sh = (uint64_t)t.s & 7u;
  for (int j = 1; j < t.s; ++j)
    for (int m = 0; m < j; ++m)
      if (t.a[j][m] != 0.0) sh |= shape_a_bit(j, m);
  for (int m = 0; m < t.s; ++m)
    if (t.b[m] != 0.0) sh |= shape_b_bit(m);
  return sh;
}

// Shapes with tile kernels compiled for them (4 sites per thread): the classical RK4 tableau
// (the generic kernel runs it with second-neighbour coupling) and Dormand-Prince 5 (7 stages,
// a_61 = 0, b_1 = b_6 = 0).  Other tableaux run the kernel that reads the pattern at run time.
constexpr uint64_t kShapeRK4 = 4u | shape_a_bit(1, 0) | shape_a_bit(2, 1) | shape_a_bit(3, 2) | shape_b_bit(0) |
                               shape_b_bit(1) | shape_b_bit(2) | shape_b_bit(3);
constexpr uint64_t kShapeDopri5 =
    7u | shape_a_bit(1, 0) | shape_a_bit(2, 0) | shape_a_bit(2, 1) | shape_a_bit(3, 0) | shape_a_bit(3, 1) |
    shape_a_bit(3, 2) | shape_a_bit(4, 0) | shape_a_bit(4, 1) | shape_a_bit(4, 2) | shape_a_bit(4, 3) |
    shape_a_bit(5, 0) | shape_a_bit(5, 1) | shape_a_bit(5, 2) | shape_a_bit(5, 3) | shape_a_bit(5, 4) |
    shape_a_bit(6, 0) | shape_a_bit(6, 2) | shape_a_bit(6, 3) | shape_a_bit(6, 4) | shape_a_bit(6, 5) |
    shape_b_bit(0) | shape_b_bit(2) | shape_b_bit(3) | shape_b_bit(4) | shape_b_bit(5);

// Eq. (4): stage state of stage j from the step's start y and the earlier slopes.
template <typename R, int D, uint64_t SHAPE = 0>
__device__ __forceinline__ void gen_stage_state(int j, const Tableau<R> &tb, const R *y, const R (*k)[D], R *u) {
#pragma unroll
  for (int d = 0; d < D; ++d) u[d] = y[d];
#pragma unroll
  for (int m = 0; m < kMaxStages; ++m) {
    if (m < j && gen_a_nonzero<SHAPE>(tb, j, m)) {
#pragma unroll
      for (int d = 0; d < D; ++d) u[d] = fma(tb.adt[j][m], k[m][d], u[d]);
    }
  }
}

// Eq. (3) with coupling range 1 (the RK4 kernels' slope) or 2 (second neighbours added
// inside the coupling term).
template <typename R, int MODEL, int RANGE>
__device__ __forceinline__ void slope_gen(const R *u, R xl, R xr, R xl2, R xr2, const Coef<R> &cf, R kappa2,
                                          R *k) {
  if constexpr (RANGE == 1) {
    slope<R, MODEL>(u, xl, xr, cf, k);
  } else {
    constexpr bool kFmaAdd = sizeof(R) == 8;  // FP64: additions as DFMA (see Coef::one)
    const R lap = fma(R(-2), u[0], kFmaAdd ? fma(xl, cf.one, xr) : add(xl, xr));
    const R lap2 = fma(R(-2), u[0], kFmaAdd ? fma(xl2, cf.one, xr2) : add(xl2, xr2));
    if constexpr (MODEL == ROESSLER) {
      k[0] = fma(cf.kappa, lap, fma(kappa2, lap2, -(kFmaAdd ? fma(u[1], cf.one, u[2]) : add(u[1], u[2]))));
      k[1] = fma(cf.a, u[1], u[0]);
      if constexpr (sizeof(R) == 8)
        k[2] = fma(u[2], u[0], fma(-cf.c, u[2], cf.b));  // as slope(): two DFMA, no DADD
      else
        k[2] = fma(u[2], sub(u[0], cf.c), cf.b);
    } else {
      k[0] = u[1];
      k[1] = fma(cf.kappa, lap, fma(kappa2, lap2, -mul(cf.w2, u[0])));
    }
  }
}

// Eq. (5): y += sum_m b_m dt k_m, in FP64 or with a Kahan-compensated update in FP32.
template <typename R, int D, bool KAHAN, uint64_t SHAPE = 0>
__device__ __forceinline__ void gen_combine(const Tableau<R> &tb, const R (*k)[D], R *y, R *cmp) {
#pragma unroll
  for (int d = 0; d < D; ++d) {
    R inc = R(0);
#pragma unroll
    for (int m = 0; m < kMaxStages; ++m)
      if (m < gen_stages<SHAPE>(tb) && gen_b_nonzero<SHAPE>(tb, m)) inc = fma(tb.bdt[m], k[m][d], inc);
    if constexpr (KAHAN) {
      const R s = sub(inc, cmp[d]);
      const R t = add(y[d], s);
      cmp[d] = sub(sub(t, y[d]), s);
      y[d] = t;
    } else {
      y[d] = add(y[d], inc);
    }
  }
}

// ---- one-stage-per-launch sweeps: one site i -------------------------------------------------

template <typename R, int D>
__device__ __forceinline__ void gen_state_site(const GenStagedJob &job, const Tableau<R> &tb, int64_t i, int j) {
  const R *Y = static_cast<const R *>(job.y);
  const R *K = static_cast<const R *>(job.k);
  R *U = static_cast<R *>(job.u);
  const size_t plane = (size_t)job.total * D;
  R y[D], k[kMaxStages][D], u[D];
#pragma unroll
  for (int d = 0; d < D; ++d) y[d] = Y[i * D + d];
#pragma unroll
  for (int m = 0; m < kMaxStages; ++m)
#pragma unroll
    for (int d = 0; d < D; ++d) k[m][d] = (m < j) ? K[m * plane + i * D + d] : R(0);
  gen_stage_state<R, D>(j, tb, y, k, u);
#pragma unroll
  for (int d = 0; d < D; ++d) U[i * D + d] = u[d];
}

// The chain of site i, number ci; its coupling strength goes into c.
template <typename R>
__device__ __forceinline__ ChainDesc gen_site_chain(const GenStagedJob &job, int64_t i, Coef<R> &c, int &ci) {
  ci = 0;
  if (job.nchains == 1) return job.one;
  ci = site_chain(job.chains, job.nchains, i);
  const ChainDesc ch = job.chains[ci];
  c.kappa = (R)ch.kappa;
  return ch;
}
// Index in the state of site q of a chain (boundary-resolved), or -1 beyond a fixed end.
__device__ __forceinline__ int64_t gen_site(const GenStagedJob &job, const ChainDesc &ch, int64_t q) {
  const int64_t g = (ch.bc == PERIODIC) ? ch.off + wrap(q, ch.n) : ((q < 0 || q >= ch.n) ? -1 : ch.off + q);
  return g < 0 || !bounds_ok(job.hdr, in_range(g, 1, job.total)) ? -1 : g;
}

template <typename R, int MODEL, int RANGE>
__device__ __forceinline__ void gen_slope_site(const GenStagedJob &job, const ChainDesc &ch, const Coef<R> &c, R kappa2,
                                               int64_t i, int j) {
  constexpr int D = Dim<MODEL>::D;
  const R *src = static_cast<const R *>(j == 0 ? job.y : job.u);
  R *K = static_cast<R *>(job.k) + (size_t)j * job.total * D;
  const int64_t li = i - ch.off;
  auto xat = [&](int64_t q) -> R {  // coupling coordinate of chain site q
    const int64_t g = gen_site(job, ch, q);
    return g < 0 ? R(0) : src[g * D];
  };
  R u[D], k[D];
#pragma unroll
  for (int d = 0; d < D; ++d) u[d] = src[i * D + d];
  slope_gen<R, MODEL, RANGE>(u, xat(li - 1), xat(li + 1), RANGE == 2 ? xat(li - 2) : R(0),
                             RANGE == 2 ? xat(li + 2) : R(0), c, kappa2, k);
#pragma unroll
  for (int d = 0; d < D; ++d) K[i * D + d] = k[d];
}

template <typename R, int D, bool KAHAN>
__device__ __forceinline__ void gen_combine_site(const GenStagedJob &job, const Tableau<R> &tb, int64_t i) {
  R *Y = static_cast<R *>(job.y);
  R *CMP = static_cast<R *>(job.cmp);
  const R *K = static_cast<const R *>(job.k);
  const size_t plane = (size_t)job.total * D;
  R y[D], k[kMaxStages][D], cmp[D];
#pragma unroll
  for (int d = 0; d < D; ++d) {
    y[d] = Y[i * D + d];
    cmp[d] = KAHAN ? CMP[i * D + d] : R(0);
  }
#pragma unroll
  for (int m = 0; m < kMaxStages; ++m)
#pragma unroll
    for (int d = 0; d < D; ++d) k[m][d] = (m < tb.s) ? K[m * plane + i * D + d] : R(0);
  gen_combine<R, D, KAHAN>(tb, k, y, cmp);
  bool bad = false;
#pragma unroll
  for (int d = 0; d < D; ++d) {
    Y[i * D + d] = y[d];
    if constexpr (KAHAN) CMP[i * D + d] = cmp[d];
    bad |= nonfinite(y[d]);
  }
  if (bad && job.hdr) atomicOr(&job.hdr->status, ST_NONFINITE);
}

inline int64_t staged_grid(int64_t total) {
  int64_t g = (total + 255) / 256;
  const int64_t cap = (int64_t)sm_count() * 64;
  return g > cap ? cap : (g < 1 ? 1 : g);
}

// ---- advancing a tile ----------------------------------------------------------------------

// Two values of the working precision as one 8- or 16-byte shared-memory access.
template <typename R> struct Pair;
template <> struct Pair<float> { using T = float2; };
template <> struct Pair<double> { using T = double2; };

// Advance one tile's registers K steps of the generic scheme.  `edge`: gen_edge_values(V)
// values of shared memory, two parities of [(first, second) coupling coordinate of each thread
// | (second-last, last) of each thread].  Every stage each thread stores its two pairs (two
// vector stores) and, after the stage's one barrier, reads its left neighbour's last pair and
// its right neighbour's first pair (two vector loads, conflict-free): four shared-memory
// instructions for the range-2 coupling, where shuffles plus warp-edge slots took 12 (FP32) or
// 16 (FP64).  The two tile ends read a stand-in (their own pair), which only reaches halo sites.
template <typename R, int MODEL, int V, int RANGE, bool KAHAN, bool MASK, uint64_t SHAPE>
__device__ __forceinline__ void gen_tile_advance(R (&y)[V][Dim<MODEL>::D], R (&cmp)[V][Dim<MODEL>::D],
                                                 uint32_t ghost, int K, const Coef<R> &cf, R kappa2,
                                                 const Tableau<R> &tb, R *edge) {
  constexpr int D = Dim<MODEL>::D;
  static_assert(V >= 2, "the generic kernel holds at least two sites per thread");
  constexpr int NT = kGenEdgeThreads;
  using R2 = typename Pair<R>::T;
  const int tid = threadIdx.x;
  const int lt = tid > 0 ? tid - 1 : tid;                           // left neighbour thread
  const int rt = tid < (int)blockDim.x - 1 ? tid + 1 : tid;          // right neighbour thread
  R k[V][kMaxStages][D];

  int parity = 0;  // edge slots alternate strictly from stage to stage (s may be odd)
#pragma unroll 1
  for (int s = 0; s < K; ++s) {
#pragma unroll
    for (int j = 0; j < kMaxStages; ++j) {
      if (j >= gen_stages<SHAPE>(tb)) break;
      if (!gen_stage_needed<SHAPE>(j)) continue;  // a compiled shape's dead stage: nothing reads it
      R u[V][D];
      R ext[V + 4];  // ext[2 + v] = x of site v; two neighbours on each side
      R2 *head = reinterpret_cast<R2 *>(edge) + parity * 2 * NT;  // (first, second) per thread
      R2 *tail = head + NT;                                         // (second-last, last) per thread
      parity ^= 1;
#pragma unroll
      for (int v = 0; v < V; ++v) {
        gen_stage_state<R, D, SHAPE>(j, tb, y[v], k[v], u[v]);
        ext[2 + v] = (MASK && ((ghost >> v) & 1u)) ? R(0) : u[v][0];
      }
      R2 hv, tv;
      hv.x = ext[2];
      hv.y = ext[3];
      tv.x = ext[V];
      tv.y = ext[V + 1];
      head[tid] = hv;
      tail[tid] = tv;
      // each thread reads only its neighbour threads' slots: in FP64 the streaming form waits
      // for the neighbouring warps only (measured +4.6 % for Dormand-Prince 5); in FP32 the two
      // named barriers per stage cost 22 %, so it keeps the block-wide one
      if constexpr (SHAPE != 0 && sizeof(R) == 8) neighbour_warp_sync(); else __syncthreads();
      {
        const R2 l = tail[lt];
        const R2 r = head[rt];
        ext[0] = l.x;
        ext[1] = l.y;
        ext[V + 2] = r.x;
        ext[V + 3] = r.y;
      }
#pragma unroll
      for (int v = 0; v < V; ++v) {
        R kv[D];
        slope_gen<R, MODEL, RANGE>(u[v], ext[1 + v], ext[3 + v], RANGE == 2 ? ext[v] : R(0),
                                   RANGE == 2 ? ext[4 + v] : R(0), cf, kappa2, kv);
#pragma unroll
        for (int d = 0; d < D; ++d) k[v][j][d] = kv[d];
      }
    }
#pragma unroll
    for (int v = 0; v < V; ++v) gen_combine<R, D, KAHAN, SHAPE>(tb, k[v], y[v], cmp[v]);
  }
}

template <typename R>
inline Tableau<R> to_tableau(const TableauD &t, double dt) {
  Tableau<R> r{};
  r.s = t.s;
  for (int j = 0; j < kMaxStages; ++j) {
    r.anz[j] = 0;
    for (int m = 0; m < kMaxStages; ++m) {
      const double a = (j < t.s && m < j) ? t.a[j][m] : 0.0;
      r.adt[j][m] = (R)(a * dt);
      if (a != 0.0) r.anz[j] |= 1u << m;
    }
  }
  r.bnz = 0;
  for (int m = 0; m < kMaxStages; ++m) {
    const double b = m < t.s ? t.b[m] : 0.0;
    r.bdt[m] = (R)(b * dt);
    if (b != 0.0) r.bnz |= 1u << m;
  }
  return r;
}

}  // namespace rk4d
