// k_generic.cu -- any explicit Runge-Kutta tableau (up to 7 stages) and coupling range 1 or 2
// (nearest or next-nearest neighbours), the generalisations the paper names in Sec. 2 ("any
// other explicit Runge-Kutta method") and Sec. 5 ("next-nearest-neighbour couplings need twice
// as long overlaps").  Temporal blocking then needs a halo of s * range sites per side per
// step (s stages, each reaching `range` sites further).
//
// Two schemes share one per-site operation sequence (so they agree bit for bit):
//   * k_gen_state / k_gen_slope / k_gen_combine: the standard implementation, one sweep per
//     stage-state evaluation, one per slope evaluation and one for the combination (2s+1 sweeps
//     per step, Sec. 2.2);
//   * k_gen_blocked: tiles of W = block * v sites advanced k steps per launch in registers.
//
// Per-site operation order (fixed):
//   stage state  u = y; for m < j with a_jm != 0:  u = fma(a_jm dt, k_m, u)        (Eq. (4))
//   slope        range 1: as the RK4 kernels; range 2 adds lap2 = fma(-2, x, x_{i-2} + x_{i+2})
//                inside the coupling: kx = fma(kappa, lap, fma(kappa2, lap2, -(y + z)))
//   combine      inc = 0; for m with b_m != 0: inc = fma(b_m dt, k_m, inc)          (Eq. (5))
//                FP64: y = y + inc;  FP32-Kahan: s = inc - c; t = y + s; c = (t - y) - s; y = t
#include <algorithm>

#include "rk4_generic.cuh"

namespace rk4d {

// ---- one-stage-per-launch reference ------------------------------------------------------

template <typename R, int D>
__global__ void __launch_bounds__(256) k_gen_state(GenStagedJob job, Tableau<R> tb, int j) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < job.total; i += stride) gen_state_site<R, D>(job, tb, i, j);
}
template <typename R, int MODEL, int RANGE>
__global__ void __launch_bounds__(256) k_gen_slope(GenStagedJob job, Coef<R> cf, R kappa2, int j) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < job.total; i += stride) {
    Coef<R> c = cf;
    int ci;
    const ChainDesc ch = gen_site_chain(job, i, c, ci);
    gen_slope_site<R, MODEL, RANGE>(job, ch, c, kappa2, i, j);
  }
}
template <typename R, int D, bool KAHAN>
__global__ void __launch_bounds__(256) k_gen_combine(GenStagedJob job, Tableau<R> tb) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < job.total; i += stride) gen_combine_site<R, D, KAHAN>(job, tb, i);
}

// ---- temporally blocked generic kernel ----------------------------------------------------

// The generic tile kernel.  With a compiled tableau shape (STREAM) it runs as a streaming
// loop: a resident set of blocks (grid sized by the host to what fits on the GPU) walks the
// tiles, block b taking tiles b, b + gridDim.x, ...  While a block computes one tile, the next
// one's window is already on its way into the second of two shared-memory buffers (cp.async),
// so a tile's load latency is hidden behind the previous tile's arithmetic.  That lets short
// launches (small k, and so a small halo of redundant sites) run without exposed load time,
// which matters here: the generic scheme's halo is s' x range sites per side and step (12 for
// Dormand-Prince 5 with second neighbours).  The run-time-shape form (SHAPE = 0) processes one
// tile per block (a loop around it would keep the tableau's coefficients in registers).
// Shared memory: edge[gen_edge_values(V)] | buffer 0: tile[W*D] (+ ctile[W*D]) | buffer 1
// (streaming only).
template <typename R, int MODEL, int V, int RANGE, bool KAHAN, uint64_t SHAPE = 0>
__global__ void __launch_bounds__(GenBounds<R, V, SHAPE>::threads) k_gen_blocked(BlockedJob job, Coef<R> cf,
                                                                                 R kappa2, Tableau<R> tb, int H) {
  constexpr int D = Dim<MODEL>::D;
  constexpr bool STREAM = SHAPE != 0;
  extern __shared__ __align__(16) unsigned char smem[];
  R *edge = reinterpret_cast<R *>(smem);
  const int W = blockDim.x * V;
  const int G = job.G;
  const int tsize = W * D * (KAHAN ? 2 : 1);  // one buffer: tile and compensation tile
  R *const buf0 = edge + gen_edge_values(V);
  const R *in = static_cast<const R *>(job.in);
  const R *cin = static_cast<const R *>(job.cin);

  // chain, chain-local tile index and coupling of item `it`
  auto locate = [&](int64_t it, ChainDesc &ch, int64_t &tile, Coef<R> &c) {
    c = cf;
    if (job.nchains == 1) {
      ch = job.one;
      tile = it;
    } else {
      int ci;
      if (job.bt.tile_chain) {
        const int2 tc = __ldg(&job.bt.tile_chain[it]);
        ci = tc.x;
        tile = tc.y;
      } else {
        ci = find_chain_warp(job.bt.full_prefix, job.nchains, it);  // every warp, three rounds of loads
        tile = it - job.bt.full_prefix[ci];
      }
      ch = job.chains[ci];
      c.kappa = (R)ch.kappa;
    }
  };
  auto issue = [&](int64_t it, R *buf) {
    ChainDesc ch;
    int64_t tile;
    Coef<R> c;
    locate(it, ch, tile, c);
    const int64_t t0 = tile * (int64_t)G - H;
    tile_load<R, D, false>(buf, in, ch.off, ch.n, ch.bc, t0, W, job.total, job.hdr);
    if constexpr (KAHAN) tile_load<R, D, false>(buf + W * D, cin, ch.off, ch.n, ch.bc, t0, W, job.total, job.hdr);
    cp_async_commit();
  };

  int64_t item = blockIdx.x;
  if (item >= job.ntiles) return;
  issue(item, buf0);
  int cur = 0;
  for (;;) {
    const int64_t next = item + gridDim.x;
    if (STREAM && next < job.ntiles) {
      issue(next, buf0 + (cur ^ 1) * tsize);  // that buffer was released by the last iteration's barrier
      cp_async_wait<1>();                     // this tile's copies are complete, the next one's may run on
    } else {
      cp_async_wait<0>();
    }
    __syncthreads();
    R *tl = buf0 + cur * tsize;
    R *ctl = tl + W * D;
    ChainDesc ch;
    int64_t tile;
    Coef<R> c;
    locate(item, ch, tile, c);
    const int64_t t0 = tile * (int64_t)G - H;
    R y[V][D], cmp[V][D];
    const int base = threadIdx.x * V;
#pragma unroll
    for (int v = 0; v < V; ++v)
#pragma unroll
      for (int d = 0; d < D; ++d) {
        y[v][d] = tl[(base + v) * D + d];
        if constexpr (KAHAN) cmp[v][d] = ctl[(base + v) * D + d]; else cmp[v][d] = R(0);
      }
    const bool edge_tile = (ch.bc == FIXED) && (t0 < 0 || t0 + W > ch.n);
    if (edge_tile) {
      uint32_t ghost = 0;
#pragma unroll
      for (int v = 0; v < V; ++v) {
        const int64_t g = t0 + base + v;
        if (g < 0 || g >= ch.n) ghost |= 1u << v;
      }
      gen_tile_advance<R, MODEL, V, RANGE, KAHAN, true, SHAPE>(y, cmp, ghost, job.K, c, kappa2, tb, edge);
    } else {
      gen_tile_advance<R, MODEL, V, RANGE, KAHAN, false, SHAPE>(y, cmp, 0u, job.K, c, kappa2, tb, edge);
    }
    const int64_t g0 = t0 + H;
    const int64_t rem = ch.n - g0;
    const int cnt = (int)(rem < G ? rem : G);
    bool bad = false;  // a stored (interior) value is NaN or infinite
#pragma unroll
    for (int v = 0; v < V; ++v) {
      const bool stored = base + v >= H && base + v < H + cnt;
#pragma unroll
      for (int d = 0; d < D; ++d) {
        tl[(base + v) * D + d] = y[v][d];
        if constexpr (KAHAN) ctl[(base + v) * D + d] = cmp[v][d];
        bad |= stored && nonfinite(y[v][d]);
      }
    }
    report_nonfinite(job.hdr, __syncthreads_or(bad));
    if (cnt > 0) {
      tile_store<R, D>(static_cast<R *>(job.out), tl, ch.off, H, g0, cnt, job.total, W, job.hdr);
      if constexpr (KAHAN) tile_store<R, D>(static_cast<R *>(job.cout), ctl, ch.off, H, g0, cnt, job.total, W, job.hdr);
    }
    if constexpr (!STREAM) break;
    __syncthreads();  // the buffer is refilled two iterations on; nobody may still read it
    cur ^= 1;
    item = next;
    if (item >= job.ntiles) break;
  }
}

// The compiled shape a tableau runs with at v sites per thread (0: the run-time-shape kernel).
static uint64_t compiled_shape(const TableauD &t, int v) {
  if (v != 4) return 0;
  const uint64_t sh = tableau_shape(t);
  return (sh == kShapeDopri5 || sh == kShapeRK4) ? sh : 0;
}

bool gen_compiled(const TableauD &t) { return compiled_shape(t, 4) != 0; }

template <typename R, int MODEL, int V, int RANGE, bool KAHAN, uint64_t SHAPE>
static int gen_max_threads_s() {
  cudaFuncAttributes a;
  if (cudaFuncGetAttributes(&a, k_gen_blocked<R, MODEL, V, RANGE, KAHAN, SHAPE>) != cudaSuccess) return 0;
  return a.maxThreadsPerBlock;
}

template <typename R, int MODEL, int V, int RANGE, bool KAHAN>
static int gen_max_threads_one(uint64_t shape) {
  if constexpr (V == 4) {
    if (shape == kShapeDopri5) return gen_max_threads_s<R, MODEL, V, RANGE, KAHAN, kShapeDopri5>();
    if (shape == kShapeRK4) return gen_max_threads_s<R, MODEL, V, RANGE, KAHAN, kShapeRK4>();
  }
  return gen_max_threads_s<R, MODEL, V, RANGE, KAHAN, 0>();
}

template <int MODEL, int RANGE>
static int gen_max_threads_m(bool fp32, int v, uint64_t sh) {
  if (v == 2) return fp32 ? gen_max_threads_one<float, MODEL, 2, RANGE, true>(sh) : gen_max_threads_one<double, MODEL, 2, RANGE, false>(sh);
  if (v == 4) return fp32 ? gen_max_threads_one<float, MODEL, 4, RANGE, true>(sh) : gen_max_threads_one<double, MODEL, 4, RANGE, false>(sh);
  return 0;
}

int gen_blocked_max_threads(int model, bool fp32, int range, int v, const TableauD &tb) {
  const uint64_t sh = compiled_shape(tb, v);
  if (model == ROESSLER) return range == 1 ? gen_max_threads_m<ROESSLER, 1>(fp32, v, sh) : gen_max_threads_m<ROESSLER, 2>(fp32, v, sh);
  return range == 1 ? gen_max_threads_m<HARMONIC, 1>(fp32, v, sh) : gen_max_threads_m<HARMONIC, 2>(fp32, v, sh);
}

size_t gen_blocked_smem_bytes(int model, bool fp32, int v, int block, const TableauD &tb) {
  const int D = model == ROESSLER ? 3 : 2;
  const size_t rs = fp32 ? 4 : 8;
  const size_t buffers = compiled_shape(tb, v) != 0 ? 2 : 1;  // the streaming form double-buffers
  return (size_t)gen_edge_values(v) * rs + buffers * (size_t)block * v * D * rs * (fp32 ? 2 : 1);
}

// ---- launchers ------------------------------------------------------------------------------

template <typename R, int MODEL, int RANGE, bool KAHAN>
static cudaError_t gen_staged_t(const GenStagedJob &job, const CoefD &cfd, const TableauD &td, double dt,
                                cudaStream_t st) {
  constexpr int D = Dim<MODEL>::D;
  if (job.total <= 0) return cudaSuccess;
  const Tableau<R> tb = to_tableau<R>(td, dt);
  const Coef<R> cf = to_coef<R>(cfd, cfd.kappa);
  const unsigned grid = (unsigned)staged_grid(job.total);
  for (int j = 0; j < td.s; ++j) {
    if (j > 0) k_gen_state<R, D><<<grid, 256, 0, st>>>(job, tb, j);
    k_gen_slope<R, MODEL, RANGE><<<grid, 256, 0, st>>>(job, cf, (R)cfd.kappa2, j);
  }
  k_gen_combine<R, D, KAHAN><<<grid, 256, 0, st>>>(job, tb);
  return cudaGetLastError();
}

cudaError_t launch_gen_staged_step(int model, bool fp32, int range, const GenStagedJob &job, const CoefD &cf,
                                   const TableauD &tb, double dt, cudaStream_t st) {
  if (job.split) return launch_gen_split_step(model, range, job, cf, tb, dt, st);
#define RK4_GEN_STAGED(MODEL)                                                                            \
  if (range == 1)                                                                                        \
    return fp32 ? gen_staged_t<float, MODEL, 1, true>(job, cf, tb, dt, st)                              \
                : gen_staged_t<double, MODEL, 1, false>(job, cf, tb, dt, st);                            \
  return fp32 ? gen_staged_t<float, MODEL, 2, true>(job, cf, tb, dt, st)                                 \
              : gen_staged_t<double, MODEL, 2, false>(job, cf, tb, dt, st);
  if (model == ROESSLER) {
    RK4_GEN_STAGED(ROESSLER)
  }
  RK4_GEN_STAGED(HARMONIC)
#undef RK4_GEN_STAGED
}

template <typename R, int MODEL, int V, int RANGE, bool KAHAN, uint64_t SHAPE>
static cudaError_t gen_blocked_s(int block, const BlockedJob &job, const CoefD &cfd, const TableauD &td, double dt,
                                 int H, cudaStream_t st) {
  static PerDevice attr;
  const cudaError_t attr_err = set_smem_limit_once(k_gen_blocked<R, MODEL, V, RANGE, KAHAN, SHAPE>, 200 * 1024, attr);
  if (attr_err != cudaSuccess) return attr_err;
  if (job.ntiles <= 0) return cudaSuccess;
  const size_t smem = gen_blocked_smem_bytes(MODEL, KAHAN, V, block, td);
  int64_t grid = job.ntiles;  // one tile per block, or
  if constexpr (SHAPE != 0) {  // the streaming form: as many blocks as stay resident together
    int per_sm = 0;
    cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(
        &per_sm, k_gen_blocked<R, MODEL, V, RANGE, KAHAN, SHAPE>, block, smem);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) return cudaErrorInvalidConfiguration;
    grid = std::min<int64_t>(job.ntiles, (int64_t)per_sm * sm_count());
  }
  k_gen_blocked<R, MODEL, V, RANGE, KAHAN, SHAPE><<<(unsigned)grid, block, smem, st>>>(
      job, to_coef<R>(cfd, cfd.kappa), (R)cfd.kappa2, to_tableau<R>(td, dt), H);
  return cudaGetLastError();
}

template <typename R, int MODEL, int V, int RANGE, bool KAHAN>
static cudaError_t gen_blocked_t(int block, const BlockedJob &job, const CoefD &cfd, const TableauD &td, double dt,
                                 int H, cudaStream_t st) {
  if constexpr (V == 4) {
    const uint64_t sh = compiled_shape(td, V);
    if (sh == kShapeDopri5) return gen_blocked_s<R, MODEL, V, RANGE, KAHAN, kShapeDopri5>(block, job, cfd, td, dt, H, st);
    if (sh == kShapeRK4) return gen_blocked_s<R, MODEL, V, RANGE, KAHAN, kShapeRK4>(block, job, cfd, td, dt, H, st);
  }
  return gen_blocked_s<R, MODEL, V, RANGE, KAHAN, 0>(block, job, cfd, td, dt, H, st);
}

template <int MODEL, int RANGE>
static cudaError_t gen_blocked_m(bool fp32, int v, int block, const BlockedJob &job, const CoefD &cf,
                                 const TableauD &tb, double dt, int H, cudaStream_t st) {
  switch (v) {
    case 2:
      return fp32 ? gen_blocked_t<float, MODEL, 2, RANGE, true>(block, job, cf, tb, dt, H, st)
                  : gen_blocked_t<double, MODEL, 2, RANGE, false>(block, job, cf, tb, dt, H, st);
    case 4:
      return fp32 ? gen_blocked_t<float, MODEL, 4, RANGE, true>(block, job, cf, tb, dt, H, st)
                  : gen_blocked_t<double, MODEL, 4, RANGE, false>(block, job, cf, tb, dt, H, st);
    default:
      return cudaErrorInvalidValue;
  }
}

cudaError_t launch_gen_blocked(int model, bool fp32, int range, int v, int block, const BlockedJob &job,
                               const CoefD &cf, const TableauD &tb, double dt, int H, cudaStream_t st) {
  if (job.split) return launch_gen_split(model, range, block * v, job, cf, tb, dt, H, st);
  if (model == ROESSLER)
    return range == 1 ? gen_blocked_m<ROESSLER, 1>(fp32, v, block, job, cf, tb, dt, H, st)
                      : gen_blocked_m<ROESSLER, 2>(fp32, v, block, job, cf, tb, dt, H, st);
  return range == 1 ? gen_blocked_m<HARMONIC, 1>(fp32, v, block, job, cf, tb, dt, H, st)
                    : gen_blocked_m<HARMONIC, 2>(fp32, v, block, job, cf, tb, dt, H, st);
}

}  // namespace rk4d
