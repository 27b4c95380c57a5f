// rk4_internal.h -- structures shared by the host runtime and the kernels' launchers.
// Not part of the public ABI (see include/rk4chain.h).
#pragma once
#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

#include <mutex>

namespace rk4d {

// One chain of a (possibly single-chain) job.  32 bytes, stored in the workspace for batches.
struct ChainDesc {
  int64_t off;   // first site of the chain in the concatenated state
  int64_t n;     // sites
  double kappa;  // coupling strength
  int32_t bc;    // PERIODIC or FIXED
  int32_t pad;
};

// Coefficients in double; converted to the working precision once per launch on the host.
// kappa2: second-neighbour coupling (generic scheme only; 0 for the paper's chain).
struct CoefD {
  double a, b, c, kappa, w2, h2, h1, dt6, kappa2, dt3;
};

// Coefficients of the split FP64 step (rk4_split.cuh): tau = dt / 2 (generic tableaux: dt), and the
// products with it as float pairs (h + l).  at: Roessler a tau, harmonic w2 tau.  most: high words of the largest
// magnitudes a site's own parameters may have (heterogeneous chains; in their order).  The state's range
// (split_in_range): high words of the largest x and -x (Roessler; of any site's own c for heterogeneous
// chains, which far, the largest |x - c|, bounds then) and of the other components.
struct SplitCoef {
  double w;  // tau / 3 (generic tableaux: dt)
  float tauh, taul, kth, ktl, k2h, k2l, ath, atl, ch, cl;
  unsigned most[4], most_x, least_x, big;
  float far;
};

// Generic explicit Runge-Kutta tableau (strictly lower a, weights b), up to kMaxStages stages.
constexpr int kMaxStages = 7;
struct TableauD {
  int s;
  double a[kMaxStages][kMaxStages];
  double b[kMaxStages];
};

// Device status word bits (in the workspace header).  ST_BOUNDS is only ever set by a library
// built with -DRK4_DEBUG_BOUNDS (index checks on every global access; see rk4_tile.cuh).
enum : int { ST_NONFINITE = 1, ST_TIMEOUT = 2, ST_BOUNDS = 4 };

// Workspace header: status word, grid-barrier counters.  256 bytes.
struct WsHeader {
  int status;
  unsigned bar_count;
  unsigned bar_gen;
  int timeout_where;
  unsigned long long work[2];  // persistent kernel: next item of the current time block, by parity
  unsigned char pad[224];
};

// A piece of one batch chain placed in a shared ("packed") tile: the chain's last partial piece
// of interior sites (or the whole chain when it is shorter than a tile's interior), with its own
// halo of H sites on each side.  Several segments lie side by side in one tile; each thread's
// sites belong to one segment because o and L are multiples of the sites per thread.
struct SegDesc {
  int64_t g0;     // first interior site (chain-local index)
  int32_t chain;  // index into the chain table
  int32_t o;      // first tile slot of the segment's window
  int32_t cnt;    // interior sites
  int32_t L;      // window length in slots: H + cnt + H rounded up to a multiple of the sites per thread
};

// The tiles of one launch over a batch: the full tiles (G interior sites each) of every chain,
// numbered chain by chain (full_prefix: first full tile of each chain, nchains + 1 entries),
// and the packed tiles (pack_prefix: first segment of each packed tile, npacked + 1 entries,
// into segs).  The kernels process the packed tiles first.  A chain of n sites has
// floor(n / G) full tiles and, when G does not divide n, one segment.
// tile_chain, when not null, holds for each full tile its chain and chain-local tile index
// (filled on the device from full_prefix before the launches), so that a tile finds its chain
// with one load instead of a search of full_prefix.
struct BatchTiles {
  const int32_t *full_prefix;
  const int32_t *pack_prefix;
  const SegDesc *segs;
  const int2 *tile_chain;
  int64_t nfull;
  int64_t npacked;
};

// Arguments of one blocked launch (one chain, or a batch through a chain table).
struct BlockedJob {
  const void *in;    // state read by this launch
  void *out;         // state written by this launch
  const void *cin;   // Kahan compensation read (FP32) or NULL
  void *cout;        // Kahan compensation written
  int nchains;       // 1: use `one`; >1: use `chains` / `bt`
  ChainDesc one;
  const ChainDesc *chains;      // device table (batches)
  BatchTiles bt;                // batches: the tiles of the launch (full_prefix counts every tile
                                // of a chain when the batch is not packed)
  int packed;                   // 1: packed tiles (bt.npacked of them) precede the full tiles
  int K;                        // steps in this launch
  int G;                        // interior sites per tile
  int64_t ntiles;               // tiles in the launch (a packed batch: its full tiles, beside bt.npacked)
  const void *sp;               // per-site parameters of a heterogeneous chain, or NULL
  WsHeader *hdr;                // status word (non-finite results, debug bounds checks)
  int64_t total;                // sites in the state buffers
  int split;                    // 1: FP64 in the split form (rk4_split.cuh)
};

struct StagedJob {
  void *y;            // state, updated in place at the last stage
  void *cmp;          // Kahan compensation (FP32) or NULL, updated in place
  const void *uin;    // stage state read (stages 1..3)
  void *uout;         // stage state written (stages 0..2)
  void *acc;          // slope sum
  int nchains;
  ChainDesc one;
  const ChainDesc *chains;   // device table for batches (site -> chain by binary search)
  int64_t total;             // total sites
  const void *sp;            // per-site parameters of a heterogeneous chain, or NULL
  WsHeader *hdr;             // status word
  int split;                 // 1: FP64 in the split form: acc holds K1, n2 and n3 the negated
  void *n2, *n3;             // differences of stages 2 and 3 as float pairs
  int parity;                // of the step (which wide flag is read)
  unsigned *wide;            // per chain and step parity: its state has left the split's range
};

// One step of the generic standard scheme: stage states, slopes and the combination, each a
// full sweep.  k holds s slope arrays of total * D values; u one stage state.
struct GenStagedJob {
  void *y;
  void *cmp;
  void *u;
  void *k;
  int nchains;
  ChainDesc one;
  const ChainDesc *chains;
  int64_t total;
  WsHeader *hdr;  // status word
  int split;      // 1: the split form (k[0]: the first slope; the others: their remainders, and u, as float pairs)
  int parity;     // of the step (which wide flag is read)
  unsigned *wide;  // per chain and step parity: its state has left the split's range
};

struct PersistentJob {
  void *bufA, *bufB;            // state ping-pong: time block t reads A when t is even
  void *cA, *cB;                // compensation ping-pong (FP32) or NULL
  int nchains;
  ChainDesc one;
  const ChainDesc *chains;
  BatchTiles bt[4];             // batches: the tiles of a time block for each k (full, then packed)
  int nk;                       // distinct k values (1..4)
  int kval[4];                  // steps per time block
  int Gval[4];                  // interior sites per tile for each k
  int64_t ntiles[4];            // tiles per time block for each k
  int64_t cnt[4];               // time blocks of kval[0], then of kval[1], ...
  WsHeader *hdr;                // status word and barrier counters (zeroed before launch)
  long long timeout_ns;         // bound on any single barrier wait
  int extra_arrivals;           // test hook: barrier waits for this many blocks that never come
  int64_t total;                // sites in the state buffers
  int split;                    // 1: FP64 in the split form (rk4_split.cuh)
};

// Launchers (return a cudaError_t).  R is selected by `fp32` (FP32 + Kahan) or double.
cudaError_t launch_blocked(int model, bool fp32, int v, int block, const BlockedJob &job, const CoefD &cf,
                           cudaStream_t st);  // job.sp != NULL selects the heterogeneous kernel (v = 2 or 4)
// The split forms of launch_blocked, launch_persistent and persistent_max_grid (one model's
// kernels per translation unit).
template <int MODEL>
cudaError_t launch_split_blocked(int v, int block, const BlockedJob &job, const CoefD &cf, cudaStream_t st);
template <int MODEL>
cudaError_t launch_split_persistent(int v, int block, int grid, const PersistentJob &job, const CoefD &cf,
                                    cudaStream_t st);
template <int MODEL> int persistent_split_max_grid(int v, int block);
// Set the chains' flags `wide` (two words each, the first of them here) of the staged schemes' split form.
cudaError_t launch_split_scan(int model, int range, const double *state, const double *sp, int64_t total, int nchains,
                              const ChainDesc &one, const ChainDesc *chains, const CoefD &cf, unsigned *wide,
                              cudaStream_t st);
// A chain's flag: 1 when a value of its state or a site's own parameter is outside the split's range; 2 when
// a site has a slope of zero in every component, 4 when one has not.  A chain with both (a front that runs
// into sites at rest, whose far end the pairs do not hold: rk4_split.cuh) is advanced in the FP64 form too.
constexpr unsigned kWideRange = 1, kWideRest = 2, kWideMoves = 4;
__host__ __device__ constexpr bool wide_chain(unsigned f) { return (f & kWideRange) || (f & 6u) == 6u; }
// Whether every step of a handle with these coefficients (c.kappa: the largest coupling strength
// of its chains) may run in the split form, and the form's coefficients.
bool split_allowed(int model, const CoefD &c);
SplitCoef split_coef(int model, const CoefD &c, bool generic = false, bool het = false);
// The generic scheme in the split form (k_gen_split.cu): a tableau's rows and weights, as float pairs
// where they multiply the slopes' remainders, and the stages the result needs.
struct SplitTableau {
  int s, last;                                 // last: the last stage needed
  uint32_t need;
  int nb, mb[kMaxStages];                      // the stages m >= 1 of nonzero weight but `last`, in order
  int na[kMaxStages], ma[kMaxStages][kMaxStages];  // and those with a nonzero a_jm
  int slot[kMaxStages], slots;                 // where a stage's remainders lie in a thread's record
  double B, E;                                 // the weights' sum, and dt sum b_m c_m
  int unit;                                    // B is 1
  float Bl;                                    // what B's rounding leaves
  float ch[kMaxStages], cl[kMaxStages];        // row sums c_j
  float gh[kMaxStages], gl[kMaxStages];        // sum over m of a_jm c_m
  float ah[kMaxStages][kMaxStages], al[kMaxStages][kMaxStages], bh[kMaxStages], bl[kMaxStages];
};
bool split_tableau_allowed(const TableauD &t);  // whether the form takes the tableau
SplitTableau split_tableau(const TableauD &t, double dt);
cudaError_t launch_gen_split(int model, int range, int sites, const BlockedJob &job, const CoefD &cf,
                             const TableauD &tb, double dt, int H, cudaStream_t st);  // tiles of `sites` sites
cudaError_t launch_gen_split_step(int model, int range, const GenStagedJob &job, const CoefD &cf,
                                  const TableauD &tb, double dt, cudaStream_t st);
cudaError_t launch_staged(int model, bool fp32, int stage, const StagedJob &job, const CoefD &cf,
                          cudaStream_t st);
cudaError_t launch_persistent(int model, bool fp32, int v, int block, int grid, const PersistentJob &job,
                              const CoefD &cf, cudaStream_t st);
int persistent_max_grid(int model, bool fp32, int v, int block, bool split);
cudaError_t launch_energy(int model, bool fp32, const void *state, const void *cmp, int nchains,
                          const ChainDesc &one, const ChainDesc *chains, const CoefD &cf, double *partials,
                          double *out, WsHeader *hdr, cudaStream_t st);
// Energy of the chain-local sites [lo, hi) of one chain; neighbours outside the range are read
// from the state like any other site (a sub-domain's ghost zones).  out: one device double.
cudaError_t launch_energy_range(int model, bool fp32, const void *state, const void *cmp, const ChainDesc &ch,
                                int64_t lo, int64_t hi, const CoefD &cf, double *partials, double *out,
                                WsHeader *hdr, cudaStream_t st);
// One ghost zone of a sub-domain state: `ghost` rows starting at dst_row are copied from the
// rows starting at src_row.
struct GhostPair {
  int64_t dst_row, src_row;
};
// Every zone of `pairs` (a device table) in one launch, for the state and, if not NULL, the
// compensation; rows are row_bytes (a multiple of 4) long.
cudaError_t launch_ghost_copy(void *state, void *comp, const GhostPair *pairs, int npairs, int64_t ghost,
                              int row_bytes, cudaStream_t st);
// Copy `bytes` between two 16-byte-aligned buffers with a kernel (either side may be mapped
// page-locked host memory, given by its device pointer).
cudaError_t launch_copy(void *dst, const void *src, size_t bytes, cudaStream_t st);
// Fill tile_chain[t] = (chain, t - prefix[chain]) for the ntiles tiles numbered by prefix
// (nchains + 1 entries, the first tile of each chain).
cudaError_t launch_tile_chains(const int32_t *prefix, int nchains, int64_t ntiles, int2 *tile_chain, cudaStream_t st);
cudaError_t launch_fill_uniform(void *dst, int64_t count, uint64_t seed, uint64_t start, bool fp32,
                                cudaStream_t st);
cudaError_t launch_gen_staged_step(int model, bool fp32, int range, const GenStagedJob &job, const CoefD &cf,
                                   const TableauD &tb, double dt, cudaStream_t st);
cudaError_t launch_gen_blocked(int model, bool fp32, int range, int v, int block, const BlockedJob &job,
                               const CoefD &cf, const TableauD &tb, double dt, int H, cudaStream_t st);
size_t gen_blocked_smem_bytes(int model, bool fp32, int v, int block, const TableauD &tb);
int gen_blocked_max_threads(int model, bool fp32, int range, int v, const TableauD &tb);
bool gen_compiled(const TableauD &tb);  // whether FP32 tile kernels are compiled for the tableau's shape
size_t blocked_smem_bytes(int model, bool fp32, int v, int block, bool het = false);  // either FP64 form fits
int blocked_max_threads(int model, bool fp32, int v, bool het = false);

constexpr int kEnergyBlocks = 1024;  // fixed grid of the single-chain reduction (deterministic)

// Per-device state of host-side set-up that CUDA scopes to the current device (a kernel's
// shared-memory limit, a device attribute): done once for each device a process uses.
constexpr int kMaxDevices = 64;
struct PerDevice {
  std::mutex m;
  bool done[kMaxDevices] = {};
  cudaError_t err[kMaxDevices] = {};
  int value[kMaxDevices] = {};
};

// Raise `kernel`'s dynamic shared-memory limit to `bytes` on the current device, once per
// device (the attribute applies only to the device that is current when it is set).
template <typename K> inline cudaError_t set_smem_limit_once(K *kernel, int bytes, PerDevice &pd) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= kMaxDevices) return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  std::lock_guard<std::mutex> g(pd.m);
  if (!pd.done[dev]) {
    pd.err[dev] = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    pd.done[dev] = true;
  }
  return pd.err[dev];
}

// Streaming multiprocessors of the current device (cached per device); grid-stride kernels
// size their grids as a multiple of it.
inline int sm_count() {
  static PerDevice pd;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return 152;
  if (dev < 0 || dev >= kMaxDevices) {
    int n = 0;
    return cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess && n > 0 ? n : 152;
  }
  std::lock_guard<std::mutex> g(pd.m);
  if (!pd.done[dev]) {
    int n = 0;
    if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n <= 0) n = 152;
    pd.value[dev] = n;
    pd.done[dev] = true;
  }
  return pd.value[dev];
}

}  // namespace rk4d

struct rk4_chain;
namespace rk4d {
// Read-only view of a handle (model, precision, chain table on the host, coefficients, stream).
int handle_info(const rk4_chain *h, int *model, bool *fp32, int *nchains, const ChainDesc **chains, CoefD *cf,
                cudaStream_t *stream, bool *het);
// Stages of the handle's tableau and its coupling range (1, or 2 with second neighbours): one
// step reaches stages x range sites along the chain.
int scheme_reach(const rk4_chain *h, int *stages, int *range);
// For callers that capture a handle's integrations into a larger CUDA graph: a counter bumped
// by every setter (a captured graph is stale once it changes); the stream the handle enqueues
// on and its own graph replay, swapped during a capture; and the pinned host tables and
// buffers an integration of nsteps needs, prepared beforehand (preparing them may synchronise
// the stream, which must not happen while capturing).
unsigned config_version(const rk4_chain *h);
cudaStream_t swap_stream(rk4_chain *h, cudaStream_t st);
bool swap_graphs(rk4_chain *h, bool on);
int prepare_integrate(rk4_chain *h, int64_t nsteps);
// One-way integrations of a batch: with way 1 an integration of tiling.k steps is one blocked launch
// from the caller's buffers into the workspace's copy of the state (state_copy), with way 2 one
// from there back; with 0 (the default) it starts and ends in the caller's buffers.  Returns the old way.
int swap_one_way(rk4_chain *h, int way);
bool one_way_allowed(const rk4_chain *h, int64_t nsteps);
void state_copy(const rk4_chain *h, void *ws, void **state, void **comp);

}  // namespace rk4d
