// rk4_abi.cu -- host runtime behind the C ABI of include/rk4chain.h: argument checking,
// workspace layout, launch plans (k steps per launch, ping-pong buffers), CUDA-graph replay,
// the tiling autotuner, reductions and the status word.  Only host code lives here; every
// floating-point operation of the integrator runs in the kernels.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <new>
#include <vector>

#include <nvtx3/nvToolsExt.h>

#include "../../include/rk4chain.h"
#include "rk4_internal.h"

using namespace rk4d;

namespace {

constexpr size_t kAlign = 256;
constexpr int kMaxDistinctK = 4;
constexpr size_t kMaxSmem = 200 * 1024;

size_t align_up(size_t x) { return (x + kAlign - 1) / kAlign * kAlign; }

struct GraphKey {
  int kernel = -1;
  const void *state = nullptr, *comp = nullptr, *ws = nullptr;
  int64_t nsteps = -1;
  int block = 0, v = 0, k = 0;
  long long timeout = 0;
  const void *sp = nullptr;
  int generic = 0;
  // the plan's launches: a batch's tables are laid out by kval and its tile counts are baked into the
  // graph, and the automatic and a set tiling of the same block, v and k make different plans
  std::vector<int> kval;
  std::vector<int64_t> cnt;
  bool operator==(const GraphKey &o) const {
    return kernel == o.kernel && state == o.state && comp == o.comp && ws == o.ws && nsteps == o.nsteps &&
           block == o.block && v == o.v && k == o.k && timeout == o.timeout && sp == o.sp && generic == o.generic &&
           kval == o.kval && cnt == o.cnt;
  }
};

struct WsLayout {
  size_t hdr, partials, result, chains, prefix, tiles, state, comp, u0, u1, acc, total;
};

// One launch plan: cnt[i] launches (or time blocks) of kval[i] steps, one i after the other, and
// whether the result needs copying back from the workspace because their number is odd.
struct Plan {
  std::vector<int> kval;
  std::vector<int64_t> cnt;
  bool copy_back = false;
  void add(int k, int64_t times = 1) {
    for (size_t i = 0; i < kval.size(); ++i)
      if (kval[i] == k) {
        cnt[i] += times;
        return;
      }
    kval.push_back(k);
    cnt.push_back(times);
  }
  int64_t count() const {
    int64_t s = 0;
    for (int64_t c : cnt) s += c;
    return s;
  }
};

}  // namespace

struct rk4_chain {
  int model = 0, precision = 0, D = 3;
  bool fp32 = false;
  int nchains = 1;
  std::vector<ChainDesc> chains;
  double kappa_most = 0.0, kappa_least = 0.0;  // largest and smallest nonzero |kappa| of the chains
  int64_t total = 0;
  double dt = 0.01;
  rk4_params p{};
  cudaStream_t stream = nullptr;
  cudaStream_t cap_stream = nullptr;
  int kernel = RK4_KERNEL_AUTO;
  bool tiling_auto = true;
  rk4_tiling tiling{};
  rk4_tiling run{};  // what the current integration runs with (run_tiling)
  unsigned run_version = 0;  // config_version + 1 of the last integration with the automatic tiling
  // its last few automatic choices, by the number of steps, under one configuration
  struct {
    int64_t steps = -1;
    rk4_tiling tiling{};
  } automatic[8];
  unsigned auto_next = 0, auto_version = 0;
  int one_way = 0;  // swap_one_way: 1 state -> workspace, 2 workspace -> state, in one launch
  double t0 = 0.0;
  int64_t nstep = 0;
  bool graphs = true;
  long long timeout_ns = 2000000000LL;
  // pinned host staging: chain table followed by kMaxDistinctK per-k tile tables (see
  // ktable_bytes), in the same relative layout as in the workspace
  void *h_tables = nullptr;
  size_t tables_bytes = 0;
  std::vector<int> tables_k;  // the k values the tile tables currently describe
  int tables_W = 0;           // and the tile width they were computed for
  int tables_v = 0;           // the sites per thread (packed segments are aligned to it)
  int tables_halo = 0;        // the halo per step
  int tables_packed = -1;     // and whether they are packed (see packed_batch)
  int64_t nfull[kMaxDistinctK] = {};    // packed batches: full tiles per k slot
  int64_t npacked[kMaxDistinctK] = {};  // and packed tiles
  double *h_out = nullptr;    // pinned: reduction results (nchains doubles)
  int *h_status = nullptr;    // pinned: status word read-back
  GraphKey gkey;
  cudaGraphExec_t gexec = nullptr;
  // generic explicit RK scheme (any tableau, coupling range 1 or 2)
  bool has_tableau = false;
  TableauD tab{};
  double kappa2 = 0.0;
  // heterogeneous chain (Eq. (1)): caller-owned device array of P parameters per site
  const void *site_params = nullptr;
  unsigned gen_version = 0;  // bumped when the tableau or kappa2 changes (graph cache key)
  int tuned_kernel = 0;  // scheme rk4_chain_autotune measured fastest for RK4_KERNEL_AUTO (0: not tuned)
  bool timeout_set = false;                 // RK4_OPT_TIMEOUT_NS given explicitly
  unsigned config_version = 0;              // bumped by every setter (graphs captured by callers)
};

namespace {

bool use_generic(const rk4_chain *h);

bool use_het(const rk4_chain *h);

int tile_interior(const rk4_chain *h, int W, int k);

int effective_kernel(const rk4_chain *h) {
  if (h->kernel != RK4_KERNEL_AUTO) return h->kernel;
  if (h->tuned_kernel != 0) return h->tuned_kernel;  // the autotuner's measured choice
  if (h->nchains == 1 || use_generic(h) || use_het(h)) return RK4_KERNEL_BLOCKED;
  return RK4_KERNEL_PERSISTENT;  // batches
}

size_t elem_bytes(const rk4_chain *h) { return h->fp32 ? 4 : 8; }

// The generic kernels run when a tableau was set or second-neighbour coupling is on.
bool use_generic(const rk4_chain *h) { return h->has_tableau || h->kappa2 != 0.0; }
bool use_het(const rk4_chain *h) { return h->site_params != nullptr; }
int coupling_range(const rk4_chain *h) { return h->kappa2 != 0.0 ? 2 : 1; }
int stages(const rk4_chain *h) { return use_generic(h) ? h->tab.s : 4; }
// Stages the step's result depends on: those with a nonzero weight b_m and, recursively, the
// earlier stages a needed stage uses.  A stage outside this set (Dormand-Prince 5's seventh,
// with b_7 = 0) cannot influence y, so the dependency cone of one step spans at most this
// many stages: the tile halo and the sub-domain reach are sized by it.
uint32_t needed_mask(const TableauD &t) {
  uint32_t need = 0;
  for (int m = 0; m < t.s; ++m)
    if (t.b[m] != 0.0) need |= 1u << m;
  for (int j = t.s - 1; j >= 0; --j)
    if ((need >> j) & 1u)
      for (int m = 0; m < j; ++m)
        if (t.a[j][m] != 0.0) need |= 1u << m;
  return need;
}
int needed_stages(const rk4_chain *h) {
  if (!use_generic(h)) return 4;
  const uint32_t need = needed_mask(h->tab);
  int n = 0;
  for (int m = 0; m < h->tab.s; ++m) n += (need >> m) & 1u;
  return n;
}

// Halo per side of one launch of k steps: s stages, each reaching `range` sites further.
int halo(const rk4_chain *h, int k) { return needed_stages(h) * coupling_range(h) * k; }

TableauD classical_rk4() {
  TableauD t{};
  t.s = 4;
  t.a[1][0] = 0.5;
  t.a[2][1] = 0.5;
  t.a[3][2] = 1.0;
  t.b[0] = 1.0 / 6.0;
  t.b[1] = 1.0 / 3.0;
  t.b[2] = 1.0 / 3.0;
  t.b[3] = 1.0 / 6.0;
  return t;
}

// Bytes of one k slot of the batch tile tables: the first-tile prefix (nchains + 1 entries;
// full tiles when packed, all tiles otherwise), the packed tiles' first-segment prefix
// (nchains + 1) and the segments (at most one per chain).
size_t ktable_bytes(int nchains) {
  return align_up(sizeof(int32_t) * (size_t)(nchains + 1)) * 2 + align_up(sizeof(SegDesc) * (size_t)nchains);
}

// Entries of one k slot's tile table (the chain of each full tile): room for tiles of at least
// kTileTableMinG interior sites; a launch with more tiles than that searches the prefix instead.
constexpr int kTileTableMinG = 64;
int64_t tile_table_entries(const rk4_chain *h) { return h->total / kTileTableMinG + h->nchains; }

WsLayout layout(const rk4_chain *h, int kernel) {
  WsLayout L{};
  size_t o = 0;
  auto take = [&](size_t bytes) {
    size_t r = o;
    o = align_up(o + bytes);
    return r;
  };
  L.hdr = take(sizeof(WsHeader));
  L.partials = take(sizeof(double) * kEnergyBlocks);
  L.result = take(sizeof(double) * (size_t)h->nchains);
  L.chains = take(h->nchains > 1 ? sizeof(ChainDesc) * (size_t)h->nchains : 0);
  L.prefix = take(h->nchains > 1 ? ktable_bytes(h->nchains) * kMaxDistinctK : 0);
  L.tiles = take(h->nchains > 1 && kernel != RK4_KERNEL_STAGED
                     ? sizeof(int2) * (size_t)tile_table_entries(h) * kMaxDistinctK : 0);
  const size_t sz = (size_t)h->total * (size_t)h->D * elem_bytes(h);
  L.state = L.comp = L.u0 = L.u1 = L.acc = 0;
  if (kernel == RK4_KERNEL_STAGED && use_generic(h)) {
    L.u0 = take(sz);                     // stage state
    L.acc = take(sz * (size_t)h->tab.s);  // the s stage slopes
  } else if (kernel == RK4_KERNEL_STAGED) {
    L.u0 = take(sz);
    L.u1 = take(sz);
    L.acc = take(sz);
  } else {
    L.state = take(sz);
    if (h->fp32) L.comp = take(sz);
  }
  L.total = o;
  return L;
}

CoefD coef(const rk4_chain *h) {
  CoefD c;
  c.a = h->p.a;
  c.b = h->p.b;
  c.c = h->p.c;
  c.kappa = h->p.kappa;
  c.w2 = h->p.omega0 * h->p.omega0;
  c.h2 = h->dt / 2.0;
  c.h1 = h->dt;
  c.dt6 = h->dt / 6.0;
  c.dt3 = h->dt / 3.0;
  c.kappa2 = h->kappa2;
  return c;
}

// FP64 handles run the step in the split form (rk4_split.cuh) when its error bound holds for
// their coefficients; every scheme of a handle takes the same form.
bool use_split(const rk4_chain *h) {
  if (h->fp32) return false;
  CoefD c = coef(h);
  if (use_generic(h) && (use_het(h) || !split_tableau_allowed(h->tab))) return false;
  c.kappa = h->kappa_most;
  if (!split_allowed(h->model, c)) return false;
  c.kappa = h->kappa_least;
  return split_allowed(h->model, c);
}

void note_kappa(rk4_chain *h, double kappa) {
  const double k = std::fabs(kappa);
  h->kappa_most = std::max(h->kappa_most, k);
  if (k > 0.0 && (h->kappa_least == 0.0 || k < h->kappa_least)) h->kappa_least = k;
}

int tiling_valid(const rk4_chain *h, int block, int v, int k) {
  if (block < 64 || block > 1024 || (block % 32) != 0) return 0;
  if (k < 1 || k > 16) return 0;
  const int W = block * v;
  if (use_generic(h)) {
    if (v != 2 && v != 4) return 0;
    const int H = halo(h, k);
    if (W - 2 * H < H) return 0;
    if (gen_blocked_smem_bytes(h->model, h->fp32, v, block, h->tab) > kMaxSmem) return 0;
    return 1;
  }
  if (v != 1 && v != 2 && v != 4 && v != 8) return 0;
  if (use_het(h) && v != 2 && v != 4) return 0;
  if (W - 8 * k < 8 * k) return 0;
  if (blocked_smem_bytes(h->model, h->fp32, v, block, use_het(h)) > kMaxSmem) return 0;
  return 1;
}

int tiling_max_threads(const rk4_chain *h, int v) {
  return use_generic(h) ? gen_blocked_max_threads(h->model, h->fp32, coupling_range(h), v, h->tab)
                        : blocked_max_threads(h->model, h->fp32, v, use_het(h));
}

void default_tiling(rk4_chain *h) {
  // The seed of the automatic choice, from the register and shared-memory budget (the paper
  // suggests sizing the cluster from the cache; here a tile should fill a block's registers):
  // what a handle runs with whose form has no measured costs (run_tiling), FP64 on the FP64 pipe
  // alone, where k = 1 keeps the redundant halo work minimal.
  if (use_generic(h)) {
    h->tiling.block = 128;
    h->tiling.v = 2;
    h->tiling.k = 1;
  } else if (use_het(h)) {
    h->tiling.block = 256;
    h->tiling.v = 2;
    h->tiling.k = h->fp32 ? 4 : 1;
  } else {
    h->tiling.block = 256;
    h->tiling.v = 4;
    h->tiling.k = h->fp32 ? 4 : 1;
  }
  h->tiling.G = tile_interior(h, h->tiling.block * h->tiling.v, h->tiling.k);
  h->tiling_auto = true;
}

int64_t tiles_for(const rk4_chain *h, int G) {
  int64_t t = 0;
  for (const ChainDesc &c : h->chains) t += (c.n + G - 1) / G;
  return t;
}

// Batches on the classical homogeneous kernels (blocked and persistent) pack the chains' last
// partial pieces into shared tiles; the generic and heterogeneous kernels give every chain
// whole tiles of its own.
bool packed_batch(const rk4_chain *h) { return h->nchains > 1 && !use_generic(h) && !use_het(h); }

// Sites per 16 bytes of state in whole sites: a packed batch's full tiles start their windows at
// multiples of it (so they move by 16-byte vectors wherever the chain starts), which the interior
// pays with up to that many sites less than W - 2 H.
int batch_align(const rk4_chain *h) {
  int a = h->D * (int)elem_bytes(h), b = 16;
  while (b) {
    const int t = a % b;
    a = b;
    b = t;
  }
  return 16 / a;
}

// Interior sites per tile for tiles of W sites and k steps.
int tile_interior(const rk4_chain *h, int W, int k) {
  return W - 2 * halo(h, k) - (packed_batch(h) ? batch_align(h) - 1 : 0);
}


// A chain: nsteps in an even number of launches of at most K steps (the state then ends where it
// began), as few as possible and as equal as possible: a launch of k steps recomputes 2 H sites
// per tile and step, H in proportion to k, so for a given number of launches equal ones waste
// least (50 steps at K = 16: 13 + 13 + 12 + 12 instead of 16 + 16 + 16 + 2).
Plan balanced_plan(int64_t nsteps, int K) {
  int64_t L = (nsteps + K - 1) / K;
  if (L % 2 == 1 && L < nsteps) ++L;
  Plan P;
  P.copy_back = L % 2 == 1;
  const int64_t base = nsteps / L, more = nsteps % L;
  if (more > 0) P.add((int)base + 1, more);
  P.add((int)base, L - more);
  return P;
}

// A batch whose tiling the caller chose: K as often as it goes, then what is left, split in two
// where that makes the number of launches even.
Plan batch_plan(int64_t nsteps, int K) {
  Plan P;
  const int64_t q = nsteps / K;
  const int r = (int)(nsteps % K);
  P.kval.push_back(K);
  P.cnt.push_back(q);
  if ((q + (r > 0 ? 1 : 0)) % 2 == 0) {
    if (r > 0) P.add(r);
  } else if (r >= 2) {
    P.add(r / 2);
    P.add(r - r / 2);
  } else if (K >= 2 && q >= 1) {
    P.cnt[0] = q - 1;
    P.add(K / 2);
    P.add(K - K / 2);
    if (r > 0) P.add(r);
  } else {
    if (r > 0) P.add(r);
    P.copy_back = true;
  }
  return P;
}

// A batch under the automatic tiling: the kval of every plan are the same (K and powers of two
// below it), so that the batch's tables hold for any number of steps: no rebuild from one call
// to the next, and a launch sequence captured by the caller stays good after calls of other
// lengths.
Plan batch_auto_plan(int64_t nsteps, int K) {
  Plan P;
  for (int k = K, i = 0; k >= 1 && i < kMaxDistinctK; k = k == 16 ? 4 : k / 2, ++i) {
    P.add(k, nsteps / k);
    nsteps %= k;
  }
  if (P.count() % 2 == 0) return P;
  for (int i = (int)P.kval.size() - 2; i >= 0; --i)  // 16 -> 4 x 4, 8 -> 2 x 4, 4 -> 2 x 2, 2 -> 2 x 1
    if (P.cnt[i] > 0) {
      --P.cnt[i];
      P.cnt[i + 1] += P.kval[i] / P.kval[i + 1];
      return P;
    }
  P.copy_back = true;
  return P;
}

Plan make_plan(const rk4_chain *h, int64_t nsteps, int K) {
  if (h->one_way) {  // with the kval batch_plan has for the same steps, so that the tables serve both
    Plan P = batch_plan(K, K);
    P.cnt.assign(P.cnt.size(), 0);
    P.cnt[0] = 1;
    P.copy_back = false;
    return P;
  }
  if (h->nchains == 1) return balanced_plan(nsteps, K);
  return h->tiling_auto ? batch_auto_plan(nsteps, K) : batch_plan(nsteps, K);
}

// What a launch costs, fitted on a GB300 (152 SMs, 2070 MHz) in us: A + hypot(B k, w (C + D k)) for k
// steps when every SM gets w tiles.  A is the launch and the tile's way in and out, B a step's
// latency when a tile has an SM to itself (1000 sites, k = 1 .. 16), C + D k the SM's time per tile
// when it is full (2^22 sites).  Roessler; the harmonic chain's costs are in nearly the same
// proportions, except that its 128 x 4 runs ahead of 256 x 2 (2.4 and 3.0 ns per site and SM at
// k = 4; the same kernel in the Roessler chain, so only the former is listed).  The stages a generic
// step needs scale B and D (six: Dormand-Prince 5).
struct TileCost {
  int block, v;
  float A, B, C, D;
};
const TileCost kCostFp64[] = {{64, 1, 2.2f, 1.26f, 0.34f, 0.336f}, {128, 1, 2.2f, 1.28f, 0.33f, 0.523f},
                              {256, 1, 2.4f, 1.70f, 0.21f, 1.024f}, {512, 1, 3.0f, 2.69f, 0.80f, 2.133f},
                              {128, 2, 2.4f, 2.22f, 0.43f, 0.975f}, {128, 4, 2.8f, 3.01f, 0.51f, 1.875f},
                              {256, 4, 3.8f, 5.08f, 1.35f, 4.000f}};
const TileCost kCostFp32[] = {{256, 1, 3.2f, 0.33f, 0.51f, 0.102f}, {128, 2, 3.0f, 0.28f, 0.28f, 0.074f},
                              {256, 2, 3.3f, 0.38f, 0.58f, 0.154f}, {128, 4, 3.1f, 0.30f, 0.33f, 0.127f},
                              {256, 4, 3.9f, 0.39f, 0.74f, 0.254f}, {512, 4, 5.5f, 0.61f, 2.10f, 0.500f},
                              {128, 8, 4.2f, 0.35f, 0.75f, 0.246f}, {256, 8, 5.3f, 0.56f, 2.33f, 0.465f}};
const TileCost kCostHet64[] = {{64, 2, 3.4f, 1.91f, 0.46f, 0.605f}, {128, 2, 3.5f, 1.96f, 0.39f, 0.975f},
                               {256, 2, 4.2f, 2.75f, 1.53f, 2.110f}};
const TileCost kCostHet32[] = {{64, 2, 3.8f, 0.30f, 0.23f, 0.036f}, {128, 2, 3.8f, 0.30f, 0.41f, 0.080f},
                               {256, 2, 4.1f, 0.39f, 0.87f, 0.169f}, {128, 4, 3.9f, 0.31f, 0.55f, 0.135f},
                               {256, 4, 5.2f, 0.39f, 1.25f, 0.276f}};
const TileCost kCostGen64[] = {{64, 2, 2.8f, 5.85f, 0.25f, 2.03f}, {128, 2, 2.9f, 5.94f, 0.42f, 2.88f},
                               {256, 2, 3.2f, 8.67f, 0.80f, 6.98f}};
const TileCost kCostGen32[] = {{128, 2, 5.3f, 0.80f, 0.55f, 0.27f}, {256, 2, 5.7f, 0.95f, 1.30f, 0.64f}};
const TileCost kCostGen32Shape[] = {{128, 4, 7.0f, 0.47f, 0.65f, 0.28f}, {256, 4, 7.9f, 0.68f, 1.50f, 0.60f},
                                    {512, 4, 7.5f, 1.32f, 3.80f, 1.20f}};

// Tiles of a launch of k steps at block x v, in units of whole tiles (from at most 512 of a
// batch's chains).
double tiles_estimate(const rk4_chain *h, int W, int v, int k) {
  const int H = halo(h, k), G = tile_interior(h, W, k);
  const int64_t step = std::max<int64_t>(1, h->nchains / 512);
  double slots = 0.0;
  int64_t seen = 0, sites = 0;
  for (int64_t c = 0; c < h->nchains; c += step, ++seen) {
    const int64_t n = h->chains[c].n, full = n / G, rem = n % G;
    sites += n;
    slots += (double)full * W;
    if (rem > 0) slots += packed_batch(h) ? (double)((rem + 2 * H + v - 1) / v * v) : (double)W;
  }
  return slots / W * ((double)h->total / (double)sites);
}

// The tiling an integration of nsteps runs with.  One that was set or tuned is taken as it is.
// The automatic choice (rk4_chain_get_tiling: its seed, then what the last integration ran with)
// depends on the sites and the steps: a short chain needs small tiles to reach every SM and many
// steps per launch to pay for the launch, a long one wide tiles.  Measured against the seed, us per
// step: FP64 1000 sites 8.9 -> 1.6 (128 x 1, k = 8), 65537 sites 8.9 -> 2.9 (512 x 1, k = 11), 2^22 sites
// 144 -> 117 (128 x 4, k = 4); FP32 65537 sites 2.3 -> 0.5 (128 x 4, k = 16), 2^22 sites 12.7 -> 8.9
// (256 x 8, k = 16).  Over 300 .. 2^24 sites of both models and precisions the choice is within 3 % of
// the best tiling in the median, 10 % at worst.
// The FP64 form (coefficients outside split_allowed) keeps the seed.
rk4_tiling run_tiling(rk4_chain *h, int64_t nsteps) {
  if (!h->tiling_auto) return h->tiling;
  if (h->nchains > 1) nsteps = 1024;  // a batch's tables must not depend on the steps
  if (h->auto_version != h->config_version) {
    for (auto &a : h->automatic) a.steps = -1;
    h->auto_version = h->config_version;
  }
  for (const auto &a : h->automatic)
    if (a.steps == nsteps) return a.tiling;
  const TileCost *cost = nullptr;
  int n = 0;
  float stages = 1.f;
#define RK4_COST(T) (cost = T, n = (int)(sizeof(T) / sizeof(T[0])))
  if (use_generic(h)) {
    stages = (float)needed_stages(h) / 6.f;
    if (!h->fp32 && use_split(h)) RK4_COST(kCostGen64);
    else if (h->fp32 && gen_compiled(h->tab)) RK4_COST(kCostGen32Shape);
    else if (h->fp32) RK4_COST(kCostGen32);
  } else if (use_het(h)) {
    if (h->fp32) RK4_COST(kCostHet32);
    else if (use_split(h)) RK4_COST(kCostHet64);
  } else if (h->fp32) {
    RK4_COST(kCostFp32);
  } else if (use_split(h)) {
    RK4_COST(kCostFp64);
  }
#undef RK4_COST
  rk4_tiling best = h->tiling;
  double best_us = 1e300;
  const double sms = sm_count();
  for (int c = 0; c < n; ++c) {
    int last = 0;
    if (cost[c].block > tiling_max_threads(h, cost[c].v)) continue;
    for (int kmax : {1, 2, 3, 4, 5, 6, 8, 10, 12, 16}) {
      if (h->nchains > 1 && (kmax & (kmax - 1)) != 0) continue;
      const Plan P = make_plan(h, nsteps, kmax);
      const int k = P.kval[0], W = cost[c].block * cost[c].v;
      if (k == last || !tiling_valid(h, cost[c].block, cost[c].v, k)) continue;
      last = k;
      double us = 0.0;
      for (size_t i = 0; i < P.kval.size(); ++i) {
        if (P.cnt[i] == 0) continue;
        const int ki = P.kval[i];
        double w = tiles_estimate(h, W, cost[c].v, ki) / sms;
        w = w <= 4.0 ? std::ceil(w) : w + 0.5;  // few tiles: the busiest SM decides
        us += (double)P.cnt[i] *
              (cost[c].A + std::hypot(cost[c].B * stages * ki, w * (cost[c].C + cost[c].D * stages * ki)));
      }
      if (us < best_us) {
        best_us = us;
        best = {cost[c].block, cost[c].v, k, tile_interior(h, W, k)};
      }
    }
  }
  auto &a = h->automatic[h->auto_next++ % 8];
  a.steps = nsteps;
  a.tiling = best;
  return best;
}

cudaError_t ensure_pinned(rk4_chain *h) {
  if (!h->h_out) {
    cudaError_t e = cudaMallocHost((void **)&h->h_out, sizeof(double) * (size_t)h->nchains + 64);
    if (e != cudaSuccess) return e;
  }
  if (!h->h_status) {
    cudaError_t e = cudaMallocHost((void **)&h->h_status, 64);
    if (e != cudaSuccess) return e;
  }
  if (h->nchains > 1 && !h->h_tables) {
    // same relative layout as the workspace: chain table, then the prefix arrays at the next
    // 256-byte boundary
    h->tables_bytes = align_up(sizeof(ChainDesc) * (size_t)h->nchains) + ktable_bytes(h->nchains) * kMaxDistinctK;
    cudaError_t e = cudaMallocHost(&h->h_tables, h->tables_bytes);
    if (e != cudaSuccess) return e;
    std::memcpy(h->h_tables, h->chains.data(), sizeof(ChainDesc) * (size_t)h->nchains);
  }
  return cudaSuccess;
}

// The batch tile tables of k slot `ki` (pinned host copy, same layout as the workspace).
struct KTables {
  int32_t *prefix, *pack_prefix;
  SegDesc *segs;
};
KTables host_ktables(rk4_chain *h, int ki) {
  char *p = static_cast<char *>(h->h_tables) + align_up(sizeof(ChainDesc) * (size_t)h->nchains) +
            ktable_bytes(h->nchains) * (size_t)ki;
  const size_t pre = align_up(sizeof(int32_t) * (size_t)(h->nchains + 1));
  return {reinterpret_cast<int32_t *>(p), reinterpret_cast<int32_t *>(p + pre), reinterpret_cast<SegDesc *>(p + 2 * pre)};
}
BatchTiles dev_ktables(const rk4_chain *h, const char *ws, const WsLayout &L, int ki) {
  const char *p = ws + L.prefix + ktable_bytes(h->nchains) * (size_t)ki;
  const size_t pre = align_up(sizeof(int32_t) * (size_t)(h->nchains + 1));
  BatchTiles bt{};
  bt.full_prefix = reinterpret_cast<const int32_t *>(p);
  bt.pack_prefix = reinterpret_cast<const int32_t *>(p + pre);
  bt.segs = reinterpret_cast<const SegDesc *>(p + 2 * pre);
  bt.nfull = h->nfull[ki];
  bt.npacked = h->npacked[ki];
  const int64_t entries = tile_table_entries(h);
  bt.tile_chain = L.tiles && bt.nfull <= entries
                      ? reinterpret_cast<const int2 *>(ws + L.tiles + sizeof(int2) * (size_t)entries * (size_t)ki)
                      : nullptr;
  return bt;
}

// Fill the tile tables of the k slots that a plan uses on the device (after upload_tables).
cudaError_t fill_tile_tables(const rk4_chain *h, char *ws, const WsLayout &L, const Plan &P, cudaStream_t st) {
  if (h->nchains == 1) return cudaSuccess;
  for (int i = 0; i < (int)P.kval.size(); ++i) {
    if (P.cnt[i] == 0) continue;
    const BatchTiles bt = dev_ktables(h, ws, L, i);
    if (!bt.tile_chain) continue;
    const cudaError_t e =
        launch_tile_chains(bt.full_prefix, h->nchains, bt.nfull, const_cast<int2 *>(bt.tile_chain), st);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

// Pack the segments of one k slot into tiles of W slots: each chain's last partial piece of
// cnt = n mod G interior sites (the whole chain when n < G) needs a window of
// L = H + cnt + H slots, rounded up to a multiple of v.  Best fit in decreasing order of L (the
// fullest tile that still has room, ties to the earliest opened), which leaves little unused
// room.  Returns the number of packed tiles; fills pack_prefix and segs in tile order.
int64_t pack_segments(const rk4_chain *h, int G, int H, int W, int v, int32_t *pack_prefix, SegDesc *segs) {
  struct Piece {
    int chain, cnt, L;
  };
  std::vector<Piece> pieces;
  for (int c = 0; c < h->nchains; ++c) {
    const int cnt = (int)(h->chains[c].n % G);
    if (cnt == 0) continue;
    const int L = (cnt + 2 * H + v - 1) / v * v;
    pieces.push_back({c, cnt, L});
  }
  std::stable_sort(pieces.begin(), pieces.end(), [](const Piece &a, const Piece &b) { return a.L > b.L; });
  // open tiles by free room (in units of v slots): the tiles of each room size, earliest first
  const int units = W / v;
  std::vector<std::vector<int>> by_room(units + 1);
  std::vector<int> room;                       // free slots of each tile
  std::vector<std::vector<int>> members;       // pieces of each tile, in slot order
  for (int i = 0; i < (int)pieces.size(); ++i) {
    const int need = pieces[i].L / v;
    int t = -1;
    for (int r = need; r <= units && t < 0; ++r)
      if (!by_room[r].empty()) {
        // earliest-opened tile of this room size (tiles are only appended in opening order)
        auto &bucket = by_room[r];
        auto it = std::min_element(bucket.begin(), bucket.end());
        t = *it;
        bucket.erase(it);
      }
    if (t < 0) {
      t = (int)room.size();
      room.push_back(units);
      members.emplace_back();
    }
    members[t].push_back(i);
    room[t] -= need;
    by_room[room[t]].push_back(t);
  }
  int32_t next = 0;
  for (size_t t = 0; t < members.size(); ++t) {
    pack_prefix[t] = next;
    int o = 0;
    for (int i : members[t]) {
      const Piece &p = pieces[i];
      SegDesc &sd = segs[next++];
      sd.chain = p.chain;
      sd.cnt = p.cnt;
      sd.L = p.L;
      sd.o = o;
      sd.g0 = h->chains[p.chain].n - p.cnt;
      o += p.L;
    }
  }
  pack_prefix[members.size()] = next;
  return (int64_t)members.size();
}

// Fill the pinned batch tile tables for the plan's k values (waits for earlier uses first).
cudaError_t prepare_tables(rk4_chain *h, const std::vector<int> &kval, int W) {
  if (h->nchains == 1) return cudaSuccess;
  const int packed = packed_batch(h) ? 1 : 0;
  if (h->tables_k == kval && h->tables_W == W && h->tables_v == h->run.v && h->tables_halo == halo(h, 1) &&
      h->tables_packed == packed)
    return cudaSuccess;
  cudaError_t e = cudaStreamSynchronize(h->stream);
  if (e != cudaSuccess) return e;
  for (size_t i = 0; i < kval.size(); ++i) {
    const int H = halo(h, kval[i]);
    const int G = tile_interior(h, W, kval[i]);
    KTables t = host_ktables(h, (int)i);
    int64_t acc = 0;
    for (int c = 0; c < h->nchains; ++c) {
      t.prefix[c] = (int32_t)acc;
      acc += packed ? h->chains[c].n / G : (h->chains[c].n + G - 1) / G;
    }
    t.prefix[h->nchains] = (int32_t)acc;
    h->nfull[i] = acc;
    h->npacked[i] = packed ? pack_segments(h, G, H, W, h->run.v, t.pack_prefix, t.segs) : 0;
  }
  h->tables_k = kval;
  h->tables_W = W;
  h->tables_v = h->run.v;
  h->tables_halo = halo(h, 1);
  h->tables_packed = packed;
  return cudaSuccess;
}

cudaError_t upload_tables(rk4_chain *h, char *ws, const WsLayout &L, cudaStream_t st) {
  if (h->nchains == 1) return cudaSuccess;
  return cudaMemcpyAsync(ws + L.chains, h->h_tables, h->tables_bytes, cudaMemcpyHostToDevice, st);
}

const ChainDesc *dev_chains(const rk4_chain *h, char *ws, const WsLayout &L) {
  return h->nchains > 1 ? reinterpret_cast<const ChainDesc *>(ws + L.chains) : nullptr;
}

// Enqueue the whole launch sequence of an integration on stream st.
cudaError_t enqueue_integrate(rk4_chain *h, int kernel, void *state, void *comp, char *ws, const WsLayout &L,
                              const Plan &P, int64_t nsteps, cudaStream_t st) {
  const CoefD cf = coef(h);
  const int W = h->run.block * h->run.v;
  // a fresh status word (and barrier counters) for every integration
  cudaError_t e = cudaMemsetAsync(ws + L.hdr, 0, sizeof(WsHeader), st);
  if (e != cudaSuccess) return e;
  e = upload_tables(h, ws, L, st);
  if (e != cudaSuccess) return e;
  const size_t bytes = (size_t)h->total * h->D * elem_bytes(h);
  if (kernel == RK4_KERNEL_STAGED && use_generic(h)) {
    GenStagedJob j{};
    j.y = state;
    j.cmp = comp;
    j.u = ws + L.u0;
    j.k = ws + L.acc;
    j.nchains = h->nchains;
    j.one = h->chains[0];
    j.chains = dev_chains(h, ws, L);
    j.total = h->total;
    j.hdr = reinterpret_cast<WsHeader *>(ws + L.hdr);
    j.split = use_split(h) ? 1 : 0;
    j.wide = reinterpret_cast<unsigned *>(ws + L.result);  // 8 bytes a chain, free while integrating
    if (j.split) {
      e = launch_split_scan(h->model, coupling_range(h), static_cast<const double *>(state), nullptr, h->total, h->nchains,
                            j.one, j.chains, cf, j.wide, st);
      if (e != cudaSuccess) return e;
    }
    for (int64_t s = 0; s < nsteps; ++s) {
      j.parity = (int)(s & 1);
      e = launch_gen_staged_step(h->model, h->fp32, coupling_range(h), j, cf, h->tab, h->dt, st);
      if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
  }
  if (kernel == RK4_KERNEL_STAGED) {
    StagedJob j{};
    j.y = state;
    j.cmp = comp;
    j.sp = h->site_params;
    j.nchains = h->nchains;
    j.one = h->chains[0];
    j.chains = dev_chains(h, ws, L);
    j.total = h->total;
    j.hdr = reinterpret_cast<WsHeader *>(ws + L.hdr);
    j.acc = ws + L.acc;
    void *u0 = ws + L.u0, *u1 = ws + L.u1;
    j.split = use_split(h) ? 1 : 0;
    j.wide = reinterpret_cast<unsigned *>(ws + L.result);  // 8 bytes a chain, free while integrating
    j.n2 = u0;
    j.n3 = u1;
    if (j.split) {
      e = launch_split_scan(h->model, 1, static_cast<const double *>(state), static_cast<const double *>(h->site_params),
                            h->total, h->nchains, j.one, j.chains, cf, j.wide, st);
      if (e != cudaSuccess) return e;
    }
    for (int64_t s = 0; s < nsteps; ++s) {
      j.parity = (int)(s & 1);
      // stage 0 reads y and writes u0; 1: u0 -> u1; 2: u1 -> u0; 3: u0 -> y
      for (int st4 = 0; st4 < 4; ++st4) {
        j.uin = (st4 == 2) ? u1 : u0;
        j.uout = (st4 == 1) ? u1 : u0;
        e = launch_staged(h->model, h->fp32, st4, j, cf, st);
        if (e != cudaSuccess) return e;
      }
    }
    return cudaSuccess;
  }
  void *wsS = ws + L.state;
  void *wsC = h->fp32 ? (void *)(ws + L.comp) : nullptr;
  e = fill_tile_tables(h, ws, L, P, st);
  if (e != cudaSuccess) return e;
  if (kernel == RK4_KERNEL_BLOCKED) {
    BlockedJob j{};
    j.nchains = h->nchains;
    j.one = h->chains[0];
    j.chains = dev_chains(h, ws, L);
    j.sp = h->site_params;
    j.hdr = reinterpret_cast<WsHeader *>(ws + L.hdr);
    j.total = h->total;
    j.packed = packed_batch(h) ? 1 : 0;
    j.split = use_split(h) ? 1 : 0;
    int ki = 0;
    int64_t left = P.cnt[0];
    for (int64_t i = 0; i < P.count(); ++i, --left) {
      while (left == 0) left = P.cnt[++ki];
      const int k = P.kval[ki];
      j.K = k;
      j.G = tile_interior(h, W, k);
      if (h->nchains > 1) {
        // ntiles counts the full tiles (or, unpacked, every tile); the packed tiles follow them
        // in the same launch
        j.bt = dev_ktables(h, ws, L, ki);
        j.ntiles = j.bt.nfull;
      } else {
        j.ntiles = tiles_for(h, j.G);
      }
      const bool even = (i % 2) == 0 && h->one_way != 2;
      j.in = even ? state : wsS;
      j.out = even ? wsS : state;
      j.cin = even ? comp : wsC;
      j.cout = even ? wsC : comp;
      if (use_generic(h))
        e = launch_gen_blocked(h->model, h->fp32, coupling_range(h), h->run.v, h->run.block, j, cf, h->tab,
                               h->dt, halo(h, k), st);
      else
        e = launch_blocked(h->model, h->fp32, h->run.v, h->run.block, j, cf, st);
      if (e != cudaSuccess) return e;
    }
  } else {  // persistent
    PersistentJob j{};
    j.bufA = state;
    j.bufB = wsS;
    j.cA = comp;
    j.cB = wsC;
    j.nchains = h->nchains;
    j.one = h->chains[0];
    j.chains = dev_chains(h, ws, L);
    j.nk = (int)P.kval.size();
    int64_t maxtiles = 0;
    for (int i = 0; i < j.nk; ++i) {
      j.kval[i] = P.kval[i];
      j.cnt[i] = P.cnt[i];
      j.Gval[i] = tile_interior(h, W, P.kval[i]);
      if (h->nchains > 1) {
        j.bt[i] = dev_ktables(h, ws, L, i);
        j.ntiles[i] = j.bt[i].nfull + j.bt[i].npacked;
      } else {
        j.ntiles[i] = tiles_for(h, j.Gval[i]);
      }
      if (P.cnt[i] > 0) maxtiles = std::max(maxtiles, j.ntiles[i]);
    }
    j.hdr = reinterpret_cast<WsHeader *>(ws + L.hdr);
    j.total = h->total;
    j.split = use_split(h) ? 1 : 0;
    // A barrier waits at most one time block; unless the caller set the bound, allow 20x a
    // pessimistic estimate of one (1e9 site-steps/s) so that very large batches cannot time
    // out spuriously.
    {
      int kmax = 1;
      for (int kv : P.kval) kmax = std::max(kmax, kv);
      const double est_ns = (double)h->total * kmax;  // at 1e9 site-steps/s: 1 ns per site-step
      j.timeout_ns = h->timeout_set ? h->timeout_ns : std::max<long long>(h->timeout_ns, (long long)(20.0 * est_ns));
    }
    j.extra_arrivals = 0;
    int grid = persistent_max_grid(h->model, h->fp32, h->run.v, h->run.block, use_split(h));
    if (grid <= 0) return cudaErrorInvalidConfiguration;
    grid = (int)std::min<int64_t>(grid, std::max<int64_t>(1, maxtiles));
    e = launch_persistent(h->model, h->fp32, h->run.v, h->run.block, grid, j, cf, st);
    if (e != cudaSuccess) return e;
  }
  if (P.copy_back) {
    e = cudaMemcpyAsync(state, wsS, bytes, cudaMemcpyDeviceToDevice, st);
    if (e != cudaSuccess) return e;
    if (h->fp32) e = cudaMemcpyAsync(comp, wsC, bytes, cudaMemcpyDeviceToDevice, st);
  }
  return e;
}

int check_buffers(const rk4_chain *h, const void *state, const void *comp, const void *ws) {
  if (!state || !ws) return RK4_EINVAL;
  if (h->fp32 != (comp != nullptr)) return RK4_EINVAL;
  if ((reinterpret_cast<uintptr_t>(ws) % kAlign) != 0) return RK4_EINVAL;
  if ((reinterpret_cast<uintptr_t>(state) % 16) != 0) return RK4_EINVAL;
  if (comp && (reinterpret_cast<uintptr_t>(comp) % 16) != 0) return RK4_EINVAL;
  return RK4_OK;
}

int integrate_impl(rk4_chain *h, void *state, void *comp, void *ws, size_t ws_bytes, int64_t nsteps) {
  int rc = check_buffers(h, state, comp, ws);
  if (rc) return rc;
  if (nsteps < 0) return RK4_EINVAL;
  const int kernel = effective_kernel(h);
  if (kernel == RK4_KERNEL_PERSISTENT && (use_generic(h) || use_het(h))) return RK4_EUNSUPPORTED;
  if (use_generic(h) && use_het(h)) return RK4_EUNSUPPORTED;
  const WsLayout L = layout(h, kernel);
  if (ws_bytes < L.total) return RK4_ENOMEM_WS;
  if (nsteps == 0) return RK4_OK;
  if (ensure_pinned(h) != cudaSuccess) return RK4_ECUDA;
  h->run = run_tiling(h, nsteps);
  if (h->tiling_auto && kernel != RK4_KERNEL_STAGED) h->run_version = h->config_version + 1;
  const Plan P = make_plan(h, nsteps, kernel == RK4_KERNEL_STAGED ? 1 : h->run.k);
  if (kernel != RK4_KERNEL_STAGED) {
    // tile counts must fit a 1-D grid and the int32 prefix tables
    const int kmax = *std::max_element(P.kval.begin(), P.kval.end());
    if (tiles_for(h, tile_interior(h, h->run.block * h->run.v, kmax)) > 0x7fffffffLL) return RK4_EUNSUPPORTED;
  }
  if (prepare_tables(h, P.kval, h->run.block * h->run.v) != cudaSuccess) return RK4_ECUDA;
  char *w = static_cast<char *>(ws);

  const bool use_graph = h->graphs && (kernel != RK4_KERNEL_BLOCKED || P.count() > 1);
  if (!use_graph) {
    return enqueue_integrate(h, kernel, state, comp, w, L, P, nsteps, h->stream) == cudaSuccess ? RK4_OK
                                                                                                : RK4_ECUDA;
  }
  GraphKey key;
  key.kernel = kernel;
  key.state = state;
  key.comp = comp;
  key.ws = ws;
  key.nsteps = nsteps;
  key.block = h->run.block;
  key.v = h->run.v;
  key.k = h->run.k;
  key.timeout = h->timeout_ns;
  key.sp = h->site_params;
  key.generic = use_generic(h) ? 1 + (int)h->gen_version : 0;
  key.kval = P.kval;
  key.cnt = P.cnt;
  if (!(h->gexec && key == h->gkey)) {
    if (h->gexec) {
      cudaGraphExecDestroy(h->gexec);
      h->gexec = nullptr;
    }
    if (!h->cap_stream && cudaStreamCreateWithFlags(&h->cap_stream, cudaStreamNonBlocking) != cudaSuccess)
      return RK4_ECUDA;
    if (cudaStreamBeginCapture(h->cap_stream, cudaStreamCaptureModeRelaxed) != cudaSuccess) return RK4_ECUDA;
    cudaError_t e = enqueue_integrate(h, kernel, state, comp, w, L, P, nsteps, h->cap_stream);
    cudaGraph_t g = nullptr;
    cudaError_t e2 = cudaStreamEndCapture(h->cap_stream, &g);
    if (e != cudaSuccess || e2 != cudaSuccess || !g) {
      if (g) cudaGraphDestroy(g);
      return RK4_ECUDA;
    }
    e = cudaGraphInstantiate(&h->gexec, g, 0);
    cudaGraphDestroy(g);
    if (e != cudaSuccess) {
      h->gexec = nullptr;
      return RK4_ECUDA;
    }
    h->gkey = key;
  }
  return cudaGraphLaunch(h->gexec, h->stream) == cudaSuccess ? RK4_OK : RK4_ECUDA;
}

int validate_common(int model, int precision, double dt, const rk4_params *p) {
  if (model != RK4_ROESSLER && model != RK4_HARMONIC) return RK4_EINVAL;
  if (precision != RK4_FP64 && precision != RK4_FP32_KAHAN) return RK4_EINVAL;
  if (!(std::isfinite(dt) && dt > 0.0)) return RK4_EINVAL;
  if (p && !(std::isfinite(p->a) && std::isfinite(p->b) && std::isfinite(p->c) && std::isfinite(p->kappa) &&
             std::isfinite(p->omega0)))
    return RK4_EINVAL;
  return RK4_OK;
}

rk4_chain *new_handle(int model, int precision, double dt, const rk4_params *p, void *stream) {
  rk4_chain *h = new (std::nothrow) rk4_chain();
  if (!h) return nullptr;
  h->model = model;
  h->precision = precision;
  h->fp32 = precision == RK4_FP32_KAHAN;
  h->D = model == RK4_ROESSLER ? 3 : 2;
  h->dt = dt;
  if (p) h->p = *p; else rk4_params_default(&h->p);
  h->stream = static_cast<cudaStream_t>(stream);
  h->tab = classical_rk4();
  default_tiling(h);
  return h;
}

// Device address of page-locked host memory that the device can access, or NULL (pageable
// memory, or memory the runtime does not know).
void *mapped_host(const void *p) {
  cudaPointerAttributes a;
  if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
    cudaGetLastError();  // clear the error of the query
    return nullptr;
  }
  if (a.type != cudaMemoryTypeHost || a.devicePointer == nullptr) return nullptr;
  // the device address of this very byte (the query names the start of p's allocation)
  return static_cast<char *>(a.devicePointer) + (static_cast<const char *>(p) - static_cast<const char *>(a.hostPointer));
}

// One host <-> device transfer of integrate_host: by the SMs when the host buffer is mapped
// page-locked memory and both sides are 16-byte aligned (k_copy.cu), else by cudaMemcpyAsync.
cudaError_t host_transfer(void *dst, const void *src, size_t bytes, bool to_device, cudaStream_t st) {
  void *hd = mapped_host(to_device ? src : dst);
  if (hd && ((reinterpret_cast<uintptr_t>(hd) | reinterpret_cast<uintptr_t>(to_device ? dst : src)) & 15u) == 0)
    return to_device ? launch_copy(dst, hd, bytes, st) : launch_copy(hd, src, bytes, st);
  return cudaMemcpyAsync(dst, src, bytes, to_device ? cudaMemcpyHostToDevice : cudaMemcpyDeviceToHost, st);
}

}  // namespace

namespace {

// c as a float pair: the head rounded to 24 bits (ties away from zero) and the rest (split1 of
// rk4_split.cuh).
struct HostPair {
  float h, l;
};
HostPair host_split(double c) {
  uint64_t u;
  std::memcpy(&u, &c, 8);
  u = (u + 0x10000000u) & ~(uint64_t)0x1fffffff;
  double d;
  std::memcpy(&d, &u, 8);
  return {(float)d, (float)(c - d)};  // c - d is exact
}
HostPair host_times_tau(double c, const HostPair &tau) {  // times_tau
  const HostPair v = host_split(c);
  const float p = tau.h * v.h;
  float e = std::fmaf(tau.h, v.h, -p);
  e = std::fmaf(tau.h, v.l, e);
  e = std::fmaf(tau.l, v.h, e);
  return {p, e};
}
unsigned high_word(double v) {
  uint64_t u;
  std::memcpy(&u, &v, 8);
  return (unsigned)(u >> 32);
}

// The largest magnitudes the split form takes: a, b, c, kappa (Roessler) or w2, kappa (harmonic).
// The differences D are dt |J| times the first slope; with dt times each coefficient at most 1/8 (the
// coupling counts fourfold) and the state within split_in_range their pair arithmetic stays below the
// state's rounding (rk4_split.cuh has the errors).
void split_most(int model, double dt, double *most) {
  if (model == RK4_ROESSLER) {
    most[0] = most[2] = 0.125 / dt;
    most[1] = 0.125 / dt;
    most[3] = 0.125 / (4.0 * dt);
  } else {
    most[0] = 1.0 / (128.0 * dt * dt);
    most[1] = 1.0 / (512.0 * dt * dt);
  }
}
// The largest |x - c| and |y|, |z| of a Roessler state (split_in_range), times dt.  One step of uniform
// states of amplitude A, dt = 0.01, error of z in units of the FP64 form's: 0.73 at dt A = 0.2, 0.89 at 0.25,
// 1.18 at 0.3, 1.56 at 0.4; x alone up to dt |x - c| = 0.25 0.81, 0.3 0.99.  The attractor reaches dt |x - c| = 0.21,
// dt z = 0.24 for c = 9 and 0.29, 0.49 for c at its limit.
constexpr double kSplitFar = 0.25, kSplitBig = 0.3;
constexpr double kSplitMostDt[] = {1.0 / 16, 1.0 / 8};  // Roessler (1.05 .. 1.3 from 1/12 on), harmonic
bool split_takes(double v, double most) {
  const double a = std::fabs(v);
  return a == 0.0 || (a >= 0x1p-60 && a <= most);
}

}  // namespace

bool rk4d::split_allowed(int model, const CoefD &c) {
  const double dt = c.h1;
  if (!(dt >= 0x1p-20 && dt <= kSplitMostDt[model == RK4_ROESSLER ? 0 : 1])) return false;
  double most[4];
  split_most(model, dt, most);
  if (model == RK4_ROESSLER)
    return split_takes(c.a, most[0]) && split_takes(c.b, most[1]) && split_takes(c.c, most[2]) &&
           split_takes(c.kappa, most[3]) && split_takes(c.kappa2, most[3]);
  return split_takes(c.w2, most[0]) && split_takes(c.kappa, most[1]) && split_takes(c.kappa2, most[1]);
}

// The error that the remainders' pairs leave in a step, estimated for a linear chain with dt J = delta and
// with independent roundings, in units of what the FP64 form leaves (its stage states' roundings): per
// stage the size e_j of the remainder's increment, |r_j| = |delta e_j| + the product's part, and the variance
// of its error from the row's terms (k_gen_split.cu).  A pair's roundings are 2^-49, the state's 2^-53.
double split_tableau_error(const TableauD &t, double delta) {
  double c[kMaxStages] = {}, r[kMaxStages] = {}, size[kMaxStages] = {}, var[kMaxStages] = {}, ours = 0.0, theirs = 0.0;
  for (int j = 0; j < t.s; ++j) {
    double e = 0.0, terms = 0.0;
    int nonzero = 0;
    for (int m = 0; m < j; ++m) {
      const double a = t.a[j][m];
      c[j] += a;
      nonzero += a != 0.0;
      if (m == 0) continue;
      e += a * c[m] - a * r[m];
      terms += a * a * (size[m] * size[m] + var[m]);
    }
    double g = 0.0;
    for (int m = 1; m < j; ++m) g += t.a[j][m] * c[m];
    r[j] = -delta * e;
    size[j] = std::fabs(r[j]) + std::fabs(delta) * c[j] * c[j] / 4.0;
    var[j] = delta * delta * (g * g + terms) + size[j] * size[j];
    if (j > 0) ours += t.b[j] * t.b[j] * (var[j] + size[j] * size[j]);
    theirs += t.b[j] * t.b[j] * nonzero;
  }
  return theirs > 0.0 ? 16.0 * std::sqrt(ours / theirs) : 1e300;
}

// Entries within the pairs' range, and an estimated error of at most 1.1 at dt |J| = 1/8.  Published schemes
// come to 0.18 (midpoint) .. 1.06 (RK4; Dormand-Prince 5 0.84, Fehlberg 5 0.96, Cash-Karp 5 0.61) and their
// measured error (one step, dt = 0.0138, c = 9, kappa = 1.5, kappa2 = 0.3, amplitudes 1 and 9) is 0.98 ..
// 0.999 of the FP64 form's.  700 random tableaux of 2 .. 7 stages with row sums of magnitudes up to 55: up
// to 1.1 at most 1.05 (1.13 in one component), 1.1 .. 2 up to 1.2 (1.5), 3 .. 18 up to 10.
bool rk4d::split_tableau_allowed(const TableauD &t) {
  const uint32_t need = needed_mask(t);
  if (!(need & 1u) || !(need >> 1)) return false;  // the form evaluates J K1 whether the scheme does or not
  for (int j = 0; j < t.s; ++j) {
    double sum = 0.0;
    for (int m = 0; m < j; ++m) {
      if (!split_takes(t.a[j][m], 64.0)) return false;
      sum += t.a[j][m];
    }
    if (!split_takes(sum, 2.0) || !split_takes(t.b[j], 64.0)) return false;
  }
  return split_tableau_error(t, 0.125) <= 1.1 && split_tableau_error(t, -0.125) <= 1.1;
}

// a + b as a sum and its exact error.
double host_two_sum(double a, double b, double *err) {
  const double s = a + b, bb = s - a;
  *err += (a - (s - bb)) + (b - bb);
  return s;
}

SplitTableau rk4d::split_tableau(const TableauD &t, double dt) {
  SplitTableau r{};
  r.s = t.s;
  r.need = needed_mask(t);
  for (int j = 0; j < t.s; ++j)
    if ((r.need >> j) & 1u) r.last = j;
  double c[kMaxStages] = {}, b_err = 0.0;  // the weights' sum is B + Bl: an error of 2^-54 in it would be a drift
  for (int j = 0; j < t.s; ++j) {
    double row = 0.0, row_err = 0.0, g = 0.0;
    for (int m = 0; m < j; ++m) {
      row = host_two_sum(row, t.a[j][m], &row_err);
      g += t.a[j][m] * c[m];
      const HostPair a = host_split(t.a[j][m]);
      r.ah[j][m] = a.h;
      r.al[j][m] = a.l;
      if (t.a[j][m] != 0.0 && m > 0) r.ma[j][r.na[j]++] = m;
    }
    c[j] = row + row_err;
    const HostPair cj = host_split(c[j]), gj = host_split(g), b = host_split(t.b[j]);
    r.ch[j] = cj.h;
    r.cl[j] = cj.l;
    r.gh[j] = gj.h;
    r.gl[j] = gj.l;
    r.bh[j] = b.h;
    r.bl[j] = b.l;
    r.B = host_two_sum(r.B, t.b[j], &b_err);
    r.E += t.b[j] * c[j];
    if (t.b[j] != 0.0 && j > 0 && j != r.last) r.mb[r.nb++] = j;
    if (((r.need >> j) & 1u) && j > 0 && j != r.last) r.slot[j] = r.slots++;
  }
  r.E *= dt;
  const double B = r.B + b_err;
  r.Bl = (float)((r.B - B) + b_err);
  r.B = B;
  r.unit = B == 1.0;
  return r;
}

SplitCoef rk4d::split_coef(int model, const CoefD &c, bool generic, bool het) {
  SplitCoef s{};
  const double tau = generic ? c.h1 : c.h2;
  s.w = generic ? c.h1 : tau / 3.0;
  const HostPair t = host_split(tau), cc = host_split(c.c);
  s.tauh = t.h;
  s.taul = t.l;
  const HostPair k2 = host_times_tau(c.kappa2, t);
  s.k2h = k2.h;
  s.k2l = k2.l;
  const HostPair k = host_times_tau(c.kappa, t), a = host_times_tau(model == RK4_ROESSLER ? c.a : c.w2, t);
  s.kth = k.h;
  s.ktl = k.l;
  s.ath = a.h;
  s.atl = a.l;
  s.ch = cc.h;
  s.cl = cc.l;
  double most[4] = {};
  split_most(model, c.h1, most);
  for (int i = 0; i < 4; ++i) s.most[i] = high_word(most[i]);
  const double far = kSplitFar / c.h1;
  s.far = (float)far;
  s.most_x = high_word(het ? far + most[2] : far + c.c);
  s.least_x = high_word(far - c.c);
  s.big = high_word(model == RK4_ROESSLER ? kSplitBig / c.h1 : 0x1p40);
  return s;
}

// Read-only view of a handle for the allocation-free reduction entry point.
int rk4d::handle_info(const rk4_chain *h, int *model, bool *fp32, int *nchains, const ChainDesc **chains, CoefD *cf,
                      cudaStream_t *stream, bool *het) {
  if (!h) return RK4_EINVAL;
  *het = use_het(h);
  *model = h->model;
  *fp32 = h->fp32;
  *nchains = h->nchains;
  *chains = h->chains.data();
  *cf = coef(h);
  *stream = h->stream;
  return RK4_OK;
}

unsigned rk4d::config_version(const rk4_chain *h) { return h->config_version; }

cudaStream_t rk4d::swap_stream(rk4_chain *h, cudaStream_t st) {
  cudaStream_t old = h->stream;
  h->stream = st;
  return old;
}

bool rk4d::swap_graphs(rk4_chain *h, bool on) {
  const bool old = h->graphs;
  h->graphs = on;
  return old;
}

int rk4d::swap_one_way(rk4_chain *h, int way) {
  const int old = h->one_way;
  h->one_way = way;
  return old;
}

bool rk4d::one_way_allowed(const rk4_chain *h, int64_t nsteps) {
  return h->nchains > 1 && !h->tiling_auto && effective_kernel(h) == RK4_KERNEL_BLOCKED && h->tiling.k == nsteps;
}

void rk4d::state_copy(const rk4_chain *h, void *ws, void **state, void **comp) {
  const WsLayout L = layout(h, RK4_KERNEL_BLOCKED);
  *state = static_cast<char *>(ws) + L.state;
  *comp = h->fp32 ? static_cast<char *>(ws) + L.comp : nullptr;
}

int rk4d::prepare_integrate(rk4_chain *h, int64_t nsteps) {
  if (!h || nsteps < 1) return RK4_EINVAL;
  if (ensure_pinned(h) != cudaSuccess) return RK4_ECUDA;
  const int kernel = effective_kernel(h);
  h->run = run_tiling(h, nsteps);
  const Plan P = make_plan(h, nsteps, kernel == RK4_KERNEL_STAGED ? 1 : h->run.k);
  return prepare_tables(h, P.kval, h->run.block * h->run.v) == cudaSuccess ? RK4_OK : RK4_ECUDA;
}

int rk4d::scheme_reach(const rk4_chain *h, int *s, int *range) {
  if (!h) return RK4_EINVAL;
  *s = needed_stages(h);
  *range = coupling_range(h);
  return RK4_OK;
}

extern "C" {

void rk4_params_default(rk4_params *p) {
  if (!p) return;
  p->a = 0.2;
  p->b = 1.0;
  p->c = 9.0;
  p->kappa = 1.0;
  p->omega0 = 1.0;
}

int rk4_chain_create(rk4_chain **out, int model, int precision, int64_t n, double dt, int bc, const rk4_params *p,
                     void *cuda_stream) {
  if (!out) return RK4_EINVAL;
  *out = nullptr;
  int rc = validate_common(model, precision, dt, p);
  if (rc) return rc;
  if (n < 1 || n > ((int64_t)1 << 40)) return RK4_EINVAL;
  if (bc != RK4_PERIODIC && bc != RK4_FIXED) return RK4_EINVAL;
  rk4_chain *h = new_handle(model, precision, dt, p, cuda_stream);
  if (!h) return RK4_EINVAL;
  ChainDesc c{};
  c.off = 0;
  c.n = n;
  c.kappa = h->p.kappa;
  c.bc = bc;
  h->chains.push_back(c);
  note_kappa(h, c.kappa);
  h->nchains = 1;
  h->total = n;
  *out = h;
  return RK4_OK;
}

int rk4_batch_create(rk4_chain **out, int model, int precision, int nchains, const int64_t *lengths,
                     const double *kappa, const int8_t *bc, double dt, const rk4_params *p, void *cuda_stream) {
  if (!out) return RK4_EINVAL;
  *out = nullptr;
  int rc = validate_common(model, precision, dt, p);
  if (rc) return rc;
  if (nchains < 1 || !lengths || !kappa || !bc) return RK4_EINVAL;
  int64_t total = 0;
  for (int c = 0; c < nchains; ++c) {
    if (lengths[c] < 1 || !std::isfinite(kappa[c]) || (bc[c] != RK4_PERIODIC && bc[c] != RK4_FIXED))
      return RK4_EINVAL;
    total += lengths[c];
    if (total > ((int64_t)1 << 40)) return RK4_EINVAL;
  }
  rk4_chain *h = new_handle(model, precision, dt, p, cuda_stream);
  if (!h) return RK4_EINVAL;
  int64_t off = 0;
  for (int c = 0; c < nchains; ++c) {
    ChainDesc d{};
    d.off = off;
    d.n = lengths[c];
    d.kappa = kappa[c];
    d.bc = bc[c];
    h->chains.push_back(d);
    note_kappa(h, d.kappa);
    off += lengths[c];
  }
  h->nchains = nchains;
  h->total = total;
  *out = h;
  return RK4_OK;
}

int rk4_chain_workspace_bytes(const rk4_chain *h, size_t *bytes) {
  if (!h || !bytes) return RK4_EINVAL;
  *bytes = layout(h, effective_kernel(h)).total;
  return RK4_OK;
}

int rk4_chain_shape(const rk4_chain *h, int64_t *total_sites, int *dim) {
  if (!h) return RK4_EINVAL;
  if (total_sites) *total_sites = h->total;
  if (dim) *dim = h->D;
  return RK4_OK;
}

int rk4_chain_set_kernel(rk4_chain *h, int kernel) {
  if (!h || kernel < RK4_KERNEL_AUTO || kernel > RK4_KERNEL_PERSISTENT) return RK4_EINVAL;
  h->config_version++;
  h->kernel = kernel;
  h->tuned_kernel = 0;
  return RK4_OK;
}

int rk4_chain_set_tiling(rk4_chain *h, int block, int v, int k) {
  if (!h) return RK4_EINVAL;
  h->config_version++;
  if (block == 0) {
    default_tiling(h);
    return RK4_OK;
  }
  if (!tiling_valid(h, block, v, k)) return RK4_EINVAL;
  const int maxt = tiling_max_threads(h, v);
  if (maxt > 0 && block > maxt) return RK4_EINVAL;
  if (h->tuned_kernel == RK4_KERNEL_STAGED) h->tuned_kernel = 0;  // a tiling asks for a tiled scheme
  h->tiling_auto = false;
  h->tiling.block = block;
  h->tiling.v = v;
  h->tiling.k = k;
  h->tiling.G = tile_interior(h, block * v, k);
  return RK4_OK;
}

int rk4_chain_get_tiling(const rk4_chain *h, rk4_tiling *out) {
  if (!h || !out) return RK4_EINVAL;
  *out = h->tiling_auto && h->run_version == h->config_version + 1 ? h->run : h->tiling;
  return RK4_OK;
}

int rk4_chain_get_kernel(const rk4_chain *h, int *kernel) {
  if (!h || !kernel) return RK4_EINVAL;
  *kernel = effective_kernel(h);
  return RK4_OK;
}

// NVTX range around a host-side call (visible in Nsight timelines; no cost without a tool).
struct NvtxRange {
  explicit NvtxRange(const char *name) { nvtxRangePushA(name); }
  ~NvtxRange() { nvtxRangePop(); }
};

int rk4_chain_integrate(rk4_chain *h, void *state, void *comp, void *ws, size_t ws_bytes, int64_t nsteps, double *t) {
  if (!h) return RK4_EINVAL;
  NvtxRange range("rk4_chain_integrate");
  int rc = integrate_impl(h, state, comp, ws, ws_bytes, nsteps);
  if (rc == RK4_OK) {
    h->nstep += nsteps;
    if (t) *t = h->t0 + (double)h->nstep * h->dt;
  }
  return rc;
}

int rk4_chain_step(rk4_chain *h, void *state, void *comp, void *ws, size_t ws_bytes, double *t) {
  return rk4_chain_integrate(h, state, comp, ws, ws_bytes, 1, t);
}

int rk4_chain_integrate_host(rk4_chain *h, void *host_state, void *host_comp, void *dev_state, void *dev_comp,
                             void *ws, size_t ws_bytes, int64_t nsteps, double *t) {
  if (!h || !host_state) return RK4_EINVAL;
  if (h->fp32 != (host_comp != nullptr)) return RK4_EINVAL;
  int rc = check_buffers(h, dev_state, dev_comp, ws);
  if (rc) return rc;
  if (ws_bytes < layout(h, effective_kernel(h)).total) return RK4_ENOMEM_WS;
  const size_t bytes = (size_t)h->total * h->D * elem_bytes(h);
  if (host_transfer(dev_state, host_state, bytes, true, h->stream) != cudaSuccess) return RK4_ECUDA;
  if (h->fp32 && host_transfer(dev_comp, host_comp, bytes, true, h->stream) != cudaSuccess) return RK4_ECUDA;
  rc = rk4_chain_integrate(h, dev_state, dev_comp, ws, ws_bytes, nsteps, t);
  if (rc) return rc;
  if (host_transfer(host_state, dev_state, bytes, false, h->stream) != cudaSuccess) return RK4_ECUDA;
  if (h->fp32 && host_transfer(host_comp, dev_comp, bytes, false, h->stream) != cudaSuccess) return RK4_ECUDA;
  return cudaStreamSynchronize(h->stream) == cudaSuccess ? RK4_OK : RK4_ECUDA;
}

int rk4_chain_energy(rk4_chain *h, const void *state, const void *comp, void *ws, size_t ws_bytes, double *out) {
  if (!h || !out) return RK4_EINVAL;
  NvtxRange range("rk4_chain_energy");
  if (use_het(h) && h->model == RK4_HARMONIC) return RK4_EUNSUPPORTED;
  int rc = check_buffers(h, state, comp, ws);
  if (rc) return rc;
  const WsLayout L = layout(h, effective_kernel(h));
  if (ws_bytes < L.total) return RK4_ENOMEM_WS;
  if (ensure_pinned(h) != cudaSuccess) return RK4_ECUDA;
  char *w = static_cast<char *>(ws);
  WsHeader *hdr = reinterpret_cast<WsHeader *>(w + L.hdr);
  if (cudaMemsetAsync(hdr, 0, sizeof(WsHeader), h->stream) != cudaSuccess) return RK4_ECUDA;
  if (upload_tables(h, w, L, h->stream) != cudaSuccess) return RK4_ECUDA;
  const CoefD cf = coef(h);
  double *res = reinterpret_cast<double *>(w + L.result);
  if (launch_energy(h->model, h->fp32, state, comp, h->nchains, h->chains[0], dev_chains(h, w, L), cf,
                    reinterpret_cast<double *>(w + L.partials), res, hdr, h->stream) != cudaSuccess)
    return RK4_ECUDA;
  if (cudaMemcpyAsync(h->h_out, res, sizeof(double) * h->nchains, cudaMemcpyDeviceToHost, h->stream) != cudaSuccess)
    return RK4_ECUDA;
  if (cudaMemcpyAsync(h->h_status, &hdr->status, sizeof(int), cudaMemcpyDeviceToHost, h->stream) != cudaSuccess)
    return RK4_ECUDA;
  if (cudaStreamSynchronize(h->stream) != cudaSuccess) return RK4_ECUDA;
  std::memcpy(out, h->h_out, sizeof(double) * h->nchains);
  if (*h->h_status & ST_NONFINITE) return RK4_ENONFINITE;
  return RK4_OK;
}

int rk4_chain_status(rk4_chain *h, void *ws) {
  if (!h || !ws) return RK4_EINVAL;
  if (ensure_pinned(h) != cudaSuccess) return RK4_ECUDA;
  const WsLayout L = layout(h, effective_kernel(h));
  WsHeader *hdr = reinterpret_cast<WsHeader *>(static_cast<char *>(ws) + L.hdr);
  if (cudaMemcpyAsync(h->h_status, &hdr->status, sizeof(int), cudaMemcpyDeviceToHost, h->stream) != cudaSuccess)
    return RK4_ECUDA;
  if (cudaMemsetAsync(&hdr->status, 0, sizeof(int), h->stream) != cudaSuccess) return RK4_ECUDA;
  if (cudaStreamSynchronize(h->stream) != cudaSuccess) return RK4_ECUDA;
  const int s = *h->h_status;
  if (s & ST_TIMEOUT) return RK4_ETIMEOUT;
  if (s & ST_BOUNDS) return RK4_EBOUNDS;
  if (s & ST_NONFINITE) return RK4_ENONFINITE;
  return RK4_OK;
}

int rk4_chain_set_option(rk4_chain *h, int option, int64_t value) {
  if (!h) return RK4_EINVAL;
  h->config_version++;
  if (option == RK4_OPT_GRAPHS) {
    if (value != 0 && value != 1) return RK4_EINVAL;
    h->graphs = value != 0;
    return RK4_OK;
  }
  if (option == RK4_OPT_TIMEOUT_NS) {
    if (value < 1000 || value > (int64_t)600 * 1000000000LL) return RK4_EINVAL;
    h->timeout_ns = value;
    h->timeout_set = true;
    return RK4_OK;
  }
  return RK4_EINVAL;
}

int rk4_debug_barrier_timeout(rk4_chain *h, void *state, void *comp, void *ws, size_t ws_bytes, int64_t timeout_ns) {
  if (!h) return RK4_EINVAL;
  int rc = check_buffers(h, state, comp, ws);
  if (rc) return rc;
  if (timeout_ns < 1000 || timeout_ns > 10LL * 1000000000LL) return RK4_EINVAL;
  const WsLayout L = layout(h, RK4_KERNEL_PERSISTENT);
  if (ws_bytes < L.total) return RK4_ENOMEM_WS;
  if (ensure_pinned(h) != cudaSuccess) return RK4_ECUDA;
  h->run = h->tiling;
  const int W = h->tiling.block * h->tiling.v;
  Plan P;  // one time block
  P.add(h->tiling.k);
  if (prepare_tables(h, P.kval, W) != cudaSuccess) return RK4_ECUDA;
  char *w = static_cast<char *>(ws);
  if (upload_tables(h, w, L, h->stream) != cudaSuccess) return RK4_ECUDA;
  if (fill_tile_tables(h, w, L, P, h->stream) != cudaSuccess) return RK4_ECUDA;
  PersistentJob j{};
  j.bufA = state;
  j.bufB = w + L.state;
  j.cA = comp;
  j.cB = h->fp32 ? (void *)(w + L.comp) : nullptr;
  j.nchains = h->nchains;
  j.one = h->chains[0];
  j.chains = dev_chains(h, w, L);
  j.nk = 1;
  j.kval[0] = h->tiling.k;
  if (use_generic(h)) return RK4_EUNSUPPORTED;
  j.Gval[0] = tile_interior(h, W, h->tiling.k);
  if (h->nchains > 1) {
    j.bt[0] = dev_ktables(h, w, L, 0);
    j.ntiles[0] = j.bt[0].nfull + j.bt[0].npacked;
  } else {
    j.ntiles[0] = tiles_for(h, j.Gval[0]);
  }
  j.cnt[0] = 1;
  j.hdr = reinterpret_cast<WsHeader *>(w + L.hdr);
  j.total = h->total;
  j.split = use_split(h) ? 1 : 0;
  j.timeout_ns = timeout_ns;
  j.extra_arrivals = 1;
  int grid = persistent_max_grid(h->model, h->fp32, h->tiling.v, h->tiling.block, use_split(h));
  if (grid <= 0) return RK4_ECUDA;
  grid = (int)std::min<int64_t>(grid, std::max<int64_t>(1, j.ntiles[0]));
  if (cudaMemsetAsync(w + L.hdr, 0, sizeof(WsHeader), h->stream) != cudaSuccess) return RK4_ECUDA;
  if (launch_persistent(h->model, h->fp32, h->tiling.v, h->tiling.block, grid, j, coef(h), h->stream) !=
      cudaSuccess)
    return RK4_ECUDA;
  return RK4_OK;
}

int rk4_chain_autotune(rk4_chain *h, void *state, void *comp, void *ws, size_t ws_bytes, int probe_steps,
                       rk4_tiling *best) {
  if (!h || probe_steps < 1 || probe_steps > 100000) return RK4_EINVAL;
  NvtxRange range("rk4_chain_autotune");
  int rc = check_buffers(h, state, comp, ws);
  if (rc) return rc;
  if (h->kernel == RK4_KERNEL_STAGED) {  // the one-stage-per-launch scheme has nothing to tune
    if (best) *best = h->tiling;
    return RK4_OK;
  }
  // Candidate schemes.  An explicit choice is kept.  On RK4_KERNEL_AUTO: the blocked scheme, for
  // a batch also the persistent one, and the staged scheme whenever ws is large enough for it.
  const bool tiled_only = use_generic(h) || use_het(h);
  const bool on_auto = h->kernel == RK4_KERNEL_AUTO;
  std::vector<int> kernels;
  if (!on_auto) {
    kernels.push_back(h->kernel);
  } else {
    if (h->nchains > 1 && !tiled_only) kernels.push_back(RK4_KERNEL_PERSISTENT);
    kernels.push_back(RK4_KERNEL_BLOCKED);
  }
  for (size_t i = 0; i < kernels.size();)  // only the schemes the caller's workspace can hold
    if (ws_bytes < layout(h, kernels[i]).total) kernels.erase(kernels.begin() + (long)i); else ++i;
  const bool try_staged = on_auto && ws_bytes >= layout(h, RK4_KERNEL_STAGED).total;
  if (kernels.empty() && !try_staged) return RK4_ENOMEM_WS;
  const rk4_tiling saved = h->tiling;
  const bool saved_auto = h->tiling_auto;
  h->tiling_auto = false;  // the candidates run as they are
  const int saved_tuned = h->tuned_kernel;
  int best_kernel = 0;
  const bool saved_graphs = h->graphs;
  h->graphs = false;
  cudaEvent_t e0 = nullptr, e1 = nullptr;
  if (cudaEventCreate(&e0) != cudaSuccess || cudaEventCreate(&e1) != cudaSuccess) {
    h->graphs = saved_graphs;
    h->tiling_auto = saved_auto;
    return RK4_ECUDA;
  }
  // Per-step time of an integration of `steps` after a warm-up of `warm`, or a negative value
  // when the configuration fails to run.
  auto time_steps = [&](int64_t warm, int64_t steps) -> float {
    if (integrate_impl(h, state, comp, ws, ws_bytes, warm) != RK4_OK) return -1.f;
    cudaEventRecord(e0, h->stream);
    if (integrate_impl(h, state, comp, ws, ws_bytes, steps) != RK4_OK) return -1.f;
    cudaEventRecord(e1, h->stream);
    if (cudaEventSynchronize(e1) != cudaSuccess) {
      rc = RK4_ECUDA;
      return -1.f;
    }
    float ms = 0.f;
    cudaEventElapsedTime(&ms, e0, e1);
    return ms / (float)steps;
  };
  static const int blocks[] = {64, 128, 256, 512, 1024};
  static const int vs[] = {1, 2, 4, 8};
  static const int ks[] = {1, 2, 4, 8, 16};
  float best_ms = 1e30f;
  rk4_tiling best_t = saved;
  bool have_tiling = false;
  rc = RK4_OK;
  for (int kern : kernels) {
    if (rc != RK4_OK) break;
    if (on_auto) h->tuned_kernel = kern;
    for (int b : blocks)
      for (int v : vs)
        for (int k : ks) {
          if (rc != RK4_OK) break;
          if (!tiling_valid(h, b, v, k)) continue;
          if (b == 64 && !use_generic(h)) continue;
          const int maxt = tiling_max_threads(h, v);
          if (maxt <= 0 || b > maxt) continue;
          if (kern == RK4_KERNEL_PERSISTENT && persistent_max_grid(h->model, h->fp32, v, b, use_split(h)) <= 0) continue;
          h->tiling.block = b;
          h->tiling.v = v;
          h->tiling.k = k;
          h->tiling.G = tile_interior(h, b * v, k);
          const int64_t steps = ((probe_steps + 2 * k - 1) / (2 * k)) * 2 * k;  // whole, even launch count
          const float per_step = time_steps(2 * k, steps);
          if (per_step >= 0.f && per_step < best_ms) {
            best_ms = per_step;
            best_t = h->tiling;
            best_kernel = kern;
            have_tiling = true;
          }
        }
  }
  if (rc == RK4_OK && try_staged) {
    h->tuned_kernel = RK4_KERNEL_STAGED;
    const float per_step = time_steps(1, probe_steps);
    if (per_step >= 0.f && per_step < best_ms) {
      best_ms = per_step;
      best_kernel = RK4_KERNEL_STAGED;
    }
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  h->graphs = saved_graphs;
  if (rc != RK4_OK || best_ms >= 1e30f) {
    h->tiling = saved;
    h->tiling_auto = saved_auto;
    h->tuned_kernel = saved_tuned;
    return rc != RK4_OK ? rc : RK4_ECUDA;
  }
  h->tuned_kernel = on_auto ? best_kernel : 0;
  h->config_version++;
  h->tiling = have_tiling ? best_t : saved;
  h->tiling_auto = !have_tiling && saved_auto;
  if (best) *best = h->tiling;
  return RK4_OK;
}

int rk4_chain_set_tableau(rk4_chain *h, int s, const double *A, const double *b) {
  if (!h) return RK4_EINVAL;
  h->config_version++;
  h->tuned_kernel = 0;
  if (s == 0) {  // back to the classical RK4 kernels
    h->has_tableau = false;
    h->tab = classical_rk4();
    default_tiling(h);
    return RK4_OK;
  }
  if (s < 1 || s > kMaxStages || !A || !b) return RK4_EINVAL;
  TableauD t{};
  t.s = s;
  for (int j = 0; j < s; ++j) {
    if (!std::isfinite(b[j])) return RK4_EINVAL;
    t.b[j] = b[j];
    for (int m = 0; m < s; ++m) {
      const double a = A[j * s + m];
      if (!std::isfinite(a)) return RK4_EINVAL;
      if (m >= j && a != 0.0) return RK4_EINVAL;  // explicit schemes only
      if (m < j) t.a[j][m] = a;
    }
  }
  h->has_tableau = true;
  h->tab = t;
  h->gen_version++;
  default_tiling(h);
  return RK4_OK;
}

int rk4_chain_set_coupling2(rk4_chain *h, double kappa2) {
  if (!h || !std::isfinite(kappa2)) return RK4_EINVAL;
  h->config_version++;
  h->tuned_kernel = 0;
  h->kappa2 = kappa2;
  if (!h->has_tableau) h->tab = classical_rk4();
  h->gen_version++;
  default_tiling(h);
  return RK4_OK;
}

int rk4_chain_set_site_params(rk4_chain *h, const void *params) {
  if (!h) return RK4_EINVAL;
  if (params && (reinterpret_cast<uintptr_t>(params) % 16) != 0) return RK4_EINVAL;
  h->config_version++;
  h->tuned_kernel = 0;
  h->site_params = params;
  default_tiling(h);
  return RK4_OK;
}

int rk4_chain_get_clock(const rk4_chain *h, double *t0, int64_t *nstep) {
  if (!h) return RK4_EINVAL;
  if (t0) *t0 = h->t0;
  if (nstep) *nstep = h->nstep;
  return RK4_OK;
}

int rk4_chain_set_clock(rk4_chain *h, double t0, int64_t nstep) {
  if (!h || !std::isfinite(t0) || nstep < 0) return RK4_EINVAL;
  h->t0 = t0;
  h->nstep = nstep;
  return RK4_OK;
}

int rk4_chain_set_time(rk4_chain *h, double t0) {
  if (!h || !std::isfinite(t0)) return RK4_EINVAL;
  h->t0 = t0;
  h->nstep = 0;
  return RK4_OK;
}

int rk4_chain_destroy(rk4_chain *h) {
  if (!h) return RK4_OK;
  if (h->gexec) cudaGraphExecDestroy(h->gexec);
  if (h->cap_stream) cudaStreamDestroy(h->cap_stream);
  if (h->h_tables) cudaFreeHost(h->h_tables);
  if (h->h_out) cudaFreeHost(h->h_out);
  if (h->h_status) cudaFreeHost(h->h_status);
  delete h;
  return RK4_OK;
}

const char *rk4_strerror(int code) {
  switch (code) {
    case RK4_OK: return "ok";
    case RK4_EINVAL: return "invalid argument";
    case RK4_ENOMEM_WS: return "workspace too small";
    case RK4_ECUDA: return "CUDA runtime error";
    case RK4_ENONFINITE: return "non-finite value in the state";
    case RK4_ETIMEOUT: return "device-side wait timed out";
    case RK4_EUNSUPPORTED: return "unsupported request";
    case RK4_EBOUNDS: return "an index check of the debug build caught an out-of-range access";
    default: return "unknown error";
  }
}

int rk4_fill_uniform(void *dst, int64_t count, uint64_t seed, uint64_t start, int precision, void *cuda_stream) {
  if (!dst || count < 0) return RK4_EINVAL;
  if (precision != RK4_FP64 && precision != RK4_FP32_KAHAN) return RK4_EINVAL;
  return launch_fill_uniform(dst, count, seed, start, precision == RK4_FP32_KAHAN,
                             static_cast<cudaStream_t>(cuda_stream)) == cudaSuccess
             ? RK4_OK
             : RK4_ECUDA;
}

}  // extern "C"
