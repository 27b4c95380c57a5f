// k_persistent.cu -- one persistent, cooperative launch that integrates a whole batch of
// chains: for every block of k steps each resident thread block walks its share of the
// (chain, tile) items, then all blocks meet at a grid barrier before the next time block
// reads what the previous one wrote.  The barrier's wait is bounded: a block that waits
// longer than timeout_ns latches ST_TIMEOUT in the status word and the kernel returns.
#include "k_grid_barrier.cuh"
#include "rk4_tile.cuh"

namespace rk4d {

// A packed tile of a batch (the segments of item p).  Not inlined, as in the one-shot blocked
// kernel: the segment bookkeeping then takes registers only inside this call, and the full-tile
// path, which runs nearly every item, keeps its own allocation (inlined, the FP32 batch kernel
// spilled at the 64-register cap of four resident blocks per SM).
template <typename R, int MODEL, int V, bool KAHAN>
__device__ __noinline__ void persistent_packed_call(const R *in, R *out, const R *cin, R *cout,
                                                    const ChainDesc *chains, const SegDesc *segs,
                                                    const int32_t *pack_prefix, int64_t p, int K, Coef<R> cf,
                                                    unsigned char *smem, int64_t sites, WsHeader *hdr) {
  packed_tile_item<R, MODEL, V, KAHAN, true>(in, out, cin, cout, chains, segs, pack_prefix[p], pack_prefix[p + 1], K,
                                             cf, smem, sites, hdr);
}

// One full tile, of a single chain or (BATCH) of a batch, as a call of its own: the tile's
// arithmetic then gets the register budget it has in the one-shot blocked kernel, instead of
// sharing it with the persistent loop's state (time block, item, buffers), which the call saves
// once per tile.
template <typename R, int MODEL, int V, bool KAHAN, bool BATCH>
__device__ __noinline__ void persistent_tile_call(const PersistentJob &job, int ki, const R *in, R *out,
                                                  const R *cin, R *cout, int64_t item, int K, int G, Coef<R> cf,
                                                  unsigned char *smem) {
  if constexpr (!BATCH) {
    tile_item<R, MODEL, V, KAHAN, true>(in, out, cin, cout, job.one, item, K, G, cf, smem, job.total, job.hdr);
  } else {
    int64_t local;
    const int ci = batch_chain(job.bt[ki], job.nchains, item - job.bt[ki].npacked, smem, local);
    const ChainDesc ch = job.chains[ci];
    cf.kappa = (R)ch.kappa;
    tile_item<R, MODEL, V, KAHAN, true, false, true>(in, out, cin, cout, ch, local, K, G, cf, smem, job.total,
                                                     job.hdr);
  }
}

template <typename R, int MODEL, int V, bool KAHAN, bool BATCH>
__global__ void __launch_bounds__(max_threads_for(V), (V >= 2 && KAHAN) ? 2 : 1)  // FP32: two resident blocks
    k_persistent(PersistentJob job, Coef<R> cf) {
  extern __shared__ __align__(16) unsigned char smem[];
  persistent_loop(job, [&](int ki, const void *vin, void *vout, const void *vcin, void *vcout, int64_t item, int K,
                           int G) {
    const R *in = static_cast<const R *>(vin), *cin = static_cast<const R *>(vcin);
    R *out = static_cast<R *>(vout), *cout = static_cast<R *>(vcout);
    if (BATCH && item < job.bt[ki].npacked)
      persistent_packed_call<R, MODEL, V, KAHAN>(in, out, cin, cout, job.chains, job.bt[ki].segs,
                                                 job.bt[ki].pack_prefix, item, K, cf, smem, job.total, job.hdr);
    else
      persistent_tile_call<R, MODEL, V, KAHAN, BATCH>(job, ki, in, out, cin, cout, item, K, G, cf, smem);
  });
}

template <typename R, int MODEL, int V, bool KAHAN>
static cudaError_t setup_attr() {
  static PerDevice attr, attr_b;
  const cudaError_t e = set_smem_limit_once(k_persistent<R, MODEL, V, KAHAN, false>, 200 * 1024, attr);
  if (e != cudaSuccess) return e;
  return set_smem_limit_once(k_persistent<R, MODEL, V, KAHAN, true>, 200 * 1024, attr_b);
}

template <typename R, int MODEL, int V, bool KAHAN>
static cudaError_t launch_one(int block, int grid, const PersistentJob &job, const CoefD &cfd, cudaStream_t st) {
  cudaError_t e = setup_attr<R, MODEL, V, KAHAN>();
  if (e != cudaSuccess) return e;
  const size_t smem = blocked_smem_bytes(MODEL, KAHAN, V, block);
  Coef<R> cf = to_coef<R>(cfd, cfd.kappa);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3((unsigned)block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  if (job.nchains > 1) return cudaLaunchKernelEx(&cfg, k_persistent<R, MODEL, V, KAHAN, true>, job, cf);
  return cudaLaunchKernelEx(&cfg, k_persistent<R, MODEL, V, KAHAN, false>, job, cf);
}

template <typename R, int MODEL, int V, bool KAHAN>
static int max_grid_one(int block) {
  if (setup_attr<R, MODEL, V, KAHAN>() != cudaSuccess) return 0;
  int per_sm = 0;
  const size_t smem = blocked_smem_bytes(MODEL, KAHAN, V, block);
  int per_sm_b = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_persistent<R, MODEL, V, KAHAN, false>, block, smem) !=
          cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm_b, k_persistent<R, MODEL, V, KAHAN, true>, block, smem) !=
          cudaSuccess)
    return 0;
  return std::min(per_sm, per_sm_b) * sm_count();  // a grid that stays co-resident with either form
}

#define RK4_DISPATCH_V(FN, ...)                                                                   \
  switch (v) {                                                                                     \
    case 1: return fp32 ? FN<float, MODEL, 1, true>(__VA_ARGS__) : FN<double, MODEL, 1, false>(__VA_ARGS__); \
    case 2: return fp32 ? FN<float, MODEL, 2, true>(__VA_ARGS__) : FN<double, MODEL, 2, false>(__VA_ARGS__); \
    case 4: return fp32 ? FN<float, MODEL, 4, true>(__VA_ARGS__) : FN<double, MODEL, 4, false>(__VA_ARGS__); \
    case 8: return fp32 ? FN<float, MODEL, 8, true>(__VA_ARGS__) : FN<double, MODEL, 8, false>(__VA_ARGS__); \
    default: break;                                                                                \
  }

template <int MODEL>
static cudaError_t launch_m(bool fp32, int v, int block, int grid, const PersistentJob &job, const CoefD &cf,
                            cudaStream_t st) {
  RK4_DISPATCH_V(launch_one, block, grid, job, cf, st)
  return cudaErrorInvalidValue;
}

template <int MODEL>
static int max_grid_m(bool fp32, int v, int block) {
  RK4_DISPATCH_V(max_grid_one, block)
  return 0;
}

cudaError_t launch_persistent(int model, bool fp32, int v, int block, int grid, const PersistentJob &job,
                              const CoefD &cf, cudaStream_t st) {
  if (job.split)
    return model == ROESSLER ? launch_split_persistent<ROESSLER>(v, block, grid, job, cf, st)
                             : launch_split_persistent<HARMONIC>(v, block, grid, job, cf, st);
  return model == ROESSLER ? launch_m<ROESSLER>(fp32, v, block, grid, job, cf, st)
                           : launch_m<HARMONIC>(fp32, v, block, grid, job, cf, st);
}

int persistent_max_grid(int model, bool fp32, int v, int block, bool split) {
  if (split)
    return model == ROESSLER ? persistent_split_max_grid<ROESSLER>(v, block)
                             : persistent_split_max_grid<HARMONIC>(v, block);
  return model == ROESSLER ? max_grid_m<ROESSLER>(fp32, v, block) : max_grid_m<HARMONIC>(fp32, v, block);
}

}  // namespace rk4d
