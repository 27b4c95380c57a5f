// k_split.cuh -- the blocked and persistent FP64 kernels in the split form (rk4_split.cuh), and
// their launchers for one model.  Each model is instantiated in a translation unit of its own
// (k_split_roessler.cu, k_split_harmonic.cu), so that they compile side by side.
//
// What bounds it: 13 FP64 instructions per site-step (Roessler: 7 for the first slope, 6 for the
// update; harmonic 8) at 0.6 T/s allow 4.6e10 site-steps/s; beside them about 300 FP32
// operations (packed two sites per instruction, 40 T lane-operations/s) and 110 integer ones.
// Measured at N = 2^24 against the FP64 form (49 instructions, 1.23e10 site-steps/s): 3.64e10 at
// 256 x 4 x 4, 3.32e10 at 128 x 2 x 4; harmonic 6.4e10 (128 x 4 x 4) against 1.90e10.
#pragma once
#include "k_grid_barrier.cuh"
#include "rk4_tile.cuh"

namespace rk4d {

// Largest block an instantiation is compiled for.  With four sites per thread blocks of up to 256
// threads have an instantiation of their own, which may use more registers than the one for 512.
__host__ __device__ constexpr int split_small_block(int v) { return v == 4 ? 256 : max_threads_for(v); }
// Whether an instantiation parks (split_advance): with four sites per thread the Roessler step
// holds 241 registers, one block of 256 threads per SM (FP64 pipe 39 % busy); parked it fits 128
// and two blocks (76 %): N = 2^24, 256 x 4, k = 2: 2.3e10 -> 3.2e10 site-steps/s, k = 8 3.45e10.
// With two sites (114 registers instead of 128) it measured 2 % slower at 128 threads, and the
// harmonic step, which fits 126 registers as it is, 3 % slower.  Heterogeneous tiles already hold
// their parameters in shared memory.
__host__ __device__ constexpr bool split_parks(int model, int v, int nt, bool het) {
  return model == ROESSLER && !het && v == 4 && nt <= 256;
}
__host__ __device__ constexpr int split_min_blocks(int model, int v, int nt, bool het) {
  return split_parks(model, v, nt, het) ? 2 : 0;
}
template <int MODEL, int V, bool HET, int NT> static size_t split_smem_bytes(int block) {
  const size_t plain = blocked_smem_bytes(MODEL, false, V, block, HET);
  const size_t parked = sizeof(double) * ((size_t)edge_values(V) + (size_t)block * split_record_words<MODEL, V>());
  return split_parks(MODEL, V, NT, HET) ? std::max(plain, parked) : plain;
}

// An item outside the split's range, in the FP64 form.  Not inlined: it is rare, and its
// registers then do not add to the split's.
template <int MODEL, int V, bool COH, bool HET, bool ALN>
__device__ __noinline__ void wide_tile_call(const double *in, double *out, ChainDesc ch, int64_t tile, int K, int G,
                                            Coef<double> cf, unsigned char *smem, int64_t sites, WsHeader *hdr,
                                            const double *sp) {
  tile_item<double, MODEL, V, false, COH, HET, ALN, false>(in, out, nullptr, nullptr, ch, tile, K, G, cf, smem, sites,
                                                           hdr, sp);
}
template <int MODEL, int V, bool COH>
__device__ __noinline__ void wide_packed_call(const double *in, double *out, const ChainDesc *chains,
                                              const SegDesc *segs, int s0, int s1, int K, Coef<double> cf,
                                              unsigned char *smem, int64_t sites, WsHeader *hdr) {
  packed_tile_item<double, MODEL, V, false, COH, false>(in, out, nullptr, nullptr, chains, segs, s0, s1, K, cf, smem,
                                                        sites, hdr);
}
// A packed tile of a batch; not inlined for the reason given in k_blocked.cu.
template <int MODEL, int V, bool COH, bool PARK>
__device__ __noinline__ void split_packed_call(const double *in, double *out, const ChainDesc *chains,
                                               const SegDesc *segs, const int32_t *pack_prefix, int64_t p, int K,
                                               Coef<double> cf, const SplitCoef *sc, unsigned char *smem,
                                               int64_t sites, WsHeader *hdr) {
  const int s0 = pack_prefix[p], s1 = pack_prefix[p + 1];
  if (!packed_tile_item<double, MODEL, V, false, COH, true, PARK>(in, out, nullptr, nullptr, chains, segs, s0, s1, K, cf,
                                                            smem, sites, hdr, sc))
    wide_packed_call<MODEL, V, COH>(in, out, chains, segs, s0, s1, K, cf, smem, sites, hdr);
}

// The split form of k_blocked: one block per item, a packed batch's packed tiles first.
template <int MODEL, int V, bool HET, bool PACKED, int NT>
__global__ void __launch_bounds__(NT, split_min_blocks(MODEL, V, NT, HET)) k_split(BlockedJob job, Coef<double> cf, SplitCoef sc) {
  constexpr bool PARK = split_parks(MODEL, V, NT, HET);
  extern __shared__ __align__(16) unsigned char smem[];
  const double *in = static_cast<const double *>(job.in);
  double *out = static_cast<double *>(job.out);
  int64_t item = blockIdx.x;
  if constexpr (PACKED) {
    if (item < job.bt.npacked) {
      split_packed_call<MODEL, V, false, PARK>(in, out, job.chains, job.bt.segs, job.bt.pack_prefix, item, job.K, cf, &sc,
                                         smem, job.total, job.hdr);
      return;
    }
    item -= job.bt.npacked;
  }
  ChainDesc ch;
  int64_t tile = item;
  if (job.nchains == 1) {
    ch = job.one;
  } else {
    const int ci = batch_chain(job.bt, job.nchains, item, smem, tile);
    ch = job.chains[ci];
    cf.kappa = ch.kappa;
    split_set_kappa(sc, ch.kappa);
  }
  const double *sp = static_cast<const double *>(job.sp);
  if (!tile_item<double, MODEL, V, false, false, HET, PACKED, true, PARK>(in, out, nullptr, nullptr, ch, tile, job.K, job.G,
                                                                    cf, smem, job.total, job.hdr, sp, &sc))
    wide_tile_call<MODEL, V, false, HET, PACKED>(in, out, ch, tile, job.K, job.G, cf, smem, job.total, job.hdr, sp);
}

// One full tile of the persistent kernel as a call of its own (as persistent_tile_call).
template <int MODEL, int V, bool BATCH, bool PARK>
__device__ __noinline__ void persistent_split_call(const PersistentJob &job, int ki, const double *in, double *out,
                                                   int64_t item, int K, int G, Coef<double> cf, SplitCoef sc,
                                                   unsigned char *smem) {
  ChainDesc ch;
  int64_t tile = item;
  if constexpr (BATCH) {
    const int ci = batch_chain(job.bt[ki], job.nchains, item - job.bt[ki].npacked, smem, tile);
    ch = job.chains[ci];
    cf.kappa = ch.kappa;
    split_set_kappa(sc, ch.kappa);
  } else {
    ch = job.one;
  }
  if (!tile_item<double, MODEL, V, false, true, false, BATCH, true, PARK>(in, out, nullptr, nullptr, ch, tile, K, G, cf,
                                                                    smem, job.total, job.hdr, nullptr, &sc))
    wide_tile_call<MODEL, V, true, false, BATCH>(in, out, ch, tile, K, G, cf, smem, job.total, job.hdr, nullptr);
}

// The split form of k_persistent.
template <int MODEL, int V, bool BATCH, int NT>
__global__ void __launch_bounds__(NT, split_min_blocks(MODEL, V, NT, false))
    k_persistent_split(PersistentJob job, Coef<double> cf, SplitCoef sc) {
  constexpr bool PARK = split_parks(MODEL, V, NT, false);
  extern __shared__ __align__(16) unsigned char smem[];
  persistent_loop(job, [&](int ki, const void *in, void *out, const void *, void *, int64_t item, int K, int G) {
    const double *i = static_cast<const double *>(in);
    double *o = static_cast<double *>(out);
    if (BATCH && item < job.bt[ki].npacked)
      split_packed_call<MODEL, V, true, PARK>(i, o, job.chains, job.bt[ki].segs, job.bt[ki].pack_prefix, item, K, cf, &sc,
                                        smem, job.total, job.hdr);
    else
      persistent_split_call<MODEL, V, BATCH, PARK>(job, ki, i, o, item, K, G, cf, sc, smem);
  });
}

template <int MODEL, int V, bool HET, bool PACKED, int NT>
static cudaError_t launch_split_k(int block, int64_t grid, const BlockedJob &job, const CoefD &cfd, cudaStream_t st) {
  static PerDevice attr;
  const cudaError_t e = set_smem_limit_once(k_split<MODEL, V, HET, PACKED, NT>, 200 * 1024, attr);
  if (e != cudaSuccess) return e;
  const size_t smem = split_smem_bytes<MODEL, V, HET, NT>(block);
  if (grid > 0)
    k_split<MODEL, V, HET, PACKED, NT><<<(unsigned)grid, block, smem, st>>>(job, to_coef<double>(cfd, cfd.kappa),
                                                                          split_coef(MODEL, cfd));
  return cudaGetLastError();
}
template <int MODEL, int V, bool HET>
static cudaError_t launch_split_v(int block, const BlockedJob &job, const CoefD &cf, cudaStream_t st) {
  constexpr int S = split_small_block(V), B = max_threads_for(V);
  if constexpr (!HET) {
    if (job.nchains > 1 && job.packed) {
      const int64_t grid = job.ntiles + job.bt.npacked;
      return block <= S ? launch_split_k<MODEL, V, false, true, S>(block, grid, job, cf, st)
                        : launch_split_k<MODEL, V, false, true, B>(block, grid, job, cf, st);
    }
  }
  return block <= S ? launch_split_k<MODEL, V, HET, false, S>(block, job.ntiles, job, cf, st)
                    : launch_split_k<MODEL, V, HET, false, B>(block, job.ntiles, job, cf, st);
}

template <int MODEL>
cudaError_t launch_split_blocked(int v, int block, const BlockedJob &job, const CoefD &cf, cudaStream_t st) {
  if (job.sp) {
    switch (v) {
      case 2: return launch_split_v<MODEL, 2, true>(block, job, cf, st);
      case 4: return launch_split_v<MODEL, 4, true>(block, job, cf, st);
      default: return cudaErrorInvalidValue;
    }
  }
  switch (v) {
    case 1: return launch_split_v<MODEL, 1, false>(block, job, cf, st);
    case 2: return launch_split_v<MODEL, 2, false>(block, job, cf, st);
    case 4: return launch_split_v<MODEL, 4, false>(block, job, cf, st);
    case 8: return launch_split_v<MODEL, 8, false>(block, job, cf, st);
    default: return cudaErrorInvalidValue;
  }
}

template <int MODEL, int V, int NT>
static int persistent_split_grid_k(int block) {
  static PerDevice attr, attr_b;
  if (set_smem_limit_once(k_persistent_split<MODEL, V, false, NT>, 200 * 1024, attr) != cudaSuccess ||
      set_smem_limit_once(k_persistent_split<MODEL, V, true, NT>, 200 * 1024, attr_b) != cudaSuccess)
    return 0;
  const size_t smem = split_smem_bytes<MODEL, V, false, NT>(block);
  int a = 0, b = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&a, k_persistent_split<MODEL, V, false, NT>, block, smem) !=
          cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_persistent_split<MODEL, V, true, NT>, block, smem) !=
          cudaSuccess)
    return 0;
  return std::min(a, b) * sm_count();  // a grid that stays co-resident with either form
}
template <int MODEL, int V, int NT>
static cudaError_t launch_persistent_split_k(int block, int grid, const PersistentJob &job, const CoefD &cfd,
                                             cudaStream_t st) {
  if (persistent_split_grid_k<MODEL, V, NT>(block) < grid) return cudaErrorInvalidConfiguration;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3((unsigned)block);
  cfg.dynamicSmemBytes = split_smem_bytes<MODEL, V, false, NT>(block);
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  const Coef<double> cf = to_coef<double>(cfd, cfd.kappa);
  const SplitCoef sc = split_coef(MODEL, cfd);
  if (job.nchains > 1) return cudaLaunchKernelEx(&cfg, k_persistent_split<MODEL, V, true, NT>, job, cf, sc);
  return cudaLaunchKernelEx(&cfg, k_persistent_split<MODEL, V, false, NT>, job, cf, sc);
}

#define RK4_SPLIT_V(FN, ...)                                                                             \
  switch (v) {                                                                                           \
    case 1: return FN<MODEL, 1, max_threads_for(1)>(__VA_ARGS__);                                        \
    case 2: return FN<MODEL, 2, max_threads_for(2)>(__VA_ARGS__);                                        \
    case 4:                                                                                              \
      return block <= split_small_block(4) ? FN<MODEL, 4, split_small_block(4)>(__VA_ARGS__)             \
                                           : FN<MODEL, 4, max_threads_for(4)>(__VA_ARGS__);              \
    case 8: return FN<MODEL, 8, max_threads_for(8)>(__VA_ARGS__);                                        \
    default: break;                                                                                      \
  }

template <int MODEL>
cudaError_t launch_split_persistent(int v, int block, int grid, const PersistentJob &job, const CoefD &cf,
                                    cudaStream_t st) {
  RK4_SPLIT_V(launch_persistent_split_k, block, grid, job, cf, st)
  return cudaErrorInvalidValue;
}
template <int MODEL> int persistent_split_max_grid(int v, int block) {
  RK4_SPLIT_V(persistent_split_grid_k, block)
  return 0;
}
#undef RK4_SPLIT_V

}  // namespace rk4d
