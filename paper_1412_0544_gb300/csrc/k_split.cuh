// k_split.cuh -- the blocked and persistent FP64 kernels in the split form (rk4_split.cuh), and
// their launchers for one model.  Each model is instantiated in a translation unit of its own
// (k_split_roessler.cu, k_split_harmonic.cu), so that they compile side by side.
//
// What bounds it: 13 FP64 instructions per site-step (Roessler: 7 for the first slope, 6 for the
// update; harmonic 8) at 0.6 T/s allow 4.6e10 site-steps/s; beside them about 400 FP32
// operations (three later stages at 85, 102 for the sums and increments, 33 to convert; packed two
// sites per instruction, 40 T lane-operations/s) and 110 integer ones.
// Measured at N = 2^24 against the FP64 form (49 instructions, 1.23e10 site-steps/s): 3.67e10 at
// 256 x 2 x 4 and 128 x 4 x 4; harmonic 6.4e10 (128 x 4 x 4) against 1.90e10.
#pragma once
#include "k_grid_barrier.cuh"
#include "rk4_tile.cuh"

namespace rk4d {

// Sites per thread of the kernel that runs tiles of block x v sites.  The Roessler step takes two (a
// packed pair) for whatever v > 1, parked in 64 registers (split_advance), so that an SM holds 32
// warps: N = 2^24, 256 x 2 x 4, 3.10e10 site-steps/s unparked (128 registers, 16 warps) -> 3.68e10;
// 128 x 4 x 4 with four per thread (parked, 126 registers) 3.52e10 -> 3.68e10.  Tiles of 1024 sites,
// of which an SM holds two either way, keep four: 256 x 4 x 1 2.71e10 against 2.51e10, x 2 3.27e10
// against 3.25e10, x 8 3.57e10 against 3.54e10.  One site per thread (nothing to pack, 64 registers as
// it is) keeps a step shortest where tiles are few.  The harmonic step (98 to 128 registers, only state
// and slope to park) was faster with the tiling's own v: 128 x 4 x 4 6.43e10 against 6.09e10.
// Heterogeneous tiles hold their parameters in shared memory and have no room for records; two
// sites per thread there too, up to 512 threads (N = 2^22: 256 x 4 x 2 1.79e10 -> 1.99e10, 128 x 4 x 4
// 2.70e10 -> 2.97e10).
__host__ __device__ constexpr int split_lanes(int model, int v, int block, bool het) {
  if (model != ROESSLER || v == 1) return v;
  if (het) return block * v > 1024 ? v : 2;
  return v >= 4 && block * v == 1024 ? 4 : 2;
}
__host__ __device__ constexpr bool split_parks(int model, int v, bool het) {
  return model == ROESSLER && v >= 2 && !het;
}
// Largest block and resident blocks of an instantiation.
__host__ __device__ constexpr int split_max_threads(int model, int v, bool het) {
  return split_parks(model, v, het) ? (v == 2 ? 1024 : 256) : max_threads_for(v);
}
__host__ __device__ constexpr int split_min_blocks(int model, int v, bool het) {
  return split_parks(model, v, het) && v == 4 ? 2 : 0;
}
template <int MODEL, int V, bool HET> static size_t split_smem_bytes(int block) {
  const size_t plain = blocked_smem_bytes(MODEL, false, V, block, HET);
  const size_t parked = sizeof(double) * ((size_t)edge_values(V) + (size_t)block * split_record_words<MODEL, V>());
  return split_parks(MODEL, V, HET) ? std::max(plain, parked) : plain;
}
// fn(V, NT, threads) with V and NT compile-time, for tiles of block x v sites.
template <int MODEL, bool HET, typename R, typename F> static R split_dispatch(int v, int block, R none, F &&fn) {
  const int lanes = split_lanes(MODEL, v, block, HET), threads = block * v / lanes;
  auto with = [&](auto vc) -> R {
    return fn(vc, std::integral_constant<int, split_max_threads(MODEL, decltype(vc)::value, HET)>(), threads);
  };
  if constexpr (!HET) {
    if (lanes == 1) return with(std::integral_constant<int, 1>());
  }
  if (lanes == 2) return with(std::integral_constant<int, 2>());
  if (lanes == 4) return with(std::integral_constant<int, 4>());
  if constexpr (MODEL == HARMONIC && !HET) {
    if (lanes == 8) return with(std::integral_constant<int, 8>());
  }
  return none;
}

// An item (of a packed tile, the marked segments) outside the split's range, in the FP64 form.  Not inlined: it is rare, and its
// registers then do not add to the split's.
template <int MODEL, int V, bool HET, bool ALN>
__device__ __noinline__ void wide_tile_call(const double *in, double *out, ChainDesc ch, int64_t tile, int K, int G,
                                            Coef<double> cf, unsigned char *smem, int64_t sites, WsHeader *hdr,
                                            const double *sp) {
  tile_item<double, MODEL, V, false, false, HET, ALN, false>(in, out, nullptr, nullptr, ch, tile, K, G, cf, smem, sites,
                                                           hdr, sp);
}
template <int MODEL, int V, bool COH>
__device__ __noinline__ void wide_packed_call(const double *in, double *out, const ChainDesc *chains,
                                              const SegDesc *segs, int s0, int s1, int K, Coef<double> cf,
                                              unsigned char *smem, int64_t sites, WsHeader *hdr) {
  packed_tile_item<double, MODEL, V, false, COH, false, false, true>(in, out, nullptr, nullptr, chains, segs, s0, s1, K,
                                                                     cf, smem, sites, hdr);
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
__global__ void __launch_bounds__(NT, split_min_blocks(MODEL, V, HET)) k_split(BlockedJob job, Coef<double> cf, SplitCoef sc) {
  constexpr bool PARK = split_parks(MODEL, V, HET);
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
    wide_tile_call<MODEL, V, HET, PACKED>(in, out, ch, tile, job.K, job.G, cf, smem, job.total, job.hdr, sp);
}

// One full tile of the persistent kernel as a call of its own (as persistent_tile_call), in the split form
// or (WIDE) in the FP64 form; false when it is outside the split's range.  The FP64 form is called from the
// kernel's loop: from within the split form's call ptxas gave it registers that cost 13 % (64 chains of 64000
// sites, a state of 1e-25, 8 steps: 3308 -> 2938 us; 4096 of 1000 sites in range 1052 -> 1041).  Packed tiles,
// a few per launch, keep theirs inside (outside: 1041 -> 1054).
template <int MODEL, int V, bool BATCH, bool PARK, bool WIDE>
__device__ __noinline__ bool persistent_split_call(const PersistentJob &job, int ki, const double *in, double *out,
                                                   int64_t item, int K, int G, Coef<double> cf, SplitCoef sc,
                                                   unsigned char *smem) {
  ChainDesc ch;
  int64_t tile = item;
  if constexpr (BATCH) {
    const int ci = batch_chain(job.bt[ki], job.nchains, item - job.bt[ki].npacked, smem, tile);
    ch = job.chains[ci];
    cf.kappa = ch.kappa;
    if constexpr (!WIDE) split_set_kappa(sc, ch.kappa);
  } else {
    ch = job.one;
  }
  return tile_item<double, MODEL, V, false, true, false, BATCH, !WIDE, PARK && !WIDE>(
      in, out, nullptr, nullptr, ch, tile, K, G, cf, smem, job.total, job.hdr, nullptr, &sc);
}

// The split form of k_persistent.
template <int MODEL, int V, bool BATCH, int NT>
__global__ void __launch_bounds__(NT, split_min_blocks(MODEL, V, false)) k_persistent_split(PersistentJob job, Coef<double> cf, SplitCoef sc) {
  constexpr bool PARK = split_parks(MODEL, V, false);
  extern __shared__ __align__(16) unsigned char smem[];
  persistent_loop(job, [&](int ki, const void *in, void *out, const void *, void *, int64_t item, int K, int G) {
    const double *i = static_cast<const double *>(in);
    double *o = static_cast<double *>(out);
    if (BATCH && item < job.bt[ki].npacked)
      split_packed_call<MODEL, V, true, PARK>(i, o, job.chains, job.bt[ki].segs, job.bt[ki].pack_prefix, item, K, cf, &sc,
                                        smem, job.total, job.hdr);
    else if (!persistent_split_call<MODEL, V, BATCH, PARK, false>(job, ki, i, o, item, K, G, cf, sc, smem))
      persistent_split_call<MODEL, V, BATCH, PARK, true>(job, ki, i, o, item, K, G, cf, sc, smem);
  });
}

template <int MODEL, int V, bool HET, bool PACKED, int NT>
static cudaError_t launch_split_k(int block, int64_t grid, const BlockedJob &job, const CoefD &cfd, cudaStream_t st) {
  static PerDevice attr;
  const cudaError_t e = set_smem_limit_once(k_split<MODEL, V, HET, PACKED, NT>, 200 * 1024, attr);
  if (e != cudaSuccess) return e;
  const size_t smem = split_smem_bytes<MODEL, V, HET>(block);
  if (grid > 0)
    k_split<MODEL, V, HET, PACKED, NT><<<(unsigned)grid, block, smem, st>>>(job, to_coef<double>(cfd, cfd.kappa),
                                                                          split_coef(MODEL, cfd, false, HET));
  return cudaGetLastError();
}
template <int MODEL>
cudaError_t launch_split_blocked(int v, int block, const BlockedJob &job, const CoefD &cf, cudaStream_t st) {
  if (job.sp)
    return split_dispatch<MODEL, true>(v, block, cudaErrorInvalidValue, [&](auto vc, auto nt, int threads) {
      return launch_split_k<MODEL, decltype(vc)::value, true, false, decltype(nt)::value>(threads, job.ntiles, job, cf, st);
    });
  return split_dispatch<MODEL, false>(v, block, cudaErrorInvalidValue, [&](auto vc, auto nt, int threads) {
    constexpr int V = decltype(vc)::value, NT = decltype(nt)::value;
    if (job.nchains > 1 && job.packed)
      return launch_split_k<MODEL, V, false, true, NT>(threads, job.ntiles + job.bt.npacked, job, cf, st);
    return launch_split_k<MODEL, V, false, false, NT>(threads, job.ntiles, job, cf, st);
  });
}

template <int MODEL, int V, int NT>
static int persistent_split_grid_k(int block) {
  static PerDevice attr, attr_b;
  if (set_smem_limit_once(k_persistent_split<MODEL, V, false, NT>, 200 * 1024, attr) != cudaSuccess ||
      set_smem_limit_once(k_persistent_split<MODEL, V, true, NT>, 200 * 1024, attr_b) != cudaSuccess)
    return 0;
  const size_t smem = split_smem_bytes<MODEL, V, false>(block);
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
  cfg.dynamicSmemBytes = split_smem_bytes<MODEL, V, false>(block);
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

template <int MODEL>
cudaError_t launch_split_persistent(int v, int block, int grid, const PersistentJob &job, const CoefD &cf,
                                    cudaStream_t st) {
  return split_dispatch<MODEL, false>(v, block, cudaErrorInvalidValue, [&](auto vc, auto nt, int threads) {
    return launch_persistent_split_k<MODEL, decltype(vc)::value, decltype(nt)::value>(threads, grid, job, cf, st);
  });
}
template <int MODEL> int persistent_split_max_grid(int v, int block) {
  return split_dispatch<MODEL, false>(v, block, 0, [&](auto vc, auto nt, int threads) {
    return persistent_split_grid_k<MODEL, decltype(vc)::value, decltype(nt)::value>(threads);
  });
}

}  // namespace rk4d
