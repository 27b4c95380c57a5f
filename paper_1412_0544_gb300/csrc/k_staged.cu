// k_staged.cu -- the paper's "standard implementation" (Sec. 2.2) on the GPU: one launch per
// RK stage, each a full sweep over every site.  It is the bit-identity reference for the
// blocked and persistent kernels (all three call the same per-site functions).
#include <algorithm>

#include "rk4_generic.cuh"

namespace rk4d {

// The chain of site i, number ci (its coupling strength goes into c).
template <typename R>
__device__ __forceinline__ ChainDesc staged_chain(const StagedJob &job, int64_t i, Coef<R> &c, int &ci) {
  ci = 0;
  if (job.nchains == 1) return job.one;
  ci = site_chain(job.chains, job.nchains, i);
  const ChainDesc ch = job.chains[ci];
  c.kappa = (R)ch.kappa;
  return ch;
}

// Stage j of site i, of chain ch with coefficients c.
template <typename R, int MODEL, bool KAHAN>
__device__ __forceinline__ void staged_site(const StagedJob &job, const ChainDesc &ch, Coef<R> c, int64_t i, int j) {
  constexpr int D = Dim<MODEL>::D;
  R *Y = static_cast<R *>(job.y);
  R *CMP = static_cast<R *>(job.cmp);
  const R *src = (j == 0) ? Y : static_cast<const R *>(job.uin);
  R *UOUT = static_cast<R *>(job.uout);
  R *ACC = static_cast<R *>(job.acc);
  if (job.sp) c = site_coef<R, MODEL>(c, static_cast<const R *>(job.sp) + i * Dim<MODEL>::P);  // Eq. (1)
  const int64_t li = i - ch.off;  // index within the chain
  R u[D], y[D], acc[D], cmp[D], k[D];
#pragma unroll
  for (int d = 0; d < D; ++d) {
    u[d] = src[i * D + d];
    y[d] = Y[i * D + d];
    acc[d] = (j > 0) ? ACC[i * D + d] : R(0);
    cmp[d] = (KAHAN && j == 3) ? CMP[i * D + d] : R(0);
  }
  R xl, xr;
  if (ch.bc == PERIODIC) {
    const int64_t il = (li == 0) ? ch.n - 1 : li - 1;
    const int64_t ir = (li == ch.n - 1) ? 0 : li + 1;
    if (!bounds_ok(job.hdr, in_range(ch.off + il, 1, job.total) && in_range(ch.off + ir, 1, job.total))) return;
    xl = src[(ch.off + il) * D];
    xr = src[(ch.off + ir) * D];
  } else {
    if (!bounds_ok(job.hdr, in_range(li, 1, ch.n))) return;
    xl = (li == 0) ? R(0) : src[(i - 1) * D];
    xr = (li == ch.n - 1) ? R(0) : src[(i + 1) * D];
  }
  slope<R, MODEL>(u, xl, xr, c, k);
  stage_update<R, D, KAHAN>(j, k, y, u, acc, cmp, c);
  if (j < 3) {
#pragma unroll
    for (int d = 0; d < D; ++d) {
      UOUT[i * D + d] = u[d];
      ACC[i * D + d] = acc[d];
    }
  } else {
    bool bad = false;
#pragma unroll
    for (int d = 0; d < D; ++d) {
      Y[i * D + d] = y[d];
      if constexpr (KAHAN) CMP[i * D + d] = cmp[d];
      bad |= nonfinite(y[d]);
    }
    if (bad && job.hdr) atomicOr(&job.hdr->status, ST_NONFINITE);
  }
}

template <typename R, int MODEL, bool KAHAN>
__global__ void __launch_bounds__(256) k_staged(StagedJob job, Coef<R> cf, int j) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < job.total; i += stride) {
    Coef<R> c = cf;
    int ci;
    const ChainDesc ch = staged_chain(job, i, c, ci);
    staged_site<R, MODEL, KAHAN>(job, ch, c, i, j);
  }
}

// The same in the split form (rk4_split.cuh), bit for bit what the tile kernels compute: stage 0
// stores the first slope K1, stages 1 and 2 their negated differences, and a stage's increments
// (the site's and its neighbours') are formed again from these.  Once a value of a chain has left the
// split's range (the scan before the first step, or a step's result) the chain's further steps run
// in the FP64 form.
template <int MODEL>
__global__ void __launch_bounds__(256) k_staged_split(StagedJob job, Coef<double> cf, SplitCoef sc, int j) {
  constexpr int D = Dim<MODEL>::D;
  double *Y = static_cast<double *>(job.y);
  double *K1 = static_cast<double *>(job.acc);
  float2 *N2 = static_cast<float2 *>(job.n2), *N3 = static_cast<float2 *>(job.n3);
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < job.total; i += stride) {
    Coef<double> c = cf;
    int ci;
    const ChainDesc ch = staged_chain(job, i, c, ci);
    if (wide_chain(job.wide[2 * ci + job.parity])) {
      staged_site<double, MODEL, false>(job, ch, c, i, j);
      if (j == 3) job.wide[2 * ci + (job.parity ^ 1)] = kWideRange;
      continue;
    }
    const int64_t li = i - ch.off;
    // the neighbours' sites, or -1 beyond a fixed end
    int64_t il = li > 0 ? i - 1 : (ch.bc == PERIODIC ? ch.off + ch.n - 1 : -1);
    int64_t ir = li < ch.n - 1 ? i + 1 : (ch.bc == PERIODIC ? ch.off : -1);
    if (!bounds_ok(job.hdr, (il < 0 || in_range(il, 1, job.total)) && (ir < 0 || in_range(ir, 1, job.total)))) continue;
    const double *sp = job.sp ? static_cast<const double *>(job.sp) + i * Dim<MODEL>::P : nullptr;
    double y[D];
#pragma unroll
    for (int d = 0; d < D; ++d) y[d] = Y[i * D + d];
    if (sp) c = site_coef<double, MODEL>(c, sp);
    if (j == 0) {
      double k[D];
      slope<double, MODEL>(y, il < 0 ? 0.0 : Y[il * D], ir < 0 ? 0.0 : Y[ir * D], c, k);
#pragma unroll
      for (int d = 0; d < D; ++d) K1[i * D + d] = k[d];
      continue;
    }
    SplitCoef s = sc;
    split_set_kappa(s, c.kappa);
    if (sp) {
      const FPair<float> at = times_tau(sp[0], s), cc = split1(MODEL == ROESSLER ? sp[2] : 0.0);
      s.ath = at.h;
      s.atl = at.l;
      s.ch = cc.h;
      s.cl = cc.l;
    }
    // increments of component q (site * D + component) for stage j; N is the running sum
    auto increment = [&](int64_t q, FPair<float> &k1, FPair<float> &N) {
      k1 = split1(K1[q]);
      FPair<float> d = k1;
      for (int m = 1; m < j; ++m) {
        const float2 n = m == 1 ? N2[q] : N3[q];
        split_update<float>(m, k1, {n.x, n.y}, d, N);
      }
      return d;
    };
    FPair<float> k1[D], d[D], N[D], n[D], xl = {0.f, 0.f}, xr = {0.f, 0.f}, t0, t1;
#pragma unroll
    for (int q = 0; q < D; ++q) {
      N[q] = {0.f, 0.f};
      d[q] = increment(i * D + q, k1[q], N[q]);
    }
    if (il >= 0) xl = increment(il * D, t0, t1);
    if (ir >= 0) xr = increment(ir * D, t0, t1);
    SplitBase<float> base = {};
    if constexpr (MODEL == ROESSLER) {
      base.z = split1(y[2]);
      base.t = x_minus_c<float>(split1(y[0]), {s.ch, s.cl});
    }
    split_stage<MODEL, float>(d, xl, xr, base, stage_coef<float>(s), n);
    if (j < 3) {
      float2 *o = j == 1 ? N2 : N3;
#pragma unroll
      for (int q = 0; q < D; ++q) o[i * D + q] = make_float2(n[q].h, n[q].l);
      continue;
    }
    bool wide = false, bad = false;
#pragma unroll
    for (int q = 0; q < D; ++q) {
      split_update<float>(3, k1[q], n[q], d[q], N[q]);
      double nd;
      join(N[q], &nd, 1);
      const double r = split_final(y[q], K1[i * D + q], nd, 6.0, s.w);
      Y[i * D + q] = r;
      wide |= !split_in_range<MODEL>(r, q, MODEL == ROESSLER && sp ? sp + 2 : nullptr, s);
      bad |= nonfinite(r);
    }
    if (wide) job.wide[2 * ci + (job.parity ^ 1)] = kWideRange;
    if (bad) atomicOr(&job.hdr->status, ST_NONFINITE);
  }
}

template <int MODEL, int RANGE>
__global__ void __launch_bounds__(256) k_split_scan(StagedJob job, Coef<double> cf, double kappa2, SplitCoef sc) {
  constexpr int D = Dim<MODEL>::D, P = Dim<MODEL>::P;
  const double *Y = static_cast<const double *>(job.y), *SP = static_cast<const double *>(job.sp);
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < job.total; i += stride) {
    Coef<double> c = cf;
    int ci;
    const ChainDesc ch = staged_chain(job, i, c, ci);
    if (SP) c = site_coef<double, MODEL>(c, SP + i * P);
    unsigned f = 0;
    double y[D], k[D];
#pragma unroll
    for (int d = 0; d < D; ++d) {
      y[d] = Y[i * D + d];
      if (!split_in_range<MODEL>(y[d], d, MODEL == ROESSLER && SP ? SP + i * P + 2 : nullptr, sc)) f |= kWideRange;
    }
    if (SP) {
#pragma unroll
      for (int q = 0; q < P; ++q)
        if (!split_param_in_range(SP[i * P + q], sc.most[q])) f |= kWideRange;
    }
    auto xat = [&](int64_t q) {
      if (ch.bc == PERIODIC) q = wrap(q, ch.n);
      const int64_t g = ch.off + q;
      return q < 0 || q >= ch.n || !bounds_ok(job.hdr, in_range(g, 1, job.total)) ? 0.0 : Y[g * D];
    };
    const int64_t li = i - ch.off;
    slope_gen<double, MODEL, RANGE>(y, xat(li - 1), xat(li + 1), RANGE == 2 ? xat(li - 2) : 0.0,
                                    RANGE == 2 ? xat(li + 2) : 0.0, c, kappa2, k);
    bool rest = true;
#pragma unroll
    for (int d = 0; d < D; ++d) rest = rest && is_zero(k[d]);
    f |= rest ? kWideRest : kWideMoves;
    unsigned *flag = job.wide + 2 * ci;
    if (f & ~*static_cast<volatile unsigned *>(flag)) atomicOr(flag, f);
  }
}

static unsigned sweep_grid(int64_t total) {
  const int64_t cap = (int64_t)sm_count() * 64;
  return (unsigned)std::min<int64_t>((total + 255) / 256, cap);
}

cudaError_t launch_split_scan(int model, int range, const double *state, const double *sp, int64_t total, int nchains,
                              const ChainDesc &one, const ChainDesc *chains, const CoefD &cfd, unsigned *wide,
                              cudaStream_t st) {
  const cudaError_t e = cudaMemsetAsync(wide, 0, 2 * sizeof(unsigned) * (size_t)nchains, st);
  if (e != cudaSuccess || total <= 0) return e;
  StagedJob job{};
  job.y = const_cast<double *>(state);
  job.sp = sp;
  job.nchains = nchains;
  job.one = one;
  job.chains = chains;
  job.total = total;
  job.wide = wide;
  const Coef<double> cf = to_coef<double>(cfd, cfd.kappa);
  const SplitCoef sc = split_coef(model, cfd, false, sp != nullptr);
  const unsigned grid = sweep_grid(total);
  if (model == ROESSLER) {
    if (range == 1) k_split_scan<ROESSLER, 1><<<grid, 256, 0, st>>>(job, cf, cfd.kappa2, sc);
    else k_split_scan<ROESSLER, 2><<<grid, 256, 0, st>>>(job, cf, cfd.kappa2, sc);
  } else {
    if (range == 1) k_split_scan<HARMONIC, 1><<<grid, 256, 0, st>>>(job, cf, cfd.kappa2, sc);
    else k_split_scan<HARMONIC, 2><<<grid, 256, 0, st>>>(job, cf, cfd.kappa2, sc);
  }
  return cudaGetLastError();
}

template <int MODEL>
static cudaError_t launch_split_one(int j, const StagedJob &job, const CoefD &cfd, cudaStream_t st) {
  if (job.total <= 0) return cudaSuccess;
  k_staged_split<MODEL><<<sweep_grid(job.total), 256, 0, st>>>(job, to_coef<double>(cfd, cfd.kappa),
                                                              split_coef(MODEL, cfd, false, job.sp != nullptr), j);
  return cudaGetLastError();
}

template <typename R, int MODEL, bool KAHAN>
static cudaError_t launch_one(int j, const StagedJob &job, const CoefD &cfd, cudaStream_t st) {
  if (job.total <= 0) return cudaSuccess;
  k_staged<R, MODEL, KAHAN><<<sweep_grid(job.total), 256, 0, st>>>(job, to_coef<R>(cfd, cfd.kappa), j);
  return cudaGetLastError();
}

cudaError_t launch_staged(int model, bool fp32, int j, const StagedJob &job, const CoefD &cf, cudaStream_t st) {
  if (job.split)
    return model == ROESSLER ? launch_split_one<ROESSLER>(j, job, cf, st) : launch_split_one<HARMONIC>(j, job, cf, st);
  if (model == ROESSLER)
    return fp32 ? launch_one<float, ROESSLER, true>(j, job, cf, st) : launch_one<double, ROESSLER, false>(j, job, cf, st);
  return fp32 ? launch_one<float, HARMONIC, true>(j, job, cf, st) : launch_one<double, HARMONIC, false>(j, job, cf, st);
}

}  // namespace rk4d
