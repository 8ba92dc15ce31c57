// Instantiates the templated kernels for one fiber count PRISM_K and exposes them
// through a KernelSet. Included by prism_k<K>.cu.
#include "prism_kernels.cuh"
#include "prism_launch.h"
#include "prism_local.cuh"

#ifndef PRISM_K
#error "PRISM_K must be defined"
#endif

namespace prism {
namespace {

constexpr int kK = PRISM_K;

template <int TPV, int LOSS, bool CAL, int SHELL = 0, bool GRAD = false>
cudaError_t fused_one(const IterArgs& a, int grid, int nt, size_t smem, cudaStream_t st) {
  auto fn = k_iter_fused<kK, TPV, LOSS, CAL, SHELL, GRAD>;
  cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
  if (e != cudaSuccess) return e;
  // a programmatic dependent only after k_prior_grad (which lets it start once every one of
  // its CTAs has run past its own wait), and only where the tile queue hands each CTA two tiles
  // or more: CTAs that start early land on the SMs that k_prior_grad leaves free, and with one
  // tile per CTA nothing evens that out (a 40^3 phantom's iteration, 500 tiles on 500 CTAs,
  // took 0.101 instead of 0.075 ms; the brain's, 9.5 tiles per CTA, 0.8 % less time)
  const bool dep = a.pdl && a.nb_priors && a.ntiles >= 2 * grid;
  return launch_dep(fn, dim3(grid), dim3(nt), smem, st, dep, a);
}

template <int TPV, int LOSS, bool CAL, int SHELL = 0>
cudaError_t fused_occ(int nt, size_t smem, int* blocks) {
  auto fn = k_iter_fused<kK, TPV, LOSS, CAL, SHELL>;
  cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
  if (e != cudaSuccess) return e;
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks, fn, nt, smem);
}

// The kernels of the shell loop's general form: four lanes per voxel, and one where forms 1 and 2 do
// not apply.
template <int TPV, int LOSS, bool CAL>
struct Shell3 {
  template <bool GRAD>
  cudaError_t launch(const IterArgs& a, int grid, int nt, size_t smem, cudaStream_t st) const {
    return fused_one<TPV, LOSS, CAL, 3, GRAD>(a, grid, nt, smem, st);
  }
  cudaError_t occupancy(int nt, size_t smem, int* blocks) const { return fused_occ<TPV, LOSS, CAL, 3>(nt, smem, blocks); }
};
template <typename F>
cudaError_t shell3(int loss, int cal, int tpv, F go) {
  if (tpv == 1 && loss == kLossMSE && cal) return go(Shell3<1, kLossMSE, true>{});
  if (tpv == 1 && loss == kLossNLL) return cal ? go(Shell3<1, kLossNLL, true>{}) : go(Shell3<1, kLossNLL, false>{});
  if (tpv == 4 && loss == kLossMSE) return cal ? go(Shell3<4, kLossMSE, true>{}) : go(Shell3<4, kLossMSE, false>{});
  if (tpv == 4) return cal ? go(Shell3<4, kLossNLL, true>{}) : go(Shell3<4, kLossNLL, false>{});
  return cudaErrorInvalidValue;
}

template <int TPV, bool GRAD>
cudaError_t fused_tpv(const IterArgs& a, int loss, int cal, int grid, int nt, size_t smem, cudaStream_t st) {
  if (loss == kLossMSE) {
    return cal ? fused_one<TPV, kLossMSE, true, 0, GRAD>(a, grid, nt, smem, st)
               : fused_one<TPV, kLossMSE, false, 0, GRAD>(a, grid, nt, smem, st);
  }
  return cal ? fused_one<TPV, kLossNLL, true, 0, GRAD>(a, grid, nt, smem, st)
             : fused_one<TPV, kLossNLL, false, 0, GRAD>(a, grid, nt, smem, st);
}

template <int TPV>
cudaError_t occ_tpv(int loss, int cal, int nt, size_t smem, int* blocks) {
  if (loss == kLossMSE) {
    return cal ? fused_occ<TPV, kLossMSE, true>(nt, smem, blocks) : fused_occ<TPV, kLossMSE, false>(nt, smem, blocks);
  }
  return cal ? fused_occ<TPV, kLossNLL, true>(nt, smem, blocks) : fused_occ<TPV, kLossNLL, false>(nt, smem, blocks);
}

template <bool GRAD>
cudaError_t fused_any(const IterArgs& a, int loss, int cal, int tpv, int shell, int grid, int nt, size_t smem,
                      cudaStream_t st) {
  if (shell == 3) return shell3(loss, cal, tpv, [&](auto f) { return f.template launch<GRAD>(a, grid, nt, smem, st); });
  if (shell) {
    if (tpv != 1 || loss != kLossMSE || cal) return cudaErrorInvalidValue;
    return shell == 2 ? fused_one<1, kLossMSE, false, 2, GRAD>(a, grid, nt, smem, st)
                      : fused_one<1, kLossMSE, false, 1, GRAD>(a, grid, nt, smem, st);
  }
  switch (tpv) {
    case 1: return fused_tpv<1, GRAD>(a, loss, cal, grid, nt, smem, st);
    case 4: return fused_tpv<4, GRAD>(a, loss, cal, grid, nt, smem, st);
    case 16: return fused_tpv<16, GRAD>(a, loss, cal, grid, nt, smem, st);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t l_fused(const IterArgs& a, int loss, int cal, int tpv, int shell, int grad, int grid, int nt, size_t smem,
                    cudaStream_t st) {
  return grad ? fused_any<true>(a, loss, cal, tpv, shell, grid, nt, smem, st)
              : fused_any<false>(a, loss, cal, tpv, shell, grid, nt, smem, st);
}

cudaError_t l_fused_occupancy(int loss, int cal, int tpv, int shell, int nt, size_t smem, int* blocks) {
  if (shell == 3) return shell3(loss, cal, tpv, [&](auto f) { return f.occupancy(nt, smem, blocks); });
  if (shell) {
    if (tpv != 1 || loss != kLossMSE || cal) return cudaErrorInvalidValue;
    return shell == 2 ? fused_occ<1, kLossMSE, false, 2>(nt, smem, blocks)
                      : fused_occ<1, kLossMSE, false, 1>(nt, smem, blocks);
  }
  switch (tpv) {
    case 1: return occ_tpv<1>(loss, cal, nt, smem, blocks);
    case 4: return occ_tpv<4>(loss, cal, nt, smem, blocks);
    case 16: return occ_tpv<16>(loss, cal, nt, smem, blocks);
    default: return cudaErrorInvalidValue;
  }
}

template <typename F>
cudaError_t local_fn(int loss, int tpv, F go) {
  if (tpv == 4) return loss == kLossMSE ? go(k_iter_local<kK, 4, kLossMSE>) : go(k_iter_local<kK, 4, kLossNLL>);
  if (tpv == 16) return loss == kLossMSE ? go(k_iter_local<kK, 16, kLossMSE>) : go(k_iter_local<kK, 16, kLossNLL>);
  return cudaErrorInvalidValue;
}

cudaError_t l_local(const IterArgs& a, int loss, int tpv, int grid, size_t smem, cudaStream_t st) {
  return local_fn(loss, tpv, [&](auto fn) {
    cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
    if (e != cudaSuccess) return e;
    if (loss == kLossMSE) {
      fn<<<grid, kFusedThreads, smem, st>>>(a);
      return cudaGetLastError();
    }
    // the NLL's CTAs wait on one another: all of them resident, or the launch is refused
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(kFusedThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeCooperative;
    at[0].val.cooperative = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, fn, a);
  });
}

cudaError_t l_local_occupancy(int loss, int tpv, size_t smem, int* blocks) {
  return local_fn(loss, tpv, [&](auto fn) {
    cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
    if (e != cudaSuccess) return e;
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks, fn, kFusedThreads, smem);
  });
}

inline int nblocks(int64_t n, int b) { return static_cast<int>((n + b - 1) / b); }

cudaError_t l_transform(const IterArgs& a, int tb, int te, cudaStream_t st) {
  const int64_t n = static_cast<int64_t>(te - tb) * a.TV;
  if (n <= 0) return cudaSuccess;
  k_transform<kK><<<nblocks(n, 128), 128, 0, st>>>(a, tb, te);
  return cudaGetLastError();
}

template <int TPV>
cudaError_t synth_tpv(const IterArgs& a, const PlainArgs& p, int cal, int nt, cudaStream_t st) {
  const int g = p.tile_end - p.tile_begin;
  if (cal) k_synth<kK, TPV, true><<<g, nt, 0, st>>>(a, p);
  else k_synth<kK, TPV, false><<<g, nt, 0, st>>>(a, p);
  return cudaGetLastError();
}

cudaError_t l_synth(const IterArgs& a, const PlainArgs& p, int cal, int tpv, int nt, cudaStream_t st) {
  if (p.tile_end <= p.tile_begin) return cudaSuccess;
  switch (tpv) {
    case 1: return synth_tpv<1>(a, p, cal, nt, st);
    case 4: return synth_tpv<4>(a, p, cal, nt, st);
    case 16: return synth_tpv<16>(a, p, cal, nt, st);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t l_yhat(const IterArgs& a, int cal, const int32_t* vos, const int32_t* order, float* out, cudaStream_t st) {
  if (a.ntiles <= 0) return cudaSuccess;
  const int nt = max(128, a.TV);   // TV: 8, 32, 128 or, on a plain handle with 256-thread CTAs, up to 256
  const size_t smem = static_cast<size_t>(a.TV) * ((kYhatC + 1) * sizeof(float) + sizeof(int64_t));   // at most 36 KB
  if (cal) k_yhat<kK, true><<<a.ntiles, nt, smem, st>>>(a, vos, order, out);
  else k_yhat<kK, false><<<a.ntiles, nt, smem, st>>>(a, vos, order, out);
  return cudaGetLastError();
}

template <int TPV>
cudaError_t adjoint_tpv(const IterArgs& a, const PlainArgs& p, int cal, int nt, size_t smem, cudaStream_t st) {
  const int g = p.tile_end - p.tile_begin;
  if (cal) {
    auto fn = k_adjoint<kK, TPV, true>;
    cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
    if (e != cudaSuccess) return e;
    fn<<<g, nt, smem, st>>>(a, p);
  } else {
    k_adjoint<kK, TPV, false><<<g, nt, 0, st>>>(a, p);
  }
  return cudaGetLastError();
}

cudaError_t l_adjoint(const IterArgs& a, const PlainArgs& p, int cal, int tpv, int nt, size_t smem, cudaStream_t st) {
  if (p.tile_end <= p.tile_begin) return cudaSuccess;
  switch (tpv) {
    case 1: return adjoint_tpv<1>(a, p, cal, nt, smem, st);
    case 4: return adjoint_tpv<4>(a, p, cal, nt, smem, st);
    case 16: return adjoint_tpv<16>(a, p, cal, nt, smem, st);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t l_prior_prep(const IterArgs& a, int tb, int te, cudaStream_t st) {
  const int64_t n = static_cast<int64_t>(te - tb) * a.TV;
  if (n <= 0) return cudaSuccess;
  return launch_dep(a.n_nbr == 6 ? k_prior_prep<kK, 6> : k_prior_prep<kK, 26>, dim3(nblocks(n, 128)), dim3(128), 0, st, a.pdl != 0,
                    a, tb, te);
}

cudaError_t l_prior_grad(const IterArgs& a, int tb, int te, cudaStream_t st) {
  const int64_t n = static_cast<int64_t>(te - tb) * a.TV;
  if (n <= 0) return cudaSuccess;
  return launch_dep(a.n_nbr == 6 ? k_prior_grad<kK, 6> : k_prior_grad<kK, 26>, dim3(nblocks(n, 128)), dim3(128), 0, st, a.pdl != 0,
                    a, tb, te);
}

cudaError_t l_prior(const IterArgs& a, const PlainArgs& p, cudaStream_t st) {
  const int g = p.tile_end - p.tile_begin;
  if (g <= 0) return cudaSuccess;
  // one block of TV threads per tile (TV <= 256): the tile's prior value is one block sum
  k_prior<kK><<<dim3(1, g), (a.TV + 31) / 32 * 32, 0, st>>>(a, p);
  return cudaGetLastError();
}

cudaError_t l_fibers(const IterArgs& a, const int32_t* sov, int64_t V, float rel, float* dirs, float* fracs,
                     uint8_t* peaks, cudaStream_t st) {
  if (V <= 0) return cudaSuccess;
  k_fibers<kK><<<nblocks(V, 128), 128, 0, st>>>(a, sov, V, rel, dirs, fracs, peaks);
  return cudaGetLastError();
}
cudaError_t l_stitch(const IterArgs& a, const StitchArgs& s, cudaStream_t st) {
  if (s.n <= 0) return cudaSuccess;
  k_stitch<kK><<<nblocks(s.n, 128), 128, 0, st>>>(a, s);
  return cudaGetLastError();
}

}  // namespace

#define PRISM_CAT2(a, b) a##b
#define PRISM_CAT(a, b) PRISM_CAT2(a, b)
const KernelSet& PRISM_CAT(kernels_k, PRISM_K)() {
  static const KernelSet ks = {l_fused, l_fused_occupancy, l_local, l_local_occupancy, l_transform, l_synth, l_yhat, l_adjoint, l_prior_prep, l_prior_grad, l_prior, l_fibers, l_stitch};
  return ks;
}

}  // namespace prism
