// Fits without neighbour priors and calibration, several lanes per voxel: many iterations per launch.
//
// Nothing couples two voxels of such a fit but the noise level of the Rician NLL, which the voxels
// of a volume share. One launch therefore keeps a tile's signal, table, parameters and moments in
// shared memory and runs up to kMaxIters iterations on it. An iteration of the general fused kernel
// at these sizes is a chain of latencies (launch, queue, tile and group records, staging, three
// transforms, block-wide FP64 sums, the last CTA's tail): 13.8 us for an 8^3 patch, of which the
// arithmetic is under 1 us. Here a voxel's lanes sit in one warp: all of them carry out the voxel's
// chain rule on the summed accumulators (issue slots that a small fit leaves idle) and share its update,
// so that an iteration of the MSE has no block barrier. Measured per iteration (GB300, MSE, K = 3, N = 96):
// 8^3 voxels 2.0 us (general kernel 13.8), 16^3 3.2 (17.5) and 28^3 8.5 us (19.6 with one thread per voxel).
//
// Rician NLL: dJ/dsigma is a sum over the volume in each iteration. The tiles of a volume
// write their FP64 partials and count themselves in on a per-volume counter, before the chain rule and the
// update; after these they wait for the count of the iteration; then every tile takes the same
// fixed-order sum and updates its own copy of sigma.
// The launch is cooperative (every CTA resident, one tile each) and every wait has a limit. 16
// volumes of 10^3 voxels: 75 -> 11.5 us an iteration (N = 96; 12.2 with the partials written after the update).
#pragma once

#include "prism_kernels.cuh"

namespace prism {

constexpr int kMaxIters = 32;      // iterations per launch (Adam's constants of each in shared memory)
constexpr int kLocalRow = 7;       // float4 per measurement pair in shared memory: the six that the
                                   // uncalibrated step reads and one of padding, so that eight lanes
                                   // reading eight neighbouring rows hit different banks
// Floats per voxel of a state array in shared memory: 4K + 5 rounded up to an odd multiple of 4, so that
// eight voxels' rows fall into different banks, whether a lane reads a float or four.
__host__ __device__ constexpr int local_stride(int K) { return K <= 1 ? 12 : K <= 3 ? 20 : 28; }

__host__ __device__ inline size_t local_smem(int K, int tpv, int NP) {
  const size_t tv = kFusedThreads / tpv;
  return static_cast<size_t>(NP / 2) * kLocalRow * sizeof(float4) + static_cast<size_t>(NP) * tv * sizeof(float) +
         4 * static_cast<size_t>(local_stride(K)) * tv * sizeof(float);
}

__device__ __forceinline__ int ld_acquire(const int32_t* p) {
  int v;
  asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

// dJ/dsigma of a tile (Rician NLL), behind the objective's partials; both [kMaxIters][ntiles].
__device__ __forceinline__ double* local_dsig(const IterArgs& a, int it, int tile) {
  return a.tile_red + static_cast<size_t>(kMaxIters + it) * a.ntiles + tile;
}

// Sum of a volume's dJ/dsigma of one iteration, fixed order: strided over the warp's lanes, then a
// butterfly; every lane ends with it.
__device__ __forceinline__ double local_dsig_sum(const IterArgs& a, const GroupDev& gr, int it) {
  const double* d = local_dsig(a, it, gr.tile0);
  double s = 0.0;
#pragma unroll 4
  for (int i = threadIdx.x & 31; i < gr.ntiles; i += 32) s += __ldcg(d + i);
  return warp_sum_d(s);
}

// A volume's objective of every iteration of the launch, by the CTA that finished the volume's last
// tile, from one FP64 value per tile and iteration. A lane adds four strided sums, a butterfly the lanes. A warp
// takes an iteration; with fewer iterations than warps all of them share each (`part`: 128 doubles), in
// the same order, so that the bits do not depend on how many iterations a launch holds. (Four values per tile, summed by
// one warp where the launch holds one iteration: a call of one took 235 us for 32,760 voxels with sixteen lanes, of which the
// iteration was 40. With the launch's last CTA doing all volumes' sums one by one, 16 volumes of 10^3 voxels
// took 13.6 us an iteration instead of 7.0.)
__device__ __forceinline__ void local_objectives(const IterArgs& a, const GroupDev& gr, int group, int step, double* part) {
  constexpr int NW = kFusedThreads / 32;
  static_assert(NW == 4, "four strided sums");
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, n = gr.ntiles;
  auto store = [&](int it, double s0, double s1, double s2, double s3) {
    const double J = warp_sum_d((s0 + s1) + (s2 + s3));
    if (lane != 0) return;
    if (!isfinite(J)) atomicOr(a.status, kStNonfinite);
    if (it == a.n_it - 1) a.gloss[group] = J;
    a.hist[static_cast<size_t>((step + it) % a.hist_len) * a.G + group] = J;
  };
  if (a.n_it < NW) {
    for (int it = 0; it < a.n_it; ++it) {
      const double* red = a.tile_red + static_cast<size_t>(it) * a.ntiles + gr.tile0;
      double s = 0.0;
#pragma unroll 8
      for (int i = threadIdx.x; i < n; i += kFusedThreads) s += __ldcg(red + i);
      part[threadIdx.x] = s;
      __syncthreads();
      if (warp == 0) store(it, part[lane], part[lane + 32], part[lane + 64], part[lane + 96]);
      __syncthreads();
    }
    return;
  }
  for (int it = warp; it < a.n_it; it += NW) {
    const double* red = a.tile_red + static_cast<size_t>(it) * a.ntiles + gr.tile0;
    double s[NW] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll 4
    for (int i = lane; i < n; i += kFusedThreads) {
#pragma unroll
      for (int u = 0; u < NW; ++u)
        if (i + 32 * u < n) s[u] += __ldcg(red + i + 32 * u);
    }
    store(it, s[0], s[1], s[2], s[3]);
  }
}

template <int K, int TPV, int LOSS>
__global__ void __launch_bounds__(kFusedThreads, (K >= 4 ? 3 : 4)) k_iter_local(const IterArgs a) {
  constexpr int NF = K + 3, Q = 4 * K + 5, QS = local_stride(K), VW = 32 / TPV, TV = kFusedThreads / TPV, NW = kFusedThreads / 32;
  static_assert(TPV > 1, "one warp holds a voxel's lanes and several voxels");
  extern __shared__ __align__(16) unsigned char smem[];
  const int NPmax = a.Nmax;
  float4* s_tab = reinterpret_cast<float4*>(smem);                      // [NPmax / 2][kLocalRow]
  float* s_y = reinterpret_cast<float*>(s_tab + NPmax / 2 * kLocalRow);  // [NP][TV], packed as in HBM
  // [4][TV][QS]: theta, m, v and the gradient
  float* s_st = s_y + static_cast<size_t>(NPmax) * TV;
  __shared__ uint64_t s_bar;
  __shared__ float s_ac[2 * kMaxIters];
  __shared__ int s_last[2];   // this CTA counted in last: of the tile's volume, of the launch
  __shared__ double s_J[kMaxIters * NW];   // the warps' parts of the objective by iteration; then local_objectives' sums
  __shared__ double s_ex[NW];   // NLL: the warps' dJ/dsigma, and the volume's sigma_log of the next iteration
  __shared__ float s_sig;
  __shared__ float4 s_bess[(LOSS == kLossNLL) ? kBesselTab : 1];
  if constexpr (LOSS == kLossNLL) bessel_stage(s_bess);   // visible after the first tile's barriers
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int lv = lane % VW, js = lane / VW, vl = warp * VW + lv;
  const int Vp = a.Vpad, step = *a.step, n_it = a.n_it;
  if (tid == 0) {
    mbar_init(&s_bar, 1);
    fence_mbar_init();
  }
  if (tid < 2 * n_it)
    s_ac[tid] = adam_constant(tid, a.lr, a.beta1, a.beta2, static_cast<int64_t>(step) + 1 + (tid >> 1));
  uint32_t phase = 0;
  int cur_group = -1;
  bool failed = false;
  for (int ti = blockIdx.x; ti < a.ntiles; ti += gridDim.x) {
    const int t = a.tile_order[ti];
    const Tile tl = a.tiles[t];
    const GroupDev gr = a.groups[tl.group];
    const int N = tl.n_meas, NP = (N + 3) & ~3;
    __syncthreads();   // the previous tile's shared data are no longer read (and s_bar is set up)
    if (tid == 0 && !failed) {
      const uint32_t bytes = static_cast<uint32_t>(NP) * TV * 4u;   // multiple of 16: NP % 4 == 0
      fence_proxy_async_smem();
      mbar_expect_tx(&s_bar, bytes);
      tma_bulk_g2s(s_y, a.y + tl.y_off, bytes, &s_bar);
    }
    if (tl.group != cur_group) {
      const float4* src = reinterpret_cast<const float4*>(a.table2 + gr.table2_off);
      for (int e = tid; e < NP / 2 * 6; e += kFusedThreads) {
        const int p = e / 6, c = e - 6 * p;
        s_tab[p * kLocalRow + c] = src[8 * p + c];
      }
      cur_group = tl.group;
    }
    for (int e = tid; e < Q * TV; e += kFusedThreads) {
      const size_t ix = static_cast<size_t>(e / TV) * Vp + tl.slot0 + e % TV;
      const int at = e % TV * QS + e / TV;
      s_st[at] = a.theta[ix];
      s_st[TV * QS + at] = a.m[ix];
      s_st[2 * TV * QS + at] = a.v[ix];
    }
    if (!failed && !mbar_wait(&s_bar, phase)) {
      atomicOr(a.status, kStTimeout);
      mbar_wait(&s_bar, phase);   // let the copy land before its shared memory is released
      failed = true;
    }
    phase ^= 1;
    failed = __syncthreads_or(failed);
    // Without its signal the tile, like the CTA's later ones, still runs, so that no other tile waits for its
    // sums in vain, but stores no state (the handle's status says that the launch failed). A loop that skipped the
    // iterations would not be uniform to the compiler: 2.0 instead of 1.9 us an iteration of an 8^3 patch.
    const bool act = vl < tl.count;
    float* st = s_st + vl * QS;
    float th[Q];
#pragma unroll
    for (int q = 0; q < Q; ++q) th[q] = st[q];
    Vox<K> P;
    transform<K>(th, P);
    float slog = 0.f, sgm = 0.f, sgv = 0.f;   // the volume's noise level and its moments (NLL)
    if (LOSS == kLossNLL) {
      slog = a.gparams[gr.gp_off];
      sgm = a.gm[gr.gp_off];
      sgv = a.gv[gr.gp_off];
    }
    const float2* yc2 = reinterpret_cast<const float2*>(s_y + static_cast<size_t>(warp) * NP * VW) + lv;
    for (int it = 0; it < n_it; ++it) {
      const float inv_s2 = (LOSS == kLossNLL) ? expf(-2.f * slog) : 0.f;
      const float scale = (LOSS == kLossMSE) ? 2.f * gr.inv_M : inv_s2;
      Acc<K> A;
      acc_zero<K>(A);
      {
        VoxP<K> DP;
        AccP<K> AP;
        voxp_init<K>(P, DP, AP);
        // lane js of the voxel takes pairs js, js + TPV, ...; the leading pairs of b = 0 without the
        // fiber terms (MSE)
        const int i0 = (LOSS == kLossMSE) ? gr.nb0p : 0;
        if (i0 > js) step2_b0<K>(DP, yc2 + js * VW, TPV * VW, (i0 - js + TPV - 1) / TPV, AP);
        int p = i0 + ((js - i0) % TPV + TPV) % TPV;
        // (the rows' address runs along with the pair; with more than three fibers the signal's too, and it alone ends the
        // loop: 5 fibers, N = 600, 12^3: 14.3 -> 13.4 us an iteration, 3 fibers 9.6 -> 9.35)
        const float4* row = s_tab + p * kLocalRow;
        if constexpr (K >= 4) {
          const float2* yp = yc2 + p * VW;
#pragma unroll 1
          for (const float4* end = s_tab + N / 2 * kLocalRow; row < end; row += TPV * kLocalRow, yp += TPV * VW, p += TPV)
            step2<K, false, LOSS>(DP, reinterpret_cast<const MeasPair&>(*row), *yp, make_float2(1.f, 1.f), AP, inv_s2, s_bess);
        } else {
#pragma unroll (LOSS == kLossNLL ? 1 : 2)
          for (; p < N / 2; p += TPV, row += TPV * kLocalRow)
            step2<K, false, LOSS>(DP, reinterpret_cast<const MeasPair&>(*row), yc2[p * VW], make_float2(1.f, 1.f), AP, inv_s2,
                                  s_bess);
        }
        if (p < (N + 1) / 2)   // the last measurement of an odd count
          step2<K, true, LOSS>(DP, reinterpret_cast<const MeasPair&>(s_tab[p * kLocalRow]), yc2[p * VW],
                               make_float2(1.f, 0.f), AP, inv_s2, s_bess);
        accp_sums<K, LOSS, false>(AP, A);
      }
      acc_reduce_tpv<K, TPV, VW>(A);
      A.gS0 = acc_gS0<K>(P, A);
      float gS0, gf[NF], gd[K][3], gfin;
      data_grad<K>(P, A, scale, gS0, gf, gd, gfin);
      float dloss;
      if (LOSS == kLossMSE) {
        dloss = A.l1 * gr.inv_M;
      } else {
        dloss = 2.f * slog * N + 0.5f * inv_s2 * A.l1 - A.l3;
        const float dsig = 2.f * N - inv_s2 * (A.l1 + 2.f * A.l2);
        // the tile's part of dJ/dsigma leaves first (its last warp counts the tile in): the chain rule and the
        // update below run while the volume's other tiles arrive
        double dS = act ? static_cast<double>(dsig) : 0.0;
#pragma unroll
        for (int o = 1; o < VW; o <<= 1) dS += __shfl_xor_sync(0xffffffffu, dS, o);
        if (lane == 0) s_ex[warp] = dS;
        __syncthreads();
        if (tid == kFusedThreads - 32) {
          double ss = s_ex[0];
          for (int w = 1; w < NW; ++w) ss += s_ex[w];
          *local_dsig(a, it, t) = ss;
          __threadfence();
          atomicAdd(a.gbar + tl.group, 1);
        }
      }
      const float ploss = priors<K, true>(a, P, 0, gr.inv_M, nullptr, gS0, gf, gd);
      float g[Q];
      chain_raw<K>(P, gS0, gf, gd, gfin, g);
      const float stepsz = s_ac[2 * it], isbc2 = s_ac[2 * it + 1];
      // The voxel's lanes share the update, lane js taking parameters js, js + TPV, ...: every lane holds
      // the whole gradient, but the update's 17 instructions per parameter are a quarter of an iteration.
      if (js == 0) {
#pragma unroll
        for (int q = 0; q < Q; ++q) st[3 * TV * QS + q] = g[q];
      }
      __syncwarp();
#pragma unroll
      for (int i = 0; i < (Q + TPV - 1) / TPV; ++i) {
        float* p = st + js + TPV * i;
        if (js + TPV * i < Q) {
          float x = p[0], m = p[TV * QS], v = p[2 * TV * QS];
          const float gq = p[3 * TV * QS];
          if (a.optimizer == 0) {
            m = fmaf(a.beta1, m, (1.f - a.beta1) * gq);
            v = fmaf(a.beta2, v, (1.f - a.beta2) * gq * gq);
            x -= stepsz * m * frcp(fmaf(fsqrt(v), isbc2, a.eps));
          } else {
            rprop_update(x, m, v, gq, a.lr, a.eta_minus, a.eta_plus, a.step_min, a.step_max);
          }
          p[0] = x;
          p[TV * QS] = m;
          p[2 * TV * QS] = v;
        }
      }
      __syncwarp();
#pragma unroll
      for (int q = 0; q < Q; ++q) th[q] = st[q];
      transform<K>(th, P);
      // the warp's part of the objective: lanes 0 .. VW - 1 hold its voxels
      double J = act ? static_cast<double>(dloss) + static_cast<double>(ploss) : 0.0;
#pragma unroll
      for (int o = 1; o < VW; o <<= 1) J += __shfl_xor_sync(0xffffffffu, J, o);
      if (lane == 0) s_J[it * NW + warp] = J;
      if (LOSS == kLossNLL) {
        // the first warp alone waits for the volume's tiles and takes its sum (with every warp doing so, a
        // third of the iteration went into the exchange)
        const bool leader = t == gr.tile0;
        if (warp == 0 && (it + 1 < n_it || leader)) {
          const int want = gr.ntiles * (it + 1);
          if (!failed) {
            bool ok = true;
            if (lane == 0) {
              int polls = 0;
              while (ld_acquire(a.gbar + tl.group) < want && polls < (1 << 21)) ++polls;
              ok = polls < (1 << 21);
              if (!ok) atomicOr(a.status, kStTimeout);
            }
            failed = __any_sync(0xffffffffu, !ok);
          }
          // lane 0's acquire orders the other lanes' reads of the partials only through a warp barrier (a vote
          // orders no memory accesses)
          __syncwarp();
          const float gsig = static_cast<float>(local_dsig_sum(a, gr, it));
          if (a.optimizer == 0) {
            sgm = fmaf(a.beta1, sgm, (1.f - a.beta1) * gsig);
            sgv = fmaf(a.beta2, sgv, (1.f - a.beta2) * gsig * gsig);
            slog -= stepsz * sgm / fmaf(sqrtf(sgv), isbc2, a.eps);
          } else {
            rprop_update(slog, sgm, sgv, gsig, a.lr, a.eta_minus, a.eta_plus, a.step_min, a.step_max);
          }
          if (lane == 0) s_sig = slog;
          if (lane == 0 && leader && it == n_it - 1) {
            a.gparams_rw[gr.gp_off] = slog;
            a.gm[gr.gp_off] = sgm;
            a.gv[gr.gp_off] = sgv;
          }
        }
        __syncthreads();
        if (it + 1 < n_it) slog = s_sig;
      }
    }
    __syncthreads();
    if (tid < n_it) {   // the tile's objective of each iteration (n_it <= 32: the first warp)
      const double* w = s_J + tid * NW;
      a.tile_red[static_cast<size_t>(tid) * a.ntiles + t] = (w[0] + w[1]) + (w[2] + w[3]);
    }
    if (warp == 0) __syncwarp();
    if (tid == 0) {   // both counts in flight at once, under the stores below
      __threadfence();
      const int left = gr.ntiles - 1 - atomicAdd(a.gbar + a.G + tl.group, 1);
      int left_all = 1;
      if (ti + static_cast<int>(gridDim.x) >= a.ntiles) left_all = static_cast<int>(gridDim.x) - 1 - atomicAdd(a.done, 1);
      s_last[0] = left == 0;
      s_last[1] = left_all == 0;
    }
    for (int e = tid; e < Q * TV && !failed; e += kFusedThreads) {
      const int v = e % TV;
      if (v >= tl.count) continue;
      const size_t ix = static_cast<size_t>(e / TV) * Vp + tl.slot0 + v;
      const int at = v * QS + e / TV;
      a.theta[ix] = s_st[at];
      a.m[ix] = s_st[TV * QS + at];
      a.v[ix] = s_st[2 * TV * QS + at];
    }
    __syncthreads();
    if (s_last[0]) {
      __threadfence();
      local_objectives(a, gr, tl.group, step, s_J);
      if (tid == 0) a.gbar[a.G + tl.group] = 0;
    }
  }
  // the last CTA: step counter, the next constants, counters
  if (!s_last[1]) return;
  if (LOSS == kLossNLL)
    for (int i = tid; i < a.G; i += kFusedThreads) a.gbar[i] = 0;
  if (tid < 2)
    const_cast<float*>(a.adamc)[tid] = adam_constant(tid, a.lr, a.beta1, a.beta2, static_cast<int64_t>(step) + n_it + 1);
  if (tid == 0) {
    *const_cast<int32_t*>(a.step) = step + n_it;
    *a.done = 0;
  }
}

}  // namespace prism
