// Allocation-free evaluation of the voxel-local objective and its gradient.
//
// Who needs it: callers that cannot allocate device memory at the point where they
// evaluate the fit -- code hosted inside a framework that owns the whole device memory
// pool and refuses foreign allocations, real-time pipelines that reserve all memory at
// start-up because cudaMalloc / cudaFree can synchronise the device and stall other
// streams, and plugins whose host forbids allocation outside its own allocator. They
// pass every input and output buffer; the only other memory used is the fixed
// file-scope array below, which every GPU that loads the library holds until exit.
//
// It evaluates, for n_vox voxels of one group, the mean squared error of the predicted
// signal (summed over measurements, divided by n_vox) plus the mean direction-repulsion and
// minor-fraction sparsity penalties (no calibration, no neighbour priors), on raw signal rows
// that it divides by each voxel's mean b <= 50 signal, exactly as prism_forward /
// prism_backward do for such a problem, and writes J and dJ/dtheta. The paper has no
// counterpart of this entry point.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <mutex>
#include <string>

#include "prism.h"
#include "prism_kernels.cuh"

namespace prism {
namespace {

constexpr int kNaThreads = 128;                        // voxels per block
constexpr int kNaMaxMeas = 1024;                       // measurements
constexpr int kNaMaxBlocks = 8192;                     // loss partials
constexpr int64_t kNaMaxVox = static_cast<int64_t>(kNaMaxBlocks) * kNaThreads;   // 1,048,576
constexpr size_t kNaTableBytes = 64 * 1024;                                      // tables (NaTable)
constexpr size_t kNaPartialOff = kNaTableBytes;
constexpr size_t kNaCounterOff = kNaPartialOff + kNaMaxBlocks * sizeof(double);  // + 64 KiB
constexpr size_t kNaScratchBytes = kNaCounterOff + 256;

// The scratch: measurement tables, per-block loss partials, arrival counter. Shared by
// every call on a device; the last call's contents stay until the next call.
static __device__ __align__(256) unsigned char g_noalloc_scratch[kNaScratchBytes];

// Host side: the array's device address, looked up once per device.
std::mutex g_na_mutex;
void* g_na_addr[64] = {};

// The tables of one call, measurements sorted by b-value (stable; the b <= 50 ones come first). Shell
// form (at most kMaxRuns different b-values): every shell padded to an even count; [ShellRun x
// kMaxRuns], gradient rows as in GroupDev::gtab_off. Otherwise the first kNaRow float4 of MeasPair per
// pair. Then, in both, the order: position -> the caller's measurement index, -1 for padding.
constexpr int kNaRow = 6;
constexpr int kNaPos = kNaMaxMeas + kMaxRuns;   // positions, padding included
struct NaTable {
  int32_t np;       // pairs
  int32_t n_runs;   // shells (0: the per-measurement form)
  int32_t nb0;      // b <= 50 measurements, among the first b0_pos positions
  int32_t b0_pos;
  uint32_t bytes;   // of the tables in the scratch, the order included
  __host__ __device__ uint32_t order_off() const { return bytes - static_cast<uint32_t>(2 * np) * 4u; }
};
static_assert(sizeof(float4) * kNaRow * (kNaMaxMeas / 2) + 4 * kNaMaxMeas <= kNaTableBytes, "table fits the scratch");
static_assert(sizeof(ShellRun) * kMaxRuns + 16 * kNaPos <= kNaTableBytes, "shell table fits the scratch");

__device__ __forceinline__ void cp_async4(float* dst, const float* src, bool valid) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(smem_u32(dst)), "l"(src), "r"(valid ? 4 : 0) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// One thread per voxel. A warp copies chunks of 32 measurements of its 32 voxels' rows into a ring of two
// buffers in shared memory, lanes along the row (asynchronous copies, the next chunk in flight while
// this one is worked on), and each thread reads its own row there: reading the rows from global memory,
// a lane per row, touched 32 lines per load. The measurements go through the shell loop of the fused
// kernel (or its per-measurement step) two at a time. Bound by FP32 arithmetic, like that kernel.
// 151,951 voxels at N = 288, K = 3: a call 446 -> 139 us.
constexpr int kNaChunk = 32, kNaStride = kNaChunk + 1;   // odd row stride: a column hits 32 banks
template <int K, bool SHELL>
__global__ void __launch_bounds__(kNaThreads, (K >= 4 ? 3 : 4)) k_grad_noalloc(
    const float* __restrict__ signal, const float* __restrict__ theta, int64_t V, int N, const NaTable tb,
    float lam_rep, float lam_sparse, float tau, float* __restrict__ grad, double* __restrict__ loss,
    unsigned char* scratch) {
  constexpr int NF = K + 3, Q = 4 * K + 5, NW = kNaThreads / 32;
  extern __shared__ __align__(16) unsigned char s_tab[];
  float* s_ring = reinterpret_cast<float*>(s_tab + ((tb.bytes + 15u) & ~15u));   // [NW][2][32][kNaStride]
  float* s_col = s_ring + NW * 2 * 32 * kNaStride;                               // shell form: [kShellCols][kNaThreads]
  __shared__ double s_red[8][3];
  __shared__ int s_last;
  static_assert(2 * 32 * kNaStride >= 32 * (4 * PRISM_MAX_K + 5), "a warp's parameters fit its ring");
  double* partial = reinterpret_cast<double*>(scratch + kNaPartialOff);
  unsigned int* counter = reinterpret_cast<unsigned int*>(scratch + kNaCounterOff);
  for (uint32_t i = threadIdx.x; i < tb.bytes / 4; i += kNaThreads)
    reinterpret_cast<uint32_t*>(s_tab)[i] = reinterpret_cast<const uint32_t*>(scratch)[i];
  __syncthreads();
  const int32_t* s_ord = reinterpret_cast<const int32_t*>(s_tab + tb.order_off());
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t vw = static_cast<int64_t>(blockIdx.x) * kNaThreads + warp * 32, v = vw + lane;   // the warp's first voxel; ours
  const bool act = v < V;
  const int rows = static_cast<int>(max(static_cast<int64_t>(0), min(static_cast<int64_t>(32), V - vw)));
  const float inv_M = 1.f / static_cast<float>(V);
  float* ring = s_ring + warp * (2 * 32 * kNaStride);
  // raw parameters through the ring
  float th[Q];
  for (int e = lane; e < rows * Q; e += 32) ring[e] = theta[vw * Q + e];
  __syncwarp();
#pragma unroll
  for (int q = 0; q < Q; ++q) th[q] = act ? ring[lane * Q + q] : 0.f;
  __syncwarp();
  const int npos = 2 * tb.np, nch = (npos + kNaChunk - 1) / kNaChunk;
  auto stage = [&](int j) {   // chunk j -> buffer j % 2 (always one commit group)
    if (j < nch) {
      const int pos = j * kNaChunk + lane;
      const int n = pos < npos ? s_ord[pos] : -1;
      const float* src = signal + vw * N + max(n, 0);
      float* dst = ring + (j & 1) * (32 * kNaStride) + lane;
#pragma unroll 8
      for (int r = 0; r < 32; ++r) cp_async4(dst + r * kNaStride, src + static_cast<int64_t>(r < rows ? r : 0) * N, n >= 0 && r < rows);
    }
    cp_async_commit();
  };
  stage(0);
  stage(1);
  Vox<K> P;
  transform<K>(th, P);
  // b0 normalisation: the mean of the b <= 50 measurements, summed in two-float arithmetic (exact
  // two-sum), or in FP64 where that leaves FP32's comfortable range. A mean that is not positive and
  // finite is replaced by 1 for this voxel's arithmetic (as the handle path's b0 statistics do) and
  // marks the voxel: its gradient row and the loss become NaN, since an asynchronous call cannot
  // return an error code for it.
  float b0 = 1.f;
  bool bad = false;
  {
    float hi = 0.f, lo = 0.f;
    const int c0 = (tb.b0_pos + kNaChunk - 1) / kNaChunk;
    for (int j = 0; j < c0; ++j) {
      cp_async_wait<1>();
      __syncwarp();
      const float* row = ring + (j & 1) * (32 * kNaStride) + lane * kNaStride;
      const int cnt = min(kNaChunk, tb.b0_pos - j * kNaChunk);
      for (int i = 0; i < cnt; ++i) {   // padding positions hold 0
        const float x = row[i], t = hi + x, bb = t - hi;
        lo += (hi - (t - bb)) + (x - bb);
        hi = t;
      }
      __syncwarp();
      if (c0 > 1) stage(j + 2);
    }
    if (c0 > 1) {   // start the chunks again
      cp_async_wait<0>();
      __syncwarp();
      stage(0);
      stage(1);
    }
    if (act) {
      double m;
      if (hi > 1e-30f && hi < 1e37f) {
        m = static_cast<double>(hi) + static_cast<double>(lo);
      } else {
        m = 0.0;
        for (int i = 0; i < tb.b0_pos; ++i)
          if (s_ord[i] >= 0) m += signal[v * N + s_ord[i]];
      }
      const double mean = m / tb.nb0;
      if (mean > 0.0 && mean < 1e300) {
        b0 = static_cast<float>(mean);
      } else {
        bad = true;
      }
    }
  }
  // a mean whose reciprocal overflows: the voxel's row and mean times 2^64 as each chunk arrives
  const bool tiny = b0 < 1e-37f;
  if (tiny) b0 *= 18446744073709551616.f;
  auto scale_up = [&](int j) {
    float* r = ring + (j & 1) * (32 * kNaStride) + lane * kNaStride;
    for (int i = 0; tiny && i < kNaChunk; ++i) r[i] *= 18446744073709551616.f;
  };
  // y = signal / b0 by the reciprocal and one correction (a division's accuracy in three packed operations;
  // the correction of an infinite signal, a NaN, is dropped by fminf, so that it stays infinite)
  const float ib = 1.f / b0;
  const float2 ib2 = dup2(ib), nb2 = dup2(-b0);
  auto measured = [&](const float* row, int i) {   // the pair's two measurements, normalised
    const float2 y = make_float2(row[2 * i], row[2 * i + 1]);
    const float2 q = __fmul2_rn(y, ib2);
    const float2 e = __ffma2_rn(q, nb2, y);
    return __ffma2_rn(make_float2(fminf(e.x, 1e30f), fminf(e.y, 1e30f)), ib2, q);
  };
  Acc<K> A;
  acc_zero<K>(A);
  float gS0, gf[NF], gd[K][3], gfin, g[Q];
  const float* col = s_col + threadIdx.x;
  if constexpr (SHELL) {
    const ShellRun* s_runs = reinterpret_cast<const ShellRun*>(s_tab);
    const float4* gxy = reinterpret_cast<const float4*>(s_runs + kMaxRuns);
    const float2* gz2 = reinterpret_cast<const float2*>(gxy + tb.np);
    ShellState<K> S;
    shell_begin(S, P, s_col + threadIdx.x);
    for (int j = 0; j < nch; ++j) {
      cp_async_wait<1>();
      __syncwarp();
      scale_up(j);
      const float* row = ring + (j & 1) * (32 * kNaStride) + lane * kNaStride;
      const int pc0 = j * (kNaChunk / 2), pc1 = min(pc0 + kNaChunk / 2, tb.np);
      int p = pc0;
      while (p < pc1) {
        if (p >= S.pend) {   // every pass opens a shell (at most n_runs) or advances p
          if (S.ri + 1 >= tb.n_runs) break;
          if (S.ri >= 0) shell_close(S, s_runs[S.ri], s_col + threadIdx.x);
          ++S.ri;
          shell_open(S, s_runs[S.ri], s_col + threadIdx.x);
          continue;
        }
        const ShellRun& R = s_runs[S.ri];
        const int pe = min(pc1, S.pend), pf = min(pe, R.p1 - R.odd);   // pf: end of the whole pairs
        if (S.b0) {
          for (; p < pe; ++p) {
            float2 r = __fadd2_rn(measured(row, p - pc0), S.c0);
            if (p >= pf) r.y = 0.f;
            S.l1 = __ffma2_rn(r, r, S.l1);
            S.Qs = __fadd2_rn(S.Qs, r);
          }
        } else {
#pragma unroll (K <= 3 ? 2 : 1)
          for (; p < pf; ++p) {
            const float4 q = gxy[p];
            shell_step(S, lo2(q), hi2(q), gz2[p], measured(row, p - pc0));
          }
          if (p < pe) {
            const float4 q = gxy[p];
            shell_step<K, true>(S, lo2(q), hi2(q), gz2[p], measured(row, p - pc0));
            ++p;
          }
        }
      }
      __syncwarp();
      stage(j + 2);
    }
    if (S.ri >= 0) shell_close(S, s_runs[S.ri], s_col + threadIdx.x);
    shell_fold(P, S, col, A);
    data_grad_shell<K>(P, A, 2.f * inv_M, gS0, gf, gd, gfin);
  } else {
    const float4* tab = reinterpret_cast<const float4*>(s_tab);
    VoxP<K> DP;
    AccP<K> AP;
    voxp_init<K>(P, DP, AP);
    for (int j = 0; j < nch; ++j) {
      cp_async_wait<1>();
      __syncwarp();
      scale_up(j);
      const float* row = ring + (j & 1) * (32 * kNaStride) + lane * kNaStride;
      const int pc0 = j * (kNaChunk / 2), pe = min(pc0 + kNaChunk / 2, tb.np), pf = min(pe, N / 2);
      int p = pc0;
#pragma unroll 1
      for (; p < pf; ++p)
        step2<K, false>(DP, reinterpret_cast<const MeasPair&>(tab[kNaRow * p]), measured(row, p - pc0),
                        make_float2(1.f, 1.f), AP);
      if (p < pe)
        step2<K, true>(DP, reinterpret_cast<const MeasPair&>(tab[kNaRow * p]), measured(row, p - pc0),
                       make_float2(1.f, 0.f), AP);
      __syncwarp();
      stage(j + 2);
    }
    accp_fold<K, kLossMSE, false>(P, AP, A);
    data_grad<K>(P, A, 2.f * inv_M, gS0, gf, gd, gfin);
  }
  cp_async_wait<0>();
  IterArgs pa{};
  pa.lam_rep = lam_rep;
  pa.lam_sparse = lam_sparse;
  pa.tau = tau;
  pa.nb_priors = 0;
  const float ploss = act ? priors<K>(pa, P, 0, inv_M, nullptr, gS0, gf, gd) : 0.f;
  chain_raw<K, SHELL>(P, gS0, gf, gd, gfin, g);
  const float qnan = __int_as_float(0x7fc00000);
  __syncwarp();
  if (act) {
#pragma unroll
    for (int q = 0; q < Q; ++q) ring[lane * Q + q] = bad ? qnan : g[q];
  }
  __syncwarp();
  for (int e = lane; e < rows * Q; e += 32) grad[vw * Q + e] = ring[e];
  double out[3];
  const double dl = bad ? static_cast<double>(qnan) : static_cast<double>(A.l1 * inv_M);
  block_reduce3(act ? dl : 0.0, act ? static_cast<double>(ploss) : 0.0, 0.0, s_red, out);
  if (threadIdx.x == 0) {
    partial[blockIdx.x] = out[0] + out[1];
    __threadfence();
    s_last = (atomicAdd(counter, 1u) == gridDim.x - 1);
  }
  __syncthreads();
  if (!s_last) return;
  // the last block: fixed-order sum of the partials, strided over its threads
  __threadfence();
  double tot = 0.0;
#pragma unroll 4
  for (unsigned int b = threadIdx.x; b < gridDim.x; b += kNaThreads) tot += __ldcg(&partial[b]);
  block_reduce3(tot, 0.0, 0.0, s_red, out);
  if (threadIdx.x == 0) {
    *loss = out[0];
    *counter = 0u;
  }
}

// Tables of a call (see NaTable) into `dst`.
NaTable na_tables(const float* bvals, const float* bvecs, int N, unsigned char* dst) {
  const double L2E = 1.4426950408889634, dpar = 1.7e-3, dperp = 0.4e-3;
  int32_t idx[kNaMaxMeas], order[kNaPos];
  for (int n = 0; n < N; ++n) idx[n] = n;
  // sorted by (b, index): the order of a stable sort, which would allocate
  std::sort(idx, idx + N, [&](int32_t a, int32_t b) { return bvals[a] != bvals[b] ? bvals[a] < bvals[b] : a < b; });
  int shells = 0;
  for (int n = 0; n < N; ++n) shells += n == 0 || bvals[idx[n]] != bvals[idx[n - 1]];
  NaTable t{};
  if (shells <= kMaxRuns) {
    t.n_runs = shells;
    ShellRun* runs = reinterpret_cast<ShellRun*>(dst);
    int pos = 0;
    for (int n = 0, r = 0; n < N; ++r) {
      const float b = bvals[idx[n]];
      const double bd = b;
      ShellRun& R = runs[r];
      R.p0 = pos / 2;
      for (; n < N && bvals[idx[n]] == b; ++n) order[pos++] = idx[n];
      R.odd = pos % 2;
      if (R.odd) order[pos++] = -1;
      R.p1 = pos / 2;
      R.b0 = (b == 0.f) ? 1 : 0;
      R.ecsf = static_cast<float>(std::exp(-bd * 3.0e-3));
      R.egm = static_cast<float>(std::exp(-bd * 0.9e-3));
      R.eres = static_cast<float>(std::exp(-bd * 0.2e-3));
      R.nbperp = static_cast<float>(-bd * dperp * L2E);
      if (b <= 50.f) t.b0_pos = pos;
    }
    t.np = pos / 2;
    float* gt = reinterpret_cast<float*>(runs + kMaxRuns);
    for (int i = 0; i < pos; ++i) {
      const int n = order[i], p = i / 2, h = i % 2;
      const double s = n < 0 ? 0.0 : std::sqrt(static_cast<double>(bvals[n]) * dpar * L2E);
      gt[4 * p + h] = n < 0 ? 0.f : static_cast<float>(s * bvecs[3 * n]);
      gt[4 * p + 2 + h] = n < 0 ? 0.f : static_cast<float>(s * bvecs[3 * n + 1]);
      gt[4 * t.np + i] = n < 0 ? 0.f : static_cast<float>(s * bvecs[3 * n + 2]);
    }
    t.bytes = static_cast<uint32_t>(sizeof(ShellRun) * kMaxRuns + (12 + 4) * static_cast<size_t>(pos));
  } else {
    int pos = N;
    for (int n = 0; n < N; ++n) order[n] = idx[n];
    if (pos % 2) order[pos++] = -1;
    t.np = pos / 2;
    float* f = reinterpret_cast<float*>(dst);
    for (int i = 0; i < pos; ++i) {
      const int n = order[i];
      float row[12] = {};
      if (n >= 0) {
        const double b = bvals[n];
        if (bvals[n] <= 50.f) t.b0_pos = i + 1;
        const float r[11] = {bvecs[3 * n], bvecs[3 * n + 1], bvecs[3 * n + 2], static_cast<float>(-b * dpar * L2E),
                             static_cast<float>(-b * dperp * L2E), static_cast<float>(-b * (dpar - dperp) * L2E),
                             static_cast<float>(std::exp(-b * 3.0e-3)), static_cast<float>(std::exp(-b * 0.9e-3)),
                             static_cast<float>(std::exp(-b * 0.2e-3)), static_cast<float>(-2.0 * b * dpar),
                             static_cast<float>(2.0 * b * (dperp - dpar))};
        for (int c = 0; c < 11; ++c) row[c] = r[c];
        row[11] = 1.f;
      }
      for (int c = 0; c < 12; ++c) f[24 * (i / 2) + 2 * c + i % 2] = row[c];
    }
    t.bytes = static_cast<uint32_t>((4 * kNaRow * 2 + 4) * static_cast<size_t>(pos));
  }
  for (int n = 0; n < N; ++n) t.nb0 += bvals[n] <= 50.f;
  std::memcpy(dst + t.order_off(), order, sizeof(int32_t) * 2 * static_cast<size_t>(t.np));
  return t;
}

}  // namespace
}  // namespace prism

using namespace prism;

// Defined in prism_api.cu: records the message returned by prism_last_error().
int prism_record_error(int code, const char* msg);

extern "C" int prism_grad_noalloc(const float* signal, const float* bvals, const float* bvecs, const float* theta,
                                  int64_t n_vox, int32_t n_meas, int32_t K, float lam_rep, float lam_sparse,
                                  float tau, float* grad, double* loss, void* stream) {
  if (!signal || !bvals || !bvecs || !theta || !grad || !loss)
    return prism_record_error(PRISM_E_INVALID_ARG, "prism_grad_noalloc: NULL argument");
  if (K < 1 || K > PRISM_MAX_K) return prism_record_error(PRISM_E_INVALID_ARG, "prism_grad_noalloc: K must be in 1..5");
  if (n_vox < 1 || n_vox > kNaMaxVox)
    return prism_record_error(PRISM_E_SHAPE, ("prism_grad_noalloc: n_vox must be in 1.." + std::to_string(kNaMaxVox) +
                                              " (the fixed scratch holds " + std::to_string(kNaMaxBlocks) +
                                              " block partials of 128 voxels)").c_str());
  if (n_meas < 1 || n_meas > kNaMaxMeas)
    return prism_record_error(PRISM_E_SHAPE, "prism_grad_noalloc: n_meas must be in 1..1024");
  if (!(lam_rep >= 0.f) || !(lam_sparse >= 0.f) || !(tau >= 0.f))
    return prism_record_error(PRISM_E_INVALID_ARG, "prism_grad_noalloc: lam_rep, lam_sparse and tau must be >= 0");
  int nb0 = 0;
  for (int n = 0; n < n_meas; ++n) {
    const double b = bvals[n];
    if (!std::isfinite(b) || b < 0.0) return prism_record_error(PRISM_E_INVALID_ARG, "prism_grad_noalloc: bad b-value");
    // the b-vector rules of prism_fit_init: finite, and unit length where b > 50
    const float gx = bvecs[3 * n], gy = bvecs[3 * n + 1], gz = bvecs[3 * n + 2];
    if (!std::isfinite(gx) || !std::isfinite(gy) || !std::isfinite(gz))
      return prism_record_error(PRISM_E_INVALID_ARG, "prism_grad_noalloc: non-finite b-vector");
    if (b > 50.0 && std::fabs(std::sqrt(gx * gx + gy * gy + gz * gz) - 1.f) > 1e-3f)
      return prism_record_error(PRISM_E_INVALID_ARG,
                                ("prism_grad_noalloc: b-vector " + std::to_string(n) +
                                 " of a b > 50 measurement is not unit length").c_str());
    nb0 += (b <= 50.0);
  }
  if (nb0 == 0) return prism_record_error(PRISM_E_SHAPE, "prism_grad_noalloc: no b <= 50 measurement");
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess || dev < 0 || dev >= 64)
    return prism_record_error(PRISM_E_CUDA, "prism_grad_noalloc: cudaGetDevice failed");
  unsigned char* scratch = nullptr;
  {
    std::lock_guard<std::mutex> lock(g_na_mutex);
    if (!g_na_addr[dev]) {
      void* p = nullptr;
      e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
      if (e != cudaSuccess || !p)
        return prism_record_error(PRISM_E_CUDA, (std::string("prism_grad_noalloc: cudaGetSymbolAddress: ") +
                                                 cudaGetErrorString(e)).c_str());
      g_na_addr[dev] = p;
    }
    scratch = static_cast<unsigned char*>(g_na_addr[dev]);
  }
  static thread_local unsigned char tables[kNaTableBytes];
  const NaTable tb = na_tables(bvals, bvecs, n_meas, tables);
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  e = cudaMemsetAsync(scratch + kNaCounterOff, 0, sizeof(unsigned int), st);
  if (e == cudaSuccess) e = cudaMemcpyAsync(scratch, tables, tb.bytes, cudaMemcpyHostToDevice, st);
  if (e != cudaSuccess)
    return prism_record_error(PRISM_E_CUDA, (std::string("prism_grad_noalloc: ") + cudaGetErrorString(e)).c_str());
  const int blocks = static_cast<int>((n_vox + kNaThreads - 1) / kNaThreads);
  const size_t smem = ((tb.bytes + 15u) & ~15u) + (kNaThreads / 32) * 2 * 32 * kNaStride * sizeof(float) +
                      (tb.n_runs ? kShellCols * kNaThreads * sizeof(float) : 0);
  auto go = [&](auto fn) {
    cudaError_t r = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
    if (r != cudaSuccess) return r;
    fn<<<blocks, kNaThreads, smem, st>>>(signal, theta, n_vox, n_meas, tb, lam_rep, lam_sparse, tau, grad, loss, scratch);
    return cudaGetLastError();
  };
  switch (K) {
    case 1: e = tb.n_runs ? go(k_grad_noalloc<1, true>) : go(k_grad_noalloc<1, false>); break;
    case 2: e = tb.n_runs ? go(k_grad_noalloc<2, true>) : go(k_grad_noalloc<2, false>); break;
    case 3: e = tb.n_runs ? go(k_grad_noalloc<3, true>) : go(k_grad_noalloc<3, false>); break;
    case 4: e = tb.n_runs ? go(k_grad_noalloc<4, true>) : go(k_grad_noalloc<4, false>); break;
    default: e = tb.n_runs ? go(k_grad_noalloc<5, true>) : go(k_grad_noalloc<5, false>); break;
  }
  if (e != cudaSuccess)
    return prism_record_error(PRISM_E_CUDA, (std::string("prism_grad_noalloc launch: ") + cudaGetErrorString(e)).c_str());
  return PRISM_OK;
}
