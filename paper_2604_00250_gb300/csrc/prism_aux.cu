// Non-templated PRISM kernels: preprocessing (b0 normalisation, packing, measurement
// tables, parameter layout), the plain-path data term and Adam, and the group-level
// reductions and updates of the calibration / noise parameters (Sec. 2.3).
#include <math.h>

#include "prism_kernels.cuh"
#include "prism_launch.h"

namespace prism {

// ---------------------------------------------------------------------------
// Preprocessing (Sec. 2.5: both y and y_hat are divided by the measured b0).
// ---------------------------------------------------------------------------
// b0 mean of every voxel and the block's sum of the squared b0 deviations, part[block]: kB0Lanes lanes
// per voxel read the b <= 50 measurements (`b0n`, nb0 of them) and nothing else of the row; k_pack, which
// reads all of it, looks for the other non-finite values. The per-voxel sums are FP32 (a b0 mean of a few dozen
// positive values, stored as FP32); the squared deviations accumulate in FP64. A voxel whose mean is not
// positive, or takes in a non-finite value, is counted in *bad and stored as -1. `rows`: the voxels' rows in `sig`, or null for
// rows in order. (A warp per voxel over the whole row: 164 us of 141,000 voxels at N = 288, 30 us now.)
constexpr int kB0Lanes = 8, kB0Vox = 256 / kB0Lanes;
__global__ void __launch_bounds__(256) k_b0_stats(const float* __restrict__ sig, const int64_t* __restrict__ rows,
                                                  int64_t V, int N, const int32_t* __restrict__ b0n, int nb0,
                                                  float* __restrict__ b0mean, double* __restrict__ part, int* bad) {
  __shared__ double s[8];
  __shared__ int32_t s_n[1024];   // nb0 <= N <= 1024 (prism_fit_init checks it)
  for (int n = threadIdx.x; n < nb0; n += blockDim.x) s_n[n] = b0n[n];
  __syncthreads();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, sub = lane % kB0Lanes;
  const int64_t v = static_cast<int64_t>(blockIdx.x) * kB0Vox + threadIdx.x / kB0Lanes;
  const bool ok = v < V;
  const float* row = sig + (ok ? (rows ? rows[v] : v) : 0) * N;
  float m = 0.f;
  bool finite = true;
#pragma unroll 4
  for (int i = sub; i < nb0; i += kB0Lanes) {
    const float x = ok ? row[s_n[i]] : 0.f;
    finite = finite && isfinite(x);
    m += x;
  }
  const unsigned lanes = ((1u << kB0Lanes) - 1u) << (lane - sub);   // the voxel's
  finite = (__ballot_sync(0xffffffffu, finite) & lanes) == lanes;
#pragma unroll
  for (int o = kB0Lanes / 2; o > 0; o >>= 1) m += __shfl_xor_sync(0xffffffffu, m, o);
  m /= static_cast<float>(nb0);
  const bool good = finite && m > 0.f;
  if (ok && sub == 0) {
    b0mean[v] = good ? m : -1.f;
    if (!good) atomicAdd(bad, 1);
  }
  double acc = 0.0;
  const float inv = good ? 1.f / m : 1.f;
#pragma unroll 4
  for (int i = sub; i < nb0; i += kB0Lanes) {
    const float d = ok ? fmaf(row[s_n[i]], inv, -1.f) : 0.f;
    acc += static_cast<double>(d * d);
  }
  acc = warp_sum_d(acc);
  if (lane == 0) s[warp] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < 8; ++w) acc += s[w];
    part[blockIdx.x] = acc;
  }
}

// sigma init (Sec. 2.3 learns sigma but does not say where it starts): pooled std of the
// normalised b0 repeats, clamped >= 1e-3. One block, strided over the partials, then a fixed tree
// (one thread reading them in turn took 24 us for 550).
__global__ void __launch_bounds__(256) k_sigma_init(const double* part, int nblocks, int64_t V, int nb0, float fallback,
                                                    float* sigma_log) {
  __shared__ double s_w[8];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  double s = 0.0;
#pragma unroll 4
  for (int b = threadIdx.x; b < nblocks; b += 256) s += part[b];
  s = warp_sum_d(s);
  if (lane == 0) s_w[warp] = s;
  __syncthreads();
  if (threadIdx.x != 0) return;
  for (int w = 1; w < 8; ++w) s += s_w[w];
  double sg = fallback;
  if (nb0 >= 2) sg = fmax(sqrt(s / (static_cast<double>(V) * (nb0 - 1))), 1e-3);
  *sigma_log = static_cast<float>(log(sg));
}

// One warp column of a tile (VW voxels) per block of kPackThreads, in chunks of kPackC measurements
// staged in shared memory so that the reads run along the voxels' signal rows and the writes along the
// packed [pair][voxel][2] layout (ypos). A voxel with a non-finite measurement is counted in *bad
// (unless its b0 mean already was). Bound by the loads in flight: a block per tile, its four columns in
// turn, took 118 us for 141,000 voxels at N = 288, now 65 us.
constexpr int kPackThreads = 256, kPackC = 128;
template <int VW>
__global__ void __launch_bounds__(kPackThreads) k_pack(const IterArgs a, const float* __restrict__ sig,
                                                       const int64_t* __restrict__ rows,
                                                       const float* __restrict__ b0mean,
                                                       const int32_t* __restrict__ vox_of_slot,
                                                       const int32_t* __restrict__ order, int64_t vox0, int tile_begin,
                                                       int N, int npos, float* __restrict__ ypack, int* bad) {
  __shared__ float s[VW][kPackC + 1];
  __shared__ int64_t s_row[VW];   // the voxel's signal row (-1: padding slot)
  __shared__ float s_inv[VW];     // 1 / its b0 mean (-1 where that was refused)
  __shared__ int s_bad[VW];
  const int t = tile_begin + blockIdx.x, w = blockIdx.y;
  const Tile tl = a.tiles[t];
  const int NP = (npos + 3) & ~3;   // positions: order[] holds the measurement of each, -1 for padding
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (threadIdx.x < VW) {
    const int vl = w * VW + threadIdx.x;
    int64_t r = -1;
    float inv = 0.f;
    if (vl < tl.count) {
      const int64_t v = vox_of_slot[tl.slot0 + vl] - vox0;
      r = (rows ? rows[v] : v) * N;
      const float m = b0mean[v];
      inv = m > 0.f ? 1.f / m : -1.f;
    }
    s_row[threadIdx.x] = r;
    s_inv[threadIdx.x] = inv;
    s_bad[threadIdx.x] = 0;
  }
  __syncthreads();
  for (int n0 = 0; n0 < NP; n0 += kPackC) {
    const int C = min(kPackC, NP - n0);   // even (NP and kPackC are multiples of 4)
    int32_t on[kPackC / 32];   // the measurements this lane reads of every row (-1: padding)
#pragma unroll
    for (int q = 0; q < kPackC / 32; ++q) {
      const int n = n0 + lane + 32 * q;
      on[q] = (n < npos) ? order[n] : -1;
    }
    // a warp per voxel row, its loads and those of the next rows in flight together
#pragma unroll
    for (int j = warp; j < VW; j += kPackThreads / 32) {
      const int64_t r = s_row[j];
      const float inv = s_inv[j];
      bool nonfinite = false;
#pragma unroll
      for (int q = 0; q < kPackC / 32; ++q) {
        const float x = (r >= 0 && on[q] >= 0) ? sig[r + on[q]] : 0.f;
        nonfinite = nonfinite || !isfinite(x);
        if (lane + 32 * q < C) s[j][lane + 32 * q] = x * inv;
      }
      if (nonfinite) s_bad[j] = 1;
    }
    __syncthreads();
    float* out = ypack + tl.y_off + static_cast<size_t>(w) * NP * VW + static_cast<size_t>(n0) * VW;
#pragma unroll 8
    for (int i = threadIdx.x; i < VW * C; i += kPackThreads) {
      const int pc = i / (2 * VW), r = i - pc * 2 * VW, j = r >> 1;
      out[i] = s[j][2 * pc + (r & 1)];
    }
    __syncthreads();
  }
  if (threadIdx.x < VW && s_bad[threadIdx.x] && s_inv[threadIdx.x] >= 0.f) atomicAdd(bad, 1);
}

// Static part of the per-measurement table; exp(alpha) = 1, beta = 0 (identity, Sec. 2.3).
__global__ void k_table(const float* bvals, const float* bvecs, int N, MeasRow* rows) {
  const int n = blockIdx.x * blockDim.x + threadIdx.x;
  if (n >= N) return;
  const double b = bvals[n];
  const double L2E = 1.4426950408889634;
  const double dpar = 1.7e-3, dperp = 0.4e-3;          // Eq. 5, mm^2/s
  MeasRow r;
  r.gx = bvecs[3 * n];
  r.gy = bvecs[3 * n + 1];
  r.gz = bvecs[3 * n + 2];
  r.nkpar = static_cast<float>(-b * dpar * L2E);
  r.nkperp = static_cast<float>(-b * dperp * L2E);
  r.nkd = static_cast<float>(-b * (dpar - dperp) * L2E);
  r.ecsf = static_cast<float>(exp(-b * 3.0e-3));          // Eq. 4
  r.egm = static_cast<float>(exp(-b * 0.9e-3));
  r.eres = static_cast<float>(exp(-b * 0.2e-3));
  r.An = static_cast<float>(-2.0 * b * dpar);
  r.Bn = static_cast<float>(2.0 * b * (dperp - dpar));
  r.A = 1.f;
  r.beta = 0.f;
  r.pad0 = r.pad1 = r.pad2 = 0.f;
  rows[n] = r;
}

// Paired table of one group (MeasPair), zero past N.
__global__ void k_pair_table(const MeasRow* rows, int N, int NP, MeasPair* out) {
  const int pidx = blockIdx.x * blockDim.x + threadIdx.x;
  if (pidx >= NP / 2) return;
  const float* r0 = reinterpret_cast<const float*>(rows + 2 * pidx);
  const bool v0 = 2 * pidx < N, v1 = 2 * pidx + 1 < N;
  float f0[16], f1[16];
  for (int f = 0; f < 16; ++f) {
    f0[f] = v0 ? r0[f] : 0.f;
    f1[f] = v1 ? r0[16 + f] : 0.f;
  }
  // field order of MeasRow: gx gy gz nkpar nkperp nkd ecsf egm eres An Bn A beta pad pad pad
  MeasPair mp;
  float* o = reinterpret_cast<float*>(&mp);
  for (int f = 0; f < 16; ++f) {
    o[2 * f] = f0[f];
    o[2 * f + 1] = f1[f];
  }
  out[pidx] = mp;
}

// Slots of one volume's voxels, a block per patch: slots run over a patch's masked voxels in C order from
// its first tile on, so each thread counts its share of the patch's (x, y) lines, a block-wide
// exclusive sum gives their first slots, and a second walk writes the voxel <-> slot <-> grid tables and
// packed coordinates (and, for a slab, the voxels' rows in the whole volume). The host passes over
// every voxel that this replaces took 1.45 ms of a slab set-up of 280,000 voxels, and 20 bytes per
// grid position and voxel of uploads; the host now counts the masks (0.2 ms), and this takes 57 us.
constexpr int kPlanThreads = 128;
__global__ void __launch_bounds__(kPlanThreads) k_plan(const PlanArgs p, const GroupDev* __restrict__ groups) {
  __shared__ int s_sum[kPlanThreads / 32];
  const GroupDev gr = groups[p.g];
  const int P = p.P, py = (gr.ny + P - 1) / P, pz = (gr.nz + P - 1) / P;
  const int pi = blockIdx.x, x0 = pi / (py * pz) * P, y0 = (pi / pz) % py * P, za = pi % pz * P;
  const int wx = min(P, gr.nx - x0), wy = min(P, gr.ny - y0), zb = min(gr.nz, za + P);
  const int per = (wx * wy + kPlanThreads - 1) / kPlanThreads;
  const int l0 = min(wx * wy, static_cast<int>(threadIdx.x) * per), l1 = min(wx * wy, l0 + per);
  auto row_of = [&](int l) { return static_cast<int64_t>(x0 + l / wy) * gr.ny + (y0 + l % wy); };
  int n = 0;
  for (int l = l0; l < l1; ++l) {
    const uint8_t* m = p.mask + row_of(l) * p.stride + p.z0;
    for (int z = za; z < zb; ++z) n += m[z] != 0;
  }
  // exclusive sum over the block's threads
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int inc = n;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int u = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += u;
  }
  if (lane == 31) s_sum[warp] = inc;
  __syncthreads();
  int slot = p.ptile[pi] * p.TV + inc - n;
  for (int w = 0; w < warp; ++w) slot += s_sum[w];
  for (int l = l0; l < l1; ++l) {
    const int64_t row = row_of(l);
    const uint8_t* m = p.mask + row * p.stride + p.z0;
    int k = 0;   // masked voxels of the line before this patch
    for (int z = 0; z < za; ++z) k += m[z] != 0;
    int64_t v = gr.vox0 + p.line[row] + k, wr = 0;
    if (p.rows) {
      for (int z = -p.z0; z < 0; ++z) k += m[z] != 0;
      wr = p.wline[row] + k;
    }
    for (int z = za; z < zb; ++z) {
      const int64_t gi = gr.grid_off + row * gr.nz + z;
      if (!m[z]) {
        p.slot_of_grid[gi] = -1;
        continue;
      }
      p.slot_of_grid[gi] = slot;
      p.slot_of_vox[v] = slot;
      p.vox_of_slot[slot] = static_cast<int32_t>(v);
      p.vcoord[slot] = static_cast<uint32_t>(x0 + l / wy) | (static_cast<uint32_t>(y0 + l % wy) << 10) |
                       (static_cast<uint32_t>(z) << 20);
      if (p.rows) p.rows[v] = wr++;
      ++v;
      ++slot;
    }
  }
}

// Grid position of every masked voxel of a whole volume, a thread per (x, y) line.
__global__ void k_grid_of_vox(const uint8_t* __restrict__ mask, const int32_t* __restrict__ line, int nlines, int nz,
                              int32_t* __restrict__ grid_of_vox) {
  const int l = blockIdx.x * blockDim.x + threadIdx.x;
  if (l >= nlines) return;
  int v = line[l];
  for (int z = 0; z < nz; ++z)
    if (mask[static_cast<int64_t>(l) * nz + z]) grid_of_vox[v++] = l * nz + z;
}

// Per-slot flags and neighbours of one volume from its grid -> slot map (one thread per grid
// position): flags (bits 0-5: the face neighbour in +x, -x, +y, -y, +z, -z is in the
// mask, any patch; bits 8-12: the count of neighbours in the same patch) and the neighbour
// slots in the same patch: the six faces first, then the edges and corners of the 3x3x3 cube
// in (i, j, k) loop order.
__global__ void k_slot_data(const Tile* __restrict__ tiles, const GroupDev* __restrict__ groups, int g,
                            const int32_t* __restrict__ slot_of_grid, int Vp, int TV, int nnb,
                            uint32_t* __restrict__ vflag, int32_t* __restrict__ nbr) {
  const GroupDev gr = groups[g];
  const int64_t ng = static_cast<int64_t>(gr.nx) * gr.ny * gr.nz;
  const int64_t gi = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (gi >= ng) return;
  const int32_t* sog = slot_of_grid + gr.grid_off;
  const int slot = sog[gi];
  if (slot < 0) return;
  const int z = static_cast<int>(gi % gr.nz), y = static_cast<int>((gi / gr.nz) % gr.ny),
            x = static_cast<int>(gi / (static_cast<int64_t>(gr.nz) * gr.ny));
  const int patch = tiles[slot / TV].patch;
  uint32_t fl = 0;
  int cnt = 0;
  int next = 6;   // index of the next edge / corner neighbour
  for (int pass = 0; pass < 2; ++pass)
    for (int i = -1; i <= 1; ++i)
      for (int j = -1; j <= 1; ++j)
        for (int k = -1; k <= 1; ++k) {
          const int l1 = abs(i) + abs(j) + abs(k);
          if (l1 == 0 || (pass == 0) != (l1 == 1)) continue;
          int e;
          if (pass == 0) {
            e = (i != 0) ? (i > 0 ? 0 : 1) : (j != 0) ? (j > 0 ? 2 : 3) : (k > 0 ? 4 : 5);   // +x -x +y -y +z -z
          } else {
            if (next >= nnb) continue;
            e = next++;
          }
          const int xx = x + i, yy = y + j, zz = z + k;
          if (xx < 0 || yy < 0 || zz < 0 || xx >= gr.nx || yy >= gr.ny || zz >= gr.nz) continue;
          const int sj = sog[(static_cast<int64_t>(xx) * gr.ny + yy) * gr.nz + zz];
          if (sj < 0) continue;
          if (e < 6) fl |= 1u << e;
          if (tiles[sj / TV].patch == patch) {
            nbr[static_cast<size_t>(e) * Vp + slot] = sj;
            ++cnt;
          }
        }
  vflag[slot] = fl | (static_cast<uint32_t>(cnt) << 8);
}

// Row gather: dst[i][:] = src[rows[i]][:], a warp per row.
__global__ void __launch_bounds__(256) k_gather_rows(const float* __restrict__ src, const int64_t* __restrict__ rows,
                                                     int64_t n, int len, float* __restrict__ dst) {
  const int64_t i = static_cast<int64_t>(blockIdx.x) * 8 + (threadIdx.x >> 5);
  if (i >= n) return;
  const float* s = src + rows[i] * len;
  float* d = dst + i * len;
#pragma unroll 4
  for (int c = threadIdx.x & 31; c < len; c += 32) d[c] = s[c];
}

// Raw parameters between the caller's rows [V][Q] (mask order; `rows`: row of each voxel, or null for
// rows in order) and the kernels' [Q][Vpad] by slot, kParVox voxels per block through shared memory:
// the rows are read and written along their length, the slots along runs of consecutive voxels. Q =
// 4K + 5 is odd, so a column of the staged rows falls into 32 different banks. (Element by element, the
// strided side took a sector per value: 62 us to read out 740,110 voxels at K = 3, now 17 us.)
constexpr int kParVox = 128;
__global__ void __launch_bounds__(kParVox) k_scatter_params(const float* __restrict__ in,
                                                            const int64_t* __restrict__ rows,
                                                            const int32_t* __restrict__ slot_of_vox, int64_t V, int Q,
                                                            int Vpad, float* __restrict__ theta) {
  extern __shared__ float s_par[];   // [kParVox][Q]
  const int64_t v0 = static_cast<int64_t>(blockIdx.x) * kParVox;
  const int nv = static_cast<int>(min(static_cast<int64_t>(kParVox), V - v0));
  if (rows) {
    for (int e = threadIdx.x; e < nv * Q; e += kParVox) {
      const int v = e / Q;
      s_par[e] = in[rows[v0 + v] * Q + (e - v * Q)];
    }
  } else {
#pragma unroll 8
    for (int e = threadIdx.x; e < nv * Q; e += kParVox) s_par[e] = in[v0 * Q + e];
  }
  __syncthreads();
  if (threadIdx.x >= nv) return;
  const int slot = slot_of_vox[v0 + threadIdx.x];
#pragma unroll 8
  for (int q = 0; q < Q; ++q) theta[static_cast<size_t>(q) * Vpad + slot] = s_par[threadIdx.x * Q + q];
}

__global__ void __launch_bounds__(kParVox) k_gather_params(const float* __restrict__ theta,
                                                           const int32_t* __restrict__ slot_of_vox, int64_t V, int Q,
                                                           int Vpad, float* __restrict__ out) {
  extern __shared__ float s_par[];   // [kParVox][Q]
  const int64_t v0 = static_cast<int64_t>(blockIdx.x) * kParVox;
  const int nv = static_cast<int>(min(static_cast<int64_t>(kParVox), V - v0));
  if (threadIdx.x < nv) {
    const int slot = slot_of_vox[v0 + threadIdx.x];
#pragma unroll 8
    for (int q = 0; q < Q; ++q) s_par[threadIdx.x * Q + q] = theta[static_cast<size_t>(q) * Vpad + slot];
  }
  __syncthreads();
#pragma unroll 8
  for (int e = threadIdx.x; e < nv * Q; e += kParVox) out[v0 * Q + e] = s_par[e];
}

// Counter-based generator: splitmix64 (Steele, Lea, Flood 2014) of (seed, voxel, draw).
__device__ __forceinline__ uint64_t splitmix64(uint64_t x) {
  x += 0x9E3779B97F4A7C15ull;
  x = (x ^ (x >> 30)) * 0xBF58476D1CE4E5B9ull;
  x = (x ^ (x >> 27)) * 0x94D049BB133111EBull;
  return x ^ (x >> 31);
}
__device__ __forceinline__ float u01f(uint64_t h) {
  return (static_cast<float>(h >> 40) + 0.5f) * (1.f / 16777216.f);   // 24 bits, in (0, 1)
}

// Default start: S0 = 1, equal fractions, f_intra = 0.5, directions uniform on the sphere,
// drawn per grid position (so that a voxel starts from the same values whichever of the
// volume's voxels share the handle).
__global__ void k_default_init(const int32_t* __restrict__ slot_of_vox, const uint32_t* __restrict__ vcoord, int ny,
                               int nz, int64_t V, int K, int Vpad, uint64_t seed, float* __restrict__ theta) {
  const int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (i >= V) return;
  const int slot = slot_of_vox[i];
  int cx, cy, cz;
  unpack_coord(vcoord[slot], cx, cy, cz);
  const int64_t v = (static_cast<int64_t>(cx) * ny + cy) * nz + cz;
  theta[slot] = 0.5413248546129181f;   // log(e - 1): S0 = softplus(raw) = 1
  for (int i = 0; i < K + 3; ++i) theta[static_cast<size_t>(1 + i) * Vpad + slot] = 0.f;
  for (int k = 0; k < K; ++k) {
    // normalised Gaussian triple by the Box-Muller transform, in FP32 (u1 >= 2^-25 keeps the
    // radius above 2e-4, so the norm is never 0)
    float g[3];
    for (int c = 0; c < 3; c += 2) {
      const uint64_t base = seed * 0x100000001B3ull ^ (static_cast<uint64_t>(v) << 8) ^ (k * 4 + c);
      const float u1 = u01f(splitmix64(base)), u2 = u01f(splitmix64(base ^ 0xABCDEF12345ull));
      const float rad = sqrtf(-2.f * logf(u1));
      float sn, cs;
      sincospif(2.f * u2, &sn, &cs);
      g[c] = rad * cs;
      if (c + 1 < 3) g[c + 1] = rad * sn;
    }
    const float inv = rsqrtf(g[0] * g[0] + g[1] * g[1] + g[2] * g[2]);
    for (int c = 0; c < 3; ++c) theta[static_cast<size_t>(K + 4 + 3 * k + c) * Vpad + slot] = g[c] * inv;
  }
  theta[static_cast<size_t>(4 * K + 4) * Vpad + slot] = 0.f;
}

// ---------------------------------------------------------------------------
// Plain-path data term and voxel Adam.
// ---------------------------------------------------------------------------
__global__ void k_adam_voxel(const IterArgs a, const PlainArgs pa) {
  const int slot = pa.tile_begin * a.TV + blockIdx.x * blockDim.x + threadIdx.x;
  if (slot >= pa.tile_end * a.TV) return;
  const Tile tl = a.tiles[slot / a.TV];
  if (slot - tl.slot0 >= tl.count) return;
  const float stepsz = a.adamc[0], isbc2 = a.adamc[1];
  for (int q = 0; q < a.Q; ++q) {
    const size_t ix = static_cast<size_t>(q) * a.Vpad + slot;
    const float g = pa.grad[ix];
    if (a.optimizer == 0) {
      const float mq = fmaf(a.beta1, a.m[ix], (1.f - a.beta1) * g);
      const float vq = fmaf(a.beta2, a.v[ix], (1.f - a.beta2) * g * g);
      a.m[ix] = mq;
      a.v[ix] = vq;
      a.theta[ix] -= stepsz * mq / fmaf(sqrtf(vq), isbc2, a.eps);
    } else {
      float th = a.theta[ix], mq = a.m[ix], vq = a.v[ix];
      rprop_update(th, mq, vq, g, a.lr, a.eta_minus, a.eta_plus, a.step_min, a.step_max);
      a.theta[ix] = th;
      a.m[ix] = mq;
      a.v[ix] = vq;
    }
  }
}

// ---------------------------------------------------------------------------
// Group reductions: per-tile partials -> per-group sums, fixed order (two levels:
// splits of `split_tiles` tiles, then the last-arriving block sums the splits).
// Entries: 0 data loss, 1 dJ/dsigma_log, 2 prior loss, 3.. 3+2N alpha / beta.
// A block takes kRedE entries of a split, a quarter of its tiles per 64 threads. Bound by latency and by
// GB300's FP64 rate (an add per warp costs its SM about 16 cycles): the tiles' FP32 partials are
// summed in two-float arithmetic (Knuth's exact two-sum, error below 2^-44 of the sum of magnitudes) and
// only the few sums of sums in FP64; a split's tiles lie at one stride, so their loads go out together.
// (One FP64 chain of 64 tiles per thread, offsets looked up: 34 us for 2,048 tiles at N = 360; 17.5 us now, the adjoint's z pass, 7.4 us before, included.)
// ---------------------------------------------------------------------------
__device__ __forceinline__ void group_reduce_block(const IterArgs& a, const GroupArgs& g, int gi, int s, int ce, int what) {
  __shared__ int s_last;
  __shared__ double s_q[4][kRedE];
  const GroupDev gr = a.groups[gi];
  const int nsplit = (gr.ntiles + g.split_tiles - 1) / g.split_tiles;
  if (s >= nsplit) return;
  const int E = 3 + ((gr.calib && (what & 2)) ? 2 * gr.npos : 0);
  if (ce * kRedE >= E) return;
  const int el = threadIdx.x % kRedE, sub = threadIdx.x / kRedE, e = ce * kRedE + el;
  const int per = (g.split_tiles + 3) / 4, first = s * g.split_tiles + sub * per;
  const int n = min(per, min((s + 1) * g.split_tiles, gr.ntiles) - first);   // this quarter's tiles
  double acc = 0.0;
  if (e < E && n > 0) {
    const int t0 = gr.tile0 + first;
    if (e < 3) {
      const double* src = a.tile_red + 4 * static_cast<size_t>(t0) + e;
#pragma unroll 8
      for (int t = 0; t < n; ++t) acc += src[4 * t];
    } else {
      const float* src = a.tile_ab + a.tiles[t0].ab_off + (e - 3);   // a group's tiles follow one another
      float hi = 0.f, lo = 0.f;
#pragma unroll 8
      for (int t = 0; t < n; ++t) two_sum(hi, lo, src[static_cast<size_t>(t) * 2 * gr.npos]);
      acc = two_float(hi, lo);
    }
  }
  s_q[sub][el] = acc;
  __syncthreads();
  if (sub == 0 && e < E)
    g.part2[static_cast<size_t>(g.split_off[gi] + s) * g.max_e + e] = (s_q[0][el] + s_q[1][el]) + (s_q[2][el] + s_q[3][el]);
  __threadfence();
  __syncthreads();
  const int nce = (g.max_e + kRedE - 1) / kRedE;
  if (threadIdx.x == 0) {
    const int prev = atomicAdd(&g.counters[gi * nce + ce], 1);
    s_last = (prev == nsplit - 1);
  }
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  acc = 0.0;
  if (e < E) {
    const double* src = g.part2 + static_cast<size_t>(g.split_off[gi]) * g.max_e + e;
#pragma unroll 8
    for (int k = sub; k < nsplit; k += 4) acc += __ldcg(&src[static_cast<size_t>(k) * g.max_e]);
  }
  s_q[sub][el] = acc;
  __syncthreads();
  if (sub == 0 && e < E) {
    const double tot = (s_q[0][el] + s_q[1][el]) + (s_q[2][el] + s_q[3][el]);
    if (e == 0) {
      if (what & 1) g.gloss[gi] = tot;
    } else if (e == 1) {
      g.gred[gr.gp_off] = tot;
    } else if (e == 2) {
      if (what & 1) g.gprior[gi] = tot;
    }
    else {   // the partials run over positions, the gradients over the caller's measurements
      const bool beta = e >= 3 + gr.npos;
      const int n = g.meas_of[gr.pos_off + e - 3 - (beta ? gr.npos : 0)];
      if (n >= 0) g.gred[gr.gp_off + 4 + (beta ? gr.N4 : 0) + n] = tot;
    }
  }
  if (threadIdx.x == 0) g.counters[gi * nce + ce] = 0;
}

// dJ/db_lr[c] = sum_x w_c(x) dJ/dU(x): the adjoint of the trilinear upsampling. Its weights
// factor per axis, w_c(x, y, z) = w_cx(x) w_cy(y) w_cz(z), so the sum is taken in a fixed order
// over z (per (x, y) line), then over the corner's (x, y) support; each grid voxel is read once.
// Axis weights as in tri_weights: u = clamp((i + .5) 8 / n - .5, 0, 7), i0 = min(floor u, 6),
// corner i0 takes 1 - (u - i0) and corner i0 + 1 takes u - i0.
__device__ __forceinline__ void axis_weight(int i, int n, int& i0, float& w) {
  float u = (i + 0.5f) * (8.f / n) - 0.5f;
  u = fminf(fmaxf(u, 0.f), 7.f);
  i0 = min(static_cast<int>(floorf(u)), 6);
  w = u - i0;
}

// The voxels whose weight for corner c of an n-voxel axis can be nonzero (with a margin of
// one): [lo, hi].
__device__ __forceinline__ void axis_support(int c, int n, int& lo, int& hi) {
  const float sc = n / 8.f;
  lo = (c == 0) ? 0 : max(0, static_cast<int>(floorf((c - 0.5f) * sc - 0.5f)) - 1);
  hi = (c == kGrid - 1) ? n - 1 : min(n - 1, static_cast<int>(ceilf((c + 1.5f) * sc - 0.5f)) + 1);
}
__device__ __forceinline__ float axis_corner_weight(int i, int n, int c) {
  int i0;
  float w;
  axis_weight(i, n, i0, w);
  return (c == i0) ? 1.f - w : ((c == i0 + 1) ? w : 0.f);
}

// Pass 1: G1[x][y][cz] = sum_z w_cz(z) dJ/dU(x, y, z); one warp per (x, y) line, its lanes
// strided over z, then a fixed-order butterfly over the lanes (FP32: at most 1023 terms).
__device__ __forceinline__ void bias_grad_z(const IterArgs& a, const GroupArgs& g, int gi, int line) {
  const GroupDev gr = a.groups[gi];
  const int lane = threadIdx.x & 31;
  if (!gr.calib || line >= gr.nx * gr.ny) return;   // warp-uniform
  double* G1 = g.bscratch + g.bs_off[gi];
  float acc[kGrid];
#pragma unroll
  for (int c = 0; c < kGrid; ++c) acc[c] = 0.f;
  const int32_t* sog = g.slot_of_grid + gr.grid_off + static_cast<int64_t>(line) * gr.nz;
  for (int z = lane; z < gr.nz; z += 32) {
    const int slot = sog[z];
    if (slot < 0) continue;
    int k0;
    float wz;
    axis_weight(z, gr.nz, k0, wz);
    const float u = a.gU[slot];
#pragma unroll
    for (int c = 0; c < kGrid - 1; ++c)
      if (c == k0) {
        acc[c] = fmaf(1.f - wz, u, acc[c]);
        acc[c + 1] = fmaf(wz, u, acc[c + 1]);
      }
  }
#pragma unroll
  for (int c = 0; c < kGrid; ++c) {
    const float v = warp_sum_range<1, 16>(acc[c]);
    if (lane == 0) G1[static_cast<int64_t>(line) * kGrid + c] = v;
  }
}

// The tile sums and, in the first `nbz` blocks of a group, pass 1 of the bias-field adjoint (eight
// lines per block): neither reads what the other writes, so they share a launch.
__global__ void __launch_bounds__(256) k_group_sums(const IterArgs a, const GroupArgs g, int what, int nbz) {
  grid_dep_wait();
  grid_dep_launch();
  const int b = blockIdx.x, gi = blockIdx.y;
  if (b < nbz) {
    bias_grad_z(a, g, gi, b * 8 + (threadIdx.x >> 5));
  } else {
    const int nce = (g.max_e + kRedE - 1) / kRedE;
    group_reduce_block(a, g, gi, (b - nbz) / nce, (b - nbz) % nce, what);
  }
}

// Pass 2: dJ/db_lr[cx][cy][cz] = sum_xy w_cx(x) w_cy(y) G1[x][y][cz], a warp per corner, its lanes strided
// over the corner's (x, y) support, then a butterfly: 512 warps share the FP64 work (a thread per
// corner over x after one over y had it on a few SMs: 8.2 + 8.3 us for 64^3, 8.9 us now).
__global__ void __launch_bounds__(256) k_bias_grad_xy(const IterArgs a, const GroupArgs g) {
  grid_dep_wait();
  grid_dep_launch();
  const int gi = blockIdx.y;
  const GroupDev gr = a.groups[gi];
  if (!gr.calib) return;
  const int c = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  const int cx = c / (kGrid * kGrid), cy = (c / kGrid) % kGrid, cz = c % kGrid;
  const double* G1 = g.bscratch + g.bs_off[gi] + cz;
  int xlo, xhi, ylo, yhi;
  axis_support(cx, gr.nx, xlo, xhi);
  axis_support(cy, gr.ny, ylo, yhi);
  const int ny = yhi - ylo + 1, n = (xhi - xlo + 1) * ny;
  double acc = 0.0;
#pragma unroll 4
  for (int e = lane; e < n; e += 32) {
    const int x = xlo + e / ny, y = ylo + e % ny;
    const float wx = axis_corner_weight(x, gr.nx, cx), wy = axis_corner_weight(y, gr.ny, cy);
    const double v = G1[(static_cast<int64_t>(x) * gr.ny + y) * kGrid];
    if (wx != 0.f && wy != 0.f) acc += (static_cast<double>(wx) * static_cast<double>(wy)) * v;
  }
  acc = warp_sum_d(acc);
  if (lane == 0) g.gred[gr.gp_off + 4 + 2 * gr.N4 + c] = acc;
}

// Group finalisation (one block): objective with the calibration regularisers of Sec. 2.4
// (L2 on alpha, beta, b_lr and TV on B; the paper gives no weights: 1e-3 each by default),
// loss history, Adam on sigma_log / alpha / beta / b_lr, table refresh, step counter.
// mode bit 0: loss; bit 1: Adam + step; bit 2: export gradients. One block per group on the critical
// path of a calibrated iteration, bound by one SM's FP64 rate: the weights are divided once and each
// parameter costs five FP64 operations (with a division per parameter and 256 threads 25 us for the
// 1,236 parameters at N = 360, 15 us now).
constexpr int kGroupThreads = 512;
__global__ void __launch_bounds__(kGroupThreads) k_group_adam(const IterArgs a, const GroupArgs g, int mode) {
  __shared__ double s[kGroupThreads / 32], s_w[3];
  __shared__ int s_bad, s_last;
  grid_dep_wait();
  grid_dep_launch();
  const int tid = threadIdx.x;
  if (tid == 0) s_bad = 0;
  const int step = *a.step;
  const float stepsz = a.adamc[0], isbc2 = a.adamc[1];
  // one block per group; the last block to finish advances the step counter
  for (int gi = blockIdx.x; gi < g.G; gi += gridDim.x) {
    const GroupDev gr = a.groups[gi];
    const int base = gr.gp_off;
    const int N = gr.N, N4 = gr.N4;
    // regulariser weights of a squared alpha, beta and b_lr, and their values
    if (tid < 3) s_w[tid] = static_cast<double>(tid == 0 ? g.w_alpha : tid == 1 ? g.w_beta : g.w_blr) / (tid < 2 ? N : kNGrid);
    double ra = 0.0, rb = 0.0, rl = 0.0;
    if (gr.calib) {
      const float* p = g.gparams + base + 4;
      for (int i = tid; i < N; i += kGroupThreads) {
        const double xa = p[i], xb = p[N4 + i];
        ra = fma(xa, xa, ra);
        rb = fma(xb, xb, rb);
      }
      for (int i = tid; i < kNGrid; i += kGroupThreads) {
        const double x = p[2 * N4 + i];
        rl = fma(x, x, rl);
      }
    }
    __syncthreads();
    const double wa = s_w[0], wb = s_w[1], wl = s_w[2];
    if (mode & 1) {
      double reg = gr.calib ? warp_sum_d(fma(wa, ra, fma(wb, rb, wl * rl))) : 0.0;
      if ((tid & 31) == 0) s[tid >> 5] = reg;
      __syncthreads();
      if (tid == 0) {
        for (int w = 1; gr.calib && w < kGroupThreads / 32; ++w) reg += s[w];
        const double J = g.gloss[gi] + g.gprior[gi] + reg;
        g.gloss[gi] = J;
        if (!isfinite(J)) s_bad = 1;
        if (mode & 2) g.hist[static_cast<size_t>(step % g.hist_len) * g.G + gi] = J;
      }
    }
    __syncthreads();
    // gradients and Adam over the group's packed parameters
    const int total = 4 + 2 * N4 + kNGrid;
    for (int i = tid; i < total; i += blockDim.x) {
      float grad;
      bool train;
      const float x = g.gparams[base + i];
      if (i == 0) {
        train = (g.loss_mode == kLossNLL);
        grad = train ? static_cast<float>(g.gred[base]) : 0.f;
      } else if (i < 4) {
        train = false;
        grad = 0.f;
      } else if (i < 4 + N4) {
        train = gr.calib && (i - 4 < N);
        grad = train ? static_cast<float>(fma(2.0 * wa, static_cast<double>(x), g.gred[base + i])) : 0.f;
      } else if (i < 4 + 2 * N4) {
        train = gr.calib && (i - 4 - N4 < N);
        grad = train ? static_cast<float>(fma(2.0 * wb, static_cast<double>(x), g.gred[base + i])) : 0.f;
      } else {
        train = gr.calib;
        grad = train ? static_cast<float>(fma(2.0 * wl, static_cast<double>(x), g.gred[base + i])) : 0.f;
      }
      if (g.gexport && (mode & 4)) g.gexport[base + i] = grad;
      if ((mode & 2) && train) {
        float mq, vq, xn = x;
        if (a.optimizer == 0) {
          mq = fmaf(a.beta1, g.gm[base + i], (1.f - a.beta1) * grad);
          vq = fmaf(a.beta2, g.gv[base + i], (1.f - a.beta2) * grad * grad);
          xn = x - stepsz * mq / fmaf(sqrtf(vq), isbc2, a.eps);
        } else {
          mq = g.gm[base + i];
          vq = g.gv[base + i];
          rprop_update(xn, mq, vq, grad, a.lr, a.eta_minus, a.eta_plus, a.step_min, a.step_max);
        }
        g.gm[base + i] = mq;
        g.gv[base + i] = vq;
        g.gparams[base + i] = xn;
        if (i >= 4 && i < 4 + 2 * N4) {
          const int n = (i < 4 + N4) ? i - 4 : i - 4 - N4;
          MeasRow* row = g.table + gr.table_off + n;
          float* pr = reinterpret_cast<float*>(g.table2 + gr.table2_off + n / 2) + (n & 1);
          const int pos = g.pos_of[gr.table_off + n];
          float* pc = g.ctab + gr.ctab_off + pos / 2 * 4 + (pos & 1);
          if (i < 4 + N4) {
            row->A = expf(xn);
            pr[2 * kPairFieldA] = row->A;
            if (g.ctab) pc[0] = row->A;
          } else {
            row->beta = xn;
            pr[2 * kPairFieldBeta] = xn;
            if (g.ctab) pc[2] = xn;
          }
        }
      }
    }
    __syncthreads();
  }
  if (tid == 0 && s_bad) atomicOr(a.status, kStNonfinite);
  if (!(mode & 2)) return;
  __syncthreads();
  if (tid == 0) {
    __threadfence();
    s_last = (atomicAdd(g.gdone, 1) == static_cast<int>(gridDim.x) - 1);
  }
  __syncthreads();
  if (!s_last || tid >= 2) return;
  // constants of the next iteration, t = step + 2 (bias corrections in double)
  const_cast<float*>(a.adamc)[tid] = adam_constant(tid, a.lr, a.beta1, a.beta2, static_cast<int64_t>(step) + 2);
  if (tid == 0) {
    __threadfence();
    *g.gdone = 0;
    *const_cast<int32_t*>(a.step) = step + 1;
  }
}

// Adam constants for the coming iteration t = step + 1 (after init or a checkpoint load).
__global__ void k_adam_constants(const IterArgs a) {
  if (threadIdx.x >= 2) return;
  const_cast<float*>(a.adamc)[threadIdx.x] =
      adam_constant(threadIdx.x, a.lr, a.beta1, a.beta2, static_cast<int64_t>(*a.step) + 1);
}

// Table refresh after the caller sets group parameters (exp(alpha), beta).
__global__ void k_table_refresh(const GroupArgs g, const IterArgs a) {
  const GroupDev gr = a.groups[blockIdx.x];
  for (int n = threadIdx.x; n < gr.N; n += blockDim.x) {
    MeasRow* row = g.table + gr.table_off + n;
    row->A = gr.calib ? expf(g.gparams[gr.gp_off + 4 + n]) : 1.f;
    row->beta = gr.calib ? g.gparams[gr.gp_off + 4 + gr.N4 + n] : 0.f;
    float* pr = reinterpret_cast<float*>(g.table2 + gr.table2_off + n / 2) + (n & 1);
    pr[2 * kPairFieldA] = row->A;
    pr[2 * kPairFieldBeta] = row->beta;
    if (g.ctab) {
      const int pos = g.pos_of[gr.table_off + n];
      float* pc = g.ctab + gr.ctab_off + pos / 2 * 4 + (pos & 1);
      pc[0] = row->A;
      pc[2] = row->beta;
    }
  }
}

// ---------------------------------------------------------------------------
// Launchers.
// ---------------------------------------------------------------------------
static inline int nblk(int64_t n, int b) { return static_cast<int>((n + b - 1) / b); }

// The bounded-wait error path, exercised without a fault: one thread waits, with the bounded
// wait the fused kernel uses for its bulk copies, on the first phase of a fresh mbarrier that
// nothing completes (no copy is issued and nothing arrives). When the wait gives up after
// `polls` polls, the timeout bit of the status word is set and the kernel returns.
__global__ void k_wait_probe(int32_t* status, int polls) {
  __shared__ __align__(8) uint64_t bar;
  if (threadIdx.x != 0) return;
  mbar_init(&bar, 1);
  fence_mbar_init();
  if (!mbar_wait(&bar, 0u, polls)) atomicOr(status, kStTimeout);
}

cudaError_t launch_wait_probe(int32_t* status, int polls, cudaStream_t st) {
  k_wait_probe<<<1, 32, 0, st>>>(status, polls);
  return cudaGetLastError();
}

cudaError_t launch_group_sums(const IterArgs& a, const GroupArgs& g, int what, bool bias, cudaStream_t st) {
  const int nbz = bias ? nblk(static_cast<int64_t>(g.max_nx) * g.max_ny, 8) : 0;
  const int nred = (g.max_e + kRedE - 1) / kRedE * g.max_split;
  cudaError_t e = launch_dep(k_group_sums, dim3(nbz + nred, g.G), dim3(256), 0, st, a.pdl != 0, a, g, what, nbz);
  if (e == cudaSuccess && bias)
    e = launch_dep(k_bias_grad_xy, dim3(kNGrid / 8, g.G), dim3(256), 0, st, a.pdl != 0, a, g);
  return e;
}
cudaError_t launch_group_adam(const IterArgs& a, const GroupArgs& g, int mode, cudaStream_t st) {
  return launch_dep(k_group_adam, dim3(g.G), dim3(kGroupThreads), 0, st, a.pdl != 0, a, g, mode);
}
cudaError_t launch_loss(const IterArgs& a, const PlainArgs& p, int loss, cudaStream_t st) {
  const int nt = p.tile_end - p.tile_begin;
  if (nt <= 0) return cudaSuccess;
  if (loss == kLossMSE) k_loss<kLossMSE><<<nt, 256, 0, st>>>(a, p);
  else k_loss<kLossNLL><<<nt, 256, 0, st>>>(a, p);
  return cudaGetLastError();
}
cudaError_t launch_adam_voxel(const IterArgs& a, const PlainArgs& p, cudaStream_t st) {
  const int64_t n = static_cast<int64_t>(p.tile_end - p.tile_begin) * a.TV;
  if (n <= 0) return cudaSuccess;
  k_adam_voxel<<<nblk(n, 256), 256, 0, st>>>(a, p);
  return cudaGetLastError();
}
int b0_stat_blocks(int64_t V) { return nblk(V, kB0Vox); }
cudaError_t launch_b0_stats(const float* sig, const int64_t* rows, int64_t V, int N, const int32_t* b0n, int nb0,
                            float* b0mean, double* part, int* bad, cudaStream_t st) {
  k_b0_stats<<<b0_stat_blocks(V), 256, 0, st>>>(sig, rows, V, N, b0n, nb0, b0mean, part, bad);
  return cudaGetLastError();
}
cudaError_t launch_sigma_init(const double* part, int nblocks, int64_t V, int nb0, float fb, float* out,
                              cudaStream_t st) {
  k_sigma_init<<<1, 256, 0, st>>>(part, nblocks, V, nb0, fb, out);
  return cudaGetLastError();
}
cudaError_t launch_pack(const IterArgs& a, const float* sig, const int64_t* rows, const float* b0mean,
                        const int32_t* vox_of_slot, const int32_t* order, int64_t vox0, int tile_begin, int tile_end,
                        int N, int npos, float* ypack, int* bad, cudaStream_t st) {
  if (tile_end <= tile_begin) return cudaSuccess;
  if (a.TV % a.VW != 0) return cudaErrorInvalidValue;
  const dim3 nb(tile_end - tile_begin, a.TV / a.VW);
  switch (a.VW) {
    case 32: k_pack<32><<<nb, kPackThreads, 0, st>>>(a, sig, rows, b0mean, vox_of_slot, order, vox0, tile_begin, N, npos, ypack, bad); break;
    case 8: k_pack<8><<<nb, kPackThreads, 0, st>>>(a, sig, rows, b0mean, vox_of_slot, order, vox0, tile_begin, N, npos, ypack, bad); break;
    case 2: k_pack<2><<<nb, kPackThreads, 0, st>>>(a, sig, rows, b0mean, vox_of_slot, order, vox0, tile_begin, N, npos, ypack, bad); break;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}
cudaError_t launch_plan(const PlanArgs& p, const GroupDev* groups, int npatch, cudaStream_t st) {
  if (npatch <= 0) return cudaSuccess;
  k_plan<<<npatch, kPlanThreads, 0, st>>>(p, groups);
  return cudaGetLastError();
}
cudaError_t launch_grid_of_vox(const uint8_t* mask, const int32_t* line, int nx, int ny, int nz, int32_t* grid_of_vox,
                               cudaStream_t st) {
  k_grid_of_vox<<<nblk(static_cast<int64_t>(nx) * ny, 128), 128, 0, st>>>(mask, line, nx * ny, nz, grid_of_vox);
  return cudaGetLastError();
}
cudaError_t launch_slot_data(const Tile* tiles, const GroupDev* groups, int G, const GroupDev* host_groups,
                             const int32_t* slot_of_grid, int Vp, int TV, int nnb, uint32_t* vflag, int32_t* nbr,
                             cudaStream_t st) {
  cudaError_t e = cudaMemsetAsync(vflag, 0, sizeof(uint32_t) * Vp, st);
  if (e == cudaSuccess) e = cudaMemsetAsync(nbr, 0xff, sizeof(int32_t) * static_cast<size_t>(nnb) * Vp, st);
  if (e != cudaSuccess) return e;
  for (int g = 0; g < G; ++g) {
    const int64_t ng = static_cast<int64_t>(host_groups[g].nx) * host_groups[g].ny * host_groups[g].nz;
    k_slot_data<<<nblk(ng, 256), 256, 0, st>>>(tiles, groups, g, slot_of_grid, Vp, TV, nnb, vflag, nbr);
  }
  return cudaGetLastError();
}
cudaError_t launch_gather_rows(const float* src, const int64_t* rows, int64_t n, int len, float* dst,
                               cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  k_gather_rows<<<nblk(n, 8), 256, 0, st>>>(src, rows, n, len, dst);
  return cudaGetLastError();
}
cudaError_t launch_table(const float* bvals, const float* bvecs, int N, MeasRow* rows, cudaStream_t st) {
  k_table<<<nblk(N, 128), 128, 0, st>>>(bvals, bvecs, N, rows);
  return cudaGetLastError();
}
cudaError_t launch_pair_table(const MeasRow* rows, int N, MeasPair* out, cudaStream_t st) {
  const int NP = (N + 3) & ~3;
  k_pair_table<<<nblk(NP / 2, 128), 128, 0, st>>>(rows, N, NP, out);
  return cudaGetLastError();
}
cudaError_t launch_scatter_params(const float* in, const int64_t* rows, const int32_t* sov, int64_t V, int Q, int Vpad,
                                  float* th, cudaStream_t st) {
  if (V == 0) return cudaSuccess;
  k_scatter_params<<<nblk(V, kParVox), kParVox, sizeof(float) * kParVox * Q, st>>>(in, rows, sov, V, Q, Vpad, th);
  return cudaGetLastError();
}
cudaError_t launch_gather_params(const float* th, const int32_t* sov, int64_t V, int Q, int Vpad, float* out,
                                 cudaStream_t st) {
  if (V == 0) return cudaSuccess;
  k_gather_params<<<nblk(V, kParVox), kParVox, sizeof(float) * kParVox * Q, st>>>(th, sov, V, Q, Vpad, out);
  return cudaGetLastError();
}
cudaError_t launch_default_init(const int32_t* sov, const uint32_t* vcoord, int ny, int nz, int64_t V, int K,
                                int Vpad, uint64_t seed, float* th, cudaStream_t st) {
  if (V == 0) return cudaSuccess;
  k_default_init<<<nblk(V, 128), 128, 0, st>>>(sov, vcoord, ny, nz, V, K, Vpad, seed, th);
  return cudaGetLastError();
}
cudaError_t launch_adam_constants(const IterArgs& a, cudaStream_t st) {
  k_adam_constants<<<1, 32, 0, st>>>(a);
  return cudaGetLastError();
}
cudaError_t launch_table_refresh(const GroupArgs& g, const IterArgs& a, cudaStream_t st) {
  k_table_refresh<<<g.G, 128, 0, st>>>(g, a);
  return cudaGetLastError();
}

}  // namespace prism
