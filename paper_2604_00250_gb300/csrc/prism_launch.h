// Host-side launch interface between the C-ABI implementation and the kernels.
#pragma once

#include <cuda_runtime.h>

#include "prism_device.cuh"

namespace prism {

// Launches fn on st, as a programmatic dependent of the stream's previous kernel when `pdl`
// (the kernel then waits for it on the device before reading what it wrote).
template <typename... P, typename... A>
cudaError_t launch_dep(void (*fn)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, bool pdl, A... args) {
  if (!pdl) {
    fn<<<grid, block, smem, st>>>(args...);
    return cudaGetLastError();
  }
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, fn, args...);
}

// Stitching of a slab fit (k_stitch): the whole volume's voxels by grid position and its slices.
struct StitchArgs {
  const int32_t* grid_of_vox;
  const SliceDev* slices;
  const int32_t* slot_of_grid;
  int64_t n;
  int32_t ny, nz;
  float *s0, *fracs, *fin, *dirs;
};

// Per-K launchers of the templated kernels (one translation unit per K).
struct KernelSet {
  // shell = 1..3: the shell loop (see k_iter_fused); grad = 1: the gradient form (no update)
  cudaError_t (*fused)(const IterArgs& a, int loss, int cal, int tpv, int shell, int grad, int grid, int nt,
                       size_t smem, cudaStream_t st);
  cudaError_t (*fused_occupancy)(int loss, int cal, int tpv, int shell, int nt, size_t smem, int* blocks);
  // iterations of a fit without neighbour priors and calibration, several lanes per voxel
  cudaError_t (*local)(const IterArgs& a, int loss, int tpv, int grid, size_t smem, cudaStream_t st);
  cudaError_t (*local_occupancy)(int loss, int tpv, size_t smem, int* blocks);
  cudaError_t (*transform)(const IterArgs& a, int tb, int te, cudaStream_t st);
  cudaError_t (*synth)(const IterArgs& a, const PlainArgs& p, int cal, int tpv, int nt, cudaStream_t st);
  cudaError_t (*yhat)(const IterArgs& a, int cal, const int32_t* vox_of_slot, const int32_t* order, float* out,
                      cudaStream_t st);
  cudaError_t (*adjoint)(const IterArgs& a, const PlainArgs& p, int cal, int tpv, int nt, size_t smem,
                         cudaStream_t st);
  cudaError_t (*prior_prep)(const IterArgs& a, int tb, int te, cudaStream_t st);
  cudaError_t (*prior_grad)(const IterArgs& a, int tb, int te, cudaStream_t st);
  cudaError_t (*prior)(const IterArgs& a, const PlainArgs& p, cudaStream_t st);
  cudaError_t (*fibers)(const IterArgs& a, const int32_t* slot_of_vox, int64_t V, float rel, float* dirs,
                        float* fracs, uint8_t* peaks, cudaStream_t st);
  cudaError_t (*stitch)(const IterArgs& a, const StitchArgs& s, cudaStream_t st);
};

const KernelSet& kernels_for_k(int K);

// Group-level kernels (prism_aux.cu).
constexpr int kRedE = 64;   // entries of the group sums per block
struct GroupArgs {
  int32_t G, max_split, split_tiles, max_e;
  const int32_t* split_off;   // [G] first part2 row of the group
  double* part2;              // [sum splits][max_e]
  int32_t* counters;          // [G][ceil(max_e / kRedE)]
  double* gred;               // packed like gparams (double); loss kept separately
  double* gloss;              // [G] data term, then the full objective after finalisation
  double* gprior;             // [G] prior total
  float* gm;                  // group Adam moments (packed like gparams)
  float* gv;
  float* gparams;
  MeasRow* table;
  MeasPair* table2;   // the paired copy (its e^alpha_n and beta_n follow the rows)
  float* ctab;                // the same by position (GroupDev::ctab_off), or null
  const int32_t* pos_of;      // measurement -> position, rows as in `table`
  const int32_t* meas_of;     // position -> measurement or -1 (GroupDev::pos_off)
  const int32_t* slot_of_grid;
  double* hist;               // [H][G] loss history
  int32_t hist_len;
  float* gexport;             // packed group gradients for the caller (or null)
  int32_t loss_mode;          // kLossMSE / kLossNLL
  float w_alpha, w_beta, w_blr;
  double* bscratch;           // bias-gradient partial contractions (see bias_grad_z)
  const int64_t* bs_off;      // [G] offset of a group's [nx][ny][8] sums over z
  int32_t max_nx, max_ny;     // largest grid extents over the groups
  int32_t* gdone;             // blocks of k_group_adam that finished (last one resets it)
};

// Sums over the tiles (`what` bit 0: objective, bit 1: group gradients) and, with `bias`, the
// bias-field adjoint.
cudaError_t launch_group_sums(const IterArgs& a, const GroupArgs& g, int what, bool bias, cudaStream_t st);
cudaError_t launch_group_adam(const IterArgs& a, const GroupArgs& g, int mode, cudaStream_t st);
cudaError_t launch_loss(const IterArgs& a, const PlainArgs& p, int loss, cudaStream_t st);
cudaError_t launch_adam_voxel(const IterArgs& a, const PlainArgs& p, cudaStream_t st);

// Preprocessing and layout kernels.
int b0_stat_blocks(int64_t V);   // partials that launch_b0_stats writes
cudaError_t launch_b0_stats(const float* sig, const int64_t* rows, int64_t V, int N, const int32_t* b0n, int nb0,
                            float* b0mean, double* part, int* bad, cudaStream_t st);
cudaError_t launch_sigma_init(const double* part, int nblocks, int64_t V, int nb0, float sigma_fallback,
                              float* sigma_log_out, cudaStream_t st);
cudaError_t launch_pack(const IterArgs& a, const float* sig, const int64_t* rows, const float* b0mean,
                        const int32_t* vox_of_slot, const int32_t* order, int64_t vox0, int tile_begin, int tile_end,
                        int N, int npos, float* ypack, int* bad, cudaStream_t st);
// Slots of one volume's voxels (k_plan). `mask`, `line` (masked voxels before each (x, y) line) and
// `ptile` (first tile of each patch, -1 for none) are the volume's; `stride` and `z0` as in a slab of a
// larger mask, whose lines `wline` then counts and whose rows go to `rows`.
struct PlanArgs {
  const uint8_t* mask;
  int32_t stride, z0;
  const int32_t *line, *wline, *ptile;
  int32_t g, P, TV;
  int32_t *slot_of_grid, *slot_of_vox, *vox_of_slot;
  uint32_t* vcoord;
  int64_t* rows;
};
cudaError_t launch_plan(const PlanArgs& p, const GroupDev* groups, int npatch, cudaStream_t st);
cudaError_t launch_grid_of_vox(const uint8_t* mask, const int32_t* line, int nx, int ny, int nz, int32_t* grid_of_vox,
                               cudaStream_t st);
cudaError_t launch_slot_data(const Tile* tiles, const GroupDev* groups, int G, const GroupDev* host_groups,
                             const int32_t* slot_of_grid, int Vp, int TV, int nnb, uint32_t* vflag, int32_t* nbr,
                             cudaStream_t st);
cudaError_t launch_gather_rows(const float* src, const int64_t* rows, int64_t n, int len, float* dst,
                               cudaStream_t st);
cudaError_t launch_table(const float* bvals, const float* bvecs, int N, MeasRow* rows, cudaStream_t st);
cudaError_t launch_pair_table(const MeasRow* rows, int N, MeasPair* out, cudaStream_t st);
cudaError_t launch_scatter_params(const float* in, const int64_t* rows, const int32_t* slot_of_vox, int64_t V, int Q,
                                  int Vpad, float* theta, cudaStream_t st);
cudaError_t launch_gather_params(const float* theta, const int32_t* slot_of_vox, int64_t V, int Q, int Vpad,
                                 float* out, cudaStream_t st);
cudaError_t launch_default_init(const int32_t* slot_of_vox, const uint32_t* vcoord, int ny, int nz, int64_t V, int K,
                                int Vpad, uint64_t seed, float* theta, cudaStream_t st);
cudaError_t launch_table_refresh(const GroupArgs& g, const IterArgs& a, cudaStream_t st);
cudaError_t launch_adam_constants(const IterArgs& a, cudaStream_t st);
cudaError_t launch_wait_probe(int32_t* status, int polls, cudaStream_t st);

}  // namespace prism
