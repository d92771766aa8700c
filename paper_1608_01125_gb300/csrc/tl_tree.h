// tl_tree.h -- arguments and launchers of the exact path (tl_tree.cu), shared with
// the host runtime.
#pragma once
#include "tl_common.cuh"
#include "tl_frame.cuh"

namespace tl {

// k_order: one beam
struct OrderArgs {
  TLBeam b;
  double ct;
  float L;
  const TLFrame *frames;    // per instance (one for a single problem)
  TLGrid grid;              // a single problem's
  const TLGrid *grids;      // per instance (batches)
  const uint32_t *inst_of;  // instance of each photon (batches, else NULL)
  int inst_shift;           // bit position of the instance in the key
  int passes;               // 8-bit digits of the key
  float4 *pos_u;
  const float4 *dir_u;
  uint32_t *key;
  uint32_t *hist;           // digit counts of the passes, zero before
};

// k_boxes: the tree's beam
struct BoxArgs {
  const float4 *pos, *dir;
  const TLInst *inst;
  const uint32_t *tile_inst;  // instance of each tile (batches, else NULL)
  const TLFrame *frames;
  float Llo, Lhi, half;
  float4 *box;
  const unsigned *build_status;
};

// k_collide
struct ColArgs {
  const float4 *qpos, *qdir, *tpos, *tdir;  // sorted photons: query beam, tree's beam
  const float4 *box;                        // the tree
  const TLInst *qinst, *tinst;
  const uint32_t *tile_inst;  // instance of each query tile (batches, else NULL)
  const TLFrame *frames;
  float Llo, Lhi, half;
  TLNarrowConst nk;
  TLCounters *ctr;
  uint2 *cand;  // candidate pairs (positions in beam A's and beam B's sorted photons)
  unsigned long long cand_cap;
  long long items;  // groups of 32 query photons times slices
  int group0;       // first group of this part
  int slices;       // parts of the tree per group
  int fp64, swap;   // swap: the tree is beam A's
};

size_t moment_doubles();
cudaError_t launch_beam_moments(const TLBeam &b, const TLFrame &f, double *out, cudaStream_t s);
cudaError_t launch_inst_bounds(const TLBeam &b, const uint32_t *inst_of, const TLFrame *frames,
                               int n_inst, long long *tmp, double *out, cudaStream_t s);
cudaError_t launch_inst_frames(const double *ba, const double *bb, int n_inst, TLFrame *out,
                               cudaStream_t s);
cudaError_t launch_inst_grid(const double *ba, const double *bb, const TLFrame *frames, int n_inst,
                             double T, double L, double half, int bits, TLGrid *ga, TLGrid *gb,
                             cudaStream_t s);
cudaError_t launch_order(const OrderArgs &a, cudaStream_t s);
cudaError_t launch_boxes(const BoxArgs &a, int tiles, int n_inst, int max_top, cudaStream_t s);
cudaError_t launch_step_init(TLCounters *ctr, const unsigned *build_status,
                             const unsigned *run_status, cudaStream_t s);
cudaError_t launch_collide(const ColArgs &a, cudaStream_t s);
cudaError_t launch_part_next(TLCounters *ctr, cudaStream_t s);
cudaError_t launch_decide(const TravArgs &a, int blocks, cudaStream_t s);

}  // namespace tl
