// tl_tree.h -- arguments and launchers of the exact path (tl_tree.cu), shared with
// the host runtime.
#pragma once
#include "tl_common.cuh"
#include "tl_frame.cuh"

namespace tl {

// k_order: one beam
struct OrderArgs {
  int64_t n;
  const float4 *stat;       // p0 and energy, direction and index of every photon (FP32)
  float ct, L, half;
  const TLFrame *frames;    // per instance (one for a single problem)
  TLGrid grid;              // a single problem's
  const TLGrid *grids;      // per instance (batches)
  const uint32_t *inst_of;  // instance of each photon (batches, else NULL)
  const TLInst *inst;
  uint2 *cell;              // out: cell and rank in it (TL_NONE: meets nothing)
  uint32_t *count;          // photons per cell, zero before
  uint32_t *scan_st;        // the scan's words, cleared
  int scan_tiles;
};

// k_place: one beam's photons to their places
struct PlaceArgs {
  TLBeam b;
  double ct;
  int64_t n_pad;
  const float4 *stat;
  const uint2 *cell;
  const uint32_t *start;    // first sorted position of each cell
  const uint32_t *inst_of;  // batches
  const TLInst *inst;
  float4 *rec;
};

// k_boxes: the tree's beam
struct BoxArgs {
  const float4 *rec;
  const TLInst *inst;
  const uint32_t *start;
  const uint32_t *group_inst;  // instance of each group (batches, else NULL)
  const TLFrame *frames;
  float Llo, Lhi, half;
  int beam, needles;
  float4 *box;
  const unsigned *build_status;
};

// k_collide
struct ColArgs {
  const float4 *q, *t;  // sorted photons: query beam, tree's beam
  const float4 *box;                        // the tree
  const TLInst *qinst, *tinst;
  const uint32_t *qstart, *tstart;  // running sums of their cells
  const uint32_t *group_inst;  // instance of each query group (batches, else NULL)
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
  int needles;      // the tree's level 0 holds needles
};

int mean_doubles();  // per-block sums of launch_mean_dir
int64_t mean_count(int64_t n);  // photons it sums
cudaError_t launch_mean_dir(const TLBeam &b, double *part, cudaStream_t s);
size_t moment_doubles();
cudaError_t launch_beam_moments(const TLBeam &b, const TLFrame &f, double *out, cudaStream_t s);
cudaError_t launch_inst_bounds(const TLBeam &b, const uint32_t *inst_of, const TLFrame *frames,
                               int n_inst, long long *tmp, double *out, cudaStream_t s);
cudaError_t launch_inst_energy(const TLBeam &b, const TLInst *inst, int n_inst, double *out,
                               cudaStream_t s);
cudaError_t launch_inst_frames(const double *ba, const double *bb, const double *lea,
                               const double *leb, const TLPadTable &pads, double half, int n_inst,
                               TLFrame *out, cudaStream_t s);
cudaError_t launch_inst_grid(const double *ba, const double *bb, const TLFrame *frames,
                             const TLInst *ia, const TLInst *ib, int n_inst, double T, double L,
                             double half, TLGrid *ga, TLGrid *gb, cudaStream_t s);
cudaError_t launch_static(const TLBeam &b, float4 *stat, cudaStream_t s);
cudaError_t launch_order(const OrderArgs &a, cudaStream_t s);
int64_t scan_tiles(int64_t cells);
cudaError_t launch_cell_scan(uint32_t *count, uint32_t *start, int64_t cells, uint32_t *st,
                             long long spin, int debug_stall, unsigned *status, cudaStream_t s);
cudaError_t launch_place(const PlaceArgs &a, cudaStream_t s);
cudaError_t launch_boxes(const BoxArgs &a, int tiles, int n_inst, int max_top, cudaStream_t s);
cudaError_t launch_step_init(TLCounters *ctr, const unsigned *build_status,
                             const unsigned *run_status, cudaStream_t s);
cudaError_t launch_collide(const ColArgs &a, cudaStream_t s);
cudaError_t launch_part_next(TLCounters *ctr, cudaStream_t s);
cudaError_t launch_decide(const TravArgs &a, int blocks, cudaStream_t s);

}  // namespace tl
