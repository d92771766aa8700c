// tl_api.cu -- host runtime behind the C ABI declared in include/trilens.h:
// context and workspace, per-step build and collide sequencing on the
// caller's stream, device status checks and buffer regrowth.
#include <math.h>
#include <stdarg.h>
#include <stdio.h>
#include <stdlib.h>
#include <string.h>

#include <algorithm>
#include <string>
#include <vector>

#include "tl_ctx.h"
#include "trilens_debug.h"

namespace tl {
cudaError_t traverse_config(int fp64, int warps, int depth, int *blocks_per_sm);
cudaError_t launch_narrow(const TravArgs &a, int blocks, cudaStream_t s);
cudaError_t launch_traverse(const TravArgs &a, const uint2 *list, unsigned long long list_n,
                            int budget, int blocks, int warps, cudaStream_t s, int part,
                            int nparts);
cudaError_t launch_part_init(TLCounters *ctr, cudaStream_t s);
cudaError_t launch_band(const TravArgs &a, int blocks, cudaStream_t s);
cudaError_t launch_yield(const TravArgs &a, void *partials, int blocks, cudaStream_t s);
size_t partial_bytes();
cudaError_t launch_yield_inst(const TravArgs &a, const uint32_t *inst_of_a, double *yields,
                              int blocks, cudaStream_t s);
cudaError_t launch_pair_products(const TLBeam &a, const TLBeam &b, const uint32_t *hits,
                                 int64_t n_hits, unsigned long long seed, double *out,
                                 cudaStream_t s);
cudaError_t launch_step_finish(const TLCounters *ctr, unsigned *run_status, TLRunAcc *acc,
                               cudaStream_t s);
}  // namespace tl

enum {
  PH_PROP = 0, PH_SORT, PH_GATHER, PH_EMIT, PH_REFIT, PH_EXPAND, PH_TRAV, PH_BAND, PH_YIELD,
  PH_NARROW, PH_COUNT
};

// node pairs per traversal queue chunk and frontier item (tl_traverse.cu)
constexpr unsigned long long kQueueChunk = 32;
// the list of candidate (or leaf-bucket) pairs never grows past 2^30 pairs (8 GiB): a step that lists
// more is done in parts, each listing at most that
constexpr unsigned long long kLeafListMax = 1ull << 30;

// after a step overflowed the leaf-pair list (the largest part listed need
// pairs): a larger list, or more parts
static int leaves_for(trilens_ctx *c, unsigned long long need) {
  if (need + need / 4 + 1024 <= kLeafListMax) return grow(c, &c->leaves, &c->leaf_cap, need);
  drop_run(c);
  if (c->leaf_cap < kLeafListMax) {
    cudaFree(c->leaves);
    c->leaves = nullptr;
    c->leaf_cap = 0;
    CK(dalloc(&c->leaves, (size_t)kLeafListMax));
    c->leaf_cap = kLeafListMax;
  }
  const unsigned long long per = kLeafListMax / 2;  // room for uneven parts
  const unsigned long long more = (need + per - 1) / per;
  if ((unsigned long long)c->parts * more > 4096)
    return fail(c, TRILENS_ERR_STACK, "a step would need more than 4096 parts");
  c->parts = (int)(c->parts * more);
  return TRILENS_OK;
}

static void tmark(trilens_ctx *c, int ph, int k, int end) {
  if (!c->timing) return;
  cudaEventRecord(c->ev[ph][k][end], c->stream);
  if (end) c->ev_pending[ph][k] = true;
}

// warps of k_collide that keep every SM busy: fewer groups of 32 photons than this
// are each given several warps, on parts of the tree (2 x 2048 photons have 64 groups)
constexpr int kColWarpsPerSm = 24;

// the groups of 32 query photons of part p of the step, and the kernel's arguments
static tl::ColArgs col_args(trilens_ctx *c, int p) {
  const int q = 1 - c->tree, t = c->tree;
  tl::ColArgs a;
  memset(&a, 0, sizeof(a));
  a.q = c->w[q].rec;
  a.t = c->w[t].rec;
  a.box = c->box;
  a.qinst = c->insts[q];
  a.tinst = c->insts[t];
  a.qstart = c->w[q].start;
  a.tstart = c->w[t].start;
  a.group_inst = c->group_inst[q];
  a.frames = c->frames;
  a.Llo = c->L_lo;
  a.Lhi = c->L_hi;
  a.half = c->half;
  a.nk = c->nk;
  a.ctr = c->ctr;
  a.cand = c->leaves;
  a.cand_cap = c->leaf_cap;
  const long long groups = c->n_groups[q];
  const long long g0 = groups * p / c->parts, g1 = groups * (p + 1) / c->parts;
  a.group0 = (int)g0;
  a.slices = 1;
  if (g1 > g0)
    a.slices = (int)std::min<long long>(
        64, std::max<long long>(1, (long long)kColWarpsPerSm * c->n_sm / (g1 - g0)));
  a.items = c->n_groups[t] > 0 ? (g1 - g0) * a.slices : 0;
  a.fp64 = c->p.precision == TRILENS_FP64;
  a.swap = t == 0;
  a.needles = c->needles;
  return a;
}

// the collisions of a step up to its candidates' decisions, part by part
static int collide_parts(trilens_ctx *c, const tl::TravArgs &a) {
  for (int p = 0; p < c->parts; ++p) {
    if (p > 0) CK(tl::launch_part_next(c->ctr, c->stream));
    tmark(c, PH_TRAV, 0, 0);  // (of several parts the last is timed)
    CK(tl::launch_collide(col_args(c, p), c->stream));
    tmark(c, PH_TRAV, 0, 1);
    tmark(c, PH_NARROW, 0, 0);
    CK(tl::launch_decide(a, 8 * c->n_sm, c->stream));
    tmark(c, PH_NARROW, 0, 1);
  }
  return TRILENS_OK;
}

// the seeded traversal and its narrow phase, part by part
static int traverse_parts(trilens_ctx *c, const tl::TravArgs &a, const uint2 *seeds,
                          unsigned n_seeds) {
  for (int p = 0; p < c->parts; ++p) {
    if (p > 0) CK(tl::launch_part_init(c->ctr, c->stream));
    tmark(c, PH_TRAV, 0, 0);
    CK(tl::launch_traverse(a, seeds, n_seeds, c->budget, c->trav_blocks, c->trav_warps, c->stream,
                           p, c->parts));
    tmark(c, PH_TRAV, 0, 1);
    tmark(c, PH_NARROW, 0, 0);
    CK(tl::launch_narrow(a, 8 * c->n_sm, c->stream));
    tmark(c, PH_NARROW, 0, 1);
  }
  return TRILENS_OK;
}

// add the elapsed time of every recorded phase (the stream is synchronised)
static void tcollect(trilens_ctx *c) {
  for (int ph = 0; ph < PH_COUNT; ++ph)
    for (int k = 0; k < 2; ++k)
      if (c->ev_pending[ph][k]) {
        float ms = 0.f;
        if (cudaEventElapsedTime(&ms, c->ev[ph][k][0], c->ev[ph][k][1]) == cudaSuccess)
          c->phase_ms[ph] += ms;
        c->ev_pending[ph][k] = false;
      }
}

// ---- host-side constants (plain double; used only for conservative bounds)

static double host_sigma(double s) {
  if (!(s > 1.0)) return 0.0;
  double b = sqrt((s - 1.0) / s);
  double lg = log((1.0 + b) * (1.0 + b) * s);
  return 0.5 * TL_PI * TL_RE * TL_RE / s * ((3.0 - b * b * b * b) * lg - 2.0 * b * (2.0 - b * b));
}

// s where Eq. BWcross peaks (golden-section search; sigma is unimodal)
static double host_sigma_peak_s() {
  double lo = 1.2, hi = 4.0, g = 0.5 * (sqrt(5.0) - 1.0);
  for (int it = 0; it < 200; ++it) {
    double x1 = hi - g * (hi - lo), x2 = lo + g * (hi - lo);
    if (host_sigma(x1) < host_sigma(x2)) lo = x1;
    else hi = x2;
  }
  return 0.5 * (lo + hi);
}

static double host_sigma_max() { return host_sigma(host_sigma_peak_s()); }

// an upper bound of Eq. BWcross over s (for conservative tests elsewhere)
double tl_sigma_max_bound() { return host_sigma_max() * (1.0 + 1e-6); }

// the pads' A(q): r(s) s^q at its largest, over r_max (see tl_set_pads); in steps of 3 %
// of s - 1 up to s = 1e12 (r s^q is smooth, so 1e-3 covers the steps, and falls beyond)
static TLPadTable make_pad_table() {
  double a[kPadQ] = {};
  const double smax = host_sigma_max();
  for (double x = 1e-3; x < 1e12; x *= 1.03) {
    double v = sqrt(host_sigma(1.0 + x) / smax);
    const double p = pow(1.0 + x, 0.04);
    for (int k = 0; k < kPadQ; ++k, v *= p) a[k] = std::max(a[k], v);
  }
  TLPadTable t;
  for (int k = 0; k < kPadQ; ++k) t.a[k] = (float)(a[k] * (1.0 + 1e-3));
  return t;
}

static const TLPadTable &pad_table() {
  static const TLPadTable t = make_pad_table();
  return t;
}

static float round_up(double x) {
  float f = (float)x;
  if ((double)f < x) f = nextafterf(f, INFINITY);
  return f;
}
static float round_down(double x) {
  float f = (float)x;
  if ((double)f > x) f = nextafterf(f, -INFINITY);
  return f;
}

// constants of the FP32 narrow phase for a step of dt_fs and amplification kappa
TLNarrowConst tl_narrow_const(double dt_fs, double kappa) {
  const double u = ldexp(1.0, -24);
  const double sigma_max = host_sigma_max() * (1.0 + 1e-6);
  TLNarrowConst nk;
  nk.L = (float)(TL_C * dt_fs);
  nk.L_in = round_down((double)nk.L * (1.0 - 8.0 * u));
  nk.L_out = round_up((double)nk.L * (1.0 + 8.0 * u));
  nk.r2max = round_up(1e12 * kappa * sigma_max * (1.0 + 1e-5) / TL_PI);
  nk.kr = (float)(1e12 * kappa / TL_PI);
  nk.inv2mc4 = (float)(1.0 / (2.0 * TL_MEC2 * TL_MEC2));
  nk.pref = (float)(0.5 * TL_PI * TL_RE * TL_RE);
  // sure-miss radius per bin of s: sigma's largest value over the bin (at the
  // end nearer the peak, or the peak itself), with a relative margin
  const double s_peak = host_sigma_peak_s();
  nk.sbin[0] = 0.0f;
  for (int i = 1; i < TL_SBINS; ++i) {
    const int e = (i - 1) / TL_SBIN_OCT, k = (i - 1) % TL_SBIN_OCT;
    const double a = ldexp(1.0 + (double)k / TL_SBIN_OCT, e);
    const double b = ldexp(1.0 + (double)(k + 1) / TL_SBIN_OCT, e);
    double sig;
    if (i == TL_SBINS - 1) sig = host_sigma(a);  // [a, inf): sigma falls beyond the peak
    else if (b <= s_peak) sig = host_sigma(b);
    else if (a >= s_peak) sig = host_sigma(a);
    else sig = sigma_max;
    nk.sbin[i] = round_up(1e12 * kappa * std::min(sig * (1.0 + 1e-5), sigma_max) / TL_PI);
  }
  nk.suf[TL_SBINS - 1] = nk.sbin[TL_SBINS - 1];
  for (int i = TL_SBINS - 2; i >= 0; --i) nk.suf[i] = std::max(nk.sbin[i], nk.suf[i + 1]);
  return nk;
}

static void free_beam(tl::BuildBufs &w) {
  cudaFree(w.stat);
  cudaFree(w.rec);
  cudaFree(w.cell);
  cudaFree(w.count);
  cudaFree(w.start);
  cudaFree(w.scan_st);
  cudaFree(w.full);
  memset(&w, 0, sizeof(w));
}

// the buffers every step needs: SoAs and the counting sort's cells
static int alloc_beam(trilens_ctx *c, tl::BuildBufs &w, int64_t n, int64_t padded, int64_t cells) {
  const size_t m = (size_t)std::max<int64_t>(n, 1), mp = (size_t)std::max<int64_t>(padded, 1);
  CK(dalloc(&w.stat, 2 * m));
  CK(dalloc(&w.rec, 2 * mp));
  w.pos = w.rec;  // the statistical regime's two arrays
  w.dir = w.rec + mp;
  CK(dalloc(&w.cell, m));
  w.cells = cells;
  CK(dalloc(&w.count, (size_t)cells));
  CK(cudaMemsetAsync(w.count, 0, sizeof(uint32_t) * (size_t)cells, c->stream));
  CK(dalloc(&w.start, (size_t)cells + 1));
  CK(dalloc(&w.scan_st, (size_t)tl::scan_tiles(cells) + 1));
  return TRILENS_OK;
}

// moments of both beams in a frame, and their extremes (ext NULL: not wanted)
static int beam_moments(trilens_ctx *c, const TLFrame &f, double mom[2][15], double ext[2][14]) {
  const size_t md = tl::moment_doubles();
  double *dev = nullptr, h[2][29];
  CK(cudaMalloc((void **)&dev, sizeof(double) * 2 * md));
  cudaError_t e = cudaSuccess;
  for (int k = 0; k < 2 && !e; ++k) {
    e = tl::launch_beam_moments(c->beam[k], f, dev + k * md, c->stream);
    if (!e)
      e = cudaMemcpyAsync(h[k], dev + k * md, sizeof(h[k]), cudaMemcpyDeviceToHost, c->stream);
  }
  if (!e) e = cudaStreamSynchronize(c->stream);
  cudaFree(dev);
  CK(e);
  for (int k = 0; k < 2; ++k) {
    memcpy(mom[k], h[k], sizeof(double) * 15);
    if (ext) memcpy(ext[k], h[k] + 15, sizeof(double) * 14);
  }
  return TRILENS_OK;
}

// The statistical regime's arrays of m photons, in order in one buffer (256-byte aligned
// each); the bytes they take.
static size_t carve_full(tl::BuildBufs &w, char *base, size_t m) {
  size_t at = 0;
  auto take = [&](auto *&p, size_t count) {
    p = reinterpret_cast<std::remove_reference_t<decltype(p)>>(base + at);
    at = (at + sizeof(*p) * count + 255) & ~(size_t)255;
  };
  take(w.pos_u, m);
  take(w.dir_u, m);
  for (int q = 0; q < 2; ++q) {
    take(w.key[q], m);
    take(w.val[q], m);
  }
  take(w.sort_status, (size_t)w.sort_tiles * 256);
  take(w.sort_ep, 9);
  take(w.sort_raw, 8 * 256);
  take(w.sort_hist, 8 * 256);
  take(w.sort_tile, 8);
  take(w.nodes, m);
  take(w.parent_leaf, m);
  take(w.parent_node, m);
  take(w.rpre, 6 * m);
  take(w.rsuf, 6 * m);
  take(w.rtile, 6 * (size_t)tl::refit_tiles((int64_t)m));
  take(w.rsuper, tl::refit_super_floats((int64_t)m));
  take(w.nfirst, m);
  take(w.nlast, m);
  take(w.nlev, m);
  return at;
}

// the statistical regime's hierarchies and the seeded traversal's queues, on first use
int ensure_full(trilens_ctx *c) {
  if (c->full_ready) return TRILENS_OK;
  if (c->frame0.ident) {
    memcpy(c->moments, c->fmoments, sizeof(c->moments));
  } else {
    const int rcm = beam_moments(c, tl_ident_frame(), c->moments, nullptr);
    if (rcm) return rcm;
  }
  for (int k = 0; k < 2; ++k) {
    tl::BuildBufs &w = c->w[k];
    const size_t m = (size_t)std::max<int64_t>(c->beam[k].n, 1);
    w.sort_tiles = (int64_t)((m + TL_SORT_TILE - 1) / TL_SORT_TILE);
    w.sort_epoch = 0;
    // one allocation per beam (one by one, the arrays took a fifth of the first call)
    if (!w.full) CK(dalloc(&w.full, carve_full(w, nullptr, m)));
    carve_full(w, w.full, m);
    CK(tl::launch_static_soa(c->beam[k], w, c->stream));
    CK(cudaMemsetAsync(w.sort_raw, 0, sizeof(uint32_t) * 8 * 256, c->stream));
  }
  int lo = 0, hi = 0;
  CK(cudaDeviceGetStreamPriorityRange(&lo, &hi));
  if (!c->cut_stream)
    CK(cudaStreamCreateWithPriority(&c->cut_stream, cudaStreamNonBlocking, hi));
  if (!c->sum_stream) CK(cudaStreamCreateWithFlags(&c->sum_stream, cudaStreamNonBlocking));
  const unsigned long long warps = (unsigned long long)c->trav_blocks * c->trav_warps;
  int rc = alloc_queue(c, std::max<unsigned long long>(
                              1 << 20, 2ull * warps * (unsigned long long)c->p.stack_depth));
  if (rc) return rc;
  if ((rc = alloc_spill(c, c->spill_per_warp, warps))) return rc;
  // leaf-bucket pairs: 16 per photon to start, at most 2^29 (4 GiB) before a step
  // asks for more
  const unsigned long long cap = std::min<unsigned long long>(
      std::max<unsigned long long>(1 << 20, 16ull * (c->beam[0].n + c->beam[1].n)), 1ull << 29);
  if (c->leaf_cap < cap) {
    drop_run(c);
    cudaFree(c->leaves);
    c->leaves = nullptr;
    c->leaf_cap = 0;
    CK(dalloc(&c->leaves, (size_t)cap));
    c->leaf_cap = cap;
  }
  c->full_ready = true;
  return TRILENS_OK;
}

// Bits of the cells that order n photons: 2 to 4 cells per photon spread evenly, so up to a
// leaf's worth of photons per cell where a Gaussian bunch is densest (ten times the cells per
// photon cost more to scan than the finer order saves).  Large beams take 2^23, whose counts
// (32 MB) stay in L2 for the atomics, or half a cell per photon: both beams of 16M photons
// at 90 degrees 3.45 ms a step with 2^25, 3.21 with 2^23, 3.29 with 2^22; of 5e7 photons
// 11.8 ms with 2^27, 10.9 with 2^25, 11.5 with 2^23.
static int order_bits_for(int64_t n) {
  int lg = 0;
  while ((1ll << lg) < n) ++lg;
  return std::max(4, std::min(lg + 1, std::max(23, lg - 1)));
}

// The exact path's layout of both beams (sizes[k]: photons of every instance).
static int layout(trilens_ctx *c, const std::vector<int64_t> sizes[2]) {
  c->tree = c->beam[1].n <= c->beam[0].n ? 1 : 0;
  const size_t ni = sizes[0].size();
  for (int k = 0; k < 2; ++k) {
    std::vector<TLInst> in(ni);
    std::vector<uint32_t> group_inst;
    int64_t group = 0, cells = 0, first = 0;
    for (size_t q = 0; q < ni; ++q) {
      TLInst &I = in[q];
      memset(&I, 0, sizeof(I));
      I.n = (int)sizes[k][q];
      I.first = (int)first;
      first += sizes[k][q];
      I.bits = order_bits_for(sizes[k][q]);
      I.cell0 = (uint32_t)cells;
      cells += 1ll << in[q].bits;
      // (a tile's groups behind a small instance count as that instance's, without photons)
      if (sizes[k][q] > kTile) group = (group + 31) & ~31ll;
      if (ni > 1 && q > 0) group_inst.resize((size_t)group, (uint32_t)q - 1u);
      I.group0 = (int)group;
      group += (sizes[k][q] + 31) / 32;
      if (sizes[k][q] > kTile) group = (group + 31) & ~31ll;
      if (ni > 1) group_inst.resize((size_t)group, (uint32_t)q);
    }
    const int64_t tile = (group + 31) / 32;
    if (ni > 1) group_inst.resize((size_t)tile * 32, (uint32_t)ni - 1u);
    c->n_groups[k] = (int)tile * 32;
    if (k == c->tree) {  // levels 0..2 tile by tile, then what is above
      uint64_t up = (uint64_t)tile * (kTile + 32 + 1);
      for (size_t q = 0; q < ni; ++q) {
        in[q].lev[0] = (uint32_t)((uint64_t)in[q].group0 * 32);
        in[q].lev[1] = (uint32_t)((uint64_t)tile * kTile + (uint64_t)in[q].group0);
        in[q].lev[2] = (uint32_t)((uint64_t)tile * (kTile + 32) + (uint64_t)(in[q].group0 / 32));
        const int top = tl_top_level(in[q].n);
        for (int l = 3; l <= top; ++l) {
          in[q].lev[l] = (uint32_t)up;
          up += (uint64_t)tl_level_count(in[q].n, l);
        }
        c->max_top = std::max(c->max_top, top);
      }
      CK(dalloc(&c->box, 2 * (size_t)up));
    }
    CK(dalloc(&c->insts[k], ni));
    CK(cudaMemcpyAsync(c->insts[k], in.data(), sizeof(TLInst) * ni, cudaMemcpyHostToDevice,
                       c->stream));
    if (ni > 1) {
      CK(dalloc(&c->group_inst[k], group_inst.size()));
      CK(cudaMemcpyAsync(c->group_inst[k], group_inst.data(), sizeof(uint32_t) * group_inst.size(),
                         cudaMemcpyHostToDevice, c->stream));
    }
    const int rc = alloc_beam(c, c->w[k], c->beam[k].n, tile * kTile, cells);
    if (rc) return rc;
    // (copies from pageable memory have read the host tables when they return)
  }
  CK(dalloc(&c->frames, ni));
  return TRILENS_OK;
}

// ---- C ABI

extern "C" {

const char *trilens_version(void) { return "trilens-gb300 0.1 (sm_103a)"; }

const char *trilens_status_str(int code) {
  switch (code) {
    case TRILENS_OK: return "ok";
    case TRILENS_ERR_INVALID: return "invalid argument";
    case TRILENS_ERR_CAPACITY: return "hit buffer too small";
    case TRILENS_ERR_CUDA: return "CUDA error";
    case TRILENS_ERR_TIMEOUT: return "device wait reached its spin limit";
    case TRILENS_ERR_STACK: return "traversal overflow after retries";
    case TRILENS_ERR_NOMEM: return "device allocation failed";
    default: return "unknown status";
  }
}

const char *trilens_last_error(trilens_ctx *c) { return c ? c->msg : "no context"; }

static bool beam_ok(const trilens_beam *b) {
  if (!b || b->n < 0 || b->n >= (1ll << 27)) return false;
  if (b->n == 0) return true;
  return b->px && b->py && b->pz && b->dx && b->dy && b->dz && b->E;
}

void trilens_destroy(trilens_ctx *c) {
  if (!c) return;
  cudaSetDevice(c->device);
  if (c->stream) cudaStreamSynchronize(c->stream);
  else cudaDeviceSynchronize();
  free_beam(c->w[0]);
  free_beam(c->w[1]);
  cudaFree(c->queue);
  cudaFree(c->run_acc);
  cudaFree(c->hits);
  cudaFree(c->band);
  cudaFree(c->leaves);
  cudaFree(c->spill);
  cudaFree(c->ctr);
  cudaFree(c->partials);
  cudaFree(c->build_status);
  surrogate_free(c);
  deplete_free(c);
  cudaFreeHost(c->ctr_host);
  cudaFreeHost(c->build_status_host);
  for (int k = 0; k < 2; ++k) {
    cudaFree(c->inst_of[k]);
    cudaFree(c->inst_bounds[k]);
    cudaFree(c->insts[k]);
    cudaFree(c->group_inst[k]);
    cudaFree(c->grids[k]);
    for (int a = 0; a < 8; ++a) cudaFree(c->owned[k][a]);
  }
  cudaFree(c->frames);
  cudaFree(c->box);
  cudaFree(c->inst_tmp);
  cudaFree(c->run_status);
  cudaFreeHost(c->run_status_host);
  drop_run(c);
  if (c->cap_stream) cudaStreamDestroy(c->cap_stream);
  if (c->side_stream) cudaStreamDestroy(c->side_stream);
  if (c->sum_stream) cudaStreamDestroy(c->sum_stream);
  if (c->cut_stream) cudaStreamDestroy(c->cut_stream);
  if (c->fork_ev) cudaEventDestroy(c->fork_ev);
  if (c->join_ev) cudaEventDestroy(c->join_ev);
  for (int ph = 0; ph < PH_COUNT; ++ph)
    for (int k = 0; k < 2; ++k)
      for (int e = 0; e < 2; ++e)
        if (c->ev[ph][k][e]) cudaEventDestroy(c->ev[ph][k][e]);
  delete c;
}

}  // extern "C"

// Create a context; sizes NULL for a single problem, else the photons of every
// instance of each beam.
static int ctx_create(trilens_ctx **out, const trilens_beam *a, const trilens_beam *b,
                      const trilens_params *p, trilens_stream_t stream,
                      const std::vector<int64_t> *sizes) {
  if (!out) return TRILENS_ERR_INVALID;
  *out = nullptr;
  if (!beam_ok(a) || !beam_ok(b) || !p) return TRILENS_ERR_INVALID;
  if (!(p->dt_fs > 0.0) || !(p->kappa > 0.0) || !isfinite(p->dt_fs) || !isfinite(p->kappa))
    return TRILENS_ERR_INVALID;
  if (p->precision != TRILENS_FP64 && p->precision != TRILENS_FP32_BAND) return TRILENS_ERR_INVALID;
  if (p->leaf_bucket < 0 || p->leaf_bucket > 32) return TRILENS_ERR_INVALID;
  if (p->stack_depth != 0 && (p->stack_depth < 64 || p->stack_depth > 4096))
    return TRILENS_ERR_INVALID;
  if (p->block_shape < 0 || p->block_shape > TL_TRAV_MAX_WARPS) return TRILENS_ERR_INVALID;
  if (p->spin_limit < 0) return TRILENS_ERR_INVALID;

  trilens_ctx *c = new trilens_ctx();
  CK(cudaGetDevice(&c->device));
  c->stream = (cudaStream_t)stream;
  c->p = *p;
  if (c->p.leaf_bucket == 0) c->p.leaf_bucket = 4;
  if (c->p.stack_depth == 0) c->p.stack_depth = 512;
  if (c->p.block_shape == 0) c->p.block_shape = 4;
  if (c->p.spin_limit == 0) c->p.spin_limit = 1ll << 22;
  const trilens_beam *bs[2] = {a, b};
  for (int k = 0; k < 2; ++k) {
    TLBeam &t = c->beam[k];
    t.n = bs[k]->n;
    t.px = bs[k]->px; t.py = bs[k]->py; t.pz = bs[k]->pz;
    t.dx = bs[k]->dx; t.dy = bs[k]->dy; t.dz = bs[k]->dz;
    t.E = bs[k]->E; t.w = bs[k]->w;
  }
  int rc;
  // constants
  c->L64 = TL_C * c->p.dt_fs;
  c->sigma_max = host_sigma_max() * (1.0 + 1e-6);
  c->rmax = sqrt(1e12 * c->p.kappa * c->sigma_max / TL_PI) * (1.0 + 1e-6);
  c->L_lo = round_down(c->L64);
  c->L_hi = round_up(c->L64);
  c->half = round_up(0.5 * c->rmax * (1.0 + 1e-6) + 1e-9);
  c->nk = tl_narrow_const(c->p.dt_fs, c->p.kappa);
  // workspace
  CK(dalloc(&c->build_status, 1));
  CK(cudaMallocHost((void **)&c->build_status_host, sizeof(unsigned)));
  CK(cudaMemsetAsync(c->build_status, 0, sizeof(unsigned), c->stream));
  const std::vector<int64_t> one[2] = {{c->beam[0].n}, {c->beam[1].n}};
  if ((rc = layout(c, sizes ? sizes : one))) {
    trilens_destroy(c);
    return rc;
  }
  for (int k = 0; k < 2; ++k) {
    c->w[k].build_status = c->build_status;
    CK(tl::launch_static(c->beam[k], c->w[k].stat, c->stream));
    int64_t n = std::max<int64_t>(c->beam[k].n, 2);
    int lg = 0;
    while ((1ll << lg) < n) ++lg;
    // Morton resolution: one bit per axis beyond one cell per photon
    c->bits[k] = std::min(21, std::max(4, (lg + 2) / 3 + 1));
    c->key_bits[k] = 3 * c->bits[k];
    c->w[k].key_bits = c->key_bits[k];
  }
  if (!sizes) {
    for (int k = 0; k < 2; ++k) c->order_bits[k] = order_bits_for(c->beam[k].n);
    // one-time: the beams' mean directions (the frame), then their moments and extremes in
    // the frame, for the grids and boxes of every step
    c->frame0 = tl_ident_frame();
    double mean[2][5] = {}, le[2][2] = {};
    if (c->beam[0].n > 0 && c->beam[1].n > 0) {
      const int nd = tl::mean_doubles();
      std::vector<double> h(2 * (size_t)nd);
      double *part = nullptr;
      CK(cudaMalloc((void **)&part, sizeof(double) * h.size()));
      cudaError_t me = cudaSuccess;
      for (int k = 0; k < 2 && !me; ++k)
        me = tl::launch_mean_dir(c->beam[k], part + k * nd, c->stream);
      if (!me)
        me = cudaMemcpyAsync(h.data(), part, sizeof(double) * h.size(), cudaMemcpyDeviceToHost,
                             c->stream);
      if (!me) me = cudaStreamSynchronize(c->stream);
      cudaFree(part);
      CK(me);
      for (int k = 0; k < 2; ++k) {
        for (int q = 0; q < nd; ++q)
          mean[k][q % 5] += h[(size_t)k * nd + q] / (double)tl::mean_count(c->beam[k].n);
        le[k][0] = mean[k][3];
        le[k][1] = sqrt(std::max(mean[k][4] - mean[k][3] * mean[k][3], 0.0));
      }
      c->frame0 = tl_make_frame(mean[0], mean[1]);
    }
    if ((rc = beam_moments(c, c->frame0, c->fmoments, c->ext))) {
      trilens_destroy(c);
      return rc;
    }
    tl_set_pads(c->frame0, pad_table(), c->ext[0], c->ext[1], le[0], le[1], c->half);
    tl_set_needles(c->frame0, c->ext[0], c->ext[1], c->L64, c->half);
    CK(cudaMemcpyAsync(c->frames, &c->frame0, sizeof(TLFrame), cudaMemcpyHostToDevice, c->stream));
  }
  CK(tl::sort_prepare());
  CK(tl::refit_prepare());
  int dev_sm = 0;
  CK(cudaDeviceGetAttribute(&dev_sm, cudaDevAttrMultiProcessorCount, c->device));
  c->n_sm = dev_sm;
  c->trav_warps = c->p.block_shape;
  int bps = 0;
  CK(tl::traverse_config(c->p.precision == TRILENS_FP64, c->trav_warps, c->p.stack_depth, &bps));
  if (bps < 1) {
    trilens_destroy(c);
    return TRILENS_ERR_INVALID;
  }
  c->trav_blocks = bps * c->n_sm;
  c->hit_cap = std::max<unsigned long long>(1 << 16, 2ull * (c->beam[0].n + c->beam[1].n));
  CK(dalloc(&c->hits, c->hit_cap));
  c->band_cap = std::max<unsigned long long>(1 << 16, (c->beam[0].n + c->beam[1].n) / 4);
  CK(dalloc(&c->band, c->band_cap));
  // candidate pairs: what the first look leaves, of the order of the hits; in FP64 mode
  // every pair of overlapping boxes.  Grown when a step asks for more.
  c->leaf_cap = std::min<unsigned long long>(
      std::max<unsigned long long>(1 << 18, (c->p.precision == TRILENS_FP64 ? 16ull : 2ull) *
                                                (c->beam[0].n + c->beam[1].n)),
      1ull << 29);
  CK(dalloc(&c->leaves, c->leaf_cap));
  CK(dalloc(&c->ctr, 1));
  CK(cudaMallocHost((void **)&c->ctr_host, sizeof(TLCounters)));
  c->yield_blocks = 4 * c->n_sm;
  CK(cudaMalloc(&c->partials, tl::partial_bytes() * c->yield_blocks));
  CK(cudaStreamSynchronize(c->stream));
  *out = c;
  return TRILENS_OK;
}

extern "C" {

int trilens_create(trilens_ctx **out, const trilens_beam *a, const trilens_beam *b,
                   const trilens_params *p, trilens_stream_t stream) {
  return ctx_create(out, a, b, p, stream, nullptr);
}

}  // extern "C"

// The two beams' builds share nothing but the status word (set with atomic OR): beam
// B's runs on a side stream, forked from the context's stream and joined back before
// anything that reads them (in a captured run this is a fork and a join in the graph).
// Per-phase timing keeps them on one stream, one after the other.
static int fork_builds(trilens_ctx *c, bool *fork) {
  *fork = !c->timing && c->beam[0].n > 0 && c->beam[1].n > 0;
  if (!*fork) return TRILENS_OK;
  if (!c->side_stream) CK(cudaStreamCreateWithFlags(&c->side_stream, cudaStreamNonBlocking));
  if (!c->fork_ev) CK(cudaEventCreateWithFlags(&c->fork_ev, cudaEventDisableTiming));
  if (!c->join_ev) CK(cudaEventCreateWithFlags(&c->join_ev, cudaEventDisableTiming));
  CK(cudaEventRecord(c->fork_ev, c->stream));
  CK(cudaStreamWaitEvent(c->side_stream, c->fork_ev, 0));
  return TRILENS_OK;
}

static int join_builds(trilens_ctx *c, bool fork) {
  if (!fork) return TRILENS_OK;
  CK(cudaEventRecord(c->join_ev, c->side_stream));
  CK(cudaStreamWaitEvent(c->stream, c->join_ev, 0));
  return TRILENS_OK;
}

// Photon pairs are told by their needles (tl_set_needles) in steps where more than this
// many photons of the tree's beam have swept boxes that meet a photon's, at the beam's
// density.  Time of a step with boxes over that with needles, 75 steps of 60,000 to 4M photons
// of four shapes, head-on, at 0.6 and at 1.57 rad: 0.91 to 1.03 where 5 to 45 boxes meet a
// photon's, 0.87 to 1.09 at 45 to 65, 0.97 to 1.14 at 65 to 120, 0.99 to 1.31 at 120 to 270, 1.25
// to 1.8 at 360 to 1340 (2 x 4M photons 6.60 to 4.62 ms); below 1 beyond 65 only at 1.57 rad, by 3 %.
// Batches keep the boxes (2 x 64 instances of up to 131072 photons 6.9 and 7.2 ms).
constexpr double kNeedlePairs = 64.0;

// The ordering grids of a single problem's beams for the step with travel T to the
// swept boxes' centres: per axis of the frame the mean of the centres +- 5 standard
// deviations, in closed form from the moments (centres outside are clamped to the edge
// cells; the grid only shapes the tree), and cells in the proportions of the boxes'
// extents: pad plus the travel of a typical photon of either beam.
static void step_grids(trilens_ctx *c, double T, TLGrid g[2]) {
  double ru[3], s[3], near = 0.0;
  for (int k = 0; k < 3; ++k) {
    const TLFrame &f = c->frame0;
    ru[k] = (double)f.r[3 * k] * f.u[0] + (double)f.r[3 * k + 1] * f.u[1] +
            (double)f.r[3 * k + 2] * f.u[2];
    s[k] = 2.0 * f.typ;
    for (int h = 0; h < 2; ++h) {
      const double *m = c->fmoments[h], n = (double)std::max<int64_t>(c->beam[h].n, 1);
      const double mean = m[3 + k] / n;
      const double var = std::max(m[12 + k] / n - mean * mean, 0.0);
      s[k] += c->L64 * sqrt((mean - ru[k]) * (mean - ru[k]) + var);
    }
  }
  for (int h = 0; h < 2; ++h) {
    double lo[3], range[3];
    double vol = 15.75;  // (2 pi)^1.5: of a Gaussian beam's peak density
    for (int k = 0; k < 3; ++k) {
      const double *m = c->fmoments[h], n = (double)std::max<int64_t>(c->beam[h].n, 1);
      const double mean = (m[k] + T * m[3 + k]) / n;
      const double msq = (m[6 + k] + 2.0 * T * m[9 + k] + T * T * m[12 + k]) / n;
      const double sd5 = 5.0 * sqrt(std::max(msq - mean * mean, 0.0));
      lo[k] = mean - 0.5 * c->L64 * ru[k] - sd5;
      range[k] = 2.0 * sd5;
      vol *= 0.2 * sd5 / s[k];
    }
    if (h == c->tree) near = (double)c->beam[h].n / vol;
    g[h] = tl_make_grid(lo, range, s, c->order_bits[h]);
    const double *e = c->ext[1 - h];
    tl_beam_box(e, e[12], e[13], c->frame0, T - 0.5 * c->L64, c->L64, c->half, g[h].clo, g[h].chi);
  }
  c->needles = c->frame0.axis >= 0 && near > kNeedlePairs;
}

// The exact path's order of both beams and the tree of the smaller one.
static int build_exact(trilens_ctx *c, int64_t step) {
  const double ct = TL_C * ((double)step * c->p.dt_fs);
  const double T = ct + 0.5 * c->L64;
  const bool batch = c->n_inst > 1;
  TLGrid grid[2];
  if (batch)
    CK(tl::launch_inst_grid(c->inst_bounds[0], c->inst_bounds[1], c->frames, c->insts[0],
                            c->insts[1], c->n_inst, T, c->L64, c->half, c->grids[0], c->grids[1],
                            c->stream));
  else
    step_grids(c, T, grid);
  c->exact_step = c->full_step = -1;  // the two builds share the sorted photons
  // The root of the descent, tested on the host: where the boxes of all swept boxes of
  // the two beams do not meet (Eq. CollDet), no photon of one meets one of the other,
  // and the step has nothing to order or to test.
  c->apart = c->beam[0].n <= 0 || c->beam[1].n <= 0;
  for (int k = 0; k < 3 && !batch; ++k)
    c->apart = c->apart || grid[0].clo[k] > grid[1].chi[k] || grid[1].clo[k] > grid[0].chi[k];
  if (c->apart) {
    c->exact_step = step;
    return TRILENS_OK;
  }
  bool fork;
  if (int rc = fork_builds(c, &fork)) return rc;
  for (int k = 0; k < 2; ++k) {
    cudaStream_t st = (fork && k == 1) ? c->side_stream : c->stream;
    tl::BuildBufs &w = c->w[k];
    tmark(c, PH_PROP, k, 0);
    tl::OrderArgs o;
    memset(&o, 0, sizeof(o));
    o.n = c->beam[k].n;
    o.stat = w.stat;
    o.ct = (float)ct;
    o.L = (float)c->L64;
    o.half = c->half;
    o.frames = c->frames;
    if (!batch) o.grid = grid[k];
    o.grids = c->grids[k];
    o.inst_of = c->inst_of[k];
    o.inst = c->insts[k];
    o.cell = w.cell;
    o.count = w.count;
    o.scan_st = w.scan_st;
    o.scan_tiles = (int)tl::scan_tiles(w.cells);
    if (c->n_inst <= 1) o.inst_of = nullptr;
    CK(tl::launch_order(o, st));
    tmark(c, PH_PROP, k, 1);
    tmark(c, PH_SORT, k, 0);
    CK(tl::launch_cell_scan(w.count, w.start, w.cells, w.scan_st, c->p.spin_limit,
                            c->debug_stall_sort, c->build_status, st));
    tl::PlaceArgs pl;
    memset(&pl, 0, sizeof(pl));
    pl.b = c->beam[k];
    pl.ct = ct;
    pl.n_pad = (int64_t)c->n_groups[k] * 32;
    pl.stat = w.stat;
    pl.cell = w.cell;
    pl.start = w.start;
    pl.inst_of = o.inst_of;
    pl.inst = c->insts[k];
    pl.rec = w.rec;
    CK(tl::launch_place(pl, st));
    tmark(c, PH_SORT, k, 1);
    c->phase_launches[PH_PROP] += 1;
    c->phase_launches[PH_SORT] += 2;
    if (k != c->tree) continue;
    tmark(c, PH_REFIT, k, 0);
    tl::BoxArgs b;
    memset(&b, 0, sizeof(b));
    b.rec = w.rec;
    b.inst = c->insts[k];
    b.start = w.start;
    b.group_inst = c->group_inst[k];
    b.frames = c->frames;
    b.Llo = c->L_lo;
    b.Lhi = c->L_hi;
    b.half = c->half;
    b.beam = k;
    b.needles = c->needles;
    b.box = c->box;
    b.build_status = c->build_status;
    CK(tl::launch_boxes(b, c->n_groups[k] / 32, c->n_inst, c->max_top, st));
    tmark(c, PH_REFIT, k, 1);
    c->phase_launches[PH_REFIT] += c->max_top >= 3 ? 2 : 1;
  }
  if (int rc = join_builds(c, fork)) return rc;
  c->exact_step = step;
  return TRILENS_OK;
}

// The statistical regime's binary hierarchies of both beams, in Morton order.
static int build_full(trilens_ctx *c, int64_t step) {
  if (int rc = ensure_full(c)) return rc;
  c->exact_step = c->full_step = -1;
  const double ct = TL_C * ((double)step * c->p.dt_fs);
  const double T = ct + 0.5 * c->L64;
  bool fork;
  if (int rc = fork_builds(c, &fork)) return rc;
  for (int k = 0; k < 2; ++k) {
    const int64_t n = c->beam[k].n;
    if (n <= 0) continue;
    cudaStream_t st = (fork && k == 1) ? c->side_stream : c->stream;
    // Morton box of the step: per axis the mean of the swept boxes' centres
    // c = p0 + T d +- 5 standard deviations, in closed form from the beam's
    // moments (centres outside are clamped to the edge cells).  Unlike the
    // extreme centres, the moments of a large beam barely change from one
    // draw to the next, so neither do the cells a level of the hierarchy
    // stands for.
    float lo[3], scale[3];
    const double maxq = (double)((1u << c->bits[k]) - 1u);
    for (int a = 0; a < 3; ++a) {
      const double *m = c->moments[k], nn = (double)n;
      const double mean = (m[a] + T * m[3 + a]) / nn;
      const double msq = (m[6 + a] + 2.0 * T * m[9 + a] + T * T * m[12 + a]) / nn;
      const double h = 5.0 * std::sqrt(std::max(msq - mean * mean, 0.0));
      const float l = (float)(mean - h), u = (float)(mean + h);
      lo[a] = l;
      scale[a] = u > l ? (float)(maxq / ((double)u - (double)l)) : 0.0f;
    }
    tl::BuildBufs &w = c->w[k];
    tmark(c, PH_PROP, k, 0);
    CK(tl::launch_propagate(c->beam[k], ct, (float)c->L64, lo, scale, c->bits[k], w,
                            n > 1 ? (c->key_bits[k] + 7) / 8 : 0, st));
    tmark(c, PH_PROP, k, 1);
    tmark(c, PH_SORT, k, 0);
    CK(tl::launch_sort(w, n, c->key_bits[k], c->p.spin_limit, c->debug_stall_sort,
                       c->build_status, &c->sel[k], st));
    tmark(c, PH_SORT, k, 1);
    if (n <= 1) {  // no sort: copy the one photon (a longer beam is gathered by the sort)
      tmark(c, PH_GATHER, k, 0);
      CK(tl::launch_gather(w, n, st));
      tmark(c, PH_GATHER, k, 1);
      c->phase_launches[PH_GATHER] += 1;
    }
    tmark(c, PH_EMIT, k, 0);
    CK(tl::launch_karras(w, n, c->sel[k], c->p.leaf_bucket, st));
    tmark(c, PH_EMIT, k, 1);
    tmark(c, PH_REFIT, k, 0);
    CK(tl::launch_refit(w, n, c->L_lo, c->L_hi, c->half, c->n_sm, st));
    tmark(c, PH_REFIT, k, 1);
    c->phase_launches[PH_PROP] += 1;
    c->phase_launches[PH_SORT] += n > 1 ? 1 + (c->key_bits[k] + 7) / 8 : 0;
    c->phase_launches[PH_EMIT] += 1;
    c->phase_launches[PH_REFIT] += tl::refit_tiles(n) > 1 ? 3 : 1;
  }
  if (int rc = join_builds(c, fork)) return rc;
  c->full_step = step;
  return TRILENS_OK;
}

int need_full(trilens_ctx *c, int64_t step) {
  return c->full_step == step ? TRILENS_OK : build_full(c, step);
}

extern "C" {

int trilens_build(trilens_ctx *c, int64_t step) {
  if (!c) return TRILENS_ERR_INVALID;
  if (step < 0) return fail(c, TRILENS_ERR_INVALID, "step < 0");
  CK(cudaSetDevice(c->device));
  // a context that uses the statistical regime builds its hierarchies; a collision of
  // the whole beams builds the exact path's trees if they do not stand for the step
  const int rc = c->sur ? build_full(c, step) : build_exact(c, step);
  if (rc) return rc;
  c->built_step = step;
  return TRILENS_OK;
}

}  // extern "C"

// A step's (or a captured run's) failure from its traversal and build status
// words, or TRILENS_OK.  After a wait that expired or an invalid hierarchy the
// sort's status words are cleared before the next sort, the queue is reset to
// the sentinel (a traversal cut short may leave items in it) and the build
// status is cleared.
static int status_failure(trilens_ctx *c, unsigned trav_st, unsigned build_st) {
  if (!((trav_st | build_st) & (TL_ST_TIMEOUT | TL_ST_BADTREE))) return TRILENS_OK;
  c->exact_step = c->full_step = -1;
  c->w[0].sort_epoch = c->w[1].sort_epoch = 0;
  if (c->queue)
    CK(cudaMemsetAsync(c->queue, 0xff, sizeof(uint2) * (size_t)c->queue_cap, c->stream));
  CK(cudaMemsetAsync(c->build_status, 0, sizeof(unsigned), c->stream));
  CK(cudaStreamSynchronize(c->stream));
  if (build_st & TL_ST_TIMEOUT)
    return fail(c, TRILENS_ERR_TIMEOUT,
                "a device wait reached spin_limit=%lld (the look-back of a build's scan or sort)",
                (long long)c->p.spin_limit);
  if (trav_st & TL_ST_TIMEOUT)
    return fail(c, TRILENS_ERR_TIMEOUT,
                "a device wait reached spin_limit=%lld (a traversal warp waiting for work)",
                (long long)c->p.spin_limit);
  return fail(c, TRILENS_ERR_CUDA,
              "the refit met a node reference out of range: the step's hierarchy is invalid "
              "(internal error)");
}

tl::TravArgs trav_args(trilens_ctx *c, double ct) {
  tl::TravArgs a;
  memset(&a, 0, sizeof(a));
  for (int k = 0; k < 2; ++k) {
    TLTree &t = k ? a.B : a.A;
    const bool full = c->full_step >= 0;  // the buffers hold the statistical regime's order
    t.pos = full ? c->w[k].pos : c->w[k].rec;
    t.dir = full ? c->w[k].dir : c->w[k].rec + 1;
    t.stride = full ? 1u : 2u;
    t.nodes = c->w[k].nodes;
    t.n = c->beam[k].n;
    t.super = (uint32_t)(t.n > 1 ? t.n - 1 : 0);
  }
  a.mA = c->beam[0];
  a.mB = c->beam[1];
  a.ct = ct;
  a.dt = c->p.dt_fs;
  a.kappa = c->p.kappa;
  a.nk = c->nk;
  a.fp64 = c->p.precision == TRILENS_FP64;
  a.ctr = c->ctr;
  a.hits = c->hits;
  a.hit_cap = c->hit_cap;
  a.band = c->band;
  a.band_cap = c->band_cap;
  a.leaves = c->leaves;
  a.leaf_cap = c->leaf_cap;
  a.queue = reinterpret_cast<unsigned long long *>(c->queue);
  a.queue_cap = c->queue_cap;
  a.spill = c->spill;
  a.spill_per_warp = c->spill_per_warp;
  a.spin_limit = c->p.spin_limit;
  a.stack_depth = c->p.stack_depth;
  a.leaf_bucket = c->p.leaf_bucket;
  a.build_status = c->build_status;
  return a;
}

int run_exact(trilens_ctx *c, double ct, const uint2 *seeds, unsigned n_seeds, int *retries_out) {
  int retries = 0;
  TLCounters &h = *c->ctr_host;
  while (true) {
    tl::TravArgs a = trav_args(c, ct);
    CK(tl::launch_step_init(c->ctr, c->build_status, nullptr, c->stream));
    const int rcp = seeds ? traverse_parts(c, a, seeds, n_seeds)
                          : (c->apart ? TRILENS_OK : collide_parts(c, a));
    if (rcp) return rcp;
    c->phase_launches[PH_TRAV] += c->parts;
    c->phase_launches[PH_NARROW] += c->parts;
    if (!a.fp64) {
      tmark(c, PH_BAND, 0, 0);
      CK(tl::launch_band(a, c->n_sm * 4, c->stream));
      tmark(c, PH_BAND, 0, 1);
      c->phase_launches[PH_BAND] += 1;
    }
    tmark(c, PH_YIELD, 0, 0);
    CK(tl::launch_yield(a, c->partials, c->yield_blocks, c->stream));
    tmark(c, PH_YIELD, 0, 1);
    c->phase_launches[PH_YIELD] += 1;
    CK(cudaMemcpyAsync(&h, c->ctr, sizeof(TLCounters), cudaMemcpyDeviceToHost, c->stream));
    CK(cudaMemcpyAsync(c->build_status_host, c->build_status, sizeof(unsigned),
                       cudaMemcpyDeviceToHost, c->stream));
    CK(cudaStreamSynchronize(c->stream));
    tcollect(c);
    const unsigned st = h.status | *c->build_status_host;
    if (int rf = status_failure(c, h.status, *c->build_status_host)) return rf;
    bool again = false;
    int rc;
    if (st & TL_ST_BAND_OVF) {
      if ((rc = grow(c, &c->band, &c->band_cap, h.band))) return rc;
      again = true;
    }
    if (st & TL_ST_HIT_OVF) {
      if ((rc = grow(c, &c->hits, &c->hit_cap, h.hits + (again ? h.band : 0)))) return rc;
      again = true;
    }
    if (st & TL_ST_SPILL_OVF) {  // the queue: larger, and every slot the sentinel again
      // (a pass stops soon after the queue is full, so what it asked for says little: four
      // times as large, up to the largest)
      const unsigned long long need = kQueueChunk * (h.q_tail + h.q_tail / 4 + 1024);
      if ((rc = alloc_queue(c, std::max(need, std::min(4 * c->queue_cap, 1ull << 30))))) return rc;
      again = true;
    }
    if (st & TL_ST_PRIV_OVF) {  // a warp's spill area: twice as large
      if ((rc = alloc_spill(c, 2 * c->spill_per_warp, c->spill_warps))) return rc;
      again = true;
    }
    if (st & TL_ST_LEAFQ) {  // the leaf-pair list: larger, or the step in more parts
      if ((rc = leaves_for(c, h.max_part_leaves))) return rc;
      again = true;
    }
    if (!again) break;
    if (++retries > 16)  // each makes room for at least twice as much of something
      return fail(c, TRILENS_ERR_STACK,
                  "buffers kept overflowing (status 0x%x; queue of %llu node pairs, %llu chunks "
                  "asked for; spill areas of %u)",
                  st, c->queue_cap, (unsigned long long)h.q_tail, c->spill_per_warp);
  }
  if (retries_out) *retries_out = retries;
  return TRILENS_OK;
}

extern "C" {

int trilens_collide_step(trilens_ctx *c, int64_t step, uint32_t *hits, int64_t cap,
                         int64_t *n_hits) {
  if (!c) return TRILENS_ERR_INVALID;
  if (step != c->built_step) return fail(c, TRILENS_ERR_INVALID, "step %lld not built", (long long)step);
  if (cap < 0 || (hits == nullptr && cap > 0)) return fail(c, TRILENS_ERR_INVALID, "bad hit buffer");
  CK(cudaSetDevice(c->device));
  const double ct = TL_C * ((double)step * c->p.dt_fs);
  int retries = 0;
  int rc = TRILENS_OK;
  if (c->exact_step != step && (rc = build_exact(c, step))) return rc;
  rc = run_exact(c, ct, nullptr, 0, &retries);
  if (rc) return rc;
  TLCounters &h = *c->ctr_host;
  if (hits && (int64_t)h.count > cap) {
    // the step is not added to the cumulative yield: the caller repeats it
    // with a larger buffer (the hierarchies stay built)
    if (n_hits) *n_hits = (int64_t)h.count;
    return fail(c, TRILENS_ERR_CAPACITY, "need %llu hit slots", (unsigned long long)h.count);
  }
  trilens_step_stats &s = c->last;
  s.step = step;
  s.count = (int64_t)h.count;
  s.weighted = h.weighted;
  s.hsum = h.hsum;
  s.hxor = h.hxor;
  s.narrow_tests = (int64_t)h.narrow_tests;
  s.node_tests = (int64_t)h.node_tests;
  s.leaf_pairs = (int64_t)h.leaf_pairs;
  s.band = (int64_t)h.band;
  s.retries = retries;
  c->tot_count += (double)h.count;
  c->tot_weighted += h.weighted;
  if (n_hits) *n_hits = (int64_t)h.count;
  if (hits && cap > 0) {
    const unsigned long long ncopy = std::min<unsigned long long>(h.count, (unsigned long long)cap);
    if (ncopy)
      CK(cudaMemcpyAsync(hits, c->hits, sizeof(uint2) * ncopy, cudaMemcpyDeviceToDevice, c->stream));
  }
  return TRILENS_OK;
}

// ---- batches of independent instances ------------------------------------

static int ensure_graph(trilens_ctx *c);

static int batch_prepare(trilens_ctx *c, const trilens_beam *const src[2], int32_t n_inst) {
  // concatenate each side's instances into library-owned arrays
  std::vector<tl::InstSrc> tab(n_inst);
  int64_t tot[2] = {0, 0};
  for (int k = 0; k < 2; ++k)
    for (int q = 0; q < n_inst; ++q) tot[k] += src[k][q].n;
  for (int k = 0; k < 2; ++k) {
    int64_t off = 0;
    for (int q = 0; q < n_inst; ++q) {
      const trilens_beam &bq = src[k][q];
      const double *ps[8] = {bq.px, bq.py, bq.pz, bq.dx, bq.dy, bq.dz, bq.E, bq.w};
      for (int a = 0; a < 8; ++a) tab[q].p[a] = ps[a];
      tab[q].n = bq.n;
      tab[q].off = off;
      off += bq.n;
    }
    for (int a = 0; a < 8; ++a) CK(dalloc(&c->owned[k][a], (size_t)std::max<int64_t>(tot[k], 1)));
    CK(dalloc(&c->inst_of[k], (size_t)std::max<int64_t>(tot[k], 1)));
    tl::InstSrc *dtab = nullptr;
    double **dptr = nullptr;
    CK(cudaMalloc((void **)&dtab, sizeof(tl::InstSrc) * n_inst));
    CK(cudaMalloc((void **)&dptr, sizeof(double *) * 8));
    CK(cudaMemcpyAsync(dtab, tab.data(), sizeof(tl::InstSrc) * n_inst, cudaMemcpyHostToDevice,
                       c->stream));
    CK(cudaMemcpyAsync(dptr, c->owned[k], sizeof(double *) * 8, cudaMemcpyHostToDevice, c->stream));
    CK(tl::launch_gather_instances(dtab, n_inst, tot[k], dptr, c->inst_of[k], c->stream));
    CK(cudaStreamSynchronize(c->stream));
    cudaFree(dtab);
    cudaFree(dptr);
  }
  return TRILENS_OK;
}

int trilens_batch_create(trilens_ctx **out, const trilens_beam *a, const trilens_beam *b,
                         int32_t n_inst, const trilens_params *p, trilens_stream_t stream) {
  if (!out) return TRILENS_ERR_INVALID;
  *out = nullptr;
  if (!a || !b || !p || n_inst < 1 || n_inst > 65536) return TRILENS_ERR_INVALID;
  int64_t tot[2] = {0, 0};
  std::vector<int64_t> sizes[2];
  for (int q = 0; q < n_inst; ++q) {
    if (!beam_ok(&a[q]) || !beam_ok(&b[q])) return TRILENS_ERR_INVALID;
    sizes[0].push_back(a[q].n);
    sizes[1].push_back(b[q].n);
    tot[0] += a[q].n;
    tot[1] += b[q].n;
  }
  if (tot[0] >= (1ll << 27) || tot[1] >= (1ll << 27)) return TRILENS_ERR_INVALID;
  // a throwaway context holds the owned inputs while they are gathered
  trilens_ctx tmp;
  tmp.stream = (cudaStream_t)stream;
  trilens_ctx *c = &tmp;
  const trilens_beam *src[2] = {a, b};
  int rc = batch_prepare(c, src, n_inst);
  if (rc) return rc;
  trilens_beam cat[2];
  for (int k = 0; k < 2; ++k) {
    cat[k].n = tot[k];
    cat[k].px = tmp.owned[k][0]; cat[k].py = tmp.owned[k][1]; cat[k].pz = tmp.owned[k][2];
    cat[k].dx = tmp.owned[k][3]; cat[k].dy = tmp.owned[k][4]; cat[k].dz = tmp.owned[k][5];
    cat[k].E = tmp.owned[k][6]; cat[k].w = tmp.owned[k][7];
  }
  trilens_ctx *ctx = nullptr;
  rc = ctx_create(&ctx, &cat[0], &cat[1], p, stream, n_inst > 1 ? sizes : nullptr);
  if (rc) {
    for (int k = 0; k < 2; ++k) {
      for (int q = 0; q < 8; ++q) cudaFree(tmp.owned[k][q]);
      cudaFree(tmp.inst_of[k]);
    }
    return rc;
  }
  c = ctx;
  for (int k = 0; k < 2; ++k) {
    for (int q = 0; q < 8; ++q) {
      c->owned[k][q] = tmp.owned[k][q];
      tmp.owned[k][q] = nullptr;
    }
    c->inst_of[k] = tmp.inst_of[k];
    tmp.inst_of[k] = nullptr;
  }
  c->n_inst = n_inst;
  if (n_inst > 1) {
    CK(cudaMalloc((void **)&c->inst_tmp, sizeof(long long) * 12 * n_inst));
    for (int k = 0; k < 2; ++k) {
      CK(dalloc(&c->inst_bounds[k], (size_t)12 * n_inst));
      CK(dalloc(&c->grids[k], (size_t)n_inst));
      CK(tl::launch_inst_bounds(c->beam[k], c->inst_of[k], nullptr, n_inst, c->inst_tmp,
                                c->inst_bounds[k], c->stream));
    }
    double *le = nullptr;  // ln E of the instances, beam after beam
    CK(dalloc(&le, (size_t)4 * n_inst));
    cudaError_t fe = cudaSuccess;
    for (int k = 0; k < 2 && !fe; ++k)
      fe = tl::launch_inst_energy(c->beam[k], c->insts[k], n_inst, le + 2 * (size_t)k * n_inst,
                                  c->stream);
    if (!fe)
      fe = tl::launch_inst_frames(c->inst_bounds[0], c->inst_bounds[1], le, le + 2 * (size_t)n_inst,
                                  pad_table(), c->half, n_inst, c->frames, c->stream);
    cudaFree(le);  // (waits for the kernels)
    CK(fe);
    for (int k = 0; k < 2; ++k)  // the bounds in every instance's frame
      CK(tl::launch_inst_bounds(c->beam[k], c->inst_of[k], c->frames, n_inst, c->inst_tmp,
                                c->inst_bounds[k], c->stream));
  }
  if ((rc = ensure_graph(c))) return rc;
  CK(cudaStreamSynchronize(c->stream));
  *out = c;
  return TRILENS_OK;
}

// One step of a captured run: the collide sequence without host checks (the
// collisions need none); every overflow
// is flagged in run_status, and the step's totals are added on the device.
static int graph_collide(trilens_ctx *c, int64_t step, double *yields) {
  const double ct = TL_C * ((double)step * c->p.dt_fs);
  tl::TravArgs a = trav_args(c, ct);
  CK(tl::launch_step_init(c->ctr, c->build_status, c->run_status, c->stream));
  {
    const int rcp = collide_parts(c, a);
    if (rcp) return rcp;
  }
  if (!a.fp64) CK(tl::launch_band(a, c->n_sm * 4, c->stream));
  CK(tl::launch_yield(a, c->partials, c->yield_blocks, c->stream));
  if (yields && c->n_inst > 1)
    CK(tl::launch_yield_inst(a, c->inst_of[0], yields, c->yield_blocks, c->stream));
  CK(tl::launch_step_finish(c->ctr, c->run_status, c->run_acc, c->stream));
  return TRILENS_OK;
}

static int capture_run(trilens_ctx *c, int64_t first, int64_t steps, double *yields) {
  drop_run(c);
  const int timing = c->timing;
  c->timing = 0;
  cudaStream_t saved = c->stream;
  c->stream = c->cap_stream;
  CK(cudaStreamBeginCapture(c->cap_stream, cudaStreamCaptureModeThreadLocal));
  int rc = TRILENS_OK;
  cudaError_t e = cudaMemsetAsync(c->run_status, 0, sizeof(unsigned), c->stream);
  if (e == cudaSuccess && c->run_acc)
    e = cudaMemsetAsync(c->run_acc, 0, sizeof(TLRunAcc), c->stream);
  if (e == cudaSuccess && yields && c->n_inst > 1)
    e = cudaMemsetAsync(yields, 0, sizeof(double) * 2 * c->n_inst, c->stream);
  if (e != cudaSuccess) rc = fail(c, TRILENS_ERR_CUDA, "capture: %s", cudaGetErrorString(e));
  for (int64_t k = first; rc == TRILENS_OK && k < first + steps; ++k) {
    rc = build_exact(c, k);
    if (rc == TRILENS_OK && !c->apart) rc = graph_collide(c, k, yields);
  }
  c->exact_step = -1;  // (captured, not built)
  cudaGraph_t g = nullptr;
  e = cudaStreamEndCapture(c->cap_stream, &g);
  c->stream = saved;
  c->timing = timing;
  if (rc) {
    if (g) cudaGraphDestroy(g);
    return rc;
  }
  if (e != cudaSuccess) return fail(c, TRILENS_ERR_CUDA, "end capture: %s", cudaGetErrorString(e));
  e = cudaGraphInstantiate(&c->gexec, g, 0);
  cudaGraphDestroy(g);
  if (e != cudaSuccess) return fail(c, TRILENS_ERR_CUDA, "instantiate: %s", cudaGetErrorString(e));
  ++c->g_captures;
  c->g_first = first;
  c->g_steps = steps;
  c->g_yields = yields;
  return TRILENS_OK;
}

// Capture (if needed) and replay a multi-step run; on an overflow grow the
// buffer and run again.
static int replay_run(trilens_ctx *c, int64_t first_step, int64_t steps, double *yields) {
  for (int attempt = 0; attempt < 8; ++attempt) {
    if (!c->gexec || c->g_first != first_step || c->g_steps != steps || c->g_yields != yields) {
      int rc = capture_run(c, first_step, steps, yields);
      if (rc) return rc;
    }
    c->exact_step = c->full_step = -1;
    CK(cudaGraphLaunch(c->gexec, c->stream));
    CK(cudaMemcpyAsync(c->run_status_host, c->run_status, sizeof(unsigned), cudaMemcpyDeviceToHost,
                       c->stream));
    CK(cudaMemcpyAsync(c->build_status_host, c->build_status, sizeof(unsigned),
                       cudaMemcpyDeviceToHost, c->stream));
    CK(cudaStreamSynchronize(c->stream));
    const unsigned st = *c->run_status_host | *c->build_status_host;
    if (int rf = status_failure(c, *c->run_status_host, *c->build_status_host)) return rf;
    if (!(st & (TL_ST_HIT_OVF | TL_ST_BAND_OVF | TL_ST_LEAFQ))) {
      c->built_step = first_step + steps - 1;  // (collided again, it is ordered again)
      return TRILENS_OK;
    }
    // grow what overflowed (to the largest size a step asked for) and capture again
    TLRunAcc m;
    CK(cudaMemcpyAsync(&m, c->run_acc, sizeof(TLRunAcc), cudaMemcpyDeviceToHost, c->stream));
    CK(cudaStreamSynchronize(c->stream));
    int rc;
    if (st & TL_ST_HIT_OVF && (rc = grow(c, &c->hits, &c->hit_cap, m.max_hits + m.max_band)))
      return rc;
    if (st & TL_ST_BAND_OVF && (rc = grow(c, &c->band, &c->band_cap, m.max_band))) return rc;
    if (st & TL_ST_LEAFQ && (rc = leaves_for(c, m.max_leaves))) return rc;
  }
  return fail(c, TRILENS_ERR_STACK, "captured run kept overflowing");
}

// graph resources of a context (a batch context makes them when created)
static int ensure_graph(trilens_ctx *c) {
  if (!c->cap_stream) CK(cudaStreamCreateWithFlags(&c->cap_stream, cudaStreamNonBlocking));
  if (!c->run_status) CK(dalloc(&c->run_status, 1));
  if (!c->run_status_host) CK(cudaMallocHost((void **)&c->run_status_host, sizeof(unsigned)));
  if (!c->run_acc) CK(dalloc(&c->run_acc, 1));
  return TRILENS_OK;
}

int trilens_batch_run(trilens_ctx *c, int64_t first_step, int64_t steps, double *yields) {
  if (!c) return TRILENS_ERR_INVALID;
  if (first_step < 0 || steps < 1 || c->n_inst < 2 || !c->cap_stream)
    return fail(c, TRILENS_ERR_INVALID, "batch_run needs a batch context, first_step >= 0, steps >= 1");
  CK(cudaSetDevice(c->device));
  return replay_run(c, first_step, steps, yields);
}

int trilens_run(trilens_ctx *c, int64_t first_step, int64_t steps, trilens_step_stats *out) {
  if (!c) return TRILENS_ERR_INVALID;
  if (first_step < 0 || steps < 1 || c->n_inst > 1)
    return fail(c, TRILENS_ERR_INVALID, "run needs a single context, first_step >= 0, steps >= 1");
  CK(cudaSetDevice(c->device));
  int rc = ensure_graph(c);
  if (rc) return rc;
  if ((rc = replay_run(c, first_step, steps, nullptr))) return rc;
  TLRunAcc h;
  CK(cudaMemcpyAsync(&h, c->run_acc, sizeof(TLRunAcc), cudaMemcpyDeviceToHost, c->stream));
  CK(cudaStreamSynchronize(c->stream));
  c->tot_count += (double)h.count;
  c->tot_weighted += h.weighted;
  if (out) {
    out->step = steps;
    out->count = (int64_t)h.count;
    out->weighted = h.weighted;
    out->hsum = h.hsum;
    out->hxor = h.hxor;
    out->narrow_tests = (int64_t)h.narrow_tests;
    out->node_tests = (int64_t)h.node_tests;
    out->leaf_pairs = (int64_t)h.leaf_pairs;
    out->band = (int64_t)h.band;
    out->retries = 0;
  }
  return TRILENS_OK;
}

int trilens_collide_batch(const trilens_beam *a, const trilens_beam *b, const trilens_params *p,
                          int32_t n_inst, int64_t steps, double *yields, trilens_stream_t stream) {
  if (!yields) return TRILENS_ERR_INVALID;
  trilens_ctx *c = nullptr;
  int rc = trilens_batch_create(&c, a, b, n_inst, p, stream);
  if (rc) return rc;
  rc = trilens_batch_run(c, 0, steps, yields);
  trilens_destroy(c);
  return rc;
}

// ---- tuning ---------------------------------------------------------------

static int apply_tuning(trilens_ctx *c, int bucket, int depth, int warps, int budget) {
  if (bucket < 1 || bucket > 32 || depth < 64 || depth > 4096 || warps < 1 ||
      warps > TL_TRAV_MAX_WARPS ||
      budget < 0)
    return fail(c, TRILENS_ERR_INVALID, "tuning out of range");
  int bps = 0;
  CK(tl::traverse_config(c->p.precision == TRILENS_FP64, warps, depth, &bps));
  if (bps < 1) return fail(c, TRILENS_ERR_INVALID, "traversal shape does not fit an SM");
  c->p.leaf_bucket = bucket;
  c->p.stack_depth = depth;
  c->p.block_shape = warps;
  c->trav_warps = warps;
  c->trav_blocks = bps * c->n_sm;
  c->budget = budget;
  if (c->full_ready) {
    const unsigned long long warps_now = (unsigned long long)c->trav_blocks * c->trav_warps;
    if (warps_now > c->spill_warps) {
      const int rcs = alloc_spill(c, c->spill_per_warp, warps_now);
      if (rcs) return rcs;
    }
    const unsigned long long need_queue = 2ull * warps_now * (unsigned long long)depth;
    if (need_queue > c->queue_cap) {
      const int rcq = alloc_queue(c, need_queue);
      if (rcq) return rcq;
    }
  }
  drop_run(c);  // a captured run holds the old shapes
  c->built_step = c->exact_step = c->full_step = -1;  // the leaf bucket changes the hierarchy
  return TRILENS_OK;
}

int trilens_set_tuning(trilens_ctx *c, int32_t leaf_bucket, int32_t stack_depth,
                       int32_t block_shape, int32_t budget) {
  if (!c) return TRILENS_ERR_INVALID;
  CK(cudaSetDevice(c->device));
  return apply_tuning(c, leaf_bucket, stack_depth, block_shape, budget);
}

int trilens_get_tuning(trilens_ctx *c, int32_t out[4]) {
  if (!c || !out) return TRILENS_ERR_INVALID;
  out[0] = c->p.leaf_bucket;
  out[1] = c->p.stack_depth;
  out[2] = c->p.block_shape;
  out[3] = c->budget;
  return TRILENS_OK;
}

// key of a configuration class: sizes rounded to powers of two, precision, SM count, and
// the level and leaf bucket of a context that uses the statistical regime
static void tuning_key(trilens_ctx *c, char *key, size_t len) {
  int la = 0, lb = 0;
  while ((1ll << la) < std::max<int64_t>(c->beam[0].n, 1)) ++la;
  while ((1ll << lb) < std::max<int64_t>(c->beam[1].n, 1)) ++lb;
  const int at = snprintf(key, len, "nA2^%d_nB2^%d_inst%d_prec%d_sm%d", la, lb, c->n_inst,
                          c->p.precision, c->n_sm);
  if (surrogate_level(c) >= 0)
    snprintf(key + at, len - at, "_L%d_b%d", surrogate_level(c), c->p.leaf_bucket);
}

static bool cache_lookup(const char *path, const char *key, int v[4]) {
  if (!path) return false;
  FILE *f = fopen(path, "r");
  if (!f) return false;
  char line[512];
  bool found = false;
  while (!found && fgets(line, sizeof(line), f)) {
    char k[256];
    int a, b, cc, d;
    if (sscanf(line, " {\"key\": \"%255[^\"]\", \"leaf_bucket\": %d, \"stack_depth\": %d, "
                     "\"block_shape\": %d, \"budget\": %d", k, &a, &b, &cc, &d) == 5 &&
        strcmp(k, key) == 0) {
      v[0] = a; v[1] = b; v[2] = cc; v[3] = d;
      found = true;
    }
  }
  fclose(f);
  return found;
}

static void cache_store(const char *path, const char *key, const int v[4], double ms) {
  if (!path) return;
  // keep the other keys' lines, replace this key's
  std::vector<std::string> keep;
  if (FILE *f = fopen(path, "r")) {
    char line[512];
    while (fgets(line, sizeof(line), f)) {
      std::string l(line);
      if (l.find("\"key\"") != std::string::npos &&
          l.find(std::string("\"") + key + "\"") == std::string::npos) {
        while (!l.empty() && (l.back() == '\n' || l.back() == ',')) l.pop_back();
        keep.push_back(l);
      }
    }
    fclose(f);
  }
  char mine[512];
  snprintf(mine, sizeof(mine),
           " {\"key\": \"%s\", \"leaf_bucket\": %d, \"stack_depth\": %d, \"block_shape\": %d, "
           "\"budget\": %d, \"ms\": %.4f}",
           key, v[0], v[1], v[2], v[3], ms);
  keep.push_back(mine);
  std::string tmp = std::string(path) + ".tmp";
  FILE *f = fopen(tmp.c_str(), "w");
  if (!f) return;
  fprintf(f, "[\n");
  for (size_t i = 0; i < keep.size(); ++i)
    fprintf(f, "%s%s\n", keep[i].c_str(), i + 1 < keep.size() ? "," : "");
  fprintf(f, "]\n");
  fclose(f);
  rename(tmp.c_str(), path);
}

// The time of the sample steps with the current knobs: of what they act on, the seeded
// traversal of the steps' cut pairs, where the context uses the statistical regime, else of
// build + collide.  The faster of two passes (one is noisy enough to flip close choices).
static int time_steps(trilens_ctx *c, const int64_t *steps, int n, double *ms) {
  const bool seeded = surrogate_level(c) >= 0;
  cudaEvent_t e0, e1;
  CK(cudaEventCreate(&e0));
  CK(cudaEventCreate(&e1));
  const double keep_count = c->tot_count, keep_w = c->tot_weighted;
  double best = 1e30;
  for (int rep = 0; rep < 2; ++rep) {
    double sum = 0.0;
    CK(cudaEventRecord(e0, c->stream));
    for (int i = 0; i < n; ++i) {
      float f = 0.f;
      int rc = seeded ? surrogate_time_step(c, steps[i], &f) : trilens_build(c, steps[i]);
      if (!rc && !seeded) rc = trilens_collide_step(c, steps[i], nullptr, 0, nullptr);
      if (rc) {
        cudaEventDestroy(e0);
        cudaEventDestroy(e1);
        return rc;
      }
      sum += (double)f;
    }
    CK(cudaEventRecord(e1, c->stream));
    CK(cudaEventSynchronize(e1));
    float f = 0.f;
    CK(cudaEventElapsedTime(&f, e0, e1));
    best = std::min(best, seeded ? sum : (double)f);
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  c->tot_count = keep_count;  // tuning runs do not count towards the yield
  c->tot_weighted = keep_w;
  *ms = best;
  return TRILENS_OK;
}

int trilens_autotune(trilens_ctx *c, const int64_t *steps, int32_t n_steps,
                     const char *cache_path, int32_t chosen[4]) {
  if (!c || !steps || n_steps < 1) return TRILENS_ERR_INVALID;
  CK(cudaSetDevice(c->device));
  char key[160];
  tuning_key(c, key, sizeof(key));
  const int bucket = c->p.leaf_bucket;  // kept: it says what a cloud is (and is not a matter of time)
  int v[4];
  if (cache_lookup(cache_path, key, v)) {
    v[0] = bucket;
    int rc = apply_tuning(c, v[0], v[1], v[2], v[3]);
    if (rc) return rc;
    if (chosen)
      for (int i = 0; i < 4; ++i) chosen[i] = v[i];
    return TRILENS_OK;
  }
  // coordinate descent over the seeded traversal's knobs, each swept with the others
  // fixed at the best so far (stack depth first: a shallow stack moves work
  // to the spill areas, which would bias the other sweeps); results never
  // depend on them, only time does.  Where nothing they act on is used, the current ones stay.
  int best[4] = {bucket, c->p.stack_depth, c->p.block_shape, c->budget};
  static const int cand[4][4] = {{0, 0, 0, 0}, {256, 512, 1024, 0}, {2, 4, 8, 0}, {8, 16, 32, 64}};
  double best_ms = 1e30;
  int rc = apply_tuning(c, best[0], best[1], best[2], best[3]);
  if (rc) return rc;
  if ((rc = time_steps(c, steps, n_steps, &best_ms))) return rc;  // warm-up
  if ((rc = time_steps(c, steps, n_steps, &best_ms))) return rc;
  for (int knob = 1; knob < 4 && surrogate_level(c) >= 0; ++knob) {
    for (int j = 0; j < 4 && cand[knob][j]; ++j) {
      int t[4] = {best[0], best[1], best[2], best[3]};
      t[knob] = cand[knob][j];
      if (t[knob] == best[knob]) continue;
      if ((rc = apply_tuning(c, t[0], t[1], t[2], t[3]))) continue;  // shape does not fit
      double ms = 0;
      if ((rc = time_steps(c, steps, n_steps, &ms))) return rc;
      if (ms < best_ms) {
        best_ms = ms;
        for (int i = 0; i < 4; ++i) best[i] = t[i];
      }
    }
  }
  if ((rc = apply_tuning(c, best[0], best[1], best[2], best[3]))) return rc;
  cache_store(cache_path, key, best, best_ms);
  if (chosen)
    for (int i = 0; i < 4; ++i) chosen[i] = best[i];
  return TRILENS_OK;
}

int trilens_pair_products(const trilens_beam *a, const trilens_beam *b, const uint32_t *hits,
                          int64_t n_hits, uint64_t seed, double *out, trilens_stream_t stream) {
  if (!beam_ok(a) || !beam_ok(b) || n_hits < 0 || n_hits >= (1ll << 40)) return TRILENS_ERR_INVALID;
  if (n_hits == 0) return TRILENS_OK;
  if (!hits || !out || a->n == 0 || b->n == 0) return TRILENS_ERR_INVALID;
  TLBeam ta, tb;
  const trilens_beam *bs[2] = {a, b};
  TLBeam *ts[2] = {&ta, &tb};
  for (int k = 0; k < 2; ++k) {
    TLBeam &t = *ts[k];
    t.n = bs[k]->n;
    t.px = bs[k]->px; t.py = bs[k]->py; t.pz = bs[k]->pz;
    t.dx = bs[k]->dx; t.dy = bs[k]->dy; t.dz = bs[k]->dz;
    t.E = bs[k]->E; t.w = bs[k]->w;
  }
  if (tl::launch_pair_products(ta, tb, hits, n_hits, (unsigned long long)seed, out,
                               (cudaStream_t)stream) != cudaSuccess)
    return TRILENS_ERR_CUDA;
  return TRILENS_OK;
}

int trilens_step_stats_get(trilens_ctx *c, trilens_step_stats *out) {
  if (!c || !out) return TRILENS_ERR_INVALID;
  *out = c->last;
  return TRILENS_OK;
}

int trilens_yield(trilens_ctx *c, int32_t mode, int32_t level_L, double *count,
                  double *weighted) {
  if (!c || !count || !weighted) return TRILENS_ERR_INVALID;
  if (mode == TRILENS_YIELD_SURROGATE) {
    *count = -1.0;
    return surrogate_total(c, level_L, weighted);
  }
  if (mode != TRILENS_YIELD_EXACT) return fail(c, TRILENS_ERR_INVALID, "yield mode %d", mode);
  *count = c->tot_count;
  *weighted = c->tot_weighted;
  return TRILENS_OK;
}

int trilens_reset_yield(trilens_ctx *c) {
  if (!c) return TRILENS_ERR_INVALID;
  c->tot_count = 0;
  c->tot_weighted = 0;
  return TRILENS_OK;
}

// Test hook (not in the public header): make the first tile of the next
// builds' first sort pass withhold its published counts so that the next tile's
// bounded wait expires.  Used to check that an expired wait becomes
// TRILENS_ERR_TIMEOUT instead of a hang.
int trilens_debug_stall_sort(trilens_ctx *c, int on) {
  if (!c) return TRILENS_ERR_INVALID;
  drop_run(c);  // a captured run holds the old setting
  c->debug_stall_sort = on;
  return TRILENS_OK;
}

int trilens_debug_timing(trilens_ctx *c, int on) {
  if (!c) return TRILENS_ERR_INVALID;
  CK(cudaSetDevice(c->device));
  if (on && !c->ev[0][0][0])
    for (int ph = 0; ph < PH_COUNT; ++ph)
      for (int k = 0; k < 2; ++k)
        for (int e = 0; e < 2; ++e) CK(cudaEventCreate(&c->ev[ph][k][e]));
  c->timing = on ? 1 : 0;
  return TRILENS_OK;
}

int trilens_debug_phase_ms(trilens_ctx *c, double *out, int64_t *launches, int reset) {
  if (!c) return TRILENS_ERR_INVALID;
  for (int ph = 0; ph < PH_COUNT; ++ph) {
    if (out) out[ph] = c->phase_ms[ph];
    if (launches) launches[ph] = c->phase_launches[ph];
    if (reset) {
      c->phase_ms[ph] = 0.0;
      c->phase_launches[ph] = 0;
    }
  }
  return TRILENS_OK;
}

int trilens_debug_set_parts(trilens_ctx *c, int32_t parts) {
  if (!c || parts < 1 || parts > 4096) return TRILENS_ERR_INVALID;
  c->parts = parts;
  drop_run(c);  // a captured run holds the old part count
  return TRILENS_OK;
}

int trilens_debug_captures(trilens_ctx *c, int64_t *n) {
  if (!c || !n) return TRILENS_ERR_INVALID;
  *n = c->g_captures;
  return TRILENS_OK;
}

int trilens_debug_needles(trilens_ctx *c, int32_t *on) {
  if (!c || !on || c->exact_step < 0) return TRILENS_ERR_INVALID;
  *on = c->needles ? 1 : 0;
  return TRILENS_OK;
}

int trilens_debug_set_spin_limit(trilens_ctx *c, int64_t limit) {
  if (!c || limit < 1) return TRILENS_ERR_INVALID;
  drop_run(c);  // a captured run holds the old limit
  c->p.spin_limit = limit;
  return TRILENS_OK;
}

int trilens_debug_shrink_buffers(trilens_ctx *c, int64_t cap) {
  if (!c || cap < 1) return TRILENS_ERR_INVALID;
  CK(cudaSetDevice(c->device));
  CK(cudaStreamSynchronize(c->stream));
  drop_run(c);  // a captured run holds the old buffers
  const unsigned long long n = (unsigned long long)cap;
  cudaFree(c->hits);
  cudaFree(c->band);
  cudaFree(c->leaves);
  c->hits = c->band = c->leaves = nullptr;
  c->hit_cap = c->band_cap = c->leaf_cap = n;
  CK(dalloc(&c->hits, n));
  CK(dalloc(&c->band, n));
  CK(dalloc(&c->leaves, n));
  if (c->full_ready) {  // spill areas of cap entries per warp (at least 64), and the queue
    const int rcs = alloc_spill(c, (unsigned)std::max<int64_t>(64, std::min<int64_t>(cap, 1 << 20)),
                                c->spill_warps);
    if (rcs) return rcs;
    const int rc = alloc_queue(c, n);
    if (rc) return rc;
  }
  CK(cudaStreamSynchronize(c->stream));
  return TRILENS_OK;
}

int trilens_debug_set_key_bits(trilens_ctx *c, int32_t bits) {
  if (!c || c->n_inst > 1 || bits < 4 || bits > 21) return TRILENS_ERR_INVALID;
  for (int k = 0; k < 2; ++k) {
    c->bits[k] = bits;
    c->key_bits[k] = 3 * bits;
    c->w[k].key_bits = c->key_bits[k];
  }
  for (int k = 0; k < 2; ++k)  // at most what the cells are allocated for
    c->order_bits[k] = std::min(order_bits_for(c->beam[k].n), 3 * bits);
  drop_run(c);  // a captured run holds the old pass count
  c->built_step = c->exact_step = c->full_step = -1;
  return TRILENS_OK;
}

// There are no seed lists any more: the exact path descends one tree from its top.
int trilens_debug_set_cut_cap(trilens_ctx *c, int32_t) {
  return c ? TRILENS_OK : TRILENS_ERR_INVALID;
}

}  // extern "C"
