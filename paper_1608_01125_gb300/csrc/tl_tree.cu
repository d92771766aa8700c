// tl_tree.cu -- the exact path: order, trees and collisions of a step.
//
// Both beams are propagated and ordered by the cells of a Hilbert curve (k_order,
// k_cell_scan, k_place: one counting sort).
// The smaller beam (the tree's) gets a packed tree over its sorted photons with 32
// children per node (as in Kamel and Faloutsos, "Hilbert R-tree", VLDB 1994: leaves
// are runs of the curve, so there are no links to build): k_boxes writes every
// photon's swept box (in dense steps its needle, tl_frame.cuh) and the boxes of levels 1
// and 2, k_upper those above.  The other
// beam needs no tree: k_collide descends the tree with 32 of its consecutive photons
// at a time, one per lane, and gives the photon pairs whose boxes overlap the first
// look of the narrow phase; k_decide decides what that leaves.
#include "tl_common.cuh"
#include "tl_exact.cuh"
#include "tl_frame.cuh"
#include "tl_narrow.cuh"
#include "tl_tree.h"
#include "tl_warp.cuh"

namespace tl {

// ---------------------------------------------------------------- frames and grids

// Sums of d, ln E and ln^2 E over up to kSample photons of a beam, evenly spaced (5 FP64
// values per block, added by the host): the beam's mean direction, for the choice of the
// frame, and its typical energy, for the pads.
constexpr int kSampleBlocks = 64, kSample = 65536;

__device__ __forceinline__ float ln_energy(double E) {
  return logf(fminf(fmaxf((float)E, 1e-18f), 1e18f));
}

__global__ void __launch_bounds__(256) k_mean_dir(TLBeam b, double *part) {
  __shared__ double sm[8][5];
  const int64_t n = b.n < kSample ? b.n : kSample;
  double m[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
  for (int64_t t = blockIdx.x * 256 + threadIdx.x; t < n; t += kSampleBlocks * 256) {
    const int64_t i = t * b.n / n;
    m[0] += b.dx[i];
    m[1] += b.dy[i];
    m[2] += b.dz[i];
    const double le = (double)ln_energy(b.E[i]);
    m[3] += le;
    m[4] += le * le;
  }
  for (int q = 0; q < 5; ++q)
    for (int off = 16; off; off >>= 1) m[q] += __shfl_xor_sync(0xffffffffu, m[q], off);
  if ((threadIdx.x & 31) == 0)
    for (int q = 0; q < 5; ++q) sm[threadIdx.x >> 5][q] = m[q];
  __syncthreads();
  if (threadIdx.x < 5) {
    double t = 0.0;
    for (int w = 0; w < 8; ++w) t += sm[w][threadIdx.x];
    part[blockIdx.x * 5 + threadIdx.x] = t;
  }
}

int mean_doubles() { return 5 * kSampleBlocks; }
int64_t mean_count(int64_t n) { return n < kSample ? n : kSample; }

cudaError_t launch_mean_dir(const TLBeam &b, double *part, cudaStream_t s) {
  k_mean_dir<<<kSampleBlocks, 256, 0, s>>>(b, part);
  return cudaGetLastError();
}

// Per-axis sums of p', d', p'^2, p' d', d'^2 with p' = R p0, d' = R d (15 FP64 values),
// in a fixed order (per-block sums, then one block over the blocks), from which the means
// and variances of the swept boxes' centres follow in closed form for every step; and the
// extremes of p' and d' and the largest |p0|_1 and |d|_1 (FP32; tl_beam_box takes their
// rounding into account), 14 more values.
constexpr int kMomentBlocks = 4 * 152, kMom = 29;

__device__ __forceinline__ void turn(const TLFrame &f, double v[3]) {
  if (f.ident) return;
  const double x = v[0], y = v[1], z = v[2];
  for (int k = 0; k < 3; ++k)
    v[k] = (double)f.r[3 * k] * x + (double)f.r[3 * k + 1] * y + (double)f.r[3 * k + 2] * z;
}

// value q of two partial results joined: sums, then 6 minima, 6 maxima, 2 maxima
__device__ __forceinline__ double mom_join(int q, double a, double b) {
  return q < 15 ? a + b : (q < 21 ? fmin(a, b) : fmax(a, b));
}

__global__ void __launch_bounds__(256) k_beam_moments(TLBeam b, TLFrame f, double *part) {
  double m[15];
  float e[14];
  const float inf = __int_as_float(0x7f800000);
  for (int q = 0; q < 15; ++q) m[q] = 0.0;
  for (int q = 0; q < 14; ++q) e[q] = q < 6 ? inf : -inf;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < b.n;
       i += (int64_t)gridDim.x * blockDim.x) {
    double p[3] = {b.px[i], b.py[i], b.pz[i]}, d[3] = {b.dx[i], b.dy[i], b.dz[i]};
    e[12] = fmaxf(e[12], fabsf((float)p[0]) + fabsf((float)p[1]) + fabsf((float)p[2]));
    e[13] = fmaxf(e[13], fabsf((float)d[0]) + fabsf((float)d[1]) + fabsf((float)d[2]));
    turn(f, p);
    turn(f, d);
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      m[a] += p[a];
      m[3 + a] += d[a];
      m[6 + a] += p[a] * p[a];
      m[9 + a] += p[a] * d[a];
      m[12 + a] += d[a] * d[a];
      const float pf = (float)p[a], df = (float)d[a];
      e[a] = fminf(e[a], pf);  // (a photon at NaN meets nothing)
      e[3 + a] = fminf(e[3 + a], df);
      e[6 + a] = fmaxf(e[6 + a], pf);
      e[9 + a] = fmaxf(e[9 + a], df);
    }
  }
  __shared__ double sm[8][kMom];
  double v[kMom];
#pragma unroll
  for (int q = 0; q < kMom; ++q) {
    v[q] = q < 15 ? m[q] : (double)e[q - 15];
    for (int off = 16; off; off >>= 1)
      v[q] = mom_join(q, v[q], __shfl_xor_sync(0xffffffffu, v[q], off));
  }
  if ((threadIdx.x & 31) == 0)
#pragma unroll
    for (int q = 0; q < kMom; ++q) sm[threadIdx.x >> 5][q] = v[q];
  __syncthreads();
  if (threadIdx.x < kMom) {
    double t = sm[0][threadIdx.x];
    for (int w8 = 1; w8 < 8; ++w8) t = mom_join(threadIdx.x, t, sm[w8][threadIdx.x]);
    part[blockIdx.x * kMom + threadIdx.x] = t;
  }
}

__global__ void k_beam_moments_final(const double *part, int nparts, double *out) {
  if (threadIdx.x < kMom) {
    double t = part[threadIdx.x];
    for (int k = 1; k < nparts; ++k) t = mom_join(threadIdx.x, t, part[k * kMom + threadIdx.x]);
    out[threadIdx.x] = t;
  }
}

size_t moment_doubles() { return kMom * (1 + kMomentBlocks); }

// out: device, moment_doubles() doubles, the 29 values first
cudaError_t launch_beam_moments(const TLBeam &b, const TLFrame &f, double *out, cudaStream_t s) {
  const int64_t nb = (b.n + 255) / 256;
  const int blocks = (int)(nb < 1 ? 1 : (nb < kMomentBlocks ? nb : kMomentBlocks));
  k_beam_moments<<<blocks, 256, 0, s>>>(b, f, out + kMom);
  k_beam_moments_final<<<1, 32, 0, s>>>(out + kMom, blocks, out);
  return cudaGetLastError();
}

__device__ __forceinline__ long long ord64(double x) {
  long long i = __double_as_longlong(x);
  return i >= 0 ? i : i ^ 0x7fffffffffffffffLL;
}

// Per-instance min and max of R p0 and R d (12 ordered int64 per instance, laid out as
// p' min xyz, d' min xyz, p' max xyz, d' max xyz; frames NULL: of p0 and d).  A warp
// whose lanes share one instance reduces first and issues one atomic per quantity.
__global__ void k_inst_bounds(TLBeam b, const uint32_t *inst_of, const TLFrame *frames,
                              long long *out) {
  const int lane = threadIdx.x & 31;
  for (int64_t i0 = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) & ~31ll; i0 < b.n;
       i0 += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = i0 + lane;
    const bool valid = i < b.n;
    const uint32_t q = valid ? inst_of[i] : 0xffffffffu;
    const uint32_t q0 = __shfl_sync(0xffffffffu, q, 0);
    const bool uniform = __all_sync(0xffffffffu, !valid || q == q0);
    long long v[12];
    if (valid) {
      double x[6] = {b.px[i], b.py[i], b.pz[i], b.dx[i], b.dy[i], b.dz[i]};
      if (frames) {
        turn(frames[q], x);
        turn(frames[q], x + 3);
      }
      for (int c = 0; c < 6; ++c) v[c] = v[6 + c] = ord64(x[c]);
    } else {
      for (int c = 0; c < 6; ++c) {
        v[c] = 0x7fffffffffffffffLL;
        v[6 + c] = -0x7fffffffffffffffLL - 1;
      }
    }
    if (uniform) {
      for (int c = 0; c < 6; ++c)
        for (int off = 16; off; off >>= 1) {
          v[c] = min(v[c], __shfl_xor_sync(0xffffffffu, v[c], off));
          v[6 + c] = max(v[6 + c], __shfl_xor_sync(0xffffffffu, v[6 + c], off));
        }
      if (lane == 0)
        for (int c = 0; c < 6; ++c) {
          atomicMin(&out[12 * (size_t)q0 + c], v[c]);
          atomicMax(&out[12 * (size_t)q0 + 6 + c], v[6 + c]);
        }
    } else if (valid) {
      for (int c = 0; c < 6; ++c) {
        atomicMin(&out[12 * (size_t)q + c], v[c]);
        atomicMax(&out[12 * (size_t)q + 6 + c], v[6 + c]);
      }
    }
  }
}

__global__ void k_inst_bounds_init(long long *out, int n_inst) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t < 12 * n_inst) out[t] = (t % 12) < 6 ? 0x7fffffffffffffffLL : -0x7fffffffffffffffLL - 1;
}

__global__ void k_inst_bounds_decode(const long long *in, double *out, int n_inst) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t < 12 * n_inst) {
    long long i = in[t];
    i = i >= 0 ? i : i ^ 0x7fffffffffffffffLL;
    out[t] = __longlong_as_double(i);
  }
}

cudaError_t launch_inst_bounds(const TLBeam &b, const uint32_t *inst_of, const TLFrame *frames,
                               int n_inst, long long *tmp, double *out, cudaStream_t s) {
  const int nt = 12 * n_inst;
  k_inst_bounds_init<<<(nt + 255) / 256, 256, 0, s>>>(tmp, n_inst);
  if (b.n > 0) {
    int64_t nb = (b.n + 255) / 256;
    k_inst_bounds<<<(int)(nb < 4096 ? nb : 4096), 256, 0, s>>>(b, inst_of, frames, tmp);
  }
  k_inst_bounds_decode<<<(nt + 255) / 256, 256, 0, s>>>(tmp, out, n_inst);
  return cudaGetLastError();
}

// Mean and standard deviation of ln E over up to 1024 photons, evenly spaced, of every
// instance of a beam: a block each.
__global__ void __launch_bounds__(256) k_inst_energy(const double *E, const TLInst *inst,
                                                     double *out) {
  __shared__ double sm[8][2];
  const TLInst &I = inst[blockIdx.x];
  const int n = min(I.n, 1024);
  double m[2] = {0.0, 0.0};
  for (int t = threadIdx.x; t < n; t += 256) {
    const double le = (double)ln_energy(E[I.first + (int64_t)t * I.n / n]);
    m[0] += le;
    m[1] += le * le;
  }
  for (int q = 0; q < 2; ++q) {
    for (int off = 16; off; off >>= 1) m[q] += __shfl_xor_sync(0xffffffffu, m[q], off);
    if ((threadIdx.x & 31) == 0) sm[threadIdx.x >> 5][q] = m[q];
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < 8; ++w)
      for (int q = 0; q < 2; ++q) sm[0][q] += sm[w][q];
    const double mean = sm[0][0] / max(n, 1);
    out[2 * blockIdx.x] = mean;
    out[2 * blockIdx.x + 1] = sqrt(fmax(sm[0][1] / max(n, 1) - mean * mean, 0.0));
  }
}

cudaError_t launch_inst_energy(const TLBeam &b, const TLInst *inst, int n_inst, double *out,
                               cudaStream_t s) {
  k_inst_energy<<<n_inst, 256, 0, s>>>(b.E, inst, out);
  return cudaGetLastError();
}

// Frames of a batch's instances, from the middle of each beam's range of directions, and
// their pads; le: mean and standard deviation of ln E of either beam.
__global__ void k_inst_frames(const double *ba, const double *bb, const double *lea,
                              const double *leb, TLPadTable pads, double half, int n_inst,
                              TLFrame *out) {
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= n_inst) return;
  double a[3], b[3];
  for (int k = 0; k < 3; ++k) {
    a[k] = 0.5 * (ba[12 * q + 3 + k] + ba[12 * q + 9 + k]);
    b[k] = 0.5 * (bb[12 * q + 3 + k] + bb[12 * q + 9 + k]);
  }
  TLFrame f = tl_make_frame(a, b);  // an empty beam's bounds are NaN or infinite: the lab frame
  tl_set_pads(f, pads, ba + 12 * q, bb + 12 * q, lea + 2 * q, leb + 2 * q, half);
  out[q] = f;
}

cudaError_t launch_inst_frames(const double *ba, const double *bb, const double *lea,
                               const double *leb, const TLPadTable &pads, double half, int n_inst,
                               TLFrame *out, cudaStream_t s) {
  k_inst_frames<<<(n_inst + 127) / 128, 128, 0, s>>>(ba, bb, lea, leb, pads, half, n_inst, out);
  return cudaGetLastError();
}

// Ordering grids of both beams of a batch's instances for the step with travel
// T = c t_k + L / 2 to the swept boxes' centres: the range of the centres, and cells in
// the proportions of the boxes' extents (pad + travel of a typical photon).
__global__ void k_inst_grid(const double *ba, const double *bb, const TLFrame *frames,
                            const TLInst *ia, const TLInst *ib, int n_inst, double T, double L,
                            double half, TLGrid *ga, TLGrid *gb) {
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= n_inst) return;
  const TLFrame f = frames[q];
  const double *bd[2] = {ba + 12 * (size_t)q, bb + 12 * (size_t)q};
  double ru[3], s[3];
  for (int k = 0; k < 3; ++k) {
    ru[k] = (double)f.r[3 * k] * f.u[0] + (double)f.r[3 * k + 1] * f.u[1] +
            (double)f.r[3 * k + 2] * f.u[2];
    s[k] = 2.0 * f.typ;
    for (int h = 0; h < 2; ++h) {
      const double mean = 0.5 * (bd[h][3 + k] + bd[h][9 + k]) - ru[k];
      const double sd = 0.125 * (bd[h][9 + k] - bd[h][3 + k]);
      s[k] += L * sqrt(mean * mean + sd * sd);
    }
  }
  for (int h = 0; h < 2; ++h) {
    double lo[3], range[3];
    for (int k = 0; k < 3; ++k) {
      lo[k] = bd[h][k] + T * bd[h][3 + k] - 0.5 * L * ru[k];
      range[k] = bd[h][6 + k] + T * bd[h][9 + k] - 0.5 * L * ru[k] - lo[k];
    }
    TLGrid g = tl_make_grid(lo, range, s, (h ? ib : ia)[q].bits);
    tl_beam_box(bd[1 - h], 0.0, 0.0, f, T - 0.5 * L, L, half, g.clo, g.chi);
    (h ? gb : ga)[q] = g;
  }
}

cudaError_t launch_inst_grid(const double *ba, const double *bb, const TLFrame *frames,
                             const TLInst *ia, const TLInst *ib, int n_inst, double T, double L,
                             double half, TLGrid *ga, TLGrid *gb, cudaStream_t s) {
  k_inst_grid<<<(n_inst + 127) / 128, 128, 0, s>>>(ba, bb, frames, ia, ib, n_inst, T, L, half, ga,
                                                   gb);
  return cudaGetLastError();
}

// Concatenate the instances' input arrays into one beam and record the
// instance of every photon.
__global__ void k_gather_instances(const InstSrc *src, int n_inst, int64_t n, double *const *dst,
                                   uint32_t *inst_of) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= n) return;
  int lo = 0, hi = n_inst - 1;  // last instance whose offset <= i
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (src[mid].off <= i) lo = mid;
    else hi = mid - 1;
  }
  const InstSrc &s = src[lo];
  const int64_t j = i - s.off;
  for (int k = 0; k < 8; ++k) dst[k][i] = s.p[k] ? s.p[k][j] : 1.0;
  inst_of[i] = (uint32_t)lo;
}

cudaError_t launch_gather_instances(const InstSrc *src, int n_inst, int64_t n, double *const *dst,
                                    uint32_t *inst_of, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  k_gather_instances<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(src, n_inst, n, dst, inst_of);
  return cudaGetLastError();
}

// ---------------------------------------------------------------- order

// The step-invariant FP32 record of every photon, once per context: p0 and energy,
// direction and index.
__global__ void __launch_bounds__(256) k_static(TLBeam b, float4 *stat) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < b.n;
       i += (int64_t)gridDim.x * blockDim.x) {
    stat[2 * i] = make_float4(__double2float_rn(b.px[i]), __double2float_rn(b.py[i]),
                              __double2float_rn(b.pz[i]), __double2float_rn(b.E[i]));
    stat[2 * i + 1] = make_float4(__double2float_rn(b.dx[i]), __double2float_rn(b.dy[i]),
                                  __double2float_rn(b.dz[i]), __int_as_float((int)i));
  }
}

cudaError_t launch_static(const TLBeam &b, float4 *stat, cudaStream_t s) {
  if (b.n <= 0) return cudaSuccess;
  const int64_t nb = (b.n + 255) / 256;
  k_static<<<(unsigned)(nb < 8 * 152 ? nb : 8 * 152), 256, 0, s>>>(b, stat);
  return cudaGetLastError();
}

// Every photon's cell, from its swept box's centre in the frame (FP32), counted there:
// the count it finds is its rank in the cell.  With the cells' running sum that is its
// place, so a beam is ordered by one counting sort with 2 to 4 cells per photon, half a cell
// for beams beyond 16M photons (three or four radix passes took 29 us each for 1M photons;
// the scan takes 13 us, the move 30).
// The order inside a cell is that of the atomics and changes from run to run; it shapes
// the tree and nothing else.  A photon whose swept box misses the box of the whole other
// beam is left out of the step here: its 32 bytes are all that is read of it.  The test
// takes 2^-20 of the sums of the lengths involved for the rounding of the FP32 record
// and arithmetic (16u; 8u bound it).  Bound by memory: 32 bytes in, 8 out, one atomic
// per photon; a warp whose photons share one cell adds once, so that a beam on one point
// does not queue at one word.
constexpr int kOrderBlocks = 8 * 152;

__global__ void __launch_bounds__(256) k_order(OrderArgs a) {
  const int64_t gtid = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  for (int64_t t = gtid; t < a.scan_tiles + 1; t += (int64_t)gridDim.x * blockDim.x)
    a.scan_st[t] = 0u;
  const int lane = threadIdx.x & 31;
  const int64_t nround = (a.n + 31) & ~(int64_t)31;
  for (int64_t i = gtid; i < nround; i += (int64_t)gridDim.x * blockDim.x) {
    uint32_t cell = TL_NONE;
    if (i < a.n) {
      const float4 p0 = a.stat[2 * i], d = a.stat[2 * i + 1];
      const uint32_t q = a.inst_of ? a.inst_of[i] : 0u;
      const TLFrame &f = a.frames[q];
      const TLGrid &g = a.inst_of ? a.grids[q] : a.grid;
      const float px = fmaf(a.ct, d.x, p0.x), py = fmaf(a.ct, d.y, p0.y),
                  pz = fmaf(a.ct, d.z, p0.z);
      const float d1 = fabsf(d.x) + fabsf(d.y) + fabsf(d.z);
      const float e = a.half + 0x1p-20f * (fabsf(p0.x) + fabsf(p0.y) + fabsf(p0.z) +
                                           fmaf(a.ct, d1, a.L * (d1 + 3.0f)));
      float x[3] = {px, py, pz}, v[3] = {d.x, d.y, d.z};
      if (!f.ident) {
        const float vx = d.x - f.u[0], vy = d.y - f.u[1], vz = d.z - f.u[2];
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          x[k] = fmaf(f.r[3 * k], px, fmaf(f.r[3 * k + 1], py, f.r[3 * k + 2] * pz));
          v[k] = fmaf(f.r[3 * k], vx, fmaf(f.r[3 * k + 1], vy, f.r[3 * k + 2] * vz));
        }
      }
      bool apart = false;
      float c[3];
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        const float t = a.L * v[k];
        apart = apart || x[k] + fminf(t, 0.0f) - e > g.chi[k] || x[k] + fmaxf(t, 0.0f) + e < g.clo[k];
        c[k] = fmaf(0.5f, t, x[k]);
      }
      if (!apart) cell = (a.inst_of ? a.inst[q].cell0 : 0u) + order_key(g, c);
    }
    const uint32_t c0 = __shfl_sync(0xffffffffu, cell, 0);
    uint32_t r = 0u;
    if (__all_sync(0xffffffffu, cell == c0)) {
      if (c0 != TL_NONE) {
        if (lane == 0) r = atomicAdd(a.count + c0, 32u);
        r = __shfl_sync(0xffffffffu, r, 0) + lane;
      }
    } else if (cell != TL_NONE) {
      r = atomicAdd(a.count + cell, 1u);
    }
    if (i < a.n) a.cell[i] = make_uint2(cell, r);
  }
}

cudaError_t launch_order(const OrderArgs &a, cudaStream_t s) {
  if (a.n <= 0) return cudaSuccess;
  const int64_t nb = (a.n + 255) / 256;
  k_order<<<(int)(nb < kOrderBlocks ? nb : kOrderBlocks), 256, 0, s>>>(a);
  return cudaGetLastError();
}

// Exclusive running sum of the cells' counts, tile by tile of kScanTile cells, with the
// counts cleared for the next step.  A tile's sum is published at once; warp 0 looks back
// over the preceding tiles' words 32 at a time (Merrill and Garland 2016, "Single-pass
// parallel prefix scan with decoupled look-back").  Tiles are numbered in the order blocks
// start, so a tile only waits on running ones; every wait is bounded by spin (then
// TL_ST_TIMEOUT is recorded and the sums are not used).  Words: 2 flag bits and a 28-bit
// sum (beams hold fewer than 2^27 photons), cleared by k_order.
constexpr int kScanThreads = 1024, kScanCells = 16, kScanTile = kScanThreads * kScanCells;
constexpr uint32_t kScanSum = 1u << 30, kScanPre = 2u << 30, kScanVal = (1u << 28) - 1u;

__global__ void __launch_bounds__(kScanThreads) k_cell_scan(uint32_t *count, uint32_t *start,
                                                            int64_t cells, uint32_t *st,
                                                            long long spin, int debug_stall,
                                                            unsigned *status) {
  __shared__ uint32_t ws[32], tile_s, before_s;
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  if (t == 0) tile_s = atomicAdd(st, 1u);
  __syncthreads();
  const uint32_t tile = tile_s;
  const int64_t c0 = (int64_t)tile * kScanTile + (int64_t)t * kScanCells;
  uint4 v[kScanCells / 4];
  uint32_t sum = 0u;
#pragma unroll
  for (int q = 0; q < kScanCells / 4; ++q) {  // (cells is a multiple of 16)
    uint4 *p = reinterpret_cast<uint4 *>(count + c0) + q;
    v[q] = c0 < cells ? *p : make_uint4(0u, 0u, 0u, 0u);
    if (c0 < cells) *p = make_uint4(0u, 0u, 0u, 0u);
    sum += v[q].x + v[q].y + v[q].z + v[q].w;
  }
  uint32_t inc = sum;
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const uint32_t u = __shfl_up_sync(0xffffffffu, inc, off);
    if (lane >= off) inc += u;
  }
  if (lane == 31) ws[warp] = inc;
  __syncthreads();
  if (warp == 0) {
    uint32_t w = ws[lane];
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const uint32_t u = __shfl_up_sync(0xffffffffu, w, off);
      if (lane >= off) w += u;
    }
    ws[lane] = w;  // inclusive sums of the warps
    const uint32_t total = __shfl_sync(0xffffffffu, w, 31);
    uint32_t *my = st + 1 + tile;
    uint32_t before = 0u;
    if (tile == 0) {
      if (lane == 0 && !debug_stall) atomicExch(my, kScanPre | total);
    } else {
      if (lane == 0) atomicExch(my, kScanSum | total);
      long long j = (long long)tile - 1, spins = 0;
      while (j >= 0) {  // lane l looks at tile j - l
        uint32_t w1 = kScanPre;
        if (j - lane >= 0) w1 = *(volatile uint32_t *)(st + 1 + j - lane);
        const unsigned none = __ballot_sync(0xffffffffu, (w1 >> 30) == 0u);
        const unsigned pre = __ballot_sync(0xffffffffu, (w1 >> 30) == 2u);
        // the words up to the first prefix, or up to the first one not published
        int use = none ? __ffs(none) - 1 : 32;
        const bool done = pre && __ffs(pre) - 1 < use;
        if (done) use = __ffs(pre);
        uint32_t x = lane < use ? w1 & kScanVal : 0u;
#pragma unroll
        for (int off = 16; off; off >>= 1) x += __shfl_xor_sync(0xffffffffu, x, off);
        before += x;
        if (done) break;
        j -= use;
        if (use == 0) {
          if (++spins > spin) {
            if (lane == 0) atomicOr(status, (unsigned)TL_ST_TIMEOUT);
            break;
          }
          __nanosleep(32);
        }
      }
      if (lane == 0) atomicExch(my, kScanPre | ((before + total) & kScanVal));
    }
    if (lane == 0) before_s = before;
  }
  __syncthreads();
  uint32_t run = before_s + (warp ? ws[warp - 1] : 0u) + inc - sum;
  if (c0 >= cells) return;
  if (c0 + kScanCells == cells) start[cells] = run + sum;  // the photons in all
#pragma unroll
  for (int q = 0; q < kScanCells / 4; ++q) {
    uint4 o;
    o.x = run;
    o.y = o.x + v[q].x;
    o.z = o.y + v[q].y;
    o.w = o.z + v[q].z;
    run = o.w + v[q].w;
    reinterpret_cast<uint4 *>(start + c0)[q] = o;
  }
}

int64_t scan_tiles(int64_t cells) { return (cells + kScanTile - 1) / kScanTile; }

cudaError_t launch_cell_scan(uint32_t *count, uint32_t *start, int64_t cells, uint32_t *st,
                             long long spin, int debug_stall, unsigned *status, cudaStream_t s) {
  k_cell_scan<<<(unsigned)scan_tiles(cells), kScanThreads, 0, s>>>(count, start, cells, st, spin,
                                                                   debug_stall, status);
  return cudaGetLastError();
}

// Every photon that stays in the step to its place, at its position of the step:
// p = p0 + c t_k d in FP64 (closed form), rounded to FP32.  Coalesced reads (88 bytes),
// one full 32-byte sector written per photon; beside that it keeps GB300's FP64 pipe
// busy (six operations and three conversions per photon at 2 per clock and SM).
__global__ void __launch_bounds__(256) k_place(PlaceArgs a) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const uint2 c = i < a.b.n ? a.cell[i] : make_uint2(TL_NONE, 0u);
  if (c.x != TL_NONE) {
    int64_t to = (int64_t)__ldg(a.start + c.x) + c.y;
    const float4 s0 = a.stat[2 * i], d = a.stat[2 * i + 1];
    const double dx = a.b.dx[i], dy = a.b.dy[i], dz = a.b.dz[i];
    const float4 p =
        make_float4(__double2float_rn(__dadd_rn(a.b.px[i], __dmul_rn(a.ct, dx))),
                    __double2float_rn(__dadd_rn(a.b.py[i], __dmul_rn(a.ct, dy))),
                    __double2float_rn(__dadd_rn(a.b.pz[i], __dmul_rn(a.ct, dz))), s0.w);
    if (a.inst_of) {
      const TLInst &I = a.inst[a.inst_of[i]];
      to += (int64_t)I.group0 * 32 - (int64_t)__ldg(a.start + I.cell0);
    }
    if ((uint64_t)to < (uint64_t)a.n_pad) {  // always, unless the scan's wait expired
      a.rec[2 * to] = p;
      a.rec[2 * to + 1] = d;
    }
  }
}

cudaError_t launch_place(const PlaceArgs &a, cudaStream_t s) {
  if (a.b.n <= 0) return cudaSuccess;
  const int64_t nb = (a.b.n + 255) / 256;
  // a block per 256 photons: a fixed grid of 8 per SM leaves SMs idle at its end (both
  // beams of 16M photons at 90 degrees: 3.69 ms a step with it, 3.45 without)
  k_place<<<(unsigned)nb, 256, 0, s>>>(a);
  return cudaGetLastError();
}

// ---------------------------------------------------------------- boxes

__device__ __forceinline__ TLBox empty_box() {
  const float inf = __int_as_float(0x7f800000);
  return TLBox{inf, inf, inf, -inf, -inf, -inf};  // overlaps nothing
}

__device__ __forceinline__ void join(TLBox &a, const TLBox &b) {
  a.lx = fminf(a.lx, b.lx);
  a.ly = fminf(a.ly, b.ly);
  a.lz = fminf(a.lz, b.lz);
  a.hx = fmaxf(a.hx, b.hx);
  a.hy = fmaxf(a.hy, b.hy);
  a.hz = fmaxf(a.hz, b.hz);
}

__device__ __forceinline__ TLBox warp_union(TLBox b) {
#pragma unroll
  for (int off = 16; off; off >>= 1) {
    TLBox o;
    o.lx = __shfl_xor_sync(0xffffffffu, b.lx, off);
    o.ly = __shfl_xor_sync(0xffffffffu, b.ly, off);
    o.lz = __shfl_xor_sync(0xffffffffu, b.lz, off);
    o.hx = __shfl_xor_sync(0xffffffffu, b.hx, off);
    o.hy = __shfl_xor_sync(0xffffffffu, b.hy, off);
    o.hz = __shfl_xor_sync(0xffffffffu, b.hz, off);
    join(b, o);
  }
  return b;
}

// a box is two float4: lo xyz, hi x | hi yz, 0, 0
__device__ __forceinline__ void put_box(float4 *dst, const TLBox &b) {
  dst[0] = make_float4(b.lx, b.ly, b.lz, b.hx);
  dst[1] = make_float4(b.hy, b.hz, 0.0f, 0.0f);
}
__device__ __forceinline__ TLBox get_box(const float4 *src) {
  const float4 a = src[0];
  const float2 c = *reinterpret_cast<const float2 *>(src + 1);
  return TLBox{a.x, a.y, a.z, a.w, c.x, c.y};
}

// a needle, likewise
__device__ __forceinline__ void put_needle(float4 *dst, const TLNeedle &n) {
  dst[0] = make_float4(n.x, n.y, n.w, n.vx);
  dst[1] = make_float4(n.vy, n.h, n.e, 0.0f);
}
__device__ __forceinline__ TLNeedle get_needle(const float4 *src) {
  const float4 a = src[0], b = src[1];
  return TLNeedle{a.x, a.y, a.z, a.w, b.x, b.y, b.z};
}
// never met: no time is within its window
__device__ __forceinline__ TLNeedle no_needle() {
  return TLNeedle{0.0f, 0.0f, __int_as_float(0x7f800000), 0.0f, 0.0f, 0.0f, 0.0f};
}

// One block per tile: every photon's swept box (its needle where the frame has a closing
// axis: the box then only goes into the unions), the boxes of the tile's 32 groups of 32
// photons (level 1) and, in an instance of more than one tile, the tile's own (level 2).  One
// pass over the sorted photons; unions by shuffles, no links and no second pass.  A warp finds
// its own instance: 65536 instances of 8 photons with a tile of 1024 each took 24.7 ms and
// 6.4 GB for 16 steps, with a group of 32 each 5.2 ms and 0.4 GB.
template <bool NEEDLES>
__global__ void __launch_bounds__(kTile) k_boxes(BoxArgs a) {
  __shared__ TLBox wb[32];
  if (*a.build_status & TL_ST_TIMEOUT) return;  // keys unsorted: the build is abandoned
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5, g = blockIdx.x * 32 + warp;
  const uint32_t q = a.group_inst ? a.group_inst[g] : 0u;
  const TLInst &I = a.inst[q];
  const int n = tl_live(I, a.start);
  const int k = g - I.group0, r = k * 32 + lane;
  const bool whole = I.n > kTile;  // the tile is one instance's (the same for all its warps)
  if (whole && (k & ~31) * 32 >= n) return;
  TLBox b = empty_box();
  if (r < n) {
    const int64_t p = (int64_t)g * 32 + lane;
    const float4 pe = a.rec[2 * p];
    const float4 de = a.rec[2 * p + 1];
    const TLFrame &f = a.frames[q];
    const float pad = tl_photon_pad(f, a.beam, pe.w, a.half);
    b = swept_box(pe, de, f, a.Llo, a.Lhi, pad);
    float4 *dst = a.box + 2 * ((size_t)I.lev[0] + r);
    if (!NEEDLES) put_box(dst, b);
    else put_needle(dst, tl_needle(f, a.beam, pe, de, pad));
  }
  b = warp_union(b);
  if (lane == 0) {
    wb[warp] = b;
    if (r < n) put_box(a.box + 2 * ((size_t)I.lev[1] + k), b);
  }
  if (!whole) return;
  __syncthreads();
  if (warp == 0) {
    b = warp_union(wb[lane]);
    if (lane == 0) put_box(a.box + 2 * ((size_t)I.lev[2] + (k >> 5)), b);
  }
}

// Levels 3 and up of one instance's tree per block, a warp per node.
__global__ void __launch_bounds__(1024) k_upper(const TLInst *inst, const uint32_t *start,
                                                float4 *box, const unsigned *build_status) {
  if (*build_status & TL_ST_TIMEOUT) return;  // (k_boxes has written nothing)
  const TLInst &I = inst[blockIdx.x];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int n = tl_live(I, start), top = tl_top_level(n);
  for (int l = 3; l <= top; ++l) {
    const int cnt = tl_level_count(n, l), below = tl_level_count(n, l - 1);
    for (int j = warp; j < cnt; j += 32) {
      const int c = 32 * j + lane;
      TLBox b = c < below ? get_box(box + 2 * ((size_t)I.lev[l - 1] + c)) : empty_box();
      b = warp_union(b);
      if (lane == 0) put_box(box + 2 * ((size_t)I.lev[l] + j), b);
    }
    __syncthreads();
  }
}

cudaError_t launch_boxes(const BoxArgs &a, int tiles, int n_inst, int max_top, cudaStream_t s) {
  if (tiles <= 0) return cudaSuccess;
  if (a.needles) k_boxes<true><<<tiles, kTile, 0, s>>>(a);
  else k_boxes<false><<<tiles, kTile, 0, s>>>(a);
  if (max_top >= 3) k_upper<<<n_inst, 1024, 0, s>>>(a.inst, a.start, a.box, a.build_status);
  return cudaGetLastError();
}

// ---------------------------------------------------------------- collisions

constexpr int kColWarps = 4;
constexpr uint32_t kIdxMask = (1u << 27) - 1u;  // beams hold fewer than 2^27 photons

constexpr int kPend = 256;

struct ColSmem {
  float4 qpos[32], qdir[32];  // the warp's photons
  float4 cbox[64];            // boxes tested by every lane
  uint32_t pend[kPend];       // (lane << 27 | photon of the tree): boxes overlap
  uint32_t cand[64];          // undecided by the first look
  uint32_t mask[6], base[6];  // per level: children still to descend into
  uint8_t id[32];             // lane of each tested box
};

// Photon pairs whose boxes overlap: the first look, 32 at a time, from the end of the
// pending list; what it leaves goes to the step's candidate list.
template <bool FP64>
struct Pairs {
  const ColArgs &a;
  ColSmem &ws;
  const float *suf;
  uint32_t qpos0, tpos0;  // padded position of the warp's first photon, of the tree's
  int lane, np, nc;
  unsigned long long lbase;

  __device__ __forceinline__ void write(int cnt) {  // the last cnt (<= 32) candidates
    nc -= cnt;
    unsigned long long at = 0;
    if (lane == 0) {
      at = atomicAdd(&a.ctr->cand, (unsigned long long)cnt) - lbase;
      if (at + cnt > a.cand_cap) atomicOr(&a.ctr->status, (unsigned)TL_ST_LEAFQ);
    }
    at = __shfl_sync(0xffffffffu, at, 0);
    if (lane < cnt && at + lane < a.cand_cap) {
      const uint32_t e = ws.cand[nc + lane], q = qpos0 + (e >> 27), t = tpos0 + (e & kIdxMask);
      a.cand[at + lane] = a.swap ? make_uint2(t, q) : make_uint2(q, t);
    }
    __syncwarp();
  }
  __device__ __forceinline__ void look(int cnt) {  // the last cnt (<= 32) pending pairs
    np -= cnt;
    bool open = false;
    uint32_t e = 0u;
    if (lane < cnt) {
      e = ws.pend[np + lane];
      open = true;
      if (!FP64) {
        const size_t t = 2 * (size_t)(tpos0 + (e & kIdxMask));
        const uint32_t q = e >> 27;
        const float4 pb = __ldg(a.t + t), db = __ldg(a.t + t + 1);
        open = !tl_narrow32_sure_miss(ws.qpos[q], ws.qdir[q], pb, db, a.nk, suf);
      }
    }
    const unsigned m = __ballot_sync(0xffffffffu, open);
    if (open) ws.cand[nc + __popc(m & ((1u << lane) - 1u))] = e;
    nc += __popc(m);
    __syncwarp();
    if (nc >= 32) write(32);
  }
  // every lane's pairs: bit r of bits stands for box r of the cnt last tested, this lane
  // for its photon (by_tree) or for photon j0 + lane of the tree
  __device__ __forceinline__ void add(uint32_t bits, bool by_tree, uint32_t j0) {
    if (!__any_sync(0xffffffffu, bits != 0u)) return;
    int inc = __popc(bits);
    const int own = inc;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const int t = __shfl_up_sync(0xffffffffu, inc, off);
      if (lane >= off) inc += t;
    }
    const int total = __shfl_sync(0xffffffffu, inc, 31);
    // what does not fit the list at once (dense leaves) goes in rounds of one per lane
    if (np + total <= kPend) {
      int at = np + inc - own;
      while (bits) {
        const uint32_t k = ws.id[__ffs(bits) - 1];
        bits &= bits - 1u;
        ws.pend[at++] = by_tree ? (uint32_t)lane << 27 | (j0 + k) : k << 27 | (j0 + lane);
      }
      np += total;
      __syncwarp();
      while (np >= 32) look(32);
      return;
    }
    unsigned m;
    while ((m = __ballot_sync(0xffffffffu, bits != 0u)) != 0u) {
      if (bits) {
        const uint32_t k = ws.id[__ffs(bits) - 1];
        bits &= bits - 1u;
        ws.pend[np + __popc(m & ((1u << lane) - 1u))] =
            by_tree ? (uint32_t)lane << 27 | (j0 + k) : k << 27 | (j0 + lane);
      }
      np += __popc(m);
      __syncwarp();
      while (np >= 32) look(32);
    }
  }
  __device__ __forceinline__ void finish() {
    if (np) look(np);
    if (nc) write(nc);
  }
};

// The boxes src of the lanes in sel against box cmp of every lane: bit r of the result,
// the r-th of them overlaps.  The boxes pass through shared memory, compacted, and come
// back by broadcast: ~10 instructions for 32 box pairs.
__device__ __forceinline__ uint32_t test_boxes(ColSmem &ws, const TLBox &src, unsigned sel,
                                               const TLBox &cmp, int lane) {
  __syncwarp();
  if (sel >> lane & 1u) {
    const int r = __popc(sel & ((1u << lane) - 1u));
    put_box(ws.cbox + 2 * r, src);
    ws.id[r] = (uint8_t)lane;
  }
  __syncwarp();
  const int cnt = __popc(sel);
  uint32_t bits = 0u;
#pragma unroll 4
  for (int r = 0; r < cnt; ++r)
    if (tl_overlap(get_box(ws.cbox + 2 * r), cmp)) bits |= 1u << r;
  return bits;
}

// The same for needles, with the window lt: ~14 instructions for 32 pairs.
__device__ __forceinline__ uint32_t test_needles(ColSmem &ws, const TLNeedle &src, unsigned sel,
                                                 const TLNeedle &cmp, float lt, int lane) {
  __syncwarp();
  if (sel >> lane & 1u) {
    const int r = __popc(sel & ((1u << lane) - 1u));
    put_needle(ws.cbox + 2 * r, src);
    ws.id[r] = (uint8_t)lane;
  }
  __syncwarp();
  const int cnt = __popc(sel);
  uint32_t bits = 0u;
#pragma unroll 4
  for (int r = 0; r < cnt; ++r) {
    const float4 c = ws.cbox[2 * r];
    const float2 g = *reinterpret_cast<const float2 *>(ws.cbox + 2 * r + 1);
    const float u = c.z + cmp.w;
    const float x = fmaf(c.w - cmp.vx, u, c.x - cmp.x), y = fmaf(g.x - cmp.vy, u, c.y - cmp.y);
    if (fabsf(u) <= lt && fmaxf(fabsf(x), fabsf(y)) <= g.y + cmp.h) bits |= 1u << r;
  }
  return bits;
}

// One warp: 32 consecutive photons of the query beam, one per lane, against the tree.
// A node's 32 children are tested by 32 lanes at once against the union of the warp's
// boxes; those that overlap it are tested by every lane against its own box, and
// the node's child is descended into if any lane overlaps it.  At the photons, the two
// sides' survivors are tested against each other along the shorter list: survivors of the
// tree against all lanes, or the lanes against all 32.  What bounds it is issue: one
// coalesced load serves 32 tests, and box tests cost ~10 warp instructions for 32 pairs
// (the dual descent of two binary trees took 25 warp instructions per popped node pair
// and lane-private 64-byte records).  Few groups (small beams): the tree is cut into
// `slices` contiguous parts of its sorted photons, one warp each per group.
// Measured (with the first look, which was k_narrow's): 2 x 4M statistical step 15.0 ms
// for the dual descent and its narrow phase, 6.1 ms by boxes (half of it the first look at
// pairs whose boxes meet at different times), 3.8 ms by needles; 2 x 16M at 90 degrees
// 7.3 ms, 1.1 ms now (there the turned frame is most of it).
template <bool FP64, bool NEEDLES>
__global__ void __launch_bounds__(32 * kColWarps, 8) k_collide(ColArgs a) {
  __shared__ ColSmem wsm[kColWarps];
  __shared__ float suf[TL_SBINS];
  if (a.ctr->status & (TL_ST_TIMEOUT | TL_ST_SPILL_OVF)) return;  // the build failed
  if (!FP64) {
    for (int i = threadIdx.x; i < TL_SBINS; i += blockDim.x) suf[i] = a.nk.suf[i];
    __syncthreads();
  }
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const long long item = blockIdx.x * (long long)kColWarps + warp;
  if (item >= a.items) return;
  const int g = a.group0 + (int)(item / a.slices), slice = (int)(item % a.slices);
  const uint32_t inst = a.group_inst ? a.group_inst[g] : 0u;
  const TLInst &Q = a.qinst[inst], &T = a.tinst[inst];
  const int r0 = (g - Q.group0) * 32, qn = tl_live(Q, a.qstart);
  if (r0 >= qn) return;
  const int tn = tl_live(T, a.tstart), leaves_n = tl_level_count(tn, 1);
  const int c0 = (int)((long long)leaves_n * slice / a.slices);
  const int c1 = (int)((long long)leaves_n * (slice + 1) / a.slices);
  if (c0 == c1) return;
  ColSmem &ws = wsm[warp];
  Pairs<FP64> out{a, ws, suf, (uint32_t)g * 32u, (uint32_t)T.group0 * 32u, lane, 0, 0,
                  a.ctr->leaf_base};
  const TLFrame &f = a.frames[inst];
  TLBox own = empty_box();
  TLNeedle ndl = no_needle();
  if (r0 + lane < qn) {
    const float4 *r = a.q + 2 * ((int64_t)g * 32 + lane);
    const float4 p = r[0], d = r[1];
    const float pad = tl_photon_pad(f, a.swap, p.w, a.half);
    own = swept_box(p, d, f, a.Llo, a.Lhi, pad);
    if (NEEDLES) ndl = tl_needle(f, a.swap, p, d, pad);
    ws.qpos[lane] = p;
    ws.qdir[lane] = d;
  }
  const TLBox all = warp_union(own);
  // where and when the warp's needles are: x, y and w of the whole window
  float lt = 0.0f;
  TLBox span = empty_box();
  if (NEEDLES) {
    lt = f.lt + __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(ndl.e)));
    if (r0 + lane < qn) {
      const float ax = fmaf(fabsf(ndl.vx), lt, ndl.h), ay = fmaf(fabsf(ndl.vy), lt, ndl.h);
      span = TLBox{ndl.x - ax, ndl.y - ay, ndl.w, ndl.x + ax, ndl.y + ay, ndl.w};
    }
    span = warp_union(span);
  }
  unsigned long long node_tests = 0, narrow = 0;
  unsigned leaves = 0;
  const int top = tl_top_level(tn);
  int lev = top, base = 0;
  unsigned mask = 0u;      // children of (lev, base) to descend into
  unsigned near = 0u;      // level 1: leaves that overlap the union,
  uint32_t hits = 0u;      // and which of them overlap this lane's box
  bool fresh = true;       // the children of (lev, base) are still to be tested
  while (true) {
    if (fresh) {
      const int cnt = min(32, tl_level_count(tn, lev) - base), c = base + lane;
      const int sh = 5 * (lev - 1);
      const bool ok = lane < cnt && ((long long)c << sh) < c1 && ((long long)(c + 1) << sh) > c0;
      const TLBox b = ok ? get_box(a.box + 2 * ((size_t)T.lev[lev] + c)) : empty_box();
      near = __ballot_sync(0xffffffffu, tl_overlap(b, all));
      node_tests += (unsigned)(cnt + 32 * __popc(near));
      mask = 0u;
      if (near) {
        hits = test_boxes(ws, b, near, own, lane);
        const uint32_t any = __reduce_or_sync(0xffffffffu, hits);
        mask = __ballot_sync(0xffffffffu, (near >> lane & 1u) &&
                                              (any >> __popc(near & ((1u << lane) - 1u)) & 1u));
      }
      fresh = false;
    }
    if (lev == 1)
      while (mask) {  // leaves: 32 photons of the tree
        const int k = __ffs(mask) - 1;
        mask &= mask - 1u;
        const int j0 = (base + k) * 32;
        const bool ok = j0 + lane < tn;
        const float4 *src = a.box + 2 * ((size_t)T.lev[0] + j0 + lane);
        const unsigned mq =
            __ballot_sync(0xffffffffu, hits >> __popc(near & ((1u << k) - 1u)) & 1u);
        if (NEEDLES) {
          const TLNeedle b = ok ? get_needle(src) : no_needle();
          const float l = lt + __uint_as_float(
                                   __reduce_max_sync(0xffffffffu, __float_as_uint(b.e)));
          const float ax = fmaf(fabsf(b.vx), l, b.h), ay = fmaf(fabsf(b.vy), l, b.h);
          const unsigned mb = __ballot_sync(
              0xffffffffu, b.x + ax >= span.lx && b.x - ax <= span.hx && b.y + ay >= span.ly &&
                               b.y - ay <= span.hy && b.w + span.hz >= -l && b.w + span.lz <= l);
          ++leaves;
          const int nb = __popc(mb), nq = __popc(mq);
          narrow += (unsigned)(nb * nq);
          if (nb == 0) continue;
          const bool by_tree = nb <= nq;
          out.add(by_tree ? test_needles(ws, b, mb, ndl, l, lane)
                          : test_needles(ws, ndl, mq, b, l, lane),
                  by_tree, (uint32_t)j0);
          continue;
        }
        const TLBox b = ok ? get_box(src) : empty_box();
        const unsigned mb = __ballot_sync(0xffffffffu, tl_overlap(b, all));
        ++leaves;
        const int nb = __popc(mb), nq = __popc(mq);
        narrow += (unsigned)(nb * nq);
        if (nb == 0) continue;
        const bool by_tree = nb <= nq;
        out.add(by_tree ? test_boxes(ws, b, mb, own, lane) : test_boxes(ws, own, mq, b, lane),
                by_tree, (uint32_t)j0);
      }
    while (!mask && lev < top) {  // up to the next level with children left
      ++lev;
      mask = ws.mask[lev];
      base = (int)ws.base[lev];
    }
    if (!mask) break;
    const int k = __ffs(mask) - 1;
    mask &= mask - 1u;
    __syncwarp();
    if (lane == 0) {
      ws.mask[lev] = mask;
      ws.base[lev] = (uint32_t)base;
    }
    __syncwarp();
    base = (base + k) * 32;
    --lev;
    fresh = true;
  }
  out.finish();
  if (lane == 0) {
    if (node_tests) atomicAdd(&a.ctr->node_tests, node_tests);
    if (narrow) atomicAdd(&a.ctr->narrow_tests, narrow);
    if (leaves) atomicAdd(&a.ctr->leaf_pairs, (unsigned long long)leaves);
  }
}

cudaError_t launch_collide(const ColArgs &a, cudaStream_t s) {
  if (a.items <= 0) return cudaSuccess;
  const unsigned blocks = (unsigned)((a.items + kColWarps - 1) / kColWarps);
  auto *const k = a.needles ? (a.fp64 ? k_collide<true, true> : k_collide<false, true>)
                            : (a.fp64 ? k_collide<true, false> : k_collide<false, false>);
  k<<<blocks, 32 * kColWarps, 0, s>>>(a);
  return cudaGetLastError();
}

// Before part p > 0 of a step: its candidates start at the list's beginning again.
__global__ void k_part_next(TLCounters *ctr) {
  ctr->leaf_base = ctr->cand;
}

cudaError_t launch_part_next(TLCounters *ctr, cudaStream_t s) {
  k_part_next<<<1, 1, 0, s>>>(ctr);
  return cudaGetLastError();
}

// The candidates of the step (or part): FP32 test with its band, one pair per lane; in
// FP64 mode a division-free test first, then the definition on full warps.
template <bool FP64>
__global__ void __launch_bounds__(256) k_decide(TravArgs a) {
  __shared__ uint2 pend[8][64];
  __shared__ float sbin[TL_SBINS];
  const unsigned long long listed = a.ctr->cand - a.ctr->leaf_base;
  const unsigned long long n = min(listed, a.leaf_cap);
  if (blockIdx.x == 0 && threadIdx.x == 0) atomicMax(&a.ctr->max_part_leaves, listed);
  if (blockIdx.x * 256ull >= n) return;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (!FP64) {
    for (int i = threadIdx.x; i < TL_SBINS; i += blockDim.x) sbin[i] = a.nk.sbin[i];
    __syncthreads();
  }
  int np = 0;
  for (unsigned long long i0 = blockIdx.x * 256ull + warp * 32ull; i0 < n;
       i0 += gridDim.x * 256ull) {
    const unsigned long long i = i0 + lane;
    const bool ok = i < n;
    const uint2 pr = ok ? a.leaves[i] : make_uint2(0u, 0u);
    if (!FP64) {
      decide_pairs<FP64>(a, pr, ok, lane, sbin);
      continue;
    }
    bool open = false;
    if (ok)
      open = !tl_exact_sure_miss(
          a.mA, __float_as_uint(__ldg(a.A.dir + (size_t)pr.x * a.A.stride).w), a.mB,
          __float_as_uint(__ldg(a.B.dir + (size_t)pr.y * a.B.stride).w), a.ct, a.dt,
          (double)a.nk.r2max);
    const unsigned m = __ballot_sync(0xffffffffu, open);
    if (open) pend[warp][np + __popc(m & ((1u << lane) - 1u))] = pr;
    np += __popc(m);
    __syncwarp();
    if (np < 32) continue;
    decide_pairs<FP64>(a, pend[warp][lane], true, lane, sbin);
    np -= 32;
    const uint2 v = lane < np ? pend[warp][32 + lane] : make_uint2(0u, 0u);
    __syncwarp();
    if (lane < np) pend[warp][lane] = v;
    __syncwarp();
  }
  if (np > 0)
    decide_pairs<FP64>(a, lane < np ? pend[warp][lane] : make_uint2(0u, 0u), lane < np, lane, sbin);
}

cudaError_t launch_decide(const TravArgs &a, int blocks, cudaStream_t s) {
  if (a.fp64) k_decide<true><<<blocks, 256, 0, s>>>(a);
  else k_decide<false><<<blocks, 256, 0, s>>>(a);
  return cudaGetLastError();
}

// Zero the step's counters; a failed build, or an earlier step's queue overflow or
// expired wait in a captured run (run_status, else NULL), carries over, so that no
// later kernel of the step or run works on what is not valid.
__global__ void k_step_init(TLCounters *ctr, const unsigned *build_status,
                            const unsigned *run_status) {
  unsigned *w = reinterpret_cast<unsigned *>(ctr);
  for (int i = threadIdx.x; i < (int)(sizeof(TLCounters) / 4); i += blockDim.x) w[i] = 0u;
  __syncthreads();
  if (threadIdx.x == 0) {
    const unsigned bs = *build_status & (unsigned)TL_ST_TIMEOUT;
    const unsigned rs =
        run_status ? *run_status & (unsigned)(TL_ST_SPILL_OVF | TL_ST_TIMEOUT) : 0u;
    ctr->status = bs | rs;
  }
}

cudaError_t launch_step_init(TLCounters *ctr, const unsigned *build_status,
                             const unsigned *run_status, cudaStream_t s) {
  k_step_init<<<1, 128, 0, s>>>(ctr, build_status, run_status);
  return cudaGetLastError();
}

}  // namespace tl
