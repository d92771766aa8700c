// tl_tree.cu -- the exact path: order, trees and collisions of a step.
//
// Both beams are propagated and sorted along a Hilbert curve (k_order, tl_sort.cu).
// The smaller beam (the tree's) gets a packed tree over its sorted photons with 32
// children per node (as in Kamel and Faloutsos, "Hilbert R-tree", VLDB 1994: leaves
// are runs of the curve, so there are no links to build): k_boxes writes every
// photon's swept box and the boxes of levels 1 and 2, k_upper those above.  The other
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

// Per-axis sums of p', d', p'^2, p' d', d'^2 with p' = R p0, d' = R d (15 FP64 values),
// in a fixed order (per-block sums, then one block over the blocks).  With the
// frame the means and variances of the swept boxes' centres follow in closed form for
// every step.
constexpr int kMomentBlocks = 4 * 152;

__device__ __forceinline__ void turn(const TLFrame &f, double v[3]) {
  if (f.ident) return;
  const double x = v[0], y = v[1], z = v[2];
  for (int k = 0; k < 3; ++k)
    v[k] = (double)f.r[3 * k] * x + (double)f.r[3 * k + 1] * y + (double)f.r[3 * k + 2] * z;
}

__global__ void __launch_bounds__(256) k_beam_moments(TLBeam b, TLFrame f, double *part) {
  double m[15];
  for (int q = 0; q < 15; ++q) m[q] = 0.0;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < b.n;
       i += (int64_t)gridDim.x * blockDim.x) {
    double p[3] = {b.px[i], b.py[i], b.pz[i]}, d[3] = {b.dx[i], b.dy[i], b.dz[i]};
    turn(f, p);
    turn(f, d);
    for (int a = 0; a < 3; ++a) {
      m[a] += p[a];
      m[3 + a] += d[a];
      m[6 + a] += p[a] * p[a];
      m[9 + a] += p[a] * d[a];
      m[12 + a] += d[a] * d[a];
    }
  }
  __shared__ double sm[8][15];
  for (int q = 0; q < 15; ++q)
    for (int off = 16; off; off >>= 1) m[q] += __shfl_xor_sync(0xffffffffu, m[q], off);
  if ((threadIdx.x & 31) == 0)
    for (int q = 0; q < 15; ++q) sm[threadIdx.x >> 5][q] = m[q];
  __syncthreads();
  if (threadIdx.x < 15) {
    double t = 0.0;
    for (int w8 = 0; w8 < 8; ++w8) t += sm[w8][threadIdx.x];
    part[blockIdx.x * 15 + threadIdx.x] = t;
  }
}

__global__ void k_beam_moments_final(const double *part, int nparts, double *out) {
  if (threadIdx.x < 15) {
    double t = 0.0;
    for (int k = 0; k < nparts; ++k) t += part[k * 15 + threadIdx.x];
    out[threadIdx.x] = t;
  }
}

size_t moment_doubles() { return 15 * (1 + kMomentBlocks); }

// out: device, moment_doubles() doubles, the 15 moments first
cudaError_t launch_beam_moments(const TLBeam &b, const TLFrame &f, double *out, cudaStream_t s) {
  const int64_t nb = (b.n + 255) / 256;
  const int blocks = (int)(nb < 1 ? 1 : (nb < kMomentBlocks ? nb : kMomentBlocks));
  k_beam_moments<<<blocks, 256, 0, s>>>(b, f, out + 15);
  k_beam_moments_final<<<1, 32, 0, s>>>(out + 15, blocks, out);
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

// Frames of a batch's instances, from the middle of each beam's range of directions.
__global__ void k_inst_frames(const double *ba, const double *bb, int n_inst, TLFrame *out) {
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= n_inst) return;
  double a[3], b[3];
  for (int k = 0; k < 3; ++k) {
    a[k] = 0.5 * (ba[12 * q + 3 + k] + ba[12 * q + 9 + k]);
    b[k] = 0.5 * (bb[12 * q + 3 + k] + bb[12 * q + 9 + k]);
  }
  out[q] = tl_make_frame(a, b);  // an empty beam's bounds are NaN or infinite: the lab frame
}

cudaError_t launch_inst_frames(const double *ba, const double *bb, int n_inst, TLFrame *out,
                               cudaStream_t s) {
  k_inst_frames<<<(n_inst + 127) / 128, 128, 0, s>>>(ba, bb, n_inst, out);
  return cudaGetLastError();
}

// Ordering grids of both beams of a batch's instances for the step with travel
// T = c t_k + L / 2 to the swept boxes' centres: the range of the centres, and cells in
// the proportions of the boxes' extents (pad + travel of a typical photon).
__global__ void k_inst_grid(const double *ba, const double *bb, const TLFrame *frames, int n_inst,
                            double T, double L, double half, int bits, TLGrid *ga, TLGrid *gb) {
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= n_inst) return;
  const TLFrame f = frames[q];
  const double *bd[2] = {ba + 12 * (size_t)q, bb + 12 * (size_t)q};
  double ru[3], s[3];
  for (int k = 0; k < 3; ++k) {
    ru[k] = (double)f.r[3 * k] * f.u[0] + (double)f.r[3 * k + 1] * f.u[1] +
            (double)f.r[3 * k + 2] * f.u[2];
    s[k] = 2.0 * half;
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
    (h ? gb : ga)[q] = tl_make_grid(lo, range, s, bits);
  }
}

cudaError_t launch_inst_grid(const double *ba, const double *bb, const TLFrame *frames, int n_inst,
                             double T, double L, double half, int bits, TLGrid *ga, TLGrid *gb,
                             cudaStream_t s) {
  k_inst_grid<<<(n_inst + 127) / 128, 128, 0, s>>>(ba, bb, frames, n_inst, T, L, half, bits, ga, gb);
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

// Propagate p = p0 + c t_k d in FP64 (closed form), round to the FP32 SoA, and key
// every photon by its swept box's centre in the frame, with several instances below
// the instance's number.  Also counts the 8-bit digits of every sort pass in shared
// memory, flushed once per block.  Bound by GB300's FP64 pipe (six operations and
// three conversions per photon at 2 per clock and SM), beside which the key's integer
// work is free.  A fixed grid of at most kPropBlocks blocks, grid-stride.
constexpr int kPropBlocks = 4 * 152;

__global__ void __launch_bounds__(256) k_order(OrderArgs a) {
  __shared__ uint32_t sh[4][256];
  for (int t = threadIdx.x; t < 4 * 256; t += 256) (&sh[0][0])[t] = 0u;
  __syncthreads();
  const float halfL = 0.5f * a.L;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < a.b.n;
       i += (int64_t)gridDim.x * blockDim.x) {
    const double dx = a.b.dx[i], dy = a.b.dy[i], dz = a.b.dz[i];
    const float3 p = make_float3(__double2float_rn(__dadd_rn(a.b.px[i], __dmul_rn(a.ct, dx))),
                                 __double2float_rn(__dadd_rn(a.b.py[i], __dmul_rn(a.ct, dy))),
                                 __double2float_rn(__dadd_rn(a.b.pz[i], __dmul_rn(a.ct, dz))));
    const float4 d = a.dir_u[i];  // the FP32 direction, written once (k_static_soa)
    float *pu = reinterpret_cast<float *>(a.pos_u + i);  // x, y, z; w holds the energy
    *reinterpret_cast<float2 *>(pu) = make_float2(p.x, p.y);
    pu[2] = p.z;
    const uint32_t q = a.inst_of ? a.inst_of[i] : 0u;
    const TLFrame &f = a.frames[q];
    float c[3];
    if (f.ident) {
      c[0] = fmaf(halfL, d.x, p.x);
      c[1] = fmaf(halfL, d.y, p.y);
      c[2] = fmaf(halfL, d.z, p.z);
    } else {
      const float mx = fmaf(halfL, d.x - f.u[0], p.x), my = fmaf(halfL, d.y - f.u[1], p.y),
                  mz = fmaf(halfL, d.z - f.u[2], p.z);
#pragma unroll
      for (int k = 0; k < 3; ++k)
        c[k] = fmaf(f.r[3 * k], mx, fmaf(f.r[3 * k + 1], my, f.r[3 * k + 2] * mz));
    }
    const uint32_t key =
        a.inst_of ? (q << a.inst_shift | order_key(a.grids[q], c)) : order_key(a.grid, c);
    a.key[i] = key;
    for (int r = 0; r < a.passes; ++r) atomicAdd(&sh[r][(key >> (8 * r)) & 255u], 1u);
  }
  __syncthreads();
  for (int t = threadIdx.x; t < a.passes * 256; t += 256) {
    const uint32_t v = (&sh[0][0])[t];
    if (v) atomicAdd(&a.hist[t], v);
  }
}

cudaError_t launch_order(const OrderArgs &a, cudaStream_t s) {
  if (a.b.n <= 0) return cudaSuccess;
  const int64_t nb = (a.b.n + 255) / 256;
  k_order<<<(int)(nb < kPropBlocks ? nb : kPropBlocks), 256, 0, s>>>(a);
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

// One block per tile: every photon's swept box, the boxes of the tile's 32 runs of 32
// photons (level 1) and the tile's own (level 2).  One pass over the sorted photons;
// unions by shuffles, no links and no second pass.
__global__ void __launch_bounds__(kTile) k_boxes(BoxArgs a) {
  __shared__ TLBox wb[32];
  if (*a.build_status & TL_ST_TIMEOUT) return;  // keys unsorted: the build is abandoned
  const int tile = blockIdx.x, t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const uint32_t q = a.tile_inst ? a.tile_inst[tile] : 0u;
  const TLInst &I = a.inst[q];
  const int k = tile - I.tile0, r = k * kTile + t;
  TLBox b = empty_box();
  if (r < I.n) {
    const int64_t p = (int64_t)tile * kTile + t;
    b = swept_box(a.pos[p], a.dir[p], a.frames[q], a.Llo, a.Lhi, a.half);
    put_box(a.box + 2 * ((size_t)I.lev[0] + r), b);
  }
  b = warp_union(b);
  if (lane == 0) {
    wb[warp] = b;
    if (r < I.n) put_box(a.box + 2 * ((size_t)I.lev[1] + k * 32 + warp), b);
  }
  __syncthreads();
  if (warp == 0) {
    b = warp_union(wb[lane]);
    if (lane == 0) put_box(a.box + 2 * ((size_t)I.lev[2] + k), b);
  }
}

// Levels 3 and up of one instance's tree per block, a warp per node.
__global__ void __launch_bounds__(1024) k_upper(const TLInst *inst, float4 *box) {
  const TLInst &I = inst[blockIdx.x];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int l = 3; l <= I.top; ++l) {
    for (int j = warp; j < I.cnt[l]; j += 32) {
      const int c = 32 * j + lane;
      TLBox b = c < I.cnt[l - 1] ? get_box(box + 2 * ((size_t)I.lev[l - 1] + c)) : empty_box();
      b = warp_union(b);
      if (lane == 0) put_box(box + 2 * ((size_t)I.lev[l] + j), b);
    }
    __syncthreads();
  }
}

cudaError_t launch_boxes(const BoxArgs &a, int tiles, int n_inst, int max_top, cudaStream_t s) {
  if (tiles <= 0) return cudaSuccess;
  k_boxes<<<tiles, kTile, 0, s>>>(a);
  if (max_top >= 3) k_upper<<<n_inst, 1024, 0, s>>>(a.inst, a.box);
  return cudaGetLastError();
}

// ---------------------------------------------------------------- collisions

constexpr int kColWarps = 4;
constexpr uint32_t kIdxMask = (1u << 27) - 1u;  // beams hold fewer than 2^27 photons

struct ColSmem {
  float4 qpos[32], qdir[32];  // the warp's photons
  float4 qbox[64];            // their boxes
  float4 cbox[64];            // boxes of the visited node's children
  uint32_t pend[64];          // (lane << 27 | photon of the tree): boxes overlap
  uint32_t cand[64];          // undecided by the first look
  uint32_t mask[6], base[6];  // per level: children still to descend into
};

// Photon pairs whose boxes overlap: the first look, 32 at a time; what it leaves goes
// to the step's candidate list.
template <bool FP64>
struct Pairs {
  const ColArgs &a;
  ColSmem &ws;
  const float *suf;
  uint32_t qpos0, tpos0;  // padded position of the warp's first photon, of the tree's
  int lane, np, nc;
  unsigned long long lbase;

  __device__ __forceinline__ void write(int cnt) {  // the first cnt candidates
    unsigned long long at = 0;
    if (lane == 0) {
      at = atomicAdd(&a.ctr->cand, (unsigned long long)cnt) - lbase;
      if (at + cnt > a.cand_cap) atomicOr(&a.ctr->status, (unsigned)TL_ST_LEAFQ);
    }
    at = __shfl_sync(0xffffffffu, at, 0);
    if (lane < cnt && at + lane < a.cand_cap) {
      const uint32_t e = ws.cand[lane], q = qpos0 + (e >> 27), t = tpos0 + (e & kIdxMask);
      a.cand[at + lane] = a.swap ? make_uint2(t, q) : make_uint2(q, t);
    }
  }
  __device__ __forceinline__ void look(int cnt) {  // the first cnt (<= 32) pending pairs
    bool open = false;
    uint32_t e = 0u;
    if (lane < cnt) {
      e = ws.pend[lane];
      open = true;
      if (!FP64) {
        const uint32_t t = tpos0 + (e & kIdxMask), q = e >> 27;
        const float4 pb = __ldg(a.tpos + t), db = __ldg(a.tdir + t);
        open = !tl_narrow32_sure_miss(ws.qpos[q], ws.qdir[q], pb, db, a.nk, suf);
      }
    }
    const unsigned m = __ballot_sync(0xffffffffu, open);
    if (!m) return;
    if (open) ws.cand[nc + __popc(m & ((1u << lane) - 1u))] = e;
    nc += __popc(m);
    __syncwarp();
    if (nc < 32) return;
    write(32);
    nc -= 32;
    const uint32_t v = lane < nc ? ws.cand[32 + lane] : 0u;
    __syncwarp();
    if (lane < nc) ws.cand[lane] = v;
    __syncwarp();
  }
  __device__ __forceinline__ void add(bool ok, unsigned m, uint32_t e) {  // m = ballot(ok) != 0
    if (ok) ws.pend[np + __popc(m & ((1u << lane) - 1u))] = e;
    np += __popc(m);
    __syncwarp();
    if (np < 32) return;
    look(32);
    np -= 32;
    const uint32_t v = lane < np ? ws.pend[32 + lane] : 0u;
    __syncwarp();
    if (lane < np) ws.pend[lane] = v;
    __syncwarp();
  }
  __device__ __forceinline__ void finish() {
    if (np) look(np);
    if (nc) write(nc);
  }
};

// One warp: 32 consecutive photons of the query beam, one per lane, against the tree.
// A node's 32 children are tested by 32 lanes at once against the union of the warp's
// boxes; each that overlaps it is then tested by every lane against its own box, and
// the node is descended into if any lane overlaps.  At the photons, the two sides'
// survivors are tested against each other along the shorter list: survivors of the
// tree one by one against all lanes, or the lanes one by one against all 32.  What
// bounds it is issue: one coalesced load serves 32 tests and boxes come from shared
// memory by broadcast, so a box test costs ~12 warp instructions for 32 pairs (the
// dual descent of two binary trees took 25 warp instructions per popped node pair and
// lane-private 64-byte records).  Few groups (small beams): the tree is cut into
// `slices` contiguous parts of its sorted photons, one warp each per group.
// Measured (with the first look, which was k_narrow's): 2 x 4M statistical step 15.0 ms
// for the dual descent and its narrow phase, 6.4 ms now; 2 x 16M at 90 degrees 7.3 ms,
// 1.1 ms now (there the turned frame is most of it).
template <bool FP64>
__global__ void __launch_bounds__(32 * kColWarps) k_collide(ColArgs a) {
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
  const int tile = g >> 5;
  const uint32_t inst = a.tile_inst ? a.tile_inst[tile] : 0u;
  const TLInst &Q = a.qinst[inst], &T = a.tinst[inst];
  const int r0 = (g - Q.tile0 * 32) * 32;
  if (r0 >= Q.n || T.n == 0) return;
  const int c0 = (int)((long long)T.cnt[1] * slice / a.slices);
  const int c1 = (int)((long long)T.cnt[1] * (slice + 1) / a.slices);
  if (c0 == c1) return;
  ColSmem &ws = wsm[warp];
  Pairs<FP64> out{a, ws, suf, (uint32_t)g * 32u, (uint32_t)T.tile0 * (uint32_t)kTile, lane, 0, 0,
                  a.ctr->leaf_base};
  TLBox own = empty_box();
  if (r0 + lane < Q.n) {
    const float4 p = a.qpos[(int64_t)g * 32 + lane], d = a.qdir[(int64_t)g * 32 + lane];
    own = swept_box(p, d, a.frames[inst], a.Llo, a.Lhi, a.half);
    ws.qpos[lane] = p;
    ws.qdir[lane] = d;
  }
  put_box(ws.qbox + 2 * lane, own);
  const TLBox all = warp_union(own);
  unsigned long long node_tests = 0, narrow = 0, leaves = 0;
  const int top = T.top;
  int lev = top, base = 0;
  unsigned mask = 0u, lanes = 0u;  // children to descend into; lane c: the lanes that overlap c
  bool fresh = true;               // the children of (lev, base) are still to be tested
  while (true) {
    if (fresh) {
      const int cnt = min(32, T.cnt[lev] - base), c = base + lane;
      const int sh = 5 * (lev - 1);
      bool ok = lane < cnt && ((long long)c << sh) < c1 && ((long long)(c + 1) << sh) > c0;
      const TLBox b = ok ? get_box(a.box + 2 * ((size_t)T.lev[lev] + c)) : empty_box();
      ok = tl_overlap(b, all);
      unsigned m = __ballot_sync(0xffffffffu, ok);
      node_tests += (unsigned)(cnt + 32 * __popc(m));
      mask = 0u;
      if (m) {
        __syncwarp();
        put_box(ws.cbox + 2 * lane, b);
        __syncwarp();
        do {
          const int k = __ffs(m) - 1;
          m &= m - 1u;
          const unsigned w = __ballot_sync(0xffffffffu, tl_overlap(get_box(ws.cbox + 2 * k), own));
          if (lane == k) lanes = w;
          if (w) mask |= 1u << k;
        } while (m);
      }
      fresh = false;
    }
    if (lev == 1)
      while (mask) {  // leaves: 32 photons of the tree
        const int k = __ffs(mask) - 1;
        mask &= mask - 1u;
        const int j0 = (base + k) * 32;
        const bool ok = j0 + lane < T.n;
        const TLBox b = ok ? get_box(a.box + 2 * ((size_t)T.lev[0] + j0 + lane)) : empty_box();
        unsigned mb = __ballot_sync(0xffffffffu, tl_overlap(b, all));
        unsigned mq = __shfl_sync(0xffffffffu, lanes, k);
        ++leaves;
        const int nb = __popc(mb), nq = __popc(mq);
        narrow += (unsigned)(nb * nq);
        if (nb <= nq) {
          if (!mb) continue;
          __syncwarp();
          put_box(ws.cbox + 2 * lane, b);
          __syncwarp();
          do {
            const int j = __ffs(mb) - 1;
            mb &= mb - 1u;
            const bool hit = tl_overlap(get_box(ws.cbox + 2 * j), own);
            const unsigned m = __ballot_sync(0xffffffffu, hit);
            if (m) out.add(hit, m, (uint32_t)lane << 27 | (uint32_t)(j0 + j));
          } while (mb);
        } else {
          do {
            const int q = __ffs(mq) - 1;
            mq &= mq - 1u;
            const bool hit = tl_overlap(get_box(ws.qbox + 2 * q), b);
            const unsigned m = __ballot_sync(0xffffffffu, hit);
            if (m) out.add(hit, m, (uint32_t)q << 27 | (uint32_t)(j0 + lane));
          } while (mq);
        }
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
    if (leaves) atomicAdd(&a.ctr->leaf_pairs, leaves);
  }
}

cudaError_t launch_collide(const ColArgs &a, cudaStream_t s) {
  if (a.items <= 0) return cudaSuccess;
  const unsigned blocks = (unsigned)((a.items + kColWarps - 1) / kColWarps);
  if (a.fp64) k_collide<true><<<blocks, 32 * kColWarps, 0, s>>>(a);
  else k_collide<false><<<blocks, 32 * kColWarps, 0, s>>>(a);
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
      open = !tl_exact_sure_miss(a.mA, __float_as_uint(__ldg(a.A.dir + pr.x).w), a.mB,
                                 __float_as_uint(__ldg(a.B.dir + pr.y).w), a.ct, a.dt,
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
