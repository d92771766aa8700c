// tl_build.cu -- binary hierarchy of one beam for the statistical regime, whose clouds
// are its nodes at a Morton level (the exact path's trees are in tl_tree.cu).
//
//   propagate   positions in closed form (FP64), FP32 SoA, Morton key of the
//               swept box's centre in the step's moment box, and the radix
//               sort's digit histogram (one pass over the FP64 input)
//   gather      SoA into Morton order
//   karras      inner nodes of the binary radix tree over the sorted keys
//               (Karras 2012, "Maximizing parallelism in the construction of
//               BVHs, octrees and k-d trees"), leaf buckets of <= B photons
//   refit       every node's box as the union of its photons' swept boxes
//               (Sec. 2.1: each box covers the travel of its photons during
//               the step) over its contiguous photon range: sparse tables per
//               tile and over tiles, no atomics and no waiting
#include "tl_common.cuh"
#include "tl_frame.cuh"

namespace tl {

// ---------------------------------------------------------------- Morton

// spread the low 21 bits of x to every third bit (bit interleaving by masks)
__device__ __forceinline__ unsigned long long spread3(unsigned long long x) {
  x &= 0x1fffffull;
  x = (x | (x << 32)) & 0x1f00000000ffffull;
  x = (x | (x << 16)) & 0x1f0000ff0000ffull;
  x = (x | (x << 8)) & 0x100f00f00f00f00full;
  x = (x | (x << 4)) & 0x10c30c30c30c30c3ull;
  x = (x | (x << 2)) & 0x1249249249249249ull;
  return x;
}

__device__ __forceinline__ unsigned quant(float c, float lo, float scale, unsigned maxq) {
  float f = (c - lo) * scale;
  f = fminf(fmaxf(f, 0.0f), (float)maxq);
  return (unsigned)f;
}

// The step-invariant part of the unsorted FP32 SoA, written once per context:
// the direction rounded to FP32 with the photon's index in w (dir_u), and the
// energy in FP32 (pos_u's w; the propagation rewrites only x, y, z).  GB300's
// FP64 pipe is narrow, and these conversions were half of the propagation's
// FP64 instructions.
__global__ void __launch_bounds__(256) k_static_soa(TLBeam b, float4 *pos_u, float4 *dir_u) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < b.n;
       i += (int64_t)gridDim.x * blockDim.x) {
    dir_u[i] = make_float4(__double2float_rn(b.dx[i]), __double2float_rn(b.dy[i]),
                           __double2float_rn(b.dz[i]), __int_as_float((int)i));
    pos_u[i] = make_float4(0.0f, 0.0f, 0.0f, __double2float_rn(b.E[i]));
  }
}

cudaError_t launch_static_soa(const TLBeam &b, BuildBufs &w, cudaStream_t s) {
  if (b.n <= 0) return cudaSuccess;
  const int64_t nb = (b.n + 255) / 256;
  k_static_soa<<<(unsigned)(nb < 8 * 152 ? nb : 8 * 152), 256, 0, s>>>(b, w.pos_u, w.dir_u);
  return cudaGetLastError();
}

// Propagate p = p0 + c t_k d in FP64 (closed form), round to the FP32 SoA,
// and key every photon by the Morton code of its swept box's centre in the
// box (lo, scale).  With passes > 0 also counts the
// 8-bit digits of every radix-sort pass (the sort's histogram) in shared
// memory, flushed once per block into the zeroed raw histogram.  A fixed
// grid of at most kPropBlocks blocks, grid-stride.
constexpr int kPropBlocks = 4 * 152;

__global__ void __launch_bounds__(256) k_propagate(TLBeam b, double ct, float halfL, float3 lo,
                                                   float3 scale, unsigned maxq, float4 *pos_u,
                                                   float4 *dir_u, unsigned long long *key,
                                                   int passes, uint32_t *hist) {
  __shared__ uint32_t sh[8][256];
  if (passes > 0) {
    for (int t = threadIdx.x; t < 8 * 256; t += 256) (&sh[0][0])[t] = 0u;
    __syncthreads();
  }
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < b.n;
       i += (int64_t)gridDim.x * blockDim.x) {
    const double dx = b.dx[i], dy = b.dy[i], dz = b.dz[i];
    const double Px = __dadd_rn(b.px[i], __dmul_rn(ct, dx));
    const double Py = __dadd_rn(b.py[i], __dmul_rn(ct, dy));
    const double Pz = __dadd_rn(b.pz[i], __dmul_rn(ct, dz));
    const float3 p = make_float3(__double2float_rn(Px), __double2float_rn(Py),
                                 __double2float_rn(Pz));
    const float4 d = dir_u[i];  // the FP32 direction, written once (k_static_soa)
    float *pu = reinterpret_cast<float *>(pos_u + i);  // x, y, z; w holds the energy
    *reinterpret_cast<float2 *>(pu) = make_float2(p.x, p.y);
    pu[2] = p.z;
    const unsigned qx = quant(fmaf(halfL, d.x, p.x), lo.x, scale.x, maxq),
                   qy = quant(fmaf(halfL, d.y, p.y), lo.y, scale.y, maxq),
                   qz = quant(fmaf(halfL, d.z, p.z), lo.z, scale.z, maxq);
    const unsigned long long k = (spread3(qx) << 2) | (spread3(qy) << 1) | spread3(qz);
    key[i] = k;
    for (int q = 0; q < passes; ++q) atomicAdd(&sh[q][(k >> (8 * q)) & 255u], 1u);
  }
  if (passes > 0) {
    __syncthreads();
    for (int t = threadIdx.x; t < passes * 256; t += 256) {
      const uint32_t v = (&sh[0][0])[t];
      if (v) atomicAdd(&hist[t], v);
    }
  }
}

cudaError_t launch_propagate(const TLBeam &b, double ct, float L, const float box_lo[3],
                             const float box_scale[3], int bits, BuildBufs &w, int passes,
                             cudaStream_t s) {
  if (b.n <= 0) return cudaSuccess;
  unsigned maxq = (1u << bits) - 1u;
  const int64_t nb = (b.n + 255) / 256;
  const int blocks = (int)(nb < kPropBlocks ? nb : kPropBlocks);
  k_propagate<<<blocks, 256, 0, s>>>(
      b, ct, 0.5f * L, make_float3(box_lo[0], box_lo[1], box_lo[2]),
      make_float3(box_scale[0], box_scale[1], box_scale[2]), maxq, w.pos_u, w.dir_u, w.key[0],
      passes, w.sort_raw);
  return cudaGetLastError();
}

// ---------------------------------------------------------------- gather

// a single photon needs no sort
__global__ void __launch_bounds__(256) k_gather(int64_t n, const float4 *__restrict__ pos_u,
                                                const float4 *__restrict__ dir_u,
                                                float4 *__restrict__ pos, float4 *__restrict__ dir,
                                                const unsigned *build_status) {
  int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= n || (*build_status & TL_ST_TIMEOUT)) return;
  pos[i] = pos_u[i];
  dir[i] = dir_u[i];
}

cudaError_t launch_gather(BuildBufs &w, int64_t n, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  k_gather<<<(int)((n + 255) / 256), 256, 0, s>>>(n, w.pos_u, w.dir_u, w.pos, w.dir,
                                                  w.build_status);
  return cudaGetLastError();
}

// ---------------------------------------------------------------- Karras

// common prefix length of sorted keys i and j (ki = key i); equal keys fall
// back to the indices (so every key is distinct); -1 outside [0, n).  32-bit
// indices: a beam holds fewer than 2^27 photons.
__device__ __forceinline__ int kdelta(const unsigned long long *__restrict__ key, int n, int i,
                                      unsigned long long ki, int j) {
  if ((unsigned)j >= (unsigned)n) return -1;
  const unsigned long long kj = __ldg(key + j);
  return ki != kj ? __clzll((long long)(ki ^ kj)) : 64 + __clz(i ^ j);
}

__device__ __forceinline__ void empty_box(float4 &b1, float4 &b2) {
  // box 1 of the super root: lo = +inf, hi = -inf never overlaps
  const float inf = __int_as_float(0x7f800000);
  b1.z = inf;
  b1.w = inf;
  b2 = make_float4(inf, -inf, -inf, -inf);
}

__global__ void __launch_bounds__(256) k_karras(const unsigned long long *__restrict__ key,
                                                int64_t n, int bucket, TLNode *nodes,
                                                uint32_t *parent_leaf, uint32_t *parent_node,
                                                const unsigned *build_status, uint32_t *nfirst,
                                                uint32_t *nlast, uint8_t *nlev, int key_bits) {
  int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (*build_status & TL_ST_TIMEOUT) return;  // keys unsorted: the build is abandoned
  const uint32_t super = (uint32_t)(n > 1 ? n - 1 : 0);
  if (i == 0) {
    // the super root: one child (the whole beam) in slot 0, slot 1 empty
    TLNode sr;
    sr.b0 = make_float4(0.f, 0.f, 0.f, 0.f);
    sr.b1 = make_float4(0.f, 0.f, 0.f, 0.f);
    empty_box(sr.b1, sr.b2);
    const bool root_bucket = n <= bucket;
    int ref0 = root_bucket ? (int)(TL_FLAG | 0u) : 0;
    sr.c = make_int4(ref0, (int)TL_NONE, (int)n, 0);
    // boxes are written by the refit; write refs and the empty slot now
    nodes[super] = sr;
    if (n > 1) parent_node[0] = (super << 1) | 0u;
    else parent_leaf[0] = (super << 1) | 0u;
    nfirst[super] = 0u;
    nlast[super] = (uint32_t)(n - 1);
    nlev[super] = 0;
  }
  if (i >= n - 1) return;
  const int n32 = (int)n, i32 = (int)i;
  const unsigned long long ki = __ldg(key + i32);
  const int dl = kdelta(key, n32, i32, ki, i32 - 1), dr = kdelta(key, n32, i32, ki, i32 + 1);
  const int d = dr > dl ? 1 : -1;
  const int dmin = dr > dl ? dl : dr;
  int lmax = 2;
  while (kdelta(key, n32, i32, ki, i32 + lmax * d) > dmin) lmax <<= 1;
  int l = 0;
  for (int t = lmax >> 1; t >= 1; t >>= 1)
    if (kdelta(key, n32, i32, ki, i32 + (l + t) * d) > dmin) l += t;
  const int j32 = i32 + l * d;
  const int dnode = kdelta(key, n32, i32, ki, j32);
  int s = 0, t = l;
  do {
    t = (t + 1) >> 1;
    if (kdelta(key, n32, i32, ki, i32 + (s + t) * d) > dnode) s += t;
  } while (t > 1);
  const int64_t j = j32;
  int64_t gamma = i32 + s * d + (d < 0 ? -1 : 0);
  int64_t first = i < j ? i : j, last = i < j ? j : i;
  int64_t cl = gamma - first + 1, cr = last - gamma;
  nfirst[i] = (uint32_t)first;
  nlast[i] = (uint32_t)last;
  {
    const int lev = dnode - (64 - key_bits);  // equal keys: beyond key_bits
    nlev[i] = (uint8_t)(lev < 0 ? 0 : (lev > 255 ? 255 : lev));
  }
  int refl = cl <= bucket ? (int)(TL_FLAG | (uint32_t)first) : (int)gamma;
  int refr = cr <= bucket ? (int)(TL_FLAG | (uint32_t)(gamma + 1)) : (int)(gamma + 1);
  nodes[i].c = make_int4(refl, refr, (int)cl, (int)cr);
  if (first == gamma) parent_leaf[gamma] = ((uint32_t)i << 1) | 0u;
  else parent_node[gamma] = ((uint32_t)i << 1) | 0u;
  if (last == gamma + 1) parent_leaf[gamma + 1] = ((uint32_t)i << 1) | 1u;
  else parent_node[gamma + 1] = ((uint32_t)i << 1) | 1u;
}

cudaError_t launch_karras(BuildBufs &w, int64_t n, int sel, int bucket, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  int64_t threads = n > 1 ? n - 1 : 1;
  k_karras<<<(int)((threads + 255) / 256), 256, 0, s>>>(w.key[sel], n, bucket, w.nodes,
                                                        w.parent_leaf, w.parent_node,
                                                        w.build_status, w.nfirst, w.nlast,
                                                        w.nlev, w.key_bits);
  return cudaGetLastError();
}

// ---------------------------------------------------------------- refit

// slot 0 = floats 0..5 of the record (b0, b1.xy), slot 1 = floats 6..11
// (b1.zw, b2): one 16-byte and one 8-byte store each
__device__ __forceinline__ void write_slot(TLNode *nodes, uint32_t node, uint32_t slot,
                                           const TLBox &b) {
  TLNode &r = nodes[node];
  if (slot == 0u) {
    r.b0 = make_float4(b.lx, b.ly, b.lz, b.hx);
    *reinterpret_cast<float2 *>(&r.b1.x) = make_float2(b.hy, b.hz);
  } else {
    *reinterpret_cast<float2 *>(&r.b1.z) = make_float2(b.lx, b.ly);
    r.b2 = make_float4(b.lz, b.hx, b.hy, b.hz);
  }
}

// Refit as range unions.  Every subtree of the Karras hierarchy holds a
// contiguous range [f, l] of the Morton-ordered photons, so its box is the
// union (FP32 min / max: exact, order-free) of the photons' swept boxes over
// that range, and every node can be finished on its own, with no bottom-up
// chain of waits:
//   k_refit_tile   one block per tile of kRTile photons: the tile's leaf boxes
//                  in a shared-memory sparse table (level j holds the unions of
//                  2^j consecutive boxes), so a range inside the tile is the
//                  union of two entries.  Writes every photon's box into its
//                  parent's slot, the box of every node whose range lies in
//                  the tile into its parent's slot, the prefix and suffix
//                  unions of every photon within its tile, and the tile box.
//   k_refit_super  one block per kRSuper tiles: the same table over tile boxes.
//   k_refit_cross  nodes whose range spans tiles: suffix of the first tile +
//                  the tiles in between (two table entries per super-tile
//                  end, plus whole super-tiles) + prefix of the last tile.
// A node's range: f = first photon (written by the emit), l = f + both child
// counts - 1.  A Karras node's index is one end of its range, so a node whose
// range lies in a tile has its index there too.
constexpr int kRTile = 256, kRTileLev = 8;  // levels 0..7 cover ranges of up to 256
constexpr int kRSuper = 512, kRSuperLog = 9;

struct Box6 {
  float v[6];  // lo xyz, hi xyz
};

__device__ __forceinline__ Box6 empty6() {
  const float inf = __int_as_float(0x7f800000);
  Box6 b;
  b.v[0] = b.v[1] = b.v[2] = inf;
  b.v[3] = b.v[4] = b.v[5] = -inf;
  return b;
}

__device__ __forceinline__ void join6(Box6 &a, const Box6 &b) {
  a.v[0] = fminf(a.v[0], b.v[0]);
  a.v[1] = fminf(a.v[1], b.v[1]);
  a.v[2] = fminf(a.v[2], b.v[2]);
  a.v[3] = fmaxf(a.v[3], b.v[3]);
  a.v[4] = fmaxf(a.v[4], b.v[4]);
  a.v[5] = fmaxf(a.v[5], b.v[5]);
}

__device__ __forceinline__ TLBox to_box(const Box6 &b) {
  TLBox t;
  t.lx = b.v[0];
  t.ly = b.v[1];
  t.lz = b.v[2];
  t.hx = b.v[3];
  t.hy = b.v[4];
  t.hz = b.v[5];
  return t;
}

// shared-memory sparse table: tab[(j * 6 + q) * W + i], W entries per level
template <int W>
__device__ __forceinline__ Box6 tab_get(const float *tab, int j, int i) {
  Box6 b;
#pragma unroll
  for (int q = 0; q < 6; ++q) b.v[q] = tab[(j * 6 + q) * W + i];
  return b;
}

// union over [a, b]: two entries of level j = floor(log2(b - a + 1)), capped
// at the table's top level LEV - 1 (two top-level entries still cover any
// range of up to 2^LEV boxes)
template <int W, int LEV>
__device__ __forceinline__ Box6 tab_query(const float *tab, int a, int b) {
  const int j = min(31 - __clz(b - a + 1), LEV - 1);
  Box6 r = tab_get<W>(tab, j, a);
  join6(r, tab_get<W>(tab, j, b - (1 << j) + 1));
  return r;
}

// fills levels 1..LOG of a W-wide table whose level 0 is in place
template <int W, int LOG>
__device__ __forceinline__ void tab_build(float *tab) {
  for (int j = 1; j <= LOG; ++j) {
    const int h = 1 << (j - 1);
    for (int i = threadIdx.x; i + (1 << j) <= W; i += blockDim.x) {
#pragma unroll
      for (int q = 0; q < 6; ++q) {
        const float x = tab[((j - 1) * 6 + q) * W + i], y = tab[((j - 1) * 6 + q) * W + i + h];
        tab[(j * 6 + q) * W + i] = q < 3 ? fminf(x, y) : fmaxf(x, y);
      }
    }
    __syncthreads();
  }
}

__device__ __forceinline__ void put6(float *dst, const Box6 &b) {
  float2 *d2 = reinterpret_cast<float2 *>(dst);
  d2[0] = make_float2(b.v[0], b.v[1]);
  d2[1] = make_float2(b.v[2], b.v[3]);
  d2[2] = make_float2(b.v[4], b.v[5]);
}

__device__ __forceinline__ Box6 get6(const float *src) {
  const float2 *s2 = reinterpret_cast<const float2 *>(src);
  const float2 a = s2[0], b = s2[1], c = s2[2];
  Box6 r;
  r.v[0] = a.x;
  r.v[1] = a.y;
  r.v[2] = b.x;
  r.v[3] = b.y;
  r.v[4] = c.x;
  r.v[5] = c.y;
  return r;
}


__global__ void __launch_bounds__(kRTile) k_refit_tile(
    int64_t n, const float4 *__restrict__ pos, const float4 *__restrict__ dir, float Llo,
    float Lhi, float half, TLNode *nodes, const uint32_t *__restrict__ parent_leaf,
    const uint32_t *__restrict__ parent_node, const uint32_t *__restrict__ nfirst,
    const uint32_t *__restrict__ nlast, float *pre, float *suf, float *tilebox,
    unsigned *build_status) {
  extern __shared__ float tab[];  // kRTileLev levels x 6 x kRTile
  __shared__ unsigned abandoned;
  const int t = threadIdx.x;
  // one read for the whole block: other blocks of this kernel may set the flag
  if (t == 0) abandoned = *(volatile unsigned *)build_status & TL_ST_TIMEOUT;
  __syncthreads();
  if (abandoned) return;  // keys unsorted: the build is abandoned
  const int64_t base = blockIdx.x * (int64_t)kRTile;
  const int64_t p = base + t;
  const uint32_t super = (uint32_t)(n > 1 ? n - 1 : 0);
  const int cnt = n - base < kRTile ? (int)(n - base) : kRTile;
  // every global load first (they do not depend on the table)
  float4 ps = make_float4(0.f, 0.f, 0.f, 0.f), d = ps;
  uint32_t lref = 0u, nref = 0u;
  int64_t f = 0, l = -1;
  if (p < n) {
    ps = pos[p];
    d = dir[p];
    lref = parent_leaf[p];
  }
  const bool inner = p < (int64_t)super;  // the super root (index n - 1) has no parent
  if (inner) {
    f = nfirst[p];
    l = nlast[p];
    nref = parent_node[p];
  }
  Box6 b = empty6();
  if (p < n) {
    seg_axis(ps.x, d.x, Llo, Lhi, half, b.v[0], b.v[3]);
    seg_axis(ps.y, d.y, Llo, Lhi, half, b.v[1], b.v[4]);
    seg_axis(ps.z, d.z, Llo, Lhi, half, b.v[2], b.v[5]);
    if ((lref >> 1) <= super) write_slot(nodes, lref >> 1, lref & 1u, to_box(b));
    else atomicOr(build_status, (unsigned)TL_ST_BADTREE);
  }
#pragma unroll
  for (int q = 0; q < 6; ++q) tab[q * kRTile + t] = b.v[q];
  __syncthreads();
  tab_build<kRTile, kRTileLev - 1>(tab);
  if (p < n) {
    put6(pre + 6 * p, tab_query<kRTile, kRTileLev>(tab, 0, t));
    put6(suf + 6 * p, tab_query<kRTile, kRTileLev>(tab, t, cnt - 1));
  }
  if (t == 0) put6(tilebox + 6 * blockIdx.x, tab_query<kRTile, kRTileLev>(tab, 0, cnt - 1));
  // inner node p, if its range lies in the tile
  if (inner && f >= base && l < base + cnt) {
    if ((nref >> 1) <= super && f <= l)
      write_slot(nodes, nref >> 1, nref & 1u,
                 to_box(tab_query<kRTile, kRTileLev>(tab, (int)(f - base), (int)(l - base))));
    else atomicOr(build_status, (unsigned)TL_ST_BADTREE);
  }
}

// tables over tile boxes: stab[((s * (kRSuperLog + 1) + j) * kRSuper + i) * 6 + q]
__global__ void __launch_bounds__(kRSuper) k_refit_super(int64_t ntile, const float *tilebox,
                                                         float *stab,
                                                         const unsigned *build_status) {
  extern __shared__ float tab[];  // (kRSuperLog + 1) levels x 6 x kRSuper
  if (*build_status & TL_ST_TIMEOUT) return;
  const int64_t s = blockIdx.x, t0 = s * kRSuper;
  const int t = threadIdx.x;
  const Box6 b = t0 + t < ntile ? get6(tilebox + 6 * (t0 + t)) : empty6();
#pragma unroll
  for (int q = 0; q < 6; ++q) tab[q * kRSuper + t] = b.v[q];
  __syncthreads();
  tab_build<kRSuper, kRSuperLog>(tab);
  float *out = stab + s * (int64_t)(kRSuperLog + 1) * kRSuper * 6;
  for (int j = 0; j <= kRSuperLog; ++j)
    if (t + (1 << j) <= kRSuper) put6(out + ((int64_t)j * kRSuper + t) * 6, tab_get<kRSuper>(tab, j, t));
}

__device__ __forceinline__ Box6 super_query(const float *stab, int64_t s, int a, int b) {
  const float *tb = stab + s * (int64_t)(kRSuperLog + 1) * kRSuper * 6;
  const int j = 31 - __clz(b - a + 1);
  Box6 r = get6(tb + ((int64_t)j * kRSuper + a) * 6);
  join6(r, get6(tb + ((int64_t)j * kRSuper + b - (1 << j) + 1) * 6));
  return r;
}

// union of the tile boxes a..b (a <= b)
__device__ __forceinline__ Box6 tiles_union(const float *stab, int64_t a, int64_t b) {
  const int64_t s0 = a >> kRSuperLog, s1 = b >> kRSuperLog;
  const int a0 = (int)(a & (kRSuper - 1)), b1 = (int)(b & (kRSuper - 1));
  if (s0 == s1) return super_query(stab, s0, a0, b1);
  Box6 r = super_query(stab, s0, a0, kRSuper - 1);
  join6(r, super_query(stab, s1, 0, b1));
  for (int64_t s = s0 + 1; s < s1; ++s) join6(r, super_query(stab, s, 0, kRSuper - 1));
  return r;
}

__global__ void __launch_bounds__(256) k_refit_cross(int64_t n, TLNode *nodes,
                                                     const uint32_t *__restrict__ parent_node,
                                                     const uint32_t *__restrict__ nfirst,
                                                     const uint32_t *__restrict__ nlast,
                                                     const float *pre, const float *suf,
                                                     const float *stab, unsigned *build_status) {
  if (*build_status & TL_ST_TIMEOUT) return;
  const uint32_t super = (uint32_t)(n > 1 ? n - 1 : 0);
  for (int64_t x = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; x < (int64_t)super;
       x += (int64_t)gridDim.x * blockDim.x) {
    const int64_t f = nfirst[x], l = nlast[x];
    const int64_t t0 = f >> 8, t1 = l >> 8;
    if (t0 == t1) continue;  // finished by its tile
    if (f < 0 || l >= n || f > l) {
      atomicOr(build_status, (unsigned)TL_ST_BADTREE);
      continue;
    }
    Box6 b = get6(suf + 6 * f);
    join6(b, get6(pre + 6 * l));
    if (t1 - t0 >= 2) join6(b, tiles_union(stab, t0 + 1, t1 - 1));
    const uint32_t ref = parent_node[x];
    if ((ref >> 1) <= super) write_slot(nodes, ref >> 1, ref & 1u, to_box(b));
    else atomicOr(build_status, (unsigned)TL_ST_BADTREE);
  }
}

int64_t refit_tiles(int64_t n) { return (n + kRTile - 1) / kRTile; }
int64_t refit_supers(int64_t n) { return (refit_tiles(n) + kRSuper - 1) / kRSuper; }
size_t refit_super_floats(int64_t n) {
  return (size_t)refit_supers(n) * (kRSuperLog + 1) * kRSuper * 6;
}

cudaError_t refit_prepare() {
  cudaError_t e = cudaFuncSetAttribute(k_refit_tile, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       kRTileLev * 6 * kRTile * (int)sizeof(float));
  if (e) return e;
  return cudaFuncSetAttribute(k_refit_super, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (kRSuperLog + 1) * 6 * kRSuper * (int)sizeof(float));
}

cudaError_t launch_refit(BuildBufs &w, int64_t n, float Llo, float Lhi, float half, int n_sm,
                         cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  const int64_t tiles = refit_tiles(n), supers = refit_supers(n);
  k_refit_tile<<<(unsigned)tiles, kRTile, kRTileLev * 6 * kRTile * sizeof(float), s>>>(
      n, w.pos, w.dir, Llo, Lhi, half, w.nodes, w.parent_leaf, w.parent_node, w.nfirst, w.nlast,
      w.rpre, w.rsuf, w.rtile, w.build_status);
  if (tiles > 1) {
    k_refit_super<<<(unsigned)supers, kRSuper, (kRSuperLog + 1) * 6 * kRSuper * sizeof(float),
                    s>>>(tiles, w.rtile, w.rsuper, w.build_status);
    const int64_t nb = (n + 255) / 256;
    const int blocks = (int)(nb < 8 * n_sm ? nb : 8 * n_sm);
    k_refit_cross<<<blocks, 256, 0, s>>>(n, w.nodes, w.parent_node, w.nfirst, w.nlast, w.rpre,
                                         w.rsuf, w.rsuper, w.build_status);
  }
  return cudaGetLastError();
}

}  // namespace tl
