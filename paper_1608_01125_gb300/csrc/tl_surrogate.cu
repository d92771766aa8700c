// tl_surrogate.cu -- the statistical regime's node-pair level.
//
// The paper's ST regime treats macro-particles as continuous clouds and
// computes collision rates between whole clouds instead of testing single
// particles (Sec. 2.2).  Here the clouds are the hierarchy's nodes at level
// L (the first node on every path whose Morton prefix is at least L bits, or
// a leaf bucket): the dual traversal stops there and emits overlapping node
// pairs.  For each pair the kernels below gather 24 features (boxes, counts,
// weight sums and energy / direction moments from FP64 prefix sums over the
// Morton-ordered photons), a rate estimate of the ST form, and -- for
// training labels -- the exact yield of the pair, attributed hit by hit.
#include "tl_exact.cuh"
#include "tl_sur.h"

namespace tl {

__device__ __forceinline__ bool is_cut(const CutTree &T, uint32_t ref, int L) {
  return (ref & TL_FLAG) || T.nlev[ref] >= L;
}

__device__ __forceinline__ TLNode load_node(const TLNode *p) {
  const float4 *f = reinterpret_cast<const float4 *>(p);
  TLNode v;
  v.b0 = __ldg(f + 0);
  v.b1 = __ldg(f + 1);
  v.b2 = __ldg(f + 2);
  v.c = __ldg(reinterpret_cast<const int4 *>(f + 3));
  return v;
}

// box, first photon and count of the node a stack reference names
__device__ __forceinline__ void own(const CutTree &T, uint32_t ref, TLBox &box, uint32_t &first,
                                    uint32_t &cnt) {
  uint32_t parent, slot;
  if (ref & TL_FLAG) {
    parent = (ref & ~TL_FLAG) >> 1;
    slot = ref & 1u;
  } else {
    const uint32_t pn = T.parent_node[ref];
    parent = pn >> 1;
    slot = pn & 1u;
  }
  const TLNode v = load_node(T.nodes + parent);
  box = tl_child_box(v, (int)slot);
  cnt = (uint32_t)(slot ? v.c.w : v.c.z);
  const uint32_t cr = (uint32_t)(slot ? v.c.y : v.c.x);
  first = (ref & TL_FLAG) ? (cr & ~TL_FLAG) : T.nfirst[ref];
}

// child `slot` of inner node `ref`: box and stack reference
__device__ __forceinline__ void child(const CutTree &T, uint32_t ref, int slot, TLBox &box,
                                      uint32_t &cref) {
  const TLNode v = load_node(T.nodes + ref);
  box = tl_child_box(v, slot);
  const uint32_t cr = (uint32_t)(slot ? v.c.y : v.c.x);
  cref = (cr & TL_FLAG) ? (TL_FLAG | (ref << 1) | (uint32_t)slot) : cr;
}

// ------------------------------------------------------------ prefix moments

// Six running sums over the photons in sorted order (w, w lnE, w lnE^2, w d) in FP64, from
// which the moments of a node's contiguous range are a difference.  The order of the
// additions is part of the result (the spread of a small cloud's energies is what is left
// of two large numbers), and it is: blocks of 1024 photons, whose sums are a strided loop
// and a butterfly; a running sum over the blocks; in a block a running sum over its
// 32-photon chunks; in a chunk the Kogge-Stone scan.
//
// GB300's FP64 pipe does 2 operations per clock and SM, so what counts is the additions.
// Scanning every chunk takes 30 per photon, and only the sums at the ends of cut nodes
// are ever read: those lie where the LCA of neighbours is above level L, which their keys
// tell.  So a chunk's total is the balanced tree that the scan's last lane computes (31
// additions per chunk and sum), and the scan's value at another lane l is the same tree
// over the photons l, l - 1, .. of the chunk, evaluated at such ends alone, each by one
// thread.  2 x 1e6 photons: 433 us before (a pass for the blocks, a scan of them,
// a pass of warp scans), now 62 for the blocks, the larger of 50 and 89 for their scan and
// the tiles side by side, and 12 for the chunks.
constexpr int kPreBlock = 1024, kPreThreads = 256, kPreHalf = 3;  // kPreHalf sums at a time

// An FP32 value in FP64 by its bits (exact); the conversion instruction shares the FP64 pipe.
__device__ __forceinline__ double widen(float x) {
  const unsigned u = __float_as_uint(x), e = u & 0x7f800000u;
  if ((u << 1) == 0u) return __hiloint2double((int)u, 0);
  if (e == 0u || e == 0x7f800000u) return (double)x;  // subnormal, infinity, NaN
  return __hiloint2double((int)((u & 0x80000000u) | (((u & 0x7fffffffu) >> 3) + 0x38000000u)),
                          (int)(u << 29));
}

// balanced tree over get(0) .. get(31), neighbours first
template <int K, class F>
__device__ __forceinline__ double tree_sum(const F &get, int j) {
  if constexpr (K == 0) return get(j);
  else
    return __dadd_rn(tree_sum<K - 1>(get, j), tree_sum<K - 1>(get, j + (1 << (K - 1))));
}

// level of the LCA of the sorted photons p and p + 1 (see the emit of the hierarchy)
__device__ __forceinline__ int split_level(const unsigned long long *key, int64_t p, int key_bits) {
  const unsigned long long x = key[p] ^ key[p + 1];
  const int d = x ? __clzll((long long)x) : 64 + __clz((int)p ^ (int)(p + 1));
  return d - (64 - key_bits);
}

// energy (w) and direction of the sorted photons t, t + 256, .. of a block from the FP32
// SoA, their weights from the FP64 input (0 past the end)
__device__ __forceinline__ void load_photons(const PreBeam &a, int64_t p0, float4 d[4],
                                             double w[4]) {
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const int64_t p = p0 + k * kPreThreads;
    d[k] = make_float4(0.f, 0.f, 0.f, 1.0f);
    w[k] = 0.0;
    if (p < a.n) {
      d[k] = a.dir[p];
      const uint32_t i = __float_as_uint(d[k].w);
      d[k].w = a.pos[p].w;
      if (i < a.n) w[k] = a.w ? a.w[i] : 1.0;
    }
  }
}

// terms 0..2 (h = 0) or 3..5 of a photon
template <int H>
__device__ __forceinline__ void terms(const float4 &d, double w, double v[kPreHalf]) {
  if constexpr (H == 0) {
    const double le = widen(logf(d.w));
    v[0] = w;
    v[1] = w * le;
    v[2] = w * le * le;
  } else {
    v[0] = w * widen(d.x);
    v[1] = w * widen(d.y);
    v[2] = w * widen(d.z);
  }
}

// the blocks' sums
__global__ void __launch_bounds__(kPreThreads) k_pre_blocks(PreBeam a0, PreBeam a1) {
  const PreBeam &a = blockIdx.y ? a1 : a0;
  const PreSums &P = a.sums;
  if (blockIdx.x >= P.blocks) return;
  __shared__ double acc[6][8 * 33];  // the threads' sums, then their warps'
  const int t = threadIdx.x;
  float4 d[4];
  double w[4], sum[6] = {0, 0, 0, 0, 0, 0}, v[6];
  load_photons(a, (int64_t)blockIdx.x * kPreBlock + t, d, w);
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    terms<0>(d[k], w[k], v);
    terms<1>(d[k], w[k], v + 3);
#pragma unroll
    for (int c = 0; c < 6; ++c) sum[c] += v[c];
  }
#pragma unroll
  for (int c = 0; c < 6; ++c) acc[c][(t >> 5) * 33 + (t & 31)] = sum[c];
  __syncthreads();
  if (t < 48) {
    double *x = acc[t >> 3] + (t & 7) * 33;
    x[32] = tree_sum<5>([&](int i) { return x[__brev((unsigned)i) >> 27]; }, 0);
  }
  __syncthreads();
  if (t < 6) {
    double s = 0.0;
    for (int q = 0; q < 8; ++q) s = __dadd_rn(s, acc[t][q * 33 + 32]);
    P.bsum[(int64_t)t * P.blocks + blockIdx.x] = s;
  }
}

// A running sum over the blocks, in place: equal runs per thread, then one chain of
// additions over the threads, in registers between shared loads.  One block per sum and
// beam, beside k_pre_tile: an addition waits ~100 clocks for the one before, and twice that
// where other warps use the SM's FP64 pipe, so a block takes an SM's shared memory to
// itself (50 us for 977 blocks of photons against 105).
constexpr int kScanShared = 200 << 10;

__global__ void __launch_bounds__(1024) k_pre_scan(PreSums s0, PreSums s1) {
  const PreSums &P = blockIdx.y ? s1 : s0;
  extern __shared__ double part[];  // 1024 used
  const int64_t nb = P.blocks, per = (nb + 1023) / 1024;
  double *bs = P.bsum + (int64_t)blockIdx.x * nb;
  const int64_t lo = min(threadIdx.x * per, nb), hi = min(lo + per, nb);
  double run = 0.0;
  for (int64_t b = lo; b < hi; ++b) run = __dadd_rn(run, bs[b]);
  part[threadIdx.x] = run;
  __syncthreads();
  if (threadIdx.x == 0) {
    const int used = (int)((nb + per - 1) / per);
    double t = 0.0;
    for (int q = 0; q < used; q += 16) {  // entries past `used` are zeros of idle threads
      double x[16];
#pragma unroll
      for (int i = 0; i < 16; ++i) x[i] = part[q + i];
#pragma unroll
      for (int i = 0; i < 16; ++i) {
        part[q + i] = t;
        t = __dadd_rn(t, x[i]);
      }
    }
  }
  __syncthreads();
  run = part[threadIdx.x];
  for (int64_t b = lo; b < hi; ++b) {
    const double v = bs[b];
    bs[b] = run;
    run = __dadd_rn(run, v);
  }
}

// the sums inside a block of photons: the chunks' totals and those at the ends of cut nodes
__global__ void __launch_bounds__(kPreThreads, 5) k_pre_tile(PreBeam a0, PreBeam a1, int L) {
  const PreBeam &a = blockIdx.y ? a1 : a0;
  const PreSums &P = a.sums;
  __shared__ double m[kPreHalf][32 * 33];  // the block's photons, 33 entries per chunk
  __shared__ unsigned short ends[kPreBlock];
  __shared__ unsigned nends;
  const int64_t block = blockIdx.x, b0 = block * kPreBlock;
  if (block >= P.blocks) return;
  const int t = threadIdx.x;
  if (t == 0) nends = 0u;
  __syncthreads();
  float4 d[4];
  double w[4];
  load_photons(a, b0 + t, d, w);
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const int64_t p = b0 + t + k * kPreThreads;
    if (p < a.n && (p == a.n - 1 || split_level(a.key, p, a.key_bits) < L))
      ends[atomicAdd(&nends, 1u)] = (unsigned short)(t + k * kPreThreads);
  }
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    __syncthreads();
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int i = t + k * kPreThreads, at = (i >> 5) * 33 + (i & 31);
      double v[kPreHalf];
      if (h == 0) terms<0>(d[k], w[k], v);
      else terms<1>(d[k], w[k], v);
#pragma unroll
      for (int c = 0; c < kPreHalf; ++c) m[c][at] = v[c];
    }
    __syncthreads();
    // one tree per thread: the chunks' totals, then the ends
    const int total = kPreHalf * (32 + (int)nends);
    for (int q = t; q < total; q += kPreThreads) {
      if (q < kPreHalf * 32) {
        const int c = q >> 5, j = q & 31;
        const double *x = m[c] + j * 33;
        P.tot[((int64_t)(h * kPreHalf + c) * 32 + j) * P.blocks + block] =
            tree_sum<5>([&](int i) { return x[i]; }, 0);
      } else {
        const int e = (q - kPreHalf * 32) / kPreHalf, c = q % kPreHalf;
        const int i0 = ends[e], l = i0 & 31;
        const double *x = m[c] + (i0 >> 5) * 33 + l;
        P.end[(b0 + i0 + 1) * 6 + h * kPreHalf + c] =
            tree_sum<5>([&](int i) { return i <= l ? x[-i] : 0.0; }, 0);
      }
    }
  }
}

// from a block's running sum those of its chunks, in place (a thread per block and sum)
__global__ void __launch_bounds__(64) k_pre_chunks(PreSums s0, PreSums s1) {
  const PreSums &P = blockIdx.z ? s1 : s0;
  const int64_t b = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (b >= P.blocks) return;
  double *tot = P.tot + (int64_t)blockIdx.y * 32 * P.blocks + b;
  double r = P.bsum[blockIdx.y * P.blocks + b];
#pragma unroll
  for (int j = 0; j < 32; ++j) {
    const double x = tot[j * P.blocks];
    tot[j * P.blocks] = r;
    r = __dadd_rn(r, x);
  }
}

// running sum c up to the sorted position p (0 at the front), an end of a cut node
__device__ __forceinline__ double run_sum(const PreSums &P, int64_t p, int c) {
  if (p == 0) return 0.0;
  const int64_t q = p - 1;
  return __dadd_rn(P.tot[((int64_t)c * 32 + ((q >> 5) & 31)) * P.blocks + (q >> 10)],
                   P.end[p * 6 + c]);
}

static int64_t pre_blocks(int64_t n) { return n > 0 ? (n + kPreBlock - 1) / kPreBlock : 1; }

size_t pre_doubles(int64_t n) { return (size_t)(6 * (n + 1) + 6 * 33 * pre_blocks(n)); }

PreSums pre_sums(double *buf, int64_t n) {
  PreSums P;
  P.blocks = pre_blocks(n);
  P.bsum = buf;
  P.tot = P.bsum + 6 * P.blocks;
  P.end = P.tot + 6 * 32 * P.blocks;
  return P;
}

cudaError_t prefix_prepare() {
  return cudaFuncSetAttribute(k_pre_scan, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              kScanShared);
}

cudaError_t launch_prefix_moments(const PreBeam &a, const PreBeam &b, int L, cudaStream_t s,
                                  cudaStream_t side, cudaEvent_t blocks_ev,
                                  cudaEvent_t tile_ev) {
  const int64_t t = a.sums.blocks > b.sums.blocks ? a.sums.blocks : b.sums.blocks;
  k_pre_blocks<<<dim3((unsigned)t, 2), kPreThreads, 0, s>>>(a, b);
  cudaError_t e = cudaEventRecord(blocks_ev, s);
  if (!e) e = cudaStreamWaitEvent(side, blocks_ev, 0);
  if (e) return e;
  // on the stream's own successor, which starts before what waits for an event: the scan
  // needs its SMs before the tiles' blocks are on all of them
  k_pre_scan<<<dim3(6, 2), 1024, kScanShared, s>>>(a.sums, b.sums);
  k_pre_tile<<<dim3((unsigned)t, 2), kPreThreads, 0, side>>>(a, b, L);
  e = cudaEventRecord(tile_ev, side);
  if (!e) e = cudaStreamWaitEvent(s, tile_ev, 0);
  if (e) return e;
  k_pre_chunks<<<dim3((unsigned)((t + 63) / 64), 6, 2), 64, 0, s>>>(a.sums, b.sums);
  return cudaGetLastError();
}

// ------------------------------------------------------------ level-L cut traversal

__device__ __forceinline__ void append(bool pred, uint2 v, uint2 *buf, unsigned *cnt,
                                       unsigned cap, unsigned *status, int lane) {
  const unsigned m = __ballot_sync(0xffffffffu, pred);
  if (!m) return;
  unsigned base = 0;
  if (lane == 0) base = atomicAdd(cnt, (unsigned)__popc(m));
  base = __shfl_sync(0xffffffffu, base, 0);
  if (pred) {
    const unsigned idx = base + __popc(m & ((1u << lane) - 1u));
    if (idx < cap) buf[idx] = v;
    else atomicOr(status, (unsigned)TL_ST_FRONT_OVF);
  }
}

// One breadth-first level: pairs whose both sides are cut nodes are emitted;
// otherwise the non-cut sides are split and the overlapping child pairs go
// to the next level.
__global__ void __launch_bounds__(256) k_cut_level(CutArgs a) {
  if (*a.build_status & (TL_ST_TIMEOUT | TL_ST_BADTREE)) return;  // no valid links to follow
  const unsigned nin = min(a.counts[0], a.cap);
  const int lane = threadIdx.x & 31;
  const unsigned nround = (nin + 31u) & ~31u;
  for (unsigned i = blockIdx.x * blockDim.x + threadIdx.x; i < nround;
       i += gridDim.x * blockDim.x) {
    const bool valid = i < nin;
    const uint2 pr = valid ? a.in[i] : make_uint2(0u, 0u);
    const bool ca = valid && is_cut(a.A, pr.x, a.L), cb = valid && is_cut(a.B, pr.y, a.L);
    // emit finished pairs
    {
      const bool done = valid && ca && cb;
      const unsigned m = __ballot_sync(0xffffffffu, done);
      if (m) {
        unsigned base = 0;
        if (lane == 0) base = atomicAdd(a.cut_count, (unsigned)__popc(m));
        base = __shfl_sync(0xffffffffu, base, 0);
        if (done) {
          const unsigned idx = base + __popc(m & ((1u << lane) - 1u));
          if (idx < a.cut_cap) a.cut[idx] = make_uint4(pr.x, pr.y, 0u, 0u);
          else atomicOr(a.status, (unsigned)TL_ST_FRONT_OVF);
        }
      }
    }
    const bool split = valid && !(ca && cb);
    TLBox ba, bb;
    uint32_t fa = 0, na = 0, fb = 0, nb = 0;
    if (split && ca) own(a.A, pr.x, ba, fa, na);
    if (split && cb) own(a.B, pr.y, bb, fb, nb);
    for (int combo = 0; combo < 4; ++combo) {
      const int ia = combo >> 1, ib = combo & 1;
      bool ok = false;
      uint2 o = make_uint2(0u, 0u);
      if (split && !(ca && ia) && !(cb && ib)) {
        TLBox xa = ba, xb = bb;
        uint32_t ra = pr.x, rb = pr.y;
        if (!ca) child(a.A, pr.x, ia, xa, ra);
        if (!cb) child(a.B, pr.y, ib, xb, rb);
        ok = tl_overlap(xa, xb);
        o = make_uint2(ra, rb);
      }
      append(ok, o, a.out, a.counts + 1, a.cap, a.status, lane);
    }
  }
}

cudaError_t launch_cut_level(const CutArgs &a, int blocks, cudaStream_t s) {
  k_cut_level<<<blocks, 256, 0, s>>>(a);
  return cudaGetLastError();
}

// ------------------------------------------------------------ features

// The ST regime's rate for two clouds (Sec. 2.2, Eq. rate, Eq. reactivity).
// A cloud is a level-L node read as a box of uniform density moving rigidly
// with the mean velocity c dbar: its box at t_k is the node's swept box with
// the step's travel c dt dbar taken off, so that it sweeps the node's box
// over the step.  n_I n_II <sigma v> integrated over the overlap and the step:
//   N = W_A W_B (1e12 kappa sigma(sbar)) c |dbar_A - dbar_B|
//       * int_0^dt V_ov(t) dt / (V_A V_B),
// with the collision area 1e12 kappa sigma [um^2] and sbar from the
// geometric-mean energies and 1 - dbar_A . dbar_B.  V_ov(t) is the product of
// three piecewise-linear overlap lengths: the integral is exact, Simpson's
// rule on each piece between the times where an overlap length changes form.

// Along an axis the overlap length is min(w, p + r t, q - r t), the least width and the
// distances of the two outer ends closing with the relative velocity r, inside the times
// where that is positive; the pieces meet where p + r t or q - r t is w.
struct StAxis {
  double p, q, r, w;
};

// Minimum and maximum by the bits: two doubles of which at most one is negative order as
// their bit patterns do as integers, and integer comparisons leave the FP64 pipe free.
__device__ __forceinline__ double bit_min(double a, double b) {
  return __longlong_as_double(min(__double_as_longlong(a), __double_as_longlong(b)));
}

__device__ __forceinline__ double bit_max(double a, double b) {
  return __longlong_as_double(max(__double_as_longlong(a), __double_as_longlong(b)));
}

__device__ __forceinline__ bool sign_bit(double a) { return __double2hiint(a) < 0; }

// (p + r t and q - r t add up to the two widths: at most one is negative)
__device__ __forceinline__ double st_vol(const StAxis ax[3], double t) {
  double v = 1.0;
#pragma unroll
  for (int k = 0; k < 3; ++k)
    v *= bit_min(ax[k].w, bit_min(fma(ax[k].r, t, ax[k].p), fma(-ax[k].r, t, ax[k].q)));
  return v;
}

__device__ __forceinline__ void st_order(double &a, double &b) {
  const double lo = bit_min(a, b), hi = bit_max(a, b);
  a = lo;
  b = hi;
}

// Exact integral of the overlap volume over [0, T]: the support of all three lengths, cut
// at the (at most six) times between pieces.  FP64 bound: one reciprocal per axis and at
// most seven pieces within the support, in registers (in absolute coordinates over all of
// [0, T] it was four divisions per axis, 13 pieces and a sort in local memory).
__device__ double st_overlap_time_integral(const StAxis ax[3], double T) {
  double t0 = 0.0, t1 = T, br[6];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const StAxis &x = ax[k];
    if (x.r == 0.0) {
      if (!(x.p > 0.0 && x.q > 0.0)) return 0.0;
      br[2 * k] = br[2 * k + 1] = T;
    } else {
      const double inv = 1.0 / x.r, a = -x.p * inv, b = x.q * inv;
      t0 = bit_max(t0, sign_bit(x.r) ? b : a);
      t1 = bit_min(t1, sign_bit(x.r) ? a : b);
      br[2 * k] = (x.w - x.p) * inv;
      br[2 * k + 1] = (x.q - x.w) * inv;
    }
  }
  if (!(t1 > t0)) return 0.0;
#pragma unroll
  for (int i = 0; i < 6; ++i) br[i] = bit_min(bit_max(br[i], t0), t1);
  // a sorting network of six
  st_order(br[0], br[5]);
  st_order(br[1], br[3]);
  st_order(br[2], br[4]);
  st_order(br[1], br[2]);
  st_order(br[3], br[4]);
  st_order(br[0], br[3]);
  st_order(br[2], br[5]);
  st_order(br[0], br[1]);
  st_order(br[2], br[3]);
  st_order(br[4], br[5]);
  st_order(br[1], br[2]);
  st_order(br[3], br[4]);
  double I = 0.0, ta = t0, fa = st_vol(ax, t0);
#pragma unroll
  for (int i = 0; i < 7; ++i) {
    const double tb = i < 6 ? br[i] : t1;
    if (__double_as_longlong(tb) > __double_as_longlong(ta)) {
      const double fb = st_vol(ax, tb);
      I += (tb - ta) * (fa + 4.0 * st_vol(ax, 0.5 * (ta + tb)) + fb);
      ta = tb;
      fa = fb;
    }
  }
  return I * (1.0 / 6.0);
}

// 24 features per node pair, and the ST rate above (FP64 from the FP32 node
// boxes and the FP64 prefix moments).  L = c dt [um].
// FP64 bound (some 40 operations per clock and SM below the FP32 rate): one reciprocal of
// each weight sum, the integral above; the row leaves in 16-byte stores.  Blocks of two
// warps spread a few ten thousand pairs evenly over the SMs.  47,493 pairs:
// 157 us before, 65 us now.
__global__ void __launch_bounds__(64) k_features(CutTree A, CutTree B, const uint4 *cut,
                                                 const unsigned *cut_count, unsigned cap,
                                                 float *feat, float *st, double L, double dt,
                                                 double kappa, const unsigned *build_status) {
  if (*build_status & (TL_ST_TIMEOUT | TL_ST_BADTREE)) return;  // no valid hierarchies
  const unsigned n = min(*cut_count, cap);
  for (unsigned p = blockIdx.x * blockDim.x + threadIdx.x; p < n; p += gridDim.x * blockDim.x) {
    const uint4 c = cut[p];
    TLBox ba, bb;
    uint32_t fa, na, fb, nb;
    own(A, c.x, ba, fa, na);
    own(B, c.y, bb, fb, nb);
    double ma[6], mb[6];
#pragma unroll
    for (int q = 0; q < 6; ++q) {
      ma[q] = run_sum(A.pre, (int64_t)fa + na, q) - run_sum(A.pre, fa, q);
      mb[q] = run_sum(B.pre, (int64_t)fb + nb, q) - run_sum(B.pre, fb, q);
    }
    float4 *f = reinterpret_cast<float4 *>(feat + (size_t)p * 24);
    const float cax = 0.5f * (ba.lx + ba.hx), cay = 0.5f * (ba.ly + ba.hy), caz = 0.5f * (ba.lz + ba.hz);
    const float cbx = 0.5f * (bb.lx + bb.hx), cby = 0.5f * (bb.ly + bb.hy), cbz = 0.5f * (bb.lz + bb.hz);
    f[0] = make_float4(cbx - cax, cby - cay, cbz - caz, 0.5f * (ba.hx - ba.lx));
    f[1] = make_float4(0.5f * (ba.hy - ba.ly), 0.5f * (ba.hz - ba.lz), 0.5f * (bb.hx - bb.lx),
                       0.5f * (bb.hy - bb.ly));
    const double swa = fmax(ma[0], 1e-300), swb = fmax(mb[0], 1e-300);
    const double iwa = 1.0 / swa, iwb = 1.0 / swb;
    f[2] = make_float4(0.5f * (bb.hz - bb.lz), logf((float)na), logf((float)nb), (float)log(swa));
    const double mla = ma[1] / swa, mlb = mb[1] / swb;
    f[3] = make_float4((float)log(swb), (float)mla, (float)mlb,
                       (float)sqrt(fmax(ma[2] / swa - mla * mla, 0.0)));
    const double dax = ma[3] * iwa, day = ma[4] * iwa, daz = ma[5] * iwa;
    const double dbx = mb[3] * iwb, dby = mb[4] * iwb, dbz = mb[5] * iwb;
    f[4] = make_float4((float)sqrt(fmax(mb[2] / swb - mlb * mlb, 0.0)), (float)dax, (float)day,
                       (float)daz);
    const double omc = 1.0 - (dax * dbx + day * dby + daz * dbz);
    f[5] = make_float4((float)dbx, (float)dby, (float)dbz, (float)omc);
    // the ST rate
    const double sbar = exp(mla + mlb) * omc / (2.0 * TL_MEC2 * TL_MEC2);
    const double sig = tl_sigma64(sbar);
    const float loA[3] = {ba.lx, ba.ly, ba.lz}, hiA[3] = {ba.hx, ba.hy, ba.hz};
    const float loB[3] = {bb.lx, bb.ly, bb.lz}, hiB[3] = {bb.hx, bb.hy, bb.hz};
    const double dA[3] = {dax, day, daz}, dB[3] = {dbx, dby, dbz};
    StAxis ax[3];
    double VA = 1.0, VB = 1.0, dv2 = 0.0;
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      const double DA = L * dA[q], DB = L * dB[q];
      const double la = widen(loA[q]) - (sign_bit(DA) ? DA : 0.0);
      const double ua = widen(hiA[q]) - (sign_bit(DA) ? 0.0 : DA);
      const double lb = widen(loB[q]) - (sign_bit(DB) ? DB : 0.0);
      const double ub = widen(hiB[q]) - (sign_bit(DB) ? 0.0 : DB);
      const double wa = ua - la, wb = ub - lb, r = TL_C * dA[q] - TL_C * dB[q];
      VA *= wa;
      VB *= wb;
      dv2 += r * r;
      ax[q].p = ua - lb;
      ax[q].q = ub - la;
      ax[q].r = r;
      ax[q].w = fmin(wa, wb);
    }
    double rate = 0.0;
    if (sig > 0.0 && VA > 0.0 && VB > 0.0) {
      const double I = st_overlap_time_integral(ax, dt);
      if (I > 0.0) rate = swa * swb * (1e12 * kappa * sig) * sqrt(dv2) * I / (VA * VB);
    }
    st[p] = (float)rate;
  }
}

cudaError_t launch_features(const CutTree &A, const CutTree &B, const uint4 *cut,
                            const unsigned *cut_count, unsigned cap, float *feat, float *st,
                            double dt, double kappa, const unsigned *build_status, int blocks,
                            cudaStream_t s) {
  k_features<<<blocks, 64, 0, s>>>(A, B, cut, cut_count, cap, feat, st, TL_C * dt, dt, kappa,
                                   build_status);
  return cudaGetLastError();
}

// ------------------------------------------------------------ exact labels

// The level-L frontier of one tree: inner nodes at or past level L whose
// parent is not, and leaf buckets of inner nodes before level L.  Each gets
// an id; every photon learns the id of the frontier node that holds it.
__global__ void k_frontier_mark(CutTree T, int L, uint32_t *cid_node, uint32_t *cid_slot,
                                uint2 *flist, unsigned *fcount, unsigned fcap) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int64_t ninner = T.n > 1 ? T.n - 1 : 0;
  if (i > ninner) return;  // inner nodes 0..n-2 and the super root (index n-1 or 0)
  const uint32_t node = (i == ninner) ? T.super : (uint32_t)i;
  if (node == T.super && i != ninner) return;
  const bool cut_here = node != T.super && T.nlev[node] >= L;
  if (cut_here) {
    TLBox b;
    uint32_t f, c;
    own(T, node, b, f, c);
    // a node of at most `bucket` photons is a leaf bucket or lies inside one:
    // buckets are frontier nodes through their parent's slot (below)
    if (c <= (uint32_t)T.bucket) return;
    const uint32_t pn = T.parent_node[node];
    const uint32_t parent = pn >> 1;
    const bool parent_cut = parent != T.super && T.nlev[parent] >= L;
    if (!parent_cut) {
      const unsigned id = atomicAdd(fcount, 1u);
      cid_node[node] = id;
      if (id < fcap) flist[id] = make_uint2(f, c);
    }
    return;
  }
  // not cut: its bucket children are frontier nodes -- unless the node is
  // itself a bucket or inside one (then its parent's slot names it)
  if (node != T.super) {
    TLBox b;
    uint32_t f, c;
    own(T, node, b, f, c);
    if (c <= (uint32_t)T.bucket) return;
  }
  const TLNode v = load_node(T.nodes + node);
  for (int slot = 0; slot < 2; ++slot) {
    const uint32_t cr = (uint32_t)(slot ? v.c.y : v.c.x);
    const uint32_t cnt = (uint32_t)(slot ? v.c.w : v.c.z);
    if ((cr & TL_FLAG) && cr != TL_NONE && cnt > 0) {
      const unsigned id = atomicAdd(fcount, 1u);
      cid_slot[2 * (size_t)node + slot] = id;
      if (id < fcap) flist[id] = make_uint2(cr & ~TL_FLAG, cnt);
    }
  }
}

// photon (sorted position) -> frontier id; one warp per frontier node
__global__ void k_frontier_fill(const uint2 *flist, const unsigned *fcount, unsigned fcap,
                                uint32_t *cut_of) {
  const unsigned nf = min(*fcount, fcap);
  const unsigned w = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  for (unsigned f = w; f < nf; f += (gridDim.x * blockDim.x) >> 5) {
    const uint2 r = flist[f];
    for (uint32_t p = r.x + lane; p < r.x + r.y; p += 32) cut_of[p] = f;
  }
}

// input index -> sorted position
__global__ void k_inverse(const float4 *dir, int64_t n, uint32_t *inv) {
  const int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (p < n) inv[__float_as_uint(dir[p].w)] = (uint32_t)p;
}

__device__ __forceinline__ uint32_t cid_of(const CutTree &T, uint32_t ref, const uint32_t *cid_node,
                                           const uint32_t *cid_slot) {
  if (ref & TL_FLAG) return cid_slot[2 * (size_t)((ref & ~TL_FLAG) >> 1) + (ref & 1u)];
  return cid_node[ref];
}

__device__ __forceinline__ uint32_t hash64(unsigned long long k) {
  k ^= k >> 33;
  k *= 0xff51afd7ed558ccdull;
  k ^= k >> 33;
  return (uint32_t)k;
}

// cut pair p: record (cidA, cidB) and insert key -> p into an open-addressing table
__global__ void k_pair_index(CutTree A, CutTree B, uint4 *cut, const unsigned *cut_count,
                             unsigned cap, const uint32_t *cnA, const uint32_t *csA,
                             const uint32_t *cnB, const uint32_t *csB, unsigned long long *hkey,
                             uint32_t *hval, unsigned hmask, unsigned *status) {
  const unsigned n = min(*cut_count, cap);
  for (unsigned p = blockIdx.x * blockDim.x + threadIdx.x; p < n; p += gridDim.x * blockDim.x) {
    uint4 c = cut[p];
    c.z = cid_of(A, c.x, cnA, csA);
    c.w = cid_of(B, c.y, cnB, csB);
    cut[p] = c;
    const unsigned long long key = ((unsigned long long)c.z << 32) | c.w;
    uint32_t h = hash64(key) & hmask;
    bool placed = false;
    for (unsigned probe = 0; probe <= hmask; ++probe) {
      const unsigned long long prev = atomicCAS(&hkey[h], ~0ull, key);
      if (prev == ~0ull || prev == key) {
        hval[h] = p;
        placed = true;
        break;
      }
      h = (h + 1) & hmask;
    }
    if (!placed) atomicOr(status, (unsigned)TL_ST_FRONT_OVF);
  }
}

// every hit adds w_i w_j to the label of the node pair that holds it
__global__ void k_attribute(const uint2 *hits, const unsigned long long *nhits,
                            unsigned long long hcap, const TLBeam mA, const TLBeam mB,
                            const uint32_t *invA, const uint32_t *invB, const uint32_t *cutA,
                            const uint32_t *cutB, const unsigned long long *hkey,
                            const uint32_t *hval, unsigned hmask, double *label,
                            unsigned *status) {
  const unsigned long long n = min(*nhits, hcap);
  for (unsigned long long t = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; t < n;
       t += (unsigned long long)gridDim.x * blockDim.x) {
    const uint2 h = hits[t];
    const unsigned long long key =
        ((unsigned long long)cutA[invA[h.x]] << 32) | cutB[invB[h.y]];
    uint32_t s = hash64(key) & hmask;
    bool found = false;
    for (unsigned probe = 0; probe <= hmask; ++probe) {
      const unsigned long long k = hkey[s];
      if (k == key) {
        const double w = (mA.w ? mA.w[h.x] : 1.0) * (mB.w ? mB.w[h.y] : 1.0);
        atomicAdd(&label[hval[s]], w);
        found = true;
        break;
      }
      if (k == ~0ull) break;
      s = (s + 1) & hmask;
    }
    if (!found) atomicOr(status, (unsigned)TL_ST_FRONT_OVF);
  }
}

cudaError_t launch_labels_prep(const CutTree &T, int L, uint32_t *cid_node, uint32_t *cid_slot,
                               uint2 *flist, unsigned *fcount, unsigned fcap, uint32_t *cut_of,
                               uint32_t *inv, cudaStream_t s) {
  const int64_t ninner = T.n > 1 ? T.n - 1 : 0;
  k_frontier_mark<<<(unsigned)((ninner + 1 + 255) / 256), 256, 0, s>>>(T, L, cid_node, cid_slot,
                                                                       flist, fcount, fcap);
  k_frontier_fill<<<1024, 256, 0, s>>>(flist, fcount, fcap, cut_of);
  k_inverse<<<(unsigned)((T.n + 255) / 256), 256, 0, s>>>(T.dir, T.n, inv);
  return cudaGetLastError();
}

cudaError_t launch_pair_index(const CutTree &A, const CutTree &B, uint4 *cut,
                              const unsigned *cut_count, unsigned cap, const uint32_t *cnA,
                              const uint32_t *csA, const uint32_t *cnB, const uint32_t *csB,
                              unsigned long long *hkey, uint32_t *hval, unsigned hmask,
                              unsigned *status, int blocks, cudaStream_t s) {
  k_pair_index<<<blocks, 256, 0, s>>>(A, B, cut, cut_count, cap, cnA, csA, cnB, csB, hkey, hval,
                                      hmask, status);
  return cudaGetLastError();
}

cudaError_t launch_attribute(const uint2 *hits, const unsigned long long *nhits,
                             unsigned long long hcap, const TLBeam &mA, const TLBeam &mB,
                             const uint32_t *invA, const uint32_t *invB, const uint32_t *cutA,
                             const uint32_t *cutB, const unsigned long long *hkey,
                             const uint32_t *hval, unsigned hmask, double *label,
                             unsigned *status, int blocks, cudaStream_t s) {
  k_attribute<<<blocks, 256, 0, s>>>(hits, nhits, hcap, mA, mB, invA, invB, cutA, cutB, hkey, hval,
                                     hmask, label, status);
  return cudaGetLastError();
}

// ------------------------------------------------------------ surrogate estimate

// Pair yield from the network's (mu, s): the predicted mean (B + 1) e^mu over
// the baseline B = st_scale * st (the network is trained with a Poisson-type
// deviance whose minimiser is the conditional mean).  Pairs whose
// predicted standard deviation exceeds tau are flagged for the exact
// fallback (their refs copied out).  With `sums`, the predictions and the ST rates of all
// pairs are added into sums[0] and sums[1] on the way.
__global__ void k_estimate(const float *out, const float *st, float st_scale, const uint4 *cut,
                           const unsigned *cut_count, unsigned cap, float tau, double *pred,
                           uint2 *fb, unsigned *fb_count, unsigned fb_cap, uint8_t *flag,
                           double *sums) {
  const unsigned n = min(*cut_count, cap);
  const int lane = threadIdx.x & 31;
  double acc = 0.0, sst = 0.0;  // the predictions and ST rates of this thread's pairs
  const unsigned nround = (n + 31u) & ~31u;
  for (unsigned p = blockIdx.x * blockDim.x + threadIdx.x; p < nround;
       p += gridDim.x * blockDim.x) {
    bool fall = false;
    uint2 r = make_uint2(0u, 0u);
    if (p < n) {
      const float mu = out[2 * p], s = fminf(fmaxf(out[2 * p + 1], -12.f), 12.f);
      const float var = __expf(s);
      fall = sqrtf(var) > tau;
      // the predicted mean (B + 1) e^mu with baseline B = st_scale * st
      const double e = ((double)st_scale * (double)st[p] + 1.0) * exp(fmin((double)mu, 30.0));
      const double y = fall ? 0.0 : fmax(e, 0.0);
      pred[p] = y;
      acc += y;
      sst += (double)st[p];
      if (flag) flag[p] = fall ? 1 : 0;
      const uint4 c = cut[p];
      r = make_uint2(c.x, c.y);
    }
    const unsigned m = __ballot_sync(0xffffffffu, fall);
    if (m) {
      unsigned base = 0;
      if (lane == 0) base = atomicAdd(fb_count, (unsigned)__popc(m));
      base = __shfl_sync(0xffffffffu, base, 0);
      if (fall) {
        const unsigned idx = base + __popc(m & ((1u << lane) - 1u));
        if (idx < fb_cap) fb[idx] = r;
      }
    }
  }
  if (sums) {
    for (int off = 16; off; off >>= 1) {
      acc += __shfl_xor_sync(0xffffffffu, acc, off);
      sst += __shfl_xor_sync(0xffffffffu, sst, off);
    }
    if (lane == 0 && (acc != 0.0 || sst != 0.0)) {
      atomicAdd(sums, acc);
      atomicAdd(sums + 1, sst);
    }
  }
}

cudaError_t launch_estimate(const float *out, const float *st, float st_scale, const uint4 *cut,
                            const unsigned *cut_count, unsigned cap, float tau, double *pred,
                            uint2 *fb, unsigned *fb_count, unsigned fb_cap, int blocks,
                            cudaStream_t s, uint8_t *flag, double *sums) {
  k_estimate<<<blocks, 256, 0, s>>>(out, st, st_scale, cut, cut_count, cap, tau, pred, fb,
                                    fb_count, fb_cap, flag, sums);
  return cudaGetLastError();
}

// ------------------------------------------------------------ helpers

__global__ void k_sur_misc(int op, const void *a, void *c, int64_t n) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  double acc = 0.0;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += stride) {
    if (op == 0) {
      const uint4 v = reinterpret_cast<const uint4 *>(a)[i];
      reinterpret_cast<uint2 *>(c)[i] = make_uint2(v.x, v.y);
    } else if (op == 1) {
      reinterpret_cast<float *>(c)[i] = (float)log1p(reinterpret_cast<const double *>(a)[i]);
    } else if (op == 2) {
      acc += reinterpret_cast<const double *>(a)[i];
    } else {
      acc += (double)reinterpret_cast<const float *>(a)[i];
    }
  }
  if (op >= 2) {
    for (int off = 16; off; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
    if ((threadIdx.x & 31) == 0 && acc != 0.0) atomicAdd(reinterpret_cast<double *>(c), acc);
  }
}

cudaError_t launch_sur_misc(int op, const void *a, const void *b, void *c, int64_t n,
                            cudaStream_t s) {
  (void)b;
  if (n <= 0) return cudaSuccess;
  int64_t blocks = (n + 255) / 256;
  if (blocks > 4096) blocks = 4096;
  k_sur_misc<<<(unsigned)blocks, 256, 0, s>>>(op, a, c, n);
  return cudaGetLastError();
}

}  // namespace tl
