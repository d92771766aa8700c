// tl_swarm.cu -- the IP regime (Sec. 2.2): macro-photons split into swarms of
// real photons.
//
// A macro-photon (MP) of integer weight w stands for w real photons with its
// energy and direction spread as evenly as possible over its volume, taken as
// an axis-aligned cube of side h (one h per beam) centred on the MP: photon k
// sits at p0 + h u_k, u_k,d = frac(0.5 + k alpha_d) - 0.5, alpha = (1/g, 1/g^2,
// 1/g^3), g the real root > 1 of x^4 = x + 1 (Roberts' R_3 low-discrepancy
// sequence; u_0 = 0, so a weight-1 MP is its own photon).  The paper splits two
// MPs when they collide and builds an octree over each swarm for that
// collision; here the MPs that can collide at all during a run are marked
// first, their swarms are written out as real photons, and the real photons go
// through the exact path (Morton LBVH, dual traversal, FP64 decision), which
// finds every real-photon pair of every colliding MP pair at once.
//
//   k_swarm_mark      all MP pairs: can a photon of MP i meet a photon of MP j
//                     during the run's time window?  (s > 1 up to a relative
//                     1e-9, and the centres' closest approach within the window
//                     at most r_max + the swarms' half-diagonals, with margins
//                     for rounding; FP32 with an error bound decides all but the
//                     pairs near the limit, FP64 those).  A superset of the pairs with real hits, so the
//                     hit set does not depend on it.
//   k_swarm_block_sums, k_swarm_scan_sums, k_swarm_offsets
//                     exclusive prefix sum of the marked MPs' weights.
//   k_swarm_expand    photon q of the expanded beam: its MP by binary search in
//                     the offsets, k = q - offset, position p0 + h u_k.
#include "tl_ctx.h"

namespace {

constexpr int kThreads = 256;
constexpr int kMarkGroup = 32;     // MPs of B per word of marks
constexpr int kMarkBMin = 64;      // MPs of B per block of the marking, smallest and
constexpr int kMarkBMax = 1024;    // largest slice (see trilens_swarm_mark)
constexpr int kSwarmTab = 256;     // swarm offsets kept in shared memory by the expansion
constexpr int kScanItems = 4;                     // per thread
constexpr int kScanBlock = kThreads * kScanItems;  // items per block

// 1/g, 1/g^2, 1/g^3 as the nearest doubles, g^4 = g + 1 (Roberts' R_3)
__constant__ double kR3[3] = {0.81917251339616448, 0.67104360670378926, 0.5497004779019703};

struct MarkArgs {
  TLBeam A, B;
  double T0, T1;   // the run's time window [fs]
  double lim2;     // (r_max + half-diagonals)^2 with margins [um^2]
  double s_floor;  // (2 m_e c^2) m_e c^2 (1 - 1e-9)
  uint8_t *mark_a, *mark_b;
  float T0f, T1f;  // the window in FP32
  float R;         // sqrt(lim2) in FP32
  float sf;        // s_floor in FP32
  double kT;       // FP32 error of a position at any time of the window per unit of |d|_1
  int slice;       // MPs of B per block
};

// The FP64 decision of one pair (the marks are exactly what it says): the invariant
// above the floor and the centres' closest approach in the window within the limit.
__device__ __noinline__ bool mark_exact(const MarkArgs &g, long long i, long long j) {
  const double dxi = g.A.dx[i], dyi = g.A.dy[i], dzi = g.A.dz[i];
  const double dxj = g.B.dx[j], dyj = g.B.dy[j], dzj = g.B.dz[j];
  const double px = g.A.px[i] - g.B.px[j], py = g.A.py[i] - g.B.py[j], pz = g.A.pz[i] - g.B.pz[j];
  const double cs = dxi * dxj + dyi * dyj + dzi * dzj;
  if (!(g.A.E[i] * g.B.E[j] * (1.0 - cs) > g.s_floor)) return false;  // below threshold
  const double vx = TL_C * (dxi - dxj), vy = TL_C * (dyi - dyj), vz = TL_C * (dzi - dzj);
  const double a = vx * vx + vy * vy + vz * vz;
  if (a == 0.0) return false;  // parallel: never a hit
  const double b = px * vx + py * vy + pz * vz;
  const double pp = px * px + py * py + pz * pz;
  const double Tm = fmax(fabs(g.T0), fabs(g.T1));
  const double lim = g.lim2 + 1e-13 * (pp + a * Tm * Tm);  // rounding of what follows
  if (-b <= a * g.T0 || -b >= a * g.T1) {
    // closest approach at an end of the window
    const double T = (-b <= a * g.T0) ? g.T0 : g.T1;
    const double qx = px + T * vx, qy = py + T * vy, qz = pz + T * vz;
    return qx * qx + qy * qy + qz * qz <= lim;
  }
  // inside: distance^2 = |p x v|^2 / |v|^2
  const double cx = py * vz - pz * vy, cy = pz * vx - px * vz, cz = px * vy - py * vx;
  return cx * cx + cy * cy + cz * cz <= lim * a;
}

// An MP as the FP32 test sees it: position, c d, energy, and its share of the bound
// on the test's distance.  The smallest distance in the window is a 1-Lipschitz
// function of the relative position and of T times the relative velocity, so FP32
// inputs move it by at most 2^-23 |p|_1 + T 2^-22 |c d|_1 per MP, and evaluating it
// in FP32 by at most 2^-20 of the same sums; e = 2^-19 (|p|_1 + T |c d|_1) covers
// both twice.  |d|_1 > 1.8 (not a unit vector) or a NaN: e = inf, FP64 decides.
struct MarkMP {
  float x, y, z, e, vx, vy, vz, E;
};
__device__ __forceinline__ MarkMP mark_mp(const TLBeam &b, long long i, double kT) {
  MarkMP m;
  const double px = b.px[i], py = b.py[i], pz = b.pz[i];
  const double dx = b.dx[i], dy = b.dy[i], dz = b.dz[i];
  m.x = (float)px;
  m.y = (float)py;
  m.z = (float)pz;
  m.vx = (float)(TL_C * dx);
  m.vy = (float)(TL_C * dy);
  m.vz = (float)(TL_C * dz);
  m.E = (float)b.E[i];
  const float p1 = fabsf(m.x) + fabsf(m.y) + fabsf(m.z);
  const float v1 = fabsf(m.vx) + fabsf(m.vy) + fabsf(m.vz);
  const float e = 0x1p-19f * p1 + (float)kT * v1;
  m.e = (v1 <= 1.8f * (float)TL_C && e < 1e30f) ? e : __int_as_float(0x7f800000);
  return m;
}

// Block (x, y): 256 MPs of A, one per thread, against the y-th slice of MPs of B,
// staged in shared memory.  What bounds it is instruction issue: ~35 FP32
// instructions per pair of a warp's 32 MPs with one of B, and no FP64 but for the
// pairs within the error bound of the limit (about 1 in 1000; GB300 does 2 FP64
// operations per clock and SM).  A pair whose two MPs are marked already can only set
// marks that are set: a warp whose 32 MPs are all marked visits only the unmarked MPs
// of B, by the bits of one word per 32.  2 x 16384 MPs: 19.2 ms with FP64 differences
// for every pair and an FP64 decision for every near one, 0.34 ms now.
__global__ void __launch_bounds__(kThreads) k_swarm_mark(MarkArgs g) {
  __shared__ float4 sp[kMarkBMax], sv[kMarkBMax];  // (x, y, z, e), (c d, E)
  __shared__ unsigned sm[kMarkBMax / kMarkGroup];  // marks of B, known or found
  __shared__ unsigned s0[kMarkBMax / kMarkGroup];  // ... as they were at the start
  const int tid = threadIdx.x, lane = tid & 31;
  const long long jb = blockIdx.y * (long long)g.slice;
  const int m = (int)min((long long)g.slice, (long long)g.B.n - jb);
  const long long i = blockIdx.x * (long long)kThreads + tid;
  const bool live = i < g.A.n;
  bool known = !live || *(volatile uint8_t *)(g.mark_a + i) != 0;
  {  // earlier blocks have marked all of the block's MPs: nothing left to find
    bool done = known;
    for (int t = tid; t < m && done; t += kThreads)
      done = *(volatile uint8_t *)(g.mark_b + jb + t) != 0;
    if (__syncthreads_and(done)) return;
  }
  for (int t = tid; t < ((m + 31) & ~31); t += kThreads) {
    bool marked = true;  // past the end: nothing to find
    if (t < m) {
      const MarkMP q = mark_mp(g.B, jb + t, g.kT);
      sp[t] = make_float4(q.x, q.y, q.z, q.e);
      sv[t] = make_float4(q.vx, q.vy, q.vz, q.E);
      marked = g.mark_b[jb + t] != 0;
    }
    const unsigned w = __ballot_sync(0xffffffffu, marked);
    if (lane == 0) sm[t >> 5] = s0[t >> 5] = w;
  }
  MarkMP a{};
  if (live) a = mark_mp(g.A, i, g.kT);
  const bool known0 = known;
  const float Rh = g.R * 1.000001f + a.e, Rl = g.R * 0.999999f - a.e;
  constexpr float ic2 = (float)(1.0 / (TL_C * TL_C));
  __syncthreads();
  const int groups = (m + kMarkGroup - 1) / kMarkGroup;
  const int w0 = (tid >> 5) % groups;  // warps start apart: one's finds spare the others' tests
  for (int gi = 0; gi < groups; ++gi) {
    const int gr = gi + w0 < groups ? gi + w0 : gi + w0 - groups;
    // one lane reads the word, which other warps add to: bm, todo and all are the warp's
    unsigned bm = lane == 0 ? *(volatile unsigned *)&sm[gr] : 0u;
    bm = __shfl_sync(0xffffffffu, bm, 0);
    const unsigned bm0 = bm;
    const int cnt = min(kMarkGroup, m - gr * kMarkGroup);
    unsigned todo = cnt == 32 ? 0xffffffffu : (1u << cnt) - 1u;
    bool all = __all_sync(0xffffffffu, known);
    if (all) todo &= ~bm;
    while (todo) {
      const int t = __ffs(todo) - 1;
      todo &= todo - 1u;
      const float4 p = sp[gr * kMarkGroup + t], v = sv[gr * kMarkGroup + t];
      const float qx = a.x - p.x, qy = a.y - p.y, qz = a.z - p.z;
      const float ux = a.vx - v.x, uy = a.vy - v.y, uz = a.vz - v.z;
      const float aa = fmaf(ux, ux, fmaf(uy, uy, uz * uz));
      const float b = fmaf(qx, ux, fmaf(qy, uy, qz * uz));
      const float T = fminf(fmaxf(__fdividef(-b, aa), g.T0f), g.T1f);
      const float ex = fmaf(T, ux, qx), ey = fmaf(T, uy, qy), ez = fmaf(T, uz, qz);
      const float d2 = fmaf(ex, ex, fmaf(ey, ey, ez * ez));
      // 1 - cos off by less than 2^-18; E E (1 - cos) against the floor
      const float cs = fmaf(a.vx, v.x, fmaf(a.vy, v.y, a.vz * v.z)) * ic2;
      const float ee = a.E * v.w, omc = 1.0f - cs;
      const float hi = Rh + p.w, lo = Rl - p.w;
      const bool apart = aa >= 0.01f;  // else the closest approach is ill-conditioned
      const bool miss = hi < 1e30f && ((apart && d2 > hi * hi) ||
                                       ee * (omc + 0x1p-18f) < g.sf * 0.99999f);
      bool cand = apart && lo > 0.0f && d2 < lo * lo && ee * (omc - 0x1p-18f) > g.sf * 1.00001f;
      // undecided by FP32, and its marks still matter (dead lanes are `known`)
      if (live && !miss && !cand && !(known && (bm >> t & 1u)))
        cand = mark_exact(g, i, jb + gr * kMarkGroup + t);
      cand = cand && live;
      known = known || cand;
      if (__any_sync(0xffffffffu, cand)) bm |= 1u << t;
      if (!all && __all_sync(0xffffffffu, known)) {
        all = true;
        todo &= ~bm;
      }
    }
    if (lane == 0 && bm != bm0) atomicOr(&sm[gr], bm);
    __syncwarp();
  }
  if (known && !known0) g.mark_a[i] = 1;
  __syncthreads();
  for (int t = tid; t < m; t += kThreads)
    if ((sm[t >> 5] & ~s0[t >> 5]) >> (t & 31) & 1u) g.mark_b[jb + t] = 1;
}

// an MP's photons if it is marked; *bad is set if its weight is no whole number
__device__ __forceinline__ long long swarm_weight(const TLBeam &mp, const uint8_t *mark,
                                                  long long i, bool *bad) {
  const double w = mp.w ? mp.w[i] : 1.0;
  if (!(w >= 1.0 && w < 4294967296.0 && w == floor(w))) {
    *bad = true;
    return 0;
  }
  return mark[i] ? (long long)w : 0;
}

__device__ __forceinline__ long long block_exclusive_scan(long long v, long long *total,
                                                          long long *ws) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  long long x = v;
  for (int o = 1; o < 32; o <<= 1) {
    const long long y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) ws[w] = x;
  __syncthreads();
  if (w == 0) {
    long long s = lane < kThreads / 32 ? ws[lane] : 0;
    for (int o = 1; o < 32; o <<= 1) {
      const long long y = __shfl_up_sync(0xffffffffu, s, o);
      if (lane >= o) s += y;
    }
    if (lane < kThreads / 32) ws[lane] = s;
  }
  __syncthreads();
  const long long before = (w ? ws[w - 1] : 0) + x - v;
  *total = ws[kThreads / 32 - 1];
  __syncthreads();
  return before;
}

// The offsets need no scratch: a block's sum stands in the place of its first MP's
// offset, negative if a weight of the block is bad, until that block's offsets are
// written; the total (negative: bad) ends up in offsets[n].
__global__ void __launch_bounds__(kThreads) k_swarm_block_sums(TLBeam mp, const uint8_t *mark,
                                                               long long *offsets) {
  __shared__ long long ws[kThreads / 32];
  const long long base = blockIdx.x * (long long)kScanBlock + threadIdx.x * kScanItems;
  long long s = 0;
  bool bad = false;
  for (int q = 0; q < kScanItems; ++q)
    if (base + q < mp.n) s += swarm_weight(mp, mark, base + q, &bad);
  long long tot;
  block_exclusive_scan(s, &tot, ws);
  bad = __syncthreads_or(bad);
  if (threadIdx.x == 0) offsets[blockIdx.x * (long long)kScanBlock] = bad ? -1 : tot;
}

// one block: the blocks' sums -> exclusive prefix sums in place, offsets[n] = total
__global__ void __launch_bounds__(kThreads) k_swarm_scan_sums(long long *offsets, long long nb,
                                                              long long n) {
  __shared__ long long ws[kThreads / 32];
  long long carry = 0;
  bool bad = false;
  for (long long c0 = 0; c0 < nb; c0 += kThreads) {
    const long long c = c0 + threadIdx.x;
    const long long v = c < nb ? offsets[c * kScanBlock] : 0;
    bad = bad || v < 0;
    long long tot;
    const long long ex = block_exclusive_scan(v, &tot, ws);
    if (c < nb) offsets[c * kScanBlock] = carry + ex;
    carry += tot;
  }
  bad = __syncthreads_or(bad);
  if (threadIdx.x == 0) offsets[n] = bad ? -1 : carry;
}

__global__ void __launch_bounds__(kThreads) k_swarm_offsets(TLBeam mp, const uint8_t *mark,
                                                            long long *offsets) {
  __shared__ long long ws[kThreads / 32];
  const long long base = blockIdx.x * (long long)kScanBlock + threadIdx.x * kScanItems;
  const long long first = offsets[blockIdx.x * (long long)kScanBlock];
  long long v[kScanItems], s = 0;
  bool bad = false;
  for (int q = 0; q < kScanItems; ++q) {
    v[q] = base + q < mp.n ? swarm_weight(mp, mark, base + q, &bad) : 0;
    s += v[q];
  }
  long long tot;
  long long run = first + block_exclusive_scan(s, &tot, ws);  // (its barriers: first is read)
  for (int q = 0; q < kScanItems; ++q) {
    if (base + q < mp.n) offsets[base + q] = run;
    run += v[q];
  }
}

struct ExpandArgs {
  TLBeam mp;
  double h;
  const long long *offsets;
  long long total;
  double *out[8];  // px py pz dx dy dz E w (w may be null)
  uint32_t *owner, *kof;
};

// u_k of the swarm's sequence, times h: the offset of photon k from its MP
__device__ __forceinline__ double swarm_offset(double h, long long k, int d) {
  const double x = __dadd_rn(0.5, __dmul_rn((double)k, kR3[d]));
  return __dmul_rn(h, __dsub_rn(__dsub_rn(x, floor(x)), 0.5));
}

// Bound by its 72 bytes per photon once the FP64 work is out of the way: the offset
// depends on k and h alone, so each block tabulates the first kSwarmTab of them (21
// FP64 operations each) and a photon then costs three FP64 additions instead of 24
// operations; and a block searches the whole offset list only for its first and last
// photon.  2 x 1.63e6 photons: 172 us before, 111 us now (126 us with the table alone).
__global__ void __launch_bounds__(kThreads) k_swarm_expand(ExpandArgs g) {
  __shared__ double tab[3][kSwarmTab];
  for (int t = threadIdx.x; t < kSwarmTab; t += kThreads)
    for (int d = 0; d < 3; ++d) tab[d][t] = swarm_offset(g.h, t, d);
  __syncthreads();
  __shared__ long long ends[2];
  for (long long q0 = blockIdx.x * (long long)kThreads; q0 < g.total;
       q0 += (long long)gridDim.x * kThreads) {
    // the MPs of the block's first and last photon (two searches of the whole
    // list), then each thread searches between them
    __syncthreads();
    if ((threadIdx.x & 31) == 0 && threadIdx.x < 64) {
      const long long qe = threadIdx.x ? min(q0 + kThreads, g.total) - 1 : q0;
      long long lo = 0, hi = g.mp.n;  // offsets[lo] <= qe < offsets[hi]
      while (hi - lo > 1) {
        const long long mid = (lo + hi) >> 1;
        if (g.offsets[mid] <= qe) lo = mid;
        else hi = mid;
      }
      ends[threadIdx.x >> 5] = lo;
    }
    __syncthreads();
    const long long q = q0 + threadIdx.x;
    if (q >= g.total) continue;
    long long lo = ends[0], hi = ends[1] + 1;
    while (hi - lo > 1) {
      const long long mid = (lo + hi) >> 1;
      if (g.offsets[mid] <= q) lo = mid;
      else hi = mid;
    }
    const long long k = q - g.offsets[lo];
    double u[3];
    for (int d = 0; d < 3; ++d) u[d] = k < kSwarmTab ? tab[d][k] : swarm_offset(g.h, k, d);
    g.out[0][q] = __dadd_rn(g.mp.px[lo], u[0]);
    g.out[1][q] = __dadd_rn(g.mp.py[lo], u[1]);
    g.out[2][q] = __dadd_rn(g.mp.pz[lo], u[2]);
    g.out[3][q] = g.mp.dx[lo];
    g.out[4][q] = g.mp.dy[lo];
    g.out[5][q] = g.mp.dz[lo];
    g.out[6][q] = g.mp.E[lo];
    if (g.out[7]) g.out[7][q] = 1.0;
    g.owner[q] = (uint32_t)lo;
    g.kof[q] = (uint32_t)k;
  }
}

bool beam_valid(const trilens_beam *b) {
  if (!b || b->n < 0 || b->n >= (1ll << 32)) return false;
  if (b->n == 0) return true;
  return b->px && b->py && b->pz && b->dx && b->dy && b->dz && b->E;
}

TLBeam to_tl(const trilens_beam *b) {
  TLBeam t;
  t.n = b->n;
  t.px = b->px; t.py = b->py; t.pz = b->pz;
  t.dx = b->dx; t.dy = b->dy; t.dz = b->dz;
  t.E = b->E; t.w = b->w;
  return t;
}

int sm_count() {
  int dev = 0, n = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    return 0;
  return n;
}

}  // namespace

extern "C" int trilens_swarm_mark(const trilens_beam *a, const trilens_beam *b, double h_a,
                                  double h_b, const trilens_params *p, int64_t first_step,
                                  int64_t steps, uint8_t *mark_a, uint8_t *mark_b,
                                  trilens_stream_t stream) {
  if (!beam_valid(a) || !beam_valid(b) || !p || !(p->dt_fs > 0.0) || !(p->kappa > 0.0) ||
      !(h_a >= 0.0) || !(h_b >= 0.0) || !(h_a < 1e30) || !(h_b < 1e30) || first_step < 0 ||
      steps < 1 || (a->n > 0 && !mark_a) || (b->n > 0 && !mark_b))
    return TRILENS_ERR_INVALID;
  cudaStream_t s = (cudaStream_t)stream;
  if (a->n > 0 && cudaMemsetAsync(mark_a, 0, (size_t)a->n, s) != cudaSuccess)
    return TRILENS_ERR_CUDA;
  if (b->n > 0 && cudaMemsetAsync(mark_b, 0, (size_t)b->n, s) != cudaSuccess)
    return TRILENS_ERR_CUDA;
  if (a->n == 0 || b->n == 0) return TRILENS_OK;
  MarkArgs g{};
  g.A = to_tl(a);
  g.B = to_tl(b);
  g.T0 = (double)first_step * p->dt_fs;
  g.T1 = (double)(first_step + steps) * p->dt_fs;
  const double rmax = 1e6 * sqrt(p->kappa * tl_sigma_max_bound() / TL_PI);
  const double reach = (rmax + 0.8660254037844387 * (h_a + h_b)) * (1.0 + 1e-6) + 1e-9;
  g.lim2 = reach * reach + 1e-9;
  g.s_floor = (2.0 * TL_MEC2) * TL_MEC2 * (1.0 - 1e-9);
  g.mark_a = mark_a;
  g.mark_b = mark_b;
  g.T0f = (float)g.T0;
  g.T1f = (float)g.T1;
  g.R = (float)sqrt(g.lim2);
  g.sf = (float)g.s_floor;
  g.kT = 0x1p-19 * std::max(fabs(g.T0), fabs(g.T1));
  // The slice of B per block.  A warp with an MP that never gets marked visits its
  // whole slice, one dependent test after the other, and later blocks skip what
  // earlier ones marked: short slices, until there are 16 blocks per SM (2 x 16384
  // MPs: 1024 per block 742 us, 256 per block 341 us).
  const long long ax = (a->n + kThreads - 1) / kThreads;
  const int n_sm = sm_count();
  if (n_sm == 0) return TRILENS_ERR_CUDA;
  g.slice = kMarkBMax;
  while (g.slice > kMarkBMin && ax * ((b->n + g.slice - 1) / g.slice) < 16ll * n_sm) g.slice >>= 1;
  const dim3 grid((unsigned)ax, (unsigned)((b->n + g.slice - 1) / g.slice));
  if (b->n > 65535ll * kMarkBMax) return TRILENS_ERR_INVALID;  // b->n above 2^26 MPs
  k_swarm_mark<<<grid, kThreads, 0, s>>>(g);
  return cudaGetLastError() == cudaSuccess ? TRILENS_OK : TRILENS_ERR_CUDA;
}

extern "C" int trilens_swarm_count(const trilens_beam *mp, const uint8_t *mark, int64_t *offsets,
                                   int64_t *total, trilens_stream_t stream) {
  if (!beam_valid(mp) || !offsets || !total || (mp->n > 0 && !mark)) return TRILENS_ERR_INVALID;
  cudaStream_t s = (cudaStream_t)stream;
  const long long n = mp->n;
  const long long nb = (n + kScanBlock - 1) / kScanBlock;
  const TLBeam t = to_tl(mp);
  long long *off = reinterpret_cast<long long *>(offsets);
  if (nb > 0) k_swarm_block_sums<<<(unsigned)nb, kThreads, 0, s>>>(t, mark, off);
  k_swarm_scan_sums<<<1, kThreads, 0, s>>>(off, nb, n);
  if (nb > 0) k_swarm_offsets<<<(unsigned)nb, kThreads, 0, s>>>(t, mark, off);
  long long tot_h = 0;
  if (cudaGetLastError() != cudaSuccess ||
      cudaMemcpyAsync(&tot_h, off + n, sizeof tot_h, cudaMemcpyDeviceToHost, s) != cudaSuccess ||
      cudaStreamSynchronize(s) != cudaSuccess)
    return TRILENS_ERR_CUDA;
  if (tot_h < 0) return TRILENS_ERR_INVALID;
  *total = tot_h;
  return TRILENS_OK;
}

extern "C" int trilens_swarm_expand(const trilens_beam *mp, double h, const int64_t *offsets,
                                    int64_t total, double *const *out, uint32_t *owner,
                                    uint32_t *index_in_swarm, trilens_stream_t stream) {
  if (!beam_valid(mp) || !offsets || total < 0 || !(h >= 0.0) || !(h < 1e30))
    return TRILENS_ERR_INVALID;
  if (total == 0) return TRILENS_OK;
  if (mp->n == 0 || !out || !owner || !index_in_swarm) return TRILENS_ERR_INVALID;
  for (int k = 0; k < 7; ++k)
    if (!out[k]) return TRILENS_ERR_INVALID;
  ExpandArgs g{};
  g.mp = to_tl(mp);
  g.h = h;
  g.offsets = reinterpret_cast<const long long *>(offsets);
  g.total = total;
  for (int k = 0; k < 8; ++k) g.out[k] = out[k];
  g.owner = owner;
  g.kof = index_in_swarm;
  const int n_sm = sm_count();
  if (n_sm == 0) return TRILENS_ERR_CUDA;
  const long long nblk = (total + kThreads - 1) / kThreads;
  const int blocks = (int)std::min<long long>(nblk, 8ll * n_sm);
  k_swarm_expand<<<blocks, kThreads, 0, (cudaStream_t)stream>>>(g);
  return cudaGetLastError() == cudaSuccess ? TRILENS_OK : TRILENS_ERR_CUDA;
}
