// tl_frame.cuh -- the frame of the exact path's boxes, the swept box of a photon
// in it, and the cells its photons are ordered by.
//
// Two photons that come within a distance r at one time do so in every frame
// that moves uniformly and is turned: boxes may be swept in any frame the two
// beams share.  The frame here moves with the mean of the two beams' mean
// directions, ubar, and its third axis is their difference: there both beams
// move along that axis only (but for their divergence), so a photon's swept box
// is a needle, whatever the crossing angle; axis-aligned boxes in the lab frame
// are as wide across the motion as along it for beams that cross.
#pragma once
#include <math.h>

#include "tl_common.cuh"

// x' = R x, v' = R (d - u) (v in units of c): exactly these FP32 numbers define the
// frame, so rounding them costs nothing.  ident: R = 1, u = 0.
struct TLFrame {
  float r[9];
  float u[3];
  int ident;
  // half-width across its path of a photon's box of beam k: amp[k] E^xp (tl_photon_pad);
  // typ: that of a typical photon
  float amp[2], xp, typ;
  // photon pairs compared at the time they pass each other (tl_set_needles): closing axis
  // (-1: none), 1 / closing velocity, half the step, window, and the pads' terms
  int axis;
  float inv, hl, lt, gain, add, ep, ec;
  int fill[3];
};

// Ordering grid of one instance and step: cell = (x' - lo) scale, nb bits per axis,
// axes by falling nb (perm); and the box that holds every swept box of the other beam's
// photons: a photon whose own misses it can meet none of them.
struct TLGrid {
  float lo[3], scale[3];
  int nb[3], perm[3];
  float clo[3], chi[3];
};

// One instance's photons of one beam in the exact path's layout: groups of 32 sorted photons
// from group0 on, and its tree, an implicit one with 32 children per
// node over the sorted photons: level 0 the photons, level l nodes of 32^l.  An instance of
// more than 1024 photons starts on a tile of 32 groups and takes whole tiles (its level 2);
// smaller ones, whose trees end at level 1, share tiles.  Only the
// photons that can meet the other beam in a step are sorted; how many, the running sum
// of the cells tells (tl_live).
struct TLInst {
  int n;            // photons,
  int first;        // from this one of the input on
  int group0;       // first group
  int bits;         // its photons are ordered by 2^bits cells,
  uint32_t cell0;   // from this one on
  uint32_t lev[6];  // first box of each level
};

// nodes of level l over n photons
__host__ __device__ inline int tl_level_count(int n, int l) {
  return (int)(((long long)n + (1ll << (5 * l)) - 1) >> (5 * l));
}
// the lowest level (>= 1) with at most 32 nodes
__host__ __device__ inline int tl_top_level(int n) {
  int l = 1;
  while (l < 5 && tl_level_count(n, l) > 32) ++l;
  return l;
}

constexpr int kTile = 1024;  // sorted photons per tile (a level-2 node of a larger instance)

__host__ __device__ inline TLFrame tl_ident_frame() {
  TLFrame f{};  // (no pads: set by tl_set_pads)
  f.r[0] = f.r[4] = f.r[8] = 1.0f;
  f.ident = 1;
  return f;
}

// The frame of two beams with mean directions a and b.  The lab frame itself when
// they are (nearly) parallel or have no common direction, or when the turn would be
// below ~1e-2, the order of a beam's own divergence: then the lab's boxes are as
// good and need a third of the work.
__host__ __device__ inline TLFrame tl_make_frame(const double a[3], const double b[3]) {
  double w[3], u[3], wl = 0.0;
  for (int k = 0; k < 3; ++k) {
    w[k] = a[k] - b[k];
    u[k] = 0.5 * (a[k] + b[k]);
    wl += w[k] * w[k];
  }
  wl = sqrt(wl);
  if (!(wl > 0.1) || !(wl < 10.0)) return tl_ident_frame();
  double uw = 0.0, wmax = 0.0;
  for (int k = 0; k < 3; ++k) {
    w[k] /= wl;
    uw += u[k] * w[k];
    wmax = fmax(wmax, fabs(w[k]));
  }
  double e[3], el = 0.0;  // the drift across the axis
  for (int k = 0; k < 3; ++k) {
    e[k] = u[k] - uw * w[k];
    el += e[k] * e[k];
  }
  el = sqrt(el);
  if (wmax >= 0.9999 && el <= 0.02) return tl_ident_frame();
  if (el < 1e-3) {  // any axis across w
    int m = 0;
    for (int k = 1; k < 3; ++k)
      if (fabs(w[k]) < fabs(w[m])) m = k;
    el = 0.0;
    for (int k = 0; k < 3; ++k) {
      e[k] = (k == m ? 1.0 : 0.0) - w[m] * w[k];
      el += e[k] * e[k];
    }
    el = sqrt(el);
  }
  TLFrame f{};
  for (int k = 0; k < 3; ++k) {
    e[k] /= el;
    f.u[k] = (float)u[k];
  }
  const double g[3] = {w[1] * e[2] - w[2] * e[1], w[2] * e[0] - w[0] * e[2],
                       w[0] * e[1] - w[1] * e[0]};
  for (int k = 0; k < 3; ++k) {
    f.r[k] = (float)e[k];
    f.r[3 + k] = (float)g[k];
    f.r[6 + k] = (float)w[k];
  }
  return f;
}

// Pads by energy.  A pair collides within r(s), s = E_i E_j (1 - cos) / (2 m^2 c^4), and r
// falls with s beyond its peak at s ~ 2 (r^2 ~ ln s / s): most pairs meet far inside r_max.
// With r(s) <= A r_max s^-q for every s (A = max of r s^q / r_max) and s >= s_i s_j,
// s_k = lambda_k E_k sqrt(cmin / 2) / m c^2 (cmin: least 1 - cos of the beams;
// lambda_a lambda_b = 1), r <= A r_max s_i^-q s_j^-q <= A r_max (s_i^-2q + s_j^-2q) / 2:
// a pad of its own for each photon, whose sums cover every pair.  A photon's pad
// is at most r_max, which covers its pairs alone.  q is the one with the least pads near
// the beams' mean ln E, 0 (r_max / 2 for all) where none is below that.  64 steps of
// 2 x 1M photons of 5 MeV 12.3 ms with r_max / 2, 10.1 ms now; a step of 2 x 4M with a
// broad spectrum 7.16 ms, 6.60 ms.
constexpr int kPadQ = 12;  // q = 0.04 k
struct TLPadTable {
  float a[kPadQ];
};

// e: 12 values each, the beams' extremes as in tl_beam_box, whose directions bound cos
// (2e-5 covers their FP32 rounding and that of the frame); mean and standard deviation of
// ln E of each beam.
__host__ __device__ inline void tl_set_pads(TLFrame &f, const TLPadTable &t, const double *ea,
                                            const double *eb, const double la[2],
                                            const double lb[2], double half) {
  double cmin = 1.0 - 2e-5;
  for (int k = 0; k < 3; ++k) {
    const double a0 = ea[3 + k], a1 = ea[9 + k], b0 = eb[3 + k], b1 = eb[9 + k];
    cmin -= fmax(fmax(a0 * b0, a0 * b1), fmax(a1 * b0, a1 * b1));
  }
  const double m2 = TL_MEC2 * TL_MEC2, st = 0.5 * cmin * exp(la[0] + lb[0]) / m2;
  const double sd = fmax(la[1], lb[1]);
  int best = 0;
  double least = 0.95;
  for (int k = 1; k < kPadQ && cmin > 1e-3 && st > 0.0; ++k) {
    const double c = (double)t.a[k] * exp(0.04 * k * (2.0 * sd - log(st)));
    if (c < least) {
      least = c;
      best = k;
    }
  }
  f.xp = -0.08f * (float)best;
  f.axis = -1;
  for (int k = 0; k < 2; ++k) {
    const double lam = exp(0.5 * (k ? la[0] - lb[0] : lb[0] - la[0]));
    f.amp[k] = best ? (float)(half * (double)t.a[best] * (1.0 + 1e-5) *
                              exp((double)f.xp * log(lam * sqrt(0.5 * cmin / m2))))
                    : (float)half;
  }
  f.typ = (float)(best ? half * (double)t.a[best] * exp(-0.04 * best * log(st)) : half);
}

// Needles.  Where the beams close along one axis of the frame with nearly one velocity vc,
// a pair that collides does so close to the time lambda0 = -dZ0 / vc (in units of length, 0
// to L in the step) at which it would pass with exactly that velocity: the closest approach
// within hs, the sum of the pads, has |dZ| <= hs, so with vlo the least closing velocity and
// delta the largest |dV / vc - 1| it lies within Terr = (hs / vlo) (1 + delta) + L delta of
// lambda0, and across the axis |dX(lambda0)| <= hs + DV Terr, DV the largest difference of
// velocities there.  So a pair can be told by u = lambda0 - L / 2 in the window
// |u| <= L / 2 + Terr, and |dXm + dVx u| <= hs (1 + DV (1 + delta) / vlo) + DV L delta,
// Xm the middle of the photon's path: a square of the pads' size, where swept boxes also
// hold all of both photons' travel (1 % of the pairs that they leave is left of a step of
// 2 x 4M photons).  u is the sum of -Z / vc - L / 2 of beam A's photon and Z / vc of beam
// B's.  FP32: a coordinate is off by 6u of the sum of the lengths turned (u = 2^-24), in u
// by that over vc; ep and ec take 16u and more of each (tl_needle).
// Beams without such an axis (delta > 0.1) keep the boxes, and so do those whose photons
// travel less than kNeedleTravel pads across it in a step (the spread of directions taken as
// an eighth of their range): there the two tests leave the same pairs.
constexpr double kNeedleTravel = 3.0;

inline void tl_set_needles(TLFrame &f, const double *ea, const double *eb,
                                               double L, double half) {
  f.axis = -1;
  double best = 0.0;
  int m = -1;
  for (int k = 0; k < 3; ++k) {
    const double c = fabs(ea[3 + k] + ea[9 + k] - eb[3 + k] - eb[9 + k]);
    if (c > best) {
      best = c;
      m = k;
    }
  }
  if (m < 0) return;
  // closing velocities of a pair, 1e-6 for the rounding of the extremes and of the frame
  const double v0 = ea[3 + m] - eb[9 + m] - 2e-6, v1 = ea[9 + m] - eb[3 + m] + 2e-6;
  const double vc = 0.5 * (v0 + v1), vlo = fmin(fabs(v0), fabs(v1));
  if (!(v0 * v1 > 0.0) || !(vlo > 0.05)) return;
  const double delta = 0.5 * (v1 - v0) / fabs(vc) + 1e-6;
  if (!(delta < 0.1)) return;
  double DV = 0.0, sd = 0.0;
  for (int k = 0; k < 3; ++k)
    if (k != m) {
      const double ra = 0.125 * (ea[9 + k] - ea[3 + k]), rb = 0.125 * (eb[9 + k] - eb[3 + k]);
      DV = fmax(DV, fmax(fabs(ea[9 + k] - eb[3 + k]), fabs(ea[3 + k] - eb[9 + k])));
      sd = fmax(sd, ra * ra + rb * rb);
    }
  if (!(L * sqrt(sd) > kNeedleTravel * 2.0 * (double)f.typ)) return;
  DV += 2e-6;
  if (!(DV < 4.0)) return;
  const double up = 1.0 + 1e-5;
  f.axis = m;
  f.inv = (float)(1.0 / vc);
  f.hl = (float)(0.5 * L);
  f.lt = (float)((0.5 * L + 4.0 * half / vlo * (1.0 + delta) + L * delta) * up);
  f.gain = (float)((1.0 + DV * (1.0 + delta) / vlo) * up);
  f.add = (float)(0.5 * DV * L * delta * up);
  f.ep = (float)(0x1p-20 * (1.0 + fabs(1.0 / vc)) * (1.0 + DV) * up);
  f.ec = (float)(0x1p-18 * (L + (double)f.lt) * (1.0 + DV) * up);
}

// The grid of `bits` bits in all over [lo, lo + range]: each bit halves the cells of
// the axis that are longest in units of s, the extent of two photons' boxes there.
// Cells (and so the 32 photons of a leaf) in the proportions of s overlap the fewest
// other boxes for their volume.
__host__ __device__ inline TLGrid tl_make_grid(const double lo[3], const double range[3],
                                               const double s[3], int bits) {
  TLGrid g{};
  double rel[3];
  for (int k = 0; k < 3; ++k) rel[k] = range[k] > 0.0 && s[k] > 0.0 ? range[k] / s[k] : 0.0;
  for (int b = 0; b < bits; ++b) {
    int m = 0;
    for (int k = 1; k < 3; ++k)
      if (rel[k] > rel[m]) m = k;
    if (g.nb[m] >= 16) break;
    ++g.nb[m];
    rel[m] *= 0.5;
  }
  for (int k = 0; k < 3; ++k) {
    g.lo[k] = (float)lo[k];
    g.scale[k] = range[k] > 0.0 ? (float)((double)(1u << g.nb[k]) / range[k]) : 0.0f;
    g.perm[k] = k;
  }
  for (int i = 0; i < 2; ++i)  // by falling bits
    for (int k = 0; k < 2; ++k)
      if (g.nb[g.perm[k]] < g.nb[g.perm[k + 1]]) {
        const int t = g.perm[k];
        g.perm[k] = g.perm[k + 1];
        g.perm[k + 1] = t;
      }
  return g;
}

// The box of every swept box of a beam at the step: from the extremes pmin, dmin,
// pmax, dmax of R p0 and R d (e[0..11]), ct = c t_k >= 0, the travel L and the pad half.
// p1, d1: the largest |p0|_1 and |d|_1 where the extremes were found in FP32 (each is off
// by less than 2^-22 of them), else 0.
__host__ __device__ inline void tl_beam_box(const double *e, double p1, double d1,
                                            const TLFrame &f, double ct, double L, double half,
                                            float clo[3], float chi[3]) {
  for (int k = 0; k < 3; ++k) {
    const double ru = (double)f.r[3 * k] * f.u[0] + (double)f.r[3 * k + 1] * f.u[1] +
                      (double)f.r[3 * k + 2] * f.u[2];
    const double lo = e[k] + ct * e[3 + k], hi = e[6 + k] + ct * e[9 + k];
    const double m = half + 1e-6 * (1.0 + fabs(lo) + fabs(hi) + ct + L + p1 + (ct + L) * d1);
    clo[k] = (float)(lo + fmin(0.0, L * (e[3 + k] - ru)) - m);
    chi[k] = (float)(hi + fmax(0.0, L * (e[9 + k] - ru)) + m);
  }
}

#ifdef __CUDACC__

// photons of an instance that are sorted this step (never more than it has, also where the
// running sum is not valid: a wait of its scan ran out)
__device__ __forceinline__ int tl_live(const TLInst &I, const uint32_t *start) {
  const int n = (int)(__ldg(start + I.cell0 + (1u << I.bits)) - __ldg(start + I.cell0));
  return max(0, min(n, I.n));
}

// Swept interval of one axis in FP32 interval arithmetic with directed rounding: the
// position lies within ep of p and the velocity within ev of v; the segment is
// P + lambda v for lambda in [0, L], L in [Llo, Lhi]; half = r_max / 2 plus margin.
__device__ __forceinline__ void swept_axis(float p, float ep, float v, float ev, float Llo,
                                           float Lhi, float half, float &lo, float &hi) {
  const float plo = __fsub_rd(p, ep), phi = __fadd_ru(p, ep);
  const float vlo = __fsub_rd(v, ev), vhi = __fadd_ru(v, ev);
  const float ldlo = vlo >= 0.f ? __fmul_rd(Llo, vlo) : __fmul_rd(Lhi, vlo);
  const float ldhi = vhi >= 0.f ? __fmul_ru(Lhi, vhi) : __fmul_ru(Llo, vhi);
  lo = __fsub_rd(fminf(plo, __fadd_rd(plo, ldlo)), half);
  hi = __fadd_ru(fmaxf(phi, __fadd_ru(phi, ldhi)), half);
}

// In the lab frame: the FP64 position of the definition lies within |P32| 2^-23 of
// P32, and likewise the direction.
__device__ __forceinline__ void seg_axis(float p, float dc, float Llo, float Lhi, float half,
                                         float &lo, float &hi) {
  swept_axis(p, __fmaf_ru(fabsf(p), 1.1920928955078125e-7f, 1e-30f), dc,
             __fmaf_ru(fabsf(dc), 1.1920928955078125e-7f, 1e-30f), Llo, Lhi, half, lo, hi);
}

// A photon's pad (E in FP32): the margin in amp covers the rounding of the power.
__device__ __forceinline__ float tl_photon_pad(const TLFrame &f, int beam, float E, float half) {
  if (f.xp == 0.0f) return half;
  return fminf(2.0f * half, fmaf(f.amp[beam], exp2f(f.xp * log2f(E)), 1e-9f));
}

// A photon as a needle: middle of its path across the closing axis, time, velocities across,
// pad, and the rounding of its time.
struct TLNeedle {
  float x, y, w, vx, vy, h, e;
};

__device__ __forceinline__ TLNeedle tl_needle(const TLFrame &f, int beam, const float4 p,
                                              const float4 d, float pad) {
  float X[3] = {p.x, p.y, p.z}, V[3] = {d.x, d.y, d.z};
  if (!f.ident) {
    const float vx = d.x - f.u[0], vy = d.y - f.u[1], vz = d.z - f.u[2];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      X[k] = fmaf(f.r[3 * k], p.x, fmaf(f.r[3 * k + 1], p.y, f.r[3 * k + 2] * p.z));
      V[k] = fmaf(f.r[3 * k], vx, fmaf(f.r[3 * k + 1], vy, f.r[3 * k + 2] * vz));
    }
  }
  const int m = f.axis;
  const float z = m == 0 ? X[0] : (m == 1 ? X[1] : X[2]);
  TLNeedle n;
  n.vx = m == 0 ? V[1] : V[0];
  n.vy = m == 2 ? V[1] : V[2];
  n.x = fmaf(n.vx, f.hl, m == 0 ? X[1] : X[0]);
  n.y = fmaf(n.vy, f.hl, m == 2 ? X[1] : X[2]);
  n.w = beam ? z * f.inv : fmaf(-z, f.inv, -f.hl);
  n.e = fmaf(f.ep, fabsf(p.x) + fabsf(p.y) + fabsf(p.z), f.ec);
  n.h = (fmaf(f.gain, pad, f.add) + n.e) * (1.0f + 0x1p-20f);
  return n;
}

// A photon's swept box in the frame.  Each coordinate of R P from the rounded inputs
// is off by at most 4u sum |R||P| (u = 2^-24: u of the inputs, 3u of the sum), each of
// R (d - ubar) by 5u sum |R|(|d| + |ubar|); 6u is taken for both.
__device__ __forceinline__ TLBox swept_box(const float4 p, const float4 d, const TLFrame &f,
                                           float Llo, float Lhi, float half) {
  TLBox b;
  if (f.ident) {
    seg_axis(p.x, d.x, Llo, Lhi, half, b.lx, b.hx);
    seg_axis(p.y, d.y, Llo, Lhi, half, b.ly, b.hy);
    seg_axis(p.z, d.z, Llo, Lhi, half, b.lz, b.hz);
    return b;
  }
  const float e6 = 6.0f * 5.9604644775390625e-8f;
  const float vx = d.x - f.u[0], vy = d.y - f.u[1], vz = d.z - f.u[2];
  const float ax = fabsf(d.x) + fabsf(f.u[0]), ay = fabsf(d.y) + fabsf(f.u[1]),
              az = fabsf(d.z) + fabsf(f.u[2]);
  float lo[3], hi[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const float rx = f.r[3 * k], ry = f.r[3 * k + 1], rz = f.r[3 * k + 2];
    const float q = fmaf(rx, p.x, fmaf(ry, p.y, rz * p.z));
    const float m = fmaf(fabsf(rx), fabsf(p.x), fmaf(fabsf(ry), fabsf(p.y), fabsf(rz) * fabsf(p.z)));
    const float v = fmaf(rx, vx, fmaf(ry, vy, rz * vz));
    const float mv = fmaf(fabsf(rx), ax, fmaf(fabsf(ry), ay, fabsf(rz) * az));
    swept_axis(q, __fmaf_ru(m, e6, 1e-30f), v, __fmaf_ru(mv, e6, 1e-30f), Llo, Lhi, half, lo[k],
               hi[k]);
  }
  b.lx = lo[0];
  b.ly = lo[1];
  b.lz = lo[2];
  b.hx = hi[0];
  b.hy = hi[1];
  b.hz = hi[2];
  return b;
}

// Index along the n-dimensional Hilbert curve of 2^b cells a side (J. Skilling,
// "Programming the Hilbert curve", AIP Conf. Proc. 707, 2004): neighbouring indices
// are neighbouring cells, so 32 consecutive photons fill a compact region.
template <int N>
__device__ __forceinline__ uint32_t hilbert(uint32_t *x, int b) {
  for (int q = b - 1; q > 0; --q) {
    const uint32_t low = (1u << q) - 1u;
#pragma unroll
    for (int i = 0; i < N; ++i) {
      const bool set = x[i] >> q & 1u;  // invert the low bits of axis 0, or swap them with axis i's
      const uint32_t t = set ? low : (x[0] ^ x[i]) & low;
      x[0] ^= t;
      if (!set) x[i] ^= t;
    }
  }
#pragma unroll
  for (int i = 1; i < N; ++i) x[i] ^= x[i - 1];  // Gray encode
  uint32_t t = x[N - 1];
  t ^= t >> 1;
  t ^= t >> 2;
  t ^= t >> 4;
  t ^= t >> 8;
  t >>= 1;
  uint32_t h = 0u;  // interleave, axis 0 highest
#pragma unroll
  for (int i = 0; i < N; ++i) {
    uint32_t v = (x[i] ^ t) & ((1u << b) - 1u);
    if (N == 3) {  // up to 10 bits
      v = (v | v << 16) & 0x030000ffu;
      v = (v | v << 8) & 0x0300f00fu;
      v = (v | v << 4) & 0x030c30c3u;
      v = (v | v << 2) & 0x09249249u;
    } else {  // up to 16 bits
      v = (v | v << 8) & 0x00ff00ffu;
      v = (v | v << 4) & 0x0f0f0f0fu;
      v = (v | v << 2) & 0x33333333u;
      v = (v | v << 1) & 0x55555555u;
    }
    h |= v << (N - 1 - i);
  }
  return h;
}

// Order key of a point of the frame: the excess bits of the longest axis, then a 2D
// Hilbert index of the two longest axes' excess over the shortest, then a 3D one of
// what all three have.
__device__ __forceinline__ uint32_t order_key(const TLGrid &g, const float c[3]) {
  uint32_t x[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const int a = g.perm[k];
    const float v = a == 0 ? c[0] : (a == 1 ? c[1] : c[2]);
    const float fq = fminf(fmaxf((v - g.lo[a]) * g.scale[a], 0.0f), (float)((1u << g.nb[a]) - 1u));
    x[k] = (uint32_t)fq;
  }
  const int b1 = g.nb[g.perm[1]], b2 = g.nb[g.perm[2]];
  uint32_t key = x[0] >> b1;
  uint32_t y[2] = {(x[0] & ((1u << b1) - 1u)) >> b2, x[1] >> b2};
  key = key << (2 * (b1 - b2)) | hilbert<2>(y, b1 - b2);
  const uint32_t low = (1u << b2) - 1u;
  uint32_t z[3] = {x[0] & low, x[1] & low, x[2] & low};
  return key << (3 * b2) | hilbert<3>(z, b2);
}

#endif
