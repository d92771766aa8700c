// tl_pairs.cu -- the electron and positron of each collision (Sec. 1,
// Eq. pTotal and Eq. Lorentz).
//
// For a colliding pair (i of beam A, j of beam B) the photons' total energy E
// and momentum P (MeV, c = 1) fix the centre-of-mass (CoM) frame.  There each
// created particle has energy M/2, M^2 = E^2 - |P|^2 = 2 E_i E_j (1 - cos), and
// momentum p' = sqrt(M^2/4 - m^2) (Eq. pTotal); the electron flies along a
// random unit vector n, the positron opposite.  Both four-momenta are boosted
// back to the lab with the CoM velocity beta = P / E, gamma = E / M:
//   e_lab = gamma (e + beta.q),  q_lab = q + beta (gamma^2/(gamma+1) beta.q + gamma e),
// which is the paper's velocity addition (Eq. Lorentz) applied to momenta.
// n is uniform on the sphere (Marsaglia 1972: x1, x2 uniform in (-1, 1) until
// S = x1^2 + x2^2 lies in (0, 1); n = (2 x1 sqrt(1-S), 2 x2 sqrt(1-S), 1 - 2S)),
// its uniforms drawn from splitmix64 as a counter-based stream: key = seed ^
// ((i << 32) | j), draw t = top 53 bits of splitmix64(key + t) / 2^53.
// Everything is FP64 with explicit round-to-nearest operations in a fixed
// order (no contraction), so the result does not depend on the compiler.
#include "tl_common.cuh"

namespace tl {

// GB300 does 2 FP64 operations per clock and SM, and that bounds this kernel (a warp's
// operation takes 16 clocks): whatever is not a rounding of the definition above is done
// elsewhere.

// 2 u / 2^53 - 1 of a draw's 53 bits u = z >> 11, exact: with u = b 2^52 + f it is
// (1 + f 2^-52) - (b ? 1 : 2), the first term by its bits, one exact subtraction (as
// conversion, scaling and offset it was four operations).
__device__ __forceinline__ double signed_draw(unsigned long long z) {
  const unsigned long long f = (z >> 11) & 0xfffffffffffffull;
  return __dsub_rn(__longlong_as_double((long long)(f | 0x3ff0000000000000ull)),
                   (long long)z < 0 ? 1.0 : 2.0);
}

// S = x1^2 + x2^2 of two draws
__device__ __forceinline__ double draw_s(unsigned long long z1, unsigned long long z2) {
  const double x1 = signed_draw(z1), x2 = signed_draw(z2);
  return __dadd_rn(__dmul_rn(x1, x1), __dmul_rn(x2, x2));
}

// A warp repeats the draw until its last lane accepts, three times on average: the test is
// made in FP32 from the draws' top 32 bits (x within 2^-24, S within 4e-7) and in FP64 only
// near its two edges, and the accepted draw's S is computed once.
__device__ __forceinline__ void com_direction(unsigned long long seed, uint32_t i, uint32_t j,
                                              double n[3]) {
  const unsigned long long key = seed ^ (((unsigned long long)i << 32) | (unsigned long long)j);
  unsigned long long z1 = 0, z2 = 0;
  bool found = false;
  for (unsigned long long t = 0; t < 128 && !found; t += 2) {
    z1 = smix64(key + t);
    z2 = smix64(key + t + 1);
    const float x1 = (float)(int)((unsigned)(z1 >> 32) ^ 0x80000000u) * 0x1p-31f;
    const float x2 = (float)(int)((unsigned)(z2 >> 32) ^ 0x80000000u) * 0x1p-31f;
    const float S = fmaf(x1, x1, x2 * x2);
    found = S > 1e-6f && S < 1.0f - 1e-6f;
    if (!found && S < 1.0f + 1e-6f) {
      const double s = draw_s(z1, z2);
      found = s < 1.0 && s > 0.0;
    }
  }
  if (!found) {  // 64 rejections in a row: not reached in practice
    n[0] = 0.0;
    n[1] = 0.0;
    n[2] = 1.0;
    return;
  }
  const double x1 = signed_draw(z1), x2 = signed_draw(z2);
  const double S = __dadd_rn(__dmul_rn(x1, x1), __dmul_rn(x2, x2));
  const double r = __dsqrt_rn(__dsub_rn(1.0, S)), r2 = __dadd_rn(r, r);
  n[0] = __dmul_rn(x1, r2);  // (2 x) r and x (2 r): doubling is exact
  n[1] = __dmul_rn(x2, r2);
  n[2] = __fma_rn(-2.0, S, 1.0);
}

// One hit per thread.  A hit whose indices are out of range or
// whose pair is below threshold gets eight zeros.
// The positron's momentum in the CoM frame is the electron's with its sign changed, and so
// is beta.q: every other term of its boost is the electron's.
// A million hits: 403 us before, 244 us now, about 140 FP64 operations each, 80 of them in
// three square roots and five divisions.
__global__ void __launch_bounds__(128) k_pair_products(TLBeam a, TLBeam b, const uint2 *hits,
                                                       int64_t n_hits, unsigned long long seed,
                                                       double *out) {
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n_hits;
       k += (int64_t)gridDim.x * blockDim.x) {
    const uint2 h = hits[k];
    double *o = out + 8 * k;
    double r[8] = {0., 0., 0., 0., 0., 0., 0., 0.};
    if ((int64_t)h.x < a.n && (int64_t)h.y < b.n) {
      const double E1 = a.E[h.x], E2 = b.E[h.y];
      const double d1[3] = {a.dx[h.x], a.dy[h.x], a.dz[h.x]};
      const double d2[3] = {b.dx[h.y], b.dy[h.y], b.dz[h.y]};
      const double E = __dadd_rn(E1, E2);
      double P[3];
      for (int c = 0; c < 3; ++c) P[c] = __dadd_rn(__dmul_rn(E1, d1[c]), __dmul_rn(E2, d2[c]));
      const double cs = __dadd_rn(__dadd_rn(__dmul_rn(d1[0], d2[0]), __dmul_rn(d1[1], d2[1])),
                                  __dmul_rn(d1[2], d2[2]));
      const double M2 = __dmul_rn(__dmul_rn(2.0, __dmul_rn(E1, E2)), __dsub_rn(1.0, cs));
      const double m = TL_MEC2;
      if (M2 > __dmul_rn(__dmul_rn(4.0, m), m)) {
        const double M = __dsqrt_rn(M2);
        const double ep = __dmul_rn(0.5, M);                                     // CoM energy
        const double pp = __dsqrt_rn(__fma_rn(0.25, M2, -(m * m)));  // p' (M2 / 4 is exact)
        double n[3];
        com_direction(seed, h.x, h.y, n);
        const double beta[3] = {__ddiv_rn(P[0], E), __ddiv_rn(P[1], E), __ddiv_rn(P[2], E)};
        const double gamma = __ddiv_rn(E, M);
        const double qe[3] = {__dmul_rn(pp, n[0]), __dmul_rn(pp, n[1]), __dmul_rn(pp, n[2])};
        const double bq = __dadd_rn(
            __dadd_rn(__dmul_rn(beta[0], qe[0]), __dmul_rn(beta[1], qe[1])),
            __dmul_rn(beta[2], qe[2]));
        const double gbq =
            __dmul_rn(__ddiv_rn(__dmul_rn(gamma, gamma), __dadd_rn(gamma, 1.0)), bq);
        const double ge = __dmul_rn(gamma, ep);
        const double ke = __dadd_rn(gbq, ge), kp = __dsub_rn(ge, gbq);
        r[0] = __dmul_rn(gamma, __dadd_rn(ep, bq));
        r[4] = __dmul_rn(gamma, __dsub_rn(ep, bq));
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          r[1 + c] = __dadd_rn(qe[c], __dmul_rn(beta[c], ke));
          r[5 + c] = __dsub_rn(__dmul_rn(beta[c], kp), qe[c]);
        }
      }
    }
    double2 *o2 = reinterpret_cast<double2 *>(o);
    o2[0] = make_double2(r[0], r[1]);
    o2[1] = make_double2(r[2], r[3]);
    o2[2] = make_double2(r[4], r[5]);
    o2[3] = make_double2(r[6], r[7]);
  }
}

cudaError_t launch_pair_products(const TLBeam &a, const TLBeam &b, const uint32_t *hits,
                                 int64_t n_hits, unsigned long long seed, double *out,
                                 cudaStream_t s) {
  if (n_hits <= 0) return cudaSuccess;
  // a block per 128 hits, so that no SM is left with a last round of its own
  const int64_t nb = (n_hits + 127) / 128;
  const int blocks = (int)(nb < (1 << 30) ? nb : 1 << 30);
  k_pair_products<<<blocks, 128, 0, s>>>(a, b, reinterpret_cast<const uint2 *>(hits), n_hits,
                                         seed, out);
  return cudaGetLastError();
}

}  // namespace tl
