// tl_warp.cuh -- warp-wide output of hits and band pairs, shared by the narrow phases.
#pragma once
#include "tl_common.cuh"
#include "tl_exact.cuh"
#include "tl_narrow.cuh"

namespace tl {

// warp-aggregated append of (x, y) for lanes with pred
__device__ __forceinline__ void emit(bool pred, uint32_t x, uint32_t y, uint2 *buf,
                                     unsigned long long cap, unsigned long long *counter,
                                     unsigned *status, unsigned ovf_bit, int lane) {
  const unsigned m = __ballot_sync(0xffffffffu, pred);
  if (!m) return;
  unsigned long long base = 0;
  if (lane == 0) base = atomicAdd(counter, (unsigned long long)__popc(m));
  base = __shfl_sync(0xffffffffu, base, 0);
  if (pred) {
    const unsigned long long idx = base + __popc(m & ((1u << lane) - 1u));
    if (idx < cap) buf[idx] = make_uint2(x, y);
  }
  if (lane == 0 && base + __popc(m) > cap) atomicOr(status, ovf_bit);
}

// The full test of one photon pair per lane (pr: positions in the two beams' sorted
// photons; lanes without ok have none); hits and band pairs leave with one atomic per
// warp each.
template <bool FP64>
__device__ __forceinline__ void decide_pairs(const TravArgs &a, const uint2 pr, bool ok, int lane,
                                             const float *sbin) {
  int outcome = TL_MISS;
  uint32_t oi = 0u, oj = 0u;
  if (ok) {
    const size_t ia = (size_t)pr.x * a.A.stride, jb = (size_t)pr.y * a.B.stride;
    const float4 da = __ldg(a.A.dir + ia), db = __ldg(a.B.dir + jb);
    oi = __float_as_uint(da.w);
    oj = __float_as_uint(db.w);
    if (FP64) {
      outcome = tl_exact_hit(a.mA, oi, a.mB, oj, a.ct, a.dt, a.kappa) ? TL_HIT : TL_MISS;
    } else {
      const float4 pa = __ldg(a.A.pos + ia), pb = __ldg(a.B.pos + jb);
      outcome = tl_narrow32(pa, da, pb, db, a.nk, sbin);
    }
  }
  emit(outcome == TL_HIT, oi, oj, a.hits, a.hit_cap, &a.ctr->hits, &a.ctr->status,
       TL_ST_HIT_OVF, lane);
  if (!FP64)
    emit(outcome == TL_BAND, oi, oj, a.band, a.band_cap, &a.ctr->band, &a.ctr->status,
         TL_ST_BAND_OVF, lane);
}

}  // namespace tl
