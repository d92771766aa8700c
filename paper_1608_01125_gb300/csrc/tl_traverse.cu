// tl_traverse.cu -- dual traversal of two binary hierarchies from a list of node pairs,
// its narrow phase, the FP64 band re-test and the per-step yield reduction.
//
// The statistical regime works on pairs of the hierarchies' level-L nodes: its exact
// labels and its exact fallback are the collisions below given node pairs.  Persistent
// warps take pairs of the list and descend depth first (Sec. 2.2; a failed overlap
// test, Eq. CollDet, skips the whole subtree pair) with a stack of node pairs in shared
// memory, handing large items on to a device work queue (see k_traverse).  Each
// iteration a warp pops up to 32 pairs, one per lane; a lane loads both
// node records of its pair once and tests the up-to-4 child combinations
// (both children of each side); survivors are pushed (or, when both sides
// are leaf buckets, appended to the step's leaf-pair list in blocks of at
// least 32) with ballot/popc compaction.  A separate kernel (k_narrow) then tests the
// listed bucket pairs' photon pairs.  (The exact path of whole beams is tl_tree.cu.)
#include "tl_common.cuh"
#include "tl_exact.cuh"
#include "tl_narrow.cuh"
#include "tl_warp.cuh"
#include "tl_yield.cuh"

namespace tl {


__device__ __forceinline__ uint32_t pack_bucket(uint32_t first, uint32_t cnt) {
  return first | ((cnt - 1u) << 27);
}

// Child i (0 or 1) of one side of a popped pair, from the side's node record
// rec: for an inner node (ref without FLAG) its child i; for a bucket (ref =
// FLAG | parent << 1 | slot, rec = the parent's record) the bucket itself
// (i = 0 only).
struct Kid {
  TLBox box;
  uint32_t sref;  // stack reference
  uint32_t pack;  // bucket as (first photon | (count - 1) << 27)
  bool bucket;
};

__device__ __forceinline__ Kid kid_of(const TLNode &rec, uint32_t ref, int i) {
  Kid k;
  uint32_t node, sl;
  if (ref & TL_FLAG) {
    node = (ref & ~TL_FLAG) >> 1;
    sl = ref & 1u;
  } else {
    node = ref;
    sl = (uint32_t)i;
  }
  k.box = tl_child_box(rec, (int)sl);
  const uint32_t cr = (uint32_t)(sl ? rec.c.y : rec.c.x);
  const uint32_t cnt = (uint32_t)(sl ? rec.c.w : rec.c.z);
  k.bucket = (cr & TL_FLAG) != 0u;
  k.pack = pack_bucket(cr & ~TL_FLAG, cnt);
  k.sref = (ref & TL_FLAG) ? ref : (k.bucket ? (TL_FLAG | (node << 1) | sl) : cr);
  return k;
}

__device__ __forceinline__ TLNode node_record(const TLTree &T, uint32_t ref) {
  const uint32_t node = (ref & TL_FLAG) ? ((ref & ~TL_FLAG) >> 1) : ref;
  const float4 *f = reinterpret_cast<const float4 *>(T.nodes + node);
  TLNode v;
  v.b0 = __ldg(f + 0);
  v.b1 = __ldg(f + 1);
  v.b2 = __ldg(f + 2);
  v.c = __ldg(reinterpret_cast<const int4 *>(f + 3));
  return v;
}

// ------------------------------------------------------------ narrow phase

// a traversal warp's leaf-pair queue: fewer than 32 entries before an iteration,
// at most 4 new ones per lane in it
constexpr int kLeafQ = 32 + 4 * 32;

struct TravSmem {
  uint2 leafq[kLeafQ];
};

constexpr int kItemsPerLane = 16;  // photon pairs of a leaf pair per pass

struct NarrowSmem {
  uint2 leafq[32];
  uint2 pend[64];  // photon pairs the first look left undecided
  uint16_t items[32 * kItemsPerLane];
};

// the full test of the first cnt (<= 32) pending photon pairs
template <bool FP64>
__device__ __forceinline__ void decide_pending(const TravArgs &a, const NarrowSmem &ws, int cnt,
                                               int lane, const float *sbin) {
  decide_pairs<FP64>(a, lane < cnt ? ws.pend[lane] : make_uint2(0u, 0u), lane < cnt, lane, sbin);
}

// ------------------------------------------------------------ traversal

// Persistent warps share one work queue.  Its items come first from the
// list, in groups of up to 32 node pairs (indices below nf), then from
// the queue's chunks of up to 32 node pairs each (256 bytes).  A warp that
// waits for a chunk is counted in ctr->hungry while it waits; a warp that
// has spent `budget` iterations on its item while h > 0 warps wait hands on
// up to h chunks.  A warp's own stack has two
// levels: the top in shared memory (D entries), the bottom in its private
// spill area in global memory.  A warp pops at most P = min(32, D / 8) pairs
// per iteration (so it pushes at most 4P); when the next iteration's pushes
// might not fit its shared stack, the bottom of it (up to D / 2 entries)
// moves to the spill area, and when the shared stack runs dry it is refilled from the
// spill area's top.  So no work leaves a warp except the chunks it hands on
// to waiting warps, taken from the bottom of its spill area first (the
// shallowest pairs it holds), else from the bottom of its shared stack.
// Unused and free entries hold a sentinel.  A writer fills a chunk's entries
// 1..31, fences, then swaps entry 0 in; a taker swaps the sentinel back into
// entry 0 as it reads it (atomic exchange) and waits while it is still free
// and work is in flight.  The traversal ends when the items finished equal
// nf plus the chunks handed on.  Every wait is bounded by spin_limit (then
// TL_ST_TIMEOUT).
constexpr unsigned long long kQFree = 0xffffffffffffffffull;
constexpr int kGroup = 32;  // listed pairs per item, node pairs per queue chunk

__device__ __forceinline__ unsigned long long pack2(uint2 v) {
  return (unsigned long long)v.x | ((unsigned long long)v.y << 32);
}

// chunks a working warp hands on per waiting warp, at most
#ifndef TL_DONATE_MAX
#define TL_DONATE_MAX 1
#endif

// Launch bounds: at most 8 warps per block and registers for 4 such blocks
// per SM (63 registers, no spills; the narrow phase is a kernel of its own).
#ifndef TL_TRAV_MINBLOCKS
#define TL_TRAV_MINBLOCKS 4
#endif
// A warp's queued leaf pairs to the step's list (one atomic per warp), from
// the current part's start lbase.  The count keeps every leaf pair; pairs
// past the list's end are dropped and the step is flagged (TL_ST_LEAFQ): the
// host grows the list, or splits the step into more parts, and repeats it.
__device__ __forceinline__ void spill_leaves(const TravArgs &a, const TravSmem &ws, int nq,
                                             int lane, unsigned long long lbase) {
  unsigned long long base = 0;
  if (lane == 0) base = atomicAdd(&a.ctr->leaf_pairs, (unsigned long long)nq) - lbase;
  base = __shfl_sync(0xffffffffu, base, 0);
  for (int e = lane; e < nq; e += 32)
    if (base + e < a.leaf_cap) a.leaves[base + e] = ws.leafq[e];
  if (lane == 0 && base + nq > a.leaf_cap) atomicOr(&a.ctr->status, (unsigned)TL_ST_LEAFQ);
}

__global__ void __launch_bounds__(TL_TRAV_MAX_WARPS * 32, TL_TRAV_MINBLOCKS) k_traverse(
    TravArgs a, const uint2 *list, unsigned long long list_n, int budget, int part, int nparts) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int D = a.stack_depth;
  uint2 *stack = reinterpret_cast<uint2 *>(smem_raw) + (size_t)warp * D;
  TravSmem &ws = reinterpret_cast<TravSmem *>(
      smem_raw + sizeof(uint2) * (size_t)D * (blockDim.x >> 5))[warp];
  TLCounters *ctr = a.ctr;
  // After a queue overflow or an expired wait in this step (an earlier part)
  // or this run, the queue may hold chunks that no warp will take: a warp
  // taking one would count an item the counters never handed on, and the
  // step's end would no longer be seen.  The host repeats the step (or run)
  // with the queue reset, so nothing more is traversed here.
  if (*(volatile unsigned *)&ctr->status & (TL_ST_SPILL_OVF | TL_ST_TIMEOUT)) return;
  // this launch's part of the list: the parts split the step's work
  const unsigned long long lo = list_n * (unsigned long long)part / (unsigned long long)nparts;
  const unsigned long long hi = list_n * (unsigned long long)(part + 1) / (unsigned long long)nparts;
  const uint2 *src0 = list + lo;
  const unsigned long long n0 = hi - lo;
  const unsigned long long lbase = ctr->leaf_base;  // the list of this part starts here
  const unsigned long long nf = (n0 + kGroup - 1) / kGroup;  // groups of listed pairs
  unsigned long long *Q = a.queue;
  const unsigned long long qcap = a.queue_cap / kGroup;  // chunks
  const unsigned lt = (1u << lane) - 1u;
  // the private spill area: entries [gbot, gtop) hold the stack's bottom
  uint2 *gs = a.spill + (size_t)(blockIdx.x * (blockDim.x >> 5) + warp) * a.spill_per_warp;
  const int W = (int)a.spill_per_warp;
  const int P = min(32, D >> 3);  // pops per iteration at most
  int gbot = 0, gtop = 0;
  int sp = 0, nq = 0, iters = 0;
  bool holding = false;  // this warp holds an item (counted in flight)
  bool handed = false;   // ... and has handed pieces of it on
  unsigned long long node_tests = 0;
  while (true) {
    // the bottom of a shared stack that could not take the next iteration's
    // pushes (min(sp, P) pops, 4 pushes each) moves to the spill area
    if (sp + 3 * min(sp, P) > D) {
      const int m = min(D >> 1, sp - P);
      if (gbot > 0 && gtop + m > W) {  // compact the spill area first
        const int cnt = gtop - gbot;
        for (int e0 = 0; e0 < cnt; e0 += 32) {
          uint2 v = make_uint2(0u, 0u);
          if (e0 + lane < cnt) v = gs[gbot + e0 + lane];
          __syncwarp();
          if (e0 + lane < cnt) gs[e0 + lane] = v;
          __syncwarp();
        }
        gtop = cnt;
        gbot = 0;
      }
      if (gtop + m <= W) {
        for (int e = lane; e < m; e += 32) gs[gtop + e] = stack[e];
        __syncwarp();
        for (int e0 = 0; e0 < sp - m; e0 += 32) {
          uint2 v = make_uint2(0u, 0u);
          if (e0 + lane < sp - m) v = stack[m + e0 + lane];
          __syncwarp();
          if (e0 + lane < sp - m) stack[e0 + lane] = v;
          __syncwarp();
        }
        gtop += m;
        sp -= m;
      } else if (lane == 0) {
        atomicOr(&ctr->status, (unsigned)TL_ST_PRIV_OVF);  // the host grows it, repeats the step
      }
    }
    // the shared stack ran dry: refill it from the spill area's top
    if (sp == 0 && gtop > gbot) {
      const int m = min(gtop - gbot, D >> 1);
      for (int e = lane; e < m; e += 32) stack[e] = gs[gtop - m + e];
      __syncwarp();
      gtop -= m;
      sp = m;
      if (gtop == gbot) gtop = gbot = 0;
    }
    if ((sp > 1 || gtop > gbot) && budget > 0 && iters >= budget) {
      unsigned h = 0;
      if (lane == 0) h = *(volatile unsigned *)&ctr->hungry;
      h = __shfl_sync(0xffffffffu, h, 0);
      iters = 0;
      if (h > 0u) {
        // hand on chunks of 32 to the waiting warps, at most TL_DONATE_MAX
        // per waiting warp: the spill area's entries (its bottom first), then
        // all but the top 32 entries of the shared stack (or half of a stack
        // of at most 64); they are counted (q_tail) before this item is
        // counted finished
        // chunks available, each non-empty: the spill area's, then those the
        // loop below cuts from the shared stack (every reserved chunk must be
        // published, so the count follows the loop's own cuts)
        int avail = (gtop - gbot + kGroup - 1) / kGroup;
        for (int r = sp; ; ) {
          const int g = min(kGroup, r > 2 * kGroup ? r - kGroup : r / 2);
          if (g < 1) break;
          ++avail;
          r -= g;
        }
        const int nch = (int)min((unsigned)avail, (unsigned)TL_DONATE_MAX * h);
        unsigned long long base = 0;
        if (lane == 0) base = atomicAdd(&ctr->q_tail, (unsigned long long)nch);
        handed = true;
        base = __shfl_sync(0xffffffffu, base, 0);
        for (int c = 0; c < nch; ++c) {
          const bool fs = gtop > gbot;
          const int give = fs ? min(kGroup, gtop - gbot)
                              : min(kGroup, sp > 2 * kGroup ? sp - kGroup : sp / 2);
          const uint2 *src = fs ? gs + gbot : stack;
          if (base + c < qcap) {
            if (lane >= 1)
              Q[(base + c) * kGroup + lane] = lane < give ? pack2(src[lane]) : kQFree;
            __threadfence();
            __syncwarp();
            if (lane == 0 && atomicExch(Q + (base + c) * kGroup, pack2(src[0])) != kQFree)
              atomicOr(&ctr->status, (unsigned)TL_ST_SPILL_OVF);  // a chunk was not free
          } else if (lane == 0) {
            atomicOr(&ctr->status, (unsigned)TL_ST_SPILL_OVF);
          }
          __syncwarp();
          if (fs) {
            gbot += give;
            if (gbot == gtop) gbot = gtop = 0;
          } else {  // the kept entries move to the bottom
            const int keep = sp - give;
            for (int e0 = 0; e0 < keep; e0 += 32) {
              uint2 v = make_uint2(0u, 0u);
              if (e0 + lane < keep) v = stack[give + e0 + lane];
              __syncwarp();
              if (e0 + lane < keep) stack[e0 + lane] = v;
              __syncwarp();
            }
            sp = keep;
          }
        }
      }
    }
    if (sp == 0) {
      int got = 0;  // 1: a group of listed pairs; 2: a queue chunk
      unsigned long long idx = 0;
      uint2 item = make_uint2(0u, 0u);
      if (lane == 0) {
        if (holding) {
          if (handed) __threadfence();  // this item's hand-ons (q_tail) before its finish
          atomicAdd(&ctr->q_done, 1ull);
          holding = false;
        }
        handed = false;
        const unsigned long long i = atomicAdd(&ctr->q_head, 1ull);
        if (i < nf) {
          idx = i;
          got = 1;
        } else if (i - nf < qcap) {
          idx = i - nf;
          unsigned long long *slot = Q + idx * kGroup;
          long long spins = 0;
          unsigned ns = 32;
          bool waiting = false;
          while (true) {
            const unsigned long long v = atomicExch(slot, kQFree);
            if (v != kQFree) {
              item = make_uint2((unsigned)v, (unsigned)(v >> 32));
              got = 2;
              __threadfence();  // entry 0 seen: the chunk's other entries are written
              break;
            }
            if (!waiting) {  // working warps see that a warp waits for work
              waiting = true;
              atomicAdd(&ctr->hungry, 1u);
            }
            // finished items first, then hand-ons: equal means nothing was in
            // flight at the first read, so nothing more can come
            const unsigned long long done = *(volatile unsigned long long *)&ctr->q_done;
            __threadfence();
            const unsigned long long tail = *(volatile unsigned long long *)&ctr->q_tail;
            if (done >= nf + tail) break;
            if (*(volatile unsigned *)&ctr->status & (TL_ST_SPILL_OVF | TL_ST_TIMEOUT)) break;
            if (++spins > a.spin_limit) {
              atomicOr(&ctr->status, (unsigned)TL_ST_TIMEOUT);
              break;
            }
            __nanosleep(ns);
            if (ns < 1024) ns <<= 1;
          }
          if (waiting) atomicSub(&ctr->hungry, 1u);
        }
        // an index past the queue's end: its producer flagged the overflow
      }
      got = __shfl_sync(0xffffffffu, got, 0);
      if (!got) break;
      idx = __shfl_sync(0xffffffffu, idx, 0);
      if (got == 1) {  // up to 32 listed pairs
        const unsigned long long f = idx * kGroup + (unsigned long long)lane;
        const bool have = f < n0;
        if (have) stack[lane] = __ldcg(src0 + f);
        sp = __popc(__ballot_sync(0xffffffffu, have));
      } else {  // entries 1..31 of the chunk: the written ones come first
        unsigned long long v = kQFree;
        if (lane >= 1) v = __ldcg(Q + idx * kGroup + lane);
        const unsigned mv = __ballot_sync(0xffffffffu, v != kQFree);
        if (v != kQFree) stack[lane] = make_uint2((unsigned)v, (unsigned)(v >> 32));
        if (lane == 0) stack[0] = item;
        sp = 1 + __popc(mv);
      }
      if (lane == 0) holding = true;
      __syncwarp();
      iters = 0;
    }
    ++iters;
    // one popped pair per lane
    const int npop = min(sp, P);
    sp -= npop;
    const bool active = lane < npop;
    const uint2 pr = active ? stack[sp + lane] : make_uint2(0u, 0u);
    __syncwarp();
    const bool bka = (pr.x & TL_FLAG) != 0u, bkb = (pr.y & TL_FLAG) != 0u;
    TLNode ra, rb;
    if (active) {
      ra = node_record(a.A, pr.x);
      rb = node_record(a.B, pr.y);
    }
    // a bucket pair taken from the list was tested when it was produced
    const bool pass = active && bka && bkb;
    int tested = 0;
#pragma unroll
    for (int combo = 0; combo < 4; ++combo) {
      const int ia = combo >> 1, ib = combo & 1;
      bool ok = false, leaf = false;
      uint2 o = make_uint2(0u, 0u);
      if (pass) {
        if (combo == 0) {
          const Kid ka = kid_of(ra, pr.x, 0), kb = kid_of(rb, pr.y, 0);
          ok = leaf = true;
          o = make_uint2(ka.pack, kb.pack);
        }
      } else if (active && !(bka && ia) && !(bkb && ib)) {
        const Kid ka = kid_of(ra, pr.x, ia), kb = kid_of(rb, pr.y, ib);
        ++tested;
        ok = tl_overlap(ka.box, kb.box);
        leaf = ka.bucket && kb.bucket;
        o = leaf ? make_uint2(ka.pack, kb.pack) : make_uint2(ka.sref, kb.sref);
      }
      const unsigned mpush = __ballot_sync(0xffffffffu, ok && !leaf);
      const unsigned mleaf = __ballot_sync(0xffffffffu, ok && leaf);
      if (sp + __popc(mpush) > D) handed = true;  // (warp-uniform)
      if (ok && !leaf) {
        const int slot = sp + __popc(mpush & lt);
        if (slot < D) {
          stack[slot] = o;
        } else {  // the stack is full: this pair goes to the queue as a chunk of one
          const unsigned long long qi = atomicAdd(&ctr->q_tail, 1ull);
          if (qi < qcap) {
            for (int k = 1; k < kGroup; ++k) Q[qi * kGroup + k] = kQFree;
            __threadfence();
            if (atomicExch(Q + qi * kGroup, pack2(o)) != kQFree)
              atomicOr(&ctr->status, (unsigned)TL_ST_SPILL_OVF);
          } else {
            atomicOr(&ctr->status, (unsigned)TL_ST_SPILL_OVF);
          }
        }
      }
      sp = min(sp + __popc(mpush), D);
      if (ok && leaf) ws.leafq[nq + __popc(mleaf & lt)] = o;
      nq += __popc(mleaf);
    }
    for (int off = 16; off; off >>= 1) tested += __shfl_xor_sync(0xffffffffu, tested, off);
    if (lane == 0) node_tests += (unsigned long long)tested;
    __syncwarp();
    if (nq >= 32) {
      spill_leaves(a, ws, nq, lane, lbase);
      nq = 0;
    }
  }
  if (nq) spill_leaves(a, ws, nq, lane, lbase);
  if (lane == 0 && node_tests) atomicAdd(&ctr->node_tests, node_tests);
}

// The narrow phase of the step's listed leaf pairs.  What bounds it is instruction
// issue (most photon pairs need only the first look, ~60 FP32 instructions), so the
// work around that look is kept small: a warp takes 32 leaf pairs, one per lane, each
// lane writes its photon pairs (lane, i, j) to a list in shared memory, at most
// kItemsPerLane per pass (all of a pair of 4-photon buckets), and the warp then takes
// the list 32 at a time with every lane busy.  The pairs the first look leaves
// undecided are queued and given the full test 32 at a time, so that the long path
// runs on full warps too.  FP64 mode: the first look is tl_exact_sure_miss, the full
// test the definition.  2 x 4M statistical step, 1.6e9 photon pairs: 14.6 ms when each
// lane found its pair by a binary search over a scan of the pair sizes and a division
// (9.4 warp instructions per photon pair), 9.5 ms now.
template <bool FP64>
__global__ void __launch_bounds__(256) k_narrow(TravArgs a) {
  __shared__ NarrowSmem wsm[8];
  __shared__ float sbin[TL_SBINS], suf[TL_SBINS];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const unsigned lt = (1u << lane) - 1u;
  NarrowSmem &ws = wsm[warp];
  const unsigned long long listed = a.ctr->leaf_pairs - a.ctr->leaf_base;  // this part's
  const unsigned long long n = min(listed, a.leaf_cap);
  if (blockIdx.x == 0 && threadIdx.x == 0) atomicMax(&a.ctr->max_part_leaves, listed);
  const unsigned long long stride = (unsigned long long)gridDim.x * 8ull * 32ull;
  if ((unsigned long long)blockIdx.x * 8ull * 32ull >= n) return;
  if (!FP64) {
    for (int i = threadIdx.x; i < TL_SBINS; i += blockDim.x) {
      sbin[i] = a.nk.sbin[i];
      suf[i] = a.nk.suf[i];
    }
    __syncthreads();
  }
  unsigned long long tests = 0;
  int npend = 0;
  for (unsigned long long base = ((unsigned long long)blockIdx.x * 8ull + warp) * 32ull; base < n;
       base += stride) {
    uint32_t ca = 0u, cb = 0u;
    if (base + lane < n) {
      const uint2 q = a.leaves[base + lane];
      ca = (q.x >> 27) + 1u;
      cb = (q.y >> 27) + 1u;
      ws.leafq[lane] = make_uint2(q.x & 0x7FFFFFFu, q.y & 0x7FFFFFFu);
    }
    uint32_t left = ca * cb, ia = 0u, jb = 0u;  // this lane's pairs not listed yet, the next one
    while (__any_sync(0xffffffffu, left > 0u)) {
      const int c = (int)min(left, (uint32_t)kItemsPerLane);
      int inc = c;
#pragma unroll
      for (int off = 1; off < 32; off <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, inc, off);
        if (lane >= off) inc += t;
      }
      const int total = __shfl_sync(0xffffffffu, inc, 31);
      for (int k = inc - c; k < inc; ++k) {
        ws.items[k] = (uint16_t)((uint32_t)lane | ia << 5 | jb << 10);
        if (++jb == cb) {
          jb = 0u;
          ++ia;
        }
      }
      left -= (uint32_t)c;
      __syncwarp();
      tests += (unsigned long long)total;
      for (int t0 = 0; t0 < total; t0 += 32) {
        bool undecided = false;
        uint32_t si = 0u, sj = 0u;
        if (t0 + lane < total) {
          const uint32_t it = ws.items[t0 + lane];
          const uint2 q = ws.leafq[it & 31u];
          si = q.x + (it >> 5 & 31u);
          sj = q.y + (it >> 10);
          const float4 da = __ldg(a.A.dir + si), db = __ldg(a.B.dir + sj);
          if (FP64) {
            undecided = !tl_exact_sure_miss(a.mA, __float_as_uint(da.w), a.mB,
                                            __float_as_uint(db.w), a.ct, a.dt, (double)a.nk.r2max);
          } else {
            const float4 pa = __ldg(a.A.pos + si), pb = __ldg(a.B.pos + sj);
            undecided = !tl_narrow32_sure_miss(pa, da, pb, db, a.nk, suf);
          }
        }
        const unsigned mu = __ballot_sync(0xffffffffu, undecided);
        if (!mu) continue;
        if (undecided) ws.pend[npend + __popc(mu & lt)] = make_uint2(si, sj);
        npend += __popc(mu);
        __syncwarp();
        if (npend >= 32) {
          decide_pending<FP64>(a, ws, 32, lane, sbin);
          // the rest (fewer than 32) move to the front
          const int rest = npend - 32;
          uint2 v = make_uint2(0u, 0u);
          if (lane < rest) v = ws.pend[32 + lane];
          __syncwarp();
          if (lane < rest) ws.pend[lane] = v;
          __syncwarp();
          npend = rest;
        }
      }
      __syncwarp();
    }
  }
  if (npend > 0) decide_pending<FP64>(a, ws, npend, lane, sbin);
  if (lane == 0 && tests) atomicAdd(&a.ctr->narrow_tests, tests);
}

// ------------------------------------------------------------ band re-test

__global__ void __launch_bounds__(256) k_band(TravArgs a) {
  const int lane = threadIdx.x & 31;
  const unsigned long long n = min(a.ctr->band, a.band_cap);
  const unsigned long long stride = (unsigned long long)gridDim.x * blockDim.x;
  const unsigned long long nround = (n + 31ull) & ~31ull;
  for (unsigned long long i = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; i < nround;
       i += stride) {
    bool hit = false;
    uint2 q = make_uint2(0u, 0u);
    if (i < n) {
      q = a.band[i];
      hit = tl_exact_hit(a.mA, q.x, a.mB, q.y, a.ct, a.dt, a.kappa);
    }
    emit(hit, q.x, q.y, a.hits, a.hit_cap, &a.ctr->hits, &a.ctr->status, TL_ST_HIT_OVF, lane);
  }
}

// ------------------------------------------------------------ yield

// Sum over the step's hits of w_i w_j (FP64), the count and the order-free
// checksums.  Per-block partials are combined by the last block to finish,
// in a fixed order.
__global__ void __launch_bounds__(256) k_yield(TravArgs a, YieldPartial *partials) {
  __shared__ YieldPartial sp[8];
  __shared__ bool last;
  const unsigned long long n = min(a.ctr->hits, a.hit_cap);
  YieldPartial p = yield_zero();
  for (unsigned long long i = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; i < n;
       i += (unsigned long long)gridDim.x * blockDim.x) {
    const uint2 h = a.hits[i];
    yield_hit(p, h.x, h.y, a.mA.w ? a.mA.w[h.x] : 1.0, a.mB.w ? a.mB.w[h.y] : 1.0);
  }
  const YieldPartial b = yield_block_reduce(p, sp);
  if (threadIdx.x == 0) {
    partials[blockIdx.x] = b;
    __threadfence();
    last = atomicAdd(&a.ctr->reduce_done, 1u) == gridDim.x - 1u;
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  YieldPartial t = yield_zero();
  for (unsigned q = threadIdx.x; q < gridDim.x; q += blockDim.x) yield_add(t, yield_load_volatile(partials + q));
  const YieldPartial tot = yield_block_reduce(t, sp);
  if (threadIdx.x == 0) {
    a.ctr->count = tot.count;
    a.ctr->weighted = tot.weighted;
    a.ctr->hsum = tot.hsum;
    a.ctr->hxor = tot.hxor;
  }
}

// Per-instance yield: count and sum of w_i w_j of each instance's hits,
// accumulated into yields[2 * inst], yields[2 * inst + 1].  A warp's hits mostly belong
// to one instance: its lanes are summed first, one pair of atomics per run of equal
// instances (two per hit on a few addresses took 4.8 ms of a 64-instance run of 16
// steps, this takes 0.29 ms).
__global__ void __launch_bounds__(256) k_yield_inst(TravArgs a, const uint32_t *inst_of_a,
                                                    double *yields) {
  const unsigned long long n = min(a.ctr->hits, a.hit_cap);
  const unsigned long long nround = (n + 31ull) & ~31ull;
  const int lane = threadIdx.x & 31;
  for (unsigned long long i = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; i < nround;
       i += (unsigned long long)gridDim.x * blockDim.x) {
    uint32_t q = TL_NONE;
    double w = 0.0;
    if (i < n) {
      const uint2 h = a.hits[i];
      w = (a.mA.w ? a.mA.w[h.x] : 1.0) * (a.mB.w ? a.mB.w[h.y] : 1.0);
      q = inst_of_a[h.x];
    }
    unsigned left = __ballot_sync(0xffffffffu, i < n);
    while (left) {
      const uint32_t q0 = __shfl_sync(0xffffffffu, q, __ffs(left) - 1);
      const unsigned m = __ballot_sync(0xffffffffu, q == q0);
      double s = q == q0 ? w : 0.0;
#pragma unroll
      for (int off = 16; off; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
      if (lane == 0) {
        atomicAdd(&yields[2 * (size_t)q0], (double)__popc(m));
        atomicAdd(&yields[2 * (size_t)q0 + 1], s);
      }
      left &= ~m;
    }
  }
}

// End of a step in graph mode: keep the step's status bits and add the
// step's yield and counters to the run's totals (acc may be NULL).
__global__ void k_step_finish(const TLCounters *ctr, unsigned *run_status, TLRunAcc *acc) {
  const unsigned st = ctr->status;
  if (st) atomicOr(run_status, st);
  if (acc) {
    acc->count += ctr->count;
    acc->weighted += ctr->weighted;
    acc->hsum += ctr->hsum;
    acc->hxor ^= ctr->hxor;
    acc->narrow_tests += ctr->narrow_tests;
    acc->node_tests += ctr->node_tests;
    acc->leaf_pairs += ctr->leaf_pairs;
    acc->band += ctr->band;
    if (ctr->hits > acc->max_hits) acc->max_hits = ctr->hits;
    if (ctr->band > acc->max_band) acc->max_band = ctr->band;
    if (ctr->max_part_leaves > acc->max_leaves) acc->max_leaves = ctr->max_part_leaves;
  }
}

// ------------------------------------------------------------ host launchers

size_t traverse_smem(int warps, int depth) {
  return sizeof(uint2) * (size_t)depth * warps + sizeof(TravSmem) * (size_t)warps;
}

cudaError_t traverse_config(int fp64, int warps, int depth, int *blocks_per_sm) {
  (void)fp64;  // the traversal is the same for both precisions (the narrow phase differs)
  const size_t smem = traverse_smem(warps, depth);
  cudaError_t e;
  if ((e = cudaFuncSetAttribute(k_traverse, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)smem)))
    return e;
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, k_traverse, warps * 32, smem);
}

cudaError_t launch_traverse(const TravArgs &a, const uint2 *list, unsigned long long list_n,
                            int budget, int blocks, int warps, cudaStream_t s, int part,
                            int nparts) {
  // a warp only waits for work that warps holding items (running ones) hand
  // on, so no block needs another to be resident
  const size_t smem = traverse_smem(warps, a.stack_depth);
  k_traverse<<<blocks, warps * 32, smem, s>>>(a, list, list_n, budget, part, nparts);
  return cudaGetLastError();
}

// Before part p > 0 of a step: the leaf list starts again (at the count so
// far) and the work queue's counters are cleared for the next traversal.
__global__ void k_part_init(TLCounters *ctr) {
  ctr->leaf_base = ctr->leaf_pairs;
  ctr->q_head = ctr->q_done = ctr->q_tail = 0ull;
  ctr->hungry = 0u;
}

cudaError_t launch_part_init(TLCounters *ctr, cudaStream_t s) {
  k_part_init<<<1, 1, 0, s>>>(ctr);
  return cudaGetLastError();
}

cudaError_t launch_narrow(const TravArgs &a, int blocks, cudaStream_t s) {
  if (a.fp64) k_narrow<true><<<blocks, 256, 0, s>>>(a);
  else k_narrow<false><<<blocks, 256, 0, s>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_band(const TravArgs &a, int blocks, cudaStream_t s) {
  k_band<<<blocks, 256, 0, s>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_yield(const TravArgs &a, void *partials, int blocks, cudaStream_t s) {
  k_yield<<<blocks, 256, 0, s>>>(a, reinterpret_cast<YieldPartial *>(partials));
  return cudaGetLastError();
}

size_t partial_bytes() { return sizeof(YieldPartial); }

cudaError_t launch_yield_inst(const TravArgs &a, const uint32_t *inst_of_a, double *yields,
                              int blocks, cudaStream_t s) {
  k_yield_inst<<<blocks, 256, 0, s>>>(a, inst_of_a, yields);
  return cudaGetLastError();
}

cudaError_t launch_step_finish(const TLCounters *ctr, unsigned *run_status, TLRunAcc *acc,
                               cudaStream_t s) {
  k_step_finish<<<1, 1, 0, s>>>(ctr, run_status, acc);
  return cudaGetLastError();
}

}  // namespace tl
