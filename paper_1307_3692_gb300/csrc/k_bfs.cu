// Round-synchronous, delayed-start multi-source BFS (Algorithm 1 step 3;
// Section 4 of Miller, Peng, Xu 2013), as one persistent cooperative kernel.
//
// State: key[v] = level and tie-break (KeyFmt, ldd_internal.cuh), initialised to
// v's own start label.  Levels run from that of the largest floor the loop
// handles.  Round r expands the frontier F_r = {v : final level of v is r}:
// every arc (v, w) offers key[v], one level further out, to w with a 64-bit
// atomicMin.  Because key[v] is final once round r - 1 has finished, and an
// offer made in round r carries level r + 1, the minimum over all offers is the
// exact label the paper's super-source shortest path assigns (Section 4),
// including the fraction tie-break.  Wherever two direct keys that differ only
// in their ids meet -- at a vertex, in the minimum that a bottom-up round stops
// at, between that minimum and a start that it passes over, or between a pivot and
// the frontier's other keys -- the meeting is listed (note_tie) and finalize
// compares the exact fractions, so a decomposition that ends without an error bit
// is exact.
//
// Start buckets.  With direct keys the loop itself fills the buckets, some
// levels ahead at a time (build_buckets): it passes over the blocks of vertices
// whose largest floor is too small and drops the vertices that somebody has
// claimed, so the buckets hold about as many vertices as pieces, not all of
// them.
//
// F_{r+1} is built during round r from two disjoint sources:
//   * pushes: the one atomicMin that lowers w's level from > r + 1 to r + 1
//     appends w (its return value identifies it uniquely);
//   * delayed starts (Section 4: the super-source edge of length L is used
//     when the frontier reaches L): vertices of start bucket r + 1 whose key
//     still has level r + 1.  A push in round r can only lower their rank
//     part, so this test is stable while round r runs.
// Appends are warp-aggregated: one 64-bit atomicAdd per warp reserves
// (items << 32 | edges), giving every appended vertex its queue slot and the
// exclusive edge offset of its adjacency list in the next frontier.  The next
// round then splits the frontier's edges into equal spans, one per CTA step,
// whatever the degree skew: a CTA loads the window of queue items that cover
// its span into shared memory and finds each edge's item with a block-wide
// max-scan.
//
// Direction-optimising rounds (Beamer, Asanovic, Patterson 2012): when the
// frontier's arcs outweigh the arcs of the still-unsettled vertices, a round
// runs bottom-up instead: every unsettled vertex w scans its neighbours for
// keys of level r and keeps the smallest key + 2^32.  The scan can stop once it
// holds (r + 1, minrank_r), where minrank_r is the smallest tie-break among level-r
// keys: nothing can beat it.  minrank_r is tracked exactly during round r - 1
// as the minimum over every successful key update and every appended start
// (each final level-r key is one of these, and each of these is >= the final
// key of its vertex).  Only w's own thread writes key[w] in such a round, and a
// vertex being lowered to level r + 1 is never read as a level-r key, so no
// atomics are needed.  On a union of graphs (k_union.cu) the floor is per
// member: the smallest level-r rank of w's own member, since no other member's
// key can reach w; it is computed when a round goes bottom-up, by one pass
// over the frontier list (every level-r vertex is on it) and one more grid
// barrier.  The first bottom-up round of a run examines every
// vertex the BFS owns; each round lists the vertices still above level r + 1,
// and the next bottom-up round examines only those.  Large bottom-up rounds
// stop at a pivot instead of the floor and have a second pass (pull_rest).
//
// Rounds with an empty frontier jump straight to the next non-empty start
// bucket; the loop stops as soon as every vertex with an arc is settled.
// Graphs whose vertices have at most kLdMaxDegree arcs run low-degree rounds
// (a plain vertex list and padded neighbour rows; a thread per frontier vertex,
// or eight lanes while the frontier is thin) and relax several levels between two
// grid barriers (windows of levels, below).  All device-side waits are bounded:
// a barrier that does not complete within the spin limit sets kErrTimeout and
// the kernel returns.
#include <cstddef>

#include "ldd_internal.cuh"

namespace ldd {

namespace {

constexpr u32 kFull = 0xffffffffu;
constexpr int kEdgeBatch = 4;  // arcs per thread in flight
constexpr int kWinBatch = 3;   // window items per thread in flight
// candidates per lane in flight in a bottom-up round: three with one CTA per
// SM (up to 128 registers), two with two CTAs per SM (64 registers: more
// would spill); measured on R-MAT 22 (0.132 ms against 0.140 with two, 0.137
// with four) and on 64 R-MAT 20 copies as a union (3.4 ms against 4.0 with
// three)
constexpr int pull_width(int per_sm) { return per_sm >= 2 ? 2 : 3; }
constexpr int kPullLong = 32;  // longer adjacency lists are scanned by the whole warp
// Bottom-up rounds of at least kDeferMin candidates stop their scans at a
// pivot rank and have a second, edge-balanced pass (pull_rest); smaller rounds
// save its grid barrier.
constexpr u32 kDeferMin = 1u << 16;
// A warp with at least kDeferLanes scans still going after kPullShort
// neighbours puts them all off to that pass, any other warp those with at
// least kDeferLong neighbours left.
constexpr int kPullShort = 8;
constexpr u32 kDeferLanes = 32;
constexpr int kDeferLong = 2048;
// Start buckets are filled kBuildMin vertices at a time at least, at first a
// 2^-kBuildShift share of the handled ones, then eight times as many: most
// loops end long before the buckets that hold most vertices.
constexpr u32 kBuildShift = 10;
constexpr u32 kBuildMin = 1024;
constexpr int kRestBatch = 8;   // the second pass: neighbours per lane in flight
constexpr u32 kPushFlag = 1u << 31;  // on its list: a frontier vertex that pushes
constexpr int kRestSide = 2;    // the side of the frontier arrays that holds the list
// the pivot is the kPivotSkip-th smallest (from 0) of kPivotSamples sampled ranks
constexpr u32 kPivotSamples = 128;
constexpr u32 kPivotSkip = 2;
constexpr int kPullCoop = 4;   // neighbours per lane per step of a warp-wide scan
// Unions of at most this many members keep their per-member floors and pivots
// in shared memory (after Smem: 24 bytes per member, 30 KB, so that two CTAs
// per SM still fit); larger unions use the global tables directly.
constexpr u32 kSmemMembers = 1280;
// Low-degree expansions give an item a thread, or eight lanes when the items then
// still take at most this many passes of the threads (the CTA's for a local
// queue, the grid's for the frontier).  A thread per item issues up to eight
// atomics and pushes one after the other with few warps active, eight lanes one:
// a level of a window with 11 items per CTA (1000 x 1000 grid) went from 3.0 to
// 1.9 us.  With many items the divergent atomics' number is what counts, and a
// thread per item keeps more of them in flight (256^3 grid: 2.76 ms with a thread
// always, 2.67 with up to 2 passes, 2.79 with up to 4; 150 k geometric graph .60,
// .46, .46 ms; two, four lanes per item in between gained nothing).
constexpr u32 kLdGroupPasses = 2;

__device__ __forceinline__ void note_tie(const BfsArgs& a, u32 w, u64 x, u64 y) {
  note_tie(a.ctl, a.f, w, x, y);
}

// atomicMin(p, v) where `on`, else `other`, without a branch: the offers of a
// batch are all on their way before the first one's answer is looked at.
// Written as `if (on) { old = atomicMin(..); if (old > v) .. }` per offer, the
// compiler kept each offer's use of its answer beside it, so a batch waited for
// one round trip per offer, 40 % of a level's time in the windows of levels.
// Round loops: 1000^2 grid, beta 0.01, 1.97 -> 1.57 ms; 256^3 grid 3.49 -> 2.79
// ms; random geometric graph of 150,001 vertices 0.73 -> 0.46 ms.
__device__ __forceinline__ u64 offer_min(u64* p, u64 v, bool on, u64 other) {
  u64 old;
  asm volatile(
      "{\n\t.reg .pred on;\n\t"
      "setp.ne.s32 on, %4, 0;\n\t"
      "mov.b64 %0, %3;\n\t"
      "@on atom.relaxed.gpu.global.min.u64 %0, [%1], %2;\n\t}"
      : "=&l"(old)
      : "l"(p), "l"(v), "l"(other), "r"((int)on)
      : "memory");
  return old;
}

struct Smem {
  int owner[kBfsMaxSpan];
  int rowd[kBfsMaxSpan + 1];
  u64 cand[kBfsMaxSpan + 1];
  int wtot[kBfsThreads / 32];
  u64 minlow[kBfsThreads / 32];  // each warp's smallest successful next-level tie-break
  u32 stop;     // thread 0 saw an error bit: the whole CTA leaves the loop
  // the next round's frontier counter, bottom-up floor and unsettled-list
  // length, read by thread 0 as the barrier releases
  u64 next_c;
  u64 next_rest;         // a large bottom-up round's list for its second pass
  u64 next_minlow;
  u32 next_ucnt;
  int next_lo, next_hi;  // the next round's start bucket (lvl + 1) bounds
  u32 next_ovf;          // the next round's overflow-list length (windows)
  u32 lcnt[3];           // windows: local-queue lengths, rotating (read, fill, clear)
  u32 nstart;            // a scan's result, shared by the CTA
  u64 pivot;             // the round's pivot
  int built;             // build_buckets: the last level filled
};
// Windows of levels keep two local queues whose entries carry a vertex and the
// key it was pushed with (12 bytes, as two arrays).
// The first queue sits in the memory the edge-balanced rounds use for their
// span windows.  With two CTAs per SM the second shares it; with one, which
// has the room, it gets as much again after Smem.
constexpr size_t kSpanBytes = sizeof(int) * kBfsMaxSpan * 2 + sizeof(u64) * kBfsMaxSpan;
static_assert(offsetof(Smem, owner) == 0 && offsetof(Smem, rowd) < offsetof(Smem, cand) &&
                  offsetof(Smem, cand) + sizeof(u64) * (kBfsMaxSpan + 1) >= kSpanBytes,
              "the span-window arrays lead Smem and cover its first kSpanBytes bytes");
constexpr size_t kLqEntry = sizeof(u64) + sizeof(u32);
constexpr int lq_cap(int per_sm) {
  return (int)((per_sm >= 2 ? kSpanBytes / 2 : kSpanBytes) / kLqEntry) / 32 * 32;
}
constexpr size_t lq_extra(int per_sm) { return per_sm >= 2 ? 0 : kSpanBytes; }
// the entries a local queue takes: the tuning's limit, if any, else all that fit
template <int kCap>
__device__ __forceinline__ u32 lq_limit(const BfsArgs& a) {
  return a.window_queue ? min(a.window_queue, (u32)kCap) : (u32)kCap;
}
struct LocalQueue {
  u64* key;
  u32* v;
};
template <int kCap>
__device__ __forceinline__ LocalQueue lq_buf(Smem& s, int b) {
  unsigned char* span = reinterpret_cast<unsigned char*>(&s.owner[0]);
  unsigned char* base;
  if ((size_t)kCap * kLqEntry * 2 <= kSpanBytes) base = span + (size_t)b * kCap * kLqEntry;
  else base = b == 0 ? span : reinterpret_cast<unsigned char*>(&s) + sizeof(Smem);
  LocalQueue q;
  q.key = reinterpret_cast<u64*>(base);
  q.v = reinterpret_cast<u32*>(q.key + kCap);
  return q;
}

// 64-bit minimum and maximum over the warp: of the high words, then of the low
// words of the lanes that have it.
__device__ __forceinline__ u64 warp_min64(u64 x) {
  const u32 hi = (u32)(x >> 32), h = __reduce_min_sync(kFull, hi);
  return (u64)h << 32 | __reduce_min_sync(kFull, hi == h ? (u32)x : 0xffffffffu);
}
__device__ __forceinline__ u64 warp_max64(u64 x) { return ~warp_min64(~x); }

// Grid-wide barrier on a monotonic arrival counter: the k-th barrier of a
// launch completes when the counter reaches k * nblocks (+ phantom), so
// arrival is one fire-and-forget add and nobody has to reset anything.
// Before arriving, thread 0 publishes this CTA's smallest next-level tie-break to
// ctl->minlow[post] (and resets the CTA value).  The poll is an acquire
// load, so once it sees every arrival the round's writes of all CTAs are
// visible.  The wait is bounded: it ends after a.spin_limit polls, with
// kErrTimeout, or once any CTA has recorded an error.  Thread 0 then reads,
// in one round trip, the error word and the next round's state (slot `post`
// of the frontier counter, bottom-up floor and unsettled-list length, and the
// bounds of start bucket blevel, of levels from lv0 on, unless it is negative)
// into shared memory, so that every thread of the CTA sees the same values and
// takes the same branch after the barrier (a thread that left the loop alone
// would leave the others at a CTA barrier).  a.bar_phantom > 0 waits for CTAs that
// do not exist: the barrier can then only end by running out of polls, which
// is how the timeout path is tested.
constexpr u32 kNoPost = 0xffffffffu;  // grid_barrier: a barrier inside a round

template <bool kTrack>
__device__ __forceinline__ void grid_barrier(const BfsArgs& a, u32& gen, u32 post, int lv0,
                                             int blevel, Smem& s) {
  Control* ctl = a.ctl;
  __syncthreads();
  u64 mine = ~0ull;  // this CTA's smallest next-level tie-break
  if (kTrack && post != kNoPost && threadIdx.x < 32) {
    const u64 x = threadIdx.x < kBfsThreads / 32 ? s.minlow[threadIdx.x] : ~0ull;
    mine = warp_min64(x);
    if (x != ~0ull) note_tie(a, 0, x, mine);
  }
  if (threadIdx.x == 0) {
    if (mine != ~0ull)
      asm volatile("red.relaxed.gpu.global.min.u64 [%0], %1;" ::"l"(&ctl->minlow[post]), "l"(mine)
                   : "memory");
    ++gen;
    const u64 target = (u64)gen * gridDim.x + a.bar_phantom;
    // release, after the CTA barrier above: covers the whole CTA's writes
    asm volatile("red.release.gpu.global.add.u64 [%0], %1;" ::"l"(&ctl->bar), "l"(1ull) : "memory");
    u32 spins = 0;
    for (;;) {
      u64 seen;
      asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(seen) : "l"(&ctl->bar) : "memory");
      if (seen >= target) break;
      if (ld_acquire_u32(&ctl->err) != 0u) break;  // another CTA has left the loop
      if (++spins > a.spin_limit) {
        atomicOr(&ctl->err, kErrTimeout);
        __threadfence();
        break;
      }
      if (spins > 64) __nanosleep(20);
    }
    const u32 err = ld_cg_u32(&ctl->err);
    if (post != kNoPost) {
      s.next_c = ld_cg_u64(&ctl->qctr[post]);
      s.next_minlow = ld_cg_u64(&ctl->minlow[post]);
      if (mine != ~0ull) note_tie(a, 0, mine, s.next_minlow);
      s.next_ucnt = ld_cg_u32(&ctl->ucnt[post]);
      s.next_ovf = ld_cg_u32(&ctl->ovf[post]);
      s.next_rest = ld_cg_u64(&ctl->rest[post]);
      s.next_lo = s.next_hi = 0;
      if (blevel >= 0) {  // bounds of start bucket blevel, for the round after the barrier
        s.next_lo = __ldg(a.bptr + (blevel - lv0));
        s.next_hi = (int)ld_cg_u32(a.rcur + (blevel - lv0));
      }
    }
    s.stop = err != 0u ? 1u : 0u;
  }
  __syncthreads();
}

// Exclusive prefix over the warp of small counts x < 2^kBits (and, in *tot,
// their sum), by one ballot per bit instead of a chain of shuffles.
template <int kBits>
__device__ __forceinline__ u32 warp_excl_small(u32 x, u32* tot) {
  const u32 lt = lanemask_lt();
  u32 pre = 0, sum = 0;
#pragma unroll
  for (int b = 0; b < kBits; ++b) {
    const u32 m = __ballot_sync(kFull, (x >> b) & 1u);
    pre += (u32)__popc(m & lt) << b;
    sum += (u32)__popc(m) << b;
  }
  *tot = sum;
  return pre;
}
template <int K>
constexpr int bits_for() { return K < 2 ? 1 : K < 4 ? 2 : K < 8 ? 3 : K < 16 ? 4 : K < 32 ? 5 : 6; }


// First item of this warp in a grid-stride loop over groups of 32 x k items,
// numbered so that consecutive groups go to different CTAs (warp w of CTA b
// takes group w * gridDim.x + b): a round with fewer items than threads still
// spreads over every SM instead of filling the leading CTAs.  The stride is
// gridDim.x * blockDim.x * k.  rev: CTAs in reverse order.
__device__ __forceinline__ u32 warp_first_item(u32 k, bool rev = false) {
  const u32 b = rev ? gridDim.x - 1 - blockIdx.x : blockIdx.x;
  return ((threadIdx.x >> 5) * gridDim.x + b) * 32u * k;
}

// Records a successful next-level key k for the bottom-up floor of the next
// round: the thread's smallest tie-break, folded into the CTA's and the grid's
// at the barrier.  Unions and low-degree rounds track nothing here: they go
// bottom-up rarely, and their floors are then computed from the frontier list
// (member_floors, list_floor).  In a union the floor is per member (another
// member's smaller tie-break can never reach v), and keeping up to kmem minima
// per CTA in every round cost more than the rare bottom-up rounds of a batch
// gain from it; in the thin rounds of a low-degree graph the bookkeeping cost
// 2 % of the loop.
template <bool kTrack>
__device__ __forceinline__ void note_low(const BfsArgs& a, bool valid, u64 k, u64& mylow) {
  if (!kTrack || !valid) return;
  const u64 low = key_low(a.f, k);
  note_tie(a, 0, low, mylow);
  mylow = min(mylow, low);
}

// Unions: the per-member floors of level-L keys (the smallest tie-break among
// each member's keys of the frontier's level) from the frontier list qv of Q
// vertices, into slot `slot` of a.mlow (all ~0 on entry), and with kPivot
// every member's frontier vertex of the largest degree into a.mpivot (as
// (degree << 32) | vertex, all zero on entry; see pull_rest).  A warp whose
// vertices share one member makes one update; small unions gather both per CTA
// in shared memory (s_acc, s_piv) and flush them.  The caller then waits at a
// grid barrier before they are read.
template <bool kPivot>
__device__ __forceinline__ void member_floors(const BfsArgs& a, const u32* qv, u32 Q, u32 slot,
                                              u64* s_acc, u64* s_piv) {
  const u32 lane = threadIdx.x & 31;
  const u32 stride = gridDim.x * blockDim.x;
  for (u32 base = warp_first_item(1); base < Q; base += stride) {
    const u32 i = base + lane;
    const bool valid = i < Q;
    u32 v = 0, m = 0xffffffffu;
    u64 r = ~0ull, pv = 0;
    if (valid) {
      v = ld_cg_u32(qv + i);
      m = __ldg(a.wmem + (v >> 5));
      r = key_low(a.f, ld_cg_u64(a.key + v));
      if (kPivot) pv = (u64)(u32)(__ldg(a.row_ptr + v + 1) - __ldg(a.row_ptr + v)) << 32 | v;
    }
    const u32 act = __ballot_sync(kFull, valid);
    const u32 m0 = __shfl_sync(kFull, m, __ffs(act) - 1);
    const bool one = __all_sync(kFull, !valid || m == m0);
    u64 rr = r;
    if (one) {
      rr = warp_min64(r);
      if (valid) note_tie(a, v, r, rr);
    }
    const u64 pp = kPivot && one ? warp_max64(pv) : pv;
    if ((one && lane == (u32)(__ffs(act) - 1)) || (!one && valid)) {
      const u32 mm = one ? m0 : m;
      u64* p = s_acc ? s_acc + mm : a.mlow + (size_t)slot * a.kmem + mm;
      const u64 seen = s_acc ? *(volatile u64*)p : ld_cg_u64(p);
      if (rr < seen) note_tie(a, v, rr, atomicMin(p, rr));
      else note_tie(a, v, rr, seen);
      if (kPivot) {
        u64* q = s_acc ? s_piv + mm : a.mpivot + (size_t)slot * a.kmem + mm;
        if (pp > (s_acc ? *(volatile u64*)q : ld_cg_u64(q))) atomicMax(q, pp);
      }
    }
  }
}

// Union: the CTA's per-member minima into slot `slot` of a.mlow (and the
// pivots into a.mpivot), and the shared tables reset.  Called by the whole CTA
// between __syncthreads.
template <bool kPivot>
__device__ __forceinline__ void flush_members(const BfsArgs& a, u32 slot, u64* s_acc,
                                              u64* s_piv) {
  for (u32 m = threadIdx.x; m < a.kmem; m += blockDim.x) {
    const u64 r = s_acc[m];
    if (r != ~0ull) {
      u64* p = a.mlow + (size_t)slot * a.kmem + m;
      const u64 seen = ld_cg_u64(p);
      const u64 met = r < seen ? atomicMin(p, r) : seen;
      if (met != ~0ull) note_tie(a, __ldg(a.voff + m), met, r);
      s_acc[m] = ~0ull;
      if (kPivot) {
        u64* q = a.mpivot + (size_t)slot * a.kmem + m;
        if (s_piv[m] > ld_cg_u64(q)) atomicMax(q, s_piv[m]);
        s_piv[m] = 0;
      }
    }
  }
}

// Union: what a bottom-up scan of w may stop at, the smallest tie-break of its
// member's level-L keys or (pivot) that of the member's pivot; ~0 when the
// member has no level-L key.  s_floor: the CTA's copy, already the one of the two.
__device__ __forceinline__ u64 member_floor(const BfsArgs& a, u32 w, u32 slot, const u64* s_floor,
                                            bool pivot) {
  const u32 m = __ldg(a.wmem + (w >> 5));
  if (s_floor) return s_floor[m];
  if (!pivot) return ld_cg_u64(a.mlow + (size_t)slot * a.kmem + m);
  const u64 pv = ld_cg_u64(a.mpivot + (size_t)slot * a.kmem + m);
  return pv ? key_low(a.f, ld_cg_u64(a.key + (u32)pv)) : ~0ull;
}

// Appends to the frontier every vertex v[i] whose bit i is set in `mask`, for
// up to K candidates per lane, with one atomicAdd per warp: the warp scans
// (count << 32 | degree sum) over its lanes, reserves that many queue slots
// and edge offsets, and every lane writes its vertices in slot order.
// qi: frontier counter index (rotates over 3), qb: queue buffer (ping-pong).
// Low-degree mode: the frontier is the plain vertex list qv (items in the
// counter's high word, its low word unused), so an append is one reservation
// per warp and one store per vertex, with no adjacency range to load.
template <int K>
__device__ __forceinline__ void warp_append_ld(u32 mask, const u32 (&v)[K], const BfsArgs& a,
                                               int qi, int qb) {
  const u32 lane = threadIdx.x & 31;
  u32 tot;
  const u32 excl = warp_excl_small<bits_for<K>()>(__popc(mask), &tot);
  if (tot == 0) return;
  u32 base = 0;
  if (lane == 0) base = (u32)(atomicAdd(&a.ctl->qctr[qi], (u64)tot << 32) >> 32);
  u32 slot = __shfl_sync(kFull, base, 0) + excl;
#pragma unroll
  for (int i = 0; i < K; ++i)
    if (mask >> i & 1u) a.qv[qb][slot++] = v[i];
}

template <int K, bool LD>
__device__ __forceinline__ void warp_append(u32 mask, const u32 (&v)[K], const BfsArgs& a, int qi,
                                            int qb) {
  if (LD) {
    warp_append_ld<K>(mask, v, a, qi, qb);
    return;
  }
  const u32 lane = threadIdx.x & 31;
  int rs[K], dg[K];
#pragma unroll
  for (int i = 0; i < K; ++i) {
    rs[i] = 0;
    dg[i] = 0;
    if (mask >> i & 1u) {
      rs[i] = __ldg(a.row_ptr + v[i]);
      dg[i] = __ldg(a.row_ptr + v[i] + 1) - rs[i];
    }
  }
  u32 cnt = 0, dsum = 0;
#pragma unroll
  for (int i = 0; i < K; ++i)
    if (dg[i] <= 0) {
      mask &= ~(1u << i);  // a vertex without arcs has nothing to expand
    } else {
      ++cnt;
      dsum += (u32)dg[i];
    }
  if (!__any_sync(kFull, mask != 0u)) return;
  const u64 mine = ((u64)cnt << 32) | dsum;
  u64 incl = mine;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const u64 y = __shfl_up_sync(kFull, incl, o);
    if (lane >= (u32)o) incl += y;
  }
  const u64 tot = __shfl_sync(kFull, incl, 31);
  u64 base = 0;
  if (lane == 0) base = atomicAdd(&a.ctl->qctr[qi], tot);
  base = __shfl_sync(kFull, base, 0) + (incl - mine);
  u32 slot = (u32)(base >> 32), off = (u32)base;
#pragma unroll
  for (int i = 0; i < K; ++i)
    if (mask >> i & 1u) {
      a.qv[qb][slot] = v[i];
      a.qrow[qb][slot] = rs[i];
      a.qoff[qb][slot] = off;
      const u32 end = off + (u32)dg[i];
      for (u32 c = (off + kBfsBase - 1) / kBfsBase; c * kBfsBase < end; ++c) a.cf[qb][c] = slot;
      ++slot;
      off = end;
    }
}

// Unclaimed vertices of start bucket rr (entries lo .. hi of rv) join the
// frontier of level rr.
template <bool U>
__device__ __forceinline__ void append_bucket(const BfsArgs& a, int rr, int lo, int hi, int qi,
                                              int qb, u64& mylow) {
  const u32 cnt = (u32)(hi - lo);
  const u32 lane = threadIdx.x & 31;
  const u32 stride = gridDim.x * blockDim.x;
  // trailing CTAs first: in a small round the leading CTAs are expanding
  for (u32 base = warp_first_item(1, true); base < cnt; base += stride) {
    const u32 i = base + lane;
    u32 u[1] = {0};
    bool want = false;
    u64 k = 0;
    if (i < cnt) {
      u[0] = ld_cg_u32(a.rv + lo + i);
      k = ld_cg_u64(a.key + u[0]);
      want = key_level(a.f, k) == (u32)rr;
    }
    note_low<!U>(a, want, k, mylow);
    warp_append<1, false>(want ? 1u : 0u, u, a, qi, qb);
  }
}

// Direct keys: fills the start buckets of levels from .. to, to the last level
// (at least from) that keeps their vertices, claimed ones included, within
// `most`; returns it, the same in every CTA.  The buckets' room follows from
// the counts of all floors (bptr); an entry is a vertex whose key still names
// itself.  The caller waits at a grid barrier before they are read.  first: from
// is the loop's first level, lv0; its vertices start the frontier (slot 0) at
// once, without a pass over their bucket and its barrier.
template <bool U, bool LD>
__device__ __forceinline__ int build_buckets(const BfsArgs& a, Smem& s, int lv0, int from, int A,
                                             u32 most, bool first, u64& mylow) {
  // the last of blockDim.x evenly spaced levels within `most`
  const int step = (A - from) / (int)blockDim.x + 1;
  __syncthreads();
  if (threadIdx.x == 0) s.built = from;
  __syncthreads();
  {
    const int r = min(from + (int)threadIdx.x * step, A);
    const int room = __ldg(a.bptr + (r + 1 - lv0)) - __ldg(a.bptr + (from - lv0));
    if ((u32)room <= most) atomicMax(&s.built, r);
  }
  __syncthreads();
  const int to = s.built;
  const u32 lane = threadIdx.x & 31;
  const u32 least = a.f.cap - (u32)to + 1;  // a block's entry in bmax: its largest floor plus one
  const u32 nblk = (a.n + kMaxBlock - 1) / kMaxBlock;
  // block after block to different warps, 32 of a warp's own looked up at once
  const u32 W = gridDim.x * (blockDim.x >> 5);
  for (u32 b0 = (threadIdx.x >> 5) * gridDim.x + blockIdx.x; b0 < nblk; b0 += 32 * W) {
    const u32 b = b0 + lane * W;
    u32 have = __ballot_sync(kFull, b < nblk && __ldg(a.bmax + b) >= least);
    while (have) {
      const u32 v0 = (b0 + (u32)(__ffs(have) - 1) * W) * kMaxBlock + lane;
      have &= have - 1;
      u64 k[kMaxBlock / 32];
#pragma unroll
      for (int q = 0; q < (int)kMaxBlock / 32; ++q)
        k[q] = v0 + (u32)q * 32 < a.n ? ld_cg_u64(a.key + v0 + (u32)q * 32) : ~0ull;
#pragma unroll
      for (int q = 0; q < (int)kMaxBlock / 32; ++q) {
        const u32 v = v0 + (u32)q * 32;
        const int lev = (int)key_level(a.f, k[q]);
        bool take = v < a.n && lev >= from && lev <= to;
        if (take && ((__ldg(a.excl + (v >> 5)) >> lane) & 1u)) take = false;
        if (take)  // unclaimed: the key names its own vertex
          take = key_id(a.f, k[q]) == (U ? v - __ldg(a.voff + __ldg(a.wmem + (v >> 5))) : v);
        if (!__any_sync(kFull, take)) continue;
        if (first) {
          const u32 vv[1] = {v};
          const bool start = take && lev == from;
          note_low<!U && !LD>(a, start, k[q], mylow);
          warp_append<1, LD>(start ? 1u : 0u, vv, a, 0, 0);
          take = take && !start;
        }
        // one reservation per level and warp
        const u32 peers = __match_any_sync(kFull, take ? lev : -1);
        const int leader = __ffs(peers) - 1;
        u32 at = 0;
        if (take && (int)lane == leader) at = atomicAdd(a.rcur + (lev - lv0), (u32)__popc(peers));
        at = __shfl_sync(kFull, at, leader);
        if (take) a.rv[at + (u32)__popc(peers & lanemask_lt())] = v;
      }
    }
  }
  return to;
}

template <bool U>
__device__ __forceinline__ void expand(const BfsArgs& a, Smem& s, int cur, u32 Q, u32 E, int lvl,
                                       int qi, int qb, u64& mylow) {
  const u32 nb = (E + kBfsBase - 1) / kBfsBase;
  u32 k = (nb + gridDim.x - 1) / gridDim.x;
  k = max(1u, min(k, a.span / kBfsBase));
  const u32 nsuper = (nb + k - 1) / k;
  const u32* cf = a.cf[cur];
  const u32* qv = a.qv[cur];
  const int* qrow = a.qrow[cur];
  const u32* qoff = a.qoff[cur];
  const u32 lvl_next = (u32)lvl + 1;
  const bool probe = E >= a.probe_min_arcs;  // smaller frontiers skip the key probe
  for (u32 sc = blockIdx.x; sc < nsuper; sc += gridDim.x) {
    const u32 b0 = sc * k, b1 = min(b0 + k, nb);
    const u32 e0 = b0 * kBfsBase, e1 = min(b1 * kBfsBase, E);
    const u32 i0 = ld_cg_u32(cf + b0);
    const u32 ilast = (b1 < nb) ? ld_cg_u32(cf + b1) : Q - 1;
    const int nwin = (int)(ilast - i0) + 1;
    const int len = (int)(e1 - e0);
    if (nwin > kBfsMaxSpan + 1 || nwin < 1 || ilast >= Q) {  // window invariant broken
      if (threadIdx.x == 0) atomicOr(&a.ctl->err, kErrInternal);
      return;
    }
    for (int j = threadIdx.x; j < len; j += kBfsThreads) s.owner[j] = 0;
    __syncthreads();
    // window: queue items covering [e0, e1); loads batched for memory-level parallelism
    for (int j0 = 0; j0 < nwin; j0 += kBfsThreads * kWinBatch) {
      u32 off[kWinBatch], v[kWinBatch];
      int row[kWinBatch];
#pragma unroll
      for (int i = 0; i < kWinBatch; ++i) {
        const int j = j0 + i * kBfsThreads + (int)threadIdx.x;
        off[i] = e1;
        if (j < nwin) {
          off[i] = ld_cg_u32(qoff + i0 + j);
          v[i] = ld_cg_u32(qv + i0 + j);
          row[i] = ld_cg_i32(qrow + i0 + j);
        }
      }
      u64 kv[kWinBatch];
#pragma unroll
      for (int i = 0; i < kWinBatch; ++i)
        if (off[i] < e1) kv[i] = ld_cg_u64(a.key + v[i]);
#pragma unroll
      for (int i = 0; i < kWinBatch; ++i)
        if (off[i] < e1) {
          const int j = j0 + i * kBfsThreads + (int)threadIdx.x;
          s.rowd[j] = row[i] - (int)off[i];
          s.cand[j] = key_up(a.f, kv[i]);
          atomicMax(&s.owner[off[i] > e0 ? off[i] - e0 : 0u], j);
        }
    }
    __syncthreads();
    block_max_scan<kBfsThreads, kBfsMaxSpan>(s.owner, len, s.wtot);
    __syncthreads();
    // edges: all loads of a batch first, then all probes, then the atomics
    for (int base = 0; base < len; base += kBfsThreads * kEdgeBatch) {
      u32 w[kEdgeBatch];
      u64 cand[kEdgeBatch];
#pragma unroll
      for (int i = 0; i < kEdgeBatch; ++i) {
        const int kk = base + i * kBfsThreads + (int)threadIdx.x;
        w[i] = 0xffffffffu;
        cand[i] = 0;
        if (kk < len) {
          const int j = s.owner[kk];
          cand[i] = s.cand[j];
          w[i] = (u32)__ldg(a.col + (s.rowd[j] + (int)(e0 + kk)));
        }
      }
      u64 cur[kEdgeBatch];  // probe before the atomic only when there are many arcs
#pragma unroll
      for (int i = 0; i < kEdgeBatch; ++i)
        cur[i] = (w[i] < a.n) ? (probe ? ld_cg_u64(a.key + w[i]) : ~0ull) : 0ull;
      u32 mask = 0, won = 0, off = 0;
#pragma unroll
      for (int i = 0; i < kEdgeBatch; ++i) {
        const bool on = cand[i] < cur[i];
        if (on) off |= 1u << i;
        cur[i] = offer_min(a.key + (on ? w[i] : 0u), cand[i], on, cur[i]);
      }
#pragma unroll
      for (int i = 0; i < kEdgeBatch; ++i)
        if (off >> i & 1u) {
          if (cur[i] > cand[i]) won |= 1u << i;
          if (key_level(a.f, cur[i]) > lvl_next) mask |= 1u << i;
        }
      bool tie = false;  // one branch for the batch: meetings are rare
#pragma unroll
      for (int i = 0; i < kEdgeBatch; ++i) tie |= w[i] < a.n && key_near(cand[i], cur[i]);
      if (tie) {
#pragma unroll
        for (int i = 0; i < kEdgeBatch; ++i)
          if (w[i] < a.n) note_tie(a, w[i], cand[i], cur[i]);
      }
#pragma unroll
      for (int i = 0; i < kEdgeBatch; ++i) note_low<!U>(a, (won >> i) & 1u, cand[i], mylow);
      warp_append<kEdgeBatch, false>(mask, w, a, qi, qb);
    }
    __syncthreads();
  }
}

// Low-degree rounds read neighbours from the padded rows (BfsArgs::ell), a chunk
// of eight at a time by a group of 8 / P lanes, P words (one load, two for P = 8)
// per lane: words P * q .. of v's chunk ch, q the lane's place in its group; ~0
// past the row's end, and all ~0 unless `on`.  Returns whether the row may go on
// (the chunk's last word is a neighbour), the same for the group.  Every lane of
// the warp calls this.
template <int P>
__device__ __forceinline__ bool ell_load(const BfsArgs& a, u32 v, u32 ch, bool on, u32 (&w)[P]) {
  constexpr u32 G = 8 / P;
  const u32 lane = threadIdx.x & 31;
  if (on) {
    const u32* p = a.ell + ((size_t)v * a.ell_s + 8 * ch + P * (lane & (G - 1)));
    if constexpr (P == 1) {
      w[0] = __ldg(p);
    } else if constexpr (P == 2) {
      const uint2 x = __ldg(reinterpret_cast<const uint2*>(p));
      w[0] = x.x;
      w[1] = x.y;
    } else {
#pragma unroll
      for (int h = 0; h < P; h += 4) {
        const uint4 x = __ldg(reinterpret_cast<const uint4*>(p + h));
        w[h] = x.x;
        w[h + 1] = x.y;
        w[h + 2] = x.z;
        w[h + 3] = x.w;
      }
    }
  } else {
#pragma unroll
    for (int h = 0; h < P; ++h) w[h] = ~0u;
  }
  if (8 * (ch + 1) >= a.ell_s) return false;  // the same for the whole grid
  const u32 b = __ballot_sync(kFull, on && w[P - 1] != ~0u);
  return b >> (lane | (G - 1)) & 1u;
}

// Low-degree round (every vertex of the graph has at most kLdMaxDegree
// arcs): one pass over Q frontier vertices (the list qv_cur) and the cnt
// entries of start bucket rb (from lo in rv), 8 / P lanes per item.
//   * A frontier vertex v offers key[v], one level further out, to each of its
//     neighbours (64-bit atomicMin, after a probe of the key when `probe`), P
//     arcs per lane and step, and appends the neighbours whose level it lowered to lvl + 1.
//   * A start-bucket entry u joins the next frontier if its key still has its
//     start level rb (Section 4's delayed start; stable during the round, see
//     the file comment).
// v's key and first neighbours, and the bucket entries' keys, load in one round
// trip, and the bucket test runs beside the expansion instead of after it: a
// thin round is a short chain of dependent loads.  `pushed` adds the arcs
// offered.
template <bool U, int P>
__device__ __forceinline__ void expand_ld(const BfsArgs& a, const u32* qv_cur, u32 Q, u32 lvl_next,
                                          int lo, u32 cnt, u32 rb, bool probe, int qi, int qb,
                                          u64& pushed) {
  constexpr u32 G = 8 / P;  // lanes per item
  const u32 lane = threadIdx.x & 31;
  const u32 total = Q + cnt;
  const u32 stride = gridDim.x * blockDim.x / G;
  for (u32 base = warp_first_item(1) / G; base < total; base += stride) {
    const u32 i = base + lane / G;
    const bool front = i < Q, buck = !front && i < total && (lane & (G - 1)) == 0;
    u32 v[1] = {0};
    if (front) v[0] = ld_cg_u32(qv_cur + i);
    else if (buck) v[0] = ld_cg_u32(a.rv + lo + (int)(i - Q));
    u64 kv = 0;
    if (front || buck) kv = ld_cg_u64(a.key + v[0]);
    u32 w[P];
    bool more = ell_load<P>(a, v[0], 0, front, w);
    warp_append<1, true>(buck && key_level(a.f, kv) == rb ? 1u : 0u, v, a, qi, qb);
    const u64 cand = key_up(a.f, kv);
    if (!__any_sync(kFull, front)) continue;
    for (u32 ch = 0;;) {
      u64 cur[P];
#pragma unroll
      for (int x = 0; x < P; ++x) {
        pushed += w[x] < a.n ? 1u : 0u;
        cur[x] = (w[x] < a.n) ? (probe ? ld_cg_u64(a.key + w[x]) : ~0ull) : 0ull;
      }
      u32 mask = 0;
#pragma unroll
      for (int x = 0; x < P; ++x) {
        const bool on = cand < cur[x];
        if (on) mask |= 1u << x;
        cur[x] = offer_min(a.key + (on ? w[x] : 0u), cand, on, cur[x]);
      }
#pragma unroll
      for (int x = 0; x < P; ++x)
        if (key_level(a.f, cur[x]) <= lvl_next) mask &= ~(1u << x);
      bool tie = false;  // one branch for the batch: meetings are rare
#pragma unroll
      for (int x = 0; x < P; ++x) tie |= w[x] < a.n && key_near(cand, cur[x]);
      if (tie) {
#pragma unroll
        for (int x = 0; x < P; ++x)
          if (w[x] < a.n) note_tie(a, w[x], cand, cur[x]);
      }
      warp_append<P, true>(mask, w, a, qi, qb);
      if (!__any_sync(kFull, more)) break;
      more = ell_load<P>(a, v[0], ++ch, more, w);
    }
  }
}

// ---------------------------------------------------------------- windows of levels
// Low-degree rounds may run a window of levels [L, H) between two grid
// barriers instead of one level.  Each CTA expands its share of the level-L
// frontier (and of the overflow list of the last window), then keeps going on
// its own: every vertex whose key it lowers to a level below H goes into the
// CTA's local queue (shared memory) and is expanded by the same CTA at the
// next local level, with only a CTA barrier in between; vertices lowered to
// level H go to the global queue for the next round.  Start bucket lv + 1 is
// checked at local level lv, as in a one-level round.
//
// Exactness: keys only decrease, and the fixed point of the min over all
// offers does not depend on the order in which they are made (Section 4's
// shortest path, label-correcting).  Every successful atomicMin makes its
// vertex be expanded again: it is pushed with the level it got, to a local
// queue, to the global queue (the first time it reaches level H), or -- when
// a local queue is full -- to the overflow list that the next round expands.
// A global-queue or overflow entry whose vertex has meanwhile been lowered to
// a smaller level is skipped, since its lowerer pushed it again; a local entry
// carries the key it was pushed with, and if that key is outdated, its offers
// are dominated by those of the better one.  Past level H - 1 a CTA works its
// local queue down until it is empty.  A CTA may run ahead of another
// inside a window, so a vertex can first get a worse key and be expanded
// twice (the statistics count every expansion); the result is the same.  A
// start test inside a window may let a vertex start that a slower CTA lowers
// later: it is expanded again with the better key.  At the end of a window
// every key below level H is final unless an overflow entry is pending, and
// the loop then runs another window before any bottom-up round.
//
// Once a window has run, the number of settled vertices is no longer counted
// exactly; an empty frontier then scans the start buckets from the current
// level for the next one that still holds an unclaimed vertex (one pass and
// one grid barrier) instead of stopping when every vertex is settled.

// Pushes vertex w[i] with the lane's key k for every bit i of mask: to the CTA's
// local queue nb while it has room, the rest (as vertex and level) to the
// overflow list of the next round.
template <int K, int kCap>
__device__ __forceinline__ void window_push(u32 mask, const u32 (&w)[K], u64 k, const BfsArgs& a,
                                            Smem& s, int nb, int nc, int qi, int qb) {
  const u32 lane = threadIdx.x & 31;
  u32 tot;
  const u32 excl = warp_excl_small<bits_for<K>()>(__popc(mask), &tot);
  if (tot == 0) return;
  u32 base = 0;
  if (lane == 0) base = atomicAdd(&s.lcnt[nc], tot);
  base = __shfl_sync(kFull, base, 0) + excl;
  const LocalQueue lq = lq_buf<kCap>(s, nb);
  const u32 cap = lq_limit<kCap>(a);
  u32 spill = 0;
#pragma unroll
  for (int i = 0; i < K; ++i)
    if (mask >> i & 1u) {
      if (base < cap) {
        lq.key[base] = k;
        lq.v[base] = w[i];
      } else {
        spill |= 1u << i;
      }
      ++base;
    }
  // a full local queue: the rest waits for the next round on the overflow list
  if (!__any_sync(kFull, spill != 0u)) return;
  u32 stot;
  const u32 sexcl = warp_excl_small<bits_for<K>()>(__popc(spill), &stot);
  u32 sbase = 0;
  if (lane == 0) sbase = atomicAdd(&a.ctl->ovf[qi], stot);
  sbase = __shfl_sync(kFull, sbase, 0) + sexcl;
#pragma unroll
  for (int i = 0; i < K; ++i)
    if (spill >> i & 1u) {
      if (sbase < a.n) {
        reinterpret_cast<u32*>(a.qrow[qb])[sbase] = w[i];
        a.qoff[qb][sbase] = key_level(a.f, k);
      } else {
        atomicOr(&a.ctl->err, kErrInternal);  // more pushes than vertices: cannot happen
      }
      ++sbase;
    }
}

// Expands one item per lane -- valid: vertex v with key kv -- in a window whose
// end is H: kv, one level further out, is offered to the neighbours, whose first
// chunk is w, with more to load if `more`.  Winners
// below H go to the local queue nb with the key they got, winners at H that
// reach it for the first time to the global queue qb.  A kv that is no longer
// the vertex's key (it was lowered again, and its lowerer pushed it again) only
// makes offers that the better key dominates.  Every lane of the warp calls
// this.
template <bool U, int kCap, int P>
__device__ __forceinline__ void window_expand(const BfsArgs& a, Smem& s, bool valid, u64 kv, u32 v,
                                              u32 (&w)[P], bool more, u32 H, int nb, int nc,
                                              int qi, int qb, u64& pushed, u64& expanded) {
  if (valid && (threadIdx.x & (8 / P - 1)) == 0) ++expanded;
  const u64 cand = key_up(a.f, kv);
  const u32 cl = key_level(a.f, cand);
  for (u32 ch = 0;;) {
    u64 met[P];
    u32 local = 0, glob = 0;
#pragma unroll
    for (int q = 0; q < P; ++q) {
      const bool on = w[q] < a.n;
      met[q] = offer_min(a.key + (on ? w[q] : 0u), cand, on, cand);
    }
    // thin levels: the rows that the next level reads come into L1 while the
    // offers are on their way (1000 x 1000 grid 1290 -> 1203 us)
    if (P == 1 && w[0] < a.n)
      asm volatile("prefetch.global.L1 [%0];" ::"l"(a.ell + (size_t)w[0] * a.ell_s));
#pragma unroll
    for (int q = 0; q < P; ++q) {
      pushed += w[q] < a.n ? 1u : 0u;
      if (met[q] > cand) {
        if (cl < H) local |= 1u << q;
        else if (key_level(a.f, met[q]) > H) glob |= 1u << q;
      }
    }
    bool tie = false;  // one branch for the batch: meetings are rare
#pragma unroll
    for (int q = 0; q < P; ++q) tie |= key_near(cand, met[q]);
    if (tie) {
#pragma unroll
      for (int q = 0; q < P; ++q) note_tie(a, w[q], cand, met[q]);
    }
    window_push<P, kCap>(local, w, cand, a, s, nb, nc, qi, qb);
    warp_append<P, true>(glob, w, a, qi, qb);
    if (!__any_sync(kFull, more)) break;
    more = ell_load<P>(a, v, ++ch, more, w);
  }
}

// A window's first level: the global frontier (Q entries of side qcur) and the
// overflow list up to item `total`, whose keys are loaded here.
template <bool U, int kCap, int P>
__device__ __forceinline__ void window_first(const BfsArgs& a, Smem& s, u32 Q, u32 total, int qcur,
                                             u32 L, u32 H, int nb, int nc, int qi, int qb,
                                             u64& pushed, u64& expanded) {
  constexpr u32 G = 8 / P;
  const u32 sub = (threadIdx.x & 31) / G;
  for (u32 base = warp_first_item(1) / G; base < total; base += gridDim.x * blockDim.x / G) {
    const u32 i = base + sub;
    u32 v = 0, lev = L;
    if (i < Q) {
      v = ld_cg_u32(a.qv[qcur] + i);
    } else if (i < total) {
      v = ld_cg_u32(reinterpret_cast<const u32*>(a.qrow[qcur]) + (i - Q));
      lev = ld_cg_u32(a.qoff[qcur] + (i - Q));
    }
    u64 kv = 0;
    bool ok = i < total;
    if (ok) kv = ld_cg_u64(a.key + v);
    u32 w[P];
    bool more = ell_load<P>(a, v, 0, ok, w);
    ok = ok && key_level(a.f, kv) >= lev;  // lowered since: its lowerer pushed it again
    if (!ok) {
      more = false;
#pragma unroll
      for (int q = 0; q < P; ++q) w[q] = ~0u;
    }
    window_expand<U, kCap, P>(a, s, ok, kv, v, w, more, H, nb, nc, qi, qb, pushed, expanded);
  }
}

// The CTA's local queue lb: nloc entries.
template <bool U, int kCap, int P>
__device__ __forceinline__ void window_local(const BfsArgs& a, Smem& s, u32 nloc, int lb, u32 H,
                                             int nb, int nc, int qi, int qb, u64& pushed,
                                             u64& expanded) {
  constexpr u32 G = 8 / P;
  const LocalQueue lq = lq_buf<kCap>(s, lb);
  const u32 sub = (threadIdx.x & 31) / G;
  for (u32 base = (threadIdx.x & ~31u) / G; base < nloc; base += blockDim.x / G) {
    const u32 i = base + sub;
    const bool ok = i < nloc;
    const u32 v = ok ? lq.v[i] : 0u;
    u32 w[P];
    const bool more = ell_load<P>(a, v, 0, ok, w);
    window_expand<U, kCap, P>(a, s, ok, ok ? lq.key[i] : 0ull, v, w, more, H, nb, nc, qi, qb,
                              pushed, expanded);
  }
}

// One window of levels [L, H): the level-L frontier (Q entries of qv_cur) and
// the nov overflow entries of the last round (qrow/qoff of side qcur, vertex
// and level), then local levels L .. H - 1, then whatever the CTA's local
// queue still holds.
// Only pushes that find the local queue full wait for the next round (on the
// overflow list).  `expanded` counts expansions.
//
// Start buckets are read one level ahead: at level lv this thread's first entry
// of bucket lv + 1 is known (its key is requested as the level starts, beside the
// expansions) and its first entry of bucket lv + 2 and the bounds of bucket
// lv + 3 are requested.  A key read before the level's expansions can only be
// higher than after them: a start taken on it that a correction undercuts is an
// entry that its expansion skips.  What a window has read ahead as it ends is
// kept for the next one (BucketsAhead), which starts at the level it is for
// unless the CTA ran past the window's end or buckets were filled since.  A
// window's start is a chain of round trips that every CTA waits for: with this,
// the depth found by 32 lanes at once and the first level's rows requested
// beside its keys, the 1000 x 1000 grid went from 1353 to 1290 us, the 256^3 grid
// from 2667 to 2558.
constexpr u32 kNoItem = 0xffffffffu;
struct BucketsAhead {
  u32 lv = kNoItem;                    // read for a window that starts at this level
  int lo1 = 0, hi1 = 0, lo2 = 0, hi2 = 0;  // buckets lv + 1 and lv + 2
  u32 first = kNoItem;                 // this thread's first entry of bucket lv + 1
};

template <bool U, int kCap>
__device__ __forceinline__ void window_ld(const BfsArgs& a, Smem& s, int lv0, int A, int built,
                                          BucketsAhead& ahead, u32 Q, u32 nov, int qcur, u32 L, u32 H,
                                          int qi, int qb, u64& pushed, u64& expanded) {
  const int* bp = a.bptr - lv0;    // start buckets by level
  const u32* rc = a.rcur - lv0;
  const u32* rv = a.rv;
  const u32 lane = threadIdx.x & 31;
  const u32 i0 = warp_first_item(1, true) + lane;  // this thread's first entry of a bucket
  const u32 gstride = gridDim.x * blockDim.x;
  const int filled = min(A, built);
  auto bucket_ok = [&](u32 r) { return (int)r <= filled; };
  int b1lo = ahead.lo1, b1hi = ahead.hi1, b2lo = ahead.lo2, b2hi = ahead.hi2;
  u32 pu = ahead.first;
  if (ahead.lv != L) {  // the same for the whole CTA
    b1lo = b1hi = b2lo = b2hi = 0;
    if (bucket_ok(L + 1)) {
      b1lo = __ldg(bp + L + 1);
      b1hi = (int)ld_cg_u32(rc + L + 1);
    }
    if (bucket_ok(L + 2)) {
      b2lo = __ldg(bp + L + 2);
      b2hi = (int)ld_cg_u32(rc + L + 2);
    }
    pu = kNoItem;
    if (i0 < (u32)(b1hi - b1lo)) pu = ld_cg_u32(rv + b1lo + (int)i0);
  }
  int lb = 0;  // the local queue being read (level lv); the other one is filled
  int cr = 0;  // the counter of the queue being read; (cr + 1) % 3 counts the filled one
  for (u32 lv = L;; ++lv) {
    const int nb = lb ^ 1;
    const int nc = cr == 2 ? 0 : cr + 1;
    // the third counter, read last at level lv - 1 and filled next at level
    // lv + 1, is cleared now: one CTA barrier per level
    if (threadIdx.x == 0) s.lcnt[nc == 2 ? 0 : nc + 1] = 0;
    const u32 nloc = min(s.lcnt[cr], lq_limit<kCap>(a));  // the same for the whole CTA
    // Past the window's last level the CTA goes on with its own queue until
    // it is empty: entries of overflow from an earlier window run behind the
    // frontier, and their chains end here instead of one hop per round.
    if (lv >= H && nloc == 0) {
      ahead.lv = lv;
      ahead.lo1 = b1lo;
      ahead.hi1 = b1hi;
      ahead.lo2 = b2lo;
      ahead.hi2 = b2hi;
      ahead.first = pu;
      break;
    }
    u64 pk = 0;  // its key
    if (pu != kNoItem) pk = ld_cg_u64(a.key + pu);
    u32 pu2 = kNoItem;
    if (i0 < (u32)(b2hi - b2lo)) pu2 = ld_cg_u32(rv + b2lo + (int)i0);
    int b3lo = 0, b3hi = 0;
    if (bucket_ok(lv + 3)) {
      b3lo = __ldg(bp + lv + 3);
      b3hi = (int)ld_cg_u32(rc + lv + 3);
    }
    // (1) the window's first level: the global frontier and the overflow list,
    // whose keys are loaded here
    if (lv == L) {
      const u32 total = Q + nov;
      if (total <= gstride / 8 * kLdGroupPasses)
        window_first<U, kCap, 1>(a, s, Q, total, qcur, L, H, nb, nc, qi, qb, pushed, expanded);
      else
        window_first<U, kCap, 8>(a, s, Q, total, qcur, L, H, nb, nc, qi, qb, pushed, expanded);
    }
    // (2) this CTA's local queue of level lv: keys come with the entries
    if (nloc <= blockDim.x / 8 * kLdGroupPasses)
      window_local<U, kCap, 1>(a, s, nloc, lb, H, nb, nc, qi, qb, pushed, expanded);
    else
      window_local<U, kCap, 8>(a, s, nloc, lb, H, nb, nc, qi, qb, pushed, expanded);
    // (3) start bucket lv + 1: a vertex whose key still has its start level joins level lv + 1
    if (lv < H && bucket_ok(lv + 1)) {
      const u32 cnt = (u32)(b1hi - b1lo);
      for (u32 base = i0 - lane; base < cnt; base += gstride) {  // warp-uniform
        const u32 i = base + lane;
        u32 u[1] = {0};
        u64 k = 0;
        bool start = false;
        if (i < cnt) {
          if (i == i0) {  // the entry read ahead
            u[0] = pu;
            k = pk;
          } else {
            u[0] = ld_cg_u32(rv + b1lo + (int)i);
            k = ld_cg_u64(a.key + u[0]);
          }
          start = key_level(a.f, k) == lv + 1;
        }
        if (lv + 1 < H) {
          window_push<1, kCap>(start ? 1u : 0u, u, k, a, s, nb, nc, qi, qb);
        } else {
          warp_append<1, true>(start ? 1u : 0u, u, a, qi, qb);
        }
      }
    }
    __syncthreads();  // every push of level lv + 1 is in; level lv's queue is read
    lb = nb;
    cr = nc;
    pu = pu2;
    b1lo = b2lo;
    b1hi = b2hi;
    b2lo = b3lo;
    b2hi = b3hi;
  }
}

// The smallest start level in from .. to among start-bucket entries whose key
// still has their start level (a vertex nobody has claimed), into
// ctl->nstart[slot] as ~level by atomicMax (0 if none); the caller waits at a
// grid barrier.  A thread takes one place of the buckets' room at a time and
// finds its bucket by a search in bptr.
__device__ __forceinline__ void scan_unclaimed(const BfsArgs& a, int lv0, int from, int to,
                                               u32 slot) {
  const int* bp = a.bptr - lv0;
  const int lo = __ldg(bp + from), hi = __ldg(bp + to + 1);
  u32 best = 0;
  for (int i = lo + (int)(blockIdx.x * blockDim.x + threadIdx.x); i < hi;
       i += (int)(gridDim.x * blockDim.x)) {
    int r = from, r1 = to;  // the last bucket that starts at or before i
    while (r < r1) {
      const int mid = (r + r1 + 1) >> 1;
      if (__ldg(bp + mid) <= i) r = mid;
      else r1 = mid - 1;
    }
    if (i >= (int)ld_cg_u32(a.rcur + (r - lv0))) continue;  // room not used
    if (key_level(a.f, ld_cg_u64(a.key + ld_cg_u32(a.rv + i))) == (u32)r)
      best = max(best, ~(u32)r);
  }
  best = __reduce_max_sync(kFull, best);
  if ((threadIdx.x & 31) == 0 && best) atomicMax(&a.ctl->nstart[slot], best);
}

// Leaves the warp's smallest tie-break for the barrier and resets the thread's.
template <bool kTrack>
__device__ __forceinline__ void post_cta_min(const BfsArgs& a, Smem& s, u64& mylow) {
  if (!kTrack) return;
  const u64 wm = warp_min64(mylow);
  if (mylow != ~0ull) note_tie(a, 0, mylow, wm);
  if ((threadIdx.x & 31) == 0) s.minlow[threadIdx.x >> 5] = wm;
  mylow = ~0ull;
}

// The two appends of a bottom-up step in one pass.  The vertices of `mask`
// join the next frontier; their adjacency ranges [rs, re) are known already,
// so, unlike warp_append, no row_ptr round trip comes first.  The vertices of
// `keep` join the list of the next bottom-up round.  Lane 0 sends both
// reservations before waiting for either.
template <int K, bool LD>
__device__ __forceinline__ void pull_append(u32 mask, u32 keep, const u32 (&v)[K],
                                            const int (&rs)[K], const int (&re)[K],
                                            const BfsArgs& a, int qi, int qb, u32* list,
                                            u32* lcount) {
  const u32 lane = threadIdx.x & 31;
  u32 cnt = 0, dsum = 0;
#pragma unroll
  for (int i = 0; i < K; ++i)
    if (mask >> i & 1u) {
      if (re[i] <= rs[i]) {
        mask &= ~(1u << i);  // a vertex without arcs has nothing to expand
      } else {
        ++cnt;
        dsum += (u32)(re[i] - rs[i]);
      }
    }
  const u32 kc = __popc(keep);
  if (!__any_sync(kFull, mask != 0u || keep != 0u)) return;
  const u64 mine = ((u64)cnt << 32) | (LD ? 0u : dsum);
  u64 incl = mine;
  u32 kincl = kc;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const u64 y = __shfl_up_sync(kFull, incl, o);
    const u32 ky = __shfl_up_sync(kFull, kincl, o);
    if (lane >= (u32)o) {
      incl += y;
      kincl += ky;
    }
  }
  const u64 tot = __shfl_sync(kFull, incl, 31);
  const u32 ktot = __shfl_sync(kFull, kincl, 31);
  u64 base = 0;
  u32 kbase = 0;
  if (lane == 0) {
    if (tot) base = atomicAdd(&a.ctl->qctr[qi], tot);
    if (ktot) kbase = atomicAdd(lcount, ktot);
  }
  base = __shfl_sync(kFull, base, 0) + (incl - mine);
  kbase = __shfl_sync(kFull, kbase, 0) + (kincl - kc);
  u32 slot = (u32)(base >> 32), off = (u32)base;
#pragma unroll
  for (int i = 0; i < K; ++i)
    if (mask >> i & 1u) {
      a.qv[qb][slot] = v[i];
      if (!LD) {
        const u32 dg = (u32)(re[i] - rs[i]);
        a.qrow[qb][slot] = rs[i];
        a.qoff[qb][slot] = off;
        const u32 end = off + dg;
        for (u32 c = (off + kBfsBase - 1) / kBfsBase; c * kBfsBase < end; ++c) a.cf[qb][c] = slot;
        off = end;
      }
      ++slot;
    }
#pragma unroll
  for (int i = 0; i < K; ++i)
    if (keep >> i & 1u) list[kbase++] = v[i];
}

// Low-degree rounds of a single graph: the floor of a bottom-up round, from its
// frontier list, with a grid barrier.
__device__ __forceinline__ u64 list_floor(const BfsArgs& a, Smem& s, const u32* qv, u32 Q, u32 slot,
                                          u32& gen, int lv0) {
  u64 low = ~0ull;
  for (u32 i = blockIdx.x * blockDim.x + threadIdx.x; i < Q; i += gridDim.x * blockDim.x)
    note_low<true>(a, true, ld_cg_u64(a.key + ld_cg_u32(qv + i)), low);
  post_cta_min<true>(a, s, low);
  grid_barrier<true>(a, gen, slot, lv0, -1, s);
  return s.next_minlow;
}

// Puts vertices w[i] (bits of mask; with kPushFlag: see pull_rest) with the
// arcs [e[i], re[i]) on the list that pull_rest works off, in the frontier's
// own format (vertex, first arc, exclusive arc offset, first slot of every base
// chunk) on side kRestSide of the frontier arrays.
template <int K>
__device__ __forceinline__ void defer_append(u32 mask, const u32 (&w)[K], const int (&e)[K],
                                             const int (&re)[K], const BfsArgs& a, u64* ctr) {
  if (!__any_sync(kFull, mask != 0u)) return;
  const u32 lane = threadIdx.x & 31;
  u64 mine = 0;
#pragma unroll
  for (int i = 0; i < K; ++i)
    if (mask >> i & 1u) mine += kLevelOne | (u32)(re[i] - e[i]);
  u64 incl = mine;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const u64 y = __shfl_up_sync(kFull, incl, o);
    if (lane >= (u32)o) incl += y;
  }
  u64 base = 0;
  if (lane == 31) base = atomicAdd(ctr, incl);
  base = __shfl_sync(kFull, base, 31) + (incl - mine);
  u32 slot = (u32)(base >> 32), off = (u32)base;
#pragma unroll
  for (int i = 0; i < K; ++i)
    if (mask >> i & 1u) {
      a.qv[kRestSide][slot] = w[i];
      a.qrow[kRestSide][slot] = e[i];
      a.qoff[kRestSide][slot] = off;
      const u32 end = off + (u32)(re[i] - e[i]);
      for (u32 c = (off + kBfsBase - 1) / kBfsBase; c * kBfsBase < end; ++c)
        a.cf[kRestSide][c] = slot;
      ++slot;
      off = end;
    }
}

// A bottom-up round's pivot (single graphs): kPivotSamples evenly spaced
// samples of the frontier's E arcs, each with its vertex's tie-break; the
// kPivotSkip-th smallest.  Every CTA takes the same samples of a list that no
// longer changes, so all get the same pivot without a barrier.
__device__ __forceinline__ u64 pivot_low(const BfsArgs& a, Smem& s, int cur, u32 Q, u32 E) {
  const u32 nb = (E + kBfsBase - 1) / kBfsBase;
  u64* smp = s.cand;
  u64 r = 0;
  __syncthreads();
  if (threadIdx.x < kPivotSamples) {
    const u32 slot = ld_cg_u32(a.cf[cur] + (u32)((u64)threadIdx.x * nb / kPivotSamples));
    r = key_low(a.f, ld_cg_u64(a.key + ld_cg_u32(a.qv[cur] + min(slot, Q - 1))));
    smp[threadIdx.x] = r;
  }
  __syncthreads();
  if (threadIdx.x < kPivotSamples) {
    u32 less = 0, same = 0;
#pragma unroll 8
    for (u32 i = 0; i < kPivotSamples; ++i) {
      const u64 x = smp[i];
      less += x < r ? 1u : 0u;
      same += x == r ? 1u : 0u;
    }
    if (less <= kPivotSkip && kPivotSkip < less + same) s.pivot = r;  // one value
  }
  __syncthreads();
  return s.pivot;
}

// The frontier vertices whose tie-break lies below the pivot (their member's
// pivot), or differs from it only in the id, go on pull_rest's list, to push.
template <bool U>
__device__ __forceinline__ void list_pushes(const BfsArgs& a, int cur, u32 Q, u64 pivot,
                                            u32 mslot, int qi, const u64* s_floor) {
  const u32 lane = threadIdx.x & 31;
  const u32 stride = gridDim.x * blockDim.x;
  for (u32 base = warp_first_item(1); base < Q; base += stride) {
    const u32 i = base + lane;
    u32 v[1] = {0};
    int rs[1] = {0}, re[1] = {0};
    bool push = false;
    if (i < Q) {
      v[0] = ld_cg_u32(a.qv[cur] + i);
      const u64 r = key_low(a.f, ld_cg_u64(a.key + v[0]));
      const u64 pv = U ? member_floor(a, v[0], mslot, s_floor, true) : pivot;
      push = r < pv || key_tie(a.f, r, pv);
      if (push) {
        note_tie(a, v[0], r, pv);  // a scan may stop at r, the pivot's own offer unread
        rs[0] = __ldg(a.row_ptr + v[0]);
        re[0] = __ldg(a.row_ptr + v[0] + 1);
        v[0] |= kPushFlag;
      }
    }
    defer_append<1>(push && rs[0] < re[0] ? 1u : 0u, v, rs, re, a, &a.ctl->rest[qi]);
  }
}

// Second pass of a large bottom-up round.  The first pass stops a scan at the
// first key of level L whose rank is at most the pivot, a rank that most of
// the frontier's arcs carry (the floor itself may belong to a center that
// hardly any candidate can reach; scans that wait for it read every arc).
// What can beat such a key comes from the few frontier vertices of smaller
// rank, which push instead.  The list (Q entries, E arcs) holds these, marked
// with kPushFlag, and the scans that the first pass put off.
//
// Arcs are dealt out in equal shares whatever the rows' lengths: a lane takes
// 8 k consecutive ones (a warp 256 k), k up to 4 once every warp has work, and
// finds their first row by a search between the slots of the chunk's ends.  It
// reads kRestBatch neighbours at a time.  A scan keeps its smallest offer and
// sends one atomicMin per row and lane (one per warp when all lanes end in the
// same row), and is passed over once its key cannot be beaten; a push sends
// one atomicMin per neighbour it improves.
//
// What bounded such rounds was the number of arcs scanned (up to 123 of R-MAT
// 22's 128 M) and the chain of one warp alone on a 160,000-arc row; now it is
// the latency of the first pass.  R-MAT 22's round loop, 24 shift seeds at
// beta 0.02 / 0.1 / 0.5: mean 189 / 205 / 605 -> 183 / 183 / 197 us, worst
// 289 / 385 / 4794 -> 279 / 281 / 301 us.  Putting scans off without the pivot
// left the mean at 339 us at beta 0.5; a grid barrier inside the round instead
// of a second one only when something is listed cost 20 us per decomposition.
// The pivot needs a frontier of fewer vertices than there are candidates (else
// listing the pushes costs more than the scans: 8 -> 42 us in R-MAT 22's second
// bottom-up round) and at least kDeferMin candidates.
template <bool U>
__device__ __forceinline__ void pull_rest(const BfsArgs& a, u32 Q, u32 E, int lvl, u64 pivot,
                                          u32 mslot, int qi, int qb, u64& mylow,
                                          const u64* s_floor) {
  constexpr u32 kNone = 0xffffffffu;
  const u32 lane = threadIdx.x & 31;
  const u32 L = (u32)lvl;
  const u64 lvl_key = level_key(a.f, L + 1);
  const u32 nchunk = (E + kBfsBase - 1) / kBfsBase;
  const u32 W = gridDim.x * (blockDim.x >> 5);
  const u32 k = max(1u, min(nchunk / W, 4u));
  const u32 nunit = (nchunk + k - 1) / k;
  const u32* qv = a.qv[kRestSide];
  const int* qrow = a.qrow[kRestSide];
  const u32* qoff = a.qoff[kRestSide];
  const u32* cf = a.cf[kRestSide];
  u32 scanned = 0, pushed = 0;
  for (u32 unit = (threadIdx.x >> 5) * gridDim.x + blockIdx.x; unit < nunit; unit += W) {
    const u32 c0 = unit * k, c1 = min(c0 + k, nchunk);
    u32 lo = ld_cg_u32(cf + c0);
    u32 hi = c1 < nchunk ? ld_cg_u32(cf + c1) : Q - 1;
    u32 p = c0 * kBfsBase + lane * (k * (kBfsBase / 32));
    const u32 p1 = min(min(p + k * (kBfsBase / 32), c1 * kBfsBase), E);
    if (lo >= Q || hi >= Q) {  // chunk table broken: cannot happen
      atomicOr(&a.ctl->err, kErrInternal);
      return;
    }
    if (p < p1)
      while (lo < hi) {  // the last slot whose first arc is at most p
        const u32 mid = (lo + hi + 1) >> 1;
        if (ld_cg_u32(qoff + mid) <= p) lo = mid;
        else hi = mid - 1;
      }
    u32 slot = lo, w = kNone, end = p;  // end == p: the row at p is not open yet
    int rowd = 0;
    u64 kw = 0, fl = 0, best = ~0ull;
    bool fresh = true, push = false;
    while (__any_sync(kFull, p < p1)) {
      if (p < p1 && p == end) {  // open the row of slot: its range, key and floor
        if (!fresh) ++slot;
        fresh = false;
        w = ld_cg_u32(qv + slot);
        push = (w & kPushFlag) != 0;
        w &= ~kPushFlag;
        const u32 off = ld_cg_u32(qoff + slot);
        rowd = ld_cg_i32(qrow + slot) - (int)off;
        end = slot + 1 < Q ? ld_cg_u32(qoff + slot + 1) : E;
        kw = ld_cg_u64(a.key + w);
        fl = lvl_key | (U ? member_floor(a, w, mslot, s_floor, true) : pivot);
        best = ~0ull;
      }
      const u32 stop = min(end, p1);
      if (!push && p < stop && min(kw, best) <= fl) p = stop;  // nothing can beat it
      u32 vv[kRestBatch];
#pragma unroll
      for (int q = 0; q < kRestBatch; ++q)
        vv[q] = p + q < stop ? (u32)__ldg(a.col + (rowd + (int)(p + q))) : kNone;
      u64 kv[kRestBatch];
#pragma unroll
      for (int q = 0; q < kRestBatch; ++q) kv[q] = vv[q] < a.n ? ld_cg_u64(a.key + vv[q]) : ~0ull;
      u32 got = p < stop ? min(stop - p, (u32)kRestBatch) : 0u;
      u32 join = 0;
      if (push) {
        const u64 cand = key_up(a.f, kw);
        bool won = false, tie = false;
        pushed += got;
#pragma unroll
        for (int q = 0; q < kRestBatch; ++q) {
          const bool on = vv[q] < a.n && cand < kv[q];
          if (on) join |= 1u << q;
          kv[q] = offer_min(a.key + (on ? vv[q] : 0u), cand, on, kv[q]);
        }
#pragma unroll
        for (int q = 0; q < kRestBatch; ++q) {
          if (join >> q & 1u) {
            won |= kv[q] > cand;
            if (key_level(a.f, kv[q]) <= L + 1) join &= ~(1u << q);
          }
          tie |= vv[q] < a.n && key_near(cand, kv[q]);
        }
        note_low<!U>(a, won, cand, mylow);
        if (tie) {
#pragma unroll
          for (int q = 0; q < kRestBatch; ++q)
            if (vv[q] < a.n) note_tie(a, vv[q], cand, kv[q]);
        }
      } else {
        scanned += got;
#pragma unroll
        for (int q = 0; q < kRestBatch; ++q)
          if (vv[q] < a.n && key_level(a.f, kv[q]) == L) {
            const u64 cand = key_up(a.f, kv[q]);
            note_tie(a, w, cand, best);
            best = min(best, cand);
          }
      }
      warp_append<kRestBatch, false>(join, vv, a, qi, qb);
      p += got;
      // the end of a scan, or of this lane's share of it: offer what was found
      const bool offer = !push && w != kNone && p == stop && best < kw;
      if (!push && w != kNone && p == stop && best > kw) {
        note_tie(a, w, best, kw);
        best = ~0ull;  // once
      }
      const u32 om = __ballot_sync(kFull, offer);
      if (om) {
        const int first = __ffs(om) - 1;
        const u32 w0 = __shfl_sync(kFull, w, first);
        bool mine = offer;
        if (__all_sync(kFull, !offer || w == w0)) {
          const u64 b = warp_min64(offer ? best : ~0ull);
          if (offer) {
            note_tie(a, w, best, b);
            best = b;
          }
          mine = (int)lane == first;
        }
        u32 won = 0;
        if (mine) {
          const u64 old = atomicMin(a.key + w, best);
          note_tie(a, w, best, old);
          note_low<!U>(a, old > best, best, mylow);
          if (key_level(a.f, old) > L + 1) won = 1;
        }
        const u32 ww[1] = {w};
        warp_append<1, false>(won, ww, a, qi, qb);
        if (offer) kw = best;  // not offered again
      }
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    scanned += __shfl_xor_sync(kFull, scanned, o);
    pushed += __shfl_xor_sync(kFull, pushed, o);
  }
  if (lane == 0 && scanned) atomicAdd(&a.ctl->pull_arcs, (u64)scanned);
  if (lane == 0 && pushed) atomicAdd(&a.ctl->push_arcs, (u64)pushed);
}

// Bottom-up round from level lvl (see the file comment).  Candidates are every
// vertex not in excl (from_list = false; a.active lists them when it is set)
// or the list `cand` of ncand vertices.
// Each lane takes kPullV candidates at a time and advances their neighbour
// scans in lock-step, one neighbour each per step, so that up to kPullV
// independent loads are in flight per lane.  A scan's first probe is the
// candidate's first neighbour from the per-graph table (when there is one),
// loaded beside its key, so it needs no col round trip.  Adds the arcs it
// scans and the vertices it examines to the statistics.
template <bool U, bool LD, int kPullV>
__device__ __forceinline__ void pull_round(const BfsArgs& a, int lvl, u64 stop_low, u32 mslot,
                                           int qi, int qb, bool from_list, const u32* cand,
                                           u32 ncand, u32* ulist_out, u32* ucnt_out,
                                           u64& mylow, const u64* s_floor, bool defer) {
  constexpr u32 kNone = 0xffffffffu;
  u32 scanned = 0, examined = 0;
  const u32 lane = threadIdx.x & 31;
  const u32 L = (u32)lvl;
  if (!from_list && a.active) {  // the first bottom-up round: the BFS's own vertices
    from_list = true;
    cand = a.active;
    ncand = a.n_active;
  }
  const u32 total = from_list ? ncand : a.n;
  // Units of 32 kPullV candidates.  A single graph deals about three fifths
  // of them out in advance, kd per warp (warps interleaved across CTAs as
  // everywhere), a union only every warp's first; the rest go to whichever
  // warp asks next, one atomic ticket per unit, so a warp held up by hub scans
  // takes fewer units instead of holding the round.  (R-MAT 22 round loop
  // 0.143 -> 0.136 ms; 64 R-MAT 20 copies as a union 5.2 -> 4.0 ms, where
  // dealing three fifths in advance gave 4.9 ms.)
  constexpr u32 kUnit = 32u * kPullV;
  const u32 W = gridDim.x * (blockDim.x >> 5);
  const u32 kd = U ? 1u : max(1u, ((total + kUnit - 1) / kUnit / W) * 3 / 5);
  u32* const next_unit = &a.ctl->pull_ctr[mslot];
  auto unit_base = [&](u32 ticket) {  // lane 0's ticket: the unit's first candidate
    return (kd * W + __shfl_sync(kFull, ticket, 0)) * kUnit;
  };
  // The passes are software-pipelined: pass p + 1's candidates are requested
  // when pass p starts, and their keys and adjacency ranges while pass p makes
  // its appends, so a pass waits only on its neighbour scans and its appends.
  auto load_ids = [&](u32 b, u32 (&w)[kPullV]) {
#pragma unroll
    for (int j = 0; j < kPullV; ++j) {
      const u32 i = b + (u32)j * 32 + lane;
      w[j] = kNone;
      if (from_list) {
        if (i < total) w[j] = ld_cg_u32(cand + i);
      } else if (i < total) {
        const u32 ex = __ldg(a.excl + (i >> 5));  // same word for the whole warp
        if (!((ex >> lane) & 1u)) w[j] = i;
      }
    }
  };
  // the key, the adjacency range and the first neighbour together: one round
  // trip, and the scan's first probe needs no col load
  auto load_keys = [&](const u32 (&w)[kPullV], u64 (&kw)[kPullV], int (&e)[kPullV],
                       int (&re)[kPullV], u32 (&f)[kPullV]) {
#pragma unroll
    for (int j = 0; j < kPullV; ++j) {
      kw[j] = 0ull;
      e[j] = 0;
      re[j] = 0;
      f[j] = kNone;
      if (w[j] != kNone) {
        kw[j] = ld_cg_u64(a.key + w[j]);
        e[j] = __ldg(a.row_ptr + w[j]);
        re[j] = __ldg(a.row_ptr + w[j] + 1);
        if (a.first) f[j] = __ldg(a.first + w[j]);
      }
    }
  };
  u32 base = warp_first_item(kPullV);
  u32 w[kPullV], f[kPullV];
  u64 kw[kPullV];
  int e[kPullV], re[kPullV];
  load_ids(base, w);
  load_keys(w, kw, e, re, f);
  const u32 gw = base / kUnit;  // this warp's first unit
  auto dealt_base = [&](u32 p) { return (p * W + gw) * kUnit; };  // its pass p < kd
  u32 pass = 0, ticket = 0;
  if (lane == 0 && kd <= 1 && base < total) ticket = atomicAdd(next_unit, 1u);
  u32 nbase = kd > 1 ? dealt_base(1) : (base < total ? unit_base(ticket) : total);
  while (base < total) {
    u32 wn[kPullV];  // the next pass's candidates, in flight during this pass
    load_ids(nbase, wn);
    // the ticket for the pass after the next: its atomic returns during this pass
    if (lane == 0 && pass + 2 >= kd && nbase < total) ticket = atomicAdd(next_unit, 1u);
    int rs0[kPullV], re0[kPullV];  // the adjacency ranges, for the appends
#pragma unroll
    for (int j = 0; j < kPullV; ++j) {
      rs0[j] = e[j];
      re0[j] = re[j];
    }
    u64 best[kPullV];
    u64 fr[kPullV];  // nothing beats (L + 1, fr); union: w's own member's
#pragma unroll
    for (int j = 0; j < kPullV; ++j) {
      fr[j] = stop_low;
      if (U && w[j] != kNone) fr[j] = member_floor(a, w[j], mslot, s_floor, !LD && defer);
    }
    const u64 lvl_key = level_key(a.f, L + 1);
#pragma unroll
    for (int j = 0; j < kPullV; ++j) {
      best[j] = kw[j];
      if (w[j] != kNone) ++examined;
      if (!(key_level(a.f, kw[j]) > L && kw[j] > (lvl_key | fr[j]))) re[j] = e[j];  // settled or unbeatable
      if (U && fr[j] == ~0ull) re[j] = e[j];  // w's member has no level-L key
    }
    // a start of level L + 1 may only tie with the floor or pivot that it is passed over for
    bool tie = false;
#pragma unroll
    for (int j = 0; j < kPullV; ++j) tie |= key_near(kw[j], lvl_key | fr[j]);
    if (tie) {
#pragma unroll
      for (int j = 0; j < kPullV; ++j)
        if (w[j] != kNone) note_tie(a, w[j], kw[j], lvl_key | fr[j]);
    }
    // the first neighbour of every candidate, then two of every one still
    // scanning per step, for about kPullLong neighbours: most scans stop at the
    // first, and the warp's slowest lane sets the pass (one per step: 64 R-MAT 20
    // copies 5.98 ms a call against 5.86, a batch of three of R-MAT 20 .645 against .625)
    bool all_off = false;
    for (int step = 0; step < kPullLong / 2; ++step) {
      if (!LD && defer && step == kPullShort / 2) {
        u32 going = 0;
#pragma unroll
        for (int j = 0; j < kPullV; ++j) going += e[j] < re[j] ? 1u : 0u;
        all_off = __reduce_add_sync(kFull, going) >= kDeferLanes;
        if (all_off) break;
      }
      bool any = false;
      u32 vv[kPullV];
#pragma unroll
      for (int j = 0; j < kPullV; ++j) {
        vv[j] = kNone;
        if (e[j] < re[j]) {
          vv[j] = (step == 0 && a.first) ? f[j] : (u32)__ldg(a.col + e[j]);
          ++e[j];
          ++scanned;
          any = true;
        }
      }
      u32 vx[kPullV];
#pragma unroll
      for (int j = 0; j < kPullV; ++j) {
        vx[j] = kNone;
        if (step > 0 && e[j] < re[j]) {
          vx[j] = (u32)__ldg(a.col + e[j]);
          ++e[j];
          ++scanned;
        }
      }
      if (!LD && defer ? !__any_sync(kFull, any) : !any) break;  // with defer: the warp together
      u64 kv[kPullV];
#pragma unroll
      for (int j = 0; j < kPullV; ++j) kv[j] = (vv[j] < a.n) ? ld_cg_u64(a.key + vv[j]) : ~0ull;
      u64 kx[kPullV];
#pragma unroll
      for (int j = 0; j < kPullV; ++j) kx[j] = (vx[j] < a.n) ? ld_cg_u64(a.key + vx[j]) : ~0ull;
#pragma unroll
      for (int j = 0; j < kPullV; ++j) {
        if (vv[j] < a.n && key_level(a.f, kv[j]) == L) {
          const u64 cand = key_up(a.f, kv[j]);
          note_tie(a, w[j], cand, best[j]);
          best[j] = min(best[j], cand);
        }
        if (vx[j] < a.n && key_level(a.f, kx[j]) == L) {
          const u64 cand = key_up(a.f, kx[j]);
          note_tie(a, w[j], cand, best[j]);
          best[j] = min(best[j], cand);
        }
        if (best[j] <= (lvl_key | fr[j])) re[j] = e[j];  // nothing can beat (L + 1, fr)
      }
    }
    // scans still going (no early exit): put off to pull_rest, or the warp
    // takes them one at a time, 32 x kPullCoop coalesced neighbours per step,
    // with the same early exit per step
    if (!LD && defer) {
      u32 dm = 0;
#pragma unroll
      for (int j = 0; j < kPullV; ++j)
        if (e[j] < re[j] && (all_off || re[j] - e[j] >= kDeferLong)) dm |= 1u << j;
      defer_append<kPullV>(dm, w, e, re, a, &a.ctl->rest[qi]);
#pragma unroll
      for (int j = 0; j < kPullV; ++j)
        if (dm >> j & 1u) e[j] = re[j];
    }
#pragma unroll
    for (int j = 0; j < kPullV; ++j) {
      u32 lm = __ballot_sync(kFull, e[j] < re[j]);
      while (lm) {
        const int src = __ffs(lm) - 1;
        lm &= lm - 1;
        const int eb = __shfl_sync(kFull, e[j], src), ee = __shfl_sync(kFull, re[j], src);
        const u64 fj = lvl_key | __shfl_sync(kFull, fr[j], src);
        u64 b = __shfl_sync(kFull, best[j], src);
        const u32 ws = __shfl_sync(kFull, w[j], src);
        int pos = eb;
        while (pos < ee) {
          u32 vq[kPullCoop];
#pragma unroll
          for (int q = 0; q < kPullCoop; ++q) {
            const int idx = pos + q * 32 + (int)lane;
            vq[q] = idx < ee ? (u32)__ldg(a.col + idx) : kNone;
          }
          u64 lb = ~0ull;
#pragma unroll
          for (int q = 0; q < kPullCoop; ++q) {
            const u64 kq = vq[q] < a.n ? ld_cg_u64(a.key + vq[q]) : ~0ull;
            if (vq[q] < a.n && key_level(a.f, kq) == L) {
              const u64 cand = key_up(a.f, kq);
              note_tie(a, ws, cand, lb);
              note_tie(a, ws, cand, b);
              lb = min(lb, cand);
            }
          }
          const u64 wb = warp_min64(lb);
          if (lb != ~0ull) note_tie(a, ws, lb, wb);
          b = min(b, wb);
          pos += 32 * kPullCoop;
          if (b <= fj) break;  // warp-uniform: nothing can beat (L + 1, minrank)
        }
        if ((int)lane == src) {
          best[j] = b;
          scanned += (u32)(min(pos, ee) - eb);
        }
      }
    }
    u64 kwn[kPullV];  // the next pass's keys and ranges, beside this pass's appends
    int en[kPullV], ren[kPullV];
    u32 fnn[kPullV];
    load_keys(wn, kwn, en, ren, fnn);
    u32 mask = 0, keep = 0, won = 0;
#pragma unroll
    for (int j = 0; j < kPullV; ++j) {
      const bool pending = w[j] != kNone && key_level(a.f, kw[j]) > L;
      if (pending && best[j] < kw[j]) {
        a.key[w[j]] = best[j];  // only this thread writes key[w] in a bottom-up round
        won |= 1u << j;
        if (key_level(a.f, kw[j]) > L + 1) mask |= 1u << j;
      }
      // still above level L + 1: examined again by a following bottom-up round
      if (pending && key_level(a.f, min(best[j], kw[j])) > L + 1) keep |= 1u << j;
    }
#pragma unroll
    for (int j = 0; j < kPullV; ++j)
      note_low<!U && !LD>(a, (won >> j) & 1u, best[j], mylow);
    pull_append<kPullV, LD>(mask, keep, w, rs0, re0, a, qi, qb, ulist_out, ucnt_out);
#pragma unroll
    for (int j = 0; j < kPullV; ++j) {
      w[j] = wn[j];
      kw[j] = kwn[j];
      e[j] = en[j];
      re[j] = ren[j];
      f[j] = fnn[j];
    }
    base = nbase;
    ++pass;
    nbase = pass + 1 < kd ? dealt_base(pass + 1) : (base < total ? unit_base(ticket) : total);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    scanned += __shfl_xor_sync(kFull, scanned, o);
    examined += __shfl_xor_sync(kFull, examined, o);
  }
  if (lane == 0) {
    if (scanned) atomicAdd(&a.ctl->pull_arcs, (u64)scanned);
    if (examined) atomicAdd(&a.ctl->pull_verts, (u64)examined);
  }
}

// U: a union of graphs (per-member bottom-up floors); a separate instance so
// that the plain kernel carries none of it.  kPerSm: the CTAs per SM the
// instance is built for.  One CTA per SM leaves it 128 registers per thread
// (no spills) and the cheapest grid barrier, the best for thin frontiers and
// single graphs; two give twice the warps, the best for the wide bottom-up
// rounds of many-seed unions.  The launch parameter bfs_blocks_per_sm picks
// the instance.
template <bool U, int kPerSm, bool LD>
__global__ void __launch_bounds__(kBfsThreads, kPerSm) k_bfs(BfsArgs a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  Smem& s = *reinterpret_cast<Smem*>(smem_raw);
  // union with few enough members: per-member next-level minima and
  // current-level floors in shared memory, after Smem
  u64* s_acc = (U && a.kmem <= kSmemMembers)
                   ? reinterpret_cast<u64*>(smem_raw + sizeof(Smem) + (LD ? lq_extra(kPerSm) : 0))
                   : nullptr;
  u64* s_floor = s_acc ? s_acc + kSmemMembers : nullptr;
  u64* s_piv = s_acc ? s_acc + 2 * kSmemMembers : nullptr;
  if (s_acc)
    for (u32 m = threadIdx.x; m < a.kmem; m += blockDim.x) {
      s_acc[m] = ~0ull;
      s_piv[m] = 0;
    }
  Control* ctl = a.ctl;
  if (threadIdx.x == 0) {
    s.stop = ld_acquire_u32(&ctl->err) != 0u ? 1u : 0u;  // validation failed upstream
    s.lcnt[0] = s.lcnt[1] = s.lcnt[2] = 0;  // a window leaves them at zero
  }
  __syncthreads();
  if (s.stop) return;  // CTA-uniform: read once by thread 0
  // levels lv0 .. A: with direct keys those of the handled vertices' floors
  const int lv0 = a.f.cap ? (int)a.f.cap - ctl->Ab : 0;
  const int A = a.f.cap ? (int)a.f.cap : ctl->A;
  constexpr bool kTrack = !U && !LD;
  u32 gen = 0;
  u64 mylow = ~0ull;  // this thread's smallest successful next-level tie-break
  // start buckets filled so far, and the room for the next ones
  int built = a.f.cap ? lv0 - 1 : A;
  u32 room = max(a.n_active >> kBuildShift, kBuildMin);
  u64 pushed = 0;  // low-degree mode: arcs offered by this thread
  // Level lv0: the vertices with the largest integer shift part start.
  if (a.f.cap) {
    built = build_buckets<U, LD>(a, s, lv0, lv0, A, room, true, mylow);
  } else {
    const int lo = __ldg(a.bptr), hi = (int)ld_cg_u32(a.rcur);
    if (LD)
      expand_ld<U, 8>(a, nullptr, 0, 0, lo, (u32)(hi - lo), (u32)lv0, false, 0, 0, pushed);
    else
      append_bucket<U>(a, lv0, lo, hi, 0, 0, mylow);
  }
  post_cta_min<kTrack>(a, s, mylow);
  grid_barrier<kTrack>(a, gen, 0, lv0, A > lv0 && built > lv0 ? lv0 + 1 : -1, s);
  const bool profiler = blockIdx.x == 0 && threadIdx.x == 0;
  if (profiler) {
    const long long t = clock64();
    ctl->round_clk[0][0] = ctl->round_clk[0][1] = ctl->round_clk[0][2] = t;
    ctl->round_kind[0] = kRoundSkip;
  }

  u64 settled = 0, edges = 0;
  u64 items = 0;     // vertices expanded (a window may expand a vertex twice)
  u64 expanded = 0;  // this thread's expansions inside windows
  u32 phase = 0, pulls = 0, nwin = 0, overflowed = 0;
  u32 wdepth = a.window_levels;  // levels of the next window
  u64 push_arcs = 0;
  int lvl = lv0;
  BucketsAhead ahead;  // windows
  bool pulling = false;
  bool windowed = false;  // a window has run: settled vertices are no longer counted exactly
  // No correct run needs more rounds than this (each round settles a level or
  // jumps to a start bucket); a loop that would is stopped with an error
  // instead of holding the GPU.
  const u64 max_rounds = 2ull * ((u64)a.n_active + (u64)(A - lv0)) + 1024;
  for (;;) {
    if (s.stop) break;  // set by the last barrier, the same for every thread of the CTA
    if (phase > max_rounds) {  // the same for every thread of every CTA
      if (blockIdx.x == 0 && threadIdx.x == 0) atomicOr(&ctl->err, kErrInternal);
      break;
    }
    const u64 c = s.next_c;  // slot phase % 3, read as the last barrier released
    int nb_lo = s.next_lo, nb_hi = s.next_hi;  // start bucket lvl + 1 (if lvl + 1 <= A)
    const u32 Q = (u32)(c >> 32);
    // overflow entries of the last window (more than n cannot have been written:
    // that sets kErrInternal, and the loop stops at the barrier)
    const u32 nov = LD ? min(s.next_ovf, a.n) : 0u;
    // low-degree mode keeps no arc count: the frontier's arcs are estimated
    // from the mean degree (direction choice and probe threshold only)
    const u32 E = LD ? (u32)min((u64)Q * a.nnz_active / max(a.n_active, 1u), 0xffffffffull)
                     : (u32)c;
    settled += Q;
    if (!windowed && settled >= a.n_active) break;  // every vertex the BFS owns has its final key
    const u64 minlow = s.next_minlow;
    const u32 ncand = s.next_ucnt;
    if (blockIdx.x == 0 && threadIdx.x == 0) {
      ctl->qctr[(phase + 2) % 3] = 0;
      ctl->minlow[(phase + 2) % 3] = ~0ull;
      ctl->ucnt[(phase + 2) % 3] = 0;
      ctl->ovf[(phase + 2) % 3] = 0;
      ctl->nstart[(phase + 2) % 3] = 0;
      ctl->pull_ctr[(phase + 2) % 3] = 0;
      ctl->rest[(phase + 2) % 3] = 0;
    }
    if (U)  // the members' floors of the slot that the next round fills
      for (u32 m = blockIdx.x * blockDim.x + threadIdx.x; m < a.kmem; m += gridDim.x * blockDim.x) {
        a.mlow[(size_t)((phase + 2) % 3) * a.kmem + m] = ~0ull;
        if (!LD) a.mpivot[(size_t)((phase + 2) % 3) * a.kmem + m] = 0;
      }
    const int qi = (int)((phase + 1) % 3), qb = (int)((phase + 1) & 1);
    int nlvl;
    bool defer = false;  // a bottom-up round with a second pass ...
    u64 stop_low = 0;    // ... and the tie-break its scans stop at
    if (lvl + 1 <= A && lvl + 1 > built) {  // the next start buckets; each time more at once
      room = room >= (a.n >> 3) ? a.n : room << 3;
      built = build_buckets<U, LD>(a, s, lv0, lvl + 1, A, room, false, mylow);
      ahead.lv = kNoItem;
      grid_barrier<kTrack>(a, gen, kNoPost, lv0, -1, s);
      if (s.stop) break;
      nb_lo = __ldg(a.bptr + (lvl + 1 - lv0));
      nb_hi = (int)ld_cg_u32(a.rcur + (lvl + 1 - lv0));
    }
    // a window of levels: low-degree rounds whose frontier is thin enough, and
    // always while overflow entries of the last window wait
    bool window = false;
    u32 H = 0;
    if (LD && a.window_levels > 1 && (nov > 0 || (Q > 0 && Q <= a.window_max_q))) {
      // The window's depth adapts: halved while the last window's local queues
      // overflowed by more than a quarter of the frontier, doubled again (up
      // to the tuning's) once nothing overflowed; and cut before the first
      // start bucket it would take in locally (buckets lvl + 1 .. H - 1) that
      // holds more than window_max_q vertices.  One level only drains the
      // overflow.  The same for every thread: nov, Q and bptr are.
      if (nov > (Q >> 2)) wdepth = max(wdepth >> 1, 1u);
      else if (nov == 0) wdepth = min(wdepth << 1, a.window_levels);
      // Buckets lvl + 1 .. H must be filled.
      const u32 dmax = built < A ? min(wdepth, (u32)(built - lvl)) : wdepth;
      u32 d = 1;
      for (; d < dmax; d += 32) {  // 32 buckets at once
        const u32 x = d + (threadIdx.x & 31);
        const int r = lvl + (int)x - lv0;
        const u32 big = __ballot_sync(
            kFull, x < dmax && r <= A - lv0 &&
                       (u32)(__ldg(a.bptr + r + 1) - __ldg(a.bptr + r)) > a.window_max_q);
        if (big) {
          d += (u32)__ffs(big) - 1;
          break;
        }
      }
      d = min(d, max(dmax, 1u));
      window = d > 1 || nov > 0;
      H = (u32)lvl + d;
    }
    if (window) {
      edges += E;
      pulling = false;
      window_ld<U, lq_cap(kPerSm)>(a, s, lv0, A, built, ahead, Q, nov, (int)(phase & 1),
                                   (u32)lvl, H, qi, qb, pushed, expanded);
      if (profiler && phase + 1 < (u32)kRoundProfile) ctl->round_clk[phase + 1][0] = clock64();
      windowed = true;
      ++nwin;
      overflowed += nov;
      nlvl = (int)H;
    } else if (Q > 0) {
      items += Q;
      edges += E;
      const u64 unsettled_arcs = a.nnz_active > edges ? a.nnz_active - edges : 0;
      const bool was_pulling = pulling;
      if (!pulling && (u64)E * a.pull_alpha > unsettled_arcs &&
          (u64)E * a.pull_gamma > a.n_active)
        pulling = true;
      else if (pulling && (u64)Q * a.pull_beta < a.n_active)
        pulling = false;
      if (pulling) {
        // large rounds stop at a pivot rank and have a second pass
        defer = !LD && max(Q, kDeferMin) <= (was_pulling ? ncand : a.n_active);
        stop_low = minlow;
        if (U) {  // this level's per-member floors and pivots, from the frontier list
          member_floors<!LD>(a, a.qv[phase & 1], Q, phase % 3, s_acc, s_piv);
          if (s_acc) {
            __syncthreads();
            flush_members<!LD>(a, phase % 3, s_acc, s_piv);
          }
          grid_barrier<kTrack>(a, gen, kNoPost, lv0, -1, s);
          if (s.stop) break;
          if (s_floor) {  // read once per CTA
            for (u32 m = threadIdx.x; m < a.kmem; m += blockDim.x) {
              u64 f = ld_cg_u64(a.mlow + (size_t)(phase % 3) * a.kmem + m);
              if (defer && f != ~0ull) {
                const u64 pv = ld_cg_u64(a.mpivot + (size_t)(phase % 3) * a.kmem + m);
                f = key_low(a.f, ld_cg_u64(a.key + (u32)pv));
              }
              s_floor[m] = f;
            }
            __syncthreads();
          }
        } else if (LD) {
          stop_low = list_floor(a, s, a.qv[phase & 1], Q, phase % 3, gen, lv0);
          if (s.stop) break;
        } else if (defer) {
          stop_low = pivot_low(a, s, (int)(phase & 1), Q, E);
        }
        if (!LD && defer && (U || stop_low > minlow))
          list_pushes<U>(a, (int)(phase & 1), Q, stop_low, phase % 3, qi, s_floor);
        pull_round<U, LD, pull_width(kPerSm)>(a, lvl, stop_low, phase % 3, qi, qb, was_pulling,
                                              a.ulist[phase & 1], ncand, a.ulist[(phase + 1) & 1],
                                              &ctl->ucnt[qi], mylow, s_floor, defer);
        ++pulls;
        if (profiler && phase + 1 < (u32)kRoundProfile) ctl->round_clk[phase + 1][0] = clock64();
        if (lvl + 1 <= A) {
          if (LD) {
            expand_ld<U, 8>(a, nullptr, 0, 0, nb_lo, (u32)(nb_hi - nb_lo), (u32)lvl + 1, false, qi,
                            qb, pushed);
          } else {
            append_bucket<U>(a, lvl + 1, nb_lo, nb_hi, qi, qb, mylow);
          }
        }
      } else if (LD) {  // expansion and start bucket lvl + 1 in one pass
        const bool probe = E >= a.probe_min_arcs;
        const u32* qv = a.qv[phase & 1];
        if (Q + (u32)(nb_hi - nb_lo) <= gridDim.x * blockDim.x / 8 * kLdGroupPasses)
          expand_ld<U, 1>(a, qv, Q, (u32)lvl + 1, nb_lo, (u32)(nb_hi - nb_lo), (u32)lvl + 1, probe,
                          qi, qb, pushed);
        else
          expand_ld<U, 8>(a, qv, Q, (u32)lvl + 1, nb_lo, (u32)(nb_hi - nb_lo), (u32)lvl + 1, probe,
                          qi, qb, pushed);
        if (profiler && phase + 1 < (u32)kRoundProfile) ctl->round_clk[phase + 1][0] = clock64();
      } else {
        expand<U>(a, s, (int)(phase & 1), Q, E, lvl, qi, qb, mylow);
        push_arcs += E;
        if (profiler && phase + 1 < (u32)kRoundProfile) ctl->round_clk[phase + 1][0] = clock64();
        if (lvl + 1 <= A) append_bucket<U>(a, lvl + 1, nb_lo, nb_hi, qi, qb, mylow);
      }
      nlvl = lvl + 1;
    } else {
      if (lvl + 1 > A) break;
      // the next start level that still holds an unclaimed vertex
      scan_unclaimed(a, lv0, lvl + 1, built, phase % 3);
      grid_barrier<kTrack>(a, gen, kNoPost, lv0, -1, s);
      if (s.stop) break;
      if (threadIdx.x == 0) s.nstart = ld_cg_u32(&ctl->nstart[phase % 3]);
      __syncthreads();
      if (s.nstart == 0u) {  // none in the buckets filled so far
        if (built >= A) break;  // every vertex the BFS owns is settled
        lvl = built;
        continue;
      }
      const int rr = (int)~s.nstart;
      if (profiler && phase + 1 < (u32)kRoundProfile) ctl->round_clk[phase + 1][0] = clock64();
      const int lo = __ldg(a.bptr + (rr - lv0)), hi = (int)ld_cg_u32(a.rcur + (rr - lv0));
      if (LD)
        expand_ld<U, 8>(a, nullptr, 0, 0, lo, (u32)(hi - lo), (u32)rr, false, qi, qb, pushed);
      else
        append_bucket<U>(a, rr, lo, hi, qi, qb, mylow);
      // this round left no unsettled list: a bottom-up round after it starts
      // from every vertex the loop owns
      pulling = false;
      nlvl = rr;
    }
    if (profiler && phase + 1 < (u32)kRoundProfile) ctl->round_clk[phase + 1][1] = clock64();
    post_cta_min<kTrack>(a, s, mylow);
    grid_barrier<kTrack>(a, gen, (u32)qi, lv0, nlvl + 1 <= A ? nlvl + 1 : -1, s);
    if (!LD && defer && !s.stop && (u32)s.next_rest) {  // pushes and put-off scans are listed
      const u64 first_low = s.next_minlow;
      pull_rest<U>(a, (u32)(s.next_rest >> 32), (u32)s.next_rest, lvl, stop_low, phase % 3, qi, qb,
                   mylow, s_floor);
      post_cta_min<kTrack>(a, s, mylow);
      grid_barrier<kTrack>(a, gen, (u32)qi, lv0, nlvl + 1 <= A ? nlvl + 1 : -1, s);
      // the CTAs compared what they posted before with the minimum of the first pass: it
      // stands for them all
      if (kTrack && profiler) note_tie(a, 0, first_low, s.next_minlow);
    }
    ++phase;
    lvl = nlvl;
    if (profiler && phase < (u32)kRoundProfile) {
      ctl->round_clk[phase][2] = clock64();
      ctl->round_kind[phase] = Q == 0 ? kRoundSkip : (pulling ? kRoundPull : kRoundPush);
    }
  }
  if (LD) {  // every thread's offered arcs (the estimate above is not a count) and expansions
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      pushed += __shfl_xor_sync(kFull, pushed, o);
      expanded += __shfl_xor_sync(kFull, expanded, o);
    }
    if ((threadIdx.x & 31) == 0 && pushed) atomicAdd(&ctl->push_arcs, pushed);
    if ((threadIdx.x & 31) == 0 && expanded) atomicAdd(&ctl->items, expanded);
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    ctl->pull_rounds = pulls;
    if (!LD) atomicAdd(&ctl->push_arcs, push_arcs);
    ctl->rounds = phase;
    ctl->last_level = lvl - lv0;
    atomicAdd(&ctl->items, windowed ? items : settled);
    ctl->edges = edges;
    ctl->windows = nwin;
    ctl->overflowed = overflowed;
  }
}

}  // namespace

size_t bfs_smem_bytes() { return sizeof(Smem); }

namespace {
size_t bfs_smem(bool u, int per_sm, bool ld) {
  return sizeof(Smem) + (ld ? lq_extra(per_sm) : 0) + (u ? 3 * kSmemMembers * sizeof(u64) : 0);
}

const void* bfs_kernel(bool u, int per_sm, bool ld) {
  if (ld) {
    if (u) return per_sm >= 2 ? (const void*)k_bfs<true, 2, true> : (const void*)k_bfs<true, 1, true>;
    return per_sm >= 2 ? (const void*)k_bfs<false, 2, true> : (const void*)k_bfs<false, 1, true>;
  }
  if (u) return per_sm >= 2 ? (const void*)k_bfs<true, 2, false> : (const void*)k_bfs<true, 1, false>;
  return per_sm >= 2 ? (const void*)k_bfs<false, 2, false> : (const void*)k_bfs<false, 1, false>;
}
}  // namespace

int bfs_grid_size(int num_sms, int* blocks_per_sm) {
  static bool attr_set[64] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) == cudaSuccess && dev >= 0 && dev < 64 && !attr_set[dev]) {
    for (int u = 0; u < 2; ++u)
      for (int p = 1; p <= 2; ++p)
        for (int ld = 0; ld < 2; ++ld)
          cudaFuncSetAttribute(bfs_kernel(u != 0, p, ld != 0),
                               cudaFuncAttributeMaxDynamicSharedMemorySize,
                               (int)bfs_smem(u != 0, p, ld != 0));
    attr_set[dev] = true;
  }
  // the most CTAs per SM (1 or 2) that every instance built for it reaches
  int per_sm = 2;
  for (int u = 0; u < 2; ++u)
    for (int p = 1; p <= 2; ++p)
      for (int ld = 0; ld < 2; ++ld) {
        int got = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&got, bfs_kernel(u != 0, p, ld != 0),
                                                          kBfsThreads, bfs_smem(u != 0, p, ld != 0)) !=
            cudaSuccess)
          return -1;
        if (got < 1) return -1;
        if (got < p) per_sm = min(per_sm, got);
      }
  *blocks_per_sm = per_sm;
  return per_sm * num_sms;
}

int launch_bfs(const BfsArgs& a, int grid, int per_sm, cudaStream_t s, cudaError_t* err) {
  BfsArgs copy = a;
  void* args[] = {&copy};
  *err = cudaLaunchCooperativeKernel(bfs_kernel(a.mlow != nullptr, per_sm, a.low_degree != 0),
                                     dim3(grid),
                                     dim3(kBfsThreads), args,
                                     bfs_smem(a.mlow != nullptr, per_sm, a.low_degree != 0), s);
  return *err == cudaSuccess ? 1 : -1;
}

}  // namespace ldd
