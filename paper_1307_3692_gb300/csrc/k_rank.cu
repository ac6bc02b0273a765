// Start keys of the delayed-start BFS (Section 4 of Miller, Peng, Xu 2013).
//
//  1. split (Algorithm 1 step 2, Section 4): a_u = floor(delta_u),
//     f_u = delta_u - a_u (exact in FP64), A = max a_u = floor(delta_max).
//  2. tie-break inside a level (Section 4): larger f_u first, then smaller u.
//  3. keys (KeyFmt in ldd_internal.cuh): u's own start label.
//  4. start buckets (Section 4: the super-source edge of length L is looked at
//     when the frontier reaches distance L): the vertices the BFS handles,
//     grouped by start round R_u = A - a_u (any order inside a group).
//
// Direct keys (the usual path, k_direct): level, the leading bits of f_u and u
// in one word, from one pass over the shifts that also counts the floors; an
// exclusive scan of the counts gives the buckets' offsets (bptr).  The round
// loop fills the buckets as it reaches them, with the vertices nobody has
// claimed by then, which are few: bmax, the largest floor of every kMaxBlock
// vertices, lets it pass over the others.
//
// Ranked keys (shifts whose codes tie too often, or levels and ids too wide for
// a code): a stable LSD radix sort of the order-preserving bits of f (8
// "onesweep" passes of 8 bits) over all vertices gives the rank; the start
// buckets are a counting sort by R_u (histogram while the keys are built, an
// exclusive scan that is bptr, and a scatter in which each CTA reserves its
// range of every group with one atomic).
//
// Batches (disjoint unions of member graphs, k_union.cu): every member's
// floors are lifted by one integer, lift_s = max_t A_t - A_s, so that each
// member's own largest shift starts at round 0 and the members' rounds run in
// step.  A constant added to every level of one member changes no comparison
// inside that member, and members never compete.
#include <algorithm>

#include "ldd_internal.cuh"

namespace ldd {

namespace {

constexpr u32 kFull = 0xffffffffu;
constexpr int kScanThreads = 256;
constexpr int kScanIpt = 16;
constexpr int kScanTile = kScanThreads * kScanIpt;
constexpr u32 kRBins = 4096;                  // start rounds counted in shared memory
constexpr int kRChunk = 16;                   // vertices per thread in the start-bucket scatter

__device__ __forceinline__ bool failed(const Control* ctl) {
  return *(volatile const u32*)&ctl->err != 0u;
}

// Adds one count per valid lane to sh[digit]: one atomic when the warp agrees.
__device__ __forceinline__ void hist_add(u32* sh, u32 digit, bool valid, u32 lane) {
  const u32 act = __ballot_sync(kFull, valid);
  if (act == 0) return;
  const int first = __ffs(act) - 1;
  const u32 d0 = __shfl_sync(kFull, digit, first);
  if (__all_sync(kFull, !valid || digit == d0)) {
    if ((int)lane == first) atomicAdd(&sh[d0], (u32)__popc(act));
  } else if (valid) {
    atomicAdd(&sh[digit], 1u);
  }
}

__device__ __forceinline__ void finish_split(u32 err, int amax, Control* ctl) {
  __shared__ int s_amax;
  __shared__ u32 s_err;
  if (threadIdx.x == 0) {
    s_amax = 0;
    s_err = 0;
  }
  __syncthreads();
  if (err) atomicOr(&s_err, err);
  atomicMax(&s_amax, amax);
  __syncthreads();
  if (threadIdx.x == 0) {
    if (s_err) atomicOr(&ctl->err, s_err);
    atomicMax(&ctl->A, s_amax);
  }
}

// ---------------------------------------------------------------- direct keys
// The only pass over the shifts (vertices u0 .. n-1 per launch; one launch per
// chunk while the shifts are still arriving, u0 a multiple of kMaxBlock): every
// vertex's direct key, the counts of the floors among the vertices the BFS
// handles (acnt; the start-round histogram in reverse order, all zero on
// entry), and bmax.  A warp takes kMaxBlock consecutive vertices per step, four
// per lane with all loads first.  In a union the shifts are in the caller's
// layout (a 32-vertex word belongs to one member) and the id is the vertex's
// place in its member; pads get no key.  Errors: bad shifts, a floor beyond the
// level field (kErrLevelCap) or beyond the count table.
//
// Bound by memory: 8 bytes read and 8 written per vertex.  Ranks by a bucket
// sort of the fractions (16-byte records scattered by bucket, ranked in shared
// memory, keys and full start buckets scattered again) were bound by their
// sectors.  Keys and buckets, before and now: 256^3 grid 1236 -> 149 us, R-MAT
// 22 145-168 -> 32-42 us, 64 copies of R-MAT 20 as a union 3700 -> 410 us (and
// its lifts 1300 -> 200), 1000^2 grid 81 -> 32 us.
//
// Then bound by instruction issue (119 per 32 vertices of a union, issue slots 55
// % busy at 2.5 TB/s): the split works on one fixed-point word, the floors are
// counted without grouping equal ones, and a warp whose vertices belong to one
// member (nearly all) reads the member's offsets once: 64 copies of R-MAT 20 408 -> 237 us (and the
// lifts' pass alike), 256^3 grid 149 -> 73 us, R-MAT 22 32-42 -> 28-36 us.
constexpr int kDirectIpt = kMaxBlock / 32;

template <bool U>
__global__ void __launch_bounds__(256) k_direct(const double* __restrict__ delta,
                                                const u32* __restrict__ excl, u32 u0, u32 n,
                                                KeyFmt f, u64* __restrict__ key, u32* acnt,
                                                u32 cap, u32* __restrict__ bmax,
                                                const u32* __restrict__ wmem,
                                                const u32* __restrict__ voff,
                                                const u32* __restrict__ ooff,
                                                const int* __restrict__ lift, Control* ctl) {
  __shared__ u32 sh[kRBins];
  __shared__ int s_ab;
  const u32 tid = threadIdx.x, lane = tid & 31;
  for (u32 i = tid; i < kRBins; i += blockDim.x) sh[i] = 0;
  if (tid == 0) s_ab = 0;
  __syncthreads();
  u32 amax = 0, err = 0, ab = 0;  // ab: largest handled floor of this warp's blocks, plus one
  const u32 code_shift = 32 - f.cb;
  const u32 stride = gridDim.x * (blockDim.x / 32) * kMaxBlock;
  for (u32 wb = u0 + (blockIdx.x * (blockDim.x / 32) + (tid >> 5)) * kMaxBlock; wb < n;
       wb += stride) {
    double d[kDirectIpt];
    u32 id[kDirectIpt], ex[kDirectIpt], lf[kDirectIpt];
    bool live[kDirectIpt];
    u32 m0 = 0, m1 = 0;  // the members of the first and last word
    if (U) {
      m0 = __ldg(wmem + (wb >> 5));
      m1 = __ldg(wmem + (min(wb + kMaxBlock, n) - 1) / 32);
    }
    if (!U || m0 == m1) {
      u32 base = 0, at = 0, size = n, lift0 = 0;
      if (U) {
        base = __ldg(voff + m0);
        at = __ldg(ooff + m0);
        size = __ldg(ooff + m0 + 1) - at;
        lift0 = (u32)__ldg(lift + m0);
      }
#pragma unroll
      for (int k = 0; k < kDirectIpt; ++k) {
        id[k] = wb + (u32)k * 32 + lane - base;
        live[k] = id[k] < size;  // else a pad, or past the end
        if (!U) live[k] = live[k] && id[k] < n;
        lf[k] = lift0;
        d[k] = live[k] ? __ldcs(delta + at + id[k]) : 0.0;
      }
    } else {
#pragma unroll
      for (int k = 0; k < kDirectIpt; ++k) {
        const u32 u = wb + (u32)k * 32 + lane;
        live[k] = u < n;
        id[k] = lf[k] = 0;
        d[k] = 0.0;
        if (live[k]) {
          const u32 m = __ldg(wmem + (u >> 5)), o = __ldg(ooff + m);
          id[k] = u - __ldg(voff + m);
          live[k] = o + id[k] < __ldg(ooff + m + 1);
          lf[k] = (u32)__ldg(lift + m);
          if (live[k]) d[k] = __ldcs(delta + o + id[k]);
        }
      }
    }
#pragma unroll
    for (int k = 0; k < kDirectIpt; ++k) {
      const u32 word = (wb >> 5) + (u32)k;
      ex[k] = word * 32 < n ? __ldg(excl + word) : 0xffffffffu;
    }
    u32 top = 0;
#pragma unroll
    for (int k = 0; k < kDirectIpt; ++k) {
      bool ok;
      const u64 x = fixed_shift(d[k], &ok);
      if (!ok) {
        int a;
        u64 fb;
        split_bits(d[k], err, a, fb);
        continue;
      }
      if (!live[k]) continue;
      const u32 a = (u32)(x >> 32) + lf[k];
      amax = max(amax, a);
      key[wb + (u32)k * 32 + lane] =
          level_key(f, f.cap - a) | ((u64)(~(u32)x >> code_shift) << f.ib) | id[k];
      if ((ex[k] >> lane) & 1u) continue;
      top = max(top, a + 1u);
      if (a < kRBins) atomicAdd(&sh[a], 1u);
      else if ((u64)a + 2 <= cap) atomicAdd(acnt + a, 1u);
      else err |= kErrBucketCap;
    }
    top = __reduce_max_sync(kFull, top);
    ab = max(ab, top);
    if (lane == 0) bmax[wb / kMaxBlock] = top;
  }
  if (amax > f.cap) err |= kErrLevelCap;
  if (lane == 0 && ab) atomicMax(&s_ab, (int)(ab - 1));
  __syncthreads();
  for (u32 i = tid; i < kRBins; i += blockDim.x)
    if (sh[i] && (u64)i + 2 <= cap) atomicAdd(acnt + i, sh[i]);
    else if (sh[i]) err |= kErrBucketCap;
  if (tid == 0 && s_ab) atomicMax(&ctl->Ab, s_ab);
  finish_split(err, (int)min(amax, 0x7fffffffu), ctl);
}

// ---------------------------------------------------------------- exact path
__global__ void __launch_bounds__(256) k_split64(const double* __restrict__ delta, u32 n,
                                                 int* __restrict__ a_out, u64* __restrict__ kout,
                                                 u32* __restrict__ vout,
                                                 const u32* __restrict__ wmem,
                                                 const int* __restrict__ lift, Control* ctl) {
  __shared__ u32 sh[kFracDigits][256];
  const u32 tid = threadIdx.x, lane = tid & 31;
  for (u32 i = tid; i < kFracDigits * 256; i += blockDim.x) (&sh[0][0])[i] = 0;
  __syncthreads();
  int amax = 0;
  u32 err = 0;
  const u32 stride = gridDim.x * blockDim.x;
  for (u32 base = blockIdx.x * blockDim.x + (tid & ~31u); base < n; base += stride) {
    const u32 idx = base + lane;
    const bool valid = idx < n;
    u64 key = 0;
    if (valid) {
      int a;
      u64 fb;
      split_bits(delta[idx], err, a, fb);
      if (lift) a += __ldg(lift + __ldg(wmem + (idx >> 5)));
      key = ~fb;  // ascending key: f descending
      a_out[idx] = a;
      kout[idx] = key;
      vout[idx] = idx;
      amax = max(amax, a);
    }
#pragma unroll
    for (int dg = 0; dg < kFracDigits; ++dg)
      hist_add(sh[dg], (u32)(key >> (8 * dg)) & 255u, valid, lane);
  }
  __syncthreads();
  for (u32 i = tid; i < kFracDigits * 256; i += blockDim.x) {
    const u32 c = (&sh[0][0])[i];
    if (c) atomicAdd(&(&ctl->hist_f[0][0])[i], c);
  }
  finish_split(err, amax, ctl);
}

// Exclusive offsets of every digit histogram; a digit whose keys all share
// one value needs no pass.  One CTA of 256 threads.
__global__ void __launch_bounds__(256) k_scan_digits(const u32* __restrict__ hist,
                                                     u32* __restrict__ off, u32* mask, int ndig,
                                                     u32 n) {
  __shared__ u32 s_warp[8];
  __shared__ int s_const;
  const int t = threadIdx.x, lane = t & 31, w = t >> 5;
  u32 m = 0;
  for (int d = 0; d < ndig; ++d) {
    const u32 h = hist[d * 256 + t];
    if (t == 0) s_const = 0;
    __syncthreads();
    if (h == n) s_const = 1;
    u32 x = h;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const u32 y = __shfl_up_sync(kFull, x, o);
      if (lane >= o) x += y;
    }
    if (lane == 31) s_warp[w] = x;
    __syncthreads();
    u32 wbase = 0;
    for (int i = 0; i < w; ++i) wbase += s_warp[i];
    off[d * 256 + t] = wbase + x - h;
    if (!s_const) m |= 1u << d;
    __syncthreads();
  }
  if (t == 0) *mask = (n == 0) ? 0u : m;
}

constexpr int kSortWarps = kSortThreads / 32;

struct SortSmem {
  u64 keys[kSortTile];         // the tile, staged in sorted order for the write-out
  u32 vals[kSortTile];
  u32 whist[kSortWarps][256];  // per-warp digit counts, then per-warp offsets
  u32 tile_excl[256];          // start of each digit's run inside the tile
  u32 base[256];               // global start of this tile's run of each digit
  u32 wsum[kSortWarps];
  u32 tile;
  u32 bad;
};

// One stable LSD pass on digit `pass` (bits shift..shift+7) of 64-bit keys.
// Buffers are a ping-pong pair; the input side is the parity of the passes run
// before.  Each 4096-key tile ranks its keys per digit in shared memory with
// warp match, finds its global offsets by decoupled look-back over the
// preceding tiles, and writes each digit's run out contiguously.
__global__ void __launch_bounds__(kSortThreads) k_onesweep(
    u64* __restrict__ k0, u32* __restrict__ v0, u64* __restrict__ k1, u32* __restrict__ v1, u32 n,
    int pass, int shift, const u32* __restrict__ mask_ptr, const u32* __restrict__ digit_off,
    u64* __restrict__ status, u32* __restrict__ tile_ctr, u32 epoch, u32* err, u32 spin_limit) {
  const u32 mask = *mask_ptr;
  if (!((mask >> pass) & 1u) || *(volatile u32*)err != 0u) return;
  const int par = __popc(mask & ((1u << pass) - 1u)) & 1;
  const u64* kin = par ? k1 : k0;
  const u32* vin = par ? v1 : v0;
  u64* kout = par ? k0 : k1;
  u32* vout = par ? v0 : v1;

  extern __shared__ __align__(16) unsigned char sort_smem_raw[];
  SortSmem& sm = *reinterpret_cast<SortSmem*>(sort_smem_raw);
  const u32 tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (tid == 0) {
    sm.tile = atomicAdd(tile_ctr, 1u);
    sm.bad = 0;
  }
  for (u32 i = tid; i < kSortWarps * 256; i += kSortThreads) (&sm.whist[0][0])[i] = 0;
  __syncthreads();
  const u32 tile = sm.tile;
  const u32 tile0 = tile * kSortTile;
  const u32 base = tile0 + warp * (32 * kSortIpt);

  u64 key[kSortIpt];
  u32 val[kSortIpt];
  u32 rk[kSortIpt];
#pragma unroll
  for (int k = 0; k < kSortIpt; ++k) {
    const u32 idx = base + k * 32 + lane;
    key[k] = (idx < n) ? kin[idx] : 0ull;
    val[k] = (idx < n) ? vin[idx] : 0u;
  }
  const u32 lt = lanemask_lt();
#pragma unroll
  for (int k = 0; k < kSortIpt; ++k) {
    const u32 idx = base + k * 32 + lane;
    const bool valid = idx < n;
    const u32 dg = (u32)(key[k] >> shift) & 255u;
    const u32 d = valid ? dg : 256u + lane;
    const u32 peers = __match_any_sync(kFull, d);
    const u32 cnt = valid ? sm.whist[warp][dg] : 0u;
    rk[k] = cnt + __popc(peers & lt);
    __syncwarp();
    if (valid && (peers & lt) == 0) sm.whist[warp][dg] = cnt + __popc(peers);
    __syncwarp();
  }
  __syncthreads();
  const u32 dg = tid;  // thread tid owns digit tid
  u32 run = 0;
#pragma unroll
  for (int w = 0; w < kSortWarps; ++w) {
    const u32 c = sm.whist[w][dg];
    sm.whist[w][dg] = run;
    run += c;
  }
  u64* mine = status + (u64)tile * 256 + dg;
  const u64 tag = (u64)epoch << 32;
  if (tile == 0) st_volatile_u64(mine, tag | (2ull << 30) | run);
  else st_volatile_u64(mine, tag | (1ull << 30) | run);
  {
    u32 x = run;  // exclusive scan of the digit totals over the tile
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const u32 y = __shfl_up_sync(kFull, x, o);
      if (lane >= (u32)o) x += y;
    }
    if (lane == 31) sm.wsum[warp] = x;
    __syncthreads();
    u32 pre = 0;
    for (u32 w = 0; w < warp; ++w) pre += sm.wsum[w];
    sm.tile_excl[dg] = pre + x - run;
  }
  u32 excl = 0;
  if (tile > 0) {
    int p = (int)tile - 1;
    u32 spins = 0;
    while (p >= 0) {
      const u64 sv = ld_volatile_u64(status + (u64)p * 256 + dg);
      if ((u32)(sv >> 32) != epoch) {
        if (++spins > spin_limit) {
          atomicOr(err, kErrTimeout);
          sm.bad = 1;
          break;
        }
        if (spins > 16) __nanosleep(64);
        continue;
      }
      excl += (u32)sv & 0x3fffffffu;
      if ((((u32)sv) >> 30) == 2u) break;
      --p;
    }
    st_volatile_u64(mine, tag | (2ull << 30) | (excl + run));
  }
  sm.base[dg] = digit_off[dg] + excl;
  __syncthreads();
  if (sm.bad) return;  // offsets unknown: write nothing
#pragma unroll
  for (int k = 0; k < kSortIpt; ++k) {
    const u32 idx = base + k * 32 + lane;
    if (idx < n) {
      const u32 d = (u32)(key[k] >> shift) & 255u;
      const u32 local = sm.tile_excl[d] + sm.whist[warp][d] + rk[k];
      sm.keys[local] = key[k];
      sm.vals[local] = val[k];
    }
  }
  __syncthreads();
  const u32 tile_n = min((u32)kSortTile, n - tile0);
  for (u32 i = tid; i < tile_n; i += kSortThreads) {
    const u64 kv = sm.keys[i];
    const u32 d = (u32)(kv >> shift) & 255u;
    const u32 pos = sm.base[d] + (i - sm.tile_excl[d]);
    if (pos < n) {
      kout[pos] = kv;
      vout[pos] = sm.vals[i];
    }
  }
}

// order[p] = u and rank[u] = p for the sorted fraction order (exact path).
__global__ void __launch_bounds__(256) k_rank_scatter(const u32* __restrict__ v0,
                                                      const u32* __restrict__ v1, Control* ctl,
                                                      u32 n, u32* __restrict__ order,
                                                      u32* __restrict__ rank) {
  if (failed(ctl)) return;
  const u32* vals = (__popc(ctl->mask_f) & 1u) ? v1 : v0;
  const u32 stride = gridDim.x * blockDim.x;
  for (u32 p = blockIdx.x * blockDim.x + threadIdx.x; p < n; p += stride) {
    u32 u = vals[p];
    if (u >= n) {  // cannot happen for a permutation; never index with it
      atomicOr(&ctl->err, kErrInternal);
      u = 0;
    }
    order[p] = u;
    rank[u] = p;
  }
}

// ---------------------------------------------------------------- device scan
// In-place exclusive scan of data[0 .. len), single pass with decoupled
// look-back over 4096-element tiles.  len = A + 2 when len_from_A (the
// start-round histogram), else len_host.  With rev_src (direct keys), A is the
// largest floor among the vertices the BFS handles, the input is the floor
// histogram read in reverse, data[r] = rev_src[A - r] for
// r = 0 .. A and 0 for r = A + 1, and rev_src is cleared on the way (all zero
// for the next decomposition); a table of fewer than A + 2 entries (cap) sets
// kErrBucketCap.  Optionally copies the result to copy[].  Tiles take tickets in
// order, so every tile's predecessors are running or done; every wait is bounded
// (spin_limit polls, then kErrTimeout).  One warp looks back over 32 predecessor
// tiles at a time.
// stall = 1 makes tile 0 wait, like the others, on a predecessor that does not
// exist, so that every look-back runs out of polls (tests of the timeout path).
__global__ void __launch_bounds__(kScanThreads) k_scan_excl(u32* data, u32* copy, u32 len_host,
                                                            int len_from_A, u64* __restrict__ status,
                                                            u32 epoch, u32* tile_ctr, u32* rev_src,
                                                            u32 cap, Control* ctl,
                                                            u32 spin_limit, u32 stall) {
  __shared__ u32 s_tile, s_excl, s_bad;
  __shared__ u32 s_wsum[kScanThreads / 32];
  if (failed(ctl)) {
    // an upstream error skips the scan; the floor counts are still cleared, so
    // a decomposition queued behind this one starts from zero counts
    if (rev_src) {
      const u32 end = (u32)min((u64)(u32)ctl->Ab + 1, (u64)cap);
      for (u32 r = blockIdx.x * blockDim.x + threadIdx.x; r < end; r += gridDim.x * blockDim.x)
        rev_src[r] = 0;
    }
    return;
  }
  const u32 tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (rev_src && blockIdx.x == 0 && tid < 3) ctl->minlow[tid] = ~0ull;  // for the round loop
  if (tid == 0) {
    s_tile = atomicAdd(tile_ctr, 1u);
    s_bad = 0;
    s_excl = 0;
  }
  __syncthreads();
  const u32 tile = s_tile;
  const int A = rev_src ? ctl->Ab : ctl->A;
  if (rev_src && (u64)A + 2 > cap) {
    if (tile == 0 && tid == 0) atomicOr(&ctl->err, kErrBucketCap);
    for (u32 r = tile * kScanTile + tid; r < min(cap, (tile + 1) * kScanTile); r += blockDim.x)
      rev_src[r] = 0;  // cleared as above
    return;
  }
  const u32 len = len_from_A ? (u32)A + 2u : len_host;
  const u32 t0 = tile * kScanTile;
  if (t0 >= len) return;  // tiles past the end: no later tile needs them
  const u32 my0 = t0 + tid * kScanIpt;
  u32 v[kScanIpt];
  u32 tot = 0;
#pragma unroll
  for (int i = 0; i < kScanIpt; ++i) {
    const u32 r = my0 + i;
    if (rev_src) {
      v[i] = 0;
      if (r <= (u32)A) {
        v[i] = rev_src[(u32)A - r];
        rev_src[(u32)A - r] = 0;
      }
    } else {
      v[i] = (r < len) ? data[r] : 0u;
    }
    tot += v[i];
  }
  u32 x = tot;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const u32 y = __shfl_up_sync(kFull, x, o);
    if (lane >= (u32)o) x += y;
  }
  if (lane == 31) s_wsum[warp] = x;
  __syncthreads();
  u32 wpre = 0, tile_tot = 0;
  for (u32 w = 0; w < kScanThreads / 32; ++w) {
    if (w < warp) wpre += s_wsum[w];
    tile_tot += s_wsum[w];
  }
  if (warp == 0) {
    const u64 tag = (u64)epoch << 32;
    u64* mine = status + tile;
    if (tile == 0 && !stall) {
      if (lane == 0) st_volatile_u64(mine, tag | (2ull << 30) | tile_tot);
    } else {
      if (lane == 0) st_volatile_u64(mine, tag | (1ull << 30) | tile_tot);
      u32 excl = 0;
      int p = (int)tile - 1;
      u32 spins = 0;
      bool bad = false;
      while (p >= 0 || stall) {
        // lane l looks at tile p - l; "before tile 0" counts as an inclusive
        // prefix of 0 (with stall: as a tile that never reports)
        const int q = p - (int)lane;
        const u64 sv = (q >= 0) ? ld_volatile_u64(status + q) : (stall ? 0ull : (tag | (2ull << 30)));
        const bool ready = (u32)(sv >> 32) == epoch;
        const bool pref = ready && ((((u32)sv) >> 30) == 2u);
        const u32 pmask = __ballot_sync(kFull, pref);
        const u32 limit = pmask ? (u32)(__ffs(pmask) - 1) : 31u;  // lanes 0..limit are needed
        const u32 rmask = __ballot_sync(kFull, ready);
        const u32 need = (limit == 31u) ? kFull : ((2u << limit) - 1u);
        if ((rmask & need) != need) {
          if (++spins > spin_limit) {
            bad = true;
            break;
          }
          if (spins > 16) __nanosleep(64);
          continue;
        }
        u32 val = (lane <= limit) ? ((u32)sv & 0x3fffffffu) : 0u;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) val += __shfl_xor_sync(kFull, val, o);
        excl += val;
        if (pmask) break;
        p -= 32;
      }
      if (lane == 0) {
        if (bad) {
          atomicOr(&ctl->err, kErrTimeout);
          s_bad = 1;
        } else {
          st_volatile_u64(mine, tag | (2ull << 30) | (excl + tile_tot));
        }
        s_excl = excl;
      }
    }
  }
  __syncthreads();
  if (s_bad) return;
  u32 run = s_excl + wpre + x - tot;
#pragma unroll
  for (int i = 0; i < kScanIpt; ++i) {
    if (my0 + i < len) {
      data[my0 + i] = run;
      if (copy) copy[my0 + i] = run;
    }
    run += v[i];
  }
}

// ---------------------------------------------------------------- keys and start buckets
__global__ void __launch_bounds__(256) k_zero_rounds(int* bptr, u32 cap, Control* ctl) {
  if (failed(ctl)) return;
  if ((u64)ctl->A + 2 > cap) {
    if (blockIdx.x == 0 && threadIdx.x == 0) atomicOr(&ctl->err, kErrBucketCap);
    return;
  }
  const u32 len = (u32)ctl->A + 2u;
  for (u32 r = blockIdx.x * blockDim.x + threadIdx.x; r < len; r += gridDim.x * blockDim.x)
    bptr[r] = 0;
}

// In vertex order: key_u = ((A - a_u) << 32) | rank_u, and the count of every
// start round R_u among the vertices the BFS handles (into rcnt).
__global__ void __launch_bounds__(256) k_keys(const int* __restrict__ a,
                                              const u32* __restrict__ rank,
                                              const u32* __restrict__ excl, Control* ctl, u32 n,
                                              u64* __restrict__ key, u32* rcnt) {
  __shared__ u32 sh[kRBins];
  if (failed(ctl)) return;
  const int A = ctl->A;
  const bool small = (u32)A + 1u <= kRBins;
  const u32 tid = threadIdx.x, lane = tid & 31;
  if (small)
    for (u32 i = tid; i <= (u32)A; i += blockDim.x) sh[i] = 0;
  __syncthreads();
  const u32 stride = gridDim.x * blockDim.x;
  for (u32 base = blockIdx.x * blockDim.x + (tid & ~31u); base < n; base += stride) {
    const u32 u = base + lane;
    bool count = false;
    u32 R = 0;
    if (u < n) {
      R = (u32)(A - a[u]);
      key[u] = ((u64)R << 32) | rank[u];
      count = !(excl[u >> 5] >> (u & 31) & 1u);
    }
    const u32 act = __ballot_sync(kFull, count);
    if (act) {
      const u32 peers = __match_any_sync(kFull, count ? R : 0xffffffffu) & act;
      if (count && (peers & lanemask_lt()) == 0) {
        const u32 c = __popc(peers);
        if (small) atomicAdd(&sh[R], c);
        else atomicAdd(rcnt + R, c);
      }
    }
  }
  __syncthreads();
  if (small)
    for (u32 i = tid; i <= (u32)A; i += blockDim.x)
      if (sh[i]) atomicAdd(rcnt + i, sh[i]);
}

// Start-bucket scatter: bv[pos] = u for every vertex the BFS handles.  With few rounds, each CTA counts its chunk in shared memory and
// reserves its range of every group with one atomic; otherwise one atomic per
// warp and round.
__global__ void __launch_bounds__(256) k_rscatter(const int* __restrict__ a,
                                                  const u32* __restrict__ excl, Control* ctl,
                                                  u32 n, u32* cursor, u32* __restrict__ bv) {
  __shared__ u32 s_cnt[kRBins];
  if (failed(ctl)) return;
  const int A = ctl->A;
  const bool small = (u32)A + 1u <= kRBins;
  const u32 tid = threadIdx.x, lane = tid & 31;
  const u32 chunk = blockDim.x * kRChunk;
  for (u32 c0 = blockIdx.x * chunk; c0 < n; c0 += gridDim.x * chunk) {
    if (small) {
      for (u32 i = tid; i <= (u32)A; i += blockDim.x) s_cnt[i] = 0;
      __syncthreads();
    }
    u32 R[kRChunk];
    u32 local[kRChunk];
#pragma unroll
    for (int k = 0; k < kRChunk; ++k) {
      const u32 u = c0 + (u32)k * blockDim.x + tid;
      bool take = false;
      R[k] = 0xffffffffu;
      if (u < n) {
        take = !(excl[u >> 5] >> (u & 31) & 1u);
        if (take) R[k] = (u32)(A - a[u]);
      }
      local[k] = 0;
      const u32 act = __ballot_sync(kFull, take);
      if (act) {
        const u32 peers = __match_any_sync(kFull, R[k]) & act;
        const int leader = take ? __ffs(peers) - 1 : (int)lane;
        u32 got = 0;
        if (take && (int)lane == leader)
          got = small ? atomicAdd(&s_cnt[R[k]], (u32)__popc(peers))
                      : atomicAdd(cursor + R[k], (u32)__popc(peers));
        got = __shfl_sync(kFull, got, leader);
        local[k] = got + __popc(peers & lanemask_lt());
      }
    }
    if (small) {
      __syncthreads();
      for (u32 i = tid; i <= (u32)A; i += blockDim.x) {
        const u32 c = s_cnt[i];
        s_cnt[i] = c ? atomicAdd(cursor + i, c) : 0u;  // this chunk's base in group i
      }
      __syncthreads();
    }
#pragma unroll
    for (int k = 0; k < kRChunk; ++k) {
      const u32 u = c0 + (u32)k * blockDim.x + tid;
      if (R[k] != 0xffffffffu) {
        const u32 pos = (small ? s_cnt[R[k]] : 0u) + local[k];
        if (pos < n) bv[pos] = u;
      }
    }
    if (small) __syncthreads();
  }
}

// ---------------------------------------------------------------- ranked variant
// Section 4: the fractional parts of the shifts only order the vertices of one
// integer level, and a random permutation of the vertices can stand in for
// them.  Input: the integer parts a_u (levels[u] >= 0) and the permutation
// (perm[u] = u's tie-break position, smaller first).  The rank is perm itself;
// order[perm[u]] = u, with a duplicate position detected by the exchange
// (order is all ones on entry).  Bad input sets kErrPermArg.
__global__ void __launch_bounds__(256) k_ranked_split(const int* __restrict__ levels,
                                                      const int* __restrict__ perm, u32 n,
                                                      int* __restrict__ a_out, u32* order,
                                                      Control* ctl) {
  int amax = 0;
  u32 err = 0;
  for (u32 u = blockIdx.x * blockDim.x + threadIdx.x; u < n; u += gridDim.x * blockDim.x) {
    const int a = levels[u];
    const int p = perm[u];
    if (a < 0 || p < 0 || (u32)p >= n) {
      err |= kErrPermArg;
      a_out[u] = 0;
      continue;
    }
    a_out[u] = a;
    amax = max(amax, a);
    if (atomicExch(order + p, u) != 0xffffffffu) err |= kErrPermArg;  // p taken twice
  }
  finish_split(err, amax, ctl);
}

u32 grid_stride_blocks(u32 n, int num_sms) {
  return (u32)max(1ll, min((long long)(n + 255) / 256, (long long)num_sms * 8));
}

// CTAs of a k_direct instance resident on one SM: its grid is one full wave.
int direct_blocks_per_sm(bool u) {
  static int per_sm[2][64] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 4;
  int& b = per_sm[u ? 1 : 0][dev];
  if (b <= 0) {
    const void* fn = u ? (const void*)k_direct<true> : (const void*)k_direct<false>;
    int got = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&got, fn, 256, 0) != cudaSuccess || got < 1) {
      cudaGetLastError();
      got = 4;
    }
    b = got;
  }
  return b;
}

void allow_sort_smem() {
  static bool done[64] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return;
  if (!done[dev]) {
    cudaFuncSetAttribute(k_onesweep, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)sizeof(SortSmem));
    done[dev] = true;
  }
}

}  // namespace

size_t scan_status_words(u32 bptr_cap) {
  return ((size_t)bptr_cap + kScanTile - 1) / kScanTile;
}

int launch_rank_and_buckets(const RankBufs& r, bool exact64, cudaStream_t s,
                            const ShiftChunks* chunks) {
  const u32 n = r.n;
  Control* ctl = r.ctl;
  const u32 gs = grid_stride_blocks(n, r.num_sms);
  int launches = 0;
  const u32 rtiles = (r.bptr_cap + kScanTile - 1) / kScanTile;
  u32* rcnt = reinterpret_cast<u32*>(r.bptr);
  if (!exact64) {
    // keys and floor counts, then the start buckets' offsets
    if (r.acnt_dirty) cudaMemsetAsync(r.acnt, 0, (size_t)r.bptr_cap * 4, s);
    const int nchunk = chunks ? chunks->n : 0;
    const bool u = r.wmem != nullptr;
    u32 lo = 0;
    for (int c = 0; c <= nchunk; ++c) {
      // chunk c is vertices [lo, hi), complete once its event has fired
      const u32 hi = c < nchunk ? std::min(chunks->end[c], n) : n;
      if (c < nchunk) cudaStreamWaitEvent(s, chunks->ev[c], 0);
      if (hi <= lo) continue;
      const u32 per_cta = 8 * kMaxBlock;
      const u32 grid = (u32)min(((long long)(hi - lo) + per_cta - 1) / per_cta,
                                (long long)r.num_sms * direct_blocks_per_sm(u));
      if (u)
        k_direct<true><<<grid, 256, 0, s>>>(r.shift, r.excl, lo, hi, r.f, r.key, r.acnt,
                                            r.bptr_cap, r.bmax, r.wmem, r.voff, r.ooff, r.lift,
                                            ctl);
      else
        k_direct<false><<<grid, 256, 0, s>>>(r.shift, r.excl, lo, hi, r.f, r.key, r.acnt,
                                             r.bptr_cap, r.bmax, nullptr, nullptr, nullptr,
                                             nullptr, ctl);
      ++launches;
      lo = hi;
    }
    // no floor exceeds f.cap, so neither do the rounds
    const u32 tiles = (u32)((std::min<u64>(r.bptr_cap, (u64)r.f.cap + 2) + kScanTile - 1) /
                            kScanTile);
    k_scan_excl<<<tiles, kScanThreads, 0, s>>>(rcnt, r.rcur, 0, 1, r.status, ++(*r.epoch),
                                               &ctl->tile_ctr[1], r.acnt, r.bptr_cap, ctl,
                                               r.lookback_limit, r.stall_lookback);
    return launches + 1;
  }
  // exact path: stable LSD radix sort of all fractions, then keys and the
  // start-round counting sort (groups in any order inside)
  u32* rank = reinterpret_cast<u32*>(r.k1) + n;  // k1 holds 2 max(n, 64) 32-bit words
  if (chunks)
    for (int c = 0; c < chunks->n; ++c) cudaStreamWaitEvent(s, chunks->ev[c], 0);
  allow_sort_smem();
  k_split64<<<gs, 256, 0, s>>>(r.shift, n, r.a, r.k0, r.v0, r.wmem, r.lift, ctl);
  k_scan_digits<<<1, 256, 0, s>>>(&ctl->hist_f[0][0], &ctl->off_f[0][0], &ctl->mask_f,
                                  kFracDigits, n);
  launches += 2;
  const u32 ntiles = (n + kSortTile - 1) / kSortTile;
  for (int d = 0; d < kFracDigits; ++d) {
    k_onesweep<<<ntiles, kSortThreads, sizeof(SortSmem), s>>>(
        r.k0, r.v0, r.k1, r.v1, n, d, 8 * d, &ctl->mask_f, ctl->off_f[d], r.status,
        &ctl->tile_ctr[2 + d], ++(*r.epoch), &ctl->err, r.lookback_limit);
    ++launches;
  }
  k_rank_scatter<<<gs, 256, 0, s>>>(r.v0, r.v1, ctl, n, r.order, rank);
  k_zero_rounds<<<grid_stride_blocks(r.bptr_cap, r.num_sms), 256, 0, s>>>(r.bptr, r.bptr_cap,
                                                                            ctl);
  k_keys<<<gs, 256, 0, s>>>(r.a, rank, r.excl, ctl, n, r.key, rcnt);
  k_scan_excl<<<rtiles, kScanThreads, 0, s>>>(rcnt, r.rcur, 0, 1, r.status, ++(*r.epoch),
                                               &ctl->tile_ctr[1], nullptr, 0, ctl,
                                               r.lookback_limit, r.stall_lookback);
  k_rscatter<<<(u32)min((long long)(n + 256 * kRChunk - 1) / (256 * kRChunk),
                        (long long)r.num_sms * 8),
               256, 0, s>>>(r.a, r.excl, ctl, n, r.rcur, r.v0);
  return launches + 5;
}

int launch_exclusive_scan(u32* data, u32 len, u64* status, u32* epoch, u32* tile_ctr,
                          Control* ctl, u32 spin_limit, cudaStream_t s, u32* copy) {
  const u32 tiles = (len + kScanTile - 1) / kScanTile;
  if (tiles == 0) return 0;
  k_scan_excl<<<tiles, kScanThreads, 0, s>>>(data, copy, len, 0, status, ++(*epoch), tile_ctr,
                                             nullptr, 0, ctl, spin_limit, 0);
  return 1;
}

int launch_ranked_and_buckets(const RankBufs& r, const int* levels, const int* perm,
                              cudaStream_t s) {
  const u32 n = r.n;
  Control* ctl = r.ctl;
  const u32 gs = grid_stride_blocks(n, r.num_sms);
  const u32 rtiles = (r.bptr_cap + kScanTile - 1) / kScanTile;
  u32* rcnt = reinterpret_cast<u32*>(r.bptr);
  const u32* rank = reinterpret_cast<const u32*>(perm);
  cudaMemsetAsync(r.order, 0xff, (size_t)n * 4, s);
  k_ranked_split<<<gs, 256, 0, s>>>(levels, perm, n, r.a, r.order, ctl);
  k_zero_rounds<<<grid_stride_blocks(r.bptr_cap, r.num_sms), 256, 0, s>>>(r.bptr, r.bptr_cap,
                                                                            ctl);
  k_keys<<<gs, 256, 0, s>>>(r.a, rank, r.excl, ctl, n, r.key, rcnt);
  k_scan_excl<<<rtiles, kScanThreads, 0, s>>>(rcnt, r.rcur, 0, 1, r.status, ++(*r.epoch),
                                               &ctl->tile_ctr[1], nullptr, 0, ctl,
                                               r.lookback_limit, r.stall_lookback);
  k_rscatter<<<(u32)min((long long)(n + 256 * kRChunk - 1) / (256 * kRChunk),
                        (long long)r.num_sms * 8),
               256, 0, s>>>(r.a, r.excl, ctl, n, r.rcur, r.v0);
  return 5;
}

}  // namespace ldd
