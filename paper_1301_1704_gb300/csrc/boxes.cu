// boxes.cu -- non-empty boxes, bookmarks, parents and children at every
// level (Alg. 3, Sec. 2.2), from keys sorted by their top 3*Lb bits, fused
// with the finishing sort of the point order inside each box.
//
// Alg. 3 scans a dense histogram of all 8^lmax boxes.  Here nothing dense is
// built: sorted point i opens a box at level l exactly when its level-l key
// differs from that of point i-1, i.e. for every l >= d_i where d_i is fixed
// by the highest bit in which the two keys differ.  One pass over the sorted
// keys therefore flags the box starts of all levels at once, and a
// multi-level prefix sum (one decoupled look-back chain per level) gives each
// start its rank at every level it opens.  The rank of a start is the box's
// index in SrcNonEmptyBoxIndex / RecvNonEmptyBoxIdx and its position is the
// bookmark.
#include "fmm_internal.cuh"

namespace fmm {

uint32_t boxes_tiles(uint32_t n) {
  const uint64_t t = ((uint64_t)n + kBoxTile - 1) / kBoxTile;
  return t == 0 ? 1u : (uint32_t)t;
}

constexpr int kWin = kBoxTile + kBoxHalo;  // points held per tile
// Shared memory: keys [kWin + 2] (u64: the two points before the tile, then
// the window, so that a bulk copy can start 16-byte aligned), then the
// per-point first differing levels [kWin] (u8, 16-byte aligned for vector
// reads), then the indices [kWin] (u32).
constexpr size_t kBoxDdOff = (sizeof(uint64_t) * (kWin + 2) + 15) & ~(size_t)15;
constexpr size_t kBoxValOff = kBoxDdOff + kWin;
constexpr size_t kBoxSmem = kBoxValOff + sizeof(uint32_t) * kWin;
static_assert(kWin % 16 == 0 && kBoxValOff % 16 == 0, "shared layout alignment");

// First level at which a key differs from the key before it (22: equal keys;
// the keys use bits 0..62, level l owns bits 63-3l .. 65-3l).
__device__ __forceinline__ uint32_t first_diff_level(uint64_t a, uint64_t b) {
  const uint64_t x = a ^ b;
  return x == 0 ? 22u : (uint32_t)((2 + __clzll((long long)x)) / 3);
}

// (Four blocks an SM, which shared memory allows: with three, 512 sets of 7.4e7 points
// take 788 us for 737.)
__global__ void __launch_bounds__(kBoxThreads, 4) finish_boxes_kernel(const Seg* __restrict__ segs,
                                                                   const Slot* __restrict__ slots,
                                                                   uint32_t nslots, DevStatus* st,
                                                                   uint64_t wait_ns) {
  constexpr int W = kBoxThreads / 32;
  __shared__ uint32_t s_tile, s_abort, s_ttot, s_texcl;
  __shared__ uint32_t s_wtot[W];
  __shared__ __align__(8) uint64_t s_bar;
  extern __shared__ __align__(16) uint64_t s_key[];  // s_key[j + 2] = key of point t0 + j
  uint64_t* const sk = s_key + 1;                     // sk[j + 1] = key of point t0 + j
  uint8_t* s_dd = reinterpret_cast<uint8_t*>(s_key) + kBoxDdOff;  // first differing level
  uint32_t* s_val = reinterpret_cast<uint32_t*>(reinterpret_cast<uint8_t*>(s_key) + kBoxValOff);

  grid_wait(segs, slots);
  const Seg& sg = segs[slots[find_slot(slots, nslots, blockIdx.x)].seg];
  const uint64_t* __restrict__ keys = sg.skeys;
  const uint32_t* __restrict__ vals = sg.svals;
  const uint32_t n = sg.n;
  const int Lb = sg.Lb, Ls = sg.Ls;
  const LevelArrays& lv = sg.lv;
  uint32_t* __restrict__ perm = sg.perm;
  uint64_t* status = sg.bstatus;
  const uint32_t ntiles = sg.btiles;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (threadIdx.x == 0) {
    s_tile = atomicAdd(&sg.tickets[0], 1u);
    s_abort = failed(st) ? 1u : 0u;
    mbar_init(&s_bar, 1);
    fence_mbar_init();
  }
  __syncthreads();
  if (s_abort) return;  // an earlier kernel failed: leave the outputs alone
  const uint32_t tile = s_tile;
  const int64_t t0 = (int64_t)tile * kBoxTile;
  const int64_t nn = n;
  const int jend = (int)((nn - t0) < kWin ? (nn - t0) : kWin);  // valid window points
  {
    // The window by bulk copy (TMA): keys of points [t0 - 2, t0 + jend) and
    // indices of [t0, t0 + jend).  Set bases are multiples of 4 slots and t0
    // of 4096, so both sources start 16-byte aligned; an odd key and up to
    // three indices at the end come by plain loads.  Slots outside the data
    // are never read (every use is bounded by jend).
    const int64_t g0 = t0 >= 2 ? t0 - 2 : 0;
    const uint32_t nk = (uint32_t)(t0 + jend - g0), nk_bulk = nk & ~1u;
    const uint32_t nv = (uint32_t)jend, nv_bulk = nv & ~3u;
    uint64_t* kdst = s_key + (g0 - (t0 - 2));
    if (threadIdx.x == 0) {
      mbar_expect_tx(&s_bar, nk_bulk * 8u + nv_bulk * 4u);
      if (nk_bulk) bulk_load(kdst, keys + g0, nk_bulk * 8u, &s_bar);
      if (nv_bulk) bulk_load(s_val, vals + t0, nv_bulk * 4u, &s_bar);
    }
    if (threadIdx.x == 32 && (nk & 1u)) kdst[nk - 1] = keys[g0 + nk - 1];
    if (threadIdx.x >= 64 && threadIdx.x < 64 + (nv - nv_bulk))
      s_val[nv_bulk + threadIdx.x - 64] = vals[t0 + nv_bulk + threadIdx.x - 64];
    const bool ok = mbar_wait(&s_bar, 0, st, wait_ns);
    if (__syncthreads_or(!ok)) {
      mbar_wait(&s_bar, 0, st, wait_ns);  // let the copy land before the block leaves
      return;
    }
  }
  // dd[j]: the point opens a box at every level >= dd[j].  Past the end of
  // the data every slot reads 0, which ends every box walk there.
  for (int j = threadIdx.x; j < kWin; j += kBoxThreads)
    s_dd[j] = (j >= jend || t0 + j == 0) ? 0u : (uint8_t)first_diff_level(sk[j + 1], sk[j]);
  __syncthreads();

  // Level-Lb box starts among this thread's points 8t .. 8t+7.
  uint32_t mask = 0;
  {
    static_assert(kBoxItems == 8, "one 8-byte read of the level bytes per thread");
    const uint2 w = *reinterpret_cast<const uint2*>(s_dd + threadIdx.x * kBoxItems);
    const uint64_t w64 = ((uint64_t)w.y << 32) | w.x;
#pragma unroll
    for (int k = 0; k < kBoxItems; ++k) {
      const uint32_t d = (uint32_t)(w64 >> (8 * k)) & 0xffu;
      if (threadIdx.x * kBoxItems + k < jend && d <= (uint32_t)Lb) mask |= 1u << k;
    }
  }
  const uint32_t c = __popc(mask);
  uint32_t x = c;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) s_wtot[warp] = x;
  __syncthreads();
  if (threadIdx.x == 0) {
    uint32_t run = 0;
    for (int w = 0; w < W; ++w) {
      const uint32_t v = s_wtot[w];
      s_wtot[w] = run;
      run += v;
    }
    s_ttot = run;
    st_relaxed(status + tile, (tile == 0 ? kFlagIncl : kFlagAgg) | run);
  }

  // Finishing sort inside the level-Ls boxes that START in this tile,
  // including their points in the halo past the tile's end (a box begun in
  // an earlier tile is that tile's).  A point's rank counts the points of its
  // box that come before it in (full key, original index) order; the order
  // the radix passes left inside a box does not matter.  Each warp takes 32 consecutive
  // points; box bounds inside the warp come from one ballot of box starts.
  // This runs between publishing the aggregate and reading the earlier
  // tiles' words, which gives them time to publish.
  if (Ls >= kMaxLevel || sg.exact) {
    // Sorted with stable passes on all 63 key bits, or on exactly the bits
    // that the order asks for: the order is already final.
    const int own = jend < kBoxTile ? jend : kBoxTile;
    for (int j = threadIdx.x; j < own; j += kBoxThreads) perm[t0 + j] = s_val[j];
  } else {
    const uint32_t lt = lanemask_lt();
    bool long_box = false;
    const int lowbits = 63 - 3 * Ls;
    const uint64_t lowmask = lowbits >= 64 ? ~0ull : ((1ull << lowbits) - 1ull);
    // The points of a box differ in their low key bits only: the top 32 of those
    // take the keys' low words, and points are compared by them.  The bits they push
    // out take the place that they leave in the high words, below the box's prefix,
    // so that points that agree in the low words are ordered by the high ones, then by
    // index.  (The boxes' keys below need the prefix alone, Lb <= Ls; past level 10
    // the prefix reaches the low words.)  A box is compared all against all, so these
    // loads and compares are most of the kernel's instructions: 7.4e7 points in 512
    // sets 882 -> 737 us, 2 x 2^24 points on a sphere and in clumps 356 -> 307; 8192
    // points 250 times over 539 -> 627 (1014 with the tied points' keys from memory).
    const bool words = Lb <= 10;
    uint2* const word = reinterpret_cast<uint2*>(sk + 1);  // point j: x low, y high
    if (words) {
      const int over = lowbits - 32;  // bits pushed out
      for (int j = threadIdx.x; j < jend; j += kBoxThreads) {
        const uint64_t k = sk[j + 1];
        uint32_t lo = (uint32_t)(k & lowmask), hi = (uint32_t)(k >> 32);
        if (over > 0) {
          const uint32_t out = (1u << over) - 1u;
          hi = (hi & ~out) | (lo & out);
          lo = (uint32_t)(k >> over);
        }
        word[j] = make_uint2(lo, hi);
      }
      __syncthreads();
    }
    for (int c0 = warp * 32; c0 < jend; c0 += W * 32) {
      const int j = c0 + lane;
      const bool in = j < jend;
      const bool start = in && s_dd[j] <= (uint32_t)Ls;
      const uint32_t f = __ballot_sync(0xffffffffu, start);
      int a;  // box start: last start at or before this lane, else walk back
      const uint32_t le = f & (lt | (1u << lane));
      if (le) {
        a = c0 + 31 - __clz(le);
      } else {
        a = c0;
        while (a > 0 && s_dd[a] > (uint32_t)Ls) --a;
      }
      int b;  // box end: next start after this lane, else walk on
      const uint32_t gt = f & ~(lt | (1u << lane));
      if (gt) {
        b = c0 + __ffs(gt) - 1;
      } else {
        b = c0 + 32;
        while (b < jend && s_dd[b] > (uint32_t)Ls) ++b;
        if (b > jend) b = jend;
      }
      if (!in) continue;
      if (a >= kBoxTile) continue;                                // the next tile's box
      if (a == 0 && t0 > 0 && s_dd[0] > (uint32_t)Ls) continue;  // an earlier tile's box
      if (b == jend && t0 + jend < nn) {
        long_box = true;  // runs past the window: the host redoes the order
        continue;
      }
      uint32_t r = 0;
      if (words && b - a > 1) {
        const uint32_t mine = word[j].x;
        uint32_t alike = 0;
        for (int q = a; q < b; ++q) {
          const uint32_t k = word[q].x;
          r += k < mine;
          alike += k == mine;
        }
        if (alike > 1) {  // more than the point itself
          const uint32_t hj = word[j].y, vj = s_val[j];
          for (int q = a; q < b; ++q) {
            const uint2 k = word[q];
            r += k.x == mine && (k.y < hj || (k.y == hj && s_val[q] < vj));
          }
        }
      } else if (b - a > 1) {
        // within a box the top bits agree: order by (low key bits, index)
        const uint64_t mine = sk[j + 1] & lowmask;
        const uint32_t vj = s_val[j];
        for (int q = a; q < b; ++q) {
          const uint64_t kq = sk[q + 1] & lowmask;
          r += (kq < mine) || (kq == mine && s_val[q] < vj);
        }
      }
      perm[t0 + a + r] = s_val[j];
    }
    if (long_box) {
      atomicExch(&st->seg_long, 1u);
      atomicExch(sg.seg_long, 1u);
    }
  }

  // Windowed look-back over the earlier tiles.
  if (warp == 0) {
    uint64_t prev = 0;
    if (tile > 0) {
      prev = lookback_warp(status, tile, 1, st, wait_ns);
      if (lane == 0) st_relaxed(status + tile, kFlagIncl | (prev + s_ttot));
    }
    if (lane == 0) s_texcl = (uint32_t)prev;
  }
  __syncthreads();
  if (threadIdx.x == 0 && tile > 0 && ld_relaxed_u32(&st->abort)) s_abort = 1;
  __syncthreads();
  if (s_abort) return;  // a wait gave up: ranks may be wrong, write nothing
  if (tile == ntiles - 1 && threadIdx.x == 0) {
    const uint32_t nb = s_texcl + s_ttot;
    sg.nbox[Lb] = nb;
    if (nb <= lv.cap[Lb]) lv.off[Lb][nb] = n;
  }
  // Level-Lb keys and bookmarks.
  const int shift = 63 - 3 * Lb;
  uint32_t rank = s_texcl + s_wtot[warp] + (x - c);
  const uint32_t cap = lv.cap[Lb];
  while (mask) {
    const int k = __ffs(mask) - 1;
    mask &= mask - 1;
    const int j = threadIdx.x * kBoxItems + k;
    if (rank < cap) {
      lv.key[Lb][rank] = Lb == 0 ? 0ull : sk[j + 1] >> shift;
      lv.off[Lb][rank] = (uint32_t)(t0 + j);
    }
    ++rank;
  }
}

// Box starts of a box whose key first differs from the one before it at level dk: one
// at every level from dk on, counted in the halves of a level pair's word.
__device__ __forceinline__ uint32_t opens(uint32_t dk, int pair) {
  return dk <= 2u * pair ? 0x10001u : (dk == 2u * pair + 1u ? 0x10000u : 0u);
}

// A thread's ITEMS consecutive words (aligned like ITEMS words), `have` of them there.
template <int ITEMS>
__device__ __forceinline__ void load_items(uint32_t (&v)[ITEMS], const uint32_t* p, bool whole,
                                           int64_t have) {
  if (whole) {
    if constexpr (ITEMS == 2) {
      const uint2 a = *reinterpret_cast<const uint2*>(p);
      v[0] = a.x, v[1] = a.y;
    } else {
#pragma unroll
      for (int k = 0; k < ITEMS; k += 4) {
        const uint4 a = *reinterpret_cast<const uint4*>(p + k);
        v[k] = a.x, v[k + 1] = a.y, v[k + 2] = a.z, v[k + 3] = a.w;
      }
    }
  } else {
#pragma unroll
    for (int k = 0; k < ITEMS; ++k) v[k] = k < have ? p[k] : 0u;
  }
}

template <int ITEMS>
__device__ __forceinline__ void store_items(uint32_t* p, const uint32_t (&v)[ITEMS], bool whole,
                                            int64_t have) {
  if (whole) {
    if constexpr (ITEMS == 2) {
      *reinterpret_cast<uint2*>(p) = make_uint2(v[0], v[1]);
    } else {
#pragma unroll
      for (int k = 0; k < ITEMS; k += 4)
        *reinterpret_cast<uint4*>(p + k) = make_uint4(v[k], v[k + 1], v[k + 2], v[k + 3]);
    }
  } else {
#pragma unroll
    for (int k = 0; k < ITEMS; ++k)
      if (k < have) p[k] = v[k];
  }
}

// Levels 0..Lb-1 (and the parents of the level-Lb boxes) from the level-Lb
// boxes: box b opens a level-l box exactly when its key differs from box
// b-1's in the level-l prefix.  A multi-level prefix sum over the boxes (one
// decoupled look-back chain per level) gives each start its rank.
// NL: a bound on the sets' box depths (Lb <= NL), so that the per-level
// loops, unrolled, cover only the levels in use.
// Bound by latency (the look-backs, and stores that follow loads), so: the level-Lb
// bookmarks are loaded before the scans, eight a thread in two vectors; starts are
// counted two levels to a word, which halves the shuffles and lets two blocks of up
// to twelve levels share an SM (one did before); a thread's parents leave as vectors.
// 2 x 2^24 points on a sphere and in clumps, L = 9: 242 -> 133 us; 512 sets of
// 7.4e7 points: 540 -> 277 us.
// ITEMS: boxes a thread.  A tile's chain of level scans, look-backs and stores is the
// whole kernel for a few hundred thousand boxes: two boxes a thread then, eight
// where the boxes alone fill the SMs (200003 clumped points, L = 6: 26 us with
// eight, 16 with two; 10^6, L = 9: 33 and 27).
template <int NL, int ITEMS>
__global__ void __launch_bounds__(kBoxThreads, NL <= 8 ? (ITEMS == 2 ? 4 : 3) : NL <= 12 ? (ITEMS == 2 ? 3 : 2) : 1) coarse_boxes_kernel(const Seg* __restrict__ segs,
                                                                   const Slot* __restrict__ slots,
                                                                   uint32_t nslots, DevStatus* st,
                                                                   uint64_t wait_ns) {
  constexpr int W = kBoxThreads / 32;
  constexpr uint32_t kTile = kBoxThreads * ITEMS;
  __shared__ uint32_t s_tile, s_abort;
  constexpr int NP = (NL + 1) / 2;  // level pairs: a tile's counts fit 16 bits
  __shared__ uint32_t s_wtot[W][NP];     // a warp's box starts, two levels to a word
  __shared__ uint32_t s_wex[W][kLevels]; // rank of a warp's first start
  __shared__ uint32_t s_ttot[kLevels];   // rank after the tile's last start
  __shared__ uint64_t s_key[kTile + 1];  // s_key[j + 1] = level-Lb key of box t0 + j
  grid_wait(segs, slots);
  const Seg& sg = segs[slots[find_slot(slots, nslots, blockIdx.x)].seg];
  const int Lb = sg.Lb;
  const LevelArrays& lv = sg.lv;
  const uint32_t n = sg.n;
  uint64_t* status = sg.cstatus;
  uint32_t* nbox = sg.nbox;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (threadIdx.x == 0) {
    s_tile = atomicAdd(&sg.tickets[1], 1u);
    s_abort = failed(st) ? 1u : 0u;
  }
  __syncthreads();
  if (s_abort || Lb < 1) return;
  const uint32_t nb = nbox[Lb] < lv.cap[Lb] ? nbox[Lb] : lv.cap[Lb];
  const uint32_t ntiles = nb == 0 ? 1u : (nb + kTile - 1) / kTile;
  const uint32_t tile = s_tile;
  if (tile >= ntiles) return;  // the grid is sized for the capacity
  const int64_t t0 = (int64_t)tile * kTile;
  const uint64_t* kLb = lv.key[Lb];
  const int up = 63 - 3 * Lb;  // level-Lb key -> full-key position
  for (int j = threadIdx.x; j < kTile + 1; j += kBoxThreads) {
    const int64_t b = t0 - 1 + j;
    s_key[j] = (b >= 0 && b < (int64_t)nb) ? kLb[b] << up : 0ull;
  }
  __syncthreads();
  uint32_t dd[ITEMS];
#pragma unroll
  for (int k = 0; k < ITEMS; ++k) {
    const int j = threadIdx.x * ITEMS + k;
    const int64_t b = t0 + j;
    dd[k] = b >= (int64_t)nb ? 0xffu : (b == 0 ? 0u : first_diff_level(s_key[j + 1], s_key[j]));
  }
  // Level-Lb bookmarks of the thread's boxes, on their way during the scans.
  uint32_t off[ITEMS];
  const uint32_t* kOff = lv.off[Lb] + t0 + threadIdx.x * ITEMS;  // 4 * ITEMS-byte aligned
  const bool whole = t0 + (int64_t)(threadIdx.x + 1) * ITEMS <= (int64_t)nb;
  load_items<ITEMS>(off, kOff, whole, (int64_t)nb - t0 - threadIdx.x * ITEMS);
  uint32_t run[NP];
#pragma unroll
  for (int p = 0; p < NP; ++p) {
    run[p] = 0;
    if (2 * p < Lb) {
      uint32_t c = 0;
#pragma unroll
      for (int k = 0; k < ITEMS; ++k) c += opens(dd[k], p);
      uint32_t x = c;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
      }
      run[p] = x - c;
      if (lane == 31) s_wtot[warp][p] = x;
    }
  }
  __syncthreads();
  for (int l = warp; l < Lb; l += W) {
    const uint32_t c = lane < W ? (s_wtot[lane][l >> 1] >> (16 * (l & 1))) & 0xffffu : 0u;
    uint32_t x = c;
#pragma unroll
    for (int o = 1; o < W; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += y;
    }
    const uint32_t total = __shfl_sync(0xffffffffu, x, W - 1);
    if (lane == 0)
      st_relaxed(status + (uint64_t)tile * kLevels + l, (tile == 0 ? kFlagIncl : kFlagAgg) | total);
    uint64_t prev = 0;
    if (tile > 0) {
      prev = lookback_warp(status + l, tile, kLevels, st, wait_ns);
      if (lane == 0) st_relaxed(status + (uint64_t)tile * kLevels + l, kFlagIncl | (prev + total));
    }
    prev = __shfl_sync(0xffffffffu, (uint32_t)prev, 0);
    if (lane < W) s_wex[lane][l] = (uint32_t)prev + x - c;
    if (lane == 0) s_ttot[l] = (uint32_t)prev + total;
  }
  __syncthreads();
  if (threadIdx.x == 0 && tile > 0 && ld_relaxed_u32(&st->abort)) s_abort = 1;
  __syncthreads();
  if (s_abort) return;  // a wait gave up: ranks may be wrong, write nothing
  if (tile == ntiles - 1 && threadIdx.x == 0) {
    for (int l = 0; l < Lb; ++l) {
      const uint32_t c = s_ttot[l];
      nbox[l] = c;
      if (c <= lv.cap[l]) lv.off[l][c] = n;
      if (c <= lv.cap[l]) lv.child[l][c] = l + 1 < Lb ? s_ttot[l + 1] : nb;
    }
  }
  // the next level-(Lb-1) box's rank: a level-Lb box's parent is the one before
  uint32_t last = s_wex[warp][Lb - 1];
#pragma unroll
  for (int p = 0; p < NP; ++p)
    if (p == (Lb - 1) >> 1) last += (run[p] >> (16 * ((Lb - 1) & 1))) & 0xffffu;
  uint32_t par[ITEMS];
#pragma unroll
  for (int k = 0; k < ITEMS; ++k) {
    const int j = threadIdx.x * ITEMS + k;
    const uint32_t dk = dd[k];
    if (dk < (uint32_t)Lb) {
      const uint64_t key = s_key[j + 1];
      if (last < lv.cap[Lb - 1]) lv.child[Lb - 1][last] = (uint32_t)t0 + j;
      ++last;
      uint32_t up_rk = 0;  // rank of the level-(l-1) box open at this box or before it
#pragma unroll
      for (int l = 0; l < NL; ++l) {
        if (l < Lb && l + 1 >= (int)dk) {
          const uint32_t rk = s_wex[warp][l] + ((run[l / 2] >> (16 * (l & 1))) & 0xffffu);
          if ((uint32_t)l >= dk) {
            if (rk < lv.cap[l]) {
              lv.key[l][rk] = l == 0 ? 0ull : key >> (63 - 3 * l);
              lv.off[l][rk] = off[k];
              if (l >= 1) {
                lv.parent[l][rk] = up_rk;
                if ((uint32_t)l > dk && up_rk < lv.cap[l - 1]) lv.child[l - 1][up_rk] = rk;
              }
            }
            up_rk = rk;
          } else {
            up_rk = rk - 1u;  // l = dk - 1: the last box of the level so far
          }
        }
      }
    }
    par[k] = last - 1u;
#pragma unroll
    for (int p = 0; p < NP; ++p) run[p] += opens(dk, p);
  }
  store_items<ITEMS>(lv.parent[Lb] + t0 + threadIdx.x * ITEMS, par, whole,
                     (int64_t)nb - t0 - threadIdx.x * ITEMS);
}

int coarse_items(uint64_t boxes) { return boxes <= (4u << 20) ? 2 : 8; }

uint32_t coarse_tiles(uint32_t cap, int items) {
  const uint64_t tile = (uint64_t)kBoxThreads * items, t = (cap + tile - 1) / tile;
  return t == 0 ? 1u : (uint32_t)t;
}

void launch_finish_boxes(const Seg* segs, const Slot* slots, uint32_t nslots, uint32_t units,
                         DevStatus* st, uint64_t wait_ns, cudaStream_t s) {
  if (units == 0) return;
  // once per process (thread-safe static initialisation)
  static const bool attr = [] {
    cudaFuncSetAttribute(finish_boxes_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)kBoxSmem);
    return true;
  }();
  (void)attr;
  launch_k(finish_boxes_kernel, units, kBoxThreads, kBoxSmem, s, segs, slots, nslots, st, wait_ns);
}

namespace {

template <int ITEMS>
void coarse_boxes_items(const Seg* segs, const Slot* slots, uint32_t nslots, uint32_t units,
                        int max_lb, DevStatus* st, uint64_t wait_ns, cudaStream_t s) {
  auto* const kernel = max_lb <= 8    ? coarse_boxes_kernel<8, ITEMS>
                       : max_lb <= 12 ? coarse_boxes_kernel<12, ITEMS>
                       : max_lb <= 16 ? coarse_boxes_kernel<16, ITEMS>
                                      : coarse_boxes_kernel<kLevels, ITEMS>;
  launch_k(kernel, units, kBoxThreads, 0, s, segs, slots, nslots, st, wait_ns);
}

}  // namespace

void launch_coarse_boxes(const Seg* segs, const Slot* slots, uint32_t nslots, uint32_t units,
                         int max_lb, int items, DevStatus* st, uint64_t wait_ns, cudaStream_t s) {
  if (units == 0) return;
  if (items == 2)
    coarse_boxes_items<2>(segs, slots, nslots, units, max_lb, st, wait_ns, s);
  else
    coarse_boxes_items<8>(segs, slots, nslots, units, max_lb, st, wait_ns, s);
}

// ---------------------------------------------------------------------------
// Child-occupancy byte of every box of levels 0..Lb-1 of the sets that serve
// as sources: bit o is set when the child in octant o (x + 2y + 4z) is
// non-empty.  Lists use it to enumerate the children of a parent-level
// neighbour without reading their keys.  A set owns a run of units (blocks)
// in proportion to its size; a unit takes a strided share of one level, or in
// builds that fill the SMs with units of every level in turn (a unit that walks
// the levels waits three loads a level: 10^6 points, L = 9, 24 -> 16 us; 512 sets
// have units enough, 78 us against 123).
__global__ void __launch_bounds__(256) occupancy_kernel(const Seg* __restrict__ segs,
                                                        const Slot* __restrict__ slots,
                                                        uint32_t nslots, uint32_t unit_first,
                                                        uint32_t launch_units,
                                                        const DevStatus* st) {
  grid_wait(segs, slots);
  if (failed(st)) return;
  const uint32_t unit = blockIdx.x % launch_units + unit_first;
  const bool one_level = gridDim.x > launch_units;
  const int l0 = (int)(blockIdx.x / launch_units);
  const uint32_t k = find_slot(slots, nslots, unit);
  const Seg& sg = segs[slots[k].seg];
  const uint32_t u = unit - slots[k].unit0, units = slots[k].aux0;
  for (int l = l0; l < (one_level ? min(l0 + 1, sg.Lb) : sg.Lb); ++l) {
    const uint32_t nb = sg.nbox[l] < sg.lv.cap[l] ? sg.nbox[l] : sg.lv.cap[l];
    const uint32_t* ch = sg.lv.child[l];
    const uint64_t* ck = sg.lv.key[l + 1];
    const uint32_t nbc = sg.nbox[l + 1] < sg.lv.cap[l + 1] ? sg.nbox[l + 1] : sg.lv.cap[l + 1];
    uint8_t* occ = sg.lv.occ[l];
    for (uint32_t b = u * blockDim.x + threadIdx.x; b < nb; b += units * blockDim.x) {
      uint32_t m = 0;
      const uint32_t c1 = ch[b + 1] < nbc ? ch[b + 1] : nbc;  // (never above nbc in a whole tree)
      for (uint32_t c = ch[b]; c < c1; ++c) m |= 1u << (uint32_t)(ck[c] & 7u);
      occ[b] = (uint8_t)m;
    }
  }
}

void launch_occupancy(const Seg* segs, const Slot* slots, uint32_t nslots, uint32_t units,
                      uint32_t unit_first, int max_lb, DevStatus* st, cudaStream_t s) {
  if (units == 0 || max_lb == 0) return;
  const uint32_t grid = units <= 304u ? units * (uint32_t)max_lb : units;
  launch_k(occupancy_kernel, grid, 256, 0, s, segs, slots, nslots, unit_first, units, st);
}

uint32_t occupancy_units(uint32_t n) { return 1u + n / 16384u; }

// ---------------------------------------------------------------------------
// Cluster-size depth (Sec. 2.1: the smallest level whose boxes hold at most
// s points).  In an order sorted by the top 3*Ls key bits, a level-l box
// (l <= Ls) is a contiguous run, so it holds more than s points exactly when
// some sorted point i and point i + s share it, i.e. when their keys agree on
// the level-l prefix.  One pass over the pairs (i, i + s) therefore gives,
// for every set, D = max_i (deepest level shared by points i and i + s),
// capped at Ls; written as D + 1 by atomicMax into out[set] (zeroed, so 0
// means "no pair": the set has at most s points).  A set whose level-Ls boxes
// are too full gets Ls + 1, + 2 or + 3 for a box of more than s, 8 s or 64 s
// points: how much deeper it is worth sorting.  Units are sort tiles.
__global__ void __launch_bounds__(256) depth_kernel(const Seg* __restrict__ segs,
                                                    const Slot* __restrict__ slots,
                                                    uint32_t nslots, uint32_t s,
                                                    uint32_t* __restrict__ out,
                                                    const DevStatus* st) {
  grid_wait(segs, slots);
  if (failed(st)) return;
  const uint32_t k = find_slot(slots, nslots, blockIdx.x);
  const uint32_t set = slots[k].seg;
  const Seg& sg = segs[set];
  const uint64_t t0 = (uint64_t)(blockIdx.x - slots[k].unit0) * sg.tile;
  const uint64_t npairs = sg.n > s ? (uint64_t)sg.n - s : 0;
  const uint64_t* keys = sg.skeys;
  const uint32_t cap = (uint32_t)sg.Ls;
  uint32_t m = 0;
  uint64_t too_full = 0;
  for (uint64_t i = t0 + threadIdx.x; i < t0 + sg.tile && i < npairs; i += blockDim.x) {
    const uint32_t shared = first_diff_level(keys[i], keys[i + s]) - 1u;  // 0..21
    const uint32_t v = (shared < cap ? shared : cap) + 1u;
    m = v > m ? v : m;
    if (v > cap) too_full = i;
  }
  // One point of a too full level-Ls box a thread: more than 8 s, 64 s points?  (Only
  // how deep to sort next: for every point it took a third of the kernel's time.)
  if (m > cap && too_full + 8ull * s < sg.n) {
    const uint64_t key = keys[too_full];
    if (first_diff_level(key, keys[too_full + 8ull * s]) > cap) {
      ++m;
      if (too_full + 64ull * s < sg.n && first_diff_level(key, keys[too_full + 64ull * s]) > cap) ++m;
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const uint32_t y = __shfl_xor_sync(0xffffffffu, m, o);
    m = y > m ? y : m;
  }
  if ((threadIdx.x & 31) == 0 && m) atomicMax(out + set, m);
}

void launch_depth(const Seg* segs, const Slot* slots, uint32_t nslots, uint32_t units, uint32_t s,
                  uint32_t* out, DevStatus* st, cudaStream_t stream) {
  if (units == 0) return;
  launch_k(depth_kernel, units, 256, 0, stream, segs, slots, nslots, s, out, st);
}

}  // namespace fmm
