// lists.cu -- E2 neighbour lists and E4 (M2L) interaction lists, levels 2..L.
//
// Alg. 4 builds E2 by a search of the 27 cells around each receiver box.  Here
// both lists come from the level above, with no search: the children of the
// source boxes in E2(parent(r), l-1) are exactly E2(r, l) + E4(r, l) (Sec. 1.4
// item 4, E4 = E2(parent) minus E2).  The level-2 case uses the fact that all
// level-1 boxes touch, so E2 at level 1 is "every non-empty source box".
//
// For a parent-level neighbour Q at offset delta (per axis -1, 0, +1) from
// parent(r), and r in octant rho of its parent, a child of Q in octant o is in
// E2(r) iff on every axis |2 delta + o - rho| <= 1, i.e.
//     delta = 0: any child bit;  delta = +1: bit 0, only if rho = 1;
//     delta = -1: bit 1, only if rho = 0.
// So E2 children of Q = occ(Q) & mask(delta, rho) and the E4 children are the
// rest of occ(Q), where occ(Q) is Q's child-occupancy byte.  A child's rank is
// child(Q) + popc(occ(Q) below its octant), so neither list reads child keys,
// and walking Q in ascending rank, children in ascending octant, yields
// ascending ranks.
//
// Two launches a level (one for small levels of one job).  The count kernel finds every parent's E2 and E4
// entries and their prefix sums (of its receiver children together); the fill kernel
// writes rows and entries, one warp a parent, no warp waiting for another.
// Both walk the parents in chunks of four that never cross a job (a job's last
// chunk may hold fewer): a warp takes a chunk at a time, so that the loads of
// four parents are in flight together.
#include <algorithm>
#include <type_traits>

#include "fmm_internal.cuh"

namespace fmm {

constexpr int kChunk = 4;      // parents of a chunk
constexpr int kNbor = 27;      // neighbours of a parent, at most
constexpr int kCand = 27 * 8;  // candidates: the neighbours' children
constexpr int kCountWarps = kListThreads / 32;
constexpr int kCountPasses = 8;              // chunks a count warp takes in a row, at most
constexpr uint32_t kCountGrid = 152u * 8u;   // eight blocks an SM
constexpr int kFillWarps = kListThreads / 32;
constexpr uint32_t kFillGrid = 152u * 4u;    // four blocks an SM

__device__ __forceinline__ uint32_t axis_mask(int delta, uint32_t rho_bit, uint32_t lo_oct,
                                              uint32_t hi_oct) {
  // lo_oct / hi_oct: octants with child bit 0 / 1 on this axis.
  if (delta == 0) return lo_oct | hi_oct;
  if (delta == 1) return rho_bit ? lo_oct : 0u;
  return rho_bit ? 0u : hi_oct;  // delta == -1
}

__device__ __forceinline__ uint32_t e2_child_mask(int dx, int dy, int dz, uint32_t rho) {
  return axis_mask(dx, rho & 1u, 0x55u, 0xaau) & axis_mask(dy, (rho >> 1) & 1u, 0x33u, 0xccu) &
         axis_mask(dz, (rho >> 2) & 1u, 0x0fu, 0xf0u);
}

// Population count of each byte.
__device__ __forceinline__ uint32_t byte_popc(uint32_t v) {
  v -= (v >> 1) & 0x55555555u;
  v = (v & 0x33333333u) + ((v >> 2) & 0x33333333u);
  return (v + (v >> 4)) & 0x0f0f0f0fu;
}

// Sum of the bytes of v (below 256 in all).
__device__ __forceinline__ uint32_t byte_sum(uint32_t v) { return (v * 0x01010101u) >> 24; }

// Bytes 0..3: all ones where bit 0..3 of m is set.
__device__ __forceinline__ uint32_t byte_mask(uint32_t m) {
  return (((m & 0xfu) * 0x00204081u) & 0x01010101u) * 0xffu;
}

// Inclusive prefix sum over the warp (the shuffle's own predicate says whether
// the lane that far below exists).
__device__ __forceinline__ uint32_t warp_incl(uint32_t x) {
#pragma unroll
  for (int o = 1; o < 32; o <<= 1)
    asm volatile(
        "{\n\t.reg .pred p;\n\t.reg .b32 y;\n\tshfl.sync.up.b32 y|p, %0, %1, 0, "
        "0xffffffff;\n\t@p add.u32 %0, %0, y;\n\t}"
        : "+r"(x)
        : "r"(o));
  return x;
}

__device__ __forceinline__ uint64_t warp_incl(uint64_t x) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint64_t y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  return x;
}

// Position of octant o among the 3 x 3 x 3 offsets: its part of an offset code.
__host__ __device__ constexpr uint32_t oct_pos(uint32_t o) {
  return (o & 1u) + 3u * ((o >> 1) & 1u) + 9u * (o >> 2);
}

// Of a neighbour at offset code (dx+1) + 3(dy+1) + 9(dz+1): byte rho = its children
// in sibling rho's E2.
__device__ __forceinline__ uint2 code_masks(uint32_t code) {
  const int dx = (int)(code % 3u) - 1, dy = (int)(code / 3u % 3u) - 1, dz = (int)(code / 9u) - 1;
  uint32_t m[2] = {0, 0};
  for (uint32_t rho = 0; rho < 8; ++rho)
    m[rho >> 2] |= e2_child_mask(dx, dy, dz, rho) << (8 * (rho & 3));
  return make_uint2(m[0], m[1]);
}

// Chunks a count warp takes in a row in a level of `chunks`: small levels are
// spread over the SMs, one chunk a warp.
__host__ __device__ inline uint32_t count_passes(uint32_t chunks) {
  const uint32_t p = chunks / (kCountGrid * kCountWarps);
  return p < 1u ? 1u : (p > (uint32_t)kCountPasses ? (uint32_t)kCountPasses : p);
}

// Chunks of a count block: whole tiles of its warps' passes, one range a block.
__device__ __forceinline__ uint32_t count_range(uint32_t chunks) {
  const uint32_t tile = count_passes(chunks) * kCountWarps;
  const uint32_t tiles = (chunks + tile - 1) / tile;
  return tile * ((tiles + kCountGrid - 1) / kCountGrid);
}

// Chunks of a job with np parents at level l.
__device__ __forceinline__ uint32_t job_chunks(const Job& J, const Seg* segs, int l) {
  return J.L < l ? 0u : (segs[J.recv].nbox[l - 1] + kChunk - 1) / kChunk;
}

// Chunks of a level of at most `cap` parents in all, at most.
uint32_t list_chunks(uint64_t cap, uint32_t njobs) { return (uint32_t)(cap / kChunk) + njobs; }
uint32_t list_blocks() { return kCountGrid; }
uint32_t list_small_tiles(uint64_t parents) {
  return (uint32_t)std::max<uint64_t>((parents + kFillWarps - 1) / kFillWarps, 1u);
}

// Per level (one block each): the chunks before each job.
__global__ void __launch_bounds__(1024) list_plan_kernel(const Seg* __restrict__ segs,
                                                         const Job* __restrict__ jobs,
                                                         uint32_t njobs, const ListLevel* lvls,
                                                         const DevStatus* st) {
  __shared__ uint32_t s_sum[33];
  grid_wait(segs, jobs);
  if (failed(st)) return;
  const int l = 2 + blockIdx.x;
  const ListLevel& LV = lvls[l];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint32_t before = 0;
  for (uint32_t c = 0; c < njobs; c += blockDim.x) {
    const uint32_t j = c + threadIdx.x;
    const uint32_t v = j < njobs ? job_chunks(jobs[j], segs, l) : 0u;
    const uint32_t x = warp_incl(v);
    __syncthreads();
    if (lane == 31) s_sum[warp] = x;
    __syncthreads();
    if (warp == 0) {
      const uint32_t w = s_sum[lane], y = warp_incl(w);
      s_sum[lane] = y - w;
      if (lane == 31) s_sum[32] = y;
    }
    __syncthreads();
    if (j < njobs) LV.jchunks[j] = before + s_sum[warp] + x - v;
    before += s_sum[32];
  }
  if (threadIdx.x == 0) LV.jchunks[njobs] = before;
}

void launch_list_plan(const Seg* segs, const Job* jobs, uint32_t njobs, int Lmax,
                      const ListLevel* lvls, DevStatus* st, cudaStream_t s) {
  if (njobs <= 1 || Lmax < 2) return;  // one job: its chunks follow from its box counts
  launch_k(list_plan_kernel, (uint32_t)(Lmax - 1), 1024, 0, s, segs, jobs, njobs, lvls, st);
}

// Job whose chunks hold chunk c: jc[j] <= c < jc[j + 1].
__device__ __forceinline__ uint32_t find_job(const uint32_t* jc, uint32_t njobs, uint32_t c) {
  uint32_t lo = 0, hi = njobs;
  while (hi - lo > 1) {
    const uint32_t mid = (lo + hi) >> 1;
    if (jc[mid] <= c)
      lo = mid;
    else
      hi = mid;
  }
  return lo;
}

// A warp's current job at level l.
struct WarpJob : LevelJob {
  uint64_t base2, base4;    // the level's entries before the job
  uint32_t j, chunk0, chunk1, np, nsrc1;
};

__host__ __device__ inline LevelJob make_level_job(const Job& J, const Seg& S, const Seg& R, int l,
                                                   const ListLevel& up) {
  LevelJob v;
  v.off_up = J.out2[l - 1];
  v.idx_up = l > 2 ? up.idx2 + 27ull * J.slot[l - 1] : nullptr;
  v.code_up = l > 2 ? up.code2 + 27ull * J.slot[l - 1] : nullptr;
  v.rchild = R.lv.child[l - 1];
  v.rkey = R.lv.key[l];
  v.rkey1 = R.lv.key[1];
  v.socc = S.lv.occ[l - 1];
  v.schild = S.lv.child[l - 1];
  v.skey1 = S.lv.key[1];
  v.rnbox = R.nbox;
  v.snbox = S.nbox;
  v.out2 = J.out2[l];
  v.out4 = J.out4[l];
  v.slot = J.slot[l];
  return v;
}

LevelJob level_job(const Job& J, const Seg& src, const Seg& recv, int l, const ListLevel& up) {
  return make_level_job(J, src, recv, l, up);
}

// The job of chunk c (one lane).  one, np1: the only job and its parents, when
// njobs = 1.
__device__ void load_job(WarpJob& W, const Seg* segs, const Job* jobs, uint32_t njobs, int l,
                         const ListLevel& LV, const ListLevel& up, const LevelJob& one,
                         uint32_t np1, uint32_t c) {
  if (njobs == 1) {
    static_cast<LevelJob&>(W) = one;
    W.j = W.chunk0 = 0;
    W.np = np1;
    W.chunk1 = (np1 + kChunk - 1) / kChunk;
    W.nsrc1 = l == 2 ? min(one.snbox[1], 8u) : 0u;
    return;
  }
  const uint32_t j = find_job(LV.jchunks, njobs, c);
  const Job& J = jobs[j];
  const LevelJob v = make_level_job(J, segs[J.src], segs[J.recv], l, up);
  const uint32_t np = v.rnbox[l - 1], ns = v.snbox[1], c0 = LV.jchunks[j], c1 = LV.jchunks[j + 1];
  static_cast<LevelJob&>(W) = v;
  W.j = j;
  W.np = np;
  W.chunk0 = c0;
  W.chunk1 = c1;
  W.nsrc1 = min(ns, 8u);
}

// At level 2 every pair of level-1 boxes touches: the offset code follows from
// their octants.
__device__ __forceinline__ uint32_t level1_code(uint32_t source, uint32_t receiver) {
  return 13u + oct_pos(source) - oct_pos(receiver);
}

// Counts: per receiver child r of parent p, |E2(r)| = sum over the parent's
// neighbours Q of popc(occ(Q) & mask(delta_Q, rho_r)), and |E2| + |E4| = the
// number of non-empty children of all Q.  Eight lanes a parent, four parents a
// warp pass; the eight sibling octants are counted at once, as bytes.  The
// kernel waits on chains of dependent loads (row start, entry, occupancy), so
// it keeps many warps in flight.  off2 / off4: a parent's first entries, from
// the block's first; the last block to finish turns the blocks' totals
// into their prefix sums and closes the jobs' rows.  Offsets a parent, not a
// receiver box, and no separate prefix sum over them: 116 us for levels 2..7
// of 2^24 uniform points, against 187 us for a warp a parent, counts a receiver
// box and a prefix sum launch a level.
__global__ void __launch_bounds__(kListThreads, 6) list_count_kernel(
    const Seg* __restrict__ segs, const Job* __restrict__ jobs, uint32_t njobs, int l,
    const __grid_constant__ ListLevel LV, const __grid_constant__ ListLevel up,
    const __grid_constant__ LevelJob one, DevStatus* st) {
  __shared__ uint2 s_mask[kNbor];
  __shared__ WarpJob s_job[kCountWarps];
  __shared__ uint64_t s_sum[2][kCountWarps + 1];
  __shared__ uint32_t s_last;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (tid < kNbor) s_mask[tid] = code_masks(tid);
  grid_wait(segs, jobs);
  const int sub = lane >> 3, l8 = lane & 7;
  const uint32_t np1 = njobs == 1 ? one.rnbox[l - 1] : 0u;
  const uint32_t chunks = njobs == 1 ? (np1 + kChunk - 1) / kChunk : LV.jchunks[njobs];
  if (failed(st)) return;  // set before this launch: the same for every thread
  const uint32_t passes = count_passes(chunks), range = count_range(chunks);
  const uint32_t b0 = blockIdx.x * range;
  const uint32_t nblocks = range ? (chunks + range - 1) / range : 0u;
  if (blockIdx.x >= max(nblocks, 1u)) return;
  __syncthreads();
  WarpJob& W = s_job[warp];
  uint32_t jend = 0;
  uint64_t run2 = 0, run4 = 0;  // the block's entries so far
  const uint32_t b1 = min(b0 + range, chunks);
  for (uint32_t t0 = b0; t0 < b1; t0 += passes * kCountWarps) {
    const uint32_t c0 = t0 + warp * passes;
    uint32_t keep2 = 0, keep4 = 0;  // lane 4 k + i: parent i of the warp's chunk k
    for (uint32_t k = 0; k < passes; ++k) {
      const uint32_t c = c0 + k;
      uint32_t n2 = 0, n4 = 0;
      if (c < b1) {
        if (c >= jend) {  // c only grows
          __syncwarp();
          if (lane == 0) load_job(W, segs, jobs, njobs, l, LV, up, one, np1, c);
          __syncwarp();
          jend = W.chunk1;
        }
        const uint32_t p = (c - W.chunk0) * kChunk + sub;
        const bool in = p < W.np;
        uint32_t first = 0, m = 0, r0 = 0, nch = 0;
        if (in) {
          r0 = W.rchild[p];
          nch = min(W.rchild[p + 1] - r0, 8u);
          if (l == 2) {
            m = W.nsrc1;
          } else {
            first = W.off_up[p];
            m = min(W.off_up[p + 1] - first, (uint32_t)kNbor);
          }
        }
        uint32_t q[4], code[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const uint32_t i = l8 + 8 * u;
          q[u] = i;
          code[u] = 13;
          if (i < m) {
            if (l == 2) {
              code[u] = level1_code((uint32_t)W.skey1[i], (uint32_t)W.rkey1[p]);
            } else {
              q[u] = W.idx_up[first + i];
              code[u] = W.code_up[first + i];
            }
          }
        }
        const uint32_t oct = (uint32_t)l8 < nch ? 1u << (uint32_t)(W.rkey[r0 + l8] & 7u) : 0u;
        uint32_t lo = 0, hi = 0, tp = oct << 16;  // tp: candidates | octants of the children << 16
        uint32_t occ[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) occ[u] = (uint32_t)l8 + 8 * u < m ? W.socc[q[u]] : 0u;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const uint2 mk = s_mask[code[u]];
          const uint32_t occ4 = occ[u] * 0x01010101u;
          lo += byte_popc(mk.x & occ4);
          hi += byte_popc(mk.y & occ4);
          tp += __popc(occ[u]);
        }
#pragma unroll
        for (int o = 1; o < 8; o <<= 1) {
          lo += __shfl_xor_sync(0xffffffffu, lo, o);
          hi += __shfl_xor_sync(0xffffffffu, hi, o);
          tp += __shfl_xor_sync(0xffffffffu, tp, o);
        }
        const uint32_t present = tp >> 16;
        n2 = byte_sum(lo & byte_mask(present)) + byte_sum(hi & byte_mask(present >> 4));
        n4 = (uint32_t)__popc(present) * (tp & 0xffffu) - n2;
      }
      // lane 4 k + i takes parent i's counts (its group: lanes 8 i ..)
      const uint32_t v2 = __shfl_sync(0xffffffffu, n2, (lane & 3) * 8);
      const uint32_t v4 = __shfl_sync(0xffffffffu, n4, (lane & 3) * 8);
      if ((uint32_t)(lane >> 2) == k) {
        keep2 = v2;
        keep4 = v4;
      }
    }
    const uint32_t x2 = warp_incl(keep2), x4 = warp_incl(keep4);
    if (lane == 31) {
      s_sum[0][warp] = x2;
      s_sum[1][warp] = x4;
    }
    __syncthreads();
    uint64_t w2 = run2, w4 = run4;
#pragma unroll
    for (int w = 0; w < kCountWarps; ++w) {
      const uint64_t a = s_sum[0][w], b = s_sum[1][w];
      if (w < warp) {
        w2 += a;
        w4 += b;
      }
      run2 += a;
      run4 += b;
    }
    __syncthreads();
    const uint32_t c = c0 + (lane >> 2);
    if ((uint32_t)(lane >> 2) < passes && c < b1) {
      LV.off2[(uint64_t)c * kChunk + (lane & 3)] = (uint32_t)w2 + x2 - keep2;
      LV.off4[(uint64_t)c * kChunk + (lane & 3)] = (uint32_t)w4 + x4 - keep4;
    }
  }
  if (tid == 0) {
    LV.bbase[2 * blockIdx.x] = run2;
    LV.bbase[2 * blockIdx.x + 1] = run4;
  }
  __threadfence();
  __syncthreads();
  if (tid == 0) s_last = atomicAdd(LV.ticket, 1u) + 1u == max(nblocks, 1u);
  __syncthreads();
  if (!s_last) return;
  __threadfence();

  // The last block: the blocks' first entries, then per job its first entry,
  // its totals and its closing rows.  (Reads past L1: other blocks wrote them.)
  constexpr int kPer = (kCountGrid + kListThreads - 1) / kListThreads;
  uint64_t tot[2] = {0, 0};
#pragma unroll
  for (int d = 0; d < 2; ++d) {
    uint64_t v[kPer], sum = 0;
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
      const uint32_t b = tid * kPer + k;
      v[k] = b < nblocks ? __ldcg(LV.bbase + 2 * b + d) : 0ull;
      sum += v[k];
    }
    const uint64_t x = warp_incl(sum);
    if (lane == 31) s_sum[d][warp] = x;
    __syncthreads();
    uint64_t e = x - sum;
    for (int w = 0; w < kCountWarps; ++w) {
      if (w < warp) e += s_sum[d][w];
      tot[d] += s_sum[d][w];
    }
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
      const uint32_t b = tid * kPer + k;
      if (b < nblocks) LV.bbase[2 * b + d] = e;
      e += v[k];
    }
    __syncthreads();
  }
  if (njobs == 1) {  // its totals are the level's
    if (tid < 2) {
      const uint64_t n = tot[tid];
      LV.nnz[tid] = n;
      (tid ? one.out4 : one.out2)[one.rnbox[l]] = (uint32_t)n;
      if (n >> 32) set_error(st, FMM_ERR_CAPACITY);
    }
    return;
  }
  for (uint32_t j = tid; j < njobs; j += kListThreads) {
    const Job& J = jobs[j];
    if (J.L < l) continue;
    const auto entry = [&](uint32_t c, int d) -> uint64_t {
      if (c >= chunks) return tot[d];
      return LV.bbase[2 * (c / range) + d] + __ldcg((d ? LV.off4 : LV.off2) + (uint64_t)c * kChunk);
    };
    const uint32_t nrecv = segs[J.recv].nbox[l];
    for (int d = 0; d < 2; ++d) {
      const uint64_t a = entry(LV.jchunks[j], d), n = entry(LV.jchunks[j + 1], d) - a;
      LV.jbase[2 * j + d] = a;
      LV.nnz[2 * j + d] = n;
      (d ? J.out4[l] : J.out2[l])[nrecv] = (uint32_t)n;
      if (n >> 32) set_error(st, FMM_ERR_CAPACITY);
    }
  }
}

// Fill.  Per parent p, the candidate list C -- the non-empty children of p's
// neighbours in ascending rank -- is built in shared memory.  p's receiver
// children, its siblings, are numbered 0..nsib-1 in order.  Every candidate
// carries its rank, a flag per sibling whose E2 it belongs to, and a byte per
// sibling: the parent's E2 entries before this candidate's, were it in that
// sibling's E2 -- all of the earlier siblings' and those of the earlier
// candidates (216 at most).  That byte is the candidate's place among the parent's
// E2 entries, and its place among the parent's E4 entries is
// (sibling) |C| + (index in C) - byte.  So a warp turns 32 candidates into one
// sibling's entries with a byte extract, a flag test, an add, an address and a
// store -- no ballot, no population count, no cursor: the loop is bound by
// instructions issued, not by memory.  Bytes are counted four siblings to a
// word; a parent of up to four siblings needs one word, and is half of all
// parents of clumped and surface-like sets.
//
// Entries are stored directly where the parent's lists are short.  From kStageMin
// candidates on (and more than four siblings) four siblings' E4 entries are
// gathered in shared memory, aligned like the output, and leave by one bulk
// copy: DRAM and L2 see whole lines, and the loop's stores stay on chip.  Both
// sides measured, levels 2..7 of 2^24 uniform points (216 candidates nearly
// everywhere): 455 us gathered, 714 us stored directly; levels 2..9 of 2^24
// points on a sphere and in clumps (60 to 100 candidates): 565 us with every
// parent gathered, 506 us with this rule.  With one ballot, two population
// counts and a cursor per 32 entries these took 636 and 716 us.
//
// kCodes: also write the E2 entries' offset codes for the next level (every
// level but the last).
constexpr uint32_t kStageMin = 128;   // candidates of a parent whose E4 entries are gathered first
constexpr uint32_t kStage = 4 * 189;  // E4 entries gathered at a time: four siblings'
struct FillWarp {
  uint4 cand[kCand];    // rank, flags (sibling j: bit 8 j, or 8 (j - 4) + 4), bytes 0..3, 4..7
  __align__(16) uint32_t stage[kStage + 4];
  uint8_t pos[kCand];   // position among the children of the parent's neighbours, plus 13
  uint8_t near[72];     // the candidates in some sibling's E2 (the 4x4x4 block)
};
static_assert(sizeof(FillWarp) % 16 == 0, "stage alignment");
struct FillSmem {
  FillWarp w[kFillWarps];
  uint2 mask[kNbor];
  uint32_t sel[256];    // per set of octants present: byte selectors of siblings 0..3, 4..7 << 16
};

// v to global / to shared memory (a byte address) where flag bit kBit is set /
// clear: one test and one predicated store.
template <uint32_t kBit>
__device__ __forceinline__ void put_if(uint32_t* p, uint32_t v, uint32_t flags) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t.reg .b32 t;\n\tand.b32 t, %2, %3;\n\tsetp.ne.u32 p, t, 0;\n\t"
      "@p st.global.u32 [%0], %1;\n\t}" ::"l"(p), "r"(v), "r"(flags), "n"(kBit)
      : "memory");
}
template <uint32_t kBit>
__device__ __forceinline__ void put_unless(uint32_t* p, uint32_t v, uint32_t flags) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t.reg .b32 t;\n\tand.b32 t, %2, %3;\n\tsetp.eq.u32 p, t, 0;\n\t"
      "@p st.global.cs.u32 [%0], %1;\n\t}" ::"l"(p), "r"(v), "r"(flags), "n"(kBit)
      : "memory");
}
template <uint32_t kBit>
__device__ __forceinline__ void stage_unless(uint32_t p, uint32_t v, uint32_t flags) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t.reg .b32 t;\n\tand.b32 t, %2, %3;\n\tsetp.eq.u32 p, t, 0;\n\t"
      "@p st.shared.u32 [%0], %1;\n\t}" ::"r"(p), "r"(v), "r"(flags), "n"(kBit)
      : "memory");
}

// One lane: `bytes` (a multiple of 16) from shared to global memory by a bulk
// copy; stage_wait: the stage may be written again (and the warp's last one
// has left shared memory).
__device__ __forceinline__ void stage_store(uint32_t* dst, const uint32_t* src, uint32_t bytes) {
  asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;\n\t"
               "cp.async.bulk.commit_group;" ::"l"(dst),
               "r"(smem_u32(src)), "r"(bytes)
               : "memory");
}
__device__ __forceinline__ void stage_wait() {
  asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
}

// Candidate e's place: the eight children of a lane's neighbour are 128 bytes
// apart from the next lane's; swapping places inside each eight keeps the
// lanes' stores of one octant off each other's banks.
__device__ __forceinline__ uint32_t cand_at(uint32_t e) { return e ^ ((e >> 3) & 7u); }

// f(integral_constant j) for the siblings j < nsib: of eight (more than four
// are there), or of four.
template <bool kWide, class F>
__device__ __forceinline__ void each_sibling(uint32_t nsib, const F& f) {
  f(std::integral_constant<int, 0>{});
  if (kWide || nsib > 1) f(std::integral_constant<int, 1>{});
  if (kWide || nsib > 2) f(std::integral_constant<int, 2>{});
  if (kWide || nsib > 3) f(std::integral_constant<int, 3>{});
  if constexpr (kWide) {
    f(std::integral_constant<int, 4>{});
    if (nsib > 5) f(std::integral_constant<int, 5>{});
    if (nsib > 6) f(std::integral_constant<int, 6>{});
    if (nsib > 7) f(std::integral_constant<int, 7>{});
  }
}

// The job's lists of the level: rows, entries and offset codes.
struct FillOut {
  uint32_t *out2, *out4, *idx2, *idx4;
  uint8_t* code2;
};
// A parent's first entries in the job's lists; no place: a wait gave up.
struct Place {
  uint64_t e2, e4;
  bool ok;
};

// One parent: its siblings' rows and entries.  kWide: more than four siblings.  c0:
// its first receiver child; place(E2 entries, E4 entries) gives its place.
template <bool kCodes, bool kWide, class PlaceFn>
__device__ __forceinline__ void fill_parent(FillWarp& F, uint2 mk, uint32_t sel, uint32_t nsib,
                                            uint32_t occ, uint32_t code, uint32_t rank,
                                            uint32_t present, uint32_t c0, const FillOut& o_,
                                            const PlaceFn& place) {
  const int lane = threadIdx.x & 31;
  // child masks of the siblings, in their order; none for absent ones
  uint32_t m0 = __byte_perm(mk.x, mk.y, sel), m1 = 0;
  if (kWide) {
    m1 = __byte_perm(mk.x, mk.y, sel >> 16) & (0xffffffffu >> (8u * (8u - nsib)));
  } else {
    m0 &= 0xffffffffu >> (8u * (4u - nsib));
  }
  // per lane (neighbour): candidates before it, and those in each sibling's E2
  const uint32_t occ4 = occ * 0x01010101u;
  const uint32_t lo0 = byte_popc(m0 & occ4), hi0 = kWide ? byte_popc(m1 & occ4) : 0u;
  uint32_t any = (m0 | m1) & occ4;
  any |= any >> 16;
  any |= any >> 8;
  const uint32_t cn = (uint32_t)__popc(occ) | ((uint32_t)__popc(any & 0xffu) << 16);
  const uint32_t xl = warp_incl(lo0), xh = kWide ? warp_incl(hi0) : 0u;
  const uint32_t xc = warp_incl(cn);
  const uint32_t tl = __shfl_sync(0xffffffffu, xl, 31);
  const uint32_t tc = __shfl_sync(0xffffffffu, xc, 31);
  const uint32_t total = tc & 0xffffu, nnear = tc >> 16;
  const uint32_t f0 = tl * 0x01010100u;  // E2 entries of the siblings before each
  uint32_t f1 = 0, tw = 0;
  if (kWide) {
    tw = __shfl_sync(0xffffffffu, xh, 31);
    f1 = tw * 0x01010100u + byte_sum(tl) * 0x01010101u;
  }
  const uint32_t n2 = byte_sum(tl) + (kWide ? byte_sum(tw) : 0u);
  const Place at = place(n2, nsib * total - n2);
  if (!at.ok) return;
  uint32_t* const e2 = o_.idx2 + at.e2;
  uint32_t* const e4 = o_.idx4 + at.e4;
  uint8_t* const codes = kCodes ? o_.code2 + at.e2 : nullptr;
  if ((uint32_t)lane < nsib) {
    const uint32_t f = ((kWide && lane >= 4 ? f1 : f0) >> (8 * (lane & 3))) & 0xffu;
    o_.out2[c0 + lane] = (uint32_t)at.e2 + f;
    o_.out4[c0 + lane] = (uint32_t)at.e4 + lane * total - f;
  }
  uint32_t lo = xl - lo0 + f0, hi = xh - hi0 + f1;
  uint32_t e = (xc - cn) & 0xffffu, ne = (xc - cn) >> 16;
#pragma unroll
  for (int o = 0; o < 8; ++o) {
    if ((occ >> o) & 1u) {
      const uint32_t i0 = (m0 >> o) & 0x01010101u, i1 = kWide ? (m1 >> o) & 0x01010101u : 0u;
      const uint32_t fl = i0 + 16u * i1;
      F.cand[cand_at(e)] = make_uint4(rank, fl, lo, hi);
      if (kCodes) F.pos[e] = (uint8_t)(2u * code + oct_pos(o));
      if (fl) F.near[ne++] = (uint8_t)e;
      ++e;
      ++rank;
      lo += i0;
      if (kWide) hi += i1;
    }
  }
  __syncwarp();
  // E2: the near candidates
  for (uint32_t i = lane; i < nnear; i += 32) {
    const uint32_t c = F.near[i];
    const uint4 v = F.cand[cand_at(c)];
    const uint32_t ps = kCodes ? F.pos[c] - 13u : 0u;
    uint32_t oct = present;  // the sibling's octant is the lowest set bit
    each_sibling<kWide>(nsib, [&](auto jt) {
      constexpr int j = decltype(jt)::value;
      constexpr uint32_t bit = 1u << (j < 4 ? 8 * j : 8 * (j - 4) + 4);
      const uint32_t x = __byte_perm(j < 4 ? v.z : v.w, 0, 0x4440 + (j & 3));
      put_if<bit>(e2 + x, v.x, v.y);
      if (kCodes) {  // position of the child among the parent's, less the sibling's
        if (v.y & bit) codes[x] = (uint8_t)(ps - oct_pos(__ffs(oct) - 1));
        oct &= oct - 1u;
      }
    });
  }
  // E4: every candidate where it is not in E2
  if (!kWide || total < kStageMin) {
    for (uint32_t i = lane; i < total; i += 32) {
      const uint4 v = F.cand[cand_at(i)];
      uint32_t at = i;
      each_sibling<kWide>(nsib, [&](auto jt) {
        constexpr int j = decltype(jt)::value;
        constexpr uint32_t bit = 1u << (j < 4 ? 8 * j : 8 * (j - 4) + 4);
        const uint32_t x = __byte_perm(j < 4 ? v.z : v.w, 0, 0x4440 + (j & 3));
        put_unless<bit>(e4 + (at - x), v.x, v.y);
        at += total;
      });
    }
    __syncwarp();
    return;
  }
  const uint32_t half = 4 * total - (f1 & 0xffu);  // E4 entries of the first four
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const uint32_t from = h ? 4 * total - half : 0u;
    uint32_t* const dst = e4 + (h ? half : 0u);
    const uint32_t n = h ? nsib * total - half - (f1 >> 24) - (tw >> 24) : half;
    const uint32_t a0 = (uint32_t)(reinterpret_cast<uintptr_t>(dst) >> 2) & 3u;
    const uint32_t base = smem_u32(F.stage) + 4u * (a0 + from);  // the stage is aligned like dst
    for (uint32_t i = lane; i < total; i += 32) {
      const uint4 v = F.cand[cand_at(i)];
      const uint32_t b = h ? v.w : v.z, fl = h ? v.y >> 4 : v.y;
      uint32_t at = base + 4u * i;
      each_sibling<false>(h ? nsib - 4 : 4u, [&](auto jt) {
        constexpr int j = decltype(jt)::value;
        const uint32_t x = __byte_perm(b, 0, 0x4440 + j);
        stage_unless<(1u << (8 * j))>(at - 4u * x, v.x, fl);
        at += 4u * total;
      });
    }
    fence_proxy_async();
    __syncwarp();
    // head and tail one by one, the rest by a bulk copy
    uint32_t* const d0 = dst - a0;
    const uint32_t a1 = a0 + n, v0 = min((a0 + 3u) & ~3u, a1), v1 = max(a1 & ~3u, v0);
    if (lane == 0 && v1 > v0) stage_store(d0 + v0, F.stage + v0, 4u * (v1 - v0));
    if ((uint32_t)lane < v0 - a0) d0[a0 + lane] = F.stage[a0 + lane];
    if ((uint32_t)lane < a1 - v1) d0[v1 + lane] = F.stage[v1 + lane];
    if (lane == 0) stage_wait();
    __syncwarp();
  }
}

template <bool kCodes>
__global__ void __launch_bounds__(kListThreads, 4) list_fill_kernel(
    const Seg* __restrict__ segs, const Job* __restrict__ jobs, uint32_t njobs, int l,
    const __grid_constant__ ListLevel LV, const __grid_constant__ ListLevel up,
    const __grid_constant__ LevelJob one, DevStatus* st) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  FillSmem& sm = *reinterpret_cast<FillSmem*>(smem_raw);
  __shared__ WarpJob s_job[kFillWarps];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (tid < kNbor) sm.mask[tid] = code_masks(tid);
  for (int t = tid; t < 256; t += kListThreads) {
    uint32_t sel = 0, n = 0;
    for (uint32_t rho = 0; rho < 8; ++rho)
      if ((t >> rho) & 1) sel |= rho << (4 * n++);
    sm.sel[t] = sel;
  }
  grid_wait(segs, jobs);
  const uint32_t np1 = njobs == 1 ? one.rnbox[l - 1] : 0u;
  const uint32_t chunks = njobs == 1 ? (np1 + kChunk - 1) / kChunk : LV.jchunks[njobs];
  if (failed(st)) return;  // set before this launch: the same for every thread
  // A warp takes whole chunks, or in small levels a part of one.
  const uint32_t warps = gridDim.x * kFillWarps;
  const uint32_t split = 4u * chunks <= warps ? 4u : (2u * chunks <= warps ? 2u : 1u);
  if (blockIdx.x * kFillWarps >= chunks * split) return;
  __syncthreads();
  const uint32_t range = count_range(chunks);
  FillWarp& F = sm.w[warp];
  WarpJob& W = s_job[warp];
  uint32_t jend = 0;
  for (uint32_t u = blockIdx.x * kFillWarps + warp; u < chunks * split; u += warps) {
    const uint32_t c = u / split;  // (a power of two)
    if (c >= jend) {  // c only grows
      __syncwarp();   // every lane has read the last job
      if (lane == 0) {
        load_job(W, segs, jobs, njobs, l, LV, up, one, np1, c);
        W.base2 = njobs == 1 ? 0ull : LV.jbase[2 * W.j];
        W.base4 = njobs == 1 ? 0ull : LV.jbase[2 * W.j + 1];
      }
      __syncwarp();
      jend = W.chunk1;
    }
    const uint32_t p0 = (c - W.chunk0) * kChunk, np = W.np;
    // 1. The chunk's parents, every load of one step of the chain (row start ->
    // entry -> child and occupancy) in flight together.
    // lanes 0..4: E2 rows of the level above, 8..12: children, 16..19 / 24..27:
    // first E2 / E4 entries
    const int sub = lane >> 3, l8 = lane & 7;
    uint32_t head = 0;
    if (sub < 2 ? l8 <= kChunk : l8 < kChunk) {
      const uint32_t* src;
      if (sub == 0)
        src = l == 2 ? nullptr : W.off_up + min(p0 + l8, np);
      else if (sub == 1)
        src = W.rchild + min(p0 + l8, np);
      else
        src = (sub == 2 ? LV.off2 : LV.off4) + (uint64_t)c * kChunk + l8;
      if (src) head = *src;
    }
    const uint64_t g2 = LV.bbase[2 * (c / range)] - W.base2;  // (job-relative)
    const uint64_t g4 = LV.bbase[2 * (c / range) + 1] - W.base4;
    uint32_t cc[kChunk], ch[kChunk];  // occupancy | code << 8, first child
    {
      uint32_t q[kChunk];
      bool in[kChunk];
#pragma unroll
      for (int k = 0; k < kChunk; ++k) {
        const uint32_t first = __shfl_sync(0xffffffffu, head, k);
        const uint32_t end = __shfl_sync(0xffffffffu, head, k + 1);
        const uint32_t m = l == 2 ? (p0 + k < np ? W.nsrc1 : 0u) : min(end - first, (uint32_t)kNbor);
        in[k] = (uint32_t)lane < m;
        q[k] = lane;
        cc[k] = 13u << 8;
        if (in[k]) {
          if (l == 2) {
            cc[k] = level1_code((uint32_t)W.skey1[lane], (uint32_t)W.rkey1[p0 + k]) << 8;
          } else {
            q[k] = W.idx_up[first + lane];
            cc[k] = (uint32_t)W.code_up[first + lane] << 8;
          }
        }
      }
#pragma unroll
      for (int k = 0; k < kChunk; ++k) {
        cc[k] |= in[k] ? W.socc[q[k]] : 0u;
        ch[k] = in[k] ? W.schild[q[k]] : 0u;
      }
    }
    uint32_t octs;  // lanes 8 k ..: octants of parent k's receiver children
    {
      const uint32_t r0 = __shfl_sync(0xffffffffu, head, 8 + sub);
      const uint32_t nch = min(__shfl_sync(0xffffffffu, head, 9 + sub) - r0, 8u);
      octs = (uint32_t)l8 < nch ? 1u << (uint32_t)(W.rkey[r0 + l8] & 7u) : 0u;
#pragma unroll
      for (int o = 1; o < 8; o <<= 1) octs |= __shfl_xor_sync(0xffffffffu, octs, o);
    }
    // 2. The parents, one after another.
    const uint32_t k0 = (u % split) * (kChunk / split), k1 = min(k0 + kChunk / split, np - p0);
    for (uint32_t k = 0; k < k1; ++k) {
      const uint32_t co = cc[0], rank = ch[0];
#pragma unroll
      for (int i = 0; i + 1 < kChunk; ++i) {
        cc[i] = cc[i + 1];
        ch[i] = ch[i + 1];
      }
      if (k < k0) continue;
      const uint32_t present = __shfl_sync(0xffffffffu, octs, 8 * k);
      const uint32_t c0 = __shfl_sync(0xffffffffu, head, 8 + k);
      const Place at{g2 + __shfl_sync(0xffffffffu, head, 16 + k),
                     g4 + __shfl_sync(0xffffffffu, head, 24 + k), true};
      const auto place = [&](uint32_t, uint32_t) { return at; };
      const uint32_t nsib = __popc(present);
      const uint64_t slot = W.slot;
      const FillOut out{W.out2, W.out4, LV.idx2 + 27ull * slot, LV.idx4 + 189ull * slot,
                        kCodes ? LV.code2 + 27ull * slot : nullptr};
      const uint2 mk = sm.mask[co >> 8];
      const uint32_t sel = sm.sel[present];
      if (nsib > 4)
        fill_parent<kCodes, true>(F, mk, sel, nsib, co & 0xffu, co >> 8, rank, present, c0, out, place);
      else if (nsib > 0)
        fill_parent<kCodes, false>(F, mk, sel, nsib, co & 0xffu, co >> 8, rank, present, c0, out, place);
    }
  }
}

// Levels of one job whose parents fit one a warp of a resident grid: counts, prefix
// sums and entries in one launch.  A block takes eight parents (in order, by
// ticket); their counts go up a decoupled look-back over the blocks, E2 by warp 0
// and E4 by warp 1, while the parents' candidates wait in registers.  Levels 2..4
// of 16384 points: 32 us in three launches, 58 in the six of count and fill; above
// a resident grid's parents the look-backs and barriers cost more than a second
// launch (512 sets in one launch a level: 5.96 ms, 3.47 in two).
template <bool kCodes>
__global__ void __launch_bounds__(kListThreads, 4) list_small_kernel(
    int l, const __grid_constant__ ListLevel LV, const __grid_constant__ ListLevel up,
    const __grid_constant__ LevelJob W, DevStatus* st, uint64_t wait_ns) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  FillSmem& sm = *reinterpret_cast<FillSmem*>(smem_raw);
  __shared__ uint32_t s_tile, s_stop, s_n[2][kFillWarps];
  __shared__ uint64_t s_base[2];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (tid < kNbor) sm.mask[tid] = code_masks(tid);
  if (tid < 256) {
    uint32_t sel = 0, n = 0;
    for (uint32_t rho = 0; rho < 8; ++rho)
      if ((tid >> rho) & 1) sel |= rho << (4 * n++);
    sm.sel[tid] = sel;
  }
  grid_wait();
  const uint32_t np = W.rnbox[l - 1];
  if (tid == 0) {
    s_stop = failed(st) ? 1u : 0u;
    s_tile = atomicAdd(LV.ticket, 1u);
  }
  __syncthreads();
  const uint32_t tile = s_tile, tiles = max((np + kFillWarps - 1) / kFillWarps, 1u);
  if (s_stop || tile >= tiles) return;
  const uint32_t p = tile * kFillWarps + warp;

  // The parent's row, children, neighbours (one a lane) and receiver octants.
  uint32_t co = 13u << 8, rank = 0, present = 0, c0 = 0;
  if (p < np) {
    const uint32_t head = lane < 2   ? (l == 2 ? 0u : W.off_up[p + lane])
                          : lane < 4 ? W.rchild[p + lane - 2]
                                     : 0u;
    const uint32_t first = __shfl_sync(0xffffffffu, head, 0);
    const uint32_t m = l == 2 ? min(W.snbox[1], 8u)
                              : min(__shfl_sync(0xffffffffu, head, 1) - first, (uint32_t)kNbor);
    c0 = __shfl_sync(0xffffffffu, head, 2);
    const uint32_t nch = min(__shfl_sync(0xffffffffu, head, 3) - c0, 8u);
    const uint32_t oct = (uint32_t)lane < nch ? 1u << (uint32_t)(W.rkey[c0 + lane] & 7u) : 0u;
    if ((uint32_t)lane < m) {
      uint32_t q = lane;
      if (l == 2) {
        co = level1_code((uint32_t)W.skey1[lane], (uint32_t)W.rkey1[p]) << 8;
      } else {
        q = W.idx_up[first + lane];
        co = (uint32_t)W.code_up[first + lane] << 8;
      }
      co |= W.socc[q];
      rank = W.schild[q];
    }
    present = __reduce_or_sync(0xffffffffu, oct);
  }
  // The block's counts and their place.  Every warp comes here once, from its own
  // call of fill_parent or, without a parent, from below: named barriers.
  const auto place = [&](uint32_t n2, uint32_t n4) {
    if (lane == 0) {
      s_n[0][warp] = n2;
      s_n[1][warp] = n4;
    }
    __syncwarp();
    asm volatile("barrier.sync 1, %0;" ::"n"(kListThreads) : "memory");
    if (warp < 2) {
      uint64_t* const chain = warp ? LV.status4 : LV.status2;
      const uint32_t v = lane < kFillWarps ? s_n[warp][lane] : 0u;
      const uint32_t x = warp_incl(v), tot = __shfl_sync(0xffffffffu, x, 31);
      uint64_t prev = 0;
      if (lane == 0) st_relaxed(chain + tile, (tile == 0 ? kFlagIncl : kFlagAgg) | tot);
      if (tile > 0) {
        prev = lookback_warp(chain, tile, 1, st, wait_ns);
        if (lane == 0) st_relaxed(chain + tile, kFlagIncl | (prev + tot));
      }
      if (lane < kFillWarps) s_n[warp][lane] = x - v;
      if (lane == 0) {
        s_base[warp] = prev;
        if (tile > 0 && ld_relaxed_u32(&st->abort)) s_stop = 1;
        if (tile + 1 == tiles) {  // the last block closes the rows
          const uint64_t n = prev + tot;
          (warp ? W.out4 : W.out2)[W.rnbox[l]] = (uint32_t)n;
          LV.nnz[warp] = n;
          if (n >> 32) set_error(st, FMM_ERR_CAPACITY);
        }
      }
      __syncwarp();
    }
    asm volatile("barrier.sync 1, %0;" ::"n"(kListThreads) : "memory");
    return Place{s_base[0] + s_n[0][warp], s_base[1] + s_n[1][warp], s_stop == 0};
  };
  const uint32_t nsib = __popc(present);
  const FillOut out{W.out2, W.out4, LV.idx2 + 27ull * W.slot, LV.idx4 + 189ull * W.slot,
                    kCodes ? LV.code2 + 27ull * W.slot : nullptr};
  const uint2 mk = sm.mask[co >> 8];
  const uint32_t sel = sm.sel[present];
  if (nsib > 4)
    fill_parent<kCodes, true>(sm.w[warp], mk, sel, nsib, co & 0xffu, co >> 8, rank, present, c0, out, place);
  else if (nsib > 0)
    fill_parent<kCodes, false>(sm.w[warp], mk, sel, nsib, co & 0xffu, co >> 8, rank, present, c0, out, place);
  else
    place(0, 0);
}

bool list_small(uint32_t njobs, uint64_t parents) {
  return njobs == 1 && parents <= (uint64_t)kFillGrid * kFillWarps;
}

void launch_list_small(int l, const ListLevel& lv, const ListLevel& up, const LevelJob& one,
                       uint64_t parents, DevStatus* st, uint64_t wait_ns, cudaStream_t s) {
  static const bool attr = [] {
    cudaFuncSetAttribute(list_small_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)sizeof(FillSmem));
    cudaFuncSetAttribute(list_small_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)sizeof(FillSmem));
    return true;
  }();
  (void)attr;
  const uint32_t grid = list_small_tiles(parents);
  launch_k(lv.code2 ? list_small_kernel<true> : list_small_kernel<false>, grid, kListThreads,
           sizeof(FillSmem), s, l, lv, up, one, st, wait_ns);
}

void launch_list_count(const Seg* segs, const Job* jobs, uint32_t njobs, int l,
                       const ListLevel& lv, const ListLevel& up, const LevelJob& one,
                       uint32_t max_chunks, DevStatus* st, cudaStream_t s) {
  const uint32_t grid = std::min((max_chunks + kCountWarps - 1) / kCountWarps, kCountGrid);
  launch_k(list_count_kernel, std::max(grid, 1u), kListThreads, 0, s, segs, jobs, njobs, l, lv, up, one,
             st);
}

void launch_list_fill(const Seg* segs, const Job* jobs, uint32_t njobs, int l,
                      const ListLevel& lv, const ListLevel& up, const LevelJob& one,
                      uint32_t max_chunks, DevStatus* st, cudaStream_t s) {
  static const bool attr = [] {
    cudaFuncSetAttribute(list_fill_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)sizeof(FillSmem));
    cudaFuncSetAttribute(list_fill_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)sizeof(FillSmem));
    return true;
  }();
  (void)attr;
  const uint64_t units = 4ull * max_chunks;  // a warp takes one parent at least
  const uint32_t grid = (uint32_t)std::max<uint64_t>(
      std::min<uint64_t>((units + kFillWarps - 1) / kFillWarps, kFillGrid), 1u);
  if (lv.code2)
    launch_k(list_fill_kernel<true>, grid, kListThreads, sizeof(FillSmem), s, segs, jobs, njobs, l, lv, up, one,
             st);
  else
    launch_k(list_fill_kernel<false>, grid, kListThreads, sizeof(FillSmem), s, segs, jobs, njobs, l, lv, up, one,
             st);
}

// ---------------------------------------------------------------------------
// Exclusive prefix sum of u32 counts in place, single pass with decoupled
// look-back (the CSR row starts NeighborBookmark of Alg. 4).
__host__ __device__ inline uint32_t scan_tiles_of(uint32_t cap) {
  const uint64_t t = ((uint64_t)cap + kScanTile - 1) / kScanTile;
  return t == 0 ? 1u : (uint32_t)t;
}

uint32_t scan_tiles(uint32_t cap) { return scan_tiles_of(cap); }

__global__ void __launch_bounds__(kScanThreads) scan_u32_kernel(uint32_t* data, uint64_t* status,
                                                               uint64_t* total64,
                                                               const uint32_t* count_dev,
                                                               uint32_t cap, uint32_t* counter,
                                                               DevStatus* st, uint64_t wait_ns) {
  constexpr int W = kScanThreads / 32;
  __shared__ uint32_t s_tile;
  __shared__ uint32_t s_wsum[W];
  __shared__ uint64_t s_prev;
  grid_wait();
  const uint32_t count = (count_dev && *count_dev < cap) ? *count_dev : cap;
  const uint32_t need = scan_tiles_of(count);
  if (threadIdx.x == 0) s_tile = atomicAdd(counter, 1u);
  __syncthreads();
  const uint32_t tile = s_tile;
  if (tile >= need) return;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint64_t i0 = (uint64_t)tile * kScanTile + (uint64_t)threadIdx.x * kScanItems;
  uint32_t v[kScanItems];
  uint32_t sum = 0;
  // A thread's items are consecutive: four 16-byte loads (and stores) when
  // the array is 16-byte aligned and all of them are in range.
  const bool vec = ((reinterpret_cast<uintptr_t>(data) & 15u) == 0) && i0 + kScanItems <= count;
  if (vec) {
    const uint4* p4 = reinterpret_cast<const uint4*>(data + i0);
#pragma unroll
    for (int k = 0; k < kScanItems / 4; ++k) {
      const uint4 q = p4[k];
      v[4 * k] = q.x;
      v[4 * k + 1] = q.y;
      v[4 * k + 2] = q.z;
      v[4 * k + 3] = q.w;
    }
  } else {
#pragma unroll
    for (int k = 0; k < kScanItems; ++k) v[k] = (i0 + k < count) ? data[i0 + k] : 0u;
  }
#pragma unroll
  for (int k = 0; k < kScanItems; ++k) sum += v[k];
  uint32_t x = sum;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) s_wsum[warp] = x;
  __syncthreads();
  if (warp == 0) {
    uint32_t run = 0;
    if (lane == 0) {
      for (int w = 0; w < W; ++w) {
        const uint32_t c = s_wsum[w];
        s_wsum[w] = run;
        run += c;
      }
    }
    run = __shfl_sync(0xffffffffu, run, 0);
    uint64_t prev = 0;
    if (tile == 0) {
      if (lane == 0) st_relaxed(status, kFlagIncl | run);
    } else {
      if (lane == 0) st_relaxed(status + tile, kFlagAgg | run);
      prev = lookback_warp(status, tile, 1, st, wait_ns);
      if (lane == 0) st_relaxed(status + tile, kFlagIncl | (prev + run));
    }
    if (lane == 0) {
      s_prev = prev;
      if (tile == need - 1) {
        const uint64_t total = prev + run;
        if (total64) *total64 = total;
        data[count] = (uint32_t)total;
        if (total >> 32) set_error(st, FMM_ERR_CAPACITY);
      }
    }
  }
  __syncthreads();
  uint64_t off = s_prev + s_wsum[warp] + (x - sum);
  if (vec) {
    uint4* p4 = reinterpret_cast<uint4*>(data + i0);
#pragma unroll
    for (int k = 0; k < kScanItems / 4; ++k) {
      uint4 q;
      q.x = (uint32_t)off;
      off += v[4 * k];
      q.y = (uint32_t)off;
      off += v[4 * k + 1];
      q.z = (uint32_t)off;
      off += v[4 * k + 2];
      q.w = (uint32_t)off;
      off += v[4 * k + 3];
      p4[k] = q;
    }
  } else {
#pragma unroll
    for (int k = 0; k < kScanItems; ++k) {
      if (i0 + k < count) data[i0 + k] = (uint32_t)off;
      off += v[k];
    }
  }
}

void launch_scan_u32(uint32_t* data, const uint32_t* count_dev, uint32_t cap, uint64_t* status,
                     uint32_t* counter, uint64_t* total64, DevStatus* st, uint64_t wait_ns,
                     cudaStream_t s) {
  launch_k(scan_u32_kernel, scan_tiles(cap), kScanThreads, 0, s, data, status, total64, count_dev, cap,
                                                           counter, st, wait_ns);
}

}  // namespace fmm
