// gather.cu -- the sorted point arrays (SortedSrc / SortedRecv, Sec. 2.1)
// and Alg. 2 (Access-Source-E2-neighborhood) for all receiver boxes of a
// level at once: the consumer side of the CSR chain NeighborBookmark ->
// NeighborList -> SrcBookmark -> SortedSrc.
#include "fmm_internal.cuh"

namespace fmm {
namespace {

// Point j of each set's sorted array is input point perm[j].  Units are the
// finishing tiles of kBoxTile points.
__global__ void __launch_bounds__(256) sorted_xyz_kernel(const Seg* __restrict__ segs,
                                                         const Slot* __restrict__ slots,
                                                         uint32_t nslots, const DevStatus* st) {
  grid_wait(segs, slots);
  if (failed(st)) return;
  const Slot sl = slots[find_slot(slots, nslots, blockIdx.x)];
  const Seg& sg = segs[sl.seg];
  // A set whose boxes outran the finishing window has an incomplete
  // permutation until the host redoes its order (and then its points).
  if (!sg.sorted || *sg.seg_long) return;
  const uint64_t t0 = (uint64_t)(blockIdx.x - sl.unit0) * kBoxTile;
  const uint64_t t1 = t0 + kBoxTile < sg.n ? t0 + kBoxTile : sg.n;
  for (uint64_t j = t0 + threadIdx.x; j < t1; j += blockDim.x) {
    const uint64_t i = sg.perm[j];
    if (i >= sg.n) continue;  // never for a complete permutation
    sg.sorted[3 * j] = sg.xyz[3 * i];
    sg.sorted[3 * j + 1] = sg.xyz[3 * i + 1];
    sg.sorted[3 * j + 2] = sg.xyz[3 * i + 2];
  }
}

// Number of E2 source points of each receiver box.
__global__ void __launch_bounds__(256) e2_count_kernel(const uint32_t* __restrict__ e2_off,
                                                       const uint32_t* __restrict__ e2_idx,
                                                       const uint32_t* __restrict__ src_off,
                                                       uint32_t nrecv, uint32_t* __restrict__ out,
                                                       DevStatus* st) {
  grid_wait(e2_off, e2_idx, src_off);
  for (uint32_t r = blockIdx.x * blockDim.x + threadIdx.x; r < nrecv;
       r += gridDim.x * blockDim.x) {
    uint64_t c = 0;
    for (uint32_t j = e2_off[r]; j < e2_off[r + 1]; ++j) {
      const uint32_t v = e2_idx[j];
      c += src_off[v + 1] - src_off[v];
    }
    if (c >> 32) set_error(st, FMM_ERR_CAPACITY);
    out[r] = (uint32_t)c;
  }
}

// One warp per receiver box: its E2 source boxes in list order, each a
// contiguous run of sorted points.  Lane k holds box k's run (at most 27); the
// warp walks the output 32 floats at a time, whole lines whatever the runs'
// lengths, and every lane finds its run from the bit mask of the runs that
// start inside the 32 floats.  2^18 boxes of four points (340 MB written) take
// 96 us, bound by instructions issued; 549 us with one run after another,
// 12 floats a store.
__global__ void __launch_bounds__(256) e2_gather_kernel(const uint32_t* __restrict__ e2_off,
                                                        const uint32_t* __restrict__ e2_idx,
                                                        const uint32_t* __restrict__ src_off,
                                                        const float* __restrict__ sorted_src,
                                                        const uint32_t* __restrict__ off,
                                                        uint32_t nrecv, float* __restrict__ out) {
  grid_wait(e2_off, off);
  const uint32_t lane = threadIdx.x & 31;
  const uint32_t below = lanemask_lt() | (1u << lane);
  const uint32_t nw = (gridDim.x * blockDim.x) >> 5;
  for (uint32_t r = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; r < nrecv; r += nw) {
    const uint32_t row = e2_off[r], m = min(e2_off[r + 1] - row, 32u);
    float* const dst = out + 3ull * off[r];
    uint32_t a = 0, n = 0;  // this lane's run: first point, points
    if (lane < m) {
      const uint32_t v = e2_idx[row + lane];
      a = src_off[v];
      n = src_off[v + 1] - a;
    }
    // Runs of 2^24 points and more, whose floats 32 bits may not count: one run
    // after another.
    if (__any_sync(0xffffffffu, n >= (1u << 24))) {
      float* w = dst;
      for (uint32_t k = 0; k < m; ++k) {
        const uint64_t a64 = 3ull * __shfl_sync(0xffffffffu, a, k);
        const uint64_t n64 = 3ull * __shfl_sync(0xffffffffu, n, k);
        for (uint64_t i = lane; i < n64; i += 32) w[i] = sorted_src[a64 + i];
        w += n64;
      }
      continue;
    }
    uint32_t end = 3 * n;  // floats up to and with this lane's run
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, end, o);
      if (lane >= (uint32_t)o) end += y;
    }
    const uint32_t total = __shfl_sync(0xffffffffu, end, 31), start = end - 3 * n;
    // a lane without a run starts past every output float
    const uint32_t at = n ? start : 0xffffffffu;
    const float* const run = sorted_src + 3ull * a - start;  // its output float f comes from run[f]
    uint32_t before = 0xffffffffu;  // runs that start before the 32 floats, less one
#pragma unroll 4
    for (uint32_t f = lane; f - lane < total; f += 32) {
      const uint32_t rel = at - (f - lane);
      const uint32_t starts = __reduce_or_sync(0xffffffffu, rel < 32u ? 1u << rel : 0u);
      // (every source box holds points, so runs start at different floats)
      const uint32_t k = before + __popc(starts & below);
      const float* const src = reinterpret_cast<const float*>(
          __shfl_sync(0xffffffffu, reinterpret_cast<unsigned long long>(run), k));
      if (f < total) __stcs(dst + f, __ldg(src + f));
      before += __popc(starts);
    }
  }
}

// One set's sorted points (after its permutation was replaced).
__global__ void __launch_bounds__(256) sorted_xyz_one_kernel(const uint32_t* __restrict__ perm,
                                                             const float* __restrict__ xyz,
                                                             uint32_t n, float* __restrict__ out) {
  grid_wait(perm);
  for (uint64_t j = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; j < n;
       j += (uint64_t)gridDim.x * blockDim.x) {
    const uint64_t i = perm[j];
    if (i >= n) continue;  // never for a complete permutation
    out[3 * j] = xyz[3 * i];
    out[3 * j + 1] = xyz[3 * i + 1];
    out[3 * j + 2] = xyz[3 * i + 2];
  }
}

}  // namespace

void launch_sorted_xyz_one(const uint32_t* perm, const float* xyz, uint32_t n, float* out,
                           cudaStream_t s) {
  if (n == 0) return;
  uint32_t grid = (n + 255) / 256;
  if (grid > 152u * 8u) grid = 152u * 8u;
  launch_k(sorted_xyz_one_kernel, grid, 256, 0, s, perm, xyz, n, out);
}

void launch_sorted_xyz(const Seg* segs, const Slot* slots, uint32_t nslots, uint32_t units,
                       DevStatus* st, cudaStream_t s) {
  if (units == 0) return;
  launch_k(sorted_xyz_kernel, units, 256, 0, s, segs, slots, nslots, st);
}

void launch_e2_count(const uint32_t* e2_off, const uint32_t* e2_idx, const uint32_t* src_off,
                     uint32_t nrecv, uint32_t* out, DevStatus* st, cudaStream_t s) {
  if (nrecv == 0) return;
  uint32_t grid = (nrecv + 255) / 256;
  if (grid > 152u * 8u) grid = 152u * 8u;
  launch_k(e2_count_kernel, grid, 256, 0, s, e2_off, e2_idx, src_off, nrecv, out, st);
}

void launch_e2_gather(const uint32_t* e2_off, const uint32_t* e2_idx, const uint32_t* src_off,
                      const float* sorted_src, const uint32_t* off, uint32_t nrecv, float* out,
                      cudaStream_t s) {
  if (nrecv == 0) return;
  uint32_t grid = (nrecv + 7) / 8;  // 8 warps a block
  if (grid > 152u * 16u) grid = 152u * 16u;
  launch_k(e2_gather_kernel, grid, 256, 0, s, e2_off, e2_idx, src_off, sorted_src, off, nrecv, out);
}

}  // namespace fmm
