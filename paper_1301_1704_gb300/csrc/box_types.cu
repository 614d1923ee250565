// box_types.cu -- the source-box types of Alg. 6 (Sec. 3.2) for node J of a
// partition of the space at level l_par: DOMESTIC, EXPORT, IMPORT, ROOT or
// OTHERS for every source box of levels 2..L, from the source tree built
// against itself (its E4 lists are the M2L neighbours).
//
// Readings of the printed algorithm (the oracle takes the same): a box of
// level >= l_par is on J when its ancestor at l_par is owned by J; the
// children of an l_crit box that decide its type are its descendants at
// l_par; the IMPORT marks that one box's thread sets on another survive the
// final assignment (a box not on J is IMPORT when a box on J has it as an
// M2L neighbour, else OTHERS).  No races: a box reads its
// own E4 row instead of being written by its neighbours' threads.
//
// Below l_par a box is on J exactly when its parent is, and its E2 and E4 boxes
// are children of its parent's E2 boxes.  So a box whose parent has all of its
// E2 on its own side has none across J's border, and neither have its
// children: only boxes along the border read their lists, eight lanes a box.
// All levels of 2^20 points, L = 7 (45 M list entries): 83 us in 8 launches, most
// of it launches and chains of dependent loads; 417 us in 11 with a thread
// walking each box's row.
#include "fmm_internal.cuh"

namespace fmm {
namespace {

// on[b] for the boxes of level l_par, from the owners.
__global__ void __launch_bounds__(256) on_node_kernel(const uint32_t* __restrict__ owner,
                                                      uint32_t nbox, uint32_t node,
                                                      uint8_t* __restrict__ on) {
  grid_wait(owner);
  for (uint32_t b = blockIdx.x * blockDim.x + threadIdx.x; b < nbox; b += gridDim.x * blockDim.x)
    on[b] = owner[b] == node;
}

// The boxes of l_crit: bit 0 = some descendant at l_par on J, bit 1 = some
// descendant off J.  Their children at l_par when l_crit < l_par (child
// ranges); the boxes themselves when l_crit = l_par (child = null).
__global__ void __launch_bounds__(256) child_sides_kernel(const uint32_t* __restrict__ child,
                                                          const uint8_t* __restrict__ on_par,
                                                          uint32_t nbox, uint8_t* __restrict__ sides) {
  grid_wait(child, on_par);
  for (uint32_t b = blockIdx.x * blockDim.x + threadIdx.x; b < nbox; b += gridDim.x * blockDim.x) {
    uint32_t s = 0;
    if (!child)
      s = on_par[b] ? 1u : 2u;
    else
      for (uint32_t c = child[b]; c < child[b + 1] && s != 3u; ++c) s |= on_par[c] ? 1u : 2u;
    sides[b] = (uint8_t)s;
  }
}

// Whether any of the list entries idx[a..b) has its byte of `side` pass `hit`,
// for the box of an eight-lane group (uniform over the group); the whole warp
// calls.  (Counted from the row's first entry: a level's entries may end at 2^32 - 1.)
template <class Hit>
__device__ __forceinline__ bool any_entry(const uint32_t* __restrict__ idx, uint32_t a, uint32_t b,
                                          const uint8_t* __restrict__ side, const Hit& hit) {
  const uint32_t lane = threadIdx.x & 31u, l8 = lane & 7u, group = 0xffu << (lane & 24u);
  const uint32_t* const row = idx + a;
  const uint32_t n = b - a;  // at most 189
  bool found = false;
  for (uint32_t i = 0; __any_sync(0xffffffffu, !found && i < n); i += 32) {
    bool h = false;
    if (!found) {
#pragma unroll
      for (int u = 0; u < 4; ++u) {  // the loads of 32 entries together
        const uint32_t j = i + l8 + 8u * u;
        if (j < n) h |= hit(side[row[j]]);
      }
    }
    found |= (__ballot_sync(0xffffffffu, h) & group) != 0;
  }
  return found;
}

// The types of one level, eight lanes a box.  mode 1: l_crit, from `side` (the
// child sides); mode 2: deeper, from `side` (on J); mode 0: all DOMESTIC.
// border_up: per box of the level above, whether its E2 crosses J's border (null:
// unknown, every box looks).  From l_par on also, for the level below (child
// non-null): whether this level's boxes' E2 crosses the border, and the on-J
// flags of their children.
struct TypeArgs {
  const uint32_t *e4_off, *e4_idx, *e2_off, *e2_idx, *parent, *child;
  const uint8_t *side, *on, *border_up;
  uint8_t *border, *on_next, *type;
};

__global__ void __launch_bounds__(256) box_type_kernel(TypeArgs g, uint32_t nbox, int mode) {
  grid_wait();
  const uint32_t l8 = threadIdx.x & 7u;
  const uint32_t g0 = (blockIdx.x * blockDim.x + threadIdx.x) >> 3, groups = (gridDim.x * blockDim.x) >> 3;
  for (uint32_t w0 = g0 & ~3u; w0 < nbox; w0 += groups) {  // (the same rounds for a whole warp)
    const uint32_t k = w0 + (g0 & 3u);
    const bool in = k < nbox;
    uint8_t t = FMM_BOX_DOMESTIC;
    uint32_t a = 0, b = 0;
    if (mode == 1) {
      const uint32_t s = in ? g.side[k] : 0u;
      if (in && s == 1u) {  // all descendants on J
        a = g.e4_off[k];
        b = g.e4_off[k + 1];
      }
      const bool out = any_entry(g.e4_idx, a, b, g.side, [](uint8_t v) { return (v & 2u) != 0; });
      t = !(s & 1u) ? FMM_BOX_IMPORT : (s & 2u) ? FMM_BOX_ROOT : out ? FMM_BOX_EXPORT : t;
    } else if (mode == 2) {
      const bool mine = in && g.side[k] != 0;
      const bool look = in && (!g.border_up || g.border_up[g.parent[k]] != 0);
      const auto other = [mine](uint8_t v) { return (v != 0) != mine; };
      if (look) {
        a = g.e4_off[k];
        b = g.e4_off[k + 1];
      }
      const bool across = any_entry(g.e4_idx, a, b, g.side, other);
      t = mine ? (across ? FMM_BOX_EXPORT : FMM_BOX_DOMESTIC)
               : (across ? FMM_BOX_IMPORT : FMM_BOX_OTHERS);
    }
    if (g.child) {
      const bool mine = in && g.on[k] != 0;
      if (in && (!g.border_up || g.border_up[g.parent[k]] != 0)) {
        a = g.e2_off[k];
        b = g.e2_off[k + 1];
      } else {
        a = b = 0;
      }
      const bool border =
          any_entry(g.e2_idx, a, b, g.on, [mine](uint8_t v) { return (v != 0) != mine; });
      if (in) {
        if (l8 == 0) g.border[k] = border;
        const uint32_t c = g.child[k] + l8;
        if (c < g.child[k + 1]) g.on_next[c] = mine;
      }
    }
    if (in && l8 == 0) g.type[k] = t;
  }
}

uint32_t grid_for(uint32_t n) {
  uint32_t g = (n + 255) / 256;
  if (g > 152u * 8u) g = 152u * 8u;
  return g == 0 ? 1u : g;
}

}  // namespace

void launch_on_node(const uint32_t* owner, uint32_t nbox, uint32_t node, uint8_t* on,
                    cudaStream_t s) {
  if (nbox == 0) return;
  launch_k(on_node_kernel, grid_for(nbox), 256, 0, s, owner, nbox, node, on);
}

void launch_child_sides(const uint32_t* child, const uint8_t* on_par, uint32_t nbox,
                        uint8_t* sides, cudaStream_t s) {
  if (nbox == 0) return;
  launch_k(child_sides_kernel, grid_for(nbox), 256, 0, s, child, on_par, nbox, sides);
}

void launch_box_type(const fmm_tree& t, int l, int mode, const uint8_t* side, const uint8_t* on,
                     const uint8_t* border_up, uint8_t* border, uint8_t* on_next, uint8_t* type,
                     cudaStream_t s) {
  const uint32_t nbox = t.nbox_src[l];
  if (nbox == 0) return;
  TypeArgs g{t.e4_off[l], t.e4_idx[l], t.e2_off[l], t.e2_idx[l], t.parent_src[l],
             on_next ? t.child_src[l] : nullptr, side, on, border_up, border, on_next, type};
  uint32_t grid = (nbox + 31) / 32;  // 32 boxes a block
  if (grid > 152u * 8u) grid = 152u * 8u;
  launch_k(box_type_kernel, grid, 256, 0, s, g, nbox, mode);
}

}  // namespace fmm
