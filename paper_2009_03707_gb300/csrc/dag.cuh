// The DAG of 1-2 gradient pairs (Sec. 3.2, Fig. "msc-max-min-dag" (d)), read straight from
// the packed gradient words.
//
// Nodes are 1-cells (1-saddles and 1-cells paired with a quad) and 2-saddles.  For a 1-cell e,
// each cofacet quad q other than e's own partner gives an out-edge: to q itself if q is
// critical (a 2-saddle), to the 1-cell that q is paired with if q is paired with a facet, and
// nothing if q is paired with a cube.  Following an out-edge walks a V-path backwards, so
// traversals move against the gradient (Sec. 3.5).  Out-degree <= 4 (Sec. 3.2).
//
// A 1-cell is named by its owner vertex and axis: handle = (vertex index << 2) | axis, where
// the cell is (2x+1,2y,2z), (2x,2y+1,2z) or (2x,2y,2z+1) for axis 0, 1, 2.  A 2-saddle target
// is named by its owner vertex and slot.  All index arithmetic is 32-bit: a plan's cell ids
// fit in 32 bits, so its vertex count is below 2^29.
#pragma once

#include "geom.cuh"

namespace msc {

__host__ __device__ __forceinline__ uint32_t edge_handle(uint32_t v, int axis) { return (v << 2) | uint32_t(axis); }

struct Vtx {
    int x, y, z;
};

__host__ __device__ __forceinline__ Vtx vtx_of(const Geom& g, uint32_t v) {
    Vtx r;
    const uint32_t q = g.div_nx.div(v);
    r.x = int(v - q * uint32_t(g.nx));
    r.z = int(g.div_ny.div(q));
    r.y = int(q - uint32_t(r.z) * uint32_t(g.ny));
    return r;
}

__host__ __device__ __forceinline__ uint32_t vid32(const Geom& g, int x, int y, int z) {
    return uint32_t(x) + uint32_t(g.nx) * (uint32_t(y) + uint32_t(g.ny) * uint32_t(z));
}

// Slot of the 1-cell along `axis` in its owner's word: a=1 (slot 1), b=1 (slot 2), c=1 (slot 4).
__host__ __device__ __forceinline__ int edge_slot(int axis) { return 1 << axis; }

// The i-th of three values, without an indexed array (which would live in local memory).
__host__ __device__ __forceinline__ int pick3(int i, int a0, int a1, int a2) { return i == 0 ? a0 : i == 1 ? a1 : a2; }

// Per-node record of every reachable 1-cell that is not a 1-saddle: whether the node is a dead
// end, a branch point (out-degree > 1), or else its one successor.  A 1-cell successor is its
// handle; a 2-saddle successor has bit 31 set and (owner << 2 | even axis).  Records are stored
// one plane per axis (info_index), so a row of cells writes a contiguous run.
constexpr uint32_t INFO_DEAD = 0xFFFFFFFFu;
__host__ __device__ __forceinline__ uint32_t info_index(const Geom& g, uint32_t handle) {
    return (handle & 3u) * uint32_t(g.nverts) + (handle >> 2);
}
constexpr uint32_t INFO_BRANCH = 0xFFFFFFFEu;

}  // namespace msc
