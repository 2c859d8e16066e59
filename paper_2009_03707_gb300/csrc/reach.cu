// (a4) Saddle-saddle reachability and (a5, first half) junction nodes.
//
// Sec. 3.2 and Sec. 3.5 "Saddle-Saddle reachability": the 1-cells reachable from the
// 1-saddles in the DAG of 1-2 gradient pairs, level by level; the traversal ends when a level
// adds nothing.  The paper runs a frontier BFS (expand, then stream-compact a 4x candidate
// array).  Here the same level sets are computed by pulling instead of pushing, on the 1-cell
// bitmap itself:
//
//  * A 1-cell e has in-edges only if it is paired with a quad q; they come from the other three
//    facets of q (a facet f of q has the out-edge f -> e because q is a cofacet of f that is not
//    f's own partner).  So with R_k the set reached within k levels,
//        R_{k+1} = R_k  u  { e paired with a quad q : some other facet of q is in R_k },
//    R_0 = the 1-saddles.  That is one data-parallel sweep per level over the bitmap rows:
//    for each 32-cell word, four pairing-direction masks select which neighbouring rows (shifted
//    by one bit where the step is along x) feed it.  Sweep k+1 changes the bitmap iff BFS level
//    k+1 is non-empty, so the level count is the paper's.
//  * Every access is a coalesced word of a row, where a queue frontier scatters a 4-byte access
//    per node over the whole grid.  One loop iteration is two sweeps (A -> B, B -> A, so the
//    set always ends in A) and a one-thread decision kernel; the loop is a conditional WHILE node
//    when the pipeline runs as a graph, so no level needs a host round trip.
//  * A sweep costs the same however few cells it adds, and most levels add few (512^3 blob field:
//    153 levels, 7.9 M new cells at level 1, 1.4 M at level 11, then 3 % fewer each; 256^3 GRF: 14
//    levels, 8.4 M at level 2, 0.1 M at level 6).  So the sweeps stop once a level is sparse, the
//    cells of that last level become a queue, and the other levels are pushed: each new cell's
//    out-edges set their targets' bits and append the targets that were not set.  The level sets are
//    the same.  Large grids push with the whole device while a level is large; the last levels --
//    and on a small grid all of them -- run in one kernel of one thread-block cluster, whose
//    hardware barrier between levels costs far less than a kernel boundary.
//    Reachability stage of a replayed pass, against sweeps for every level: 512^3 blobs 15.9 -> 3.8 ms,
//    256^3 GRF 0.395 -> 0.200, 61 x 75 x 49 GRF 0.102 -> 0.064, 32^3 lattice (19 levels) 0.127 -> 0.061 (0.74
//    and 0.095 ms of the first two were the bitmaps, which a replay makes in the gradient stage since).
//
// Sec. 3.3 / Sec. 3.5 "Gradient path counting": a junction is a reachable 1-cell that is not a
// 1-saddle and has out-degree > 1.  One warp per bitmap word (a lane per 1-cell) evaluates the
// out-edges of each reachable cell, marks junctions, and records each node's successor for the
// path tracer.  Junctions are stream-compacted in cell-id order (scan.cuh), which also gives
// O(1) ranks for the minor's matrix indices.
#include <cooperative_groups.h>

#include "dag.cuh"
#include "scan.cuh"
#include "word_bitmaps.cuh"

namespace cg = cooperative_groups;

namespace msc {

namespace {

constexpr int THREADS = 256;

// Word addressing of the bitmaps, per thread: the 1-cell row layout is
//   edge_word(z, c, y, b, w) = z*sz + y*sy + off[axis] + w   (sz = 4 ny W, sy = 2 W),
// and the quad bitmaps hold one row per (even axis k, z, y): quad_word = ((k nz + z) ny + y) W + w.
// Word indices are 32-bit: a plan's bitmaps have fewer than 2^28 words (nverts < 2^29).
struct Rows {
    int w, y, z;  // this thread's word: x = 32w .. 32w+31 of row (y, z)
    int W, ny, nz;
    int sy, sz;   // 1-cell layout strides
    int base;     // z*sz + y*sy + w
    int qbase;    // (z ny + y) W + w
    int qplane;   // nz ny W
    __device__ Rows(const Geom& g, int64_t t) {
        const uint32_t q = g.div_W.div(uint32_t(t));
        w = int(uint32_t(t) - q * uint32_t(g.W));
        const uint32_t q2 = g.div_ny.div(q);
        y = int(q - q2 * uint32_t(g.ny));
        z = int(q2);
        W = g.W;
        ny = g.ny;
        nz = g.nz;
        sy = 2 * W;
        sz = 4 * ny * W;
        base = z * sz + y * sy + w;
        qbase = (z * ny + y) * W + w;
        qplane = nz * ny * W;
    }
    template <int AX>
    __device__ __forceinline__ int edge(int dy, int dz) const {
        return base + (AX == 1 ? W : AX == 2 ? 2 * ny * W : 0) + dy * sy + dz * sz;
    }
    template <int DY, int DZ>
    __device__ __forceinline__ bool in_range() const {
        return (DY >= 0 || y > 0) && (DY <= 0 || y < ny - 1) && (DZ >= 0 || z > 0) && (DZ <= 0 || z < nz - 1);
    }
};

// Bits of a row word at index `at` (the word of x = 32w..), shifted so that bit i refers to x + DX.
template <int DX>
__device__ __forceinline__ uint32_t shifted(const uint32_t* __restrict__ R, int at, const Rows& r) {
    const uint32_t mid = R[at];
    if (DX == 0) return mid;
    if (DX > 0) return __funnelshift_r(mid, r.w + 1 < r.W ? R[at + 1] : 0u, 1);
    return __funnelshift_l(r.w > 0 ? R[at - 1] : 0u, mid, 1);
}

// Reach bits of the AX-cells owned by vertex (x + DX, y + DY, z + DZ); 0 outside the grid.
template <int AX, int DX, int DY, int DZ>
__device__ __forceinline__ uint32_t reach_row(const uint32_t* __restrict__ R, const Rows& r) {
    if (!r.in_range<DY, DZ>()) return 0;
    return shifted<DX>(R, r.edge<AX>(DY, DZ), r);
}

// Cells of axis A whose partner is the quad on side S along axis B (mask m) and that have a
// facet of that quad in R: the quad's other facets are the parallel A-cell one vertex along
// S u_B and the two B-cells at the ends of the A-cell, owned by v (+ u_A) (- u_B if S < 0).
template <int A, int B, int S>
__device__ __forceinline__ uint32_t pull(uint32_t m, const uint32_t* __restrict__ R, const Rows& r) {
    if (!m) return 0;
    constexpr int back = S < 0 ? 1 : 0;
    constexpr int ux = A == 0, uy = A == 1, uz = A == 2, bx = B == 0, by = B == 1, bz = B == 2;
    const uint32_t p = reach_row<A, S * bx, S * by, S * bz>(R, r) |
                       reach_row<B, ux - back * bx, uy - back * by, uz - back * bz>(R, r) |
                       reach_row<B, -back * bx, -back * by, -back * bz>(R, r);
    return m & p;
}

template <int A>
__device__ __forceinline__ uint32_t sweep_word(const Rows& r, const uint4* __restrict__ masks,
                                           const uint32_t* __restrict__ Rin, uint32_t* __restrict__ Rout) {
    constexpr int B1 = A == 0 ? 1 : 0, B2 = A == 2 ? 1 : 2;
    const int i = r.edge<A>(0, 0);
    const uint32_t cur = Rin[i];
    const uint4 m = masks[i];
    uint32_t add = 0;
    if ((m.x | m.y | m.z | m.w) & ~cur)
        add = pull<A, B1, -1>(m.x & ~cur, Rin, r) | pull<A, B1, 1>(m.y & ~cur, Rin, r) |
              pull<A, B2, -1>(m.z & ~cur, Rin, r) | pull<A, B2, 1>(m.w & ~cur, Rin, r);
    Rout[i] = cur | add;
    return __popc(add);
}

// One level: Rout = Rin | cells whose partner quad has another facet in Rin.  A thread takes one
// vertex-row word at a time for all three axes (one neighbourhood check, three independent chains
// of loads).  Adds the number of new cells to *added.
// Rows (y, z) are stamped with 1 + the last sweep that changed them (1: the start).  A cell's
// predecessors lie within one step in y and z, so a row none of whose 3 x 3 neighbour rows changed
// in the previous sweep cannot change now; it is skipped, Rout included: that buffer already
// holds the row's value from two sweeps ago, which is still its value.  Fronts that move slowly
// through a large grid (many levels) then cost only the rows near the front.
__global__ void __launch_bounds__(THREADS, 4) reach_sweep(Geom g, const uint4* __restrict__ masks,
                                                       const uint32_t* __restrict__ Rin, uint32_t* __restrict__ Rout,
                                                       uint32_t* __restrict__ stamp, const Summary* __restrict__ sum,
                                                       int parity, uint32_t* __restrict__ added) {
    if (!sum->loop_flag[3]) return;  // a replayed pass has swept enough
    const int64_t nrw = int64_t(g.nz) * g.ny * g.W;
    const uint32_t k = 2u * uint32_t(sum->sweep_iters) + 1u + uint32_t(parity);  // this sweep
    uint32_t grew = 0;
    // grid-stride over the row words (a few tiles of THREADS words per CTA): a sweep in which few
    // rows are near a front then costs fewer CTA launches for the rest
    for (int64_t t = int64_t(blockIdx.x) * THREADS + threadIdx.x; t < nrw; t += int64_t(gridDim.x) * THREADS) {
        const Rows r(g, t);
        uint32_t recent = 0;
        for (int dz = -1; dz <= 1; ++dz)
            for (int dy = -1; dy <= 1; ++dy) {
                const int y = r.y + dy, z = r.z + dz;
                if (y >= 0 && y < g.ny && z >= 0 && z < g.nz) recent = max(recent, stamp[int64_t(z) * g.ny + y]);
            }
        if (recent >= k) {
            const uint32_t n = sweep_word<0>(r, masks, Rin, Rout) + sweep_word<1>(r, masks, Rin, Rout) +
                               sweep_word<2>(r, masks, Rin, Rout);
            if (n) stamp[int64_t(r.z) * g.ny + r.y] = k + 1;
            grew += n;
        }
    }
    grew = __reduce_add_sync(0xFFFFFFFFu, grew);
    __shared__ uint32_t part[THREADS / 32];
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = grew;
    __syncthreads();
    if (threadIdx.x == 0) {
        uint32_t n = 0;
        for (int w = 0; w < THREADS / 32; ++w) n += part[w];
        if (n) atomicAdd(added, n);
    }
}

// Level 0: the 1-saddles, if there are any.
__global__ void reach_start(Summary* sum) {
    sum->levels = sum->counts[1] > 0 ? 1 : 0;
    sum->loop_flag[3] = 1;  // the sweeps go on
}

// A replayed pass pushes a level of up to four times the cells at which a level counts as sparse without asking
// for more sweeps: a sweep iteration that other fields leave unused costs them 5 us, and a level just above
// the line costs little more pushed than swept (see follow_levels).
__device__ __forceinline__ uint32_t dense_above(uint32_t sparse) { return 4 * sparse; }

// End of one loop iteration (two sweeps): the non-empty levels found, and the continue decision: while
// the second sweep still added more than `sparse` cells, up to the iteration cap.  The cells it added
// are what the pushed levels start from.  `last`: there is no further iteration, whatever it added.
__global__ void reach_decide(Summary* sum, uint32_t sparse, int last, int64_t max_iter, cudaGraphConditionalHandle h,
                             int use_handle) {
    if (!sum->loop_flag[3]) return;
    const uint32_t c0 = sum->loop_flag[0], c1 = sum->loop_flag[1];
    sum->loop_flag[0] = 0;
    sum->loop_flag[1] = 0;
    ++sum->sweep_iters;
    sum->levels += (c0 ? 1 : 0) + (c1 ? 1 : 0);
    bool more = c1 > sparse;
    if (last) {
        sum->dense = c1 > dense_above(sparse) ? 1u : 0u;
        more = false;
    }
    uint32_t left = more ? 0u : c1;
    if (c1 && int64_t(sum->levels) >= max_iter) {
        atomicOr(&sum->status, uint32_t(ST_ITER));
        more = false;
        left = 0;
    }
    sum->push_count[3] = left;
    sum->loop_flag[3] = more ? 1u : 0u;
    if (use_handle) cudaGraphSetConditional(h, more ? 1u : 0u);
}

// ---- sparse levels ---------------------------------------------------------------------------
struct PushArgs {
    Geom g;
    const uint32_t* words;
    uint32_t* reached;     // the bitmap A
    uint32_t* queue[2];    // handles of a level's new cells
    uint32_t cap;          // room in each
    uint32_t* status;
};

// The targets of cell h's out-edges that were not reached before, marked; returns how many.  The (up to
// four) atomics go out together, so a level waits for memory once.  LOOK: read the targets' bits
// first, together too, and mark only those not set -- for large levels, which are bound by the number
// of atomics and not by one round trip more.
// The three gradient words that name the targets (the cell's owner and the vertices one step back
// along the two other axes) are loaded together and the four out-edges computed without branches, for
// the same reason.
template <bool LOOK>
__device__ __forceinline__ int push_cell(const PushArgs& a, uint32_t h, uint32_t out[4]) {
    const Geom& g = a.g;
    const uint32_t nx = uint32_t(g.nx), ny = uint32_t(g.ny), nz = uint32_t(g.nz), W = uint32_t(g.W);
    const uint32_t v = h >> 2;
    const int axis = int(h & 3u);
    const uint32_t row = g.div_nx.div(v);
    const uint32_t x = v - row * nx, z = g.div_ny.div(row), y = row - z * ny;
    const int bA = axis == 2 ? 0 : axis + 1, bB = axis == 0 ? 2 : axis - 1;
    const uint32_t cA = pick3(bA, x, y, z), cB = pick3(bB, x, y, z);
    const uint32_t nA = pick3(bA, nx, ny, nz), nB = pick3(bB, nx, ny, nz);
    const uint32_t sA = pick3(bA, 1u, nx, nx * ny), sB = pick3(bB, 1u, nx, nx * ny);
    const uint32_t w_own = __ldg(a.words + v);
    const uint32_t w_A = cA > 0 ? __ldg(a.words + (v - sA)) : 0u;
    const uint32_t w_B = cB > 0 ? __ldg(a.words + (v - sB)) : 0u;
    const uint32_t own = slot_code(w_own, 1 << axis);
    uint32_t* at[4];
    uint32_t bit[4], old[4], target[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int b = i < 2 ? bA : bB;
        const bool plus = i & 1;
        const uint32_t cb = i < 2 ? cA : cB, nb = i < 2 ? nA : nB;
        const int other = 3 - axis - b;  // the quad's even axis
        const uint32_t qc = slot_code(plus ? w_own : (i < 2 ? w_A : w_B), (1 << axis) | (1 << b));
        const int k = int(qc - 1) >> 1;  // the axis along which the quad is paired
        const bool edge = (plus ? cb + 1 < nb : cb > 0) && own != uint32_t(1 + 2 * b + (plus ? 1 : 0)) && qc != 0 && k != other;
        // the facet's owner: the quad's (one step back along b on the - side), one step on along k if
        // the quad is paired on that side
        const int back = plus ? 0 : 1, on = (qc & 1u) ? 0 : 1;
        const uint32_t tx = x - (b == 0 ? back : 0) + (k == 0 ? on : 0), ty = y - (b == 1 ? back : 0) + (k == 1 ? on : 0),
                       tz = z - (b == 2 ? back : 0) + (k == 2 ? on : 0);
        const int t_axis = k == axis ? b : axis;
        target[i] = edge_handle(tx + nx * (ty + ny * tz), t_axis);
        bit[i] = edge ? 1u << (tx & 31u) : 0u;
        at[i] = a.reached + (edge ? (((tz * 2 + (t_axis == 2)) * ny + ty) * 2 + (t_axis == 1)) * W + (tx >> 5) : 0u);
        old[i] = 0;
    }
    if (LOOK) {
#pragma unroll
        for (int i = 0; i < 4; ++i)
            if (bit[i]) old[i] = __ldcg(at[i]);
    }
#pragma unroll
    for (int i = 0; i < 4; ++i)
        if (bit[i] & ~old[i]) old[i] = atomicOr(at[i], bit[i]);
    int n = 0;
#pragma unroll
    for (int i = 0; i < 4; ++i)
        if (bit[i] & ~old[i]) out[n++] = target[i];
    return n;
}

// Exclusive place of n items among the block's (threads in order), and their sum in *total.
template <int T>
__device__ __forceinline__ uint32_t block_prefix(uint32_t n, uint32_t* total) {
    __shared__ uint32_t part[T / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t incl = n;
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
        if (lane >= o) incl += y;
    }
    __syncthreads();  // the last call's sums have been read
    if (lane == 31) part[warp] = incl;
    __syncthreads();
    uint32_t w = lane < T / 32 ? part[lane] : 0u;  // every warp scans the warps' sums for itself
    const uint32_t own = w;
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, w, o);
        if (lane >= o) w += y;
    }
    *total = __shfl_sync(0xFFFFFFFFu, w, T / 32 - 1);
    return __shfl_sync(0xFFFFFFFFu, w - own, warp) + incl - n;
}

// The cells of one row word's axis that are set in `bits`, to the queue.
__device__ __forceinline__ void emit_row(const PushArgs& a, const Rows& r, int axis, uint32_t bits, uint32_t* queue, uint32_t& at) {
    const uint32_t v0 = vid32(a.g, r.w * 32, r.y, r.z);
    for (; bits; bits &= bits - 1, ++at)
        if (at < a.cap) queue[at] = edge_handle(v0 + uint32_t(__ffs(bits) - 1), axis);
}

// The last swept level's cells (in A but not in B) to queue 0, *count of them (known beforehand).
__global__ void __launch_bounds__(THREADS) reach_frontier(PushArgs a, const uint32_t* __restrict__ A, const uint32_t* __restrict__ B,
                                                          const uint32_t* __restrict__ count, uint32_t* __restrict__ cursor) {
    const uint32_t left = *count;
    if (!left) return;
    if (left > a.cap && threadIdx.x == 0) atomicOr(a.status, ST_RETRY);
    const int64_t nrw = int64_t(a.g.nz) * a.g.ny * a.g.W;
    __shared__ uint32_t base;
    for (int64_t t0 = int64_t(blockIdx.x) * THREADS; t0 < nrw; t0 += int64_t(gridDim.x) * THREADS) {
        const int64_t t = t0 + threadIdx.x;
        const Rows r(a.g, t < nrw ? t : nrw - 1);
        uint32_t d[3] = {0, 0, 0};
        if (t < nrw) {
            const int e[3] = {r.edge<0>(0, 0), r.edge<1>(0, 0), r.edge<2>(0, 0)};
#pragma unroll
            for (int k = 0; k < 3; ++k) d[k] = A[e[k]] & ~B[e[k]];
        }
        uint32_t total;
        uint32_t at = block_prefix<THREADS>(__popc(d[0]) + __popc(d[1]) + __popc(d[2]), &total);
        if (!total) continue;  // block-uniform
        if (threadIdx.x == 0) base = atomicAdd(cursor, total);
        __syncthreads();
        at += base;
#pragma unroll
        for (int k = 0; k < 3; ++k) emit_row(a, r, k, d[k], a.queue[0], at);
    }
}

// One pushed level by the whole device: the queue `from` (count push_count[in]) to the other one (count
// push_count[out]).
__global__ void __launch_bounds__(THREADS) reach_push(PushArgs a, Summary* sum, int from, int in, int out) {
    if (block_retrying(a.status)) return;
    const uint32_t n = sum->push_count[in];
    __shared__ uint32_t base;
    for (uint64_t b = uint64_t(blockIdx.x) * THREADS; b < n; b += uint64_t(gridDim.x) * THREADS) {
        const uint64_t i = b + threadIdx.x;
        uint32_t next[4];
        const int m = i < n ? push_cell<true>(a, a.queue[from][i], next) : 0;
        uint32_t total;
        uint32_t at = block_prefix<THREADS>(uint32_t(m), &total);
        if (threadIdx.x == 0) {
            base = total ? atomicAdd(&sum->push_count[out], total) : 0u;
            if (base + total > a.cap) atomicOr(a.status, ST_RETRY);  // the queue is full: the pass sweeps instead
        }
        __syncthreads();
        at += base;
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (k < m && at + k < a.cap) a.queue[from ^ 1][at + k] = next[k];
    }
}

// End of PUSHES pushed levels: those that were not empty, and whether the last one is still too large
// for one cluster.  An iteration takes push_count[3] in and leaves its levels in 0, 1, 2 and 4.
constexpr int PUSHES = 4;
__global__ void reach_push_decide(Summary* sum, uint32_t few, uint32_t sparse, int64_t max_iter, cudaGraphConditionalHandle h, int use_handle) {
    const uint32_t c[PUSHES] = {sum->push_count[0], sum->push_count[1], sum->push_count[2], sum->push_count[4]};
    uint32_t left = c[PUSHES - 1];
    ++sum->push_iters;
    for (int i = 0; i < PUSHES; ++i) {
        sum->levels += c[i] ? 1 : 0;
        if (sum->dense && c[i] > dense_above(sparse)) ++sum->dense;
        if ((i & 1) && c[i] && int64_t(sum->levels) >= max_iter) {  // checked at every second level, as by the sweeps
            atomicOr(&sum->status, uint32_t(ST_ITER));
            left = 0;
            break;
        }
    }
    for (int i = 0; i < 5; ++i) sum->push_count[i] = 0;
    if (pass_retrying(&sum->status)) left = 0;
    sum->push_count[3] = left;
    const bool more = left > few;
    sum->loop_flag[3] = more ? 1u : 0u;
    if (use_handle) cudaGraphSetConditional(h, more ? 1u : 0u);
}

// The remaining levels in one cluster of thread blocks: queue 0 holds the current level, or (`all`)
// the levels start here, from every cell of the bitmap (the 1-saddles).  The counts live in the first
// block's shared memory; a cluster barrier ends each level.
constexpr int TAIL_THREADS = 1024;
__global__ void __launch_bounds__(TAIL_THREADS, 1) reach_tail(PushArgs a, Summary* sum, int all, uint32_t sparse, int64_t max_iter) {
    cg::cluster_group cluster = cg::this_cluster();
    __shared__ uint32_t counts[3], state[2], alone[TAIL_THREADS];
    __shared__ uint64_t state_levels, block_levels;
    __shared__ uint32_t base, level_n;
    uint32_t* const shared_counts = cluster.map_shared_rank(counts, 0);
    const uint32_t rank = cluster.block_rank(), size = cluster.num_blocks();
    if (threadIdx.x < 3) counts[threadIdx.x] = 0;
    cluster.sync();
    uint32_t n = sum->push_count[3];
    if (all) {
        const int64_t nrw = int64_t(a.g.nz) * a.g.ny * a.g.W;
        for (int64_t t0 = int64_t(rank) * TAIL_THREADS; t0 < nrw; t0 += int64_t(size) * TAIL_THREADS) {
            const int64_t t = t0 + threadIdx.x;
            const Rows r(a.g, t < nrw ? t : nrw - 1);
            uint32_t d[3] = {0, 0, 0};
            if (t < nrw) {
                d[0] = a.reached[r.edge<0>(0, 0)];
                d[1] = a.reached[r.edge<1>(0, 0)];
                d[2] = a.reached[r.edge<2>(0, 0)];
            }
            uint32_t total;
            uint32_t at = block_prefix<TAIL_THREADS>(__popc(d[0]) + __popc(d[1]) + __popc(d[2]), &total);
            if (!total) continue;  // block-uniform
            if (threadIdx.x == 0) base = atomicAdd(&shared_counts[2], total);
            __syncthreads();
            at += base;
#pragma unroll
            for (int k = 0; k < 3; ++k) emit_row(a, r, k, d[k], a.queue[0], at);
        }
        cluster.sync();
        if (threadIdx.x == 0) level_n = shared_counts[2];
        __syncthreads();
        n = level_n;
        if (n > a.cap && threadIdx.x == 0) atomicOr(a.status, ST_RETRY);
    }
    // level k reads queue k & 1 and counts its new cells in counts[k % 3]; counts[(k + 1) % 3], last read
    // before level k - 1 began, is cleared for the next level
    uint64_t levels = sum->levels;
    uint32_t dense = 0;  // levels that sweeps should have taken
    cluster.sync();  // every block has read the counts and the level number
    for (int k = 0; n;) {
        n = min(n, a.cap);
        if (n <= TAIL_THREADS) {
            // the first block goes on alone, with the level in its shared memory and no barrier but its
            // own, until the levels end or one outgrows its threads (that one goes to the queue); the others
            // wait at the cluster's barrier
            if (rank == 0) {
                uint32_t h = threadIdx.x < n ? a.queue[k & 1][threadIdx.x] : 0u;
                for (;;) {
                    uint32_t next[4], total;
                    const int m = threadIdx.x < n ? push_cell<false>(a, h, next) : 0;
                    const uint32_t at = block_prefix<TAIL_THREADS>(uint32_t(m), &total);
                    ++k;
                    n = total;
                    levels += n ? 1 : 0;
                    if (!(k & 1) && n && int64_t(levels) >= max_iter) {  // at every second level, as the sweeps
                        if (threadIdx.x == 0) atomicOr(a.status, ST_ITER);
                        n = 0;
                    }
                    if (!n) break;
                    // a level that goes on here is whole in shared memory, whatever the queues' room
                    uint32_t* to = n > TAIL_THREADS ? a.queue[k & 1] : alone;
                    const uint32_t room = n > TAIL_THREADS ? a.cap : uint32_t(TAIL_THREADS);
                    if (n > room && threadIdx.x == 0) atomicOr(a.status, ST_RETRY);
#pragma unroll
                    for (int j = 0; j < 4; ++j)
                        if (j < m && at + j < room) to[at + j] = next[j];
                    if (n > TAIL_THREADS) break;
                    __syncthreads();
                    h = threadIdx.x < n ? alone[threadIdx.x] : 0u;
                }
                if (threadIdx.x == 0) {
                    state[0] = n;
                    state[1] = uint32_t(k);
                    state_levels = levels;
                    counts[0] = counts[1] = counts[2] = 0;
                }
            }
            cluster.sync();
            if (threadIdx.x == 0) {
                level_n = *cluster.map_shared_rank(&state[0], 0);
                base = *cluster.map_shared_rank(&state[1], 0);
                block_levels = *cluster.map_shared_rank(&state_levels, 0);
            }
            __syncthreads();
            n = level_n;
            k = int(base);
            levels = block_levels;
            cluster.sync();  // the first block may change its state again
            continue;
        }
        if (rank == 0 && threadIdx.x == 0) counts[(k + 1) % 3] = 0;
        const uint32_t* from = a.queue[k & 1];
        uint32_t* to = a.queue[(k & 1) ^ 1];
        for (uint32_t b = rank * TAIL_THREADS; b < n; b += size * TAIL_THREADS) {
            uint32_t next[4];
            const int m = b + threadIdx.x < n ? push_cell<false>(a, from[b + threadIdx.x], next) : 0;
            uint32_t total;
            uint32_t at = block_prefix<TAIL_THREADS>(uint32_t(m), &total);
            if (!total) continue;  // block-uniform
            if (threadIdx.x == 0) {
                base = atomicAdd(&shared_counts[k % 3], total);
                if (base + total > a.cap) atomicOr(a.status, ST_RETRY);
            }
            __syncthreads();
            at += base;
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if (j < m && at + j < a.cap) to[at + j] = next[j];
        }
        cluster.sync();
        if (threadIdx.x == 0) level_n = shared_counts[k % 3];
        __syncthreads();
        n = level_n;
        ++k;
        levels += n ? 1 : 0;
        dense += n > dense_above(sparse) ? 1 : 0;
        if (!(k & 1) && n && int64_t(levels) >= max_iter) {
            if (rank == 0 && threadIdx.x == 0) atomicOr(a.status, ST_ITER);
            n = 0;
        }
    }
    if (rank == 0 && threadIdx.x == 0) {
        sum->levels = levels;
        if (sum->dense) sum->dense += dense;
    }
    cluster.sync();  // no block leaves while others read the first one's counts
}

// Down-quad bits of the quads with even axis K owned by vertex (x + DX, y + DY, z + DZ).
template <int K, int DX, int DY, int DZ>
__device__ __forceinline__ uint32_t quad_row(const uint32_t* __restrict__ qdown, const Rows& r) {
    if (!r.in_range<DY, DZ>()) return 0;
    return shifted<DX>(qdown, K * r.qplane + r.qbase + DY * r.W + DZ * r.ny * r.W, r);
}

// The bitmap words one axis of a vertex-row word needs: reached and critical bits, the four
// partner masks, and the down-quad rows of the quads on the - / + side along the first / second
// other axis (the order of the masks).
struct AxisIn {
    uint32_t vis, crit;
    uint4 m;
    uint32_t q[4];
};

template <int A>
__device__ __forceinline__ AxisIn load_axis(const Geom& g, const Rows& r, const uint32_t* __restrict__ visited,
                                            const uint4* __restrict__ masks, const uint32_t* __restrict__ qdown,
                                            const uint32_t* __restrict__ crit_bits) {
    constexpr int B1 = A == 0 ? 1 : 0, B2 = A == 2 ? 1 : 2;
    constexpr int K1 = 3 - A - B1, K2 = 3 - A - B2;  // even axes of the quads along B1, B2
    AxisIn in;
    in.vis = visited[r.edge<A>(0, 0)];
    in.crit = crit_bits[g.slot_word(1 << A, r.z, r.y, r.w)];
    in.m = masks[r.edge<A>(0, 0)];
    in.q[0] = quad_row<K1, -(B1 == 0), -(B1 == 1), -(B1 == 2)>(qdown, r);
    in.q[1] = quad_row<K1, 0, 0, 0>(qdown, r);
    in.q[2] = quad_row<K2, -(B2 == 0), -(B2 == 1), -(B2 == 2)>(qdown, r);
    in.q[3] = quad_row<K2, 0, 0, 0>(qdown, r);
    return in;
}

// Gradient word of the vertex one step down axis B from v (0 off the grid), loaded for a whole
// row of lanes at once.
template <int B>
__device__ __forceinline__ uint32_t minus_word(const Geom& g, const uint32_t* __restrict__ words, const Rows& r, int x,
                                               uint32_t v) {
    if (x >= g.nx) return 0u;
    if (B == 0) return x > 0 ? words[v - 1] : 0u;
    if (B == 1) return r.y > 0 ? words[v - uint32_t(g.nx)] : 0u;
    return r.z > 0 ? words[v - uint32_t(g.nx) * uint32_t(g.ny)] : 0u;
}

// The A-cells of one vertex-row word (a lane per cell).  The out-edges of a 1-cell e go through
// its cofacet quads other than its partner that are critical or paired with a facet, so with the
// down-quad rows the out-degree is a popcount.  Reachable cells that are not 1-saddles get their
// info record; a single successor is decoded from the one quad it goes through, whose owner is v
// itself (+ side) or v one step down the quad's other axis (- side, gradient word w_b1 / w_b2).
template <int A>
__device__ __forceinline__ void classify_axis(const Geom& g, const Rows& r, int lane, int x, uint32_t v,
                                              const AxisIn& in, uint32_t w_self, uint32_t w_b1, uint32_t w_b2,
                                              uint32_t* __restrict__ info, uint32_t* __restrict__ junc,
                                              unsigned long long& cnt) {
    constexpr int B1 = A == 0 ? 1 : 0, B2 = A == 2 ? 1 : 2;
    // every record of the row is written (whole sectors: no read-modify-write in L2); cells
    // that are not reached, or are 1-saddles, get a dead-end record that nothing reads
    if (lane == 0) cnt += __popc(in.vis);
    const uint32_t partner = ((in.m.x >> lane) & 1u) | (((in.m.y >> lane) & 1u) << 1) |
                             (((in.m.z >> lane) & 1u) << 2) | (((in.m.w >> lane) & 1u) << 3);
    const uint32_t out = (((in.q[0] >> lane) & 1u) | (((in.q[1] >> lane) & 1u) << 1) |
                          (((in.q[2] >> lane) & 1u) << 2) | (((in.q[3] >> lane) & 1u) << 3)) &
                         ~partner;
    const int n = __popc(out);
    const bool mine = ((in.vis & ~in.crit) >> lane) & 1u;
    uint32_t rec = INFO_DEAD;
    if (mine) {
        rec = n == 0 ? INFO_DEAD : INFO_BRANCH;
        if (n == 1) {
            const int sel = __ffs(out) - 1;
            const int b = sel < 2 ? B1 : B2;
            const int k = 3 - A - b;  // the quad's even axis
            const bool plus = sel & 1;
            uint32_t ov = v, ow = w_self;
            if (!plus) {
                ov -= b == 0 ? 1u : b == 1 ? uint32_t(g.nx) : uint32_t(g.nx) * uint32_t(g.ny);
                ow = sel < 2 ? w_b1 : w_b2;
            }
            const uint32_t qc = slot_code(ow, 7 ^ (1 << k));
            if (qc == 0) {
                rec = 0x80000000u | (ov << 2) | uint32_t(k);  // a 2-saddle
            } else {                                           // the facet the quad is paired with
                const int kk = int(qc - 1) >> 1;
                if (!(qc & 1u)) ov += kk == 0 ? 1u : kk == 1 ? uint32_t(g.nx) : uint32_t(g.nx) * uint32_t(g.ny);
                rec = edge_handle(ov, kk == A ? b : A);
            }
        }
    }
    if (x < g.nx) info[info_index(g, edge_handle(v, A))] = rec;
    const uint32_t jw = __ballot_sync(0xFFFFFFFFu, mine && n > 1);
    if (lane == 0) junc[A * r.qplane + r.qbase] = jw;
}

// One warp per vertex-row word, all three axes: every load of the word (the bitmaps of the three
// axes and the gradient words of v and of its three down neighbours, coalesced rows) is issued
// before any result is computed, so a warp has them all in flight at once.
__global__ void __launch_bounds__(THREADS, 4) classify_reached(Geom g, const uint32_t* __restrict__ words,
                                                            const uint32_t* __restrict__ visited,
                                                            const uint4* __restrict__ masks,
                                                            const uint32_t* __restrict__ qdown,
                                                            const uint32_t* __restrict__ crit_bits,
                                                            uint32_t* __restrict__ info, uint32_t* __restrict__ junc,
                                                            unsigned long long* __restrict__ n_reached) {
    const int lane = threadIdx.x & 31;
    const int64_t nrw = int64_t(g.nz) * g.ny * g.W;
    unsigned long long cnt = 0;
    for (int64_t t = (int64_t(blockIdx.x) * THREADS + threadIdx.x) >> 5; t < nrw;
         t += (int64_t(gridDim.x) * THREADS) >> 5) {  // warp-uniform
        const Rows r(g, t);
        const int x = r.w * 32 + lane;
        const uint32_t v = vid32(g, x, r.y, r.z);
        const AxisIn i0 = load_axis<0>(g, r, visited, masks, qdown, crit_bits);
        const AxisIn i1 = load_axis<1>(g, r, visited, masks, qdown, crit_bits);
        const AxisIn i2 = load_axis<2>(g, r, visited, masks, qdown, crit_bits);
        const uint32_t w0 = x < g.nx ? words[v] : 0u;
        const uint32_t wx = minus_word<0>(g, words, r, x, v), wy = minus_word<1>(g, words, r, x, v),
                       wz = minus_word<2>(g, words, r, x, v);
        classify_axis<0>(g, r, lane, x, v, i0, w0, wy, wz, info, junc, cnt);
        classify_axis<1>(g, r, lane, x, v, i1, w0, wx, wz, info, junc, cnt);
        classify_axis<2>(g, r, lane, x, v, i2, w0, wx, wy, info, junc, cnt);
    }
    __shared__ unsigned long long part[THREADS / 32];
    if (lane == 0) part[threadIdx.x >> 5] = cnt;
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned long long s = 0;
        for (int k = 0; k < THREADS / 32; ++k) s += part[k];
        if (s) atomicAdd(n_reached, s);
    }
}

int grid_for(const Plan* p, int64_t threads) {
    const int64_t want = (threads + THREADS - 1) / THREADS;
    const int64_t cap = int64_t(p->num_sms > 0 ? p->num_sms : 148) * 8;
    return int(std::max<int64_t>(1, std::min(want, cap)));
}

// Grids of at most this many row words push every level in one cluster.  What decides is the levels' sizes,
// which the grid only bounds: against sweeps first, then the cluster, it is even on smooth fields of any of
// these sizes and on rough ones up to 1024 row words (24^3 white noise 37 us either way, 32^3 GRF 49), and
// slower on rough ones near the line (2040 words: GRF k^-2 61 against 49 us, white noise 62-72 against 39-47;
// 70-82 by sweeps alone); a 7350-word GRF, whose first levels have 100 thousand cells, took 164 against 72.
constexpr int64_t TAIL_ROW_WORDS = 2048;
// A level of at most this many new cells is left to one cluster (two cells a thread; 128 thousand, eight
// a thread, took 1.5 ms of the 512^3 blob field's levels that the whole device pushes in 0.6 ms) ...
constexpr uint32_t TAIL_CELLS = 32 * 1024;
// ... and one of at most a third of a cell per row word is pushed rather than swept: a sweep takes some
// 25 ps a row word, a pushed level some 60 ps a cell and its launch.
constexpr int64_t SPARSE_DIV = 3;

struct SweepCtx {
    dim3 grid;
    const uint4* masks;
    uint32_t* a;
    uint32_t* b;
    uint32_t* stamp;
    uint32_t sparse;
    int last;
};

void sweep_body(Plan* p, cudaStream_t s, cudaGraphConditionalHandle h, void* ctx) {
    const SweepCtx& c = *static_cast<SweepCtx*>(ctx);
    reach_sweep<<<c.grid, THREADS, 0, s>>>(p->g, c.masks, c.a, c.b, c.stamp, p->dsum(), 0, &p->dsum()->loop_flag[0]);
    reach_sweep<<<c.grid, THREADS, 0, s>>>(p->g, c.masks, c.b, c.a, c.stamp, p->dsum(), 1, &p->dsum()->loop_flag[1]);
    reach_decide<<<1, 1, 0, s>>>(p->dsum(), c.sparse, c.last, p->opts.max_iterations, h, h != 0);
}

struct PushCtx {
    int grid;
    uint32_t sparse;
    PushArgs a;
};

void push_body(Plan* p, cudaStream_t s, cudaGraphConditionalHandle h, void* ctx) {
    const PushCtx& c = *static_cast<PushCtx*>(ctx);
    for (int i = 0; i < PUSHES; ++i)
        reach_push<<<c.grid, THREADS, 0, s>>>(c.a, p->dsum(), i & 1, i == 0 ? 3 : i - 1, i == PUSHES - 1 ? 4 : i);
    reach_push_decide<<<1, 1, 0, s>>>(p->dsum(), TAIL_CELLS, c.sparse, p->opts.max_iterations, h, h != 0);
}

// One cluster over as many blocks as this device can schedule together.
msc_status launch_tail(Plan* p, cudaStream_t s, const PushArgs& a, int all, uint32_t sparse) {
    msc_status st;
    if (!p->tail_cluster) {
        if ((st = check_cuda(p, cudaFuncSetAttribute(reach_tail, cudaFuncAttributeNonPortableClusterSizeAllowed, 1),
                             "cudaFuncSetAttribute(reach_tail)")))
            return st;
        for (int size : {16, 8, 4, 2, 1}) {
            cudaLaunchConfig_t cfg{};
            cfg.gridDim = dim3(unsigned(size));
            cfg.blockDim = dim3(TAIL_THREADS);
            cudaLaunchAttribute at{};
            at.id = cudaLaunchAttributeClusterDimension;
            at.val.clusterDim.x = unsigned(size);
            at.val.clusterDim.y = at.val.clusterDim.z = 1;
            cfg.attrs = &at;
            cfg.numAttrs = 1;
            int n = 0;
            if (cudaOccupancyMaxActiveClusters(&n, reach_tail, &cfg) == cudaSuccess && n > 0) {
                p->tail_cluster = size;
                break;
            }
            cudaGetLastError();
        }
        if (!p->tail_cluster) return fail(p, MSC_ERR_CUDA, "no thread-block cluster can be launched");
    }
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(unsigned(p->tail_cluster));
    cfg.blockDim = dim3(TAIL_THREADS);
    cfg.stream = s;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = unsigned(p->tail_cluster);
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    launched(p);
    return check_cuda(p, cudaLaunchKernelEx(&cfg, reach_tail, a, p->dsum(), all, sparse, p->opts.max_iterations), "reach_tail launch");
}

}  // namespace

msc_status ensure_reach_maps(Plan* p) {
    const Geom& g = p->g;
    const size_t nw = size_t(g.edge_words()), nrw = size_t(g.nz) * size_t(g.ny) * size_t(g.W);
    msc_status st;
    if ((st = ensure(p, p->visited, sizeof(uint32_t) * nw))) return st;
    if ((st = ensure(p, p->reach_tmp, sizeof(uint32_t) * nw))) return st;
    if ((st = ensure(p, p->reach_masks, sizeof(uint4) * nw))) return st;
    if ((st = ensure(p, p->reach_qdown, sizeof(uint32_t) * 3 * nrw))) return st;
    return ensure(p, p->reach_stamp, sizeof(uint32_t) * size_t(g.nz) * size_t(g.ny));
}

WordBitmaps maps_of(const Plan* p) {
    return WordBitmaps{static_cast<const uint32_t*>(p->words.ptr),     static_cast<uint32_t*>(p->crit_bits.ptr),
                       static_cast<uint4*>(p->reach_masks.ptr),        static_cast<uint32_t*>(p->visited.ptr),
                       static_cast<uint32_t*>(p->reach_tmp.ptr),       static_cast<uint32_t*>(p->reach_qdown.ptr),
                       static_cast<uint32_t*>(p->reach_stamp.ptr)};
}

static msc_status run_levels(Plan* p, cudaStream_t s) {
    const Geom& g = p->g;
    msc_status st;
    const int64_t nrw = int64_t(g.nz) * g.ny * g.W;  // vertex-row words
    if ((st = ensure_reach_maps(p))) return st;
    auto* masks = static_cast<uint4*>(p->reach_masks.ptr);
    auto* stamp = static_cast<uint32_t*>(p->reach_stamp.ptr);
    uint32_t* A = static_cast<uint32_t*>(p->visited.ptr);
    uint32_t* B = static_cast<uint32_t*>(p->reach_tmp.ptr);
    if (!p->capturing) {  // a captured pass made them with the critical bitmaps
        if ((st = check_cuda(p, launch_word_bitmaps<false, true>(g, maps_of(p), p->num_sms, s), "word_bitmaps launch"))) return st;
        launched(p);
    }
    reach_start<<<1, 1, 0, s>>>(p->dsum());
    launched(p);
    if ((st = check_cuda(p, cudaGetLastError(), "reach_start launch"))) return st;
    // sweep grid: at most 4 tiles per CTA and at least one resident wave (4 CTAs per SM).  Fewer,
    // longer CTAs would cost little alone but leave long tails when other passes share the device.
    const int64_t tiles = (nrw + THREADS - 1) / THREADS;
    const int64_t sweep_ctas = std::min<int64_t>(tiles, std::max<int64_t>(int64_t(std::max(1, p->num_sms)) * 4, (tiles + 3) / 4));
    SweepCtx ctx{dim3(unsigned(std::max<int64_t>(1, sweep_ctas)), 1), masks, A, B, stamp, 0, 0};
    if (p->capturing) p->reach_captured = 0;
    if (p->reach_sweeps_only) return run_loop(p, s, 1, 3, sweep_body, &ctx);
    // the pushed levels.  A small grid's queues hold every 1-cell; a large one's twelve times the level
    // they start from (a level of a sparse front hardly grows), and a pass that needs more asks for a
    // rerun by sweeps alone
    const bool all = nrw <= TAIL_ROW_WORDS;
    const int64_t sparse = std::max<int64_t>(TAIL_CELLS, nrw / SPARSE_DIV);
    int64_t room = all ? 3 * g.nverts : 12 * sparse;
    if (p->fault_kind == 5) room = std::max<int64_t>(1, std::min<int64_t>(room, p->fault_at));
    if ((st = ensure(p, p->reach_queue, sizeof(uint32_t) * 2 * size_t(room)))) return st;
    PushArgs a{};
    a.g = g;
    a.words = static_cast<const uint32_t*>(p->words.ptr);
    a.reached = A;
    a.queue[0] = static_cast<uint32_t*>(p->reach_queue.ptr);
    a.queue[1] = a.queue[0] + room;
    a.cap = uint32_t(room);
    a.status = p->status_word();
    if (!all) {
        ctx.sparse = uint32_t(sparse);
        if (!p->capturing) {
            if ((st = run_loop(p, s, 1, 3, sweep_body, &ctx))) return st;
        } else {
            // as many iterations as the last synchronised pass took, one after another (a conditional
            // node costs 12 us an iteration): a field that needs fewer skips the rest, one that needs
            // more pushes a larger level (see follow_levels)
            p->reach_captured = p->reach_iters;
            for (int64_t i = 0; i < p->reach_iters; ++i) {
                ctx.last = i + 1 == p->reach_iters;
                sweep_body(p, s, 0, &ctx);
                launched(p, 3);
            }
            p->loop_body_launches[1] = 0;
        }
        Summary* sum = p->dsum();
        reach_frontier<<<grid_for(p, nrw), THREADS, 0, s>>>(a, A, B, &sum->push_count[3], &sum->push_cursor);
        launched(p);
        if (sparse > TAIL_CELLS) {
            PushCtx pc{std::max(1, p->num_sms) * 8, ctx.sparse, a};
            if ((st = run_loop(p, s, 3, PUSHES + 1, push_body, &pc))) return st;
        }
    }
    if ((st = launch_tail(p, s, a, all ? 1 : 0, uint32_t(sparse)))) return st;
    if (p->capturing) return MSC_OK;
    // a synchronised pass whose queue was full (a replayed one comes here through its rerun)
    if ((st = read_summary(p, s))) return st;
    p->reach_iters = std::max<int64_t>(1, int64_t(p->hsum->sweep_iters));
    if (!(p->hsum->status & ST_RETRY)) return MSC_OK;
    p->reach_sweeps_only = true;
    const uint32_t clear[2] = {p->hsum->status & ~uint32_t(ST_RETRY), 0u};
    if ((st = check_cuda(p, cudaMemcpyAsync(p->status_word(), &clear[0], sizeof(uint32_t), cudaMemcpyHostToDevice, s), "status reset")) ||
        (st = check_cuda(p, cudaMemsetAsync(&p->dsum()->sweep_iters, 0, sizeof(unsigned long long), s), "loop reset")) ||
        (st = check_cuda(p, cudaMemsetAsync(p->dsum()->push_count, 0, sizeof(p->dsum()->push_count), s), "loop reset")) ||
        (st = check_cuda(p, cudaStreamSynchronize(s), "stream sync")))
        return st;
    return run_levels(p, s);
}

msc_status run_reachability(Plan* p, cudaStream_t s) {
    // a field whose levels outgrew the queue says nothing of the next one's; a captured pass does what the
    // last synchronised one ended with
    if (!p->capturing) p->reach_sweeps_only = false;
    return run_levels(p, s);
}

// A replayed pass sweeps as often as it was captured to, so the next one is captured for the field of this
// one if that had levels for sweeps that it had to push, or if MANY replays in a row left more than SPARE
// iterations unused.  Fields in turn do not make a plan capture again and again (0.25 ms each): the number grows
// at once, and only many replays together make it fall.  Reachability stage of a GRF that takes three
// iterations, captured with two: 140^3 (the levels go to one cluster) 171 us, 85 once captured again; 152^3 119
// and 110, 256^3 230 and 207.  An unused iteration takes 5 us.
void follow_levels(Plan* p) {
    constexpr int64_t SPARE = 1, MANY = 64;
    if (!p->reach_captured) return;
    const int64_t took = int64_t(p->hsum->sweep_iters);
    if (p->hsum->dense) {  // the handed-over level and dense - 1 after it; an iteration ends at every second level
        p->reach_iters = p->reach_captured + 1 + (int64_t(p->hsum->dense) - 1) / 2;
    } else {
        const bool spare = p->reach_captured - took > SPARE;
        p->reach_spare = spare ? p->reach_spare + 1 : 0;
        p->reach_most = spare ? std::max(p->reach_most, took) : 0;
        if (p->reach_spare < MANY) return;
        p->reach_iters = std::max<int64_t>(1, p->reach_most);
    }
    p->reach_spare = p->reach_most = 0;
    destroy_graph(p);
}

msc_status run_junctions(Plan* p, cudaStream_t s) {
    const Geom& g = p->g;
    msc_status st;
    const int64_t nrw = int64_t(g.nz) * g.ny * g.W;
    if ((st = ensure(p, p->junc_bits, sizeof(uint32_t) * 3 * size_t(nrw)))) return st;
    if ((st = ensure(p, p->junc_prefix, sizeof(uint32_t) * 3 * size_t(nrw)))) return st;
    if ((st = ensure(p, p->node_info, sizeof(uint32_t) * 3 * size_t(g.nverts)))) return st;
    classify_reached<<<grid_for(p, nrw * 32), THREADS, 0, s>>>(
        g, static_cast<const uint32_t*>(p->words.ptr), static_cast<const uint32_t*>(p->visited.ptr),
        static_cast<const uint4*>(p->reach_masks.ptr), static_cast<const uint32_t*>(p->reach_qdown.ptr),
        static_cast<const uint32_t*>(p->crit_bits.ptr), static_cast<uint32_t*>(p->node_info.ptr),
        static_cast<uint32_t*>(p->junc_bits.ptr), &p->dsum()->reached);
    launched(p);
    if ((st = check_cuda(p, cudaGetLastError(), "classify_reached launch"))) return st;
    EdgeSource src{};
    src.g = g;
    src.bits = static_cast<const uint32_t*>(p->junc_bits.ptr);
    src.prefix = static_cast<uint32_t*>(p->junc_prefix.ptr);
    src.status = p->status_word();
    if ((st = compaction_sums(p, s, src, 1, &p->dsum()->n_junctions))) return st;
    int64_t cap = p->caps.nj;
    if (!p->capturing) {  // size the list exactly
        if ((st = read_summary(p, s))) return st;
        cap = int64_t(p->hsum->n_junctions);
        p->n_junctions = cap;
    }
    if ((st = ensure(p, p->junc_cells, sizeof(uint32_t) * size_t(cap ? cap : 1)))) return st;
    src.out = static_cast<uint32_t*>(p->junc_cells.ptr);
    src.cap = uint64_t(cap);
    return compaction_emit(p, s, src, 1);
}

}  // namespace msc
