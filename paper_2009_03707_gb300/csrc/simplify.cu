// Simplification of the 1-skeleton by cancellation of critical-point pairs (Sec. 4), on request.
//
// The paper cancels, in order of persistence, pairs of critical points of consecutive index that
// are joined by exactly one arc (several arcs: a strangulation); a cancellation reroutes the upper
// point's descending arcs to the end points of the lower point's ascending arcs and deletes the
// two points.  It runs the cancellations serially inside subgrids on the CPU and reports that a
// data-parallel form -- an independent set of arcs under the 3-link neighbourhood, cancelled
// together -- is the generic alternative.  Here that form runs on the GPU, in rounds:
//   * keys: (persistence = |value(upper) - value(lower)|, cell id of the upper point, cell id of
//     the lower point), where a critical cell's value is that of its highest vertex;
//   * a round cancels every valid arc (both ends alive, consecutive index, multiplicity 1,
//     persistence <= threshold) whose key is the least among the valid arcs with an end within
//     two links of one of its ends -- so the arcs of one round are more than two links apart and
//     the nodes each cancellation touches (its ends and their neighbours) are disjoint, and the
//     globally least valid arc is always among them;
//   * rounds repeat until no valid arc is left.
// A round costs little more than what it changes:
//   * state per node: its row (start and length in a pool of (neighbour, multiplicity) entries,
//     sorted by neighbour), the least key of its valid arcs and the neighbour that arc leads to.
//     All of it changes only at the nodes a cancellation touches.
//   * an arc can be selected only if it is the least valid arc of both its ends.  Those mutual arcs
//     are kept as a list (by upper node); a pair can only become mutual where an end was touched.
//     A listed arc that was looked at and not selected sleeps: it remembers a node within two links
//     that has a smaller key, and a link goes only when one of its ends is cancelled, so nothing can
//     free the arc before that node is touched.  Most arcs sleep through most rounds.
//   * the others are looked at: one link away, then two, up to the first smaller key.
//   * the selected cancellations hand out one task per touched node: merge the node's row with the
//     neighbours it gains (or drop the arc it loses) into fresh pool space, and take its new least
//     key.  When the pool runs full, the rows are gathered into the other pool and the round goes on.
// Four launches a round, their counts on the device; the host looks once per BATCH rounds.  At the
// end one gather makes the CSR, and one stable sort by round puts the cancellations in log order.
// 256^3 GRF (6.0 M nodes, 40 M entries, 317 rounds, threshold 5 % of the range): 370 ms with every
// round sweeping all nodes and rewriting the whole CSR (1.1 ms a round), 67 ms now: looks 27, updates 14,
// the list 11, cancellations 6, gathers 2.  The price is memory: 188 B a node (161 of them in simp_node, 40 the
// two lists) and two row pools of 1.25 x 12 B an entry, 2.7 GB there, where the sweeps took 117 B and two copies
// of the rows, 1.9 GB.
#include <cooperative_groups.h>

#include "radix.cuh"

namespace cg = cooperative_groups;

namespace msc {

namespace {

constexpr int THREADS = 256;
constexpr uint32_t NO_NODE = 0xFFFFFFFFu;
constexpr int BATCH = 8;       // rounds launched between two looks by the host
constexpr int G = 8;           // lanes per row: rows have about 7 entries, and a task is latency-bound
typedef unsigned long long u64;
typedef cg::thread_block_tile<G, cg::thread_block> Tile;

struct __align__(16) Key {
    u64 hi, lo;  // persistence (bits of a non-negative double), upper cell << 32 | lower cell
};
__device__ __forceinline__ bool key_less(const Key& a, const Key& b) { return a.hi < b.hi || (a.hi == b.hi && a.lo < b.lo); }
__device__ __forceinline__ Key no_key() { return Key{~0ull, ~0ull}; }

// A node's row in the pool and the neighbour its least valid arc leads to; with that arc's key they
// share one 32-byte sector, since whoever reads one usually reads the other.
struct __align__(16) Row {
    int64_t start;
    uint32_t len, to;
};
struct __align__(32) Node {
    Key least;
    Row row;
};

struct __align__(16) NodeValue {
    double value;   // of the cell's highest vertex
    uint32_t cell;
    uint32_t pad;
};

// What one round did: the arcs listed at its end, the looks, the cancellations and the nodes they touch.
// Slot 0 of the array is the state a batch of rounds starts from.
struct RoundCount {
    unsigned int nlist, nlook, nsel, ntask;
    u64 cursor;  // pool entries used when the round began
};
struct SimpState {
    u64 cursor;           // pool entries used
    unsigned int halted;  // a round (1 + its place in the batch) found the pool full
    unsigned int pad;
    u64 alive_count[4];
    u64 cancelled, entries;
    RoundCount round[BATCH + 1];
};

// A selected cancellation: the upper node p, the lower node q, and the two ranges of neighbours that
// are joined anew: p's of q's index and q's of p's index (each range holds the other end too).
struct __align__(16) Pair {
    int64_t down_at, up_at;  // in the pool
    uint32_t down_n, up_n;
    uint32_t p, q;
};
// Roles of a touched node: it keeps an arc less (of p, of q), or it gains the other end's range.
enum Role : uint32_t { GAINS_UP = 0, GAINS_DOWN = 1, LOSES_P = 2, LOSES_Q = 3 };

struct SimpArgs {
    int64_t n;        // nodes
    int64_t base[4];  // first node of each index (minima, 1-saddles, 2-saddles, maxima)
    double threshold;
    const NodeValue* value;
    Node* node;
    uint32_t* nbr;    // the pool
    u64* mult;
    u64 cap;
    // per upper node: what its arc waits for (the node w with the smaller key), the arc's lower node and
    // the node between p or q and w (w itself if it is one link away)
    uint32_t* wait;
    uint2* wait_qv;
    uint8_t* listed;    // per upper node: it has an entry in the list
    uint32_t* touched;  // per node: 1 + the last round that touched it
    uint32_t* stamp;    // per upper node: 1 + the last round that looked at its arc
    uint32_t* list;     // upper nodes of mutual arcs (NO_NODE: an entry no longer used)
    uint2* look;        // arcs (p, q) to look at in this round
    uint8_t* alive;
    uint32_t* cround; // per upper node: the round that cancelled it, and its lower node
    uint32_t* cwith;
    Pair* pairs;      // this round's cancellations
    uint32_t* task_node;
    uint32_t* task_pair;  // pair << 2 | role
    u64* task_factor;     // multiplicity of the touched node's arc to the cancelled node
    int64_t* task_at;     // pool space of the new row
    SimpState* state;
    uint32_t* status;
};

__device__ __forceinline__ int node_index(const SimpArgs& a, uint32_t u) {
    return int(u >= a.base[1]) + int(u >= a.base[2]) + int(u >= a.base[3]);
}

// The key of the arc (u, v) of multiplicity m between live nodes if it is valid, else no_key().
// Neighbours have consecutive indices, so the upper node is the one with the larger number.
__device__ __forceinline__ Key arc_key(const SimpArgs& a, uint32_t u, const NodeValue& nu, uint32_t v, u64 m) {
    if (m != 1) return no_key();
    const NodeValue nv = a.value[v];
    const double pers = fabs(nu.value - nv.value);
    if (!(pers <= a.threshold)) return no_key();
    const uint32_t up = u > v ? nu.cell : nv.cell, lo = u > v ? nv.cell : nu.cell;
    return Key{u64(__double_as_longlong(pers)), (u64(up) << 32) | u64(lo)};
}

__device__ __forceinline__ void take_less(Key& k, uint32_t& to, const Key& other, uint32_t other_to) {
    if (key_less(other, k)) {
        k = other;
        to = other_to;
    }
}
template <class Grp>
__device__ __forceinline__ void group_least(const Grp& g, Key& k, uint32_t& to) {
    for (int o = g.size() / 2; o; o >>= 1) {
        const Key other{g.shfl_xor(k.hi, o), g.shfl_xor(k.lo, o)};
        take_less(k, to, other, g.shfl_xor(to, o));
    }
}

// First position in v[0..n) that is >= key.
__device__ __forceinline__ uint32_t lower_bound(const uint32_t* v, uint32_t n, uint32_t key) {
    uint32_t lo = 0;
    while (n) {
        const uint32_t half = n >> 1;
        if (v[lo + half] < key) {
            lo += half + 1;
            n -= half + 1;
        } else {
            n = half;
        }
    }
    return lo;
}

__global__ void __launch_bounds__(THREADS) simp_init(SimpArgs a, Geom g, const float* __restrict__ f,
                                                     const uint32_t* __restrict__ c0, const uint32_t* __restrict__ c1,
                                                     const uint32_t* __restrict__ c2, const uint32_t* __restrict__ c3,
                                                     const int64_t* __restrict__ nodeptr, NodeValue* __restrict__ value) {
    for (int64_t u = int64_t(blockIdx.x) * THREADS + threadIdx.x; u < a.n; u += int64_t(gridDim.x) * THREADS) {
        const int k = node_index(a, uint32_t(u));
        const uint32_t c = (k == 0 ? c0 : k == 1 ? c1 : k == 2 ? c2 : c3)[u - a.base[k]];
        const uint32_t q = g.div_rx.div(c);
        const int cx = int(c - q * g.rx), cz = int(g.div_ry.div(q)), cy = int(q - uint32_t(cz) * g.ry);
        float best = -INFINITY;
        for (int dz = 0; dz <= (cz & 1); ++dz)
            for (int dy = 0; dy <= (cy & 1); ++dy)
                for (int dx = 0; dx <= (cx & 1); ++dx)
                    best = fmaxf(best, f[g.vid((cx >> 1) + dx, (cy >> 1) + dy, (cz >> 1) + dz)]);
        value[u] = NodeValue{double(best), c, 0u};
        a.node[u].row = Row{nodeptr[u], uint32_t(nodeptr[u + 1] - nodeptr[u]), NO_NODE};
        a.alive[u] = 1;
        a.stamp[u] = 0;
        a.touched[u] = 0;
        a.cround[u] = NO_NODE;
    }
}

// Least valid arc of every node of the initial complex.
__global__ void __launch_bounds__(THREADS) simp_least(SimpArgs a) {
    const Tile t = cg::tiled_partition<G>(cg::this_thread_block());
    const int64_t step = int64_t(gridDim.x) * (THREADS / G);
    for (int64_t i = int64_t(blockIdx.x) * (THREADS / G) + threadIdx.x / G; i < a.n; i += step) {
        const uint32_t u = uint32_t(i);
        const NodeValue nu = a.value[u];
        const int64_t s = a.node[u].row.start;
        const uint32_t L = a.node[u].row.len;
        Key k = no_key();
        uint32_t to = NO_NODE;
        for (uint32_t e = t.thread_rank(); e < L; e += G) {
            const uint32_t v = a.nbr[s + e];
            take_less(k, to, arc_key(a, u, nu, v, a.mult[s + e]), v);
        }
        group_least(t, k, to);
        if (t.thread_rank() == 0) {
            a.node[u].least = k;
            a.node[u].row.to = to;
        }
    }
}

// One atomic per block for the places of its threads' items (n <= 32 of each): every thread of the
// block calls it.
__device__ __forceinline__ unsigned int block_places(unsigned int* counter, unsigned int n) {
    __shared__ unsigned int part[THREADS / 32 + 1];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned int incl = n;
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned int y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
        if (lane >= o) incl += y;
    }
    __syncthreads();  // the last call's places have been read
    if (lane == 31) part[warp] = incl;
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned int acc = 0;
        for (int i = 0; i < THREADS / 32; ++i) {
            const unsigned int c = part[i];
            part[i] = acc;
            acc += c;
        }
        part[THREADS / 32] = acc ? atomicAdd(counter, acc) : 0u;
    }
    __syncthreads();
    return part[THREADS / 32] + part[warp] + incl - n;
}

// The mutual arcs of the initial complex, by upper node, all awake (each waits for its own upper node,
// which counts as touched before the first round).
__global__ void __launch_bounds__(THREADS) simp_mutual(SimpArgs a) {
    for (int64_t b = int64_t(blockIdx.x) * THREADS; b < a.n; b += int64_t(gridDim.x) * THREADS) {
        const int64_t p = b + threadIdx.x;
        const uint32_t q = p < a.n ? a.node[p].row.to : NO_NODE;
        const bool mine = q != NO_NODE && q < uint32_t(p) && a.node[q].row.to == uint32_t(p);
        const unsigned int at = block_places(&a.state->round[0].nlist, mine ? 1u : 0u);
        if (mine) {
            a.list[at] = uint32_t(p);
            a.wait[p] = uint32_t(p);
            a.wait_qv[p] = make_uint2(NO_NODE, NO_NODE);
        }
        if (p < a.n) a.listed[p] = mine ? 1 : 0;
    }
}

// Which arcs are looked at this round: the listed ones whose wait is over, and the mutual arcs of the
// nodes that the last round touched, unless they sleep.  ITEMS entries a thread, their loads issued
// together (the list is the longest thing a round reads: 1.9 M arcs at first on the 256^3 GRF).
constexpr int ITEMS = 4;
__device__ __forceinline__ bool still_waits(const SimpArgs& a, uint32_t p, uint32_t q, uint32_t w, const Key& k) {
    const uint2 qv = a.wait_qv[p];
    return qv.x == q && a.alive[qv.y] && key_less(a.node[w].least, k);
}
__global__ void __launch_bounds__(THREADS) simp_wake(SimpArgs a, int slot, uint32_t round) {
    if (a.state->halted) return;
    const RoundCount* in = &a.state->round[slot];
    RoundCount* out = &a.state->round[slot + 1];
    const unsigned int nlist = in->nlist, ntask = in->ntask;
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        out->cursor = a.state->cursor;
        atomicAdd(&out->nlist, nlist);  // the look kernel appends behind the entries there are
    }
    for (uint64_t b = uint64_t(blockIdx.x) * THREADS * ITEMS; b < nlist; b += uint64_t(gridDim.x) * THREADS * ITEMS) {
        uint32_t p[ITEMS], w[ITEMS], q[ITEMS];
        unsigned int n = 0;
#pragma unroll
        for (int j = 0; j < ITEMS; ++j) {
            const uint64_t i = b + threadIdx.x + j * THREADS;
            p[j] = i < nlist ? a.list[i] : NO_NODE;
        }
#pragma unroll
        for (int j = 0; j < ITEMS; ++j) w[j] = p[j] != NO_NODE ? a.wait[p[j]] : NO_NODE;
#pragma unroll
        for (int j = 0; j < ITEMS; ++j)
            if (w[j] != NO_NODE && a.touched[w[j]] != round) p[j] = NO_NODE;  // asleep
#pragma unroll
        for (int j = 0; j < ITEMS; ++j) {
            q[j] = NO_NODE;
            if (p[j] == NO_NODE) continue;
            q[j] = a.node[p[j]].row.to;
            if (q[j] == NO_NODE || q[j] > p[j] || a.node[q[j]].row.to != p[j]) {  // cancelled, or no longer mutual
                a.list[b + threadIdx.x + j * THREADS] = NO_NODE;
                a.listed[p[j]] = 0;
                p[j] = NO_NODE;
            } else if (still_waits(a, p[j], q[j], w[j], a.node[p[j]].least) || atomicExch(&a.stamp[p[j]], round + 1) == round + 1) {
                p[j] = NO_NODE;
            }
            n += p[j] != NO_NODE;
        }
        unsigned int at = block_places(&out->nlook, n);
#pragma unroll
        for (int j = 0; j < ITEMS; ++j)
            if (p[j] != NO_NODE) a.look[at++] = make_uint2(p[j], q[j]);
    }
    for (uint64_t b = uint64_t(blockIdx.x) * THREADS; b < ntask; b += uint64_t(gridDim.x) * THREADS) {
        const uint64_t i = b + threadIdx.x;
        uint32_t p = NO_NODE, q = NO_NODE;
        if (i < ntask) {
            const uint32_t x = a.task_node[i], y = a.node[x].row.to;
            if (y != NO_NODE && a.node[y].row.to == x) {
                p = max(x, y);
                q = min(x, y);
                // listed and asleep, or taken already (it is listed and awake, or touched at both ends)
                if ((a.listed[p] && still_waits(a, p, q, a.wait[p], a.node[p].least)) ||
                    atomicExch(&a.stamp[p], round + 1) == round + 1)
                    p = NO_NODE;
            }
        }
        const unsigned int at = block_places(&out->nlook, p != NO_NODE ? 1u : 0u);
        if (p != NO_NODE) a.look[at] = make_uint2(p, q);
    }
}

// Looks around a mutual arc (p, q) of key k with a group of lanes: a node within two links of p or q
// that has a smaller least key (*w, and *v the node between), or false.  First the neighbours of both
// ends, a lane each; then the entries of the neighbours' rows, dealt out evenly: the rows of a step's
// neighbours lie one after another on the lanes, each lane taking AHEAD entries and finding an entry's
// row by a search over the lanes' offsets, so a step's gathers are in flight together whatever the
// rows' lengths (a lane per row: 1.5 times as long on the late rounds of the 256^3 GRF, whose rows
// reach 128 entries).
constexpr int AHEAD = 4;
// The lane with the greatest key among those that have one: of the smaller keys found together, the one
// likely to be there longest, since arcs go in about the order of their keys (looks on the 256^3 GRF:
// 35 ms with any of them, 28 ms so).
template <unsigned L>
__device__ __forceinline__ int greatest(const cg::thread_block_tile<L, cg::thread_block>& t, bool has, Key k) {
    if (!has) k = Key{0, 0};
    uint32_t lane = has ? t.thread_rank() + 1 : 0u;  // 0: no key
#pragma unroll
    for (unsigned o = L / 2; o; o >>= 1) {
        const Key other{t.shfl_xor(k.hi, o), t.shfl_xor(k.lo, o)};
        const uint32_t other_lane = t.shfl_xor(lane, o);
        if (key_less(k, other) || (!key_less(other, k) && other_lane > lane)) {
            k = other;
            lane = other_lane;
        }
    }
    return int(lane) - 1;
}
template <unsigned L>
__device__ __forceinline__ bool look_around(const SimpArgs& a, const cg::thread_block_tile<L, cg::thread_block>& t,
                                            uint32_t p, uint32_t q, const Key& k, uint32_t* v_out, uint32_t* w_out) {
    const uint32_t r = t.thread_rank();
    const Row pr = a.node[p].row, qr = a.node[q].row;
    const uint32_t n = pr.len + qr.len;
    auto neighbour = [&](uint32_t e) -> uint32_t {
        return e < n ? a.nbr[e < pr.len ? pr.start + e : qr.start + (e - pr.len)] : NO_NODE;
    };
    for (uint32_t e = r; e - r < n; e += L) {
        const uint32_t v = neighbour(e);
        Key kv = no_key();
        if (v != NO_NODE) kv = a.node[v].least;
        const bool less = key_less(kv, k);
        if (t.any(less)) {
            *v_out = *w_out = t.shfl(v, greatest(t, less, kv));
            return true;
        }
    }
    for (uint32_t e = r; e - r < n; e += L) {
        const uint32_t v = neighbour(e);
        Row vr{0, 0, 0};
        if (v != NO_NODE) vr = a.node[v].row;
        uint32_t first = vr.len;  // this row's first entry among the step's
#pragma unroll
        for (unsigned o = 1; o < L; o <<= 1) {
            const uint32_t y = t.shfl_up(first, o);
            if (r >= o) first += y;
        }
        const uint32_t total = t.shfl(first, L - 1);
        first -= vr.len;
        for (uint32_t j0 = 0; j0 < total; j0 += L * AHEAD) {
            uint32_t w[AHEAD], hit = NO_NODE, hit_l = 0;
            Key hit_k{0, 0};
            int own[AHEAD];
#pragma unroll
            for (int i = 0; i < AHEAD; ++i) {
                const uint32_t j = j0 + i * L + r;
                int l = 0;  // the last lane whose row starts at or before j (an empty row shares its start)
#pragma unroll
                for (int h = int(L) / 2; h; h >>= 1)
                    if (t.shfl(first, l + h) <= j) l += h;
                const int64_t at = t.shfl(vr.start, l) + (j - t.shfl(first, l));
                w[i] = j < total ? a.nbr[at] : NO_NODE;
                own[i] = l;
            }
#pragma unroll
            for (int i = 0; i < AHEAD; ++i)
                if (w[i] != NO_NODE) {
                    const Key kw = a.node[w[i]].least;
                    if (key_less(kw, k) && !key_less(kw, hit_k)) {
                        hit = w[i];
                        hit_l = own[i];
                        hit_k = kw;
                    }
                }
            if (t.any(hit != NO_NODE)) {
                const int l = greatest(t, hit != NO_NODE, hit_k);
                *w_out = t.shfl(hit, l);
                *v_out = t.shfl(v, t.shfl(hit_l, l));
                return true;
            }
        }
    }
    return false;
}

// The looks of a round, a group of L lanes each: an arc with a smaller key near it goes to sleep (and
// on the list, if it is not there), the others are this round's cancellations.
template <unsigned L>
__device__ __forceinline__ void look_at_arcs(const SimpArgs& a, RoundCount* out, unsigned int nlook) {
    const cg::thread_block_tile<L, cg::thread_block> t = cg::tiled_partition<L>(cg::this_thread_block());
    constexpr unsigned PER_WARP = 32 / L;
    const unsigned lane = threadIdx.x & 31;
    const unsigned warp = blockIdx.x * (THREADS / 32) + (threadIdx.x >> 5), nwarps = gridDim.x * (THREADS / 32);
    for (uint64_t b = uint64_t(warp) * PER_WARP; b < nlook; b += uint64_t(nwarps) * PER_WARP) {
        const uint64_t i = b + lane / L;
        uint2 pq = make_uint2(NO_NODE, NO_NODE);
        uint32_t v = NO_NODE, w = NO_NODE;
        bool blocked = false;
        if (i < nlook) {
            pq = a.look[i];
            blocked = look_around(a, t, pq.x, pq.y, a.node[pq.x].least, &v, &w);
        }
        const bool lead = i < nlook && t.thread_rank() == 0;
        bool append = false;
        if (lead && blocked) {
            a.wait[pq.x] = w;
            a.wait_qv[pq.x] = make_uint2(pq.y, v);
            append = !a.listed[pq.x];
            a.listed[pq.x] = 1;
        }
        const uint32_t more = __ballot_sync(0xFFFFFFFFu, append), take = __ballot_sync(0xFFFFFFFFu, lead && !blocked);
        unsigned int at_more = 0, at_take = 0;
        if (lane == 0) {
            if (more) at_more = atomicAdd(&out->nlist, unsigned(__popc(more)));
            if (take) at_take = atomicAdd(&out->nsel, unsigned(__popc(take)));
        }
        at_more = __shfl_sync(0xFFFFFFFFu, at_more, 0);
        at_take = __shfl_sync(0xFFFFFFFFu, at_take, 0);
        const uint32_t below = (1u << lane) - 1u;
        if (append) a.list[at_more + __popc(more & below)] = pq.x;
        if (lead && !blocked) {
            Pair* pr = &a.pairs[at_take + __popc(take & below)];
            pr->p = pq.x;
            pr->q = pq.y;
        }
    }
}
// Few looks are bound by how long the longest takes, so they get a whole warp each: late rounds of the 256^3
// GRF have some 2500 looks of up to 1850 entries.  Where there are many, eight lanes each were meant to keep
// more in flight; the measured gain is gone.  Whole call with the line at 16, 64, 128 and 256 thousand: 73.4,
// 66.9, 66.2, 66.1 ms; a warp for every look 66.1; sixteen lanes above the line 65.9, four 68.5; sixteen
// lanes below it 72.7.
constexpr unsigned int WIDE_LOOKS = 65536;
__global__ void __launch_bounds__(THREADS) simp_look(SimpArgs a, int slot) {
    if (a.state->halted) return;
    RoundCount* out = &a.state->round[slot + 1];
    const unsigned int nlook = out->nlook;
    if (nlook > WIDE_LOOKS) look_at_arcs<8>(a, out, nlook);
    else look_at_arcs<32>(a, out, nlook);
}

// The list without unused entries and cancelled nodes (between batches of rounds).
__global__ void __launch_bounds__(THREADS) simp_compact(SimpArgs a, unsigned int nlist, uint32_t* __restrict__ to) {
    for (uint64_t b = uint64_t(blockIdx.x) * THREADS; b < nlist; b += uint64_t(gridDim.x) * THREADS) {
        const uint64_t i = b + threadIdx.x;
        uint32_t p = i < nlist ? a.list[i] : NO_NODE;
        if (p != NO_NODE && !a.alive[p]) p = NO_NODE;
        const unsigned int at = block_places(&a.state->round[0].nlist, p != NO_NODE ? 1u : 0u);
        if (p != NO_NODE) to[at] = p;
    }
}

// A warp per cancellation: its nodes die, their neighbours become tasks, and the new rows get pool
// space (an upper bound of their lengths).  The shared counters see two atomics per block of eight
// cancellations: with five per cancellation they took half of the kernel (23 000 cancellations a round
// early on, 0.11 ms).
__global__ void __launch_bounds__(THREADS) simp_cancel(SimpArgs a, int slot, uint32_t round) {
    const unsigned int halted = a.state->halted;  // by an earlier round: this one sets it while it runs
    if (halted && halted <= unsigned(slot)) return;
    RoundCount* rc = &a.state->round[slot + 1];
    const unsigned int nsel = rc->nsel;
    __shared__ unsigned int tasks_of[THREADS / 32], task_base;
    __shared__ u64 room_of[THREADS / 32], room_base;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (unsigned b = blockIdx.x * (THREADS / 32); b < nsel; b += gridDim.x * (THREADS / 32)) {
        const unsigned i = b + warp;
        const bool mine = i < nsel;  // warp-uniform
        Pair pr{};
        int64_t ps = 0, qs = 0;
        uint32_t p = NO_NODE, q = NO_NODE, pn = 0, qn = 0;
        u64 room = 0;
        if (mine) {
            pr = a.pairs[i];
            p = pr.p;
            q = pr.q;
            const Row rp = a.node[p].row, rq = a.node[q].row;
            ps = rp.start;
            qs = rq.start;
            pn = rp.len;
            qn = rq.len;
            // rows are sorted by node, so each index is one range: p's neighbours of q's index come first
            // (then those above p), q's of p's index last (after those below q)
            const uint32_t above = uint32_t(a.base[node_index(a, q) + 1]);
            const uint32_t down = lower_bound(a.nbr + ps, pn, above), up = lower_bound(a.nbr + qs, qn, above);
            pr.down_at = ps;
            pr.down_n = down;
            pr.up_at = qs + up;
            pr.up_n = qn - up;
            // the new rows: one arc less, and the range of the other end without that end
            for (uint32_t e = lane; e < down; e += 32) {
                const uint32_t x = a.nbr[ps + e];
                if (x != q) room += u64(a.node[x].row.len) - 1 + (pr.up_n - 1);
            }
            for (uint32_t e = up + lane; e < qn; e += 32) {
                const uint32_t x = a.nbr[qs + e];
                if (x != p) room += u64(a.node[x].row.len) - 1 + (down - 1);
            }
            for (int o = 16; o; o >>= 1) room += __shfl_xor_sync(0xFFFFFFFFu, room, o);
        }
        // one pair of atomics per block: the tasks and the pool space of its cancellations
        __syncthreads();
        if (lane == 0) {
            tasks_of[warp] = mine ? pn + qn - 2 : 0u;
            room_of[warp] = room;
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            unsigned int t = 0;
            u64 m = 0;
            for (int k = 0; k < THREADS / 32; ++k) {
                const unsigned int tk = tasks_of[k];
                const u64 mk = room_of[k];
                tasks_of[k] = t;
                room_of[k] = m;
                t += tk;
                m += mk;
            }
            task_base = atomicAdd(&rc->ntask, t);
            room_base = atomicAdd(&a.state->cursor, m);
            if (room_base + m > a.cap) atomicMax(&a.state->halted, unsigned(slot + 1));
        }
        __syncthreads();
        if (!mine) continue;
        if (lane == 0) {
            a.pairs[i] = pr;
            a.alive[p] = a.alive[q] = 0;
            a.node[p] = a.node[q] = Node{no_key(), Row{0, 0, NO_NODE}};
            a.touched[p] = a.touched[q] = round + 1;
            a.cround[p] = round;
            a.cwith[p] = q;
        }
        unsigned int task = task_base + tasks_of[warp];
        u64 at = room_base + room_of[warp];
        for (int side = 0; side < 2; ++side) {
            const int64_t s = side == 0 ? ps : qs;
            const uint32_t n = side == 0 ? pn : qn, other = side == 0 ? q : p;
            const uint32_t extra = side == 0 ? pr.up_n - 1 : pr.down_n - 1;
            for (uint32_t e = 0; e < n; e += 32) {
                const bool in = e + lane < n;
                const uint32_t x = in ? a.nbr[s + e + lane] : other;
                const bool task_of = x != other;
                const bool gains = task_of && (side == 0 ? e + lane < pr.down_n : e + lane >= n - pr.up_n);
                const u64 want = gains ? u64(a.node[x].row.len) - 1 + extra : 0;
                u64 incl = want;
                for (int o = 1; o < 32; o <<= 1) {
                    const u64 y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
                    if (lane >= o) incl += y;
                }
                const uint32_t vote = __ballot_sync(0xFFFFFFFFu, task_of);
                if (task_of) {
                    const unsigned j = task + __popc(vote & ((1u << lane) - 1u));
                    a.task_node[j] = x;
                    a.task_pair[j] = (i << 2) | (gains ? (side == 0 ? GAINS_UP : GAINS_DOWN) : side == 0 ? LOSES_P : LOSES_Q);
                    a.task_factor[j] = a.mult[s + e + lane];
                    a.task_at[j] = int64_t(at + incl - want);
                }
                task += __popc(vote);
                at += __shfl_sync(0xFFFFFFFFu, incl, 31);
            }
        }
    }
}

// Pool space for the new rows of a round whose pool was full, in the pool its rows were gathered to
// (which has room for them).
__global__ void __launch_bounds__(THREADS) simp_place(SimpArgs a, unsigned int ntask) {
    for (unsigned j = blockIdx.x * THREADS + threadIdx.x; j < ntask; j += gridDim.x * THREADS) {
        const uint32_t role = a.task_pair[j] & 3u;
        if (role > GAINS_DOWN) continue;
        const Pair pr = a.pairs[a.task_pair[j] >> 2];
        const u64 want = u64(a.node[a.task_node[j]].row.len) - 1 + (role == GAINS_UP ? pr.up_n : pr.down_n) - 1;
        a.task_at[j] = int64_t(atomicAdd(&a.state->cursor, want));
    }
}

// A group of lanes per touched node: its new row and least valid arc.  A node that only loses an arc
// drops it in place.  One that gains a range B (less the other cancelled end) merges it with its row
// A (less the cancelled neighbour): every element finds its rank in the other list by binary search,
// so each lane places its own elements; common neighbours are written from A's side, with
// multiplicity m + factor * (B's).  B is read in `bn`, `bm`: the pool the cancellation was found in.
__global__ void __launch_bounds__(THREADS) simp_update(SimpArgs a, int slot, uint32_t round,
                                                       const uint32_t* __restrict__ bn, const u64* __restrict__ bm,
                                                       int resumed) {
    if (!resumed && a.state->halted) return;
    const unsigned int ntask = a.state->round[slot + 1].ntask;
    const Tile t = cg::tiled_partition<G>(cg::this_thread_block());
    const uint32_t r = t.thread_rank(), below = (1u << r) - 1u;
    const unsigned step = gridDim.x * (THREADS / G);
    for (unsigned j = blockIdx.x * (THREADS / G) + threadIdx.x / G; j < ntask; j += step) {
        const uint32_t x = a.task_node[j], tag = a.task_pair[j], role = tag & 3u;
        const Pair pr = a.pairs[tag >> 2];
        const uint32_t dead = (role == GAINS_UP || role == LOSES_P) ? pr.p : pr.q;
        const Node old = a.node[x];
        const int64_t s = old.row.start;
        const uint32_t L = old.row.len, old_to = old.row.to;
        const NodeValue nx = a.value[x];
        if (r == 0) a.touched[x] = round + 1;
        if (role > GAINS_DOWN) {
            // losing an arc that is not the least one leaves the least one as it is
            const bool redo = old_to == dead;
            Key k = no_key();
            uint32_t to = NO_NODE, gone = 0;
            for (uint32_t e = 0; e < L; e += G) {
                const bool in = e + r < L;
                const uint32_t v = in ? a.nbr[s + e + r] : 0u;
                const u64 m = in ? a.mult[s + e + r] : 0ull;
                const bool cut = in && v == dead;
                const uint32_t cuts = t.ballot(cut);
                t.sync();  // the reads before the writes
                if (in && !cut && (gone || (cuts & below))) {
                    a.nbr[s + e + r - 1] = v;
                    a.mult[s + e + r - 1] = m;
                }
                if (redo && in && !cut) take_less(k, to, arc_key(a, x, nx, v, m), v);
                gone |= cuts;
                t.sync();
            }
            if (redo) group_least(t, k, to);
            if (r == 0) a.node[x] = Node{redo ? k : old.least, Row{s, L - 1, redo ? to : old_to}};
            continue;
        }
        const uint32_t* A = a.nbr + s;
        const u64* Am = a.mult + s;
        const int64_t bat = role == GAINS_UP ? pr.up_at : pr.down_at;
        const uint32_t* B = bn + bat;
        const u64* Bm = bm + bat;
        const uint32_t nb = role == GAINS_UP ? pr.up_n : pr.down_n;
        const int64_t dst = a.task_at[j];
        const u64 f = a.task_factor[j];
        // the cancelled neighbour is in both lists: A's dead arc, and the end of B's range not joined
        const uint32_t a_cut = lower_bound(A, L, dead), b_cut = lower_bound(B, nb, dead);
        uint32_t at_to = NO_NODE;
        if (old_to != NO_NODE && old_to != dead) at_to = lower_bound(B, nb, old_to);
        // the old least arc stays a valid one unless it is cut or gains paths
        const bool keep = at_to != NO_NODE && !(at_to < nb && B[at_to] == old_to);
        const bool fresh = old_to != NO_NODE && !keep;  // look at every arc again
        Key k = keep ? old.least : no_key();
        uint32_t to = keep ? old_to : NO_NODE;
        bool over = false;
        uint32_t dups = 0;
        for (uint32_t e = 0; e < L; e += G) {
            const uint32_t i = e + r;
            const bool in = i < L && i != a_cut;
            const uint32_t v = in ? A[i] : 0u;
            uint32_t jb = 0;
            bool dup = false;
            if (in) {
                jb = lower_bound(B, nb, v);
                dup = jb < nb && B[jb] == v;
            }
            const uint32_t vote = t.ballot(dup);
            if (in) {
                u64 m = Am[i];
                if (dup) {
                    const u64 mb = Bm[jb], prod = f * mb;
                    over |= (mb != 0 && __umul64hi(f, mb) != 0) || m + prod < m;
                    m += prod;
                }
                const uint32_t o = (i - (i > a_cut)) + (jb - (jb > b_cut)) - (dups + __popc(vote & below));
                a.nbr[dst + o] = v;
                a.mult[dst + o] = m;
                if (fresh) take_less(k, to, arc_key(a, x, nx, v, m), v);
            }
            dups += __popc(vote);
        }
        uint32_t dups_b = 0;
        for (uint32_t e = 0; e < nb; e += G) {
            const uint32_t i = e + r;
            const bool in = i < nb && i != b_cut;
            const uint32_t v = in ? B[i] : 0u;
            uint32_t ja = 0;
            bool dup = false;
            if (in) {
                ja = lower_bound(A, L, v);
                dup = ja < L && A[ja] == v;
            }
            const uint32_t vote = t.ballot(dup);
            if (in && !dup) {
                const u64 mb = Bm[i], m = f * mb;
                over |= mb != 0 && __umul64hi(f, mb) != 0;
                const uint32_t o = (i - (i > b_cut)) + (ja - (ja > a_cut)) - (dups_b + __popc(vote & below));
                a.nbr[dst + o] = v;
                a.mult[dst + o] = m;
                take_less(k, to, arc_key(a, x, nx, v, m), v);
            }
            dups_b += __popc(vote);
        }
        if (over) atomicOr(a.status, ST_OVERFLOW);
        group_least(t, k, to);
        t.sync();
        if (r == 0) a.node[x] = Node{k, Row{dst, L - 1 + nb - 1 - dups, to}};
    }
}

// Starts a batch of rounds from what slot `from` left; the list's length comes with its compaction, or
// is `nlist`.
__global__ void simp_begin(SimpState* state, int from, unsigned int nlist) {
    const RoundCount last = state->round[from];
    __syncwarp();
    for (int i = threadIdx.x; i <= BATCH; i += blockDim.x)
        state->round[i] = i == 0 ? RoundCount{nlist, 0, 0, last.ntask, 0} : RoundCount{0, 0, 0, 0, 0};
    if (threadIdx.x == 0) state->halted = 0;
}

// Row lengths, for their scan.
__global__ void __launch_bounds__(THREADS) simp_lengths(SimpArgs a, uint32_t* __restrict__ len) {
    for (int64_t u = int64_t(blockIdx.x) * THREADS + threadIdx.x; u < a.n; u += int64_t(gridDim.x) * THREADS)
        len[u] = a.node[u].row.len;
}

// Gathers every row to its place in the other pool: a warp copies 32 consecutive rows' entries, one
// per lane, a lane finding its entry's row among the 32 row starts by shuffles.
__global__ void __launch_bounds__(THREADS) simp_gather(SimpArgs a, const int64_t* __restrict__ ptr,
                                                       uint32_t* __restrict__ nbr, u64* __restrict__ mult, int move) {
    const int lane = threadIdx.x & 31;
    const int64_t step = int64_t(gridDim.x) * THREADS;
    for (int64_t u0 = int64_t(blockIdx.x) * THREADS + (threadIdx.x & ~31); u0 < a.n; u0 += step) {
        const int64_t u = u0 + lane;
        const int64_t end = ptr[min(u0 + 32, a.n)];
        const int64_t at = u < a.n ? ptr[u] : end;
        const int64_t src = u < a.n ? a.node[u].row.start : 0;
        const int64_t first = __shfl_sync(0xFFFFFFFFu, at, 0);
        for (int64_t b = first; b < end; b += 32) {
            const int64_t o = b + lane;
            int k = 0;
#pragma unroll
            for (int h = 16; h; h >>= 1) {
                const int64_t v = __shfl_sync(0xFFFFFFFFu, at, k + h);
                if (v <= o) k += h;
            }
            const int64_t from = __shfl_sync(0xFFFFFFFFu, src, k) + (o - __shfl_sync(0xFFFFFFFFu, at, k));
            if (o < end) {
                nbr[o] = a.nbr[from];
                mult[o] = a.mult[from];
            }
        }
        if (move && u < a.n) a.node[u].row.start = at;
    }
}

// Survivors per index, and the cancelled upper nodes.
__global__ void __launch_bounds__(THREADS) simp_survivors(SimpArgs a, uint32_t* __restrict__ flag) {
    u64 c[4] = {0, 0, 0, 0};
    for (int64_t u = int64_t(blockIdx.x) * THREADS + threadIdx.x; u < a.n; u += int64_t(gridDim.x) * THREADS) {
        const int k = node_index(a, uint32_t(u));
        const u64 live = a.alive[u];
#pragma unroll
        for (int i = 0; i < 4; ++i) c[i] += i == k ? live : 0;
        flag[u] = a.cround[u] != NO_NODE ? 1u : 0u;
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        for (int o = 16; o; o >>= 1) c[i] += __shfl_xor_sync(0xFFFFFFFFu, c[i], o);
        if ((threadIdx.x & 31) == 0 && c[i]) atomicAdd(&a.state->alive_count[i], c[i]);
    }
}

__global__ void __launch_bounds__(THREADS) simp_log_pairs(SimpArgs a, const int64_t* __restrict__ pos,
                                                          uint32_t* __restrict__ key, uint32_t* __restrict__ val) {
    for (int64_t u = int64_t(blockIdx.x) * THREADS + threadIdx.x; u < a.n; u += int64_t(gridDim.x) * THREADS)
        if (a.cround[u] != NO_NODE) {
            key[pos[u]] = a.cround[u];
            val[pos[u]] = uint32_t(u);
        }
}

__global__ void __launch_bounds__(THREADS) simp_log(SimpArgs a, int64_t m, const uint32_t* __restrict__ key,
                                                    const uint32_t* __restrict__ val, uint32_t* __restrict__ log) {
    for (int64_t i = int64_t(blockIdx.x) * THREADS + threadIdx.x; i < m; i += int64_t(gridDim.x) * THREADS) {
        log[3 * i] = val[i];
        log[3 * i + 1] = a.cwith[val[i]];
        log[3 * i + 2] = key[i];
    }
}

}  // namespace

// Simplifies the plan's 1-skeleton (built by build_complex_graph) up to `threshold`; d_field is the
// field of the plan's last pass (for the critical cells' values).  Host-synchronised once per BATCH
// rounds.
msc_status run_simplify(Plan* p, const float* d_field, double threshold, cudaStream_t s) {
    const Geom& g = p->g;
    msc_status st;
    const int64_t n = p->graph_nodes, nnz0 = p->graph_nadj;
    SimpArgs a{};
    a.n = n;
    for (int k = 1; k < 4; ++k) a.base[k] = a.base[k - 1] + p->counts[k - 1];
    a.threshold = threshold;
    const size_t nn = size_t(n ? n : 1), half = nn / 2 + 1;
    // per node and per cancellation arrays, widest first
    size_t off = 0;
    auto carve = [&](size_t bytes) {
        const size_t at = off;
        off += (bytes + 255) / 256 * 256;
        return at;
    };
    const size_t o_value = carve(sizeof(NodeValue) * nn), o_state = carve(sizeof(Node) * nn);
    const size_t o_wait = carve(4 * nn), o_qv = carve(sizeof(uint2) * nn), o_touched = carve(4 * nn);
    const size_t o_look = carve(sizeof(uint2) * half);
    const size_t o_pairs = carve(sizeof(Pair) * half);
    const size_t o_factor = carve(sizeof(u64) * nn), o_at = carve(sizeof(int64_t) * nn);
    const size_t o_stamp = carve(4 * nn), o_cround = carve(4 * nn), o_cwith = carve(4 * nn);
    const size_t o_node = carve(4 * nn), o_pair = carve(4 * nn), o_listed = carve(nn);
    // a node has at most one entry in the list when it is compacted, and a round appends at most one arc
    // per two nodes
    const size_t list_room = nn + half * BATCH;
    const size_t o_list0 = carve(4 * list_room), o_list1 = carve(4 * list_room);
    if ((st = ensure(p, p->simp_node, off))) return st;
    if ((st = ensure(p, p->simp_alive, nn))) return st;
    if ((st = ensure(p, p->simp_len, sizeof(uint32_t) * (nn + 1)))) return st;
    if ((st = ensure(p, p->simp_pos, sizeof(int64_t) * (nn + 1)))) return st;
    if ((st = ensure(p, p->simp_ptr, sizeof(int64_t) * (nn + 1)))) return st;
    if ((st = ensure(p, p->simp_scan, row_scan_scratch_bytes(int64_t(nn)) + 64))) return st;
    if ((st = ensure(p, p->simp_log, sizeof(uint32_t) * 3 * half))) return st;
    if ((st = ensure(p, p->simp_round, sizeof(SimpState)))) return st;
    // both pools start a quarter larger than the complex
    auto pool = [&](int b, u64 want) {
        msc_status e = ensure(p, p->simp_nbr[b], sizeof(uint32_t) * size_t(want));
        return e ? e : ensure(p, p->simp_mult[b], sizeof(u64) * size_t(want));
    };
    u64 cap[2];
    for (int b = 0; b < 2; ++b) {
        cap[b] = u64(nnz0) + (p->fault_kind == 6 ? u64(p->fault_at) : u64(nnz0) / 4 + 256);
        if ((st = pool(b, cap[b]))) return st;
    }
    char* w = static_cast<char*>(p->simp_node.ptr);
    auto* value = reinterpret_cast<NodeValue*>(w + o_value);
    a.value = value;
    a.node = reinterpret_cast<Node*>(w + o_state);
    a.wait = reinterpret_cast<uint32_t*>(w + o_wait);
    a.wait_qv = reinterpret_cast<uint2*>(w + o_qv);
    a.touched = reinterpret_cast<uint32_t*>(w + o_touched);
    a.listed = reinterpret_cast<uint8_t*>(w + o_listed);
    a.look = reinterpret_cast<uint2*>(w + o_look);
    a.pairs = reinterpret_cast<Pair*>(w + o_pairs);
    a.task_factor = reinterpret_cast<u64*>(w + o_factor);
    a.task_at = reinterpret_cast<int64_t*>(w + o_at);
    a.stamp = reinterpret_cast<uint32_t*>(w + o_stamp);
    a.cround = reinterpret_cast<uint32_t*>(w + o_cround);
    a.cwith = reinterpret_cast<uint32_t*>(w + o_cwith);
    a.task_node = reinterpret_cast<uint32_t*>(w + o_node);
    a.task_pair = reinterpret_cast<uint32_t*>(w + o_pair);
    uint32_t* lists[2] = {reinterpret_cast<uint32_t*>(w + o_list0), reinterpret_cast<uint32_t*>(w + o_list1)};
    a.list = lists[0];
    auto* len = static_cast<uint32_t*>(p->simp_len.ptr);
    a.alive = static_cast<uint8_t*>(p->simp_alive.ptr);
    a.state = static_cast<SimpState*>(p->simp_round.ptr);
    a.status = p->status_word();
    auto* pos = static_cast<int64_t*>(p->simp_pos.ptr);
    auto* ptr = static_cast<int64_t*>(p->simp_ptr.ptr);
    auto* scan = static_cast<u64*>(p->simp_scan.ptr);
    int cur = 0;
    auto use_pool = [&](int b) {
        a.nbr = static_cast<uint32_t*>(p->simp_nbr[b].ptr);
        a.mult = static_cast<u64*>(p->simp_mult[b].ptr);
        a.cap = cap[b];
    };
    use_pool(cur);
    SimpState h{};
    h.cursor = u64(nnz0);
    auto put_state = [&] {
        return check_cuda(p, cudaMemcpyAsync(a.state, &h, sizeof(h), cudaMemcpyHostToDevice, s), "simplify state");
    };
    auto get_state = [&] {
        const msc_status e = check_cuda(p, cudaMemcpyAsync(&h, a.state, sizeof(h), cudaMemcpyDeviceToHost, s), "simplify read");
        return e ? e : check_status_word(p, s);  // synchronises
    };
    if ((st = put_state())) return st;
    if (nnz0 && ((st = check_cuda(p, cudaMemcpyAsync(a.nbr, p->graph_adj.ptr, sizeof(uint32_t) * size_t(nnz0),
                                                     cudaMemcpyDeviceToDevice, s), "simplify copy")) ||
                 (st = check_cuda(p, cudaMemcpyAsync(a.mult, p->graph_mult.ptr, sizeof(u64) * size_t(nnz0),
                                                     cudaMemcpyDeviceToDevice, s), "simplify copy"))))
        return st;
    const int all = grid_cap(p, n, THREADS);
    if (n) {
        simp_init<<<all, THREADS, 0, s>>>(a, g, d_field, static_cast<const uint32_t*>(p->cells[0].ptr),
                                          static_cast<const uint32_t*>(p->cells[1].ptr),
                                          static_cast<const uint32_t*>(p->cells[2].ptr),
                                          static_cast<const uint32_t*>(p->cells[3].ptr),
                                          static_cast<const int64_t*>(p->graph_nodeptr.ptr), value);
        simp_least<<<grid_cap(p, n * G, THREADS), THREADS, 0, s>>>(a);
        simp_mutual<<<all, THREADS, 0, s>>>(a);
        launched(p, 3);
    }
    if ((st = get_state())) return st;
    int64_t cancelled = 0, rounds = 0;
    int from = 0;  // the slot the next batch starts from
    const int64_t max_rounds = p->opts.max_iterations > 0 ? p->opts.max_iterations : (int64_t(1) << 20);
    bool more = n > 0;
    while (more) {
        if (rounds >= max_rounds) return fail(p, MSC_ERR_ITER_LIMIT, "simplification reached the iteration cap");
        const int count = int(std::min<int64_t>(BATCH, max_rounds - rounds));
        // grids for about twice the work the last round left, full ones for the first rounds (the loops
        // stride, so any grid is right)
        const RoundCount& last = h.round[from];
        const int64_t tasks = rounds ? std::min<int64_t>(n, 2 * int64_t(last.ntask) + 1024) : n;
        const int64_t looks = rounds ? std::min<int64_t>(n, 2 * int64_t(last.nlook) + 1024) : n;
        const int g_wake = grid_cap(p, std::max<int64_t>(last.nlist / ITEMS, tasks), THREADS);
        const int g_look = grid_cap(p, looks * 32, THREADS);
        const int g_cancel = grid_cap(p, tasks * 4, THREADS), g_update = grid_cap(p, tasks * G, THREADS);
        unsigned int nlist = last.nlist;
        simp_begin<<<1, 32, 0, s>>>(a.state, from, rounds ? 0u : nlist);
        if (rounds) {
            simp_compact<<<grid_cap(p, nlist, THREADS), THREADS, 0, s>>>(a, nlist, lists[1]);
            std::swap(lists[0], lists[1]);
            a.list = lists[0];
        }
        for (int i = 0; i < count; ++i) {
            const uint32_t r = uint32_t(rounds + i);
            simp_wake<<<g_wake, THREADS, 0, s>>>(a, i, r);
            simp_look<<<g_look, THREADS, 0, s>>>(a, i);
            simp_cancel<<<g_cancel, THREADS, 0, s>>>(a, i, r);
            simp_update<<<g_update, THREADS, 0, s>>>(a, i, r, a.nbr, a.mult, 0);
        }
        launched(p, (rounds ? 2 : 1) + 4 * count);
        if ((st = check_cuda(p, cudaGetLastError(), "simplify launch"))) return st;
        if ((st = get_state())) return st;
        const int ran = h.halted ? int(h.halted) : count;
        for (int i = 1; i <= ran; ++i) {
            if (!h.round[i].nsel) {
                more = false;
                break;
            }
            ++rounds;
            cancelled += int64_t(h.round[i].nsel);
        }
        from = ran;
        if (!h.halted) continue;
        // round `ran` of the batch found its cancellations but not the room for their rows: gather
        // the rows into the other pool, place the new ones behind them and finish the round
        const int other = cur ^ 1;
        u64 live = 0;
        auto* total = reinterpret_cast<u64*>(&a.state->entries);
        simp_lengths<<<all, THREADS, 0, s>>>(a, len);
        if ((st = check_cuda(p, row_scan(p, len, nullptr, n, ptr, scan, s, total), "simplify scan"))) return st;
        const u64 need = h.cursor - h.round[ran].cursor;
        const unsigned int ntask = h.round[ran].ntask;
        if ((st = get_state())) return st;
        live = h.entries;
        if (live + need + need / 2 > cap[other]) {
            cap[other] = live + live / 4 + 2 * need;
            if ((st = pool(other, cap[other]))) return st;
        }
        const uint32_t* old_nbr = a.nbr;
        const u64* old_mult = a.mult;
        simp_gather<<<all, THREADS, 0, s>>>(a, ptr, static_cast<uint32_t*>(p->simp_nbr[other].ptr),
                                            static_cast<u64*>(p->simp_mult[other].ptr), 1);
        cur = other;
        use_pool(cur);
        if ((st = check_cuda(p, cudaMemcpyAsync(&a.state->cursor, &a.state->entries, sizeof(u64), cudaMemcpyDeviceToDevice, s),
                             "simplify state")))
            return st;
        simp_place<<<grid_cap(p, ntask, THREADS), THREADS, 0, s>>>(a, ntask);
        simp_update<<<grid_cap(p, int64_t(ntask) * G, THREADS), THREADS, 0, s>>>(a, ran - 1, uint32_t(rounds - 1), old_nbr,
                                                                                old_mult, 1);
        launched(p, 4);
    }
    // the result: survivors, the rows as a CSR in the other pool, the log in (round, node) order
    const int other = cur ^ 1;
    if (n) {
        simp_lengths<<<all, THREADS, 0, s>>>(a, len);
        launched(p);
    }
    if ((st = check_cuda(p, row_scan(p, len, nullptr, n, ptr, scan, s, &a.state->entries), "simplify scan"))) return st;
    if (n) {
        auto* flag = reinterpret_cast<uint32_t*>(w + o_stamp);  // the stamps are spent
        simp_survivors<<<all, THREADS, 0, s>>>(a, flag);
        launched(p);
        if ((st = check_cuda(p, row_scan(p, flag, nullptr, n, pos, scan, s, &a.state->cancelled), "simplify scan"))) return st;
    }
    if ((st = get_state())) return st;
    if (h.entries > cap[other]) {
        cap[other] = h.entries;
        if ((st = pool(other, cap[other]))) return st;
    }
    if (n) {
        simp_gather<<<all, THREADS, 0, s>>>(a, ptr, static_cast<uint32_t*>(p->simp_nbr[other].ptr),
                                            static_cast<u64*>(p->simp_mult[other].ptr), 0);
        launched(p);
    }
    if (int64_t(h.cancelled) != cancelled) return fail(p, MSC_ERR_INTERNAL, "internal: the cancellations do not add up");
    if (cancelled) {
        // sort space: the task arrays hold the pairs, a buffer of its own the digit counts
        uint32_t* keys[2] = {reinterpret_cast<uint32_t*>(w + o_factor), reinterpret_cast<uint32_t*>(w + o_factor) + half};
        uint32_t* vals[2] = {reinterpret_cast<uint32_t*>(w + o_at), reinterpret_cast<uint32_t*>(w + o_at) + half};
        const int64_t nhist = int64_t(radix_hist_count(cancelled));
        const size_t b_offs = (sizeof(uint32_t) * size_t(nhist) + 255) / 256 * 256;
        const size_t b_scan = b_offs + (sizeof(int64_t) * size_t(nhist + 1) + 255) / 256 * 256;
        if ((st = ensure(p, p->simp_sort, b_scan + row_scan_scratch_bytes(nhist)))) return st;
        char* sp = static_cast<char*>(p->simp_sort.ptr);
        const RadixSpace ws{reinterpret_cast<uint32_t*>(sp), reinterpret_cast<int64_t*>(sp + b_offs),
                            reinterpret_cast<unsigned long long*>(sp + b_scan)};
        simp_log_pairs<<<all, THREADS, 0, s>>>(a, pos, keys[0], vals[0]);
        int k = 0;
        if ((st = check_cuda(p, radix_sort_pairs(p, keys, vals, &k, cancelled, uint32_t(rounds), ws, s), "log sort"))) return st;
        simp_log<<<grid_cap(p, cancelled, THREADS), THREADS, 0, s>>>(a, cancelled, keys[k], vals[k],
                                                                     static_cast<uint32_t*>(p->simp_log.ptr));
        launched(p, 2);
    }
    if ((st = check_cuda(p, cudaGetLastError(), "simplify launch"))) return st;
    if ((st = check_status_word(p, s))) return st;
    p->simp_cur = other;
    p->simp_nnz = int64_t(h.entries);
    p->simp_rounds = rounds;
    p->simp_cancelled = cancelled;
    for (int k = 0; k < 4; ++k) p->simp_counts[k] = int64_t(h.alive_count[k]);
    return MSC_OK;
}

}  // namespace msc
