// (a6) Saddle-saddle path counts, D* = D + sum_{k>=0} A B^k B* (Sec. 3.3 "Path counting via
// matrix operations"), evaluated right to left.
//
// The paper iterates A <- A B (SpGEMM) and accumulates A* B* + D: every 1-saddle row walks the
// whole sub-DAG below it, so a junction reached from many 1-saddles, at many depths, is expanded
// again for every one of them -- on a field with long V-path networks (the paper's noisy volumes,
// the 512^3 blob field here: 197 iterations, 1e9 frontier entries, path counts near 1.6e10)
// that repetition is most of the work.  The same matrix identity read from the right,
//     J = sum_k B^k B*  (paths from each junction to the 2-saddles),  J = B* + B J,
//     D* = D + A J,
// needs every junction's row once, in topological order of the minor (a DAG): a junction's row
// is ready as soon as the rows of the junctions it points to are.  So:
//   1. the reverse adjacency of B (junction -> the junctions pointing at it) and, per junction,
//      the number of its out-slots that point at junctions;
//   2. waves: wave 0 is the junctions with no junction successor; a junction's J row is the
//      merge of its 4 trace slots -- a 2-saddle slot is one path to that 2-saddle, a junction
//      slot adds that junction's J row -- and finishing it decrements the pending counts of its
//      predecessors; the one that takes a count to 0 appends the predecessor to the next wave's
//      queue (collected per block, one atomic on the queue's length per block and step).  So every
//      row a junction reads was complete before its wave began.  The waves run as a device loop (a
//      conditional WHILE node in a graph), WAVES of them an iteration; the non-empty ones number the
//      paper's iteration count, 1 + the longest chain of junctions;
//   3. D* row s = the same merge over 1-saddle s's slots, written to staging and gathered into
//      CSR (pathcount.cu's staging, row scan and gather).
// Rows are merged sorted by column with exact uint64 sums (an add that wraps raises the overflow
// flag).  J rows live in one pool, with one bump of its pointer per block and step.  A merge is a
// chain of dependent loads, one step per output entry, so a wave lasts as long as its longest
// merge: merges of more than LONG_ROW input entries are taken by a warp, of more than BLOCK_ROW by the
// block, which cut the columns into a slice per lane (pivots sampled from the inputs, a binary search
// per lane and input) and merge a slice each.  A wave's junctions are dealt out evenly over the blocks, so that a
// block has few of either sort in the many small waves.
// 512^3 blob field (14.5 M junctions, 178 waves, 37 M entries): path-count stage 22.0 -> 12.9 ms against
// waves that scanned a bitmap for their junctions (a thread took up to 32 of them one after another) and
// handed long merges to a second kernel; the first waves (0.4 to 2.6 M junctions) now run at the rate of
// their scattered reads, the last hundred take 11-20 us each.
#include <cstddef>
#include <type_traits>

#include "rowscan.cuh"

namespace msc {

namespace {

constexpr int THREADS = 256;
constexpr int WAVES = DP_WAVES;    // waves per iteration of the loop
// merges with more input entries are taken by a warp, and by a whole block
constexpr uint32_t LONG_ROW = 12, BLOCK_ROW = 256;
constexpr int RELEASED = 1536;     // released junctions a block collects before it appends them one by one
typedef unsigned long long u64;

struct DpArgs {
    const uint32_t* tgt;                 // 4 destination ranks per source (1-saddles, then junctions)
    const uint32_t* kinds;               // per source: byte k = kind of slot k
    const unsigned long long* n1_dev;    // 1-saddles and junctions, counted earlier in the pass
    const unsigned long long* nj_dev;
    int64_t cap1, capj;                  // the capacities the buffers were sized for
    uint32_t* pend;                      // per junction: junction slots whose rows are not ready
    uint32_t* queue[2];                  // the junctions of a wave (even and odd ones)
    uint32_t* in_cnt;                    // per junction: slots of other junctions pointing at it
    int64_t* in_ptr;                     // CSR of those predecessors
    uint32_t* in_fill;
    uint32_t* in_idx;
    u64* j_off;                          // per junction: its J row in the pool
    uint32_t* j_len;
    uint32_t* pool_col;                  // J rows: 2-saddle ranks increasing, uint64 counts
    u64* pool_cnt;
    u64 pool_cap;
    uint32_t* out_col;                   // D* rows (staging) and their place
    u64* out_cnt;
    u64 out_cap;
    int64_t* row_start;
    uint32_t* row_len;
    Summary* sum;
    uint32_t* status;
};

// The pass's counts; false (do nothing) when the pass is to be rerun.  Called by whole blocks.
__device__ __forceinline__ bool counts_of(const DpArgs& a, int64_t& n1, int64_t& nj) {
    const u64 x = *a.n1_dev, y = *a.nj_dev;
    if (block_retrying(a.status) || !count_fits(a.status, x, a.cap1) || !count_fits(a.status, y, a.capj)) return false;
    n1 = int64_t(x);
    nj = int64_t(y);
    return true;
}

// Exclusive prefix of n over the block's threads, and the sum in *total.
__device__ __forceinline__ uint32_t block_prefix(uint32_t n, uint32_t* total) {
    __shared__ uint32_t part[THREADS / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t incl = n;
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
        if (lane >= o) incl += y;
    }
    __syncthreads();  // the last call's sums have been read
    if (lane == 31) part[warp] = incl;
    __syncthreads();
    uint32_t before = 0, sum = 0;
#pragma unroll
    for (int w = 0; w < THREADS / 32; ++w) {
        const uint32_t c = part[w];
        before += w < warp ? c : 0;
        sum += c;
    }
    *total = sum;
    return before + incl - n;
}

// Merge of one source's 4 slots: a 2-saddle slot is one path to that 2-saddle, a junction slot
// contributes that junction's J row.  Inputs are sorted by column; the output is sorted with
// equal columns summed.  Returns the output length; *bound gets the sum of the input lengths.
struct Inputs {
    const uint32_t* col[4];
    const u64* cnt[4];
    uint32_t len[4];
    uint32_t single[4];  // the 2-saddle of a 2-saddle slot
    uint32_t kind[4];
};

__device__ __forceinline__ Inputs inputs_of(const DpArgs& a, int64_t src, uint32_t* bound) {
    Inputs in;
    const uint4 q = *reinterpret_cast<const uint4*>(a.tgt + 4 * src);
    const uint32_t kinds = a.kinds[src];
    const uint32_t t[4] = {q.x, q.y, q.z, q.w};
    uint32_t b = 0;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        in.kind[k] = trace_kind(kinds, k);
        in.single[k] = t[k];
        in.len[k] = 0;
        in.col[k] = nullptr;
        in.cnt[k] = nullptr;
        if (in.kind[k] == 2) {
            in.len[k] = 1;
        } else if (in.kind[k] == 1) {
            in.len[k] = a.j_len[t[k]];
            in.col[k] = a.pool_col + a.j_off[t[k]];
            in.cnt[k] = a.pool_cnt + a.j_off[t[k]];
        }
        b += in.len[k];
    }
    *bound = b;
    return in;
}

__device__ __forceinline__ uint32_t merge_into(const Inputs& in, uint32_t* out_col, u64* out_cnt, uint64_t room,
                                               u64* max_seen, uint32_t* status) {
    uint32_t pos[4] = {0, 0, 0, 0};
    uint32_t n = 0;
    bool wrapped = false;
    for (;;) {
        uint32_t c = 0xFFFFFFFFu;
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (pos[k] < in.len[k]) c = min(c, in.kind[k] == 2 ? in.single[k] : in.col[k][pos[k]]);
        if (c == 0xFFFFFFFFu) break;
        u64 s = 0;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            if (pos[k] >= in.len[k]) continue;
            const uint32_t ck = in.kind[k] == 2 ? in.single[k] : in.col[k][pos[k]];
            if (ck != c) continue;
            const u64 v = in.kind[k] == 2 ? 1ull : in.cnt[k][pos[k]];
            wrapped |= s + v < s;
            s += v;
            ++pos[k];
        }
        if (n < room) {
            out_col[n] = c;
            out_cnt[n] = s;
        }
        *max_seen = max(*max_seen, s);
        ++n;
    }
    if (wrapped) atomicOr(status, ST_OVERFLOW);
    return n;
}

// Per junction: its pending junction slots (wave 0 if none) and the reverse-adjacency counts.
__global__ void __launch_bounds__(THREADS) dp_init(DpArgs a) {
    int64_t n1, nj;
    if (!counts_of(a, n1, nj)) return;
    __shared__ uint32_t base;
    for (int64_t j0 = int64_t(blockIdx.x) * THREADS; j0 < nj; j0 += int64_t(gridDim.x) * THREADS) {
        const int64_t j = j0 + threadIdx.x;
        uint32_t pending = 1;
        if (j < nj) {
            const uint4 q = *reinterpret_cast<const uint4*>(a.tgt + 4 * (n1 + j));
            const uint32_t kinds = a.kinds[n1 + j];
            const uint32_t t[4] = {q.x, q.y, q.z, q.w};
            pending = 0;
#pragma unroll
            for (int k = 0; k < 4; ++k)
                if (trace_kind(kinds, k) == 1) {
                    ++pending;
                    atomicAdd(&a.in_cnt[t[k]], 1u);
                }
            a.pend[j] = pending;
        }
        uint32_t total;
        const uint32_t at = block_prefix(pending ? 0u : 1u, &total);
        if (threadIdx.x == 0) base = total ? atomicAdd(&a.sum->dp_queue[0], total) : 0u;
        __syncthreads();
        if (!pending) a.queue[0][base + at] = uint32_t(j);
    }
}

// The reverse adjacency: predecessors of every junction, one entry per slot.
__global__ void __launch_bounds__(THREADS) dp_fill(DpArgs a) {
    int64_t n1, nj;
    if (!counts_of(a, n1, nj)) return;
    for (int64_t j = int64_t(blockIdx.x) * THREADS + threadIdx.x; j < nj; j += int64_t(gridDim.x) * THREADS) {
        const uint4 q = *reinterpret_cast<const uint4*>(a.tgt + 4 * (n1 + j));
        const uint32_t kinds = a.kinds[n1 + j];
        const uint32_t t[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (trace_kind(kinds, k) == 1) a.in_idx[a.in_ptr[t[k]] + atomicAdd(&a.in_fill[t[k]], 1u)] = uint32_t(j);
    }
}

// One lane's slice of a merge: the columns in [lo, hi) (hi_open: no upper end) of every input,
// merged with equal columns summed; counts them, and writes them from out_col / out_cnt when
// `write` is set.
__device__ __forceinline__ uint32_t slice_merge(const Inputs& in, const uint32_t s[4], const uint32_t e[4],
                                                uint32_t lo, uint32_t hi, bool hi_open, bool write, uint32_t* out_col,
                                                u64* out_cnt, u64* max_seen, bool* wrapped) {
    uint32_t pos[4], end[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        pos[k] = s[k];
        end[k] = e[k];
        if (in.kind[k] == 2) {  // a 2-saddle slot: its one column, if it falls in the slice
            const bool mine = in.single[k] >= lo && (hi_open || in.single[k] < hi);
            pos[k] = 0;
            end[k] = mine ? 1 : 0;
        }
    }
    uint32_t n = 0;
    for (;;) {
        uint32_t c = 0xFFFFFFFFu;
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (pos[k] < end[k]) c = min(c, in.kind[k] == 2 ? in.single[k] : in.col[k][pos[k]]);
        if (c == 0xFFFFFFFFu) break;
        u64 sum = 0;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            if (pos[k] >= end[k]) continue;
            const uint32_t ck = in.kind[k] == 2 ? in.single[k] : in.col[k][pos[k]];
            if (ck != c) continue;
            if (write) {
                const u64 v = in.kind[k] == 2 ? 1ull : in.cnt[k][pos[k]];
                *wrapped |= sum + v < sum;
                sum += v;
            }
            ++pos[k];
        }
        if (write) {
            out_col[n] = c;
            out_cnt[n] = sum;
            *max_seen = max(*max_seen, sum);
        }
        ++n;
    }
    return n;
}

// A merge by N threads (a warp, or the block): N pivot columns, taken at even steps through the inputs
// laid end to end and sorted, cut the columns into slices with at most a step's worth of entries from each
// input.  Thread l merges the columns in [pivot l, pivot l+1) of every input (binary searches for its
// slice, the four inputs' steps side by side), twice -- to count, then, after a prefix of the counts, to
// write.  Returns the length.  A wave lasts as long as its longest merge, hence the block for the longest
// rows: per wave of the 512^3 blob field 72 us with a warp and pivots from the longest input alone (an
// input whose columns lay between two of them was merged by one lane), 61 us with pivots from all
// inputs, 56 us with the block (eight lanes for merges of up to 64 entries: no gain; blocks of 128: no
// gain; the block for more than 96, 160, 512 entries: stage 13.6, 13.1, 13.3 ms against 12.9).
struct Cut {
    uint32_t pivot[THREADS + 1];
    uint32_t at[4][THREADS + 1];
};
template <int N>
__device__ __forceinline__ uint32_t merge_by(const Inputs& in, uint32_t bound, uint32_t* out_col, u64* out_cnt,
                                             u64* max_seen, uint32_t* status, Cut& cut) {
    static_assert(N == 32 || N == THREADS, "a warp or the block");
    const int l = N == 32 ? int(threadIdx.x & 31) : int(threadIdx.x);
    uint32_t lo = 0, before = 0, longest = 0;
    const uint32_t at = uint32_t(u64(l) * bound / N);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        if (at >= before && at - before < in.len[k]) lo = in.kind[k] == 2 ? in.single[k] : in.col[k][at - before];
        before += in.len[k];
        if (in.kind[k] == 1) longest = max(longest, in.len[k]);
    }
    // bitonic sort of the pivots: exchanges within a warp by shuffles, wider ones through shared memory
#pragma unroll
    for (int size = 2; size <= N; size <<= 1)
#pragma unroll
        for (int step = size >> 1; step; step >>= 1) {
            uint32_t other;
            if (step < 32) {
                other = __shfl_xor_sync(0xFFFFFFFFu, lo, step);
            } else {
                __syncthreads();
                cut.pivot[l] = lo;
                __syncthreads();
                other = cut.pivot[l ^ step];
            }
            const bool low = (l & step) == 0, up = (l & size) == 0;
            lo = low == up ? min(lo, other) : max(lo, other);
        }
    if (l == 0) lo = 0;
    const bool hi_open = l == N - 1;
    uint32_t s[4], e[4], n[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        s[k] = 0;
        n[k] = in.kind[k] == 1 ? in.len[k] : 0u;
    }
    for (uint32_t left = longest; left; left >>= 1) {  // every n[k] <= left halves at every step
        uint32_t mid[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) mid[k] = n[k] ? in.col[k][s[k] + (n[k] >> 1)] : 0u;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const uint32_t half = n[k] >> 1;
            if (n[k] && mid[k] < lo) {
                s[k] += half + 1;
                n[k] -= half + 1;
            } else {
                n[k] = half;
            }
        }
    }
    // the slice ends where the next thread's begins
    uint32_t hi;
    if (N == 32) {
        hi = __shfl_down_sync(0xFFFFFFFFu, lo, 1);
#pragma unroll
        for (int k = 0; k < 4; ++k) e[k] = __shfl_down_sync(0xFFFFFFFFu, s[k], 1);
    } else {
        __syncthreads();
        cut.pivot[l] = lo;
#pragma unroll
        for (int k = 0; k < 4; ++k) cut.at[k][l] = s[k];
        __syncthreads();
        hi = cut.pivot[min(l + 1, N - 1)];
#pragma unroll
        for (int k = 0; k < 4; ++k) e[k] = cut.at[k][min(l + 1, N - 1)];
    }
#pragma unroll
    for (int k = 0; k < 4; ++k)
        if (hi_open) e[k] = in.kind[k] == 1 ? in.len[k] : 0u;
    bool wrapped = false;
    const uint32_t cnt = slice_merge(in, s, e, lo, hi, hi_open, false, nullptr, nullptr, max_seen, &wrapped);
    uint32_t from, total;
    if (N == 32) {
        uint32_t incl = cnt;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
            if (l >= o) incl += y;
        }
        from = incl - cnt;
        total = __shfl_sync(0xFFFFFFFFu, incl, 31);
    } else {
        from = block_prefix(cnt, &total);
    }
    slice_merge(in, s, e, lo, hi, hi_open, true, out_col + from, out_cnt + from, max_seen, &wrapped);
    if (wrapped) atomicOr(status, ST_OVERFLOW);
    return total;
}

// What a block keeps while it takes its share of a wave (or of the 1-saddles).
struct Share {
    u64 base;
    uint32_t n_block, n_long, n_released, at;
    uint32_t longs[THREADS];  // a warp's merges from the front, the block's from the back
    Cut cut;
    uint32_t released[RELEASED];
};

// Tells a junction's predecessor of its row; the last successor to do so puts it on the next wave's queue.
__device__ __forceinline__ void release(const DpArgs& a, Share& sh, uint32_t p, uint32_t old, uint32_t* queue, uint32_t* length) {
    if (old != 1u) return;
    const uint32_t k = atomicAdd(&sh.n_released, 1u);
    if (k < uint32_t(RELEASED)) sh.released[k] = p;
    else queue[atomicAdd(length, 1u)] = p;
}

// Merges the rows of `items` consecutive sources (a thread each; the long ones a warp each): ROWS, the D*
// rows of 1-saddles `first` .., into staging; otherwise the J rows of the junctions in `from`, into the
// pool, whose predecessors released go to `to`.
template <bool ROWS>
__device__ __forceinline__ void merge_share(const DpArgs& a, Share& sh, int64_t n1, int64_t first, uint32_t items,
                                            const uint32_t* from, uint32_t* to, uint32_t* to_length, u64* mx) {
    u64* const cursor = ROWS ? &a.sum->pc[PC_CURSOR] : &a.sum->dp_pool_used;
    uint32_t* const col = ROWS ? a.out_col : a.pool_col;
    u64* const cnt = ROWS ? a.out_cnt : a.pool_cnt;
    const u64 room = ROWS ? a.out_cap : a.pool_cap;
    if (threadIdx.x == 0) sh.n_block = sh.n_long = sh.n_released = 0;
    const bool has = threadIdx.x < items;
    uint32_t id = 0, bound = 0;
    int64_t e0 = 0, e1 = 0;
    Inputs in{};
    if (has) {
        id = ROWS ? uint32_t(first + threadIdx.x) : from[first + threadIdx.x];
        if (!ROWS) {
            e0 = a.in_ptr[id];
            e1 = a.in_ptr[id + 1];
        }
        in = inputs_of(a, ROWS ? int64_t(id) : n1 + id, &bound);
    }
    const bool mine = bound <= LONG_ROW;
    uint32_t total;
    const uint32_t at = block_prefix(mine ? bound : 0u, &total);  // a barrier: the share's counts are clear
    if (!mine) {
        if (bound <= BLOCK_ROW) sh.longs[atomicAdd(&sh.n_long, 1u)] = id;
        else sh.longs[THREADS - 1 - atomicAdd(&sh.n_block, 1u)] = id;
    }
    if (threadIdx.x == 0) sh.base = total ? atomicAdd(cursor, u64(total)) : 0ull;
    __syncthreads();
    auto done = [&](uint32_t i, u64 off, uint32_t len) {
        if (ROWS) {
            a.row_start[i] = int64_t(off);
            a.row_len[i] = len;
        } else {
            a.j_off[i] = off;
            a.j_len[i] = len;
        }
    };
    if (has && mine) {
        const u64 off = sh.base + at;
        uint32_t len = 0;
        if (off + bound <= room) len = merge_into(in, col + off, cnt + off, bound, mx, a.status);
        else atomicOr(a.status, ST_RETRY);  // too little room: the host grows it and reruns
        done(id, off, len);
        if (!ROWS)
            for (int64_t e = e0; e < e1; e += 4) {
                uint32_t p[4], old[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) p[k] = e + k < e1 ? a.in_idx[e + k] : 0u;
#pragma unroll
                for (int k = 0; k < 4; ++k) old[k] = e + k < e1 ? atomicSub(&a.pend[p[k]], 1u) : 0u;
#pragma unroll
                for (int k = 0; k < 4; ++k) release(a, sh, p[k], old[k], to, to_length);
            }
    }
    // the merges of N threads: one bump of the pool's pointer, the merge, the predecessors
    auto merge_long = [&](auto threads, uint32_t j) {
        constexpr int N = decltype(threads)::value;
        const int l = N == 32 ? int(threadIdx.x & 31) : int(threadIdx.x);
        uint32_t b;
        const Inputs rows = inputs_of(a, ROWS ? int64_t(j) : n1 + j, &b);
        u64 off = 0;
        if (N == 32) {
            if (l == 0) off = atomicAdd(cursor, u64(b));
            off = __shfl_sync(0xFFFFFFFFu, off, 0);
        } else {
            __syncthreads();
            if (l == 0) sh.base = atomicAdd(cursor, u64(b));
            __syncthreads();
            off = sh.base;
        }
        uint32_t len = 0;
        if (off + b <= room) len = merge_by<N>(rows, b, col + off, cnt + off, mx, a.status, sh.cut);  // uniform
        else if (l == 0) atomicOr(a.status, ST_RETRY);
        if (l == 0) done(j, off, len);
        if (!ROWS)
            for (int64_t e = a.in_ptr[j] + l; e < a.in_ptr[j + 1]; e += N) {
                const uint32_t p = a.in_idx[e];
                release(a, sh, p, atomicSub(&a.pend[p], 1u), to, to_length);
            }
    };
    const uint32_t n_long = sh.n_long, n_block = sh.n_block;
    for (uint32_t i = threadIdx.x / 32; i < n_long; i += THREADS / 32) merge_long(std::integral_constant<int, 32>{}, sh.longs[i]);
    for (uint32_t i = 0; i < n_block; ++i) merge_long(std::integral_constant<int, THREADS>{}, sh.longs[THREADS - 1 - i]);
    __syncthreads();
    if (!ROWS) {
        const uint32_t n = min(sh.n_released, uint32_t(RELEASED));
        if (threadIdx.x == 0) sh.at = n ? atomicAdd(to_length, n) : 0u;
        __syncthreads();
        for (uint32_t i = threadIdx.x; i < n; i += THREADS) to[sh.at + i] = sh.released[i];
        __syncthreads();
    }
}

// One wave, the `wave`-th of its loop iteration: the J rows of its queue's junctions, dealt out evenly
// over the blocks, and the queue of the next wave.
__global__ void __launch_bounds__(THREADS, 4) dp_wave(DpArgs a, int wave) {
    int64_t n1, nj;
    if (!counts_of(a, n1, nj)) return;
    const uint32_t n = a.sum->dp_queue[wave];
    if (!n) return;
    __shared__ Share sh;
    u64 mx = 0;
    const uint32_t each = (n + gridDim.x - 1) / gridDim.x;
    const uint64_t begin = uint64_t(blockIdx.x) * each, end = min(uint64_t(n), begin + each);
    for (uint64_t i = begin; i < end; i += THREADS)
        merge_share<false>(a, sh, n1, int64_t(i), uint32_t(min(uint64_t(THREADS), end - i)), a.queue[wave & 1],
                           a.queue[(wave & 1) ^ 1], &a.sum->dp_queue[wave + 1], &mx);
}

// End of WAVES waves (an even number, so the queues keep their parity): count those that had junctions, and
// go on while the next one has.
__global__ void dp_decide(Summary* sum, int64_t max_iter, cudaGraphConditionalHandle h, int use_handle) {
    ++sum->dp_iters;
    for (int i = 0; i < WAVES; ++i) {
        if (!sum->dp_queue[i]) continue;
        ++sum->pc[PC_ITER];
        sum->dp_junctions_done += sum->dp_queue[i];
    }
    const uint32_t next = sum->dp_queue[WAVES];
    for (int i = 0; i <= WAVES; ++i) sum->dp_queue[i] = i == 0 ? next : 0u;
    bool more = next != 0 && !pass_retrying(&sum->status);
    if (sum->pc[PC_ITER] && int64_t(sum->pc[PC_ITER]) >= max_iter) {
        atomicOr(&sum->status, uint32_t(ST_ITER));
        more = false;
    }
    sum->loop_flag[3] = more ? 1u : 0u;
    if (use_handle) cudaGraphSetConditional(h, more ? 1u : 0u);
}

// D* rows: the merge of each 1-saddle's slots, into staging.  Also checks that every junction
// was reached by the waves (the minor is a DAG, so it must be).
__global__ void __launch_bounds__(THREADS, 4) dp_rows(DpArgs a) {
    int64_t n1, nj;
    if (!counts_of(a, n1, nj)) return;
    if (blockIdx.x == 0 && threadIdx.x == 0 && a.sum->dp_junctions_done != u64(nj)) atomicOr(a.status, ST_INTERNAL);
    __shared__ Share sh;
    u64 mx = 0;
    for (int64_t s = int64_t(blockIdx.x) * THREADS; s < n1; s += int64_t(gridDim.x) * THREADS) {
        merge_share<true>(a, sh, n1, s, uint32_t(min(int64_t(THREADS), n1 - s)), nullptr, nullptr, nullptr, &mx);
    }
    for (int o = 16; o; o >>= 1) mx = max(mx, (u64)__shfl_xor_sync(0xFFFFFFFFu, mx, o));
    if ((threadIdx.x & 31) == 0 && mx) atomicMax(&a.sum->pc[PC_MAX], mx);
}

struct WaveCtx {
    int grid;
    DpArgs a;
};

void wave_body(Plan* p, cudaStream_t s, cudaGraphConditionalHandle h, void* ctx) {
    const WaveCtx& c = *static_cast<WaveCtx*>(ctx);
    for (int i = 0; i < WAVES; ++i) dp_wave<<<c.grid, THREADS, 0, s>>>(c.a, i);
    dp_decide<<<1, 1, 0, s>>>(p->dsum(), p->opts.max_iterations, h, h != 0);
}

}  // namespace

// Enqueues the junction DP and, unless only J is wanted, the D* rows into staging (the caller scans and
// gathers them).
// pool_cap / out_cap: capacities of the J-row pool and of the staging.
msc_status run_junction_dp(Plan* p, cudaStream_t s, uint64_t pool_cap, uint64_t out_cap) {
    msc_status st;
    const int64_t cap1 = p->capturing ? p->caps.cells[1] : p->counts[1];
    const int64_t capj = p->capturing ? p->caps.nj : p->n_junctions;
    const size_t njc = size_t(capj ? capj : 1);
    if ((st = ensure(p, p->dp_pend, sizeof(uint32_t) * njc))) return st;
    if ((st = ensure(p, p->dp_queues, sizeof(uint32_t) * 2 * njc))) return st;
    if ((st = ensure(p, p->dp_in_cnt, sizeof(uint32_t) * 2 * njc))) return st;  // counts, then fill cursors
    if ((st = ensure(p, p->dp_in_ptr, sizeof(int64_t) * (njc + 1)))) return st;
    if ((st = ensure(p, p->dp_in_idx, sizeof(uint32_t) * 4 * njc))) return st;
    if ((st = ensure(p, p->dp_j_off, sizeof(u64) * njc))) return st;
    if ((st = ensure(p, p->dp_j_len, sizeof(uint32_t) * njc))) return st;
    if ((st = ensure(p, p->dp_pool_col, sizeof(uint32_t) * size_t(pool_cap ? pool_cap : 1)))) return st;
    if ((st = ensure(p, p->dp_pool_cnt, sizeof(u64) * size_t(pool_cap ? pool_cap : 1)))) return st;
    // a scratch of its own: a captured pass keeps pointers to minor_scan, which must not grow for a J asked
    // for between its replays
    if ((st = ensure(p, p->dp_scan, row_scan_scratch_bytes(capj)))) return st;
    DpArgs a{};
    a.tgt = static_cast<const uint32_t*>(p->trace.ptr);
    a.kinds = static_cast<const uint32_t*>(p->trace_kinds.ptr);
    a.n1_dev = &p->dsum()->counts[1];
    a.nj_dev = &p->dsum()->n_junctions;
    a.cap1 = cap1;
    a.capj = capj;
    a.pend = static_cast<uint32_t*>(p->dp_pend.ptr);
    a.queue[0] = static_cast<uint32_t*>(p->dp_queues.ptr);
    a.queue[1] = a.queue[0] + njc;
    a.in_cnt = static_cast<uint32_t*>(p->dp_in_cnt.ptr);
    a.in_fill = a.in_cnt + njc;
    a.in_ptr = static_cast<int64_t*>(p->dp_in_ptr.ptr);
    a.in_idx = static_cast<uint32_t*>(p->dp_in_idx.ptr);
    a.j_off = static_cast<u64*>(p->dp_j_off.ptr);
    a.j_len = static_cast<uint32_t*>(p->dp_j_len.ptr);
    a.pool_col = static_cast<uint32_t*>(p->dp_pool_col.ptr);
    a.pool_cnt = static_cast<u64*>(p->dp_pool_cnt.ptr);
    a.pool_cap = pool_cap;
    a.out_col = static_cast<uint32_t*>(p->pc_col.ptr);
    a.out_cnt = static_cast<u64*>(p->pc_cnt.ptr);
    a.out_cap = out_cap;
    a.row_start = static_cast<int64_t*>(p->pc_rowstart.ptr);
    a.row_len = static_cast<uint32_t*>(p->pc_rowlen.ptr);
    a.sum = p->dsum();
    a.status = p->status_word();
    if ((st = check_cuda(p, cudaMemsetAsync(a.in_cnt, 0, sizeof(uint32_t) * 2 * njc, s), "memset"))) return st;
    // the wave state of the summary (a rerun of the stage starts it afresh)
    if (!p->capturing && (st = check_cuda(p, cudaMemsetAsync(&p->dsum()->dp_pool_used, 0,
                                                             offsetof(Summary, loop_flag) - offsetof(Summary, dp_pool_used), s),
                                          "memset")))
        return st;
    const int gj = grid_cap(p, capj, THREADS, 8);
    dp_init<<<gj, THREADS, 0, s>>>(a);
    launched(p);
    if ((st = check_cuda(p, row_scan(p, a.in_cnt, a.nj_dev, capj, a.in_ptr, static_cast<u64*>(p->dp_scan.ptr), s),
                         "predecessor scan")))
        return st;
    dp_fill<<<gj, THREADS, 0, s>>>(a);
    launched(p);
    if ((st = check_cuda(p, cudaGetLastError(), "junction dp launch"))) return st;
    record_event(p, p->kev0, s);
    WaveCtx ctx{grid_cap(p, capj, 4, 8), a};
    if ((st = run_loop(p, s, 2, WAVES + 1, wave_body, &ctx))) return st;
    if (p->j_only) return MSC_OK;
    dp_rows<<<grid_cap(p, cap1, THREADS, 8), THREADS, 0, s>>>(a);
    record_event(p, p->kev1, s);
    launched(p);
    return check_cuda(p, cudaGetLastError(), "junction dp launch");
}

}  // namespace msc
