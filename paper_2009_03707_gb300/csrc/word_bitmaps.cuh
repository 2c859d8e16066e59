// Bitmaps of the finished gradient words: the critical cells per slot (a2) and what the
// saddle-saddle reachability starts from (a4), each 32 vertices of a row to a word.
//
// A slot's code has three bits, and every bitmap is a function of the three.  So a warp takes the words
// of 32 vertices, a lane each, and transposes them as a 32 x 32 bit matrix (five exchanges of half the
// bits with the lane 16, 8, 4, 2 and 1 away): lane k then holds bit k of all 32, and with two shuffles
// more lane 3 s has slot s's three bits, each bitmap one logic instruction.  (One ballot per bit instead:
// votes issue too slowly, 0.138 ms for both sorts on the 256^3 GRF; one per bitmap, as two kernels that
// each read the words: 0.046 and 0.095 ms; 0.065 ms so.)  A warp takes `chunk` (4..32, a multiple of
// WB_WORDS) consecutive row words, WB_WORDS words' loads issued together, keeps their bitmaps in shared
// memory and writes all of them with one store per array, a lane a word.  Large grids take chunks of 32
// (the stores fully coalesced), small ones smaller chunks so that enough warps share the work.  A
// replayed pass makes both sorts from one reading of the words; stage by stage each is made when it is
// asked for.
#pragma once

#include "msc_internal.cuh"

namespace msc {

constexpr int WB_THREADS = 256;
constexpr int WB_WORDS = 4;

struct WordBitmaps {
    const uint32_t* words;
    uint32_t* crit_bits;  // [slot][z][y][w]
    // per vertex-row word, 1-cell row layout: for each axis the four masks of 1-cells paired with the quad
    // on the - / + side along the first / second other axis, and R_0 = the 1-saddles (R1: the second set)
    uint4* masks;
    uint32_t* R0;
    uint32_t* R1;
    uint32_t* qdown;  // [even axis][z][y][w]: quads that are critical or paired with a facet
    uint32_t* stamp;  // per row: every row is new at the start
};

// The transpose of the warp's 32 x 32 bits: lane r's result has bit c where lane c's x had bit r.  A step
// exchanges the blocks whose row and column numbers differ in one bit; `keep` and `turn` are the lane's
// own (set_up): what it keeps, and the rotation that brings the other lane's half into place.
struct Transpose {
    uint32_t keep[5], turn[5];
    __device__ __forceinline__ void set_up(int lane) {
        constexpr uint32_t M[5] = {0x0000FFFFu, 0x00FF00FFu, 0x0F0F0F0Fu, 0x33333333u, 0x55555555u};
#pragma unroll
        for (int i = 0; i < 5; ++i) {
            const int j = 16 >> i;
            keep[i] = lane & j ? ~M[i] : M[i];
            turn[i] = lane & j ? 32 - j : j;
        }
    }
    __device__ __forceinline__ uint32_t operator()(uint32_t x) const {
#pragma unroll
        for (int i = 0; i < 5; ++i) {
            const uint32_t y = __shfl_xor_sync(0xFFFFFFFFu, x, 16 >> i);
            x = (x & keep[i]) | (__funnelshift_l(y, y, turn[i]) & ~keep[i]);
        }
        return x;
    }
};

// The vertices whose code is C, from the code's three bits.
template <int C>
__device__ __forceinline__ uint32_t code_is(const uint32_t b[3]) {
    return (C & 1 ? b[0] : ~b[0]) & (C & 2 ? b[1] : ~b[1]) & (C & 4 ? b[2] : ~b[2]);
}

template <bool CRIT, bool REACH>
static __global__ void __launch_bounds__(WB_THREADS) word_bitmaps(Geom g, WordBitmaps a, int chunk) {
    // per word: 8 critical bitmaps, 3 x 4 partner masks, 3 quad bitmaps (an odd pitch: no bank conflicts)
    constexpr int PITCH = REACH ? 25 : 9, MASKS = 8, QUADS = 20;
    __shared__ uint32_t kept[WB_THREADS / 32][32 * PITCH];
    const int lane = threadIdx.x & 31;
    uint32_t* const mine = kept[threadIdx.x >> 5];
    Transpose transpose;
    transpose.set_up(lane);
    // lane 3 s stands for slot s: 1, 2, 4 are the 1-cells of axis 0, 1, 2, and 6, 5, 3 the quads of even
    // axis 0, 1, 2; codes 2 B + 1 and 2 B + 2 are the partners on the - and + side along B
    const int slot = lane % 3 == 0 && lane < 24 ? lane / 3 : -1;
    const int axis = slot == 1 ? 0 : slot == 2 ? 1 : slot == 4 ? 2 : -1;
    const int even = slot == 6 ? 0 : slot == 5 ? 1 : slot == 3 ? 2 : -1;
    const int64_t nrw = int64_t(g.nz) * g.ny * g.W;
    const int64_t step = ((int64_t(gridDim.x) * WB_THREADS) >> 5) * chunk;
    for (int64_t t0 = ((int64_t(blockIdx.x) * WB_THREADS + threadIdx.x) >> 5) * chunk; t0 < nrw; t0 += step) {
        for (int u0 = 0; u0 < chunk && t0 + u0 < nrw; u0 += WB_WORDS) {  // warp-uniform
            uint32_t word_of[WB_WORDS];
#pragma unroll
            for (int v = 0; v < WB_WORDS; ++v) {
                const uint32_t t = uint32_t(min(t0 + u0 + v, nrw - 1)), row = g.div_W.div(t);
                const uint32_t x = (t - row * uint32_t(g.W)) * 32 + lane;
                word_of[v] = x < uint32_t(g.nx) ? a.words[int64_t(row) * g.nx + x] : 0x00FFFFFFu;  // all codes 7 off-grid
            }
#pragma unroll
            for (int v = 0; v < WB_WORDS; ++v) {
                uint32_t* const to = mine + (u0 + v) * PITCH;
                if (!REACH) {  // only where a code is 0: that bit, at the code's place
                    const uint32_t w = word_of[v];
                    const uint32_t zero = transpose(~(w | (w >> 1) | (w >> 2)));
                    if (slot >= 0) to[slot] = zero;
                    continue;
                }
                uint32_t b[3];
                b[0] = transpose(word_of[v]);
                b[1] = __shfl_down_sync(0xFFFFFFFFu, b[0], 1);
                b[2] = __shfl_down_sync(0xFFFFFFFFu, b[0], 2);
                if (slot >= 0) to[slot] = code_is<0>(b);
                const uint32_t c1 = code_is<1>(b), c2 = code_is<2>(b), c3 = code_is<3>(b), c4 = code_is<4>(b),
                               c5 = code_is<5>(b), c6 = code_is<6>(b);
                if (axis >= 0) {
                    uint32_t* const m = to + MASKS + 4 * axis;
                    m[0] = axis == 0 ? c3 : c1;
                    m[1] = axis == 0 ? c4 : c2;
                    m[2] = axis == 2 ? c3 : c5;
                    m[3] = axis == 2 ? c4 : c6;
                }
                if (even >= 0)  // critical or paired with a facet: not 7 (off the grid), nor along the even axis
                    to[QUADS + even] = ~(code_is<7>(b) | (even == 0 ? c1 | c2 : even == 1 ? c3 | c4 : c5 | c6));
            }
        }
        __syncwarp();
        const int64_t t = t0 + lane;
        if (lane < chunk && t < nrw) {
            const uint32_t* const from = mine + lane * PITCH;
            if (CRIT)
#pragma unroll
                for (int s = 0; s < 8; ++s) a.crit_bits[s * nrw + t] = from[s];
            if (REACH) {
                const uint32_t row = g.div_W.div(uint32_t(t)), z = g.div_ny.div(row), y = row - z * uint32_t(g.ny);
                const int w = int(uint32_t(t) - row * uint32_t(g.W));
                const int64_t e[3] = {g.edge_word(int(z), 0, int(y), 0, w), g.edge_word(int(z), 0, int(y), 1, w),
                                      g.edge_word(int(z), 1, int(y), 0, w)};
#pragma unroll
                for (int k = 0; k < 3; ++k) {
                    const uint32_t* const m = from + MASKS + 4 * k;
                    a.masks[e[k]] = make_uint4(m[0], m[1], m[2], m[3]);
                    a.R0[e[k]] = from[1 << k];
                    a.qdown[k * nrw + t] = from[QUADS + k];
                }
                if (w == 0) a.stamp[row] = 1;
                // the unused slot of the 1-cell layout stays empty in both sets
                a.masks[e[2] + g.W] = make_uint4(0, 0, 0, 0);
                a.R0[e[2] + g.W] = 0;
                a.R1[e[2] + g.W] = 0;
            }
        }
        __syncwarp();  // read before the next words are kept
    }
}

// Row words per warp: 32 when every SM still gets 32 warps' worth, else fewer (at least 4).
template <bool CRIT, bool REACH>
inline cudaError_t launch_word_bitmaps(const Geom& g, const WordBitmaps& a, int num_sms, cudaStream_t s) {
    const int64_t nrw = int64_t(g.nz) * g.ny * g.W, sms = num_sms > 0 ? num_sms : 148;
    int chunk = 32;
    while (chunk > WB_WORDS && nrw < int64_t(chunk) * 32 * sms) chunk >>= 1;
    const int64_t want = ((nrw + chunk - 1) / chunk * 32 + WB_THREADS - 1) / WB_THREADS;
    word_bitmaps<CRIT, REACH><<<unsigned(std::max<int64_t>(1, std::min(want, sms * 8))), WB_THREADS, 0, s>>>(g, a, chunk);
    return cudaGetLastError();
}

}  // namespace msc
