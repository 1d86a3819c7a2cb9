// Suffix order of a few thousand tokens by one block, shared by the build of request trees and the online insert
// into the global tree.
#pragma once

#include "common.cuh"

namespace {

// Everything in shared memory, by prefix doubling.  After a round every suffix has the rank of its
// first k tokens, and the order by the tokens behind those is the current order moved k places back, so a
// round only has to sort by rank, stably: one or two radix passes of 7 bits.  A last round that adds fewer
// than k tokens looks at an overlapping window.  A rank also tells whether the sequence ends right
// behind the k tokens, so that suffixes of equal rank either all go on or are equal altogether, and the ones that
// have nothing k places on may take any place.  Order: by the first D tokens, a suffix that ends earlier before its
// extensions.  Bound by the latency of a pass (one block: barriers, and 32 items per warp and step ranked by
// ballots).  (A bitonic sort that compared tokens took 78 - 91 stages: 83 us for 4 x 4,096 tokens, 390 for 64 x 8,192;
// now 49 and 105.)
constexpr int BS_THREADS = 1024;               // of the kernel that sorts prompts
constexpr int BS_MAX_LEN = 16384;              // most tokens (two passes of 7 bits per round; 112 KB)
constexpr int BS_BITS = 7;
constexpr int BS_BINS = 1 << BS_BITS;
constexpr int BS_ROW = BS_BINS + 1;            // (rows of 128 counters put the eight threads that add up a digit on one bank: a sort of 4 x 4,096 tokens took 60 us, 49 now)

template <int THREADS, int ITEMS>
constexpr int block_order_smem() { return (int)(sizeof(int) * (THREADS / 32) * BS_ROW + 3 * sizeof(unsigned short) * THREADS * ITEMS); }

// All THREADS (512 or 1,024) threads call; ITEMS per thread: n <= THREADS * ITEMS tokens.  token(i) < 2^tok_bits; position i belongs to the
// sequence [begin(i), end(i)).  Returns the order (positions, in shared memory).
template <int THREADS, int ITEMS, class Tok, class Begin, class End>
__device__ __forceinline__ unsigned short* block_suffix_order(unsigned char* smem, int* wsum, int n, int tok_bits, int D, Tok token,
                                                              Begin begin, End end) {
    constexpr int WARPS = THREADS / 32, SHARE = WARPS / 4;      // threads that add up one digit, four warps' counts each
    static_assert(BS_BINS * SHARE == THREADS, "a thread per digit and four warps");
    int (*hist)[BS_ROW] = reinterpret_cast<int (*)[BS_ROW]>(smem);                  // [WARPS][BS_ROW]
    unsigned short* const rank = reinterpret_cast<unsigned short*>(smem + sizeof(int) * WARPS * BS_ROW);
    unsigned short* cur = rank + THREADS * ITEMS;                                // the order so far
    unsigned short* nxt = cur + THREADS * ITEMS;
    const int tid = threadIdx.x, lane = tid & 31, wib = tid >> 5;
    const unsigned lt = (1u << lane) - 1u;
    const int p0 = wib * 32 * ITEMS + lane;                     // a warp's places are consecutive, 32 per step

    // one stable pass: `val` of every place goes by bits [shift, shift + 7) of its key
    unsigned short val[ITEMS];
    auto pass = [&](int shift, auto key_of) {
        for (int k = lane; k < BS_BINS; k += 32) hist[wib][k] = 0;
        __syncwarp();
        int at[ITEMS];                                          // digit, and place among the warp's items of that digit
#pragma unroll
        for (int u = 0; u < ITEMS; ++u) {
            const bool in = p0 + u * 32 < n;
            const unsigned active = __ballot_sync(0xffffffffu, in);
            at[u] = 0;
            if (!active) continue;
            const int digit = in ? (int)((key_of(val[u]) >> shift) & (BS_BINS - 1)) : 0;
            unsigned peers = active;
#pragma unroll
            for (int k = 0; k < BS_BITS; ++k) {
                const unsigned m = __ballot_sync(0xffffffffu, (digit >> k) & 1);
                peers &= ((digit >> k) & 1) ? m : ~m;
            }
            int base = 0;
            if (in) base = hist[wib][digit];
            __syncwarp();
            if (in && (peers & lt) == 0u) hist[wib][digit] = base + __popc(peers);
            __syncwarp();
            at[u] = digit | ((base + __popc(peers & lt)) << BS_BITS);
        }
        __syncthreads();
        {
            // counts to first places, in the order (digit, warp): a thread takes four warps of one digit
            const int digit = tid / SHARE, w0 = tid % SHARE * 4;
            int c[4], sum = 0;
#pragma unroll
            for (int q = 0; q < 4; ++q) { c[q] = hist[w0 + q][digit]; sum += c[q]; }
            int inc = sum;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, inc, o);
                if (lane >= o) inc += y;
            }
            if (lane == 31) wsum[wib] = inc;
            __syncthreads();
            int before = lane < wib ? wsum[lane] : 0;
            before = (int)__reduce_add_sync(0xffffffffu, (unsigned)before) + inc - sum;
#pragma unroll
            for (int q = 0; q < 4; ++q) { hist[w0 + q][digit] = before; before += c[q]; }
        }
        __syncthreads();
#pragma unroll
        for (int u = 0; u < ITEMS; ++u)
            if (p0 + u * 32 < n) nxt[hist[wib][at[u] & (BS_BINS - 1)] + (at[u] >> BS_BITS)] = val[u];
        __syncthreads();
        unsigned short* const x = cur; cur = nxt; nxt = x;
    };
    auto load = [&]() {
#pragma unroll
        for (int u = 0; u < ITEMS; ++u) val[u] = p0 + u * 32 < n ? cur[p0 + u * 32] : 0;
    };
    // ranks (from 0) of the order `cur`, a new one where `differs` from the suffix before; returns their number
    auto rerank = [&](auto differs) -> int {
        load();
        unsigned flags[ITEMS];
        int mine = 0;
#pragma unroll
        for (int u = 0; u < ITEMS; ++u) {
            const int p = p0 + u * 32;
            flags[u] = __ballot_sync(0xffffffffu, p < n && (p == 0 || differs((int)val[u], (int)cur[p - 1])));
            mine += __popc(flags[u]);
        }
        if (lane == 0) wsum[wib] = mine;
        __syncthreads();                                        // all old ranks have been read
        const int c = lane < WARPS ? wsum[lane] : 0;
        int r = (int)__reduce_add_sync(0xffffffffu, lane < wib ? (unsigned)c : 0u) - 1;
        const int all = (int)__reduce_add_sync(0xffffffffu, (unsigned)c);
#pragma unroll
        for (int u = 0; u < ITEMS; ++u) {
            if (p0 + u * 32 < n) rank[val[u]] = (unsigned short)(r + __popc(flags[u] & (lt | (1u << lane))));
            r += __popc(flags[u]);
        }
        __syncthreads();
        return all;
    };

    // ---- by the first token, and whether it is the last one
    auto token_key = [&](int i) -> unsigned { return ((unsigned)token(i) << 1) | (i + 1 < end(i) ? 1u : 0u); };
#pragma unroll
    for (int u = 0; u < ITEMS; ++u) val[u] = (unsigned short)(p0 + u * 32);
    for (int shift = 0; shift < tok_bits + 1; shift += BS_BITS) {
        if (shift > 0) load();
        pass(shift, [&](int i) { return token_key(i); });
    }
    for (int k = 1, off; k < D; k += off) {
        off = min(k, D - k);
        // ranks of the first k tokens
        int ranks;
        if (k == 1) ranks = rerank([&](int i, int h) { return token_key(i) != token_key(h); });
        else {
            const int o = k >> 1;                               // (every round but the last doubles)
            ranks = rerank([&](int i, int h) {
                return rank[i] != rank[h] || (i + o < end(i) ? (int)rank[i + o] : -1) != (h + o < end(h) ? (int)rank[h + o] : -1);
            });
        }
        if (ranks == n) break;                                  // no two alike: the order is final
        // the order by what follows `off` places on, then by rank
        load();
#pragma unroll
        for (int u = 0; u < ITEMS; ++u) {
            const int q = p0 + u * 32 < n ? val[u] : 0, first = begin(q), e = end(q);
            val[u] = (unsigned short)(q - off >= first ? q - off : e - min(off, e - first) + (q - first));
        }
        __syncthreads();
        pass(0, [&](int i) { return (unsigned)rank[i]; });
        if (ranks > BS_BINS) { load(); __syncthreads(); pass(BS_BITS, [&](int i) { return (unsigned)rank[i]; }); }
    }
    return cur;
}

}  // namespace
