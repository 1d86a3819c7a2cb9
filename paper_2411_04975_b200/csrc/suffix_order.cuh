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
constexpr int BS_THREADS = 1024;               // of the kernel that sorts prompts (of up to 1,024 tokens: BS_SMALL)
constexpr int BS_SMALL = 256;
constexpr int BS_MAX_LEN = 16384;              // most tokens (two passes of 7 bits per round; 112 KB)
constexpr int BS_BITS = 7;
constexpr int BS_BINS = 1 << BS_BITS;
constexpr int BS_ROW = BS_BINS + 1;            // (rows of 128 counters put the eight threads that add up a digit on one bank: a sort of 4 x 4,096 tokens took 60 us, 49 now)

template <int THREADS, int ITEMS>
constexpr int block_order_smem() { return (int)(sizeof(int) * (THREADS / 32) * BS_ROW + 3 * sizeof(unsigned short) * THREADS * ITEMS); }

// All THREADS (256, 512 or 1,024) threads call; ITEMS per thread: n <= THREADS * ITEMS tokens.  token(i) < 2^tok_bits; position i belongs to the
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

// ---------------------------------------------------------------------------------------------
// The same by a cluster of blocks, for up to 131,072 tokens: prompts where there are fewer of them than multiprocessors, and
// small corpora.  Block c of the cluster owns THREADS x ITEMS consecutive places of the order and the ranks of as many
// positions, in its shared memory; what a pass moves goes to its place in another block's shared memory directly, ranks
// of positions elsewhere are read there, and the blocks meet at the cluster's barrier (some 300 cycles; a grid barrier takes 1.5 us
// and what crosses it comes from L2).  A pass: a warp ranks its items by ballots, the blocks tell one another their digit counts,
// and every item goes to its place.
//
// As in the corpus sort a rank's lowest bit tells whether the sequence goes on behind the tokens that it stands for.
constexpr int CS_BITS = 8;
constexpr int CS_BINS = 1 << CS_BITS;
constexpr int CS_ROW = CS_BINS + 1;
constexpr int CS_MOST = 16;                                      // blocks of a cluster

template <int THREADS, int ITEMS>
struct ClusterOrder {
    int hist[THREADS / 32][CS_ROW];
    int tot[CS_MOST][CS_BINS];                                   // digit counts of the cluster's blocks
    int base[CS_BINS];
    int ranks[CS_MOST];
    int wsum[THREADS / 32];
    unsigned rank[THREADS * ITEMS];                           // by position
    unsigned long long place[2][THREADS * ITEMS];             // position and, in the upper half, key by place
};

__device__ __forceinline__ unsigned cluster_rank() { unsigned r; asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r)); return r; }
__device__ __forceinline__ unsigned cluster_blocks() { unsigned r; asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r)); return r; }
__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release;\nbarrier.cluster.wait.acquire;" ::: "memory");
}
__device__ __forceinline__ unsigned cluster_address(const void* p, unsigned block) {
    unsigned a;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"((unsigned)__cvta_generic_to_shared(p)), "r"(block));
    return a;
}
__device__ __forceinline__ void cluster_store(const void* p, unsigned block, unsigned v) {
    asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(cluster_address(p, block)), "r"(v) : "memory");
}
__device__ __forceinline__ void cluster_store(const void* p, unsigned block, unsigned long long v) {
    asm volatile("st.shared::cluster.u64 [%0], %1;" ::"r"(cluster_address(p, block)), "l"(v) : "memory");
}
__device__ __forceinline__ unsigned long long cluster_load64(const void* p, unsigned block) {
    unsigned long long v;
    asm volatile("ld.shared::cluster.u64 %0, [%1];" : "=l"(v) : "r"(cluster_address(p, block)) : "memory");
    return v;
}
__device__ __forceinline__ unsigned cluster_load(const void* p, unsigned block) {
    unsigned v;
    asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(cluster_address(p, block)) : "memory");
    return v;
}

// All threads of all blocks of the cluster call.  n <= blocks * THREADS * ITEMS tokens; token(i) < 2^tok_bits; goes_on(i): position
// i + 1 belongs to the same sequence; back(i, off): the position off places in front of i, or, where that is another sequence, one of
// the last `off` of i's sequence, each for one of its first.  Returns this block's part of the order: place
// cluster_rank() * THREADS * ITEMS + k is in the lower half of [k].  The other blocks' shared memory is not touched any more.
template <int THREADS, int ITEMS, class Tok, class GoesOn, class Back>
__device__ __forceinline__ const unsigned long long* cluster_suffix_order(ClusterOrder<THREADS, ITEMS>& sh, int n, int tok_bits, int D, Tok token, GoesOn goes_on,
                                                                Back back) {
    constexpr unsigned FULL = 0xffffffffu;
    constexpr int PART = THREADS * ITEMS, WARPS = THREADS / 32;
    constexpr int SHARE = THREADS / CS_BINS, PER = WARPS / SHARE;                   // threads that add up one digit, PER warps' counts each
    constexpr unsigned NONE = 0xffffffffu;
    const int tid = threadIdx.x, lane = tid & 31, wib = tid >> 5;
    const unsigned blocks = cluster_blocks(), me = cluster_rank(), lt = (1u << lane) - 1u;
    const int first = (int)me * PART, p0 = wib * 32 * ITEMS + lane;                 // this block's places; a warp's are consecutive
    int cur = 0;
    auto rank_of = [&](int i) { return cluster_load(&sh.rank[i % PART], (unsigned)(i / PART)); };
    unsigned val[ITEMS], key[ITEMS];
    auto load = [&]() {
#pragma unroll
        for (int u = 0; u < ITEMS; ++u) {
            const unsigned long long x = first + p0 + u * 32 < n ? sh.place[cur][p0 + u * 32] : 0ull;
            val[u] = (unsigned)x; key[u] = (unsigned)(x >> 32);
        }
    };
    // one stable pass by bits [shift, shift + CS_BITS) of the keys; they go along
    auto pass = [&](int shift) {
        for (int k = lane; k < CS_BINS; k += 32) sh.hist[wib][k] = 0;
        int at[ITEMS];
        __syncwarp();
#pragma unroll
        for (int u = 0; u < ITEMS; ++u) {
            const bool in = first + p0 + u * 32 < n;
            unsigned peers = __ballot_sync(FULL, in);
            at[u] = 0;
            if (!peers) continue;
            const int digit = (int)((key[u] >> shift) & (CS_BINS - 1));
#pragma unroll
            for (int k = 0; k < CS_BITS; ++k) {
                const unsigned m = __ballot_sync(FULL, (digit >> k) & 1);
                peers &= ((digit >> k) & 1) ? m : ~m;
            }
            int base = 0;
            if (in) base = sh.hist[wib][digit];
            __syncwarp();
            if (in && (peers & lt) == 0u) sh.hist[wib][digit] = base + __popc(peers);
            __syncwarp();
            at[u] = digit | ((base + __popc(peers & lt)) << CS_BITS);
        }
        __syncthreads();
        {
            // counts of the warps before, and the block's count to all blocks
            const int digit = tid / SHARE, k = tid % SHARE, w0 = k * PER;
            int c[PER], sum = 0;
#pragma unroll
            for (int q = 0; q < PER; ++q) { c[q] = sh.hist[w0 + q][digit]; sum += c[q]; }
            int inc = sum;
#pragma unroll
            for (int o = 1; o < SHARE; o <<= 1) {
                const int y = __shfl_up_sync(FULL, inc, o, SHARE);
                if (k >= o) inc += y;
            }
            int before = inc - sum;
#pragma unroll
            for (int q = 0; q < PER; ++q) { sh.hist[w0 + q][digit] = before; before += c[q]; }
            const int all = __shfl_sync(FULL, inc, SHARE - 1, SHARE);
            for (unsigned b = k; b < blocks; b += SHARE) cluster_store(&sh.tot[me][digit], b, (unsigned)all);
        }
        cluster_sync();
        if (tid < CS_BINS) {
            int all = 0, mine = 0;
#pragma unroll 4
            for (unsigned b = 0; b < blocks; ++b) { const int c = sh.tot[b][tid]; all += c; mine += b < me ? c : 0; }
            int inc = all;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(FULL, inc, o);
                if (lane >= o) inc += y;
            }
            if (lane == 31) sh.wsum[wib] = inc;
            asm volatile("bar.sync 1, %0;" ::"r"(CS_BINS) : "memory");
            inc += (int)__reduce_add_sync(FULL, lane < wib ? (unsigned)sh.wsum[lane] : 0u);
            sh.base[tid] = inc - all + mine;
        }
        __syncthreads();
#pragma unroll
        for (int u = 0; u < ITEMS; ++u)
            if (first + p0 + u * 32 < n) {
                const int digit = at[u] & (CS_BINS - 1), to = sh.base[digit] + sh.hist[wib][digit] + (at[u] >> CS_BITS);
                cluster_store(&sh.place[cur ^ 1][to % PART], (unsigned)(to / PART), ((unsigned long long)key[u] << 32) | val[u]);
            }
        cluster_sync();
        cur ^= 1;
    };
    // ranks of the order, a new one where the rank or the one o places on (o > 0) differs from the place before; returns their number
    auto rerank = [&](int o) -> int {
        auto second = [&](unsigned i, unsigned a) { return o > 0 ? ((a & 1u) ? rank_of((int)i + o) : NONE) : 1u; };
        load();
        unsigned b[ITEMS], flags[ITEMS], pa = NONE, pb = NONE;
        int mine = 0;
#pragma unroll
        for (int u = 0; u < ITEMS; ++u) { b[u] = 0u; if (first + p0 + u * 32 < n) b[u] = second(val[u], key[u]); }
        const int before = first + wib * 32 * ITEMS - 1;        // the place in front of the warp's
        if (lane == 0 && before >= 0 && before + 1 < n) {
            const unsigned long long x = cluster_load64(&sh.place[cur][before % PART], (unsigned)(before / PART));
            pa = (unsigned)(x >> 32);
            pb = second((unsigned)x, pa);
        }
#pragma unroll
        for (int u = 0; u < ITEMS; ++u) {
            unsigned xa = __shfl_up_sync(FULL, key[u], 1), xb = __shfl_up_sync(FULL, b[u], 1);
            if (lane == 0) { xa = pa; xb = pb; }
            pa = __shfl_sync(FULL, key[u], 31); pb = __shfl_sync(FULL, b[u], 31);
            const int p = first + p0 + u * 32;
            flags[u] = __ballot_sync(FULL, p < n && (p == 0 || key[u] != xa || b[u] != xb));
            mine += __popc(flags[u]);
        }
        if (lane == 0) sh.wsum[wib] = mine;
        __syncthreads();
        const int c = lane < WARPS ? sh.wsum[lane] : 0;
        int r = (int)__reduce_add_sync(FULL, lane < wib ? (unsigned)c : 0u) - 1;
        const int all = (int)__reduce_add_sync(FULL, (unsigned)c);
        if ((unsigned)tid < blocks) cluster_store(&sh.ranks[me], (unsigned)tid, (unsigned)all);
        cluster_sync();                                         // (all old ranks have been read)
        int ranks = 0;
        for (unsigned q = 0; q < blocks; ++q) { const int x = sh.ranks[q]; ranks += x; r += q < me ? x : 0; }
#pragma unroll
        for (int u = 0; u < ITEMS; ++u) {
            if (first + p0 + u * 32 < n) {
                const unsigned on = key[u] & 1u & (b[u] == NONE ? 0u : b[u]);
                const unsigned to = val[u] / PART;
                cluster_store(&sh.rank[val[u] % PART], to, (unsigned)(r + __popc(flags[u] & (lt | (1u << lane)))) * 2u + on);
            }
            r += __popc(flags[u]);
        }
        cluster_sync();
        return ranks;
    };

    // ---- by the first token, and whether it is the last one
#pragma unroll
    for (int u = 0; u < ITEMS; ++u) {
        const int q = p0 + u * 32, i = first + q;
        key[u] = i < n ? ((unsigned)token(i) << 1) | (goes_on(i) ? 1u : 0u) : 0u;
        val[u] = (unsigned)i;
    }
    cluster_sync();                                             // (the others are there)
    for (int shift = 0; shift < tok_bits + 1; shift += CS_BITS) {
        if (shift > 0) load();
        pass(shift);
    }
    for (int k = 1, off; k < D; k += off) {
        off = min(k, D - k);
        const int ranks = rerank(k >> 1);                       // (every round but the last doubles)
        if (ranks == n) break;                                  // no two alike: the order is final
        // the order by what follows `off` places on, then by rank
#pragma unroll
        for (int u = 0; u < ITEMS; ++u)
            if (first + p0 + u * 32 < n) { val[u] = (unsigned)back((int)val[u], off); key[u] = rank_of((int)val[u]); }
        pass(1);                                                // (the lowest bit is the same for equal ranks)
        for (int shift = CS_BITS; ((unsigned)(ranks - 1) >> shift) != 0u; shift += CS_BITS) { load(); pass(shift + 1); }
    }
    return sh.place[cur];
}

}  // namespace
