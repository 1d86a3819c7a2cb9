// Offline build of the global suffix tree (Section 3, "Suffix Tree Construction")
// on the GPU: depth-capped suffix sort by prefix doubling, adjacent-suffix LCPs,
// then all depths at once, a lane per depth: sweeps over (lcp, len) give every node's count, children
// and place, and one kernel lays the nodes down as sorted child runs in pre-order.
// Hand-written LSD radix sort and scans (no CUB / Thrust).
// Also: sd_build_requests (the trees of a batch of new requests by the same pipeline).
#include <algorithm>
#include <atomic>
#include <new>
#include <stdio.h>
#include <string.h>
#include <type_traits>
#include <vector>

#include <cooperative_groups.h>

#include "append_core.cuh"
#include "device_memory.h"
#include "global_insert.cuh"
#include "suffix_order.cuh"
#include "tree_limits.h"

namespace cg = cooperative_groups;

namespace {

typedef unsigned long long u64;
typedef long long i64;

// ------------------------------------------------------------------ suffix order
// end_pos[i]: one past the last token of the sequence that holds position i.
__global__ void seq_end_kernel(const int64_t* seq_offsets, int n_seqs, i64 n, int* end_pos) {
    sd_chain_begin();
    i64 i = (i64)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    int lo = 0, hi = n_seqs;                          // largest s with seq_offsets[s] <= i
    while (hi - lo > 1) {
        int mid = (lo + hi) >> 1;
        if (seq_offsets[mid] <= i) lo = mid; else hi = mid;
    }
    end_pos[i] = (int)seq_offsets[lo + 1];
}

// bad[0] != 0 when a token is outside [0, V) or the offsets do not ascend from 0
__global__ void validate_kernel(const int32_t* tok, i64 n, int V, const int64_t* seq_offsets, int n_seqs, int* bad) {
    i64 i = (i64)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n && (tok[i] < 0 || tok[i] >= V)) atomicOr(bad, 1);
    if (i < n_seqs && seq_offsets[i] > seq_offsets[i + 1]) atomicOr(bad, 2);
    if (i == 0 && seq_offsets[0] != 0) atomicOr(bad, 2);
}

// Suffix order of a whole corpus by prefix doubling, in one cooperative launch.  After a round every suffix has
// the rank of its first k tokens, and the order by the tokens behind those is the current order moved k places back, so
// a round only has to sort by rank, stably, with LSD radix passes of 8 bits.  A last round that adds fewer than k
// tokens looks at an overlapping window.  A rank also tells whether the sequence ends right behind the k tokens (its
// lowest bit: the sequence goes on), so that suffixes of equal rank either all go on or are equal altogether, the ones
// that have nothing k places on may take any place, and no look-up of a sequence's end is needed.  Order: by the first D tokens, a suffix that ends earlier before its extensions.
//
// A block owns a chunk of consecutive places throughout.  A pass: digit counts per block; a warp per digit adds them up
// over the blocks; the blocks go through their chunks, SG_THREADS x ITEMS places at a time, ordering each lot in shared
// memory so that what is written is consecutive.  Three grid barriers of about 1.5 us, and for 4.2 M suffixes, which stay
// in L2, one random read per suffix for the keys, one for the new ranks, and what the lots cost in barriers and ballots.  (Separate histogram, scan and scatter launches over 64-bit
// keys, six passes a round: 2.2 ms for 4.2 M suffixes, 0.45 ms for 32,768, of 100 launches.)
constexpr int SG_THREADS = 512;
constexpr int SG_WARPS = SG_THREADS / 32;
constexpr int SG_BINS = 256;
constexpr int SG_BATCH = 8;                       // random reads in flight per thread

struct CorpusSort {
    const int32_t* tok;
    const int64_t* seq_off;
    int n_seqs;
    const int* end_pos;
    int N, chunk;                                 // chunk: a multiple of 32
    unsigned key_bits;                            // of a token and one more
    int D;
    uint32_t *key[2], *val[2];
    int* rank;                                    // [N] rank from 0, times two, + 1: the sequence goes on behind its k tokens (32 bits, unsigned)
    unsigned *flags, *go;                         // [N / 32 + 1] by place: a new rank starts, the sequence goes on
    int* table;                                   // [SG_BINS][blocks]
    int* total;                                   // [SG_BINS]
    int* count;                                   // [blocks]
    uint32_t* sa;                                 // result
};

template <int ITEMS>
struct SortShared {
    int cnt[SG_WARPS][SG_BINS];
    uint32_t key[SG_THREADS * ITEMS], val[SG_THREADS * ITEMS];
    int base[SG_BINS], start[SG_BINS], tot[SG_BINS];
    int wsum[SG_WARPS];
};

// exclusive sum over the block's threads; the total in `all`
__device__ __forceinline__ int sg_block_scan(int v, int* wsum, int tid, int& all) {
    const int lane = tid & 31, wib = tid >> 5;
    int inc = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += y;
    }
    if (lane == 31) wsum[wib] = inc;
    __syncthreads();
    const int c = lane < SG_WARPS ? wsum[lane] : 0;
    const int before = (int)__reduce_add_sync(0xffffffffu, lane < wib ? (unsigned)c : 0u);
    all = (int)__reduce_add_sync(0xffffffffu, (unsigned)c);
    __syncthreads();
    return before + inc - v;
}

template <int ITEMS>
__global__ void __launch_bounds__(SG_THREADS, 2)
corpus_sort_kernel(CorpusSort A) {
    extern __shared__ __align__(16) unsigned char sg_smem[];
    SortShared<ITEMS>& sh = *reinterpret_cast<SortShared<ITEMS>*>(sg_smem);
    cg::grid_group grid = cg::this_grid();
    constexpr int LOT = SG_THREADS * ITEMS;
    const int tid = threadIdx.x, lane = tid & 31, wib = tid >> 5;
    const int G = (int)gridDim.x, blk = (int)blockIdx.x, N = A.N;
    const i64 c0 = (i64)blk * A.chunk;
    const int p_begin = (int)min(c0, (i64)N), p_end = (int)min(c0 + A.chunk, (i64)N);
    const unsigned lt = (1u << lane) - 1u;
    int cur = 0;                                                // the order so far: val[cur], with its keys in key[cur]

    // digit counts of this block's chunk; `items` gives the keys of SG_BATCH places, SG_THREADS apart
    auto count_digits = [&](int shift, auto items) {
        for (int d = tid; d < SG_BINS; d += SG_THREADS) sh.tot[d] = 0;
        __syncthreads();
        for (int p = p_begin + tid; p < p_end; p += SG_THREADS * SG_BATCH) {
            uint32_t k[SG_BATCH];
            items(p, k);
#pragma unroll
            for (int u = 0; u < SG_BATCH; ++u)
                if (p + u * SG_THREADS < p_end) atomicAdd(&sh.tot[(k[u] >> shift) & (SG_BINS - 1)], 1);
        }
        __syncthreads();
        for (int d = tid; d < SG_BINS; d += SG_THREADS) A.table[(i64)d * G + blk] = sh.tot[d];
    };
    auto stored_keys = [&](int p, uint32_t (&k)[SG_BATCH]) {
#pragma unroll
        for (int u = 0; u < SG_BATCH; ++u) k[u] = p + u * SG_THREADS < p_end ? A.key[cur][p + u * SG_THREADS] : 0u;
    };
    // the counted pass: key / val [cur] to [cur ^ 1]
    auto scatter = [&](int shift) {
        grid.sync();
        for (int d = wib * G + blk; d < SG_BINS; d += G * SG_WARPS) {
            int* const row = A.table + (i64)d * G;
            int run = 0;
            for (int k0 = 0; k0 < G; k0 += 32 * 10) {
                int v[10];
#pragma unroll
                for (int u = 0; u < 10; ++u) { const int k = k0 + u * 32 + lane; v[u] = k < G ? row[k] : 0; }
#pragma unroll
                for (int u = 0; u < 10; ++u) {
                    const int k = k0 + u * 32 + lane;
                    int inc = v[u];
#pragma unroll
                    for (int o = 1; o < 32; o <<= 1) {
                        const int y = __shfl_up_sync(0xffffffffu, inc, o);
                        if (lane >= o) inc += y;
                    }
                    if (k < G) row[k] = run + inc - v[u];
                    run += __shfl_sync(0xffffffffu, inc, 31);
                    if (k0 + (u + 1) * 32 >= G) break;
                }
            }
            if (lane == 0) A.total[d] = run;
        }
        grid.sync();
        {
            int all;
            const int t = tid < SG_BINS ? A.total[tid] : 0;
            const int before = sg_block_scan(t, sh.wsum, tid, all);
            if (tid < SG_BINS) sh.base[tid] = before + A.table[(i64)tid * G + blk];
        }
        const uint32_t* const ki = A.key[cur];
        const uint32_t* const vi = A.val[cur];
        uint32_t* const ko = A.key[cur ^ 1];
        uint32_t* const vo = A.val[cur ^ 1];
        // lots of about the same size, every warp the same share of a lot: `per` items per thread, consecutive for the warp
        const int lots = (p_end - p_begin + LOT - 1) / LOT;
        const int per = lots > 0 ? ((p_end - p_begin + lots - 1) / lots + SG_THREADS - 1) / SG_THREADS : 1;
        for (int lot = p_begin; lot < p_end; lot += per * SG_THREADS) {
            const int m = min(per * SG_THREADS, p_end - lot);
            uint32_t key[ITEMS], val[ITEMS];
            const int q0 = wib * 32 * per + lane, q1 = min(m, (wib + 1) * 32 * per);
#pragma unroll
            for (int u = 0; u < ITEMS; ++u) {
                const int q = q0 + u * 32;
                key[u] = q < q1 ? ki[lot + q] : 0u;
                val[u] = q < q1 ? vi[lot + q] : 0u;
            }
            for (int d = lane; d < SG_BINS; d += 32) sh.cnt[wib][d] = 0;
            __syncwarp();
            int at[ITEMS];
#pragma unroll
            for (int u = 0; u < ITEMS; ++u) {
                const bool in = q0 + u * 32 < q1;
                unsigned peers = __ballot_sync(0xffffffffu, in);
                at[u] = 0;
                if (!peers) continue;
                const int digit = (int)((key[u] >> shift) & (SG_BINS - 1));
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    const unsigned b = __ballot_sync(0xffffffffu, (digit >> k) & 1);
                    peers &= ((digit >> k) & 1) ? b : ~b;
                }
                int base = 0;
                if (in) base = sh.cnt[wib][digit];
                __syncwarp();
                if (in && (peers & lt) == 0u) sh.cnt[wib][digit] = base + __popc(peers);
                __syncwarp();
                at[u] = base + __popc(peers & lt);
            }
            __syncthreads();
            int mine = 0;
            if (tid < SG_BINS) {
#pragma unroll
                for (int w = 0; w < SG_WARPS; ++w) { const int c = sh.cnt[w][tid]; sh.cnt[w][tid] = mine; mine += c; }
                sh.tot[tid] = mine;
            }
            int all;
            const int before = sg_block_scan(mine, sh.wsum, tid, all);
            if (tid < SG_BINS) sh.start[tid] = before;
            __syncthreads();
#pragma unroll
            for (int u = 0; u < ITEMS; ++u)
                if (q0 + u * 32 < q1) {
                    const int digit = (int)((key[u] >> shift) & (SG_BINS - 1));
                    const int q = sh.start[digit] + sh.cnt[wib][digit] + at[u];
                    sh.key[q] = key[u]; sh.val[q] = val[u];
                }
            __syncthreads();
            for (int q = tid; q < m; q += SG_THREADS) {
                const uint32_t k = sh.key[q];
                const int digit = (int)((k >> shift) & (SG_BINS - 1));
                const int dst = sh.base[digit] + q - sh.start[digit];
                ko[dst] = k; vo[dst] = sh.val[q];
            }
            __syncthreads();
            if (tid < SG_BINS) sh.base[tid] += sh.tot[tid];
            __syncthreads();
        }
        cur ^= 1;
        grid.sync();
    };
    // ranks (from 0) of the order, a new one where the key or what `second` makes of the value differs from the place before;
    // returns their number
    auto rerank = [&](auto second) -> int {
        const uint32_t* const k = A.key[cur];
        const uint32_t* const v = A.val[cur];
        int mine = 0;
        for (int w0 = p_begin / 32 + wib * SG_BATCH; w0 * 32 < p_end; w0 += SG_WARPS * SG_BATCH) {   // (chunks are multiples of 32)
            uint32_t kk[SG_BATCH], pk;
            int sv[SG_BATCH], ps;
#pragma unroll
            for (int u = 0; u < SG_BATCH; ++u) {
                const int p = (w0 + u) * 32 + lane;
                kk[u] = p < p_end ? k[p] : 0u;
                sv[u] = p < p_end ? (int)v[p] : 0;
            }
            pk = w0 > 0 ? k[w0 * 32 - 1] : 0u;
            ps = w0 > 0 ? (int)v[w0 * 32 - 1] : 0;
            second(kk, sv, pk, ps);
#pragma unroll
            for (int u = 0; u < SG_BATCH; ++u) {
                const int p = (w0 + u) * 32 + lane;
                uint32_t bk = __shfl_up_sync(0xffffffffu, kk[u], 1);
                int bs = __shfl_up_sync(0xffffffffu, sv[u], 1);
                if (lane == 0) { bk = pk; bs = ps; }
                pk = __shfl_sync(0xffffffffu, kk[u], 31); ps = __shfl_sync(0xffffffffu, sv[u], 31);
                const unsigned f = __ballot_sync(0xffffffffu, p < p_end && (p == 0 || kk[u] != bk || sv[u] != bs));
                // (goes on behind the first half and behind the second; the first round has no second half)
                const unsigned go = __ballot_sync(0xffffffffu, (kk[u] & 1u) != 0u && sv[u] != -1 && (sv[u] & 1) != 0);
                if (lane == 0 && (w0 + u) * 32 < p_end) { A.flags[w0 + u] = f; A.go[w0 + u] = go; mine += __popc(f); }
            }
        }
        int all;
        sg_block_scan(mine, sh.wsum, tid, all);
        if (tid == 0) A.count[blk] = all;
        grid.sync();                                            // (all old ranks have been read)
        int before = 0, ranks = 0;
        for (int b = tid; b < G; b += SG_THREADS) { const int c = A.count[b]; ranks += c; if (b < blk) before += c; }
        {
            int x;
            sg_block_scan(before, sh.wsum, tid, x);
            before = x;
            sg_block_scan(ranks, sh.wsum, tid, x);
            ranks = x;
        }
        // a thread per 32 places counts, then the warps assign
        for (int w0 = p_begin / 32; w0 * 32 < p_end; w0 += SG_THREADS) {
            const int w = w0 + tid;
            const int c = w * 32 < p_end ? __popc(A.flags[w]) : 0;
            int n_lot;
            const int off = before + sg_block_scan(c, sh.wsum, tid, n_lot);
            for (int q0 = 0; q0 < 32; q0 += SG_BATCH) {
                if ((w0 + wib * 32 + q0) * 32 >= p_end) break;
                uint32_t x[SG_BATCH];
                unsigned f[SG_BATCH], go[SG_BATCH];
#pragma unroll
                for (int u = 0; u < SG_BATCH; ++u) {
                    const int ww = w0 + wib * 32 + q0 + u, p = ww * 32 + lane;
                    x[u] = p < p_end ? v[p] : 0u;
                    f[u] = ww * 32 < p_end ? A.flags[ww] : 0u;
                    go[u] = ww * 32 < p_end ? A.go[ww] : 0u;
                }
#pragma unroll
                for (int u = 0; u < SG_BATCH; ++u) {
                    const int p = (w0 + wib * 32 + q0 + u) * 32 + lane;
                    const int o = __shfl_sync(0xffffffffu, off, q0 + u);
                    if (p < p_end) A.rank[x[u]] = (int)((unsigned)(o + __popc(f[u] & (lt | (1u << lane))) - 1) * 2u + ((go[u] >> lane) & 1u));
                }
            }
            before += n_lot;
        }
        grid.sync();
        return ranks;
    };

    // ---- by the first token, and whether it is the last one
    for (int p = p_begin + tid; p < p_end; p += SG_THREADS) {
        A.key[0][p] = ((uint32_t)A.tok[p] << 1) | (p + 1 < A.end_pos[p] ? 1u : 0u);
        A.val[0][p] = (uint32_t)p;
    }
    __syncthreads();
    for (unsigned shift = 0; shift < A.key_bits; shift += 8) {
        count_digits((int)shift, stored_keys);
        scatter((int)shift);
    }
    for (int k = 1, off; k < A.D; k += off) {
        off = min(k, A.D - k);
        const int o = k >> 1;                                   // (every round but the last doubles)
        const int ranks = k == 1 ? rerank([&](const uint32_t (&)[SG_BATCH], int (&x)[SG_BATCH], uint32_t, int& y) {
#pragma unroll
            for (int u = 0; u < SG_BATCH; ++u) x[u] = 1;
            y = 1;
        }) : rerank([&](const uint32_t (&kk)[SG_BATCH], int (&x)[SG_BATCH], uint32_t pk, int& y) {
#pragma unroll
            for (int u = 0; u < SG_BATCH; ++u) x[u] = (kk[u] & 1u) ? A.rank[x[u] + o] : -1;
            y = (pk & 1u) ? A.rank[y + o] : -1;
        });
        if (ranks == N) break;                                  // no two alike: the order is final
        // the order by what follows `off` places on, then by rank
        {
            const uint32_t* const from = A.val[cur];
            uint32_t* const ko = A.key[cur ^ 1];
            uint32_t* const vo = A.val[cur ^ 1];
            count_digits(1, [&](int p, uint32_t (&k)[SG_BATCH]) {
                int t[SG_BATCH];
                bool in[SG_BATCH], edge = false;
#pragma unroll
                for (int u = 0; u < SG_BATCH; ++u) {
                    in[u] = p + u * SG_THREADS < p_end;
                    t[u] = in[u] ? (int)from[p + u * SG_THREADS] : off;
                }
#pragma unroll
                for (int u = 0; u < SG_BATCH; ++u) k[u] = t[u] >= off ? (uint32_t)A.rank[t[u] - off] : 0u;
#pragma unroll
                for (int u = 0; u < SG_BATCH; ++u) edge |= in[u] && (k[u] & 1u) == 0u;
                if (edge) {
#pragma unroll 1
                    for (int u = 0; u < SG_BATCH; ++u) {
                        if (!in[u] || (k[u] & 1u)) continue;
                        // the sequence of the suffix `off` places back ends within its k tokens, if it is the same sequence at all
                        const int e = A.end_pos[t[u]];
                        if (t[u] >= off && A.end_pos[t[u] - off] == e) continue;
                        // one of its sequence's first `off`: it stands for one of the last, which have nothing `off` places on
                        int lo = 0, hi = A.n_seqs;              // largest q with seq_off[q] <= t
                        while (hi - lo > 1) { const int mid = (lo + hi) >> 1; if (A.seq_off[mid] <= t[u]) lo = mid; else hi = mid; }
                        const int b = (int)A.seq_off[lo];
                        t[u] = e - min(off, e - b) + (t[u] - b) + off;
                        k[u] = (uint32_t)A.rank[t[u] - off];
                    }
                }
#pragma unroll
                for (int u = 0; u < SG_BATCH; ++u)
                    if (in[u]) { ko[p + u * SG_THREADS] = k[u]; vo[p + u * SG_THREADS] = (uint32_t)(t[u] - off); }
            });
            cur ^= 1;
        }
        scatter(1);                                             // (the lowest bit is the same for equal ranks)
        for (int shift = 8; shift < 32 && ((unsigned)(ranks - 1) >> shift) != 0u; shift += 8) {
            count_digits(shift + 1, stored_keys);
            scatter(shift + 1);
        }
    }
    for (int p = p_begin + tid; p < p_end; p += SG_THREADS) A.sa[p] = A.val[cur][p];
}

template <int ITEMS>
int corpus_sort(CorpusSort& A, cudaStream_t st) {
    void* args[] = {&A};
    const int G = (A.N + A.chunk - 1) / A.chunk;
    SD_CUDA_OK(cudaFuncSetAttribute(corpus_sort_kernel<ITEMS>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(SortShared<ITEMS>)));
    SD_CUDA_OK(cudaLaunchCooperativeKernel((void*)corpus_sort_kernel<ITEMS>, dim3((unsigned)G), dim3(SG_THREADS), args,
                                           sizeof(SortShared<ITEMS>), st));
    return SD_OK;
}

// Suffix order of sequences that are sorted one by one (the trees of different requests share
// nothing, so no suffix of one request is ever compared with a suffix of another): one block per sequence.
template <int THREADS, int ITEMS>
__global__ void __launch_bounds__(THREADS, THREADS == BS_THREADS && ITEMS > 4 ? 1 : 2)
block_suffix_sort_kernel(const int32_t* tok, const int64_t* seq_off, int V, int tok_bits, int D, uint32_t* sa_out) {
    sd_chain_begin();
    extern __shared__ __align__(16) unsigned char bs_smem[];
    __shared__ int wsum[THREADS / 32];
    const i64 b = seq_off[blockIdx.x];
    const int n = (int)(seq_off[blockIdx.x + 1] - b), first_tok = (int)blockIdx.x * V;
    if (n <= 0) return;
    const int32_t* const t = tok + b;
    const unsigned short* const order = block_suffix_order<THREADS, ITEMS>(
        bs_smem, wsum, n, tok_bits, D, [&](int i) { return t[i] - first_tok; }, [](int) { return 0; }, [&](int) { return n; });
    for (int p = threadIdx.x; p < n; p += THREADS) sa_out[b + p] = (uint32_t)(b + order[p]);
}

template <int THREADS, int ITEMS>
int block_suffix_sort(const int32_t* tok, const int64_t* seq_off, int n_seqs, int V, int tok_bits, int D, uint32_t* sa, cudaStream_t st) {
    constexpr int smem = block_order_smem<THREADS, ITEMS>();
    if (smem > 48 * 1024)
        SD_CUDA_OK(cudaFuncSetAttribute(block_suffix_sort_kernel<THREADS, ITEMS>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    SD_CUDA_OK(sd_launch(block_suffix_sort_kernel<THREADS, ITEMS>, (unsigned)n_seqs, THREADS, smem, st, tok, seq_off, V, tok_bits, D, sa));
    return SD_OK;
}

// The same by clusters of blocks: one for a small corpus, or one per prompt.
constexpr int CC_THREADS = 512, CP_THREADS = 256;                // a corpus of 32,768 tokens 108 us (1,024 threads 113, 256 116), four prompts of 4,096 44 (56, 512 47)
template <int ITEMS>
__global__ void __launch_bounds__(CC_THREADS, 1)
cluster_corpus_sort_kernel(const int32_t* tok, const int* end_pos, int n, int tok_bits, int D, uint32_t* sa_out) {
    sd_chain_begin();
    extern __shared__ __align__(16) unsigned char cs_smem[];
    ClusterOrder<CC_THREADS, ITEMS>& sh = *reinterpret_cast<ClusterOrder<CC_THREADS, ITEMS>*>(cs_smem);
    const u64* const order = cluster_suffix_order<CC_THREADS, ITEMS>(
        sh, n, tok_bits, D, [&](int i) { return tok[i]; }, [&](int i) { return i + 1 < end_pos[i]; },
        [&](int i, int off) {
            const int e = end_pos[i];
            if (i >= off && end_pos[i - off] == e) return i - off;
            int lo = max(i - off, -1), hi = i;                  // the sequence begins behind lo, at hi at the latest
            while (hi - lo > 1) { const int mid = (lo + hi) >> 1; if (end_pos[mid] == e) hi = mid; else lo = mid; }
            return e - min(off, e - hi) + (i - hi);
        });
    const int first = (int)cluster_rank() * CC_THREADS * ITEMS;
    for (int k = threadIdx.x; k < CC_THREADS * ITEMS && first + k < n; k += CC_THREADS) sa_out[first + k] = (uint32_t)order[k];
}

// What clusters that have no prompt to sort do meanwhile, on multiprocessors that would be idle: a block per request, they walk to
// global match nodes, which the request's next draft goes on from as from a draft before.  First the new requests' (the last tokens of a
// prompt are known, the tree is there), then those of the other slots that an insert into the global tree has made
// stale, in records of their own (MatchRecord): otherwise every one of them walks all the way in its next draft (256 requests as a
// service: drafts behind an insert 51 us, now 43, of which 1 to take the record; the sort beside it 43 -> 47).
constexpr int MOST_REFRESHED = 1024;
// Whether this call of sd_build_requests has been refused for a token outside the vocabulary (in GlobalState, which keeps the last such
// call: nothing has to be cleared).
struct BadCall {
    int32_t* last;
    int32_t call;
    __device__ bool operator()() const { return *last == call; }
};
struct RequestWalk {
    sd_store sv;
    int n, refreshed;                             // new requests; slots that are looked at (0: there has been no insert)
    const int32_t* slot;
    const int64_t* off;
    const int32_t* tok;                           // as they came
    BadCall bad;
};

__device__ __forceinline__ void request_walk(const RequestWalk& R, int q) {
    __shared__ int tail[SD_MAX_DEPTH];                           // the last tokens
    __shared__ int sh_epoch, sh_len;
    const int tid = threadIdx.x, lane = tid & 31, d = tid / APP_LANES + 1, D = R.sv.D;
    const bool fresh = q < R.n;
    const int slot = fresh ? R.slot[q] : q - R.n;
    if (R.bad() || slot < 0 || slot >= R.sv.R) return;
    SlotState* const ss = R.sv.s_state + slot;
    MatchRecord* const rec = &ss->record;
    // An insert may be at work on the tree on another stream (the call itself has nothing to do with that tree): whoever has seen the epoch
    // of its end sees all that it wrote, and what is found before that carries an epoch that is over by then.
    bool leave = false;
    if (tid == 0) {
        sh_epoch = sd_acquire(&R.sv.g_state->epoch);
        sh_len = fresh ? (int)(R.off[q + 1] - R.off[q]) : sd_relaxed(&ss->len);
        leave = !fresh && (sh_len <= 0 || sh_len > R.sv.T || (sd_relaxed(&ss->status) & (SD_STATUS_POOL_FULL | SD_STATUS_BAD_TOKEN)) ||
                           (sd_relaxed(&ss->g_gen) == sd_relaxed(&ss->gen) && sd_relaxed(&ss->g_epoch) == sh_epoch && sd_relaxed(&ss->g_len) <= sh_len));
    }
    if (!fresh)
        for (int j = tid; j < R.n; j += CP_THREADS) leave |= R.slot[j] == slot;     // (it is another request's from now on)
    if (__syncthreads_or(leave)) return;
    const int epoch = sh_epoch, len = sh_len;
    const int32_t* const end = fresh ? R.tok + R.off[q] + len : R.sv.s_text + (i64)slot * R.sv.T + len;
    if (tid < SD_MAX_DEPTH) {
        tail[tid] = tid < len ? sd_relaxed(&end[-1 - tid]) : -1;
        leave = tid < len && (tail[tid] < 0 || tail[tid] >= R.sv.V);
    }
    if (__syncthreads_or(leave)) return;
    int node = -1;
    int2 zw = make_int2(0, 0);
    if (d <= len && d <= D) {
        node = R.sv.g_root[tail[d - 1]];
        if (node >= (int)R.sv.g_cap) node = -1;
        if (node >= 0) zw = *reinterpret_cast<const int2*>(&R.sv.g_ent[node].z);
    }
    group_walk<true>(R.sv.g_ent, (int)R.sv.g_cap, node, zw, d - 1, lane, [&](int k) { return tail[d - 2 - k]; });
    if (fresh) {
        if ((lane & (APP_LANES - 1)) == 0) ss->g_node[d - 1] = node;
        // (a new request's are no good for the one that still has the slot: requests_prepare_kernel makes them the new one's)
        if (tid == 0) { ss->g_gen = ss->gen - 1; ss->g_epoch = epoch; ss->g_len = len; ss->g_depths = D; }
        return;
    }
    if (tid == 0) { rec->version |= 1; sd_fence(); }
    __syncthreads();
    if ((lane & (APP_LANES - 1)) == 0) rec->node[d - 1] = node;
    if (tid < SD_MAX_DEPTH) rec->tail[tid] = tail[tid];
    if (tid == 0) { rec->epoch = epoch; rec->len = len; }
    __syncthreads();
    if (tid == 0) sd_release(&rec->version, rec->version + 1);
}

template <int ITEMS>
__global__ void __launch_bounds__(CP_THREADS, 1)
cluster_prompt_sort_kernel(const int32_t* tok, const int64_t* seq_off, int n_seqs, int V, int tok_bits, int D, uint32_t* sa_out, RequestWalk walk) {
    sd_chain_begin();
    extern __shared__ __align__(16) unsigned char cs_smem[];
    const int c = (int)(blockIdx.x / cluster_blocks());
    if (c >= n_seqs) {                                           // (whole clusters)
        const int q = (int)blockIdx.x - n_seqs * (int)cluster_blocks();
        if (q < n_seqs + walk.refreshed) request_walk(walk, q);
        return;
    }
    const i64 b = seq_off[c];
    const int n = (int)(seq_off[c + 1] - b), first_tok = c * V;
    if (n <= 0) return;
    const int32_t* const t = tok + b;
    const u64* const order = cluster_suffix_order<CP_THREADS, ITEMS>(
        *reinterpret_cast<ClusterOrder<CP_THREADS, ITEMS>*>(cs_smem), n, tok_bits, D, [&](int i) { return t[i] - first_tok; }, [&](int i) { return i + 1 < n; },
        [&](int i, int off) { return i >= off ? i - off : n - min(off, n) + i; });
    const int first = (int)cluster_rank() * CP_THREADS * ITEMS;
    for (int k = threadIdx.x; k < CP_THREADS * ITEMS && first + k < n; k += CP_THREADS) sa_out[b + first + k] = (uint32_t)b + (uint32_t)order[k];
}

template <class Kernel>
int allow_clusters(Kernel kernel, size_t smem, unsigned blocks) {
    SD_CUDA_OK(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    if (blocks > 8) SD_CUDA_OK(cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
    return SD_OK;
}

// f(std::integral_constant<int, ITEMS>) for the least of 1, 2, 4 .. MOST items that is enough
constexpr int CP_ITEMS = 16, CC_ITEMS = 8;        // the most
template <int MOST, class F>
int with_items(i64 per_thread, F f) {
    if (per_thread <= 1) return f(std::integral_constant<int, 1>());
    if (per_thread <= 2) return f(std::integral_constant<int, 2>());
    if (per_thread <= 4) return f(std::integral_constant<int, 4>());
    if (MOST == 8 || per_thread <= 8) return f(std::integral_constant<int, 8>());
    return f(std::integral_constant<int, MOST>());
}

unsigned cluster_for(i64 n, unsigned most, int threads) {        // blocks of a cluster for n tokens
    unsigned blocks = 2;
    while (blocks < most && (i64)blocks * threads < n) blocks *= 2;
    return blocks;
}

int cluster_corpus_sort(const int32_t* tok, const int* end_pos, int n, int tok_bits, int D, unsigned most, uint32_t* sa, cudaStream_t st) {
    const unsigned blocks = cluster_for(n, most, CC_THREADS);
    return with_items<CC_ITEMS>((n + (i64)blocks * CC_THREADS - 1) / (blocks * CC_THREADS), [&](auto items) -> int {
        constexpr int I = decltype(items)::value;
        const int rc = allow_clusters(cluster_corpus_sort_kernel<I>, sizeof(ClusterOrder<CC_THREADS, I>), blocks);
        if (rc != SD_OK) return rc;
        SD_CUDA_OK(sd_launch_clusters(cluster_corpus_sort_kernel<I>, blocks, blocks, CC_THREADS, sizeof(ClusterOrder<CC_THREADS, I>), st, tok, end_pos, n,
                                      tok_bits, D, sa));
        return SD_OK;
    });
}

int cluster_prompt_sort(const int32_t* tok, const int64_t* seq_off, int n_seqs, i64 max_len, int V, int tok_bits, int D, unsigned blocks,
                        uint32_t* sa, const RequestWalk& walk, cudaStream_t st) {
    const unsigned walks = (unsigned)n_seqs + (unsigned)walk.refreshed;
    const unsigned grid = ((unsigned)n_seqs + (walks + blocks - 1) / blocks) * blocks;
    return with_items<CP_ITEMS>((max_len + (i64)blocks * CP_THREADS - 1) / (blocks * CP_THREADS), [&](auto items) -> int {
        constexpr int I = decltype(items)::value;
        const int rc = allow_clusters(cluster_prompt_sort_kernel<I>, sizeof(ClusterOrder<CP_THREADS, I>), blocks);
        if (rc != SD_OK) return rc;
        SD_CUDA_OK(sd_launch_clusters(cluster_prompt_sort_kernel<I>, grid, blocks, CP_THREADS, sizeof(ClusterOrder<CP_THREADS, I>), st, tok, seq_off, n_seqs, V,
                                      tok_bits, D, sa, walk));
        return SD_OK;
    });
}

// The largest cluster of a device that the sorts can have: 16 blocks where its partitions hold as many, else 8, which is sure.
unsigned largest_cluster(int dev) {
    constexpr int MAX_DEVICES = 64;
    static std::atomic<unsigned> known[MAX_DEVICES];
    if (dev < 0 || dev >= MAX_DEVICES || sd_small_clusters()) return 8;
    unsigned c = known[dev].load();
    if (c == 0) {
        c = 8;
        constexpr size_t smem = sizeof(ClusterOrder<CC_THREADS, CC_ITEMS>);
        if (allow_clusters(cluster_corpus_sort_kernel<CC_ITEMS>, smem, CS_MOST) == SD_OK) {
            cudaLaunchAttribute attr;
            attr.id = cudaLaunchAttributeClusterDimension;
            attr.val.clusterDim.x = CS_MOST; attr.val.clusterDim.y = 1; attr.val.clusterDim.z = 1;
            cudaLaunchConfig_t cfg = {};
            cfg.gridDim = dim3(CS_MOST); cfg.blockDim = dim3(CC_THREADS); cfg.dynamicSmemBytes = smem;
            cfg.attrs = &attr; cfg.numAttrs = 1;
            int n = 0;
            if (cudaOccupancyMaxActiveClusters(&n, cluster_corpus_sort_kernel<CC_ITEMS>, &cfg) == cudaSuccess && n > 0) c = CS_MOST;
        }
        cudaGetLastError();
        known[dev].store(c);
    }
    return c;
}

// ------------------------------------------------------------------ all depths at once
// Everything the tree needs beyond the suffix order follows from lcp[] (common prefix of a suffix with the one
// before it) and len[], both capped at D.  Suffix j opens a node at every depth d in (lcp[j], len[j]].  A
// warp goes through a tile of suffixes with a lane per depth:
//   end_d(j)   = min{ i > j : lcp[i] < d }, else N      one past the node's range: count = end - j
//   F_d(j)     = #{ i in (j, end_d(j)) : lcp[i] == d < len[i] }  children that later suffixes open below it
//   children   = F_d(j) + 1 if d < len[j]
//   G_d(j)     = sum of F_a(j) over 1 <= a < d
// The nodes are numbered in depth-first pre-order and child runs are laid down in node order, so the run of a
// node's first child directly follows the node's own run and a chain of only children is a run of consecutive
// entries.  What lies in front of a node's run are the nodes (below depth 1) that earlier suffixes opened, those
// that j itself opened down to depth d, and the children that later suffixes will open below the node's ancestors:
//   run(j, d)  = S(j) + (d - max(lcp[j], 1)) + G_d(j),  S(j) = nodes below depth 1 opened by suffixes before j
// so a node's run needs no table of all nodes, only running state per depth:
//   from behind  (F, end): at suffix i, F_d + 1 if lcp[i] == d < len[i], both reset if lcp[i] < d.  In terms of G: G_d
//                becomes G_{lcp+1} (+ 1 if the suffix opens a node) for all d > lcp (0 if lcp is 0): one shuffle; F_d = G_{d+1} - G_d
//   from the front  R_d: the end of the run of the last node opened at depth d.  The first node that suffix j opens has
//                F_lcp(j) siblings behind it: its entry is R_lcp - 1 - F_lcp(j); every further one is its parent's
//                first child.
// Three sweeps over the suffixes: (1) lcp and what a tile does to the state from behind, (2) the R a tile leaves behind,
// (3) the entries; between them the state is carried over the tiles, a block per depth.  Per suffix that reads a row of D
// tokens twice and writes 16 B per node.  (A table of ranks per depth and suffix, and per node its range, children and
// run, written and read back by six kernels, took 2.5 ms for 4.2 M suffixes of 48.6 M nodes.)
constexpr int TS_SUB = 16;                        // suffixes whose state from behind is kept in registers
constexpr int TS_WARPS = 4;                       // tiles (warps) per block
constexpr int TS_TILES = 8192;                    // tiles are made longer to have no more of them than that, as far as
constexpr int TS_MAX_LEN = 1024;                  // the shared memory for their state goes
constexpr int TS_CARRY = 256;                     // threads per block of the carry kernels
constexpr unsigned TS_FULL = 0xffffffffu;

struct TreeScan {
    const int32_t* tok;
    const uint32_t* sa;
    const int* end_pos;
    uint8_t *lcp, *len;
    int N, D;
    int tile_len, tiles;                          // TS_SUB times a power of two
    int* f;                                       // [32][tiles] (1): children counted, bit 31: state reset; carried: F from behind
    int* e;                                       // [32][tiles] (1): first reset in the tile; carried: end from behind
    int* r;                                       // [32][tiles] (2): R left behind (-1: none); carried: R from the front
    int* s;                                       // [tiles + 1] nodes below depth 1, carried: S
    int* n1;                                      // [tiles + 1] nodes of depth 1, carried: before the tile
    TreeTotals* total;                            // in 64 bits: places are right only if these fit 32, nothing is written before the host knows
};

__device__ __forceinline__ int ts_scan(int v, int lane) {       // inclusive
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(TS_FULL, v, o);
        if (lane >= o) v += y;
    }
    return v;
}

// (1) LONG: tiles of many suffixes.
template <bool LONG>
__global__ void __launch_bounds__(TS_WARPS * 32)
ts_tiles_kernel(TreeScan T) {
    sd_chain_begin();
    const int lane = threadIdx.x & 31, tile = blockIdx.x * TS_WARPS + (threadIdx.x >> 5), d = lane + 1;
    if (tile >= T.tiles) return;
    const int t0 = tile * T.tile_len, t1 = min(T.N, t0 + T.tile_len);
    int px = -1, pl = 0;                                        // the row before: its tokens, its length
    if (t0 > 0) {
        const int q = (int)T.sa[t0 - 1];
        pl = min(T.D, T.end_pos[q] - q);
        if (lane < pl) px = T.tok[q + lane];
    }
    bool seen = false;
    int cnt = 0, first = T.N, below = 0, top = 0, least = 32;
    for (int jb = t0; jb < t1; jb += 32) {
        const int m = min(32, t1 - jb);
        int q = 0, ln = 0, own = 0;
        if (lane < m) { q = (int)T.sa[jb + lane]; ln = min(T.D, T.end_pos[q] - q); }
        for (int i0 = 0; i0 < m; i0 += 8) {
            int x[8], L[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) {                       // eight rows in flight
                const int at = __shfl_sync(TS_FULL, q, i0 + u);
                L[u] = __shfl_sync(TS_FULL, ln, i0 + u);
                x[u] = lane < L[u] ? T.tok[at + lane] : -1;
            }
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                if (i0 + u >= m) break;
                const unsigned ne = __ballot_sync(TS_FULL, x[u] != px || lane >= L[u] || lane >= pl);
                const int l = ne ? __ffs(ne) - 1 : 32;
                if (lane == i0 + u) own = l;
                if (!LONG || l <= least) {                               // (else it does nothing to a depth without a reset)
                    least = l;
                    if (!seen) {
                        cnt += l == d && L[u] > l ? 1 : 0;
                        if (l < d) { seen = true; first = jb + i0 + u; }
                    }
                }
                px = x[u]; pl = L[u];
            }
        }
        if (lane < m) {
            T.lcp[jb + lane] = (uint8_t)own; T.len[jb + lane] = (uint8_t)ln;
            below += ln - max(own, 1);
            top += own == 0 ? 1 : 0;
        }
    }
    T.f[(i64)lane * T.tiles + tile] = cnt | (seen ? (int)0x80000000 : 0);
    T.e[(i64)lane * T.tiles + tile] = first;
    below = (int)__reduce_add_sync(TS_FULL, (unsigned)below);
    top = (int)__reduce_add_sync(TS_FULL, (unsigned)top);
    if (lane == 0) { T.s[tile] = below; T.n1[tile] = top; }
}

// What lies behind (f, e: the tiles to the right; blocks 0 .. 31) or in front of a tile (s, n1: block 32).
__global__ void __launch_bounds__(TS_CARRY) ts_carry_kernel(TreeScan T) {
    sd_chain_begin();
    __shared__ int p0[TS_CARRY / 32], p1[TS_CARRY / 32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int per = (T.tiles + TS_CARRY - 1) / TS_CARRY;
    const int k0 = threadIdx.x * per, k1 = min(T.tiles, k0 + per);
    if (blockIdx.x == 32) {
        __shared__ i64 sum[TS_CARRY / 32];
        int b = 0;
        i64 a = 0;                                              // (a tile's nodes fit 32 bits, the tree's need not)
        for (int k = k0; k < k1; ++k) { a += T.s[k]; b += T.n1[k]; }
        i64 ia = a;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const i64 y = __shfl_up_sync(TS_FULL, ia, o);
            if (lane >= o) ia += y;
        }
        const int ib = ts_scan(b, lane);
        if (lane == 31) { sum[w] = ia; p1[w] = ib; }
        __syncthreads();
        i64 ra = ia - a, ta = 0;
        int rb = ib - b, tb = 0;
        for (int q = 0; q < TS_CARRY / 32; ++q) { if (q < w) { ra += sum[q]; rb += p1[q]; } ta += sum[q]; tb += p1[q]; }
        for (int k = k0; k < k1; ++k) { const int x = T.s[k]; b = T.n1[k]; T.s[k] = (int)ra; T.n1[k] = rb; ra += x; rb += b; }
        if (threadIdx.x == 0) { T.s[T.tiles] = (int)ta; T.n1[T.tiles] = tb; T.total->below = ta; T.total->top = tb; }
        return;
    }
    int* const f = T.f + (i64)blockIdx.x * T.tiles;
    int* const e = T.e + (i64)blockIdx.x * T.tiles;
    // (tile T.tiles - 1 - k: from the last to the first.)  v: children since the last reset, bit 31: there was one
    auto join = [](int& v, int& x, int nv, int nx) { if (nv < 0) { v = nv; x = nx; } else v += nv; };        // further to the left
    int v = 0, x = T.N;
    for (int k = k0; k < k1; ++k) join(v, x, f[T.tiles - 1 - k], e[T.tiles - 1 - k]);
    int iv = v, ix = x;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        int yv = __shfl_up_sync(TS_FULL, iv, o), yx = __shfl_up_sync(TS_FULL, ix, o);
        if (lane >= o) { join(yv, yx, iv, ix); iv = yv; ix = yx; }
    }
    if (lane == 31) { p0[w] = iv; p1[w] = ix; }
    int bv = __shfl_up_sync(TS_FULL, iv, 1), bx = __shfl_up_sync(TS_FULL, ix, 1);      // of the lanes before
    __syncthreads();
    int rv = 0, rx = T.N;
    for (int q = 0; q < w; ++q) join(rv, rx, p0[q], p1[q]);
    if (lane > 0) join(rv, rx, bv, bx);
    for (int k = k0; k < k1; ++k) {
        const int t = T.tiles - 1 - k;
        const int fv = f[t], fx = e[t];
        f[t] = rv & 0x7fffffff; e[t] = rx;
        join(rv, rx, fv, fx);
    }
}

// S and the depth-1 nodes in front of every request's first suffix (the requests' suffixes are consecutive in the
// order); entry n: all of them.
struct RequestBounds {
    int n;                                        // -1: no requests
    const int64_t* off;                           // [n + 1]
    int *s, *n1;                                  // [n + 1]
};

// R from the front: the last one left behind by a tile to the left (blocks 0 .. 31); the others: a request each.
__global__ void __launch_bounds__(TS_CARRY) ts_carry_front_kernel(TreeScan T, RequestBounds Q) {
    sd_chain_begin();
    __shared__ int part[TS_CARRY / 32], part1[TS_CARRY / 32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    if (blockIdx.x >= 32) {
        const int q = blockIdx.x - 32;
        const int j = (int)Q.off[q], tile = j / T.tile_len;
        int a = 0, b = 0;
        for (int i = tile * T.tile_len + threadIdx.x; i < j; i += TS_CARRY) { const int l = T.lcp[i]; a += T.len[i] - max(l, 1); b += l == 0 ? 1 : 0; }
        a = (int)__reduce_add_sync(TS_FULL, (unsigned)a);
        b = (int)__reduce_add_sync(TS_FULL, (unsigned)b);
        if (lane == 0) { part[w] = a; part1[w] = b; }
        __syncthreads();
        if (threadIdx.x == 0) {
            for (int k = 1; k < TS_CARRY / 32; ++k) { a += part[k]; b += part1[k]; }
            Q.s[q] = T.s[tile] + a; Q.n1[q] = T.n1[tile] + b;
        }
        return;
    }
    const int per = (T.tiles + TS_CARRY - 1) / TS_CARRY;
    const int k0 = threadIdx.x * per, k1 = min(T.tiles, k0 + per);
    int* const r = T.r + (i64)blockIdx.x * T.tiles;
    int v = -1;
    for (int k = k0; k < k1; ++k) { const int n = r[k]; if (n >= 0) v = n; }
    int iv = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(TS_FULL, iv, o);
        if (lane >= o && iv < 0) iv = y;
    }
    if (lane == 31) part[w] = iv;
    const int b = __shfl_up_sync(TS_FULL, iv, 1);
    __syncthreads();
    int run = -1;
    for (int q = 0; q < w; ++q) if (part[q] >= 0) run = part[q];
    if (lane > 0 && b >= 0) run = b;
    for (int k = k0; k < k1; ++k) { const int n = r[k]; r[k] = run; if (n >= 0) run = n; }
}

// The state from behind at a tile's right end: G of this lane's depth.
__device__ __forceinline__ int ts_g_in(const TreeScan& T, int tile, int lane) {
    const int f = T.f[(i64)lane * T.tiles + tile];
    return ts_scan(f, lane) - f;
}

// G in front of a suffix with lcp l and length n (uniform)
__device__ __forceinline__ int ts_g_step(int g, int l, int n, int d) {
    const int v = __shfl_sync(TS_FULL, g, min(l, 31)) + (n > l ? 1 : 0);
    return d > l ? (l == 0 ? 0 : v) : g;
}

__device__ __forceinline__ int ts_f_of(int g, int lane) {       // F from G (no node of depth 32 has children)
    const int up = __shfl_down_sync(TS_FULL, g, 1);
    return lane == 31 ? 0 : up - g;
}

// (2) TOP: also counts the long runs.
template <bool TOP>
__global__ void __launch_bounds__(TS_WARPS * 32)
ts_runs_kernel(TreeScan T) {
    sd_chain_begin();
    const int lane = threadIdx.x & 31, tile = blockIdx.x * TS_WARPS + (threadIdx.x >> 5), d = lane + 1;
    if (tile >= T.tiles) return;
    const int t0 = tile * T.tile_len, t1 = min(T.N, t0 + T.tile_len);
    int g = ts_g_in(T, tile, lane);
    int s_end = T.s[tile + 1], R = -1, n_wide = 0;
    unsigned open = TS_FULL;                                    // lanes without R
    i64 room = 0;
    for (int jb = t0 + ((t1 - t0 - 1) & ~31); jb >= t0; jb -= 32) {
        const int m = min(32, t1 - jb);
        int l_own = 0, n_own = 0, c = 0;
        if (lane < m) { l_own = T.lcp[jb + lane]; n_own = T.len[jb + lane]; c = n_own - max(l_own, 1); }
        const int inc = ts_scan(c, lane);
        const int all = __shfl_sync(TS_FULL, inc, 31);
        const int s_own = s_end - all + inc - c;
        s_end -= all;
#pragma unroll 4
        for (int i = m - 1; i >= 0; --i) {
            const int l = __shfl_sync(TS_FULL, l_own, i), n = __shfl_sync(TS_FULL, n_own, i);
            const int gl = __shfl_sync(TS_FULL, g, min(l, 31));
            // (the depths that it opens: lanes l .. n - 1)
            if ((((2u << (n - 1)) - 1u) & ~(l < 32 ? (1u << l) - 1u : TS_FULL)) & open) {
                const int kids = ts_f_of(g, lane) + (d < n ? 1 : 0);
                const int s = __shfl_sync(TS_FULL, s_own, i);
                if (d > l && d <= n && R < 0) R = s + d - max(l, 1) + g + kids;
                open = __ballot_sync(TS_FULL, R < 0);
            }
            // the nodes that it opens have as many children together, but for their own first ones, as G grows from there on
            if (TOP && __shfl_sync(TS_FULL, g, 31) - gl >= SD_TOP_MIN) {
                const int kids = ts_f_of(g, lane) + (d < n ? 1 : 0);
                if (d > l && d <= n && kids > SD_TOP_MIN) { ++n_wide; room += kids + SD_TOP_BLOCK; }
            }
            g = d > l ? (l == 0 ? 0 : gl + (n > l ? 1 : 0)) : g;                    // (ts_g_step)
        }
    }
    T.r[(i64)lane * T.tiles + tile] = R;
    if (TOP) {
        n_wide = (int)__reduce_add_sync(TS_FULL, (unsigned)n_wide);
        if (n_wide) {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) room += __shfl_xor_sync(TS_FULL, room, o);
            if (lane == 0) { atomicAdd(&T.total->n_wide, n_wide); atomicAdd((u64*)&T.total->wide, (u64)room); }
        }
    }
}

// Where the trees go: one tree (the global one), or one per request, whose suffixes are consecutive in the order.
struct TreeOut {
    int4* ent;                                    // global tree
    int32_t* root;
    int4* wide;                                   // its long runs: entry of the node, run, children, -
    sd_store sv;                                  // requests
    int n_req;
    const int32_t* slot;
    const int64_t* off;                           // [n_req + 1]
    const int *s_req, *n1_req;                    // [n_req + 1] S and depth-1 nodes before the request's first suffix
    BadCall bad;                                  // a token is outside the vocabulary, nothing may change
};

// A request's active node of depth d is the node of its suffix of d tokens, which comes first among those that begin with it:
// where that is not all of the tree's depth it is the last node that the suffix opens.
__device__ __forceinline__ void set_active(SlotState* ss, int d, int node, int run, int kids) {
    ss->active[d - 1] = node; ss->room[d - 1] = 0;
    ss->run_cb[d - 1] = kids > 0 ? run : 0; ss->run_w[d - 1] = kids > 0 ? (unsigned)kids | RUN_STATIC : 0u;
}

// What the lanes need of a suffix in one word, so that one shuffle hands it out: lcp and length (at most 32), S and the
// depth-1 nodes relative to the first of up to 32 suffixes (at most 31 * 31, 31).  ts_emit_kernel mostly shuffles: 13 -> 8
// of them per suffix, and the next sub-tile read ahead, 767 -> 569 us for 4.2 M suffixes.  (ts_runs_kernel is bound by
// its arithmetic: taking words apart made it 226 -> 251 us.)
__device__ __forceinline__ int ts_pack(int l, int n, int s, int n1) { return l | n << 6 | s << 12 | n1 << 22; }
__device__ __forceinline__ int ts_l(int w) { return w & 63; }
__device__ __forceinline__ int ts_n(int w) { return (w >> 6) & 63; }
__device__ __forceinline__ int ts_s(int w) { return (w >> 12) & 1023; }
__device__ __forceinline__ int ts_n1(int w) { return w >> 22; }

// (3)
template <bool REQ>
__global__ void __launch_bounds__(TS_WARPS * 32)
ts_emit_kernel(TreeScan T, TreeOut O) {
    sd_chain_begin();
    extern __shared__ int2 ts_state[];                          // [TS_WARPS][tile_len / TS_SUB][32]: G and end behind each sub-tile
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5, tile = blockIdx.x * TS_WARPS + wib, d = lane + 1;
    if (tile >= T.tiles || (REQ && O.bad())) return;
    const int t0 = tile * T.tile_len, t1 = min(T.N, t0 + T.tile_len);
    const int subs = (t1 - t0 + TS_SUB - 1) / TS_SUB;
    int2* const st = ts_state + (i64)wib * (T.tile_len / TS_SUB) * 32;
    {
        int g = ts_g_in(T, tile, lane), e = T.e[(i64)lane * T.tiles + tile];
        for (int c = subs - 1; c >= 0; --c) {
            st[c * 32 + lane] = make_int2(g, e);
            if (c == 0) break;
            const int jb = t0 + c * TS_SUB, m = min(TS_SUB, t1 - jb);
            const int own = lane < m ? ts_pack(T.lcp[jb + lane], T.len[jb + lane], 0, 0) : 0;
#pragma unroll 8
            for (int i = m - 1; i >= 0; --i) {
                const int w = __shfl_sync(TS_FULL, own, i), l = ts_l(w);
                g = ts_g_step(g, l, ts_n(w), d);
                if (d > l) e = jb + i;
            }
        }
        __syncwarp();
    }
    int R = T.r[(i64)lane * T.tiles + tile];
    int s_at = T.s[tile], n1_at = T.n1[tile];
    // the tree this suffix belongs to: entries, root table, what turns S into a place, first token, depth-1 nodes before it
    int4* ent = O.ent;
    int32_t* root = O.root;
    SlotState* ss = nullptr;
    int shift = 0, first_tok = 0, n1_0 = 0, q = 0, next_req = 0x7fffffff;
    bool fits = true;
    auto enter = [&]() {                                        // request q
        const int n1 = O.n1_req[q + 1] - O.n1_req[q], used = n1 + O.s_req[q + 1] - O.s_req[q], slot = O.slot[q];
        fits = used <= O.sv.spn && O.off[q + 1] - O.off[q] <= O.sv.T && slot >= 0 && slot < O.sv.R;
        ent = O.sv.s_ent + (i64)(fits ? slot : 0) * O.sv.spn;
        root = O.sv.s_root + (i64)(fits ? slot : 0) * O.sv.V;
        ss = O.sv.s_state + (fits ? slot : 0);
        shift = n1 - O.s_req[q]; n1_0 = O.n1_req[q]; first_tok = q * O.sv.V;
        next_req = (int)O.off[q + 1];
    };
    if (REQ) {
        int lo = 0, hi = O.n_req;                               // the last request that starts at or before t0
        while (hi - lo > 1) { const int mid = (lo + hi) >> 1; if (O.off[mid] <= t0) lo = mid; else hi = mid; }
        q = lo;
        enter();
    } else {
        shift = T.n1[T.tiles];
    }
    int l_own = 0, n_own = 0, sa_own = 0;                       // of the sub-tile's suffixes, read one sub-tile ahead
    auto fetch = [&](int j) {
        const bool in = lane < TS_SUB && j + lane < t1;
        l_own = in ? T.lcp[j + lane] : 0; n_own = in ? T.len[j + lane] : 0; sa_own = in ? (int)T.sa[j + lane] : 0;
    };
    fetch(t0);
    for (int c = 0; c < subs; ++c) {
        const int jb = t0 + c * TS_SUB, m = min(TS_SUB, t1 - jb);
        const int below = lane < m ? n_own - max(l_own, 1) : 0;
        const unsigned tops = __ballot_sync(TS_FULL, lane < m && l_own == 0);
        const int ib = ts_scan(below, lane);
        const int own = ts_pack(l_own, n_own, ib - below, __popc(tops & ((1u << lane) - 1u))), at_own = sa_own;
        const int s0 = s_at, n1_at0 = n1_at;
        s_at += __shfl_sync(TS_FULL, ib, 31);
        n1_at += __popc(tops);
        int x[TS_SUB], gs[TS_SUB], es[TS_SUB];
        const int2 in = st[c * 32 + lane];
        int g = in.x, e = in.y;
#pragma unroll
        for (int i = TS_SUB - 1; i >= 0; --i) {
            const int w = __shfl_sync(TS_FULL, own, i), at = __shfl_sync(TS_FULL, at_own, i), l = ts_l(w), n = ts_n(w);
            x[i] = lane < n ? T.tok[at + lane] : 0;
            gs[i] = g; es[i] = e;
            if (i < m) {
                g = ts_g_step(g, l, n, d);
                if (d > l) e = jb + i;
            }
        }
        fetch(jb + TS_SUB);
#pragma unroll
        for (int i = 0; i < TS_SUB; ++i) {
            if (i >= m) break;
            const int j = jb + i;
            if (REQ && j >= next_req) { while (j >= (int)O.off[q + 1]) ++q; enter(); }
            const int w = __shfl_sync(TS_FULL, own, i), l = ts_l(w), n = ts_n(w);
            const int run = s0 + ts_s(w) + d - max(l, 1) + gs[i], depth1 = n1_at0 + ts_n1(w) - n1_0;
            const int later = ts_f_of(gs[i], lane);
            const int kids = later + (d < n ? 1 : 0);
            const bool opens = d > l && d <= n;
            // the entry of the next depth's node: this node's first child, or the next of its other children
            const int place = __shfl_up_sync(TS_FULL, opens ? run : R - 1 - later, 1);
            if (opens) R = run + kids;
            if (opens && fits) {
                const int pos = lane == 0 ? depth1 : place + shift;
                // (the suffixes that end with a node come first among its own: the one that opens it is one of them, if there are any)
                const unsigned ends = !REQ && d == n ? RUN_ENDS : 0u;
                ent[pos] = make_int4(x[i] - first_tok, es[i] - j, kids > 0 ? run + shift : 0, kids > 0 ? (int)((unsigned)kids | RUN_STATIC | ends) : 0);
                if (lane == 0) root[x[i] - first_tok] = pos;
                if (REQ && d == n && d < T.D) set_active(ss, d, pos, run + shift, kids);
                if (!REQ && kids > SD_TOP_MIN) O.wide[atomicAdd(&T.total->listed, 1)] = make_int4(pos, run + shift, kids, 0);
            }
        }
    }
}

// Long runs of the global tree move behind the others, with room for a top block in front: first every node of one
// gets its new run (its entry may itself lie in a run that moves), then the runs are copied.
__global__ void ts_wide_place_kernel(TreeScan T, int4* wide, int4* ent, int first) {
    sd_chain_begin();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= T.total->n_wide) return;
    int4 w = wide[i];
    w.w = first + atomicAdd(&T.total->placed, w.z + SD_TOP_BLOCK);
    wide[i] = w;
    ent[w.x].z = w.w + SD_TOP_BLOCK;
    ent[w.x].w |= (int)RUN_HAS_TOP;
}

// One block per long run: the run, and in front of it the sum of its counts and the 64 best children by (count desc, token asc).
// The smallest count among them is found by halving; children that occur more often are fewer than 64 and placed by comparing
// them with one another, those with that very count follow in run (token) order.
constexpr int TOP_THREADS = 256;
__global__ void __launch_bounds__(TOP_THREADS)
ts_wide_fill_kernel(const int4* wide, int4* ent) {
    sd_chain_begin();
    __shared__ int part[TOP_THREADS / 32];
    __shared__ u64 psum[TOP_THREADS / 32];
    __shared__ int cand[64];
    __shared__ u64 ckey[64];
    __shared__ int n_cand, limit;
    const int4 w = wide[blockIdx.x];
    const int n = w.z, tid = threadIdx.x, lane = tid & 31, wib = tid >> 5;
    const int4* const from = ent + w.y;
    int4* const to = ent + w.w + SD_TOP_BLOCK;
    int4* const topb = ent + w.w;
    u64 sum = 0;
    unsigned most = 0;
    for (int i = tid; i < n; i += TOP_THREADS) {
        const int4 e = from[i];
        to[i] = e;
        sum += (unsigned)e.y;
        most = max(most, (unsigned)e.y);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(TS_FULL, sum, o);
    most = __reduce_max_sync(TS_FULL, most);
    if (lane == 0) { psum[wib] = sum; part[wib] = (int)most; }
    if (tid == 0) n_cand = 0;
    __syncthreads();
    const int want = min(n, 64);
    if (tid == 0) {
        for (int k = 1; k < TOP_THREADS / 32; ++k) { sum += psum[k]; most = max(most, (unsigned)part[k]); }
        limit = (int)most;
        topb[0] = make_int4((int)(unsigned)(sum & 0xffffffffu), (int)(unsigned)(sum >> 32), want, 0);
    }
    __syncthreads();
    // the largest count c with at least `want` children at or above it
    int lo = 1, hi = limit;
    while (lo < hi) {
        const int mid = lo + (hi - lo + 1) / 2;
        int k = 0;
        for (int i = tid; i < n; i += TOP_THREADS) k += from[i].y >= mid ? 1 : 0;
        k = (int)__reduce_add_sync(TS_FULL, (unsigned)k);
        __syncthreads();
        if (lane == 0) part[wib] = k;
        __syncthreads();
        k = 0;
        for (int q = 0; q < TOP_THREADS / 32; ++q) k += part[q];
        if (k >= want) lo = mid; else hi = mid - 1;
    }
    for (int i = tid; i < n; i += TOP_THREADS) {
        const int4 e = from[i];
        if (e.y > lo) {
            const int k = atomicAdd(&n_cand, 1);
            cand[k] = i; ckey[k] = ((u64)(unsigned)e.y << 32) | (0xffffffffu - (unsigned)e.x);
        }
    }
    __syncthreads();
    const int nc = n_cand;
    if (tid < nc) {
        int rank = 0;
        for (int q = 0; q < nc; ++q) rank += ckey[q] > ckey[tid] ? 1 : 0;
        topb[1 + rank] = from[cand[tid]];
    }
    if (wib == 0) {
        int k = nc;
        for (int base = 0; base < n && k < want; base += 32) {
            int4 e = make_int4(0, 0, 0, 0);
            if (base + lane < n) e = from[base + lane];
            const unsigned m = __ballot_sync(TS_FULL, e.y == lo);
            const int at = k + __popc(m & ((1u << lane) - 1u));
            if (e.y == lo && at < want) topb[1 + at] = e;
            k += __popc(m);
        }
    }
}

__global__ void init_global_state_kernel(GlobalState* g, int used, int live, long long tokens) {
    g->used = used; g->live = live; g->status = 0; g->epoch = 1; g->tokens = tokens; g->bad_call = 0;
}

struct DeviceArena {          // temporaries of one build: freed together, or kept in a workspace
    void* ptr[48];
    int n = 0;
    sd_workspace* keep = nullptr;                     // if set, buffers live there and are reused
    char* chunk = nullptr;                            // reserved block the next buffers are carved from
    long long chunk_left = 0;
    cudaStream_t st;                                  // the buffers belong to the work on this stream
    explicit DeviceArena(cudaStream_t stream) : st(stream) {}
    ~DeviceArena() {
        if (keep || n == 0) return;
        cudaStreamSynchronize(st);
        for (int i = 0; i < n; ++i) sd_device_free(ptr[i]);
    }
    // One allocation for the buffers to come (an allocation of its own costs far more than the
    // kernels that use a buffer).  If it fails the buffers are simply allocated one by one.
    void reserve(long long bytes) {
        if (keep || n >= 48 || bytes <= 0) return;
        void* p = nullptr;
        if (sd_device_malloc(&p, (size_t)bytes) != cudaSuccess) { cudaGetLastError(); return; }
        ptr[n++] = p;
        chunk = (char*)p; chunk_left = bytes;
    }
    template <class T> bool get(T** out, i64 count) {
        if (count < 1) count = 1;
        const long long need = (long long)count * (long long)sizeof(T);
        const long long padded = (need + 255) / 256 * 256;
        if (!keep && chunk_left >= padded) {
            *out = (T*)chunk;
            chunk += padded; chunk_left -= padded;
            return true;
        }
        if (n >= 48) return false;
        if (keep) {
            const int k = n++;
            if (keep->bytes[k] < need) {
                if (keep->ptr[k]) { cudaStreamSynchronize(st); sd_device_free(keep->ptr[k]); }
                keep->ptr[k] = nullptr; keep->bytes[k] = 0;
                const long long want = need + need / 4 + 256;
                if (sd_device_malloc(&keep->ptr[k], (size_t)want) != cudaSuccess) { cudaGetLastError(); return false; }
                keep->bytes[k] = want;
            }
            *out = (T*)keep->ptr[k];
            return true;
        }
        void* p = nullptr;
        if (sd_device_malloc(&p, (size_t)need) != cudaSuccess) { cudaGetLastError(); return false; }
        ptr[n++] = p;
        *out = (T*)p;
        return true;
    }
};

inline unsigned grid_for(i64 n, int threads) { return (unsigned)((n + threads - 1) / threads); }

int bits_for(i64 maxval) {
    int b = 1;
    while ((1ll << b) <= maxval && b < 32) ++b;
    return b;
}

}  // namespace

// Arguments of sd_build_requests for n requests: offsets, slots, a zero; and the host's flag.
static size_t stage_bytes_for(i64 n) { return (size_t)(8 * (n + 1) + 4 * n + 4 + 16) / 16 * 16 + 16; }

template <class T>
static bool store_alloc(sd_store* s, T** out, long long count) {
    void* p = nullptr;
    if (count < 1) count = 1;
    if (sd_device_malloc(&p, (size_t)count * sizeof(T)) != cudaSuccess) { cudaGetLastError(); return false; }
    s->device_bytes += count * (long long)sizeof(T);
    *out = (T*)p;
    return true;
}

// Everything up to the writing of the entries, for one array of sequences: suffix order and the sweeps over it.
struct Pipeline {
    DeviceArena tmp;
    explicit Pipeline(cudaStream_t st) : tmp(st) {}
    TreeScan ts;
    bool walked = false;                          // the new requests' global match nodes are known
};

// max_token: largest token value + 1 (sets the number of radix passes; below 2^31).  top_blocks: count the
// long runs.  per_seq_max_len > 0: the sequences are independent
// (tokens of different sequences never compare equal, sequence k's tokens below sequence k + 1's)
// and none is longer than that, so each is sorted by a cluster of its own, or a block where there are many or all are short.
// end_pos: one past the last token of every token's sequence, if that is known already.
// Nothing is read back to the host.
// Returns SD_OK, SD_ERR_NOMEM or SD_ERR_CUDA.
static int pipeline_run(Pipeline& P, const int32_t* d_tok, const int64_t* d_seq_offsets, int n_seqs, i64 N,
                        i64 max_token, int D, bool top_blocks, cudaStream_t st, i64 per_seq_max_len = 0,
                        int* end_pos = nullptr, RequestBounds bounds = RequestBounds{-1, nullptr, nullptr, nullptr},
                        const RequestWalk* walk = nullptr) {
    const int T256 = 256;
    DeviceArena& tmp = P.tmp;
    TreeScan& ts = P.ts;
    ts.N = (int)N; ts.D = D; ts.tok = d_tok;
    ts.tile_len = TS_SUB;
    while ((N + ts.tile_len - 1) / ts.tile_len > TS_TILES && ts.tile_len < TS_MAX_LEN) ts.tile_len *= 2;
    ts.tiles = (int)((N + ts.tile_len - 1) / ts.tile_len);
    int sms = 0, dev = 0;
    SD_CUDA_OK(cudaGetDevice(&dev));
    SD_CUDA_OK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    const int most_blocks = 2 * sms;
    // Prompts longer than one step of a block are sorted by a cluster of four or eight blocks each while there are at most 128 blocks then
    // (partitions of 16 multiprocessors and more hold so many at once; with clusters of two, 64 prompts of 8,192 tokens took as long as
    // by a block each, and their decode 1 % longer), else by a block each.  A corpus of up to 65,536 tokens is sorted by a cluster: whole
    // builds of 8,000 / 32,768 / 65,536 tokens 329 / 382 / 430 us by the whole device, 222 / 280 / 385 by a cluster, of 100,000 447 and 534.  (Where a sequence
    // begins is looked for among its own positions: by a search over all sequences those of 16 tokens each took longer from 50,000 tokens on
    // than by the whole device, 65,536 tokens 386 - 400 us, now 333 - 348.)
    unsigned prompt_cluster = 8;
    while (prompt_cluster > 1 && (i64)n_seqs * prompt_cluster > 128) prompt_cluster /= 2;
    if (prompt_cluster > 1) prompt_cluster = cluster_for(per_seq_max_len, prompt_cluster, CP_THREADS);
    const bool cluster_prompts = prompt_cluster >= 4 && per_seq_max_len > BS_THREADS && per_seq_max_len <= (i64)prompt_cluster * CP_THREADS * CP_ITEMS;
    const bool block_sort = !cluster_prompts && per_seq_max_len > 0 && per_seq_max_len <= BS_MAX_LEN;
    const unsigned corpus_cluster = largest_cluster(dev);
    const bool cluster_corpus = !cluster_prompts && !block_sort && N <= (i64)corpus_cluster * CC_THREADS * CC_ITEMS;
    if (!block_sort && !cluster_prompts)
        tmp.reserve((long long)N * (16 + 4 + 4 + 4 + 2 + 1) + 4ll * (100 * (i64)ts.tiles + (SG_BINS + 1) * (i64)most_blocks + SG_BINS) + 64 * 256);
    const bool have_ends = end_pos != nullptr;
    uint32_t* sa = nullptr;
    bool ok = tmp.get(&ts.lcp, N) && tmp.get(&ts.len, N) && tmp.get(&ts.f, 32 * (i64)ts.tiles) && tmp.get(&ts.e, 32 * (i64)ts.tiles) &&
              tmp.get(&ts.r, 32 * (i64)ts.tiles) && tmp.get(&ts.s, ts.tiles + 1) && tmp.get(&ts.n1, ts.tiles + 1) && tmp.get(&ts.total, 1) &&
              (have_ends || tmp.get(&end_pos, N)) && tmp.get(&sa, N);
    if (!ok) return SD_ERR_NOMEM;
    if (!have_ends) SD_CUDA_OK(sd_launch(seq_end_kernel, grid_for(N, T256), T256, 0, st, d_seq_offsets, n_seqs, N, end_pos));
    int rc;
    if (cluster_prompts) {
        const int V = (int)(max_token / n_seqs);                // (as below)
        rc = cluster_prompt_sort(d_tok, d_seq_offsets, n_seqs, per_seq_max_len, V, bits_for(V), D, prompt_cluster, sa, *walk, st);
        P.walked = true;
    } else if (cluster_corpus) {
        rc = cluster_corpus_sort(d_tok, end_pos, (int)N, bits_for(max_token), D, corpus_cluster, sa, st);
    } else if (block_sort) {
        const int V = (int)(max_token / n_seqs);                // (a sequence's tokens lie in a range of V of their own)
        const int bits = bits_for(V);
        auto sort = [&](auto kernel) { return kernel(d_tok, d_seq_offsets, n_seqs, V, bits, D, sa, st); };
        if (per_seq_max_len <= BS_SMALL) rc = sort(block_suffix_sort<BS_SMALL, 1>);
        else if (per_seq_max_len <= 2 * BS_SMALL) rc = sort(block_suffix_sort<BS_SMALL, 2>);
        else if (per_seq_max_len <= BS_THREADS) rc = sort(block_suffix_sort<BS_SMALL, 4>);
        else if (per_seq_max_len <= 2 * BS_THREADS) rc = sort(block_suffix_sort<BS_THREADS, 2>);
        else if (per_seq_max_len <= 4 * BS_THREADS) rc = sort(block_suffix_sort<BS_THREADS, 4>);
        else if (per_seq_max_len <= 8 * BS_THREADS) rc = sort(block_suffix_sort<BS_THREADS, 8>);
        else rc = sort(block_suffix_sort<BS_THREADS, 16>);
    } else {
        CorpusSort A;
        A.tok = d_tok; A.seq_off = d_seq_offsets; A.n_seqs = n_seqs; A.end_pos = end_pos; A.N = (int)N; A.D = D; A.sa = sa;
        A.key_bits = (unsigned)bits_for(max_token) + 1u;
        // small lots while every block has one at most: a pass is then as short as a block's share
        const bool small = N <= (i64)most_blocks * SG_THREADS * 2;
        const i64 lot = (i64)SG_THREADS * (small ? 2 : 8);
        const i64 lots = (N + lot - 1) / lot;
        const i64 per_block = (lots + most_blocks - 1) / most_blocks;
        // (as many blocks as fit, the last lot of each part full: a multiple of 32)
        A.chunk = (int)(per_block == 1 ? lot : ((N + most_blocks - 1) / most_blocks + 31) / 32 * 32);
        ok = tmp.get(&A.key[0], N) && tmp.get(&A.key[1], N) && tmp.get(&A.val[0], N) && tmp.get(&A.val[1], N) && tmp.get(&A.rank, N) &&
             tmp.get(&A.flags, N / 32 + 1) && tmp.get(&A.go, N / 32 + 1) && tmp.get(&A.table, (i64)SG_BINS * most_blocks) && tmp.get(&A.total, SG_BINS) &&
             tmp.get(&A.count, most_blocks);
        if (!ok) return SD_ERR_NOMEM;
        rc = small ? corpus_sort<2>(A, st) : corpus_sort<8>(A, st);
    }
    if (rc != SD_OK) return rc;
    ts.sa = sa;
    ts.end_pos = end_pos;
    const unsigned grid = (unsigned)((ts.tiles + TS_WARPS - 1) / TS_WARPS);
    if (top_blocks && cudaMemsetAsync(ts.total, 0, sizeof(TreeTotals), st) != cudaSuccess) return SD_ERR_CUDA;
    SD_CUDA_OK(sd_launch(ts.tile_len >= 256 ? ts_tiles_kernel<true> : ts_tiles_kernel<false>, grid, TS_WARPS * 32, 0, st, ts));
    SD_CUDA_OK(sd_launch(ts_carry_kernel, 33, TS_CARRY, 0, st, ts));
    if (top_blocks) SD_CUDA_OK(sd_launch(ts_runs_kernel<true>, grid, TS_WARPS * 32, 0, st, ts));
    else SD_CUDA_OK(sd_launch(ts_runs_kernel<false>, grid, TS_WARPS * 32, 0, st, ts));
    SD_CUDA_OK(sd_launch(ts_carry_front_kernel, (unsigned)(32 + bounds.n + 1), TS_CARRY, 0, st, ts, bounds));
    return SD_OK;
}

template <bool REQ>
static int emit_entries(const TreeScan& ts, const TreeOut& out, cudaStream_t st) {
    const unsigned grid = (unsigned)((ts.tiles + TS_WARPS - 1) / TS_WARPS);
    const size_t smem = sizeof(int2) * 32 * (size_t)TS_WARPS * (ts.tile_len / TS_SUB);
    if (smem > 48 * 1024)
        SD_CUDA_OK(cudaFuncSetAttribute(ts_emit_kernel<REQ>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    SD_CUDA_OK(sd_launch(ts_emit_kernel<REQ>, grid, TS_WARPS * 32, smem, st, ts, out));
    return SD_OK;
}

extern "C" int sd_build(const sd_build_params* p, const int32_t* d_corpus, const int64_t* d_seq_offsets, int32_t n_seqs,
                        void* stream, sd_store** out) {
    if (!out) return SD_ERR_INVALID_ARG;
    *out = nullptr;
    if (!p || p->vocab < 1 || p->depth_cap < 1 || p->depth_cap > SD_MAX_DEPTH || p->max_requests < 1 ||
        p->max_req_tokens < 1 || p->max_spec_cap < 1 || p->max_spec_cap > SD_MAX_SPEC || n_seqs < 0)
        return SD_ERR_INVALID_ARG;
    if (n_seqs > 0 && (!d_corpus || !d_seq_offsets)) return SD_ERR_INVALID_ARG;
    cudaStream_t st = (cudaStream_t)stream;

    i64 N = 0;
    if (n_seqs > 0) {
        SD_CUDA_OK(cudaMemcpyAsync(&N, d_seq_offsets + n_seqs, sizeof(i64), cudaMemcpyDeviceToHost, st));
        SD_CUDA_OK(cudaStreamSynchronize(st));
        if (N < 0 || N > SD_MAX_TOKENS) return SD_ERR_INVALID_ARG;
    }

    sd_store* s = new (std::nothrow) sd_store();
    if (!s) return SD_ERR_NOMEM;
    memset(s, 0, sizeof(*s));
    s->V = p->vocab; s->D = p->depth_cap; s->R = p->max_requests; s->T = p->max_req_tokens; s->M = p->max_spec_cap;
    if (cudaGetDevice(&s->device) != cudaSuccess) { delete s; return SD_ERR_CUDA; }
    s->built = N;
    const int D = s->D;
    s->spn = p->slot_pool_nodes > 0 ? p->slot_pool_nodes : 2ll * s->T * D;
    if (s->spn > SD_MAX_ENTRIES) { delete s; return SD_ERR_INVALID_ARG; }

    bool ok = store_alloc(s, &s->g_root, s->V) && store_alloc(s, &s->g_state, 1) && store_alloc(s, &s->gi, 1) &&
              store_alloc(s, &s->s_ent, (i64)s->R * s->spn) && store_alloc(s, &s->s_root, (i64)s->R * s->V) &&
              store_alloc(s, &s->s_text, (i64)s->R * s->T) && store_alloc(s, &s->s_state, s->R);
    if (!ok) { sd_store_release(s, st); return SD_ERR_NOMEM; }
    StreamSet streams;
    if (!sd_take_streams(s->device, stage_bytes_for(s->R), &streams)) { sd_store_release(s, st); return SD_ERR_CUDA; }
    s->aux = streams.aux; s->ev_fork = streams.ev_fork; s->ev_join = streams.ev_join; s->ev_check = streams.ev_check;
    s->stage = streams.stage; s->stage_bytes = streams.stage_bytes;
    cudaError_t ce = cudaMemsetAsync(s->g_root, 0xFF, sizeof(int32_t) * (size_t)s->V, st);
    if (ce == cudaSuccess) ce = cudaMemsetAsync(s->s_root, 0xFF, sizeof(int32_t) * (size_t)s->R * s->V, st);
    if (ce == cudaSuccess) ce = cudaMemsetAsync(s->s_state, 0, sizeof(SlotState) * (size_t)s->R, st);
    if (ce != cudaSuccess) { sd_store_release(s, st); return SD_ERR_CUDA; }

    Pipeline P(st);
    const int T256 = 256;
    TreeTotals total = {};
    int4* wide_list = nullptr;
    if (N > 0) {
        {
            int* bad = nullptr;
            int h_bad = 0;
            if (!P.tmp.get(&bad, 1)) { sd_store_release(s, st); return SD_ERR_NOMEM; }
            ce = cudaMemsetAsync(bad, 0, sizeof(int), st);
            validate_kernel<<<grid_for(std::max<i64>(N, n_seqs), T256), T256, 0, st>>>(d_corpus, N, s->V, d_seq_offsets,
                                                                                      n_seqs, bad);
            if (ce == cudaSuccess) ce = cudaMemcpyAsync(&h_bad, bad, sizeof(int), cudaMemcpyDeviceToHost, st);
            if (ce == cudaSuccess) ce = cudaStreamSynchronize(st);
            if (ce != cudaSuccess) { sd_store_release(s, st); return SD_ERR_CUDA; }
            if (h_bad) { sd_store_release(s, st); return SD_ERR_INVALID_ARG; }
        }
        const int rc = pipeline_run(P, d_corpus, d_seq_offsets, n_seqs, N, s->V, D, true, st);
        if (rc != SD_OK) { sd_store_release(s, st); return rc; }
        ce = cudaMemcpyAsync(&total, P.ts.total, sizeof(total), cudaMemcpyDeviceToHost, st);
        if (ce == cudaSuccess) ce = cudaStreamSynchronize(st);
        if (ce != cudaSuccess) { sd_store_release(s, st); return SD_ERR_CUDA; }
    }
    s->g_cap = sd_pool_entries(total, p->global_extra_nodes);
    if (s->g_cap < 0) { sd_store_release(s, st); return SD_ERR_INVALID_ARG; }
    const i64 n_nodes = total.below + total.top, used_entries = n_nodes + total.wide;
    if (total.n_wide > 0 && !P.tmp.get(&wide_list, total.n_wide)) { sd_store_release(s, st); return SD_ERR_NOMEM; }
    if (!store_alloc(s, &s->g_ent, s->g_cap)) { sd_store_release(s, st); return SD_ERR_NOMEM; }

    if (N > 0) {
        TreeOut out;
        memset(&out, 0, sizeof(out));
        out.ent = s->g_ent; out.root = s->g_root; out.wide = wide_list;
        const int erc = emit_entries<false>(P.ts, out, st);
        if (erc != SD_OK) { sd_store_release(s, st); return erc; }
        if (total.n_wide > 0) {
            ts_wide_place_kernel<<<grid_for(total.n_wide, T256), T256, 0, st>>>(P.ts, wide_list, s->g_ent, (int)n_nodes);
            ts_wide_fill_kernel<<<(unsigned)total.n_wide, TOP_THREADS, 0, st>>>(wide_list, s->g_ent);
        }
    }
    init_global_state_kernel<<<1, 1, 0, st>>>(s->g_state, (int)used_entries, (int)n_nodes, N);
    ce = cudaStreamSynchronize(st);
    if (ce == cudaSuccess) ce = cudaGetLastError();
    if (ce != cudaSuccess) { sd_store_release(s, st); return SD_ERR_CUDA; }
    *out = s;
    return SD_OK;
}

extern "C" const char* sd_strerror(int code) {
    switch (code) {
        case SD_OK: return "ok";
        case SD_ERR_INVALID_ARG: return "invalid argument";
        case SD_ERR_CUDA: return "CUDA runtime error";
        case SD_ERR_NOMEM: return "out of device memory";
        case SD_ERR_CAPACITY: return "capacity exceeded";
        default: return "unknown error";
    }
}

// ---------------------------------------------------------------------------------------------
// sd_build_requests: the per-request trees of a batch of new requests, built from their prompts
// by the same sort-based pipeline as the global tree instead of token by token.  The prompts
// are kept apart by giving every request its own token range (token + rank * V), so one
// suffix sort orders all of them request by request and one pre-order numbering lays every
// request's nodes down contiguously; each request's part is then written into its own pool.
namespace {

__device__ __forceinline__ int seq_rank_of(const int64_t* off, int n, i64 pos) {
    int lo = 0, hi = n;                               // largest q with off[q] <= pos
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (off[mid] <= pos) lo = mid; else hi = mid;
    }
    return lo;
}

// Offsets and slots of a few requests, as arguments of the kernel (a copy of them took 4 us of a refill's 100).
struct RequestArgs {
    static constexpr int MOST = 64;
    int64_t off[MOST + 1];
    int32_t slot[MOST];
};

// The tokens in ranges of their own, request by request, and where their request ends.  A token outside the vocabulary
// sets both flags (the host's one lies in its memory).  ARGS: also lays down the call's offsets and slots for the kernels behind it.
template <bool ARGS>
__global__ void map_tokens_kernel(const int32_t* tok, RequestArgs A, int64_t* off, int32_t* slot, int n, i64 N, int V, int32_t* out, int* end_pos,
                                  BadCall bad, int* host_bad) {
    sd_chain_begin();
    const i64 i = (i64)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t* const o = ARGS ? A.off : off;
    if (ARGS && i <= n) {
        off[i] = A.off[i];
        if (i < n) slot[i] = A.slot[i];
    }
    if (i >= N) return;
    int t = tok[i];
    if (t < 0 || t >= V) { *bad.last = bad.call; *host_bad = 1; t = 0; }
    const int q = seq_rank_of(o, n, i);
    out[i] = q * V + t;
    end_pos[i] = (int)o[q + 1];
}

// One block per request: forget the slot's old tree, store the new text, bookkeeping.  The entries and the active nodes are
// laid down behind this (ts_emit_kernel), but for active nodes that there are none of.
constexpr int PREP_THREADS = 1024;
__global__ void __launch_bounds__(PREP_THREADS)
requests_prepare_kernel(sd_store sv, int n, const int32_t* slot_ids, const int64_t* off, const int32_t* tok, const int* s_req,
                        const int* n1_req, BadCall bad, bool walked) {
    sd_chain_begin();
    const int q = blockIdx.x, tid = threadIdx.x;
    if (q >= n || bad()) return;
    const int slot = slot_ids[q];
    if (slot < 0 || slot >= sv.R) return;
    SlotState* ss = sv.s_state + slot;
    int32_t* text = sv.s_text + (i64)slot * sv.T;
    int32_t* root = sv.s_root + (i64)slot * sv.V;
    const int old_len = ss->len;
    const i64 lo = off[q], hi = off[q + 1];
    const int used = n1_req ? n1_req[q + 1] - n1_req[q] + s_req[q + 1] - s_req[q] : 0;
    const bool ok = used <= sv.spn && hi - lo <= sv.T;
    const int len = ok ? (int)(hi - lo) : 0;
    for (int k = tid; k < old_len; k += PREP_THREADS) root[text[k]] = -1;
    __syncthreads();
    if (hi - lo <= sv.T)
        for (i64 k = tid; k < hi - lo; k += PREP_THREADS) text[k] = tok[lo + k];
    // (depth D, too: its node has no children and is asked for by nobody)
    if (tid < SD_MAX_DEPTH && (tid + 1 > len || tid + 1 >= sv.D)) set_active(ss, tid + 1, -1, 0, 0);
    if (tid == 0) {
        ss->len = len; ss->used = ok ? used : 0; ss->live = ok ? used : 0;
        ss->status = ok ? 0 : SD_STATUS_POOL_FULL;
        ss->gen += 1;
        if (walked) ss->g_gen = ss->gen;                         // (request_walk has left the global match nodes)
    }
}

}  // namespace

extern "C" int sd_build_requests(sd_store* s, int32_t n, const int32_t* h_slot, const int64_t* h_offsets,
                                 const int32_t* d_tokens, void* stream) {
    if (!s || n < 0) return SD_ERR_INVALID_ARG;
    SD_CHECK_DEVICE(s);
    if (n == 0) return SD_OK;
    if (!h_slot || !h_offsets || n > s->R) return SD_ERR_INVALID_ARG;
    if (h_offsets[0] != 0) return SD_ERR_INVALID_ARG;
    try {
        std::vector<bool> seen((size_t)s->R);
        for (int q = 0; q < n; ++q) {
            if (h_offsets[q + 1] < h_offsets[q] || h_slot[q] < 0 || h_slot[q] >= s->R || seen[h_slot[q]]) return SD_ERR_INVALID_ARG;
            seen[h_slot[q]] = true;                              // a slot once per call
        }
    } catch (const std::bad_alloc&) {
        return SD_ERR_NOMEM;
    }
    const i64 N = h_offsets[n];
    if (N > 0 && !d_tokens) return SD_ERR_INVALID_ARG;
    if ((i64)n * s->V >= (1ll << 31) - 2 || N > SD_MAX_TOKENS) return SD_ERR_CAPACITY;
    cudaStream_t st = (cudaStream_t)stream;
    const int T256 = 256, D = s->D;

    Pipeline P(st);
    if (!s->ws) {
        s->ws = new (std::nothrow) sd_workspace();
        if (!s->ws) return SD_ERR_NOMEM;
        memset(s->ws, 0, sizeof(*s->ws));
    }
    P.tmp.keep = s->ws;                                          // temporaries are kept for the next call
    // Arguments go over with the first kernel, those of many requests in one copy from pinned memory.  Everything is
    // queued behind the check of the tokens and changes nothing if it fails; the host waits for the check alone, so
    // the GPU does not run dry meanwhile (it did, for some 50 us of a 185 us refill).
    const size_t arg_bytes = 8 * ((size_t)n + 1) + 4 * (size_t)n;
    unsigned char* d_args = nullptr;
    int32_t* mtok = nullptr;
    int *end_pos = nullptr, *s_req = nullptr, *n1_req = nullptr;
    bool ok = P.tmp.get(&d_args, (i64)arg_bytes) && P.tmp.get(&mtok, N) && P.tmp.get(&end_pos, N) && P.tmp.get(&s_req, n + 1) &&
              P.tmp.get(&n1_req, n + 1);
    if (!ok) return SD_ERR_NOMEM;
    int64_t* const d_off = reinterpret_cast<int64_t*>(d_args);
    int32_t* const d_slot = reinterpret_cast<int32_t*>(d_off + n + 1);
    s->request_calls = s->request_calls == 0x7fffffff ? 1 : s->request_calls + 1;
    const BadCall bad{&s->g_state->bad_call, s->request_calls};
    volatile int* const h_bad = (volatile int*)s->stage;
    *h_bad = 0;
    // (from here on the pinned memory is in use: whatever fails, the call waits for it before it returns)
    cudaError_t ce = cudaSuccess;
    const unsigned map_grid = grid_for(std::max<i64>(N, n + 1), T256);
    RequestArgs args;
    if (n <= RequestArgs::MOST && N > 0) {
        memcpy(args.off, h_offsets, 8 * ((size_t)n + 1));
        memcpy(args.slot, h_slot, 4 * (size_t)n);
        ce = sd_launch(map_tokens_kernel<true>, map_grid, T256, 0, st, d_tokens, args, d_off, d_slot, n, N, s->V, mtok, end_pos, bad, (int*)s->stage);
    } else {
        unsigned char* const h_args = (unsigned char*)s->stage + 16;
        memcpy(h_args, h_offsets, 8 * ((size_t)n + 1));
        memcpy(h_args + 8 * ((size_t)n + 1), h_slot, 4 * (size_t)n);
        ce = cudaMemcpyAsync(d_args, h_args, arg_bytes, cudaMemcpyHostToDevice, st);
        if (ce == cudaSuccess && N > 0)
            ce = sd_launch(map_tokens_kernel<false>, map_grid, T256, 0, st, d_tokens, args, d_off, d_slot, n, N, s->V, mtok, end_pos, bad, (int*)s->stage);
    }
    const cudaError_t record = cudaEventRecord(s->ev_check, st);
    int rc = ce == cudaSuccess && record == cudaSuccess ? SD_OK : SD_ERR_CUDA;
    if (rc == SD_OK && N > 0) {
        i64 max_len = 0;
        for (int q = 0; q < n; ++q) max_len = std::max<i64>(max_len, h_offsets[q + 1] - h_offsets[q]);
        const RequestWalk walk{*s, n, s->appended ? std::min(s->R, MOST_REFRESHED) : 0, d_slot, d_off, d_tokens, bad};
        rc = pipeline_run(P, mtok, d_off, n, N, (i64)n * s->V, D, false, st, max_len, end_pos, RequestBounds{n, d_off, s_req, n1_req}, &walk);
        if (P.walked) s->appended = 0;
        if (rc == SD_OK && N * D > SD_MAX_ENTRIES) {             // the trees' nodes may not fit 32 bits (up to then nothing has changed)
            TreeTotals total = {};
            if (cudaMemcpyAsync(&total, P.ts.total, sizeof(total), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
                cudaStreamSynchronize(st) != cudaSuccess) rc = SD_ERR_CUDA;
            else if (total.below + total.top > SD_MAX_ENTRIES) rc = SD_ERR_CAPACITY;
        }
    }
    if (rc == SD_OK && sd_launch(requests_prepare_kernel, (unsigned)n, PREP_THREADS, 0, st, *s, n, d_slot, d_off, d_tokens, N > 0 ? s_req : nullptr,
                                 N > 0 ? n1_req : nullptr, bad, P.walked) != cudaSuccess) rc = SD_ERR_CUDA;
    if (rc == SD_OK && N > 0) {
        TreeOut out;
        memset(&out, 0, sizeof(out));
        out.sv = *s; out.n_req = n; out.slot = d_slot; out.off = d_off; out.s_req = s_req; out.n1_req = n1_req; out.bad = bad;
        rc = emit_entries<true>(P.ts, out, st);
    }
    // (the pinned memory is free again, too)
    const cudaError_t checked = record == cudaSuccess ? cudaEventSynchronize(s->ev_check) : cudaStreamSynchronize(st);
    if (rc != SD_OK) return rc;
    if (checked != cudaSuccess) return SD_ERR_CUDA;
    if (*h_bad) return SD_ERR_INVALID_ARG;
    // (the temporaries stay in the store's workspace, and a later call on
    // another stream must be ordered behind this one by the caller like any other use of the store)
    SD_CUDA_OK(cudaGetLastError());
    return SD_OK;
}
