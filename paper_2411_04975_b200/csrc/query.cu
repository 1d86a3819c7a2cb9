// Read-only queries on a store: COUNT of token paths (the quantity Eq. 1
// divides), every node of a tree as a record, empirical entropy, per-slot and store-wide bookkeeping.
#include <algorithm>
#include <stddef.h>

#include "common.cuh"

namespace {

__global__ void query_counts_kernel(sd_store sv, int n, const int32_t* d_tree, const int64_t* d_offsets,
                                    const int32_t* d_paths, int32_t* d_counts) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int tree = d_tree[i];
    const long long b = d_offsets[i], e = d_offsets[i + 1];
    const int len = (int)(e - b);
    int count = 0;
    if (tree >= -1 && tree < sv.R && len >= 1 && len <= sv.D) {
        const int4* ent = tree < 0 ? sv.g_ent : sv.s_ent + (long long)tree * sv.spn;
        const int32_t* root = tree < 0 ? sv.g_root : sv.s_root + (long long)tree * sv.V;
        int x = d_paths[b];
        int node = (x >= 0 && x < sv.V) ? root[x] : -1;
        for (int k = 1; k < len && node >= 0; ++k) {
            const int4 pe = ent[node];
            const int cb = pe.z, nc = (int)((unsigned)pe.w & RUN_COUNT_MASK);
            x = d_paths[b + k];
            int lo = 0, hi = nc;
            while (lo < hi) {
                const int mid = (lo + hi) >> 1;
                if (ent[cb + mid].x < x) lo = mid + 1; else hi = mid;
            }
            node = (lo < nc && ent[cb + lo].x == x) ? cb + lo : -1;
        }
        if (node >= 0) count = ent[node].y;
    }
    d_counts[i] = count;
}

__global__ void slot_info_kernel(sd_store sv, int n, const int32_t* d_slot, int32_t* d_len, int32_t* d_nodes,
                                 int32_t* d_status) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int slot = d_slot[i];
    int len = 0, nodes = 0, status = SD_STATUS_BAD_SLOT;
    if (slot >= 0 && slot < sv.R) {
        const SlotState* ss = sv.s_state + slot;
        len = ss->len; nodes = ss->live; status = ss->status;
    }
    if (d_len) d_len[i] = len;
    if (d_nodes) d_nodes[i] = nodes;
    if (d_status) d_status[i] = status;
}

}  // namespace

extern "C" int sd_query_counts(sd_store* s, int32_t n, const int32_t* d_tree, const int64_t* d_offsets,
                               const int32_t* d_paths, int32_t* d_counts, void* stream) {
    if (!s || n < 0) return SD_ERR_INVALID_ARG;
    SD_CHECK_DEVICE(s);
    if (n == 0) return SD_OK;
    if (!d_tree || !d_offsets || !d_paths || !d_counts) return SD_ERR_INVALID_ARG;
    query_counts_kernel<<<(unsigned)((n + 127) / 128), 128, 0, (cudaStream_t)stream>>>(*s, n, d_tree, d_offsets, d_paths,
                                                                                     d_counts);
    SD_CUDA_OK(cudaGetLastError());
    return SD_OK;
}

extern "C" int sd_slot_info(sd_store* s, int32_t n, const int32_t* d_slot, int32_t* d_len, int32_t* d_nodes,
                            int32_t* d_status, void* stream) {
    if (!s || n < 0) return SD_ERR_INVALID_ARG;
    SD_CHECK_DEVICE(s);
    if (n == 0) return SD_OK;
    if (!d_slot) return SD_ERR_INVALID_ARG;
    slot_info_kernel<<<(unsigned)((n + 127) / 128), 128, 0, (cudaStream_t)stream>>>(*s, n, d_slot, d_len, d_nodes,
                                                                                  d_status);
    SD_CUDA_OK(cudaGetLastError());
    return SD_OK;
}

extern "C" int sd_stats(sd_store* s, sd_stats_t* out, void* stream) {
    if (!s || !out) return SD_ERR_INVALID_ARG;
    SD_CHECK_DEVICE(s);
    GlobalState g;
    SD_CUDA_OK(cudaMemcpyAsync(&g, s->g_state, sizeof(g), cudaMemcpyDeviceToHost, (cudaStream_t)stream));
    SD_CUDA_OK(cudaStreamSynchronize((cudaStream_t)stream));
    out->global_nodes = g.live;
    out->global_pool_used = g.used;
    out->global_pool_cap = s->g_cap;
    out->global_tokens = g.tokens;
    out->slot_pool_nodes = s->spn;
    out->device_bytes = s->device_bytes;
    out->global_status = g.status;
    return SD_OK;
}

// ---------------------------------------------------------------------------------------------
// Empirical entropy of a tree (Appendix "Predicting SuffixDecoding Effectiveness"): for every
// node the entropy of its children's count distribution, averaged over the nodes with the
// sibling sum as weight.  A traversal from the root table (the pools also hold abandoned runs and
// top-block copies, so a plain sweep over the pool would count too much).
//
// Every node with children is read once: 16 B per node is the floor (119 us for 48.6 M nodes at the
// measured copy rate), and what keeps a traversal from it is a chain of dependent loads per
// thread and, where every node goes through a queue, the queue.  So a lane goes on with the FIRST
// child of the node it has just done, whose run is laid down right behind the node's own (only
// children, most of a tree, never meet a queue at all); the other children that have children
// of their own are queued as (run, size), one counter update per warp.  Runs of more than 32
// children are done by the whole warp.  One launch per generation of the queue, nothing read
// back between them: a node's generation is the number of non-first children on its path.
// 48.6 M nodes: 14.8 ms as one thread per node and level with a round trip per level, of which
// 11.2 ms in the kernels (long runs by one thread, one counter update per node).
namespace {

constexpr int ENT_THREADS = 256;

__device__ __forceinline__ double entropy_term(unsigned c, double S) {      // -(c/S) log2(c/S) * S
    const double d = (double)c;
    return -d * log2(d / S);
}

// adds up over the block, one atomic each
__device__ __forceinline__ void entropy_accumulate(double part, unsigned long long w, double* acc, unsigned long long* wsum) {
    __shared__ double sp[ENT_THREADS / 32];
    __shared__ unsigned long long sw[ENT_THREADS / 32];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        part += __shfl_xor_sync(0xffffffffu, part, o);
        w += __shfl_xor_sync(0xffffffffu, w, o);
    }
    if ((threadIdx.x & 31) == 0) { sp[threadIdx.x >> 5] = part; sw[threadIdx.x >> 5] = w; }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int k = 1; k < ENT_THREADS / 32; ++k) { part += sp[k]; w += sw[k]; }
        if (part != 0.0) atomicAdd(acc, part);
        if (w) atomicAdd(wsum, w);
    }
}

// entries for `mine` items per lane in a queue: one counter update per warp
__device__ __forceinline__ int entropy_reserve(int mine, int* counter, int lane) {
    int inc = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += y;
    }
    int at = 0;
    if (lane == 31 && inc > 0) at = atomicAdd(counter, inc);
    return __shfl_sync(0xffffffffu, at, 31) + inc - mine;
}

// depth-1 nodes: total count, and the first items
__global__ void __launch_bounds__(ENT_THREADS)
entropy_root_sum_kernel(const int4* ent, const int32_t* root, int V, unsigned long long* total, int2* queue, int* n_queue) {
    const int v = blockIdx.x * ENT_THREADS + threadIdx.x, lane = threadIdx.x & 31;
    unsigned long long c = 0;
    int2 run = make_int2(0, 0);
    if (v < V) {
        const int idx = root[v];
        if (idx >= 0) {
            const int4 e = ent[idx];
            c = (unsigned)e.y;
            run = make_int2(e.z, (int)((unsigned)e.w & RUN_COUNT_MASK));
        }
    }
    const int at = entropy_reserve(run.y > 0 ? 1 : 0, n_queue, lane);
    if (run.y > 0) queue[at] = run;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
    if (lane == 0 && c) atomicAdd(total, c);
}

__global__ void __launch_bounds__(ENT_THREADS)
entropy_root_kernel(const int4* ent, const int32_t* root, int V, const unsigned long long* total, double* acc,
                    unsigned long long* wsum) {
    const int v = blockIdx.x * ENT_THREADS + threadIdx.x;
    double part = 0.0;
    const double S = (double)*total;
    if (v < V) {
        const int idx = root[v];
        if (idx >= 0) part = entropy_term((unsigned)ent[idx].y, S);
    }
    entropy_accumulate(part, v == 0 ? *total : 0ull, acc, wsum);
}

// One generation: a lane per queued run, then down its first children.
__global__ void __launch_bounds__(ENT_THREADS)
entropy_runs_kernel(const int4* __restrict__ ent, const int2* __restrict__ queue, const int* __restrict__ n_queue, int2* next,
                    int* n_next, double* acc, unsigned long long* wsum) {
    const unsigned FULL = 0xffffffffu;
    const int n_items = *n_queue, lane = threadIdx.x & 31;
    if ((int)(blockIdx.x * ENT_THREADS) >= n_items) return;      // (uniform for the block)
    const int stride = (int)gridDim.x * ENT_THREADS;
    int item = (int)blockIdx.x * ENT_THREADS + (int)threadIdx.x;
    double part = 0.0;
    unsigned long long wt = 0;
    int2 run = make_int2(0, 0);
    while (true) {
        if (run.y == 0 && item < n_items) { run = queue[item]; item += stride; }
        if (!__any_sync(FULL, run.y > 0)) break;
        // ---- runs of up to 32 children: a lane each
        const int cb = run.x, n = run.y;
        int push = 0;
        if (n > 0 && n <= 32) {
            const int4 first = ent[cb];
            unsigned S = (unsigned)first.y;
            for (int k = 1; k < n; ++k) {
                const int4 c = ent[cb + k];
                S += (unsigned)c.y;
                push += ((unsigned)c.w & RUN_COUNT_MASK) ? 1 : 0;
            }
            wt += S;
            if (n > 1) {                                         // an only child has probability 1: its term is 0
                const double dS = (double)S;
                for (int k = 0; k < n; ++k) part += entropy_term((unsigned)ent[cb + k].y, dS);
            }
            run = make_int2(first.z, (int)((unsigned)first.w & RUN_COUNT_MASK));
        }
        if (__any_sync(FULL, push > 0)) {
            int at = entropy_reserve(push, n_next, lane);
            if (push > 0)
                for (int k = 1; k < n; ++k) {
                    const int4 c = ent[cb + k];
                    const int nc = (int)((unsigned)c.w & RUN_COUNT_MASK);
                    if (nc) next[at++] = make_int2(c.z, nc);
                }
        }
        // ---- longer runs: the warp does them one after the other
        unsigned wide = __ballot_sync(FULL, n > 32);
        while (wide) {
            const int src = __ffs(wide) - 1;
            wide &= wide - 1;
            const int wcb = __shfl_sync(FULL, cb, src), wn = __shfl_sync(FULL, n, src);
            unsigned s = 0;
            for (int k = lane; k < wn; k += 32) s += (unsigned)ent[wcb + k].y;
            const unsigned S = __reduce_add_sync(FULL, s);       // (a parent's occurrences fit 31 bits)
            const double dS = (double)S;
            if (lane == 0) wt += S;
            for (int k0 = 0; k0 < wn; k0 += 32) {
                int4 c = make_int4(0, 0, 0, 0);
                if (k0 + lane < wn) { c = ent[wcb + k0 + lane]; part += entropy_term((unsigned)c.y, dS); }
                const int nc = (int)((unsigned)c.w & RUN_COUNT_MASK);
                const int at = entropy_reserve(nc > 0 ? 1 : 0, n_next, lane);
                if (nc > 0) next[at] = make_int2(c.z, nc);
            }
            if (lane == src) run.y = 0;
        }
    }
    entropy_accumulate(part, wt, acc, wsum);
}

// The whole of a global tree that is still as it was laid down offline: its n nodes are the first n entries, each
// once (long runs have a second copy behind them), so they are simply read in order, a lane per node.
//
// With f(x) = x log x, a node whose children's counts c add up to S adds f(S) - sum f(c) to the numerator and S to the
// denominator.  Over the whole tree every node below the root is a child once, so the denominator is the sum of all counts, and
// the numerator is f(all tokens) - sum of f(count) over the leaves + sum of f(S) - f(count) over the nodes with children; and S is
// the node's own count unless a sequence ends with the node (RUN_ENDS, one node for every suffix shorter than the tree is deep).  So
// only these few look at their children, and the others not even at their count.  The values are COUNTED, with their signs, in
// shared memory, and the block that ends last takes the logarithms, once per value, and adds up
// with the rounding errors carried along: equal values cancel exactly, and no node costs a division or a logarithm in double
// precision.  (Those of branching nodes' children, 32 at a time: 348 us for 41 M nodes, now 127, 5.1 TB/s.  Error against 80-bit
// sums over eight corpora: 2.9e-16 to 1.8e-15, now 1.2e-17 to 1.5e-16.)
// Large values are listed, and every block takes the logarithms of its own: mostly few, but a corpus of short sequences that occur again and
// again has tens of thousands (28 M tokens, 1,318 sequences of 20: 69 us with all of them left to the block that ends last, now 45).
constexpr int ENT_SWEEP = 512;                // threads per block
constexpr int ENT_BLOCKS = 3;                 // per SM
constexpr int ENT_VALUES = 1024;              // values below are counted, others listed
constexpr int ENT_AHEAD = 4;                  // loads in flight per lane
constexpr int ENT_OWN = 1024;                 // values that a block lists itself; more go to all blocks' list
struct __align__(16) EntropySums {
    unsigned long long wsum;
    double sum, rest;                         // the numerator in two parts
    int epoch, live;                          // of the tree
    int n_list, done;                         // blocks
    int net[ENT_VALUES];
};

__global__ void __launch_bounds__(ENT_SWEEP, ENT_BLOCKS)
entropy_sweep_kernel(const int4* __restrict__ ent, const GlobalState* __restrict__ gs, EntropySums* out, double2* parts, int* list) {
    __shared__ int net[ENT_VALUES];
    __shared__ int own[ENT_OWN], n_own;
    __shared__ int2 queue[ENT_SWEEP / 32][32 + 32 * ENT_AHEAD];  // nodes that a sequence ends with
    const unsigned FULL = 0xffffffffu;
    const int tid = threadIdx.x, lane = tid & 31, wib = tid >> 5;
    const int n = gs->live;
    if (blockIdx.x == 0 && tid == 0) { out->epoch = gs->epoch; out->live = n; }
    if (gs->epoch != 1) return;                                  // something was inserted since the build
    for (int v = tid; v < ENT_VALUES; v += ENT_SWEEP) net[v] = 0;
    if (tid == 0) n_own = 0;
    __syncthreads();
    int2* const q = queue[wib];
    const unsigned lt = (1u << lane) - 1u;
    int waiting = 0, twos = 0;                                   // (value 2, the most frequent by far, in registers)
    unsigned long long wt = 0;
    auto add = [&](unsigned v, int k) {                          // k f(v)
        if (v < 2u) return;                                      // (f(1) is 0)
        if (v == 2u) twos += k;
        else if (v < (unsigned)ENT_VALUES) atomicAdd(&net[v], k);
        else {
            const int at = atomicAdd(&n_own, 1), x = k > 0 ? (int)v : -(int)v;
            if (at < ENT_OWN) own[at] = x;
            else list[atomicAdd(&out->n_list, 1)] = x;
        }
    };
    auto ended = [&](int2 e) {                                   // children at e.x, e.y as the w field
        const int k = (int)((unsigned)e.y & RUN_COUNT_MASK);
        unsigned S = 0;
        if ((unsigned)e.y & RUN_HAS_TOP) S = (unsigned)ent[e.x - SD_TOP_BLOCK].x;    // (a parent's occurrences fit 31 bits)
        else
            for (int u0 = 0; u0 < k; u0 += 4) {
                unsigned c[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) c[u] = u0 + u < k ? (unsigned)ent[e.x + u0 + u].y : 0u;
                S += c[0] + c[1] + c[2] + c[3];
            }
        add(S, 1);
    };
    const long long stride = (long long)gridDim.x * (ENT_SWEEP * ENT_AHEAD);
    for (long long i0 = ((long long)blockIdx.x * ENT_SWEEP + (tid & ~31)) * ENT_AHEAD; i0 < n; i0 += stride) {
        int4 e[ENT_AHEAD];
#pragma unroll
        for (int a = 0; a < ENT_AHEAD; ++a) {
            e[a] = make_int4(0, 0, 0, 0);
            if (i0 + a * 32 + lane < n) e[a] = ent[i0 + a * 32 + lane];
        }
#pragma unroll
        for (int a = 0; a < ENT_AHEAD; ++a) {
            const unsigned w = (unsigned)e[a].w;
            wt += (unsigned)e[a].y;
            if ((w & RUN_COUNT_MASK) == 0u || (w & RUN_ENDS)) add((unsigned)e[a].y, -1);
            const unsigned ends = __ballot_sync(FULL, (w & RUN_ENDS) != 0u);
            if ((ends >> lane) & 1u) q[waiting + __popc(ends & lt)] = make_int2(e[a].z, e[a].w);
            waiting += __popc(ends);
        }
        __syncwarp();
        while (waiting >= 32) { waiting -= 32; ended(q[waiting + lane]); }
        __syncwarp();
    }
    if (lane < waiting) ended(q[lane]);
    twos = __reduce_add_sync(FULL, twos);
    if (lane == 0 && twos) atomicAdd(&net[2], twos);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) wt += __shfl_xor_sync(FULL, wt, o);
    if (lane == 0 && wt) atomicAdd(&out->wsum, wt);
    __syncthreads();
    for (int v = tid; v < ENT_VALUES; v += ENT_SWEEP) if (net[v]) atomicAdd(&out->net[v], net[v]);
    double hi = 0.0, lo = 0.0;
    auto plus = [&](double b, double e) {                        // exact sum of hi and b (Knuth), the rest to lo
        const double s = __dadd_rn(hi, b), bb = __dsub_rn(s, hi);
        lo = __dadd_rn(lo, __dadd_rn(e, __dadd_rn(__dsub_rn(hi, __dsub_rn(s, bb)), __dsub_rn(b, bb))));
        hi = s;
    };
    auto times_f = [&](double k, double v) {
        const double f = __dmul_rn(v, log2(v)), p = __dmul_rn(k, f);
        plus(p, __fma_rn(k, f, -p));
    };
    __shared__ double shi[ENT_SWEEP / 32], slo[ENT_SWEEP / 32];
    auto over_lanes = [&]() {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) { const double b = __shfl_xor_sync(FULL, hi, o), e = __shfl_xor_sync(FULL, lo, o); plus(b, e); }
    };
    auto over_block = [&]() {                                    // for warp 0
        over_lanes();
        if (lane == 0) { shi[wib] = hi; slo[wib] = lo; }
        __syncthreads();
        if (wib == 0) {
            hi = lane < ENT_SWEEP / 32 ? shi[lane] : 0.0; lo = lane < ENT_SWEEP / 32 ? slo[lane] : 0.0;
            over_lanes();
        }
    };
    const int mine = min(n_own, ENT_OWN);
    if (mine > 0) {
        for (int i = tid; i < mine; i += ENT_SWEEP) { const int v = own[i]; times_f(v > 0 ? 1.0 : -1.0, fabs((double)v)); }
        over_block();
    }
    if (tid == 0) parts[blockIdx.x] = make_double2(hi, lo);
    // ---- the block that ends last adds up
    __shared__ bool last;
    __threadfence();
    __syncthreads();
    if (tid == 0) last = atomicAdd(&out->done, 1) == (int)gridDim.x - 1;
    __syncthreads();
    if (!last) return;
    __threadfence();
    hi = 0.0; lo = 0.0;
    for (int b = tid; b < (int)gridDim.x; b += ENT_SWEEP) { const double2 x = __ldcg(&parts[b]); plus(x.x, x.y); }
    if (tid == 0 && n > 0) times_f(1.0, (double)gs->tokens);
    for (int v = tid; v < ENT_VALUES; v += ENT_SWEEP) { const int k = __ldcg(&out->net[v]); if (k) times_f((double)k, (double)v); }
    const int n_list = __ldcg(&out->n_list);
    for (int i = tid; i < n_list; i += ENT_SWEEP) { const int v = __ldcg(&list[i]); times_f(v > 0 ? 1.0 : -1.0, fabs((double)v)); }
    over_block();
    if (tid == 0) { out->sum = hi; out->rest = lo; }
}

}  // namespace

extern "C" int sd_entropy(sd_store* s, int32_t tree, double* h_entropy, void* stream) {
    if (!s || !h_entropy || tree < -1 || tree >= s->R) return SD_ERR_INVALID_ARG;
    SD_CHECK_DEVICE(s);
    cudaStream_t st = (cudaStream_t)stream;
    const int4* ent = tree < 0 ? s->g_ent : s->s_ent + (long long)tree * s->spn;
    const int32_t* root = tree < 0 ? s->g_root : s->s_root + (long long)tree * s->V;
    int live = 0, sms = 0;
    SD_CUDA_OK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, s->device));
    if (tree < 0) {
        // the tree as it was built, if it is; else this only tells its size
        // Values of ENT_VALUES and more: at each depth as many nodes have such a count as built / ENT_VALUES at most, and each is
        // listed twice at most.
        const size_t most = (size_t)(s->built / ENT_VALUES) * 2 * (size_t)s->D;
        EntropySums* d = nullptr;
        EntropySums h;
        const unsigned blocks = (unsigned)(sms * ENT_BLOCKS);
        if (sd_device_malloc((void**)&d, sizeof(EntropySums) + sizeof(double2) * blocks + sizeof(int) * most) != cudaSuccess) {
            cudaGetLastError();
            return SD_ERR_NOMEM;
        }
        double2* const parts = reinterpret_cast<double2*>(d + 1);
        cudaError_t ce = cudaMemsetAsync(d, 0, sizeof(EntropySums), st);
        entropy_sweep_kernel<<<blocks, ENT_SWEEP, 0, st>>>(ent, s->g_state, d, parts, reinterpret_cast<int*>(parts + blocks));
        if (ce == cudaSuccess) ce = cudaMemcpyAsync(&h, d, offsetof(EntropySums, net), cudaMemcpyDeviceToHost, st);
        const cudaError_t done = cudaStreamSynchronize(st);
        if (ce == cudaSuccess) ce = done;
        sd_device_free(d);
        if (ce == cudaSuccess) ce = cudaGetLastError();
        if (ce != cudaSuccess) return SD_ERR_CUDA;
        if (h.epoch == 1) {
            *h_entropy = h.wsum ? (h.sum + h.rest) / (double)h.wsum : 0.0;
            return SD_OK;
        }
        live = h.live;
    } else {
        SD_CUDA_OK(cudaMemcpyAsync(&live, &s->s_state[tree].live, sizeof(int), cudaMemcpyDeviceToHost, st));
        SD_CUDA_OK(cudaStreamSynchronize(st));
    }
    *h_entropy = 0.0;
    if (live <= 0) return SD_OK;
    // a queued node has a child, and no node is queued twice: at most half of the nodes per generation
    const long long room = std::max<long long>(s->V, (long long)live / 2 + 1);
    struct Small { unsigned long long total, wsum; double acc; int count[SD_MAX_DEPTH + 1]; } h_small;
    int2* queue = nullptr;
    Small* d_small = nullptr;
    if (sd_device_malloc((void**)&queue, sizeof(int2) * 2 * (size_t)room) != cudaSuccess ||
        sd_device_malloc((void**)&d_small, sizeof(Small)) != cudaSuccess) {
        cudaGetLastError();
        sd_device_free(queue); sd_device_free(d_small);
        return SD_ERR_NOMEM;
    }
    cudaError_t ce = cudaMemsetAsync(d_small, 0, sizeof(Small), st);
    const unsigned root_grid = (unsigned)((s->V + ENT_THREADS - 1) / ENT_THREADS);
    entropy_root_sum_kernel<<<root_grid, ENT_THREADS, 0, st>>>(ent, root, s->V, &d_small->total, queue, &d_small->count[0]);
    entropy_root_kernel<<<root_grid, ENT_THREADS, 0, st>>>(ent, root, s->V, &d_small->total, &d_small->acc, &d_small->wsum);
    // (a path of D nodes has at most D - 1 of them with children, so at most D - 1 generations)
    const unsigned grid = (unsigned)std::min<long long>(sms * 8, (room + ENT_THREADS - 1) / ENT_THREADS);
    for (int g = 0; g + 1 < s->D; ++g)
        entropy_runs_kernel<<<grid, ENT_THREADS, 0, st>>>(ent, queue + (g & 1) * room, &d_small->count[g], queue + ((g & 1) ^ 1) * room,
                                                          &d_small->count[g + 1], &d_small->acc, &d_small->wsum);
    if (ce == cudaSuccess) ce = cudaMemcpyAsync(&h_small, d_small, sizeof(Small), cudaMemcpyDeviceToHost, st);
    const cudaError_t done = cudaStreamSynchronize(st);
    if (ce == cudaSuccess) ce = done;
    sd_device_free(queue);
    sd_device_free(d_small);
    if (ce == cudaSuccess) ce = cudaGetLastError();
    if (ce != cudaSuccess) return SD_ERR_CUDA;
    *h_entropy = h_small.wsum ? h_small.acc / (double)h_small.wsum : 0.0;
    return SD_OK;
}

// ---------------------------------------------------------------------------------------------
// sd_enumerate: every node of a tree, level by level (a node's record comes after its parent's).
namespace {

// depth 1: the nodes the root table points at
__global__ void enumerate_root_kernel(const int4* ent, const int32_t* root, int V, long long max_nodes, int32_t* parent,
                                      int32_t* token, int32_t* count, int32_t* depth, int* next_ent, int* next_rec,
                                      int* n_next, unsigned long long* n_out) {
    const int v = blockIdx.x * blockDim.x + threadIdx.x;
    if (v >= V || root[v] < 0) return;
    const int4 e = ent[root[v]];
    const unsigned long long o = atomicAdd(n_out, 1ull);
    if ((long long)o < max_nodes) { parent[o] = -1; token[o] = e.x; count[o] = e.y; depth[o] = 1; }
    if (((unsigned)e.w & RUN_COUNT_MASK) && (long long)o < max_nodes) {
        const int q = atomicAdd(n_next, 1);
        next_ent[q] = root[v]; next_rec[q] = (int)o;
    }
}

// one thread per node of the current level: a record for each of its children
__global__ void enumerate_level_kernel(const int4* ent, const int* cur_ent, const int* cur_rec, int n, int level,
                                       long long max_nodes, int32_t* parent, int32_t* token, int32_t* count, int32_t* depth,
                                       int* next_ent, int* next_rec, int* n_next, unsigned long long* n_out) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int4 e = ent[cur_ent[i]];
    const int cb = e.z, nc = (int)((unsigned)e.w & RUN_COUNT_MASK);
    const unsigned long long o0 = atomicAdd(n_out, (unsigned long long)nc);
    for (int k = 0; k < nc; ++k) {
        const int4 c = ent[cb + k];
        const long long o = (long long)o0 + k;
        if (o >= max_nodes) break;
        parent[o] = cur_rec[i]; token[o] = c.x; count[o] = c.y; depth[o] = level;
        if ((unsigned)c.w & RUN_COUNT_MASK) {
            const int q = atomicAdd(n_next, 1);
            next_ent[q] = cb + k; next_rec[q] = (int)o;
        }
    }
}

}  // namespace

extern "C" int sd_enumerate(sd_store* s, int32_t tree, int64_t max_nodes, int32_t* d_parent, int32_t* d_token,
                            int32_t* d_count, int32_t* d_depth, int64_t* h_n, void* stream) {
    if (!s || !h_n || tree < -1 || tree >= s->R || max_nodes < 0 || max_nodes > 0x7fffffffll) return SD_ERR_INVALID_ARG;
    if (max_nodes > 0 && (!d_parent || !d_token || !d_count || !d_depth)) return SD_ERR_INVALID_ARG;
    SD_CHECK_DEVICE(s);
    cudaStream_t st = (cudaStream_t)stream;
    const int4* ent = tree < 0 ? s->g_ent : s->s_ent + (long long)tree * s->spn;
    const int32_t* root = tree < 0 ? s->g_root : s->s_root + (long long)tree * s->V;
    *h_n = 0;
    const long long room = max_nodes > 0 ? max_nodes : 1;        // nodes with children among the records written
    int *fe[2] = {nullptr, nullptr}, *fr[2] = {nullptr, nullptr};
    unsigned char* small = nullptr;                              // n_out, frontier sizes
    bool okm = sd_device_malloc((void**)&small, 64) == cudaSuccess;
    for (int b = 0; b < 2 && okm; ++b)
        okm = sd_device_malloc((void**)&fe[b], sizeof(int) * (size_t)room) == cudaSuccess &&
              sd_device_malloc((void**)&fr[b], sizeof(int) * (size_t)room) == cudaSuccess;
    auto release = [&]() {
        cudaStreamSynchronize(st);
        sd_device_free(small);
        for (int b = 0; b < 2; ++b) { sd_device_free(fe[b]); sd_device_free(fr[b]); }
    };
    if (!okm) { cudaGetLastError(); release(); return SD_ERR_NOMEM; }
    unsigned long long* n_out = (unsigned long long*)small;
    int* cnt = (int*)(small + 8);                                // cnt[0], cnt[1]: frontier sizes
    cudaError_t ce = cudaMemsetAsync(small, 0, 64, st);
    enumerate_root_kernel<<<(s->V + 255) / 256, 256, 0, st>>>(ent, root, s->V, max_nodes, d_parent, d_token, d_count, d_depth,
                                                             fe[0], fr[0], cnt, n_out);
    int n = 0, cur = 0;
    if (ce == cudaSuccess) ce = cudaMemcpyAsync(&n, cnt, sizeof(int), cudaMemcpyDeviceToHost, st);
    if (ce == cudaSuccess) ce = cudaStreamSynchronize(st);
    for (int level = 2; ce == cudaSuccess && n > 0 && level <= SD_MAX_DEPTH; ++level) {
        ce = cudaMemsetAsync(cnt + (cur ^ 1), 0, sizeof(int), st);
        enumerate_level_kernel<<<(n + 255) / 256, 256, 0, st>>>(ent, fe[cur], fr[cur], n, level, max_nodes, d_parent, d_token,
                                                               d_count, d_depth, fe[cur ^ 1], fr[cur ^ 1], cnt + (cur ^ 1), n_out);
        if (ce == cudaSuccess) ce = cudaMemcpyAsync(&n, cnt + (cur ^ 1), sizeof(int), cudaMemcpyDeviceToHost, st);
        if (ce == cudaSuccess) ce = cudaStreamSynchronize(st);
        cur ^= 1;
    }
    unsigned long long total = 0;
    if (ce == cudaSuccess) ce = cudaMemcpyAsync(&total, n_out, sizeof(total), cudaMemcpyDeviceToHost, st);
    if (ce == cudaSuccess) ce = cudaStreamSynchronize(st);
    if (ce == cudaSuccess) ce = cudaGetLastError();
    release();
    if (ce != cudaSuccess) return SD_ERR_CUDA;
    *h_n = (int64_t)total;
    return (long long)total > max_nodes ? SD_ERR_CAPACITY : SD_OK;
}
