// GenerateCandidateTree (Algorithm 1) for a whole batch.
//
// sd_speculate / sd_step: ONE launch, one thread block per request (speculate_fused_kernel):
//   - sd_step: warp 0 appends the request's accepted tokens to its tree (exactly what sd_append
//     does) while the other warps look ahead for it, match and expand; the per-request match
//     nodes are the slot's active nodes, so only jobs through the request's tree wait for it;
//   - the global match nodes are advanced from the nodes cached at the previous call by
//     descending only the tokens appended since;
//   - a (tree, p) job can be taken as soon as its match node is known, costliest first, a warp per
//     job; a job is dropped, exactly, as soon as an upper bound of its SCORE falls below a score
//     already reached;
//   - select (Section 3.2: only if SCORE > tau) and emit from shared memory.
// sd_speculate_noalloc: the two-kernel form, one warp per (request, tree, p) job with the jobs'
// records in global memory (match_expand_kernel, select_emit_kernel).
//
// fp64 rules: C = count / sibling-sum (Eq. 1), D = D(parent) * C (Eq. 2), SCORE
// adds D in insertion order; __ddiv_rn / __dmul_rn / __dadd_rn keep every
// operation a separately rounded IEEE binary64 operation (no FMA contraction).
#include <mutex>

#include "append_core.cuh"
#include "device_memory.h"

namespace {

constexpr int SPEC_WARPS = 8;                 // warps per block of the job kernel
constexpr unsigned FULL = 0xffffffffu;

struct Frontier {                             // candidates of one job, best first, ring buffer
    double d[SD_MAX_SPEC];
    int tok[SD_MAX_SPEC];
    int par[SD_MAX_SPEC];
    int cb[SD_MAX_SPEC];
    unsigned nc[SD_MAX_SPEC];
};

// strict total order of candidates: larger D, then smaller token, then smaller parent index
// (D values are non-negative, so their bit patterns order like the values: branch-free compare.)
__device__ __forceinline__ bool better(double da, int ta, int pa, double db, int tb, int pb) {
    const long long a = __double_as_longlong(da), b = __double_as_longlong(db);
    return (a > b) | ((a == b) & ((ta < tb) | ((ta == tb) & (pa < pb))));
}

// Entry index of child `x` in the sorted run ent[cb .. cb+n), or -1.  Whole warp.
__device__ int find_child(const int4* __restrict__ ent, int cb, int n, int x, int lane) {
    int lo = 0, hi = n;
    for (int it = 0; it < 6 && hi - lo > 32; ++it) {       // window shrinks 33x per round
        const int q = lo + (int)(((long long)(hi - lo) * (lane + 1)) / 33);
        const int tk = ent[cb + q].x;
        const unsigned ge = __ballot_sync(FULL, tk >= x);
        const int f = ge ? __ffs(ge) - 1 : 32;              // first probe with token >= x
        const int q_prev = __shfl_sync(FULL, q, f > 0 ? f - 1 : 0);
        const int q_at = __shfl_sync(FULL, q, f < 32 ? f : 31);
        if (f > 0) lo = q_prev + 1;
        if (f < 32) hi = q_at + 1;
    }
    int found = -1;
    for (int base = lo; base < hi && found < 0; base += 32) {   // one round unless n is huge
        const int idx = base + lane;
        const bool hit = idx < hi && ent[cb + idx].x == x;
        const unsigned eq = __ballot_sync(FULL, hit);
        if (eq) found = cb + base + __ffs(eq) - 1;
    }
    return found;
}

// Insert one candidate (same values on every lane) into the sorted frontier of at
// most K entries.  fh = ring head, fs = size.
// Returns false if at least K entries are better (nothing changes then).
__device__ bool frontier_insert(Frontier& F, int fh, int& fs, int K, double d, int tok, int par, int cb, unsigned nc,
                                int lane) {
    const int i0 = lane, i1 = lane + 32;
    const int s0 = (fh + i0) & (SD_MAX_SPEC - 1), s1 = (fh + i1) & (SD_MAX_SPEC - 1);
    const bool b0 = i0 < fs && better(F.d[s0], F.tok[s0], F.par[s0], d, tok, par);
    const bool b1 = i1 < fs && better(F.d[s1], F.tok[s1], F.par[s1], d, tok, par);
    const int pos = __popc(__ballot_sync(FULL, b0)) + __popc(__ballot_sync(FULL, b1));
    if (pos >= K) return false;
    const int ns = min(fs + 1, K);
    double md0 = 0, md1 = 0; int mt0 = 0, mt1 = 0, mp0 = 0, mp1 = 0, mc0 = 0, mc1 = 0; unsigned mn0 = 0, mn1 = 0;
    const bool mv0 = i0 > pos && i0 < ns, mv1 = i1 > pos && i1 < ns;
    if (mv0) { const int q = (s0 - 1) & (SD_MAX_SPEC - 1); md0 = F.d[q]; mt0 = F.tok[q]; mp0 = F.par[q]; mc0 = F.cb[q]; mn0 = F.nc[q]; }
    if (mv1) { const int q = (s1 - 1) & (SD_MAX_SPEC - 1); md1 = F.d[q]; mt1 = F.tok[q]; mp1 = F.par[q]; mc1 = F.cb[q]; mn1 = F.nc[q]; }
    __syncwarp();
    if (mv0) { F.d[s0] = md0; F.tok[s0] = mt0; F.par[s0] = mp0; F.cb[s0] = mc0; F.nc[s0] = mn0; }
    if (mv1) { F.d[s1] = md1; F.tok[s1] = mt1; F.par[s1] = mp1; F.cb[s1] = mc1; F.nc[s1] = mn1; }
    if (i0 == pos) { F.d[s0] = d; F.tok[s0] = tok; F.par[s0] = par; F.cb[s0] = cb; F.nc[s0] = nc; }
    if (i1 == pos) { F.d[s1] = d; F.tok[s1] = tok; F.par[s1] = par; F.cb[s1] = cb; F.nc[s1] = nc; }
    __syncwarp();
    fs = ns;
    return true;
}

// Offer every child of a node (run ent[cb .. cb+n)) to the frontier.
__device__ void push_children(const int4* __restrict__ ent, int cb, int n, double d_parent, int par_index, Frontier& F,
                              int fh, int& fs, int K, int lane) {
    if (n <= 0 || K <= 0) return;
    long long sum = 0;
    int4 first = make_int4(0, 0, 0, 0);
    for (int base = 0; base < n; base += 32) {
        const int idx = base + lane;
        int4 e = make_int4(0, 0, 0, 0);
        if (idx < n) e = ent[cb + idx];
        if (base == 0) first = e;
        sum += e.y;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(FULL, sum, o);
    const double dsum = (double)sum;                            // denominator of Eq. 1
    for (int base = 0; base < n; base += 32) {
        const int idx = base + lane;
        const bool v = idx < n;
        int4 e = first;
        if (base != 0) { e = make_int4(0, 0, 0, 0); if (v) e = ent[cb + idx]; }
        double dc = 0.0;
        if (v) dc = __dmul_rn(d_parent, __ddiv_rn((double)e.y, dsum));   // Eq. 2 with Eq. 1
        bool pass = v;
        if (v && fs == K) {                                     // cannot beat the current worst: skip
            const int last = (fh + fs - 1) & (SD_MAX_SPEC - 1);
            pass = better(dc, e.x, par_index, F.d[last], F.tok[last], F.par[last]);
        }
        unsigned m = __ballot_sync(FULL, pass);
        while (m) {
            const int src = __ffs(m) - 1;
            m &= m - 1;
            const double cd = __shfl_sync(FULL, dc, src);
            const int ct = __shfl_sync(FULL, e.x, src);
            const int cc = __shfl_sync(FULL, e.z, src);
            const unsigned cn = (unsigned)__shfl_sync(FULL, e.w, src);
            frontier_insert(F, fh, fs, K, cd, ct, par_index, cc, cn, lane);
        }
    }
}

// ExpandSpeculationTree below the node with child run [cb, cb + n) as Algorithm 1 states it, one node
// after the other: tokens and parents of the draft in insertion order, SCORE in `score`.  Whole warp.
__device__ __noinline__ int expand_serial(const int4* __restrict__ ent, int cb0, int n0, int budget, unsigned flags, Frontier& F,
                                          int32_t* out_tok, int32_t* out_par, double& score, int lane) {
    int fh = 0, fs = 0, cnt = 0;
    score = 0.0;
    push_children(ent, cb0, n0, 1.0, -1, F, fh, fs, budget, lane);
    while (cnt < budget && fs > 0) {
        const double d = F.d[fh];
        const int tok = F.tok[fh], par = F.par[fh], cb = F.cb[fh];
        const int nc = (int)(F.nc[fh] & RUN_COUNT_MASK);
        __syncwarp();
        fh = (fh + 1) & (SD_MAX_SPEC - 1);
        --fs;
        if (lane == 0) { out_tok[cnt] = tok; out_par[cnt] = par; }
        score = __dadd_rn(score, d);                            // Eq. 4, insertion order
        const int idx = cnt++;
        const int K = budget - cnt;
        if (fs > K) fs = K;
        if (flags & SD_FLAG_LINEAR) fs = 0;
        push_children(ent, cb, nc, d, idx, F, fh, fs, K, lane);
    }
    __syncwarp();
    return cnt;
}

__device__ __forceinline__ int budget_for(double alpha, int p, int cap) {
    const double b = floor(__dmul_rn(alpha, (double)p));        // Eq. 3
    if (b > (double)cap) return cap;
    if (b < 0.0) return 0;
    return (int)b;
}

__global__ void __launch_bounds__(SPEC_WARPS * 32)
match_expand_kernel(sd_store sv, int n, const int32_t* __restrict__ d_slot, int Pe, double alpha, int max_spec,
                    unsigned flags, const int32_t* __restrict__ d_budget_cap) {
    __shared__ Frontier fr[SPEC_WARPS];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const long long job = (long long)blockIdx.x * SPEC_WARPS + wib;
    if (job >= (long long)n * 2 * Pe) return;
    const int i = (int)(job / (2 * Pe));
    const int rem = (int)(job % (2 * Pe));
    const int tree = rem / Pe, p = rem % Pe + 1;
    const long long rec = ((long long)i * 2 + tree) * sv.D + (p - 1);
    int cnt = 0;
    double score = 0.0;
    const int slot = d_slot[i];
    bool live = slot >= 0 && slot < sv.R;
    if (tree == 0 && (flags & SD_FLAG_REQUEST_ONLY)) live = false;
    if (tree == 1 && (flags & SD_FLAG_GLOBAL_ONLY)) live = false;
    if (live) {
        const SlotState* ss = sv.s_state + slot;
        const int t = ss->len;
        if (ss->status & (SD_STATUS_POOL_FULL | SD_STATUS_BAD_TOKEN)) live = false;
        if (p > t) live = false;
        int cap = max_spec;
        if (d_budget_cap && d_budget_cap[i] >= 0) cap = min(cap, d_budget_cap[i]);
        const int budget = budget_for(alpha, p, cap);
        if (live && budget > 0) {
            // ---- MatchPattern
            const int4* ent;
            int node;
            if (tree == 1) {
                ent = sv.s_ent + (long long)slot * sv.spn;
                node = ss->active[p - 1];                       // node of the last p tokens
            } else {
                ent = sv.g_ent;
                const int32_t* pat = sv.s_text + (long long)slot * sv.T + (t - p);
                node = sv.g_root[pat[0]];
                for (int k = 1; k < p && node >= 0; ++k) {
                    const int4 e = ent[node];
                    node = find_child(ent, e.z, (int)((unsigned)e.w & RUN_COUNT_MASK), pat[k], lane);
                }
            }
            if (node >= 0) {
                // ---- ExpandSpeculationTree
                const int4 e = ent[node];
                cnt = expand_serial(ent, e.z, (int)((unsigned)e.w & RUN_COUNT_MASK), budget, flags, fr[wib], sv.j_tok + rec * sv.M,
                                    sv.j_par + rec * sv.M, score, lane);
            }
        }
    }
    if (lane == 0) { sv.j_n[rec] = cnt; sv.j_score[rec] = score; }
}

__global__ void select_emit_kernel(sd_store sv, int n, const int32_t* __restrict__ d_slot, int Pe, double tau, int32_t* d_n_draft,
                                   int32_t* d_tokens, int32_t* d_parents, int32_t* d_positions, uint32_t* d_mask,
                                   int32_t* d_chosen_tree, int32_t* d_chosen_p, double* d_score, int32_t* d_status) {
    __shared__ int spar[4][SD_MAX_SPEC];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const int i = blockIdx.x * 4 + wib;
    if (i >= n) return;
    const int M = sv.M, words = (M + 31) / 32;
    const int slot = d_slot[i];
    const bool ok = slot >= 0 && slot < sv.R;
    // first job in loop order (global before per-request, p ascending) with the largest score
    double best = 0.0;
    int best_o = -1;
    for (int o = lane; o < 2 * Pe; o += 32) {
        const long long rec = ((long long)i * 2 + o / Pe) * sv.D + (o % Pe);
        const double sc = sv.j_score[rec];
        if (sc > best) { best = sc; best_o = o; }               // ascending o: strict '>' keeps the first
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        const double ob = __shfl_xor_sync(FULL, best, off);
        const int oo = __shfl_xor_sync(FULL, best_o, off);
        if (oo >= 0 && (ob > best || (ob == best && (best_o < 0 || oo < best_o)))) { best = ob; best_o = oo; }
    }
    int nd = 0, tree = -1, p = 0, t = 0, status = SD_STATUS_BAD_SLOT;
    long long rec = 0;
    if (ok) {
        t = sv.s_state[slot].len;
        status = sv.s_state[slot].status;
    }
    if (ok && best_o >= 0 && best > tau) {                      // Section 3.2: only a score above the threshold is used
        tree = best_o / Pe; p = best_o % Pe + 1;
        rec = ((long long)i * 2 + tree) * sv.D + (p - 1);
        nd = sv.j_n[rec];
    } else {
        best = 0.0;
    }
    for (int j = lane; j < SD_MAX_SPEC; j += 32) spar[wib][j] = j < nd ? sv.j_par[rec * M + j] : -1;
    __syncwarp();
    for (int j = lane; j < M; j += 32) {
        int tok = -1, par = -1, pos = -1;
        unsigned long long bits = 0;
        if (j < nd) {
            tok = sv.j_tok[rec * M + j];
            par = spar[wib][j];
            int depth = 0;
            for (int a = j, hops = 0; a >= 0 && hops < SD_MAX_SPEC; a = spar[wib][a], ++hops) {
                bits |= 1ull << a;
                ++depth;
            }
            pos = t + depth - 1;
        }
        const long long o = (long long)i * M + j;
        d_tokens[o] = tok; d_parents[o] = par; d_positions[o] = pos;
        d_mask[o * words] = (uint32_t)bits;
        if (words > 1) d_mask[o * words + 1] = (uint32_t)(bits >> 32);
    }
    if (lane == 0) {
        d_n_draft[i] = nd; d_chosen_tree[i] = tree; d_chosen_p[i] = p; d_score[i] = best;
        if (d_status) d_status[i] = status;
    }
}


// ---------------------------------------------------------------------------------------------
// Fused path: one block of W warps per request (the kernel itself is described where it is
// defined).  Two blocks per SM is the usual shape.  A batch of at most one request per SM gets blocks with
// more registers, a batch of more than two requests per SM smaller ones (four per SM) to stay in one wave.
// (The usual block's size was taken when candidates lay in shared memory: drafts of 256 requests 44.2 us with 14 warps, 51.5 / 52.1 / 45.6 /
// 48.9 / 49.3 with 10 / 12 / 13 / 15 / 16; steps 58.6, with 8 / 10 / 12 / 16 63.1 / 60.1 / 59.2 / 58.6.  It has not been swept since.)
constexpr int CTA_WARPS = 14;
constexpr int CTA_WARPS_STEP = 14;             // of sd_step
// one block per SM at most, 128 registers per thread: nothing is spilled.  Drafts of 64 requests with long runs 95 us (24 warps of 80
// registers 107, 20 106, 12 108), of one request 7.3 (8.0, 7.6, 7.1); steps of 64 requests 47.4 (12 warps 49.2, 20 48.7)
constexpr int CTA_WARPS_WIDE = 16;
constexpr int CTA_WARPS_NARROW = 8;            // batches of more than two requests per SM: four blocks per SM
constexpr int CTA_WARPS_NARROW_STEP = 4;       // (sd_step: 128 registers; with 5 warps of 96 a decode of 512 requests takes 1,925 us, 1,870 now)

// Candidates of one job: not ordered, two per lane in registers.  The next node is the one with the largest D, which a
// reduction over the lanes tells; its children go to lanes with a free place, a child each, so nothing is sorted, moved or
// looked up in memory per node.
// A job is a chain of nodes (30 - 44 of them in the slowest jobs of 256 requests), each a dependent read of its children and about 130
// instructions at 6 - 9 cycles; with two blocks on an SM the busiest SMs also run out of issue slots.  (Candidates in shared
// memory, the children read as windows of 32 entries kept in registers, and a division per node: 45.3 us for a draft of 256
// requests, 43.1 now; 43.6 -> 38.5 on other text; steps 55 -> 51.  The request of a candidate's children into L2 as it is found
// is worth 1 - 2 % of that; requests into L1, or by cp.async, lost as much.  Telling the others the running SCORE one node
// later cost 3 %.)  Slower where branches of few children follow one another all the way (text that copies 19 of 20 spans, of 100
// tokens each): drafts of 8 / 64 / 256 requests 34 / 38 / 46 -> 39 / 41 / 50; windows there, too, or asking for the children as soon
// as the node is known brought nothing back with a warm L2.
struct Cand {
    unsigned hi, lo;                          // D; 0: a free place
    int tok, cb;
    unsigned np;                              // children | RUN_HAS_TOP | parent index + 1 from bit 24 on (the last node of 64 is nobody's parent)
};
constexpr unsigned CAND_RUN = RUN_COUNT_MASK | RUN_HAS_TOP;
constexpr int CAND_PAR = 24;
constexpr int POOL = 96;                      // what two places per lane hold and one node's children
struct Pool {                                 // to make room (pool_compact)
    double d[POOL];
    int tok[POOL];
    int cb[POOL];
    unsigned np[POOL];
};

// Eq. 1 for sums up to RECIP_MAX: the quotient from the correctly rounded reciprocal (Markstein, "Computation of elementary
// functions on the IBM RISC System/6000 processor", 1990, theorem 8: q = RN(a r), then RN(q + r RN(a - b q)) is RN(a / b)).  Three
// instructions in a row instead of some 30.  The reciprocals are divided by the compiler, in IEEE binary64.
constexpr int RECIP_MAX = 511;
struct __align__(16) RecipTable {
    double r[RECIP_MAX + 1];
    constexpr RecipTable() : r() {
        for (int b = 1; b <= RECIP_MAX; ++b) r[b] = 1.0 / (double)b;
    }
};
__device__ const RecipTable g_recip;

__device__ __forceinline__ double quotient(double a, double b, double r) {
    const double q = __dmul_rn(a, r);
    return __fma_rn(r, __fma_rn(-b, q, a), q);
}

struct __align__(16) WarpWork {
    Pool C;
    Frontier T;                               // children of a wide node, by count (F of a wide match node's slices)
    int one_tok[SD_MAX_SPEC];                 // its first children of count 1, in token order
    int one_cb[SD_MAX_SPEC];
    unsigned one_nc[SD_MAX_SPEC];
    int tok[2][SD_MAX_SPEC];                  // draft tokens: working buffer and best-so-far buffer
    unsigned char par[2][SD_MAX_SPEC];        // parent index + 1 (0: child of the match node)
    double best_score;
    int best_order, best_n, best_buf;
};

template <int WARPS>
struct BlockSharedT {
    WarpWork w[WARPS];
    RecipTable recip;
    int node[2][SD_MAX_DEPTH];                // match node per tree and pattern length (-1: none)
    int cb[2][SD_MAX_DEPTH];                  // its child run
    unsigned nc[2][SD_MAX_DEPTH];             // ... as the node's w field (count | flags)
    unsigned char ordp[SD_MAX_DEPTH];         // pattern lengths - 1 by the number of nodes their jobs can add at most
    int wide[2 * SD_MAX_DEPTH];               // jobs whose match node has a wide child run
    int nwide, nwide_kept;
    // per tree: jobs to be taken, a bit per place in ordp; warps whose match nodes are still to come; the request's are
    struct __align__(16) { unsigned ready[2]; int walking, appending; } board;
    int gave_up;                              // a warp waited too long for them
    int at_hand;                              // all of them are known from the call before
    long long slice_sum[WARPS];
    int slice_fs[WARPS];
    AppendShared app;
    int src_node[SD_MAX_DEPTH];               // where the walk to a global match node starts: node (-1: nowhere) ...
    int src_from[SD_MAX_DEPTH];               // ... and the first token to take
    unsigned best_hi;                         // high word of the largest SCORE reached so far: a lower
                                              // bound of it (scores are non-negative doubles), which is
                                              // all the pruning needs; 32 bits keep the atomic native
    unsigned long long anc[SD_MAX_SPEC];      // ancestors of the chosen tree's nodes
    signed char up[SD_MAX_SPEC];
};

__device__ __forceinline__ void prefetch_l2(const void* p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); }

// Start fetching the `n` entries at ent[cb ...] into L2 (whole warp; at most `max_lines` 128-byte lines per lane).
__device__ __forceinline__ void prefetch_run(const int4* __restrict__ ent, int cb, int n, int lane, int max_rounds) {
    const int lines = (n + 7) >> 3;
    for (int r = 0, l = lane; r < max_rounds && l < lines; ++r, l += 32) prefetch_l2(ent + cb + l * 8);
}

// Merge up to 32 candidates (one per lane with `pass`) into the sorted frontier of at most K
// entries in one go: every survivor's final position is its number of betters, found by
// broadcasting the candidates once; then all entries move together.
__device__ void frontier_merge(Frontier& F, int fh, int& fs, int K, bool pass, double d, int tok, int par, int cb,
                               unsigned nc, int lane) {
    const unsigned m = __ballot_sync(FULL, pass);
    if (!m) return;
    const int i0 = lane, i1 = lane + 32;
    const int s0 = (fh + i0) & (SD_MAX_SPEC - 1), s1 = (fh + i1) & (SD_MAX_SPEC - 1);
    const bool v0 = i0 < fs, v1 = i1 < fs;
    double e0d = 0.0, e1d = 0.0;
    int e0t = 0, e1t = 0, e0p = 0, e1p = 0;
    if (v0) { e0d = F.d[s0]; e0t = F.tok[s0]; e0p = F.par[s0]; }
    if (v1) { e1d = F.d[s1]; e1t = F.tok[s1]; e1p = F.par[s1]; }
    int up0 = 0, up1 = 0;                                       // candidates that go before E[i0], E[i1]
    int my_rank = 0;
    unsigned mm = m;
    while (mm) {
        const int src = __ffs(mm) - 1;
        mm &= mm - 1;
        const double bd = __shfl_sync(FULL, d, src);
        const int bt = __shfl_sync(FULL, tok, src), bp = __shfl_sync(FULL, par, src);
        const bool b0 = v0 && better(bd, bt, bp, e0d, e0t, e0p);
        const bool b1 = v1 && better(bd, bt, bp, e1d, e1t, e1p);
        up0 += b0 ? 1 : 0;
        up1 += b1 ? 1 : 0;
        const int worse_old = __popc(__ballot_sync(FULL, b0)) + __popc(__ballot_sync(FULL, b1));
        const int better_new = __popc(__ballot_sync(FULL, pass && lane != src && better(d, tok, par, bd, bt, bp)));
        if (lane == src) my_rank = (fs - worse_old) + better_new;
    }
    const int n0 = i0 + up0, n1 = i1 + up1;
    int c0 = 0, c1 = 0;
    unsigned w0 = 0, w1 = 0;
    const bool k0 = v0 && n0 < K && up0 > 0, k1 = v1 && n1 < K && up1 > 0;   // entries that move
    if (k0) { c0 = F.cb[s0]; w0 = F.nc[s0]; }
    if (k1) { c1 = F.cb[s1]; w1 = F.nc[s1]; }
    __syncwarp();
    if (k0) { const int q = (fh + n0) & (SD_MAX_SPEC - 1); F.d[q] = e0d; F.tok[q] = e0t; F.par[q] = e0p; F.cb[q] = c0; F.nc[q] = w0; }
    if (k1) { const int q = (fh + n1) & (SD_MAX_SPEC - 1); F.d[q] = e1d; F.tok[q] = e1t; F.par[q] = e1p; F.cb[q] = c1; F.nc[q] = w1; }
    if (pass && my_rank < K) {
        const int q = (fh + my_rank) & (SD_MAX_SPEC - 1);
        F.d[q] = d; F.tok[q] = tok; F.par[q] = par; F.cb[q] = cb; F.nc[q] = nc;
    }
    __syncwarp();
    fs = min(fs + __popc(m), K);
}

// Offer the first `cnt` entries of list O (ordered, ring head 0) to F.
__device__ void frontier_merge_list(Frontier& F, int fh, int& fs, int K, const Frontier& O, int cnt, int par, int lane) {
    for (int base = 0; base < cnt; base += 32) {
        const int q = base + lane;
        bool pass = q < cnt;
        double d = 0.0; int tok = 0, cb = 0; unsigned nc = 0;
        if (pass) { d = O.d[q]; tok = O.tok[q]; cb = O.cb[q]; nc = O.nc[q]; }
        if (pass && fs == K) {
            const int last = (fh + fs - 1) & (SD_MAX_SPEC - 1);
            pass = better(d, tok, par, F.d[last], F.tok[last], F.par[last]);
        }
        if (!__any_sync(FULL, pass)) break;                     // O is ordered: nothing further can enter
        frontier_merge(F, fh, fs, K, pass, d, tok, par, cb, nc, lane);
    }
}

// A WINDOW is 32 consecutive entries, one per lane, starting at `base`.  Trees are laid out so
// that the child run of a node's first (often only) child tends to follow the node's own
// child run, so one window usually holds several levels of a path at once.
__device__ __forceinline__ int4 load_window(const int4* __restrict__ ent, int base, int limit, int lane) {
    const int idx = base + lane;
    // the entries behind the window hold the rest of the node's sub-tree (pre-order layout):
    // bring the next 1.5 KB into L2 so that the following windows of this job hit there
    if (lane < 12 && base + 32 + lane * 8 < limit)
        asm volatile("prefetch.global.L2 [%0];" ::"l"(ent + base + 32 + lane * 8));
    return idx < limit ? ent[idx] : make_int4(-1, 0, 0, 0);
}

constexpr int WIDE_RUN = 256;                 // child runs longer than this are scanned by several warps

// One pass over chunks first, first + stride, ... of a child run: adds up the counts and keeps
// the K children with the largest counts (then smallest tokens) in F, ordered, with the COUNT
// in the d field.  Among the children of one parent that is the order of D (Eq. 2), so no
// division is needed while scanning.  F starts empty at ring head fh.
// Most children of a wide node occur once.  Those tie on the count and rank by token, i.e. in
// run order: the first K of them are simply copied (ones list) and appended behind the
// children that occur more often, which alone go through the ordered merge.
// Children with a count below `cmin` are known not to matter and are skipped.
__device__ void scan_run_by_count(const int4* __restrict__ ent, int cb, int n, int first, int stride, int par_index,
                                  int cmin, WarpWork& W, Frontier& F, int fh, int& fs, int K, long long& sum_out,
                                  int lane) {
    long long sum = 0;
    fs = 0;
    int ones = 0;                                               // count-1 children copied so far (warp-uniform)
    if (stride == 1) prefetch_run(ent, cb, n, lane, 64);        // the whole run, all lines in flight at once
    for (int c = first; c * 32 < n; c += 4 * stride) {
        int4 e[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {                           // four loads in flight
            const int idx = (c + u * stride) * 32 + lane;
            e[u] = make_int4(-1, 0, 0, 0);
            if (idx < n) e[u] = ent[cb + idx];
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            sum += e[u].y;
            const unsigned m1 = __ballot_sync(FULL, e[u].y == 1 && cmin <= 1);
            if (m1 && ones < K) {
                const int at = ones + __popc(m1 & ((1u << lane) - 1u));
                if (e[u].y == 1 && at < K) { W.one_tok[at] = e[u].x; W.one_cb[at] = e[u].z; W.one_nc[at] = (unsigned)e[u].w; }
                ones = min(K, ones + __popc(m1));
            }
            bool pass = e[u].y >= 2 && e[u].y >= cmin;
            if (pass && fs == K) {
                const int last = (fh + fs - 1) & (SD_MAX_SPEC - 1);
                pass = better((double)e[u].y, e[u].x, par_index, F.d[last], F.tok[last], F.par[last]);
            }
            if (pass && ((unsigned)e[u].w & RUN_COUNT_MASK)) prefetch_l2(ent + e[u].z);
            frontier_merge(F, fh, fs, K, pass, (double)e[u].y, e[u].x, par_index, e[u].z, (unsigned)e[u].w, lane);
        }
    }
    __syncwarp();
    // the count-1 children go behind the others, in token order, as far as there is room
    const int take = min(ones, K - fs);
    for (int i = lane; i < take; i += 32) {
        const int q = (fh + fs + i) & (SD_MAX_SPEC - 1);
        F.d[q] = 1.0; F.tok[q] = W.one_tok[i]; F.par[q] = par_index; F.cb[q] = W.one_cb[i]; F.nc[q] = W.one_nc[i];
    }
    fs += take;
    __syncwarp();
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(FULL, sum, o);
    sum_out = sum;
}

// counts in F.d -> D = d_parent * count / sum (Eq. 1, Eq. 2)
__device__ void counts_to_d(Frontier& F, int fh, int fs, double d_parent, long long sum, int lane) {
    const double dsum = (double)sum;
    for (int i = lane; i < fs; i += 32) {
        const int q = (fh + i) & (SD_MAX_SPEC - 1);
        F.d[q] = __dmul_rn(d_parent, __ddiv_rn(F.d[q], dsum));
    }
    __syncwarp();
}

// Leaves the `room` best of the n candidates in C (what is worse than that many others cannot be taken any more), some more
// where that is less work, but never more than 64.  Returns how many; `floor` becomes the high word of the least D that matters.
__device__ __noinline__ int pool_compact(Pool& C, int n, int room, unsigned& floor, int lane) {
    unsigned h[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) h[c] = c * 32 + lane < n ? (unsigned)__double2hiint(C.d[c * 32 + lane]) : 0u;
    unsigned lo = 1u, hi = __reduce_max_sync(FULL, max(max(h[0], h[1]), h[2]));
    int at_lo = n;                                              // the largest limit with at least `room` candidates at or above it
    for (int it = 0; it < 32 && lo < hi && (at_lo > room + 8 || at_lo > 64); ++it) {
        const unsigned mid = lo + (hi - lo + 1u) / 2u;
        int k = 0;
#pragma unroll
        for (int c = 0; c < 3; ++c) k += __popc(__ballot_sync(FULL, h[c] >= mid));
        if (k >= room) { lo = mid; at_lo = k; } else hi = mid - 1u;
    }
    Cand v[3];
    int to[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const int i = c * 32 + lane;
        to[c] = -1;
        if (h[c] < lo) continue;
        v[c] = Cand{h[c], (unsigned)__double2loint(C.d[i]), C.tok[i], C.cb[i], C.np[i]};
    }
    int k = 0;
    if (at_lo <= 64) {
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const unsigned m = __ballot_sync(FULL, h[c] >= lo);
            if (h[c] >= lo) to[c] = k + __popc(m & ((1u << lane) - 1u));
            k += __popc(m);
        }
    } else {
        // many of equal D: by token and parent then, too
        int rank[3] = {0, 0, 0};
        for (int q = 0; q < n; ++q) {
            const double d = C.d[q];
            const int tok = C.tok[q], par = (int)(C.np[q] >> CAND_PAR) & 63;
#pragma unroll
            for (int c = 0; c < 3; ++c)
                if (h[c] >= lo) rank[c] += better(d, tok, par, __hiloint2double((int)v[c].hi, (int)v[c].lo), v[c].tok, (int)(v[c].np >> CAND_PAR) & 63) ? 1 : 0;
        }
        k = room;
#pragma unroll
        for (int c = 0; c < 3; ++c) if (h[c] >= lo && rank[c] < room) to[c] = rank[c];
    }
    __syncwarp();
#pragma unroll
    for (int c = 0; c < 3; ++c)
        if (to[c] >= 0) { C.d[to[c]] = __hiloint2double((int)v[c].hi, (int)v[c].lo); C.tok[to[c]] = v[c].tok; C.cb[to[c]] = v[c].cb; C.np[to[c]] = v[c].np; }
    __syncwarp();
    if (at_lo >= room) floor = max(floor, lo);
    return k;
}

// The best children (by count, then smallest token; at most `room`) of a node with more than 32: their entries in `list`, where `room` are
// found the last one is the least of them.  They are taken from registers: all of a run of up to 128 children, else those that occur
// often (up to 128 of them; most children of a long run occur once or twice), and only what is left from the run itself, there
// one class of equal counts after the other.  `hot`: 256 words of the warp's.
// Text in which one token is every second one is bound by this: 17 runs of 33 to 128 children in the slowest jobs, with 20 places left on
// average.  Listed from registers class by class (2,900 to 5,000 cycles a run, a ballot chain per class) drafts of 64 requests took
// 98.6 us; with the least count found by halves 94.6; with that search begun at 2 and ended at sum / room, the most it can be, 80.7 (1,050
// to 1,500 cycles).  Every class by a pass over the run took 125.
__device__ __noinline__ int list_by_count(const int4* __restrict__ ent, int cb, int n, int room, int* list, int* hot, unsigned& sum_out,
                                          int lane) {
    unsigned y[4], least = 1u;                                  // counts from `least` on are in the registers
    int pos[4];
    if (n <= 128) {
        unsigned sum = 0;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            pos[u] = u * 32 + lane;
            y[u] = pos[u] < n ? (unsigned)ent[cb + pos[u]].y : 0u;
            sum += y[u];                                        // (a parent's occurrences fit 31 bits)
        }
        sum_out = __reduce_add_sync(FULL, sum);
    } else {
        constexpr int LIMITS = 8;                               // 2, 3, 5, 9, .. 129
        unsigned sum = 0, many[LIMITS] = {};
        for (int base = lane; base < n; base += 128) {
            unsigned v[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) v[u] = base + u * 32 < n ? (unsigned)ent[cb + base + u * 32].y : 0u;
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                sum += v[u];
#pragma unroll
                for (int k = 0; k < LIMITS; ++k) many[k] += v[u] > (1u << k) ? 1u : 0u;
            }
        }
        sum_out = __reduce_add_sync(FULL, sum);
        least = 0u;
#pragma unroll
        for (int k = LIMITS - 1; k >= 0; --k) if (__reduce_add_sync(FULL, many[k]) <= 128u) least = (1u << k) + 1u;
        int got = 0;
        if (least > 0u) {
            for (int base = 0; base < n; base += 128) {
                unsigned v[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) v[u] = base + u * 32 + lane < n ? (unsigned)ent[cb + base + u * 32 + lane].y : 0u;
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const unsigned m = __ballot_sync(FULL, v[u] >= least);
                    const int at = got + __popc(m & ((1u << lane) - 1u));
                    if (v[u] >= least) { hot[2 * at] = base + u * 32 + lane; hot[2 * at + 1] = (int)v[u]; }
                    got += __popc(m);
                }
            }
            __syncwarp();
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const bool in = u * 32 + lane < got;
            pos[u] = in ? hot[2 * (u * 32 + lane)] : 0;
            y[u] = in ? (unsigned)hot[2 * (u * 32 + lane) + 1] : 0u;
        }
    }
    // what they hold: those that occur more often than the last one that there is room for, then as many that occur as often, in run order.
    // `room` of them that occur `cut` times make up room * cut of the sum at least.
    unsigned cut = 1u, top = min(__reduce_max_sync(FULL, max(max(y[0], y[1]), max(y[2], y[3]))), sum_out / (unsigned)room);
    while (cut < top) {
        const unsigned mid = min(2u * cut, cut + (top - cut + 1u) / 2u);
        unsigned k = 0;
#pragma unroll
        for (int u = 0; u < 4; ++u) k += y[u] >= mid ? 1u : 0u;
        k = __reduce_add_sync(FULL, k);
        if (k >= (unsigned)room) cut = mid; else top = mid - 1u;
        if (k == (unsigned)room) {                              // these are they
            unsigned fewest = 0xffffffffu;
#pragma unroll
            for (int u = 0; u < 4; ++u) if (y[u] >= mid) fewest = min(fewest, y[u]);
            cut = __reduce_min_sync(FULL, fewest);
            break;
        }
    }
    int taken = 0;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const unsigned m = __ballot_sync(FULL, y[u] > cut);
        if (y[u] > cut) list[taken + __popc(m & ((1u << lane) - 1u))] = cb + pos[u];
        taken += __popc(m);
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const unsigned m = __ballot_sync(FULL, y[u] == cut);
        const int at = taken + __popc(m & ((1u << lane) - 1u));
        if (y[u] == cut && at < room) list[at] = cb + pos[u];
        taken += __popc(m);
    }
    // what the registers do not hold (least 0: nothing is in them)
    top = least - 1u;
    while (top > 0u && taken < room) {
        unsigned next = 0;
        for (int base = 0; base < n && taken < room; base += 128) {
            unsigned v[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) v[u] = base + u * 32 + lane < n ? (unsigned)ent[cb + base + u * 32 + lane].y : 0u;
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const unsigned m = __ballot_sync(FULL, v[u] == top);
                const int at = taken + __popc(m & ((1u << lane) - 1u));
                if (v[u] == top && at < room) list[at] = cb + base + u * 32 + lane;
                taken += __popc(m);
                if (v[u] < top) next = max(next, v[u]);
            }
        }
        top = __reduce_max_sync(FULL, next);
    }
    __syncwarp();
    return min(taken, room);
}

// ExpandSpeculationTree + SCORE for one (tree, p) job by one warp.  nseed >= 0: the match node's best
// children are in W.T (nseed of them, from ring head 0, with their D).
// ROOMY: candidates that find no lane of their own kind free go into free places of either kind before room is made, through shared memory.
// On text with long runs at many depths 42 of 54 compactions a request are not needed then (drafts of 64 requests 102.5 -> 98.6 us).
// Where blocks share an SM the registers that it takes are spilled: drafts of 256 requests 4.5 % longer.
template <bool ROOMY, class BlockShared>
__device__ __noinline__ void expand_job(BlockShared& sh, WarpWork& W, const int4* __restrict__ ent, int limit, int tree, int p,
                           int budget, unsigned flags, int nseed, int lane) {
    const int order = tree * SD_MAX_DEPTH + p;                  // loop order of Algorithm 1
    const int buf = W.best_buf ^ 1;
    const unsigned lt = (1u << lane) - 1u;
    Cand c0{0u, 0u, 0, 0, 0u}, c1{0u, 0u, 0, 0, 0u};
    unsigned floor = 1u;                                        // candidates whose D has a smaller high word do not matter
    int cnt = 0;
    double score = 0.0, left = (double)budget;                  // left: nodes that can still be added
    bool dropped = false;
    // the node whose children are to be offered next: the match node first, D(N_p) = 1
    double cur_d = 1.0;
    int cur_cb = sh.cb[tree][p - 1], cur_idx = -1;
    unsigned cur_w = sh.nc[tree][p - 1];
    bool have_cur = nseed < 0;
    if (!have_cur) {
        auto seed = [&](int q) {
            return q < nseed ? Cand{(unsigned)__double2hiint(W.T.d[q]), (unsigned)__double2loint(W.T.d[q]), W.T.tok[q], W.T.cb[q], W.T.nc[q] & CAND_RUN}
                             : Cand{0u, 0u, 0, 0, 0u};
        };
        c0 = seed(lane); c1 = seed(32 + lane);
    }
    // What is still to come is at most d each: is SCORE at most (with a margin) below one already reached?  (Any lane that
    // has seen one counts.)  The final SCORE is at least its running value: the others prune on that.
    unsigned best = 0u;
    auto hopeless = [&](double d) {
        best = *(volatile unsigned*)&sh.best_hi;
        return __any_sync(FULL, (unsigned)__double2hiint(__fma_rn(left, d, score) * 1.000000001) < best) != 0;
    };
    auto publish = [&]() { if (lane == 0 && (unsigned)__double2hiint(score) > best) atomicMax(&sh.best_hi, (unsigned)__double2hiint(score)); };
    while (true) {
        if (have_cur) {
            // ---------------- the children of `cur` become candidates
            have_cur = false;
            const int cur_n = (int)(cur_w & RUN_COUNT_MASK);
            if (cur_n == 1) {
                const unsigned top = __reduce_max_sync(FULL, max(c0.hi, c1.hi));
                if (top < (unsigned)__double2hiint(cur_d)) {
                    // An only child has C = 1, so D stays cur_d: while the best waiting candidate is
                    // strictly worse, the whole chain of only children is added in one go.
                    const int4 w = load_window(ent, cur_cb, limit, lane);
                    const bool link = cur_cb + lane < limit && ((unsigned)w.w & RUN_COUNT_MASK) == 1u && w.z == cur_cb + lane + 1;
                    const unsigned links = __ballot_sync(FULL, link);
                    const int len = min(min(32, limit - cur_cb), 1 + (links == 0xffffffffu ? 32 : __ffs(~links) - 1));
                    const int m = min(len, budget - cnt);
                    if (lane < m) {
                        W.tok[buf][cnt + lane] = w.x;
                        W.par[buf][cnt + lane] = (unsigned char)((lane == 0 ? cur_idx : cnt + lane - 1) + 1);
                    }
                    for (int q = 0; q < m; ++q) score = __dadd_rn(score, cur_d);
                    publish();
                    cnt += m;
                    left -= (double)m;
                    cur_idx = cnt - 1;
                    cur_cb = __shfl_sync(FULL, w.z, m - 1);
                    cur_w = (unsigned)__shfl_sync(FULL, w.w, m - 1);
                    if (cnt >= budget) break;
                    if (hopeless(cur_d)) { dropped = true; break; }
                    have_cur = true;
                    continue;
                }
            }
            if (cur_n > 0) {
                const unsigned par = (unsigned)(cur_idx + 1) << CAND_PAR;
                int first = cur_cb, nl = cur_n;                 // the entries to offer
                double dsum = 0.0;
                const int* list = nullptr;
                if (cur_n > 32) {
                    // a long run: only the best of its children, by count, can ever be added.  A ready-made list of them
                    // stands in front of the run, or is made here.
                    const int room = budget - cnt;
                    if (cur_w & RUN_HAS_TOP) {
                        const int4 hdr = ent[cur_cb - SD_TOP_BLOCK];
                        dsum = (double)(((unsigned long long)(unsigned)hdr.y << 32) | (unsigned long long)(unsigned)hdr.x);
                        nl = min(hdr.z, room);
                        first = cur_cb - SD_TOP_BLOCK + 1;
                    } else {
                        unsigned sum;
                        nl = list_by_count(ent, cur_cb, cur_n, room, W.one_tok, reinterpret_cast<int*>(&W.T), sum, lane);
                        dsum = (double)sum;
                        list = W.one_tok;
                    }
                }
                for (int base = 0; base < nl; base += 32) {
                    const int k = min(32, nl - base);
                    // a child per lane with a free place; where there are too few of a kind, all lanes in order, and a place is found or made
                    const unsigned f0 = __ballot_sync(FULL, c0.hi == 0u), f1 = __ballot_sync(FULL, c1.hi == 0u);
                    const bool to0 = __popc(f0) >= k, fits = to0 || __popc(f1) >= k;
                    const unsigned f = to0 ? f0 : (fits ? f1 : FULL);
                    const int r = __popc(f & lt);
                    const bool in = ((f >> lane) & 1u) != 0u && r < k;
                    int4 e = make_int4(0, 0, 0, 0);
                    if (in) e = ent[list ? list[base + r] : first + base + r];
                    double q;
                    if (cur_n <= 32) {
                        const unsigned sum = __reduce_add_sync(FULL, (unsigned)e.y);             // sibling sum: the denominator of Eq. 1
                        if (sum <= (unsigned)RECIP_MAX) q = quotient((double)e.y, (double)sum, sh.recip.r[sum]);
                        else q = __ddiv_rn((double)e.y, (double)sum);
                    } else q = __ddiv_rn((double)e.y, dsum);
                    const double dc = __dmul_rn(cur_d, q);      // Eq. 2
                    Cand c{(unsigned)__double2hiint(dc), (unsigned)__double2loint(dc), e.x, e.z, ((unsigned)e.w & CAND_RUN) | par};
                    const bool keep = in && c.hi >= floor;
                    if (keep && (c.np & RUN_COUNT_MASK)) prefetch_l2(ent + e.z);
                    if (fits) {
                        if (keep) { if (to0) c0 = c; else c1 = c; }
                    } else if (__any_sync(FULL, keep)) {
                        if (!keep) c.hi = 0u;
                        int n = 0;
                        auto stage = [&](const Cand& v) {
                            const bool on = v.hi >= floor;      // (a free place's 0 is not)
                            const unsigned m = __ballot_sync(FULL, on);
                            if (on) {
                                const int i = n + __popc(m & lt);
                                W.C.d[i] = __hiloint2double((int)v.hi, (int)v.lo); W.C.tok[i] = v.tok; W.C.cb[i] = v.cb; W.C.np[i] = v.np;
                            }
                            n += __popc(m);
                        };
                        auto back = [&](int i) {
                            return i < n ? Cand{(unsigned)__double2hiint(W.C.d[i]), (unsigned)__double2loint(W.C.d[i]), W.C.tok[i], W.C.cb[i], W.C.np[i]}
                                         : Cand{0u, 0u, 0, 0, 0u};
                        };
                        stage(c);
                        if (ROOMY && n <= __popc(f0) + __popc(f1)) {             // those that matter go into free places of either kind
                            __syncwarp();
                            if (c0.hi == 0u) c0 = back(__popc(f0 & lt));
                            if (c1.hi == 0u) c1 = back(__popc(f0) + __popc(f1 & lt));
                        } else {
                            stage(c0); stage(c1);
                            __syncwarp();
                            n = pool_compact(W.C, n, budget - cnt, floor, lane);
                            c0 = back(lane); c1 = back(32 + lane);
                        }
                        __syncwarp();
                    }
                    // as many as can still be added: what is worse than the last of them does not matter any more
                    if (cur_n > 32 && nl == budget - cnt && base + 32 >= nl) {
                        const unsigned last = __ballot_sync(FULL, in && r == k - 1);
                        floor = max(floor, __shfl_sync(FULL, c.hi, __ffs(last) - 1));
                    }
                }
            }
        }
        // ---------------- the best candidate is the next node
        const unsigned top = __reduce_max_sync(FULL, max(c0.hi, c1.hi));
        if (top == 0u) break;
        unsigned b0 = __ballot_sync(FULL, c0.hi == top), b1 = __ballot_sync(FULL, c1.hi == top);
        if ((b0 & (b0 - 1u)) | (b1 & (b1 - 1u)) | (b0 && b1 ? 1u : 0u)) {
            // several share the high word: full comparison
            const unsigned mlo = __reduce_max_sync(FULL, max(c0.hi == top ? c0.lo : 0u, c1.hi == top ? c1.lo : 0u));
            const bool t0 = c0.hi == top && c0.lo == mlo, t1 = c1.hi == top && c1.lo == mlo;
            b0 = __ballot_sync(FULL, t0); b1 = __ballot_sync(FULL, t1);
            const int ties = __popc(b0) + __popc(b1);
            if (ties > 1 && (ties > 32 || (flags & SD_FLAG_LINEAR))) {
                // smallest token, then smallest parent index
                const unsigned mt = __reduce_min_sync(FULL, min(t0 ? (unsigned)c0.tok : 0xffffffffu, t1 ? (unsigned)c1.tok : 0xffffffffu));
                const bool s0 = t0 && (unsigned)c0.tok == mt, s1 = t1 && (unsigned)c1.tok == mt;
                const unsigned p0 = (c0.np >> CAND_PAR) & 63u, p1 = (c1.np >> CAND_PAR) & 63u;
                const unsigned mp = __reduce_min_sync(FULL, min(s0 ? p0 : 64u, s1 ? p1 : 64u));
                b0 = __ballot_sync(FULL, s0 && p0 == mp); b1 = __ballot_sync(FULL, s1 && p1 == mp);
            } else if (ties > 1) {
                // Candidates of equal D take turns: smallest token first, then smallest parent index, and an
                // only child (C = 1: the same D again) takes its parent's place.  All of them are ahead of every
                // other candidate, so a lane each keeps them until one has several children or all have ended.
                // (Text that occurs a few times below the match node is just this: chains of equal D, token by token in
                // turn.  One by one through the pool a node of them costs several times as much.)
                const int i0 = __popc(b0 & lt), i1 = __popc(b0) + __popc(b1 & lt);
                if (t0) { W.one_tok[i0] = c0.tok; W.one_cb[i0] = c0.cb; W.one_nc[i0] = c0.np; }
                if (t1) { W.one_tok[i1] = c1.tok; W.one_cb[i1] = c1.cb; W.one_nc[i1] = c1.np; }
                __syncwarp();
                const bool mine = lane < ties;
                bool live = mine;
                int tok = 0, par = 0, cb = 0;
                unsigned nc = 0;
                int4 nx = make_int4(0, 0, 0, 0);                // the only child, read ahead
                if (mine) {
                    tok = W.one_tok[lane]; cb = W.one_cb[lane]; nc = W.one_nc[lane];
                    par = (int)(nc >> CAND_PAR) & 63;
                    if ((nc & RUN_COUNT_MASK) == 1u) nx = ent[cb];
                }
                cur_d = __hiloint2double((int)top, (int)mlo);
                unsigned alive = (ties == 32 ? FULL : (1u << ties) - 1u);
                while (cnt < budget) {
                    if ((cnt & 3) == 0 && hopeless(cur_d)) { dropped = true; break; }
                    const unsigned mt = __reduce_min_sync(FULL, live ? (unsigned)tok : 0xffffffffu);
                    unsigned who = __ballot_sync(FULL, live && (unsigned)tok == mt);
                    if (who & (who - 1u)) {
                        const bool in = (who >> lane) & 1u;
                        const unsigned mp = __reduce_min_sync(FULL, in ? (unsigned)par : 0xffffffffu);
                        who = __ballot_sync(FULL, in && (unsigned)par == mp);
                    }
                    const int wl = __ffs(who) - 1;
                    const int n = (int)(__shfl_sync(FULL, nc, wl) & RUN_COUNT_MASK);
                    if (lane == wl) {
                        W.tok[buf][cnt] = tok; W.par[buf][cnt] = (unsigned char)par;
                        if (n == 1) {
                            tok = nx.x; par = cnt + 1; cb = nx.z; nc = (unsigned)nx.w;
                            if ((nc & RUN_COUNT_MASK) == 1u) nx = ent[cb];
                        } else live = false;
                    }
                    score = __dadd_rn(score, cur_d);            // Eq. 4, insertion order
                    left -= 1.0;
                    ++cnt;
                    if (n == 1) continue;
                    alive &= ~(1u << wl);
                    if (n > 1) {
                        have_cur = true;
                        cur_idx = cnt - 1;
                        cur_cb = __shfl_sync(FULL, cb, wl);
                        cur_w = (unsigned)__shfl_sync(FULL, nc, wl);
                        break;
                    }
                    if (!alive) break;
                }
                if (dropped) break;
                publish();
                if (cnt >= budget) break;
                if (mine) { W.one_tok[lane] = tok; W.one_cb[lane] = cb; W.one_nc[lane] = (nc & CAND_RUN) | ((unsigned)par << CAND_PAR); }
                __syncwarp();
                const unsigned lives = __ballot_sync(FULL, live);
                if (t0) { c0.tok = W.one_tok[i0]; c0.cb = W.one_cb[i0]; c0.np = W.one_nc[i0]; if (!((lives >> i0) & 1u)) c0.hi = 0u; }
                if (t1) { c1.tok = W.one_tok[i1]; c1.cb = W.one_cb[i1]; c1.np = W.one_nc[i1]; if (!((lives >> i1) & 1u)) c1.hi = 0u; }
                __syncwarp();
                continue;
            }
        }
        {
            const bool from0 = b0 != 0u;
            const int wl = __ffs(from0 ? b0 : b1) - 1;
            const unsigned lo = from0 ? c0.lo : c1.lo, np = from0 ? c0.np : c1.np;
            const int cb = from0 ? c0.cb : c1.cb;
            cur_d = __hiloint2double((int)top, (int)__shfl_sync(FULL, lo, wl));
            cur_cb = __shfl_sync(FULL, cb, wl);
            cur_w = __shfl_sync(FULL, np, wl) & CAND_RUN;
            // everything still to come is at most cur_d each
            if (hopeless(cur_d)) { dropped = true; break; }
            if (lane == wl) {
                W.tok[buf][cnt] = from0 ? c0.tok : c1.tok; W.par[buf][cnt] = (unsigned char)((np >> CAND_PAR) & 63u);
                if (from0) c0.hi = 0u; else c1.hi = 0u;
            }
            score = __dadd_rn(score, cur_d);                    // Eq. 4, insertion order
            left -= 1.0;
            publish();
            cur_idx = cnt++;
            if (cnt >= budget) break;
            if (flags & SD_FLAG_LINEAR) { c0.hi = 0u; c1.hi = 0u; floor = 1u; }
            have_cur = true;
        }
    }
    __syncwarp();
    if (!dropped && (score > W.best_score || (score == W.best_score && score > 0.0 && order < W.best_order))) {
        if (lane == 0) {
            W.best_score = score; W.best_order = order; W.best_n = cnt; W.best_buf = buf;
            atomicMax(&sh.best_hi, (unsigned)__double2hiint(score));
        }
    }
    __syncwarp();
}

// One block of W warps per request.
//   1. match.  Global tree: the match nodes are advanced from the nodes cached at the previous
//      call by descending only the tokens appended since (full walks when the cache is stale).
//      Per-request tree: the slot's active nodes are the match nodes (sd_step: once the append
//      is done).
//   2. expand: a (tree, p) job can be taken as soon as its match node is known, costliest first; a warp per job.
//      sd_step: warp 0 appends the accepted tokens to the request's tree
//      meanwhile, exactly as sd_append would; the jobs of that tree can be taken when it is done.  (A warp that finds
//      nothing to take while something is still to come waits, but not for ever: what is left then is done behind the
//      block-wide barrier.)
//   3. jobs of either tree that start at a wide child run without top block are scanned by all
//      warps together, behind a block-wide barrier.
//   4. select + emit from shared memory; no global scratch.
// A job is skipped or dropped, exactly, as soon as an upper bound of its SCORE falls below a
// score another job of the request has already reached (the running scores are published).
constexpr int BAR_APPENDED = 1;               // a hardware barrier beside the block-wide one
constexpr int WALKERS = 8;                    // warps that walk to global match nodes, four pattern lengths each

template <bool STEP, int WARPS, int MINB>
__global__ void __launch_bounds__(WARPS * 32, MINB)
speculate_fused_kernel(sd_store sv, int n, const int32_t* __restrict__ d_slot, int Pe, double alpha, int max_spec,
                       unsigned flags, double tau, const int32_t* __restrict__ d_budget_cap, int32_t* d_n_draft,
                       int32_t* d_tokens, int32_t* d_parents, int32_t* d_positions, uint32_t* d_mask, int32_t* d_chosen_tree,
                       int32_t* d_chosen_p, double* d_score, int32_t* d_status, const int64_t* __restrict__ d_app_off,
                       const int32_t* __restrict__ d_app_tok) {
    sd_chain_begin();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    using BlockShared = BlockSharedT<WARPS>;
    constexpr int CTA_WARPS = WARPS;
    constexpr int NT = WARPS * 32;
    // the warps that do everything but the append: all of them, or all but warp 0
    constexpr int GW0 = STEP ? 1 : 0, GWARPS = WARPS - GW0, GT = GWARPS * 32;
    BlockShared& sh = *reinterpret_cast<BlockShared*>(smem_raw);
    const int tid = threadIdx.x, lane = tid & 31, wib = tid >> 5;
    const int gtid = tid - GW0 * 32, gw = wib - GW0;             // index inside that group (negative: warp 0 of sd_step)
    constexpr bool SPLIT = GWARPS > WALKERS;                     // the warps that do not walk look ahead for the append
    constexpr int WALK = SPLIT ? WALKERS : GWARPS;
    const int i = blockIdx.x;
    const int M = sv.M, words = (M + 31) / 32, D = sv.D;
    for (int q = tid; q < (int)sizeof(RecipTable) / 16; q += NT)
        reinterpret_cast<double2*>(&sh.recip)[q] = reinterpret_cast<const double2*>(&g_recip)[q];
    const int slot = d_slot[i];
    const bool ok = slot >= 0 && slot < sv.R;
    // a slot may appear once per call: a later appearance is refused (two blocks on one tree would
    // race); the answer is collected at the first barrier below, before anything is written
    int dup = 0;
    for (int j = tid; j < i; j += NT) dup |= d_slot[j] == slot ? 1 : 0;
    int t = 0, status = SD_STATUS_BAD_SLOT;
    SlotState* ss = nullptr;
    if (ok) { ss = sv.s_state + slot; t = ss->len; status = ss->status; }
    // STEP: t_old tokens are in the slot's text, the next n_new come from the append list; the
    // match below already runs on the context of t = t_old + n_new tokens
    const int t_old = t;
    const int32_t* newtok = nullptr;
    int n_new = 0;
    if (STEP && ok) {
        newtok = d_app_tok + d_app_off[i];
        n_new = (int)(d_app_off[i + 1] - d_app_off[i]);
        t = t_old + n_new;
    }
    bool usable = ok && !(status & (SD_STATUS_POOL_FULL | SD_STATUS_BAD_TOKEN)) && t > 0;
    const int32_t* text = ok ? sv.s_text + (long long)slot * sv.T : nullptr;
    if (STEP && ok) append_stage_tokens(sh.app, text, t_old, newtok, n_new, tid, NT);
    int cap = max_spec;
    if (d_budget_cap && d_budget_cap[i] >= 0) cap = min(cap, d_budget_cap[i]);
    if (tid < 2 * SD_MAX_DEPTH) { (&sh.node[0][0])[tid] = -1; (&sh.nc[0][0])[tid] = 0; }
    if (tid == 0) {
        sh.nwide = 0; sh.nwide_kept = 0; sh.best_hi = 0u; sh.board.ready[0] = 0u; sh.board.ready[1] = 0u;
        sh.board.walking = WALK; sh.board.appending = 1; sh.gave_up = 0; sh.app.ahead = 0; sh.at_hand = 0;
    }
    if (wib == WARPS - 1) {
        const int c = lane < Pe ? min(budget_for(alpha, lane + 1, cap), 2 * (D - lane - 1)) : -1;
        int rank = 0;
#pragma unroll
        for (int q = 0; q < 32; ++q) {
            const int cq = __shfl_sync(FULL, c, q);
            rank += (cq > c || (cq == c && q < lane)) ? 1 : 0;
        }
        sh.ordp[rank] = (unsigned char)lane;
    }
    WarpWork& W = sh.w[wib];
    if (lane == 0) { W.best_score = 0.0; W.best_order = 1 << 30; W.best_n = 0; W.best_buf = 0; }

    // ---------------- 1. match
    bool want_g = usable && !(flags & SD_FLAG_REQUEST_ONLY);
    bool want_r = usable && !(flags & SD_FLAG_GLOBAL_ONLY);
    // (a slot that appears twice is refused below; until then its first block may be writing what this one reads, so the lanes vote)
    if (gw == 0 && __all_sync(FULL, want_g)) {
        // the walk to the match node of the last d tokens starts at the node kept from the call before, or at the root
        const int d = lane + 1;
        int len = ss->g_len, depths = ss->g_depths, kept = ss->g_node[lane];
        bool known = __all_sync(FULL, ss->g_gen == ss->gen && ss->g_epoch == sv.g_state->epoch && len <= t);
        if (!known) {
            // (a call of sd_build_requests may be writing it)
            const MatchRecord& rec = ss->record;
            const int version = sd_acquire(&rec.version);
            len = sd_relaxed(&rec.len); depths = D; kept = sd_relaxed(&rec.node[lane]);
            known = version != 0 && (version & 1) == 0 && sd_relaxed(&rec.epoch) == sv.g_state->epoch && len > 0 && len <= t_old;
            if (known && lane < len && lane < D) known = sd_relaxed(&rec.tail[lane]) == text[len - 1 - lane];
            sd_fence();
            known = __all_sync(FULL, known && sd_relaxed(&rec.version) == version);
        }
        const int k = t - len;                                  // tokens appended since
        const int before = __shfl_sync(FULL, kept, max(d - k - 1, 0));
        // the match nodes of this very context are at hand?  (One warp tells the others: the block of a slot that appears twice in the
        // call, which is refused, reads all this while the slot's first block may be writing it.)
        if (!STEP && lane == 0) sh.at_hand = known && k == 0;
        int node = -1, from = t;
        if (d <= t && d <= Pe) {
            if (known && d > k && d - k <= depths) {
                node = before;                                  // node of the tokens before the new ones
                from = t - k;
            } else {
                const int x0 = t - d < t_old ? text[t - d] : newtok[t - d - t_old];
                node = (x0 >= 0 && x0 < sv.V) ? sv.g_root[x0] : -1;
                from = t - d + 1;
            }
        }
        if (d <= Pe) { sh.src_node[lane] = node; sh.src_from[lane] = from; }
    }
    // all cached nodes read before any is replaced; and: is this a second block for the same slot?
    const bool refused = __syncthreads_or(dup) != 0;
    if (refused) { usable = false; want_g = false; want_r = false; status = SD_STATUS_BAD_SLOT; }
    // a lane per place in the order of the jobs (by the number of nodes a job can add at most)
    const int my_p = sh.ordp[lane] + 1, my_budget = my_p <= Pe ? budget_for(alpha, my_p, cap) : 0;
    // SCORE <= number of draft nodes (every D <= 1), and SCORE <= number of levels below the
    // match node: the D values of one level of a tree add up to at most 1 (Eq. 1 shares out
    // the parent's D among its children)
    const unsigned my_limit = (unsigned)__double2hiint((double)min(my_budget, D - my_p) * 1.000000001);
    // the jobs of pattern lengths [pa, pb), whose match nodes are known, can be taken
    auto offer = [&](int tree, bool want, int pa, int pb, const int4* base) {
        __syncwarp();
        const bool job = want && my_p >= pa && my_p < pb && my_p <= t && min(my_budget, D - my_p) > 0 && sh.node[tree][my_p - 1] >= 0;
        const unsigned wf = job ? sh.nc[tree][my_p - 1] : 0u;
        const int nch = (int)(wf & RUN_COUNT_MASK);
        const bool far = nch > WIDE_RUN && !(wf & RUN_HAS_TOP);  // scanned by all warps together, later
        if (far) sh.wide[atomicAdd(&sh.nwide, 1)] = tree * SD_MAX_DEPTH + my_p - 1;
        else if (nch > 0) {
            // all first runs start their way to L2 now, before a warp gets to them
            const int4* run = base + sh.cb[tree][my_p - 1];
            for (int l = 0; l < min(4, (nch + 7) >> 3); ++l) prefetch_l2(run + l * 8);
        }
        const unsigned m = __ballot_sync(FULL, nch > 0 && !far);
        __threadfence_block();
        if (lane == 0 && m) atomicOr(&sh.board.ready[tree], m);
    };
    const int4* s_ent = ok ? sv.s_ent + (long long)slot * sv.spn : nullptr;
    const bool look_ahead = STEP && n_new >= 3 && usable;         // (one or two tokens are as soon searched for in their turn)
    if (wib == (STEP ? 0 : WARPS - 1)) {
        // ---- the request's match nodes are its active nodes
        int act = -1, cb = 0;
        unsigned w = 0;
        bool good = usable;
        if (ok && !refused) {
            act = ss->active[lane]; cb = ss->run_cb[lane]; w = ss->run_w[lane];
            if (STEP && n_new > 0) {
                // ---- sd_step: its accepted tokens go into its tree and text (as sd_append does)
                int len = ss->len, used = ss->used, live = ss->live, st = ss->status;
                if (!(st & (SD_STATUS_POOL_FULL | SD_STATUS_BAD_TOKEN))) {
                    w = append_pack(w, ss->room[lane]);
                    append_tokens<(MINB < 4)>(sh.app, sv, slot, newtok, n_new, SPLIT ? GWARPS - WALKERS : GWARPS, lane, act, cb, w, len, used, live, st);
                    append_store(ss, lane, act, cb, w);
                    if (w != RUN_UNKNOWN) w &= ~(ROOM_MASK << ROOM_SHIFT);
                }
                if (lane == 0) { ss->len = len; ss->used = used; ss->live = live; ss->status = st; }
                // an append that stopped early leaves a context the jobs were not made for
                good = good && len == t && !(st & (SD_STATUS_POOL_FULL | SD_STATUS_BAD_TOKEN));
            }
        }
        if (good && act >= 0 && w == RUN_UNKNOWN) { const int4 e = s_ent[act]; cb = e.z; w = (unsigned)e.w; }
        sh.node[1][lane] = act; sh.cb[1][lane] = cb; sh.nc[1][lane] = w;
        offer(1, good && want_r, 1, SD_MAX_DEPTH + 1, s_ent);
        __threadfence_block();
        if (lane == 0) atomicSub(&sh.board.appending, 1);
    }
    if (gw >= 0) {
        if (look_ahead && (!SPLIT || gw >= WALKERS)) {
            search_ahead(sh.app, sv, s_ent, sv.s_root + (long long)slot * sv.V, t_old, n_new, (gtid - (SPLIT ? WALKERS * 32 : 0)) / APP_LANES,
                         (GT - (SPLIT ? WALKERS * 32 : 0)) / APP_LANES, lane);
            __threadfence_block();
            __syncwarp();
            if (lane == 0) atomicAdd(&sh.app.ahead, 1);
        }
        // ---- global match nodes: eight lanes per pattern length
        if (gw < WALK) {
            if (want_g) {
                for (int p0 = 0; p0 + gw * 4 < Pe; p0 += WALK * 4) {
                    const int d = p0 + gtid / APP_LANES + 1;
                    int node = d <= Pe ? sh.src_node[d - 1] : -1;
                    const int pos = d <= Pe ? sh.src_from[d - 1] : t;
                    int2 zw = make_int2(0, 0);
                    if (node >= 0) zw = *reinterpret_cast<const int2*>(&sv.g_ent[node].z);
                    group_walk(sv.g_ent, (int)sv.g_cap, node, zw, t - pos, lane, [&](int k) {
                        const int kx = pos + k - t_old;            // (of the new tokens the first ones are at hand)
                        return kx < 0 ? text[pos + k] : (kx < APP_AHEAD ? sh.app.tok[kx + APP_SHALLOW - 1] : newtok[kx]);
                    });
                    if ((lane & (APP_LANES - 1)) == 0 && d <= Pe) {
                        ss->g_node[d - 1] = node;
                        sh.node[0][d - 1] = node;
                        if (node >= 0) { sh.cb[0][d - 1] = zw.x; sh.nc[0][d - 1] = (unsigned)zw.y; }
                    }
                    offer(0, true, p0 + gw * 4 + 1, p0 + gw * 4 + 5, sv.g_ent);
                }
                if (gtid == 0) { ss->g_gen = ss->gen; ss->g_epoch = sv.g_state->epoch; ss->g_len = t; ss->g_depths = Pe; }
            }
            __threadfence_block();
            if (lane == 0) atomicSub(&sh.board.walking, 1);
        }
    }

    // ---------------- 2. the jobs, until none is left and none can come any more.  (A queue made when all match nodes were
    // known, whose next job might have to wait for the append: steps of 1 / 64 / 256 / 512 requests 16.5 / 38 / 52 / 42 us, now
    // 16 / 36 / 48 / 40.  Taking the cheap half at once, too: 50 for 256.)
    auto work = [&]() {
        int skip = wib;                                         // (not all warps go for the same one)
        for (int spins = 0;;) {
            unsigned m0, m1, walking, appending;                // (one access: what is said to have come is there)
            asm volatile("ld.volatile.shared.v4.u32 {%0, %1, %2, %3}, [%4];"
                         : "=r"(m0), "=r"(m1), "=r"(walking), "=r"(appending) : "r"((unsigned)__cvta_generic_to_shared(&sh.board)) : "memory");
            if (__all_sync(FULL, (m0 | m1) == 0u && (walking | appending) != 0u) && ++spins <= 4096) {
                __nanosleep(400);                               // (200: steps of 512 requests 1 % longer, the append has fewer issue slots)
                skip = wib;                                     // (what comes next comes all at once)
                continue;
            }
            const unsigned best = *(volatile unsigned*)&sh.best_hi;
            const unsigned able = __ballot_sync(FULL, my_limit >= best);
            const unsigned r0 = __ballot_sync(FULL, (m0 >> lane) & 1u), r1 = __ballot_sync(FULL, (m1 >> lane) & 1u);
            // a job whose bound is below a score already reached is dropped, exactly
            if (lane == 0 && (r0 & ~able)) atomicAnd(&sh.board.ready[0], able);
            if (lane == 0 && (r1 & ~able)) atomicAnd(&sh.board.ready[1], able);
            const bool more = __any_sync(FULL, (walking | appending) != 0u);
            const bool first = __any_sync(FULL, walking != 0u);   // (the costlier half only, while costlier ones may still come)
            const unsigned v0 = r0 & able & (first ? 0xffffu : FULL), v1 = r1 & able & (first ? 0xffffu : FULL);
            const int total = __popc(v0) + __popc(v1);
            if (total == 0) {
                if (!more) break;
                if (++spins > 4096) { if (lane == 0) sh.gave_up = 1; break; }
                __nanosleep(400);
                continue;
            }
            const int k = min(skip, total - 1);
            const unsigned lt = (1u << lane) - 1u, mine0 = (v0 >> lane) & 1u;
            const int at = __popc(v0 & lt) + __popc(v1 & lt);   // the global tree's job before the request's
            const unsigned w0 = __ballot_sync(FULL, mine0 && at == k), w1 = __ballot_sync(FULL, ((v1 >> lane) & 1u) && at + (int)mine0 == k);
            const int tree = w0 ? 0 : 1, rank = __ffs(w0 | w1) - 1;
            unsigned old = 0;
            if (lane == 0) old = atomicAnd(&sh.board.ready[tree], ~(1u << rank));
            old = __shfl_sync(FULL, old, 0);
            skip = 0;
            if (!((old >> rank) & 1u)) continue;                // another warp was faster
            __threadfence_block();
            const int p = __shfl_sync(FULL, my_p, rank), budget = __shfl_sync(FULL, my_budget, rank);
            expand_job<MINB == 1>(sh, W, tree == 0 ? sv.g_ent : s_ent, tree == 0 ? (int)sv.g_cap : (int)sv.spn, tree, p, budget, flags, -1, lane);
        }
    };
    // All jobs can be taken at once: in their order, then (256 requests: 38.6 us, without the barrier 41; where the SM has one block
    // it only costs, 6.2 -> 6.8 us for one request).
    if (!STEP && MINB > 1 && sh.at_hand) __syncthreads();
    // (nothing to do before the append is done: in a hardware barrier; looking every 200 ns cost such steps 4 %, every 400 ns 2 %)
    if (STEP && !want_g) {
        if (wib == 0) asm volatile("bar.arrive %0, %1;" ::"r"(BAR_APPENDED), "r"(NT) : "memory");
        else asm volatile("bar.sync %0, %1;" ::"r"(BAR_APPENDED), "r"(NT) : "memory");
    }
    work();
    __syncthreads();                                            // sd_step: the append is done and visible

    // ---------------- 3. what had to wait: an append that stopped early, jobs that no warp waited for,
    // jobs that start at a wide child run
    if (STEP && ok && !refused) {
        status = ss->status;
        if (ss->len != t || (status & (SD_STATUS_POOL_FULL | SD_STATUS_BAD_TOKEN))) {
            // the append stopped early: no speculation for this request, and the match nodes
            // taken above describe a context that does not exist
            usable = false; want_g = false; want_r = false;
            t = ss->len;
            if (tid == 0) ss->g_gen = ss->gen - 1;
        }
    }
    if (sh.gave_up || sh.nwide > 0) {                           // (either only grows before the barrier above)
        if (sh.gave_up && usable) work();
        __syncthreads();
        // Jobs that start at a wide node (short patterns, hence small budgets): most cannot reach
        // the best score any more and are dropped here.  For the rest the warps of the block share
        // the scan of the run, then one warp merges the partial lists and finishes the job.
        if (tid == 0) {
            const double best = __hiloint2double((int)sh.best_hi, 0);
            int kept = 0;
            for (int q = 0; q < sh.nwide && usable; ++q) {
                const int p = sh.wide[q] % SD_MAX_DEPTH + 1;
                if (!((double)min(budget_for(alpha, p, cap), D - p) * 1.000000001 < best)) sh.wide[kept++] = sh.wide[q];
            }
            sh.nwide_kept = kept;
        }
        __syncthreads();
        const int nwide = sh.nwide_kept;
        for (int base = 0; base < nwide; base += CTA_WARPS) {
            const int nj = min(CTA_WARPS, nwide - base);
            const int G = CTA_WARPS / nj;                           // warps per job
            const int my_job = wib / G, my_slice = wib % G;
            const bool active = my_job < nj;
            int tree = 0, p = 1, budget = 0, fs = 0;
            const int4* ent = sv.g_ent;
            if (active) {
                const int code = sh.wide[base + my_job];
                tree = code / SD_MAX_DEPTH; p = code % SD_MAX_DEPTH + 1;
                budget = budget_for(alpha, p, cap);
                ent = tree == 0 ? sv.g_ent : s_ent;
                long long sum;
                scan_run_by_count(ent, sh.cb[tree][p - 1], (int)(sh.nc[tree][p - 1] & RUN_COUNT_MASK), my_slice, G, -1, 1, W,
                                  W.T, 0, fs, budget, sum, lane);
                if (lane == 0) { sh.slice_sum[wib] = sum; sh.slice_fs[wib] = fs; }
            }
            __syncthreads();
            if (active && my_slice == 0) {
                long long sum = sh.slice_sum[wib];
                for (int g = 1; g < G; ++g) {
                    const Frontier& O = sh.w[wib + g].T;
                    const int ofs = sh.slice_fs[wib + g];
                    sum += sh.slice_sum[wib + g];
                    frontier_merge_list(W.T, 0, fs, budget, O, ofs, -1, lane);
                }
                counts_to_d(W.T, 0, fs, 1.0, sum, lane);
                expand_job<MINB == 1>(sh, W, ent, tree == 0 ? (int)sv.g_cap : (int)sv.spn, tree, p, budget, flags, fs, lane);
            }
            __syncthreads();
        }
    }
    if (wib != 0) return;

    // ---------------- 4. select (first in loop order among the largest scores) and emit: one warp
    double best = lane < CTA_WARPS ? sh.w[lane].best_score : 0.0;
    int od = lane < CTA_WARPS ? sh.w[lane].best_order : 1 << 30;
    int win = lane;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        const double osc = __shfl_xor_sync(FULL, best, off);
        const int ood = __shfl_xor_sync(FULL, od, off);
        const int oww = __shfl_xor_sync(FULL, win, off);
        if (osc > best || (osc == best && ood < od)) { best = osc; od = ood; win = oww; }
    }
    // Section 3.2: the tree is used only if its score exceeds the threshold (tau = 0: any score above 0)
    const bool used = usable && best > 0.0 && best > tau;
    const WarpWork& B = sh.w[win];
    const int nd = used ? B.best_n : 0;
    int tok[2], par[2], up[2];
    unsigned long long bits[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int j = lane + 32 * h;
        tok[h] = -1; par[h] = -1; bits[h] = 0ull;
        if (j < nd) { tok[h] = B.tok[B.best_buf][j]; par[h] = (int)B.par[B.best_buf][j] - 1; bits[h] = 1ull << j; }
        up[h] = par[h];
        sh.anc[j] = bits[h]; sh.up[j] = (signed char)up[h];
    }
    __syncwarp();
    // ancestors by pointer doubling: bits gathered so far, and the next ancestor to ask
    while (__any_sync(FULL, up[0] >= 0 || up[1] >= 0)) {
        unsigned long long add[2];
        int nu[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            add[h] = up[h] >= 0 ? sh.anc[up[h]] : 0ull;
            nu[h] = up[h] >= 0 ? (int)sh.up[up[h]] : -1;
        }
        __syncwarp();
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            bits[h] |= add[h];
            up[h] = nu[h];
            sh.anc[lane + 32 * h] = bits[h]; sh.up[lane + 32 * h] = (signed char)up[h];
        }
        __syncwarp();
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int j = lane + 32 * h;
        if (j >= M) continue;
        const long long o = (long long)i * M + j;
        d_tokens[o] = tok[h]; d_parents[o] = par[h]; d_positions[o] = j < nd ? t + __popcll(bits[h]) - 1 : -1;
        d_mask[o * words] = (uint32_t)bits[h];
        if (words > 1) d_mask[o * words + 1] = (uint32_t)(bits[h] >> 32);
    }
    if (lane == 0) {
        d_n_draft[i] = nd;
        d_chosen_tree[i] = used ? (od - 1) / SD_MAX_DEPTH : -1;  // order = tree * 32 + p with p in 1 .. 32
        d_chosen_p[i] = used ? (od - 1) % SD_MAX_DEPTH + 1 : 0;
        d_score[i] = used ? best : 0.0;
        if (d_status) d_status[i] = status;
    }
}

}  // namespace

namespace {

constexpr int MAX_DEVICES = 64;
struct DeviceInfo { bool ready = false; int trims = 0, sm_count = 0; };
DeviceInfo g_dev[MAX_DEVICES];
std::mutex g_dev_mutex;

template <bool STEP, int WARPS, int MINB>
int raise_smem_limit() {
    return cudaFuncSetAttribute(speculate_fused_kernel<STEP, WARPS, MINB>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)sizeof(BlockSharedT<WARPS>)) == cudaSuccess ? SD_OK : SD_ERR_CUDA;
}

// once per device (and behind sd_trim): raise the kernels' dynamic shared memory limit, read the SM count
int device_setup(int dev, int* sm_count) {
    if (dev < 0 || dev >= MAX_DEVICES) return SD_ERR_INVALID_ARG;
    std::lock_guard<std::mutex> lock(g_dev_mutex);
    const int trims = sd_trims();
    if (!g_dev[dev].ready || g_dev[dev].trims != trims) {
        if (raise_smem_limit<false, CTA_WARPS, 2>() != SD_OK || raise_smem_limit<true, CTA_WARPS_STEP, 2>() != SD_OK ||
            raise_smem_limit<false, CTA_WARPS_WIDE, 1>() != SD_OK || raise_smem_limit<true, CTA_WARPS_WIDE, 1>() != SD_OK ||
            raise_smem_limit<false, CTA_WARPS_NARROW, 4>() != SD_OK ||
            raise_smem_limit<true, CTA_WARPS_NARROW_STEP, 4>() != SD_OK)
            return SD_ERR_CUDA;
        SD_CUDA_OK(cudaDeviceGetAttribute(&g_dev[dev].sm_count, cudaDevAttrMultiProcessorCount, dev));
        g_dev[dev].trims = trims;
        g_dev[dev].ready = true;
    }
    *sm_count = g_dev[dev].sm_count;
    return SD_OK;
}

}  // namespace

static int launch_fused(sd_store* s, int32_t n, const int32_t* d_slot, const sd_spec_params* prm,
                        const int32_t* d_budget_cap, int32_t* d_n_draft, int32_t* d_tokens, int32_t* d_parents,
                        int32_t* d_positions, uint32_t* d_mask, int32_t* d_chosen_tree, int32_t* d_chosen_p,
                        double* d_score, int32_t* d_status, const int64_t* d_app_off, const int32_t* d_app_tok,
                        bool step, void* stream) {
    if (!s || !prm || n < 0 || n > s->R) return SD_ERR_INVALID_ARG;
    if (prm->P < 1 || prm->max_spec < 0 || prm->max_spec > s->M || !(prm->alpha >= 0.0) || !(prm->tau >= 0.0))
        return SD_ERR_INVALID_ARG;
    if ((prm->flags & SD_FLAG_GLOBAL_ONLY) && (prm->flags & SD_FLAG_REQUEST_ONLY)) return SD_ERR_INVALID_ARG;
    SD_CHECK_DEVICE(s);
    if (n == 0) return SD_OK;
    if (!d_slot || !d_n_draft || !d_tokens || !d_parents || !d_positions || !d_mask || !d_chosen_tree || !d_chosen_p ||
        !d_score)
        return SD_ERR_INVALID_ARG;
    if (step && !d_app_off) return SD_ERR_INVALID_ARG;
    cudaStream_t st = (cudaStream_t)stream;
    const int Pe = prm->P < s->D ? prm->P : s->D;               // longer patterns never match
    int sms = 0;
    const int rc = device_setup(s->device, &sms);
    if (rc != SD_OK) return rc;
    // one block per SM is all a small batch can use: it takes more registers
    const bool wide = n <= sms;
    // more requests than two blocks per SM hold at once: smaller blocks, one wave
    const bool narrow = n > 2 * sms;
#define SD_LAUNCH_FUSED(STEP, WARPS, MINB, OFF, TOK)                                                                     \
    SD_CUDA_OK(sd_launch(speculate_fused_kernel<STEP, WARPS, MINB>, (unsigned)n, WARPS * 32, sizeof(BlockSharedT<WARPS>), st, \
                         *s, n, d_slot, Pe, prm->alpha, prm->max_spec, prm->flags, prm->tau, d_budget_cap, d_n_draft, d_tokens, \
                         d_parents, d_positions, d_mask, d_chosen_tree, d_chosen_p, d_score, d_status, OFF, TOK))
    if (step) {
        if (wide) SD_LAUNCH_FUSED(true, CTA_WARPS_WIDE, 1, d_app_off, d_app_tok);
        else if (narrow) SD_LAUNCH_FUSED(true, CTA_WARPS_NARROW_STEP, 4, d_app_off, d_app_tok);
        else SD_LAUNCH_FUSED(true, CTA_WARPS_STEP, 2, d_app_off, d_app_tok);
    } else {
        if (wide) SD_LAUNCH_FUSED(false, CTA_WARPS_WIDE, 1, nullptr, nullptr);
        else if (narrow) SD_LAUNCH_FUSED(false, CTA_WARPS_NARROW, 4, nullptr, nullptr);
        else SD_LAUNCH_FUSED(false, CTA_WARPS, 2, nullptr, nullptr);
    }
#undef SD_LAUNCH_FUSED
    SD_CUDA_OK(cudaGetLastError());
    return SD_OK;
}

extern "C" int sd_speculate(sd_store* s, int32_t n, const int32_t* d_slot, const sd_spec_params* prm,
                            const int32_t* d_budget_cap, int32_t* d_n_draft, int32_t* d_tokens, int32_t* d_parents,
                            int32_t* d_positions, uint32_t* d_mask, int32_t* d_chosen_tree, int32_t* d_chosen_p,
                            double* d_score, int32_t* d_status, void* stream) {
    return launch_fused(s, n, d_slot, prm, d_budget_cap, d_n_draft, d_tokens, d_parents, d_positions, d_mask, d_chosen_tree,
                        d_chosen_p, d_score, d_status, nullptr, nullptr, false, stream);
}

extern "C" int sd_step(sd_store* s, int32_t n, const int32_t* d_slot, const int64_t* d_offsets, const int32_t* d_new_tokens,
                       const sd_spec_params* prm, const int32_t* d_budget_cap, int32_t* d_n_draft, int32_t* d_tokens,
                       int32_t* d_parents, int32_t* d_positions, uint32_t* d_mask, int32_t* d_chosen_tree,
                       int32_t* d_chosen_p, double* d_score, int32_t* d_status, void* stream) {
    return launch_fused(s, n, d_slot, prm, d_budget_cap, d_n_draft, d_tokens, d_parents, d_positions, d_mask, d_chosen_tree,
                        d_chosen_p, d_score, d_status, d_offsets, d_new_tokens, true, stream);
}

// ---------------------------------------------------------------------------------------------
// sd_speculate_noalloc: the same two kernels, with the per-job scratch records kept in a
// fixed array that is part of the loaded library image instead of in memory obtained
// from cudaMalloc.  Meant for callers that must not touch the CUDA allocator at all
// (see the declaration in suffixspec.h).
//
// The array's name below is only meaningful to device code.  Host code holds a stand-in
// symbol of the same name, so the launch code first asks the runtime for the array's
// real device address (once per device, with that device current) and passes that on.
namespace {

constexpr long long NOALLOC_BYTES =
    (long long)SD_NOALLOC_MAX_JOBS * (sizeof(double) + sizeof(int32_t) + 2ll * SD_MAX_SPEC * sizeof(int32_t));

static __device__ __align__(256) unsigned char g_noalloc_scratch[NOALLOC_BYTES];

constexpr int NOALLOC_MAX_DEVICES = 64;
unsigned char* g_noalloc_ptr[NOALLOC_MAX_DEVICES];      // device address of the array, per device
bool g_noalloc_ready[NOALLOC_MAX_DEVICES];
std::mutex g_noalloc_mutex;

// Device address of the scratch array on the current device (looked up on first use).
int noalloc_scratch_address(unsigned char** out) {
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= NOALLOC_MAX_DEVICES) return SD_ERR_CUDA;
    std::lock_guard<std::mutex> lock(g_noalloc_mutex);
    if (!g_noalloc_ready[dev]) {
        unsigned char* p = nullptr;
        if (cudaGetSymbolAddress((void**)&p, g_noalloc_scratch) != cudaSuccess || !p) {
            cudaGetLastError();
            return SD_ERR_CUDA;
        }
        g_noalloc_ptr[dev] = p;
        g_noalloc_ready[dev] = true;
    }
    *out = g_noalloc_ptr[dev];
    return SD_OK;
}

}  // namespace

extern "C" int sd_speculate_noalloc(sd_store* s, int32_t n, const int32_t* d_slot, const sd_spec_params* prm,
                                    const int32_t* d_budget_cap, int32_t* d_n_draft, int32_t* d_tokens,
                                    int32_t* d_parents, int32_t* d_positions, uint32_t* d_mask, int32_t* d_chosen_tree,
                                    int32_t* d_chosen_p, double* d_score, int32_t* d_status, void* stream) {
    if (!s || !prm || n < 0 || n > s->R) return SD_ERR_INVALID_ARG;
    if (prm->P < 1 || prm->max_spec < 0 || prm->max_spec > s->M || !(prm->alpha >= 0.0) || !(prm->tau >= 0.0))
        return SD_ERR_INVALID_ARG;
    if ((prm->flags & SD_FLAG_GLOBAL_ONLY) && (prm->flags & SD_FLAG_REQUEST_ONLY)) return SD_ERR_INVALID_ARG;
    SD_CHECK_DEVICE(s);
    // one record per (request, tree, depth): the batch must fit the fixed array
    if ((long long)n * 2 * s->D > SD_NOALLOC_MAX_JOBS) return SD_ERR_CAPACITY;
    if (n == 0) return SD_OK;
    if (!d_slot || !d_n_draft || !d_tokens || !d_parents || !d_positions || !d_mask || !d_chosen_tree || !d_chosen_p ||
        !d_score)
        return SD_ERR_INVALID_ARG;
    unsigned char* base = nullptr;
    const int rc = noalloc_scratch_address(&base);
    if (rc != SD_OK) return rc;
    // Same record layout as the store's own scratch, carved out of the fixed array.  Every
    // record the second kernel reads is written by the first kernel of the same call, so
    // nothing left over from an earlier call is ever consumed and nothing needs clearing.
    sd_store view = *s;
    view.j_score = reinterpret_cast<double*>(base);
    view.j_n = reinterpret_cast<int32_t*>(base + (long long)SD_NOALLOC_MAX_JOBS * sizeof(double));
    view.j_tok = view.j_n + SD_NOALLOC_MAX_JOBS;
    view.j_par = view.j_tok + (long long)SD_NOALLOC_MAX_JOBS * SD_MAX_SPEC;
    cudaStream_t st = (cudaStream_t)stream;
    const int Pe = prm->P < s->D ? prm->P : s->D;
    const long long jobs = (long long)n * 2 * Pe;
    match_expand_kernel<<<(unsigned)((jobs + SPEC_WARPS - 1) / SPEC_WARPS), SPEC_WARPS * 32, 0, st>>>(
        view, n, d_slot, Pe, prm->alpha, prm->max_spec, prm->flags, d_budget_cap);
    select_emit_kernel<<<(unsigned)((n + 3) / 4), 128, 0, st>>>(view, n, d_slot, Pe, prm->tau, d_n_draft, d_tokens, d_parents,
                                                                d_positions, d_mask, d_chosen_tree, d_chosen_p, d_score,
                                                                d_status);
    SD_CUDA_OK(cudaGetLastError());
    return SD_OK;
}
