// Online update of the suffix trees: device functions shared by the kernels that append tokens
// (the batched append kernel and the fused decode-step kernel) and by those that walk a tree.
//
// Online update of the suffix trees (Section 3, "Suffix Tree Construction": the
// tokens of the ongoing request are added as they are generated, a finished
// request's output is added to the global tree).
//
// Per-request trees: one warp owns one tree for the duration of the kernel.  Appending token x at
// context length t adds one occurrence to every string that ends at x and is at
// most D tokens long: lane L extends the ACTIVE node of depth L (the node of
// the last L tokens; lane 0 extends the root) by child x, creating it or
// raising its count.  The 32 lanes work on 32 different parents at once.
//
// Placement.  A suffix that has left the known text creates one new leaf per appended token,
// each the only child of the previous one.  The first such leaf reserves room for the whole
// chain down to depth D and every later leaf goes directly behind its parent, so chains of
// only children are consecutive entries (what the wide window loads of sd_speculate exploit).
#pragma once

#include "common.cuh"

namespace {

__device__ __forceinline__ int* word(int4* e, int k) { return reinterpret_cast<int*>(e) + k; }

// The whole warp inserts child x at sorted position `pos` into the child run of `parent` (cb, n
// children): entries move 32 at a time.  `moves`: the run is full and goes to ent[fresh ...).  Returns the new
// child's entry.  All arguments are warp-uniform.
__device__ int insert_child_warp(int4* ent, int parent, int cb, int n, int pos, int x, int fresh, bool moves, int lane) {
    const int4 ne = make_int4(x, 1, 0, 0);
    int idx;
    if (moves) {
        for (int i = lane; i < n; i += 32) ent[fresh + i + (i >= pos ? 1 : 0)] = ent[cb + i];
        idx = fresh + pos;
        if (lane == 0) { ent[idx] = ne; *word(&ent[parent], 2) = fresh; }
    } else {
        for (int hi = n; hi > pos; hi -= 32) {                   // from the top down, a chunk at a time
            const int lo = max(pos, hi - 32);
            const int i = lo + lane;
            int4 e = make_int4(0, 0, 0, 0);
            if (i < hi) e = ent[cb + i];
            __syncwarp();
            if (i < hi) ent[cb + i + 1] = e;
            __syncwarp();
        }
        idx = cb + pos;
        if (lane == 0) ent[idx] = ne;
    }
    if (lane == 0) *word(&ent[parent], 3) = n + 1;
    __syncwarp();
    return idx;
}

// The same for up to four lanes at once, by eight lanes each: `src` is the lane that a group works for (-1: none), the
// other arguments are every lane's own.  Returns the new child's entry to the lanes of src's group.
__device__ int insert_child_groups(int4* ent, int src, int parent, int cb, int n, int pos, int x, int fresh, bool moves, int lane) {
    const unsigned FULL = 0xffffffffu;
    const int l = lane & 7, from = max(src, 0);
    parent = __shfl_sync(FULL, parent, from); cb = __shfl_sync(FULL, cb, from); n = __shfl_sync(FULL, n, from);
    pos = __shfl_sync(FULL, pos, from); fresh = __shfl_sync(FULL, fresh, from);
    moves = __shfl_sync(FULL, moves ? 1 : 0, from) != 0;
    const bool on = src >= 0;
    if (on && moves)
        for (int i = l; i < n; i += 8) ent[fresh + i + (i >= pos ? 1 : 0)] = ent[cb + i];
    for (int hi = on && !moves ? n : 0; __any_sync(FULL, hi > pos); hi -= 8) {
        const int i = max(pos, hi - 8) + l;
        int4 e = make_int4(0, 0, 0, 0);
        if (i < hi) e = ent[cb + i];
        __syncwarp();
        if (i < hi) ent[cb + i + 1] = e;
        __syncwarp();
    }
    const int idx = moves ? fresh + pos : cb + pos;
    if (on && l == 0) {
        ent[idx] = make_int4(x, 1, 0, 0);
        if (moves) *word(&ent[parent], 2) = fresh;
        *word(&ent[parent], 3) = n + 1;
    }
    __syncwarp();
    return idx;
}

// ---------------------------------------------------------------------------------------------
// Append to a request's tree: one warp, a lane per active node.
//
// Tokens follow one another strictly (the next one starts at the nodes this one found or made), so a
// request with 16 accepted tokens waits for 16 steps in a row, and that is what most decode steps wait
// for.  A warp gets about one instruction per seven cycles on such a chain, so what counts is how few
// there are.  Nearly all runs below the first levels have at most four children: four loads per lane, all at
// once, and no search.  The first levels' runs are long; where a token belongs in them is looked up ahead by
// other warps, for many tokens at once (search_ahead: eight lanes per search), and the lane then reads four
// entries around that place.  Where a place is not known, one or two long runs are searched by the whole warp, one after
// the other; from three on (APP_OPEN) every lane searches its own at once.  Leaves are written by their lanes, all at once;
// children that go into runs are inserted four at a time, eight lanes each, or by the whole warp where more than APP_BIG
// entries move or one is left.  (A search of up to eight entries per lane and round for every
// lane, four rounds for a long run, took 2.3 us per token with the SM to itself and 3.8 with four
// blocks on it.  Searches and inserts for one lane at a time throughout, on text with long runs at many depths: 106 us
// for a step of 256 requests, 80.5 as it is.)
constexpr int APP_AHEAD = 28;                 // tokens looked up ahead
constexpr int APP_SHALLOW = 4;                // depths looked up ahead
constexpr int APP_LANES = 8;                  // lanes per search
constexpr int APP_OPEN = 3;                   // long runs to search from which on every lane searches its own
constexpr int APP_BIG = 64;                   // entries to move from which on the whole warp does it
constexpr unsigned ROOM_SHIFT = 24, ROOM_MASK = 31u;            // room behind a node, kept in the spare bits of its w field while appending

struct AppendShared {
    int tok[APP_AHEAD + APP_SHALLOW + 2];     // the first new tokens, the few before and the two behind them (-1: none)
    int hint[APP_AHEAD][APP_SHALLOW];         // by token and parent depth: where it belonged in that run before the append (-1: unknown)
    int ahead;                                // warps that have left their hints
};

// One range of a sorted run being searched by eight lanes.
struct RunSearch {
    const int4* run;
    int lo, hi;
};

__device__ __forceinline__ int search_probe(const RunSearch& r, int k) { return r.lo + ((r.hi - r.lo) * (k + 1)) / 9; }

// All lanes of the warp call; the eight lanes of a group search for x in their run (an empty range is allowed).
// Returns its place or -1, with the child run of the entry found; `place` is where it belongs.
__device__ __forceinline__ int group_lookup(RunSearch a, int x, int lane, int& place, int2& zw) {
    const unsigned FULL = 0xffffffffu;
    const int l = lane & (APP_LANES - 1), gb = lane & ~(APP_LANES - 1);
    while (true) {
        const bool on = a.hi - a.lo > APP_LANES;
        if (!__any_sync(FULL, on)) break;
        int t = 0;
        if (on) t = a.run[search_probe(a, l)].x;
        const int c = __popc((__ballot_sync(FULL, on && t < x) >> gb) & 0xffu);          // probes below x
        if (on) {
            const int lo = c > 0 ? search_probe(a, c - 1) + 1 : a.lo;
            const int hi = c < APP_LANES ? search_probe(a, c) + 1 : a.hi;                // keep the pivot: it may be x itself
            a.lo = lo; a.hi = hi;
        }
    }
    int4 e = make_int4(-1, 0, 0, 0);
    const bool v = a.lo + l < a.hi;
    if (v) e = a.run[a.lo + l];
    const unsigned lt = (__ballot_sync(FULL, v && e.x < x) >> gb) & 0xffu;
    const unsigned eq = (__ballot_sync(FULL, v && e.x == x) >> gb) & 0xffu;
    place = a.lo + __popc(lt);
    const int k = eq ? __ffs(eq) - 1 : 0;
    zw.x = __shfl_sync(FULL, e.z, k, APP_LANES);
    zw.y = __shfl_sync(FULL, e.w, k, APP_LANES);
    return eq ? a.lo + k : -1;
}

// All lanes of the warp call; the eight lanes of a group go `steps` tokens (token(0), ...) down from `node` with child run zw; on
// return node is the node reached or -1.  The eight entries at hand hold the next levels, too, where they are only
// children (most of them are): a token then costs no load.  Long runs are searched.  MOVING: the tree may be changing meanwhile: what
// is found may be wrong, but nothing outside the `limit` entries is read.
template <bool MOVING = false, class F>
__device__ __forceinline__ void group_walk(const int4* ent, int limit, int& node, int2& zw, int steps, int lane, F token) {
    const unsigned FULL = 0xffffffffu;
    const int l = lane & (APP_LANES - 1), gb = lane & ~(APP_LANES - 1);
    int wb = -64, k = 0;
    int4 e = make_int4(-1, 0, 0, 0);
    while (true) {
        bool on = node >= 0 && k < steps;
        if (!__any_sync(FULL, on)) break;
        const int x = on ? token(k) : -1;
        int n = on ? (int)((unsigned)zw.y & RUN_COUNT_MASK) : 0;
        if (MOVING && (zw.x < 0 || zw.x > limit - n)) { n = 0; zw.x = 0; }
        const bool far = n > APP_LANES;
        if (__any_sync(FULL, far)) {
            int place;
            int2 next;
            const int at = group_lookup(RunSearch{ent + zw.x, 0, far ? n : 0}, x, lane, place, next);
            if (far) { node = at >= 0 ? zw.x + at : -1; zw = next; ++k; on = false; }
        }
        if (!__any_sync(FULL, on)) continue;
        if (on && (zw.x < wb || zw.x + n > wb + APP_LANES)) {
            wb = zw.x;
            if (wb + l < limit) e = ent[wb + l];
        }
        const int off = zw.x - wb;
        const unsigned eq = (__ballot_sync(FULL, on && l >= off && l < off + n && e.x == x) >> gb) & 0xffu;
        const int q = eq ? __ffs(eq) - 1 : 0;
        const int nz = __shfl_sync(FULL, e.z, q, APP_LANES), nw = __shfl_sync(FULL, e.w, q, APP_LANES);
        if (on) { node = eq ? wb + q : -1; zw = make_int2(nz, nw); ++k; }
    }
}

// The tokens sh.tok holds: token 0 of the append is sh.tok[APP_SHALLOW - 1].
__device__ __forceinline__ void append_stage_tokens(AppendShared& sh, const int32_t* text, int t_old, const int32_t* newtok, int n_new,
                                                    int tid, int nthreads) {
    for (int i = tid; i < APP_AHEAD + APP_SHALLOW + 2; i += nthreads) {
        const int k = i - (APP_SHALLOW - 1);
        sh.tok[i] = k < 0 ? (t_old + k >= 0 ? text[t_old + k] : -1) : (k < n_new ? newtok[k] : -1);
    }
}

// Whole warps call, `group` of `groups` groups of eight lanes: a group per start position walks APP_SHALLOW
// levels from the root and notes where each token belongs in the run it meets.  Reads the tree only (the
// appending warp may be at work: a place it has changed meanwhile is recognised when the hint is used).
__device__ __forceinline__ void search_ahead(AppendShared& sh, const sd_store& sv, const int4* ent, const int32_t* root, int t_old,
                                             int n_new, int group, int groups, int lane) {
    const int n = min(n_new, APP_AHEAD);
    for (int g0 = 0; g0 < n + APP_SHALLOW - 1; g0 += groups) {
        const int g = g0 + group, k0 = g - (APP_SHALLOW - 1);    // the path starts at token k0 of the append
        const bool on = k0 < n && t_old + k0 >= 0;
        int x = on ? sh.tok[g] : -1;
        int2 zw = make_int2(0, 0);
        bool node = false;
        if (x >= 0 && x < sv.V) {
            const int at = root[x];
            node = at >= 0;
            if (node) zw = *reinterpret_cast<const int2*>(&ent[at].z);
        }
        if ((lane & (APP_LANES - 1)) == 0 && on && k0 >= 0) sh.hint[k0][0] = -1;
#pragma unroll 1
        for (int d = 2; d <= APP_SHALLOW; ++d) {
            const int k = k0 + d - 1;                            // the token that takes the path to depth d
            const bool q = on && k < n;
            x = q ? sh.tok[g + d - 1] : -1;
            // (an entry being written may be read half old, half new: never beyond the pool)
            const bool good = q && node && zw.x >= 0 && (long long)zw.x + ((unsigned)zw.y & RUN_COUNT_MASK) <= sv.spn;
            const RunSearch r{ent + (good ? zw.x : 0), 0, good ? (int)((unsigned)zw.y & RUN_COUNT_MASK) : 0};
            int place;
            int2 next;
            const int at = group_lookup(r, x, lane, place, next);
            if ((lane & (APP_LANES - 1)) == 0 && q && k >= 0) sh.hint[k][d - 1] = node ? place : -1;
            node = at >= 0;
            zw = next;
        }
    }
}

// Place of x in the sorted run ent[cb .. cb + n), and whether it is there.  Whole warp, arguments warp-uniform.
__device__ __forceinline__ int warp_place(const int4* ent, int cb, int n, int x, int lane, bool& there) {
    const unsigned FULL = 0xffffffffu;
    int lo = 0, hi = n;
    while (hi - lo > 32) {
        const int q = lo + (int)(((long long)(hi - lo) * (lane + 1)) / 33);
        const int c = __popc(__ballot_sync(FULL, ent[cb + q].x < x));
        const int below = __shfl_sync(FULL, q, max(c - 1, 0)), at = __shfl_sync(FULL, q, min(c, 31));
        if (c > 0) lo = below + 1;
        if (c < 32) hi = at + 1;                                 // keep the pivot: it may be x itself
    }
    const int t = lo + lane < hi ? ent[cb + lo + lane].x : 0x7fffffff;
    there = __any_sync(FULL, t == x);
    return lo + __popc(__ballot_sync(FULL, t < x));
}

// All 32 lanes of a warp call: appends newtok[0 .. n_new) to the slot's tree and text.  Lane d - 1 holds the
// active node of depth d (act, -1: none) with its child run (cb, w as RUN_UNKNOWN or count | flags | room);
// len / used / live / status are warp-uniform.  A token outside the vocabulary or one the pool or the text buffer
// has no room for ends the append in front of it.  sh.tok is staged; hints are used once
// ahead_warps warps have left theirs.
// FETCH: what the first look for the next token will read in the runs found comes to L2 meanwhile (text with long runs, a
// flushed L2: steps of 64 / 256 requests 117 / 78 -> 109 / 76 us).  Not with four blocks on an SM, which have no
// issue slots to spare (512 requests: 43.3 -> 44.6 us).
template <bool FETCH>
__device__ __forceinline__ void append_tokens(AppendShared& sh, const sd_store& sv, int slot, const int32_t* newtok, int n_new, int ahead_warps,
                                              int lane, int& act, int& cb, unsigned& w, int& len, int& used, int& live, int& status) {
    const unsigned FULL = 0xffffffffu;
    int4* const ent = sv.s_ent + (long long)slot * sv.spn;
    int32_t* const root = sv.s_root + (long long)slot * sv.V;
    int32_t* const text = sv.s_text + (long long)slot * sv.T;
    const int D = sv.D;
    auto token = [&](int k) { return k < APP_AHEAD + 2 ? sh.tok[k + APP_SHALLOW - 1] : (k < n_new ? newtok[k] : -1); };
    auto root_of = [&](int x) { return x >= 0 && x < sv.V ? root[x] : -1; };
    int x1 = len >= 1 ? text[len - 1] : -1, x2 = len >= 2 ? text[len - 2] : -2;
    int x = token(0), xn = token(1);
    // the depth-1 node of the token at hand is read while the tokens before it are being taken
    int r = root_of(x), rn = root_of(xn);
    int4 re = r >= 0 ? ent[r] : make_int4(0, 0, 0, 0);
    bool hints = false;
    for (int k = 0; k < n_new; ++k) {
        if (x < 0 || x >= sv.V) { status |= SD_STATUS_BAD_TOKEN; return; }
        if (len >= sv.T) { status |= SD_STATUS_POOL_FULL; return; }
        const int parent = __shfl_up_sync(FULL, act, 1);         // node of depth `lane`
        int pcb = __shfl_up_sync(FULL, cb, 1);
        unsigned pw = __shfl_up_sync(FULL, w, 1);
        const bool valid = lane <= min(len, D - 1);
        if (!hints && k < APP_AHEAD) hints = *(volatile int*)&sh.ahead == ahead_warps;
        if (r < 0 && (x == x1 || x == x2)) { r = root[x]; if (r >= 0) re = ent[r]; }          // (made by one of the last two tokens)
        else if (r >= 0 && (x == x1 || x == x2)) re = ent[r];    // (its count and run may have changed since it was read)
        int found = -1, place = 0, n = 0, fy = 0, fz = 0;
        unsigned fw = 0;
        if (lane == 0) { found = r; fy = re.y; fz = re.z; fw = (unsigned)re.w; pw = 0; pcb = 0; }
        else if (valid) {
            if (pw == RUN_UNKNOWN) { const int2 zw = *reinterpret_cast<const int2*>(&ent[parent].z); pcb = zw.x; pw = (unsigned)zw.y; }
            n = (int)(pw & RUN_COUNT_MASK);
        }
        int lo = 0, m = n;                                       // the entries to look at
        bool known = true;
        if (n > 4) {
            known = false;
            m = 0;
            if (hints && lane < APP_SHALLOW && k < APP_AHEAD) {
                const int h = sh.hint[k][lane];
                if (h >= 0) { lo = min(max(h - 1, 0), n - 4); m = 4; }
            }
        }
        if (__popc(__ballot_sync(FULL, n > 4 && m == 0)) >= APP_OPEN) {
            // eight parts, probed at their last entries, until at most four entries are left: the first part that does
            // not lie wholly below x
            const bool mine = n > 4 && m == 0;
            int hi = mine ? n : 0;
            while (__any_sync(FULL, hi - lo > 4)) {
                if (hi - lo > 4) {
                    const int step = (hi - lo + 7) >> 3;
                    int below = 0;
#pragma unroll
                    for (int u = 0; u < 7; ++u) {
                        const int q = lo + (u + 1) * step - 1;
                        below += q < hi && ent[pcb + q].x < x ? 1 : 0;
                    }
                    lo += below * step;
                    hi = min(hi, lo + step);
                }
            }
            if (mine) { m = hi - lo; place = lo; known = true; }
        }
        if (m > 0) {
            int t[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) t[u] = u < m ? ent[pcb + lo + u].x : 0x7fffffff;
            int below = 0;
#pragma unroll
            for (int u = 0; u < 4; ++u) below += t[u] < x ? 1 : 0;
            place = lo + below;
#pragma unroll
            for (int u = 0; u < 4; ++u) if (t[u] == x) found = pcb + lo + u;
            // (a hint: the run may have grown since, or be another one by now)
            if (!known) known = found >= 0 || ((lo == 0 || below > 0) && (lo + 4 == n || below < 4));
        }
        unsigned open = __ballot_sync(FULL, !known);
        while (open) {                                           // long runs: the whole warp, one after the other
            const int src = __ffs(open) - 1;
            open &= open - 1;
            const int scb = __shfl_sync(FULL, pcb, src);
            bool there;
            const int at = warp_place(ent, scb, __shfl_sync(FULL, n, src), x, lane, there);
            if (lane == src) { place = at; found = there ? scb + at : -1; }
        }
        if (lane > 0 && found >= 0) { const int4 fe = ent[found]; fy = fe.y; fz = fe.z; fw = (unsigned)fe.w; }
        const int next_parent = __shfl_down_sync(FULL, parent, 1);
        // on to the next token's depth-1 node
        const int xnn = token(k + 2);
        const int rnn = root_of(xnn);
        const int4 ren = rn >= 0 ? ent[rn] : make_int4(0, 0, 0, 0);

        const bool need = valid && found < 0;
        const unsigned needs = __ballot_sync(FULL, need);
        int new_act = found, new_cb = fz;
        unsigned new_w = fw;
        if (found >= 0) {
            *word(&ent[found], 1) = fy + 1;
            if (lane < 31 && next_parent == found) new_w = RUN_UNKNOWN;      // the next lane may be editing this very node's run
            else if (FETCH && (fw & RUN_COUNT_MASK)) {
                const int nn = (int)(fw & RUN_COUNT_MASK), step = (nn + 7) >> 3;
                asm volatile("prefetch.global.L2 [%0];" ::"l"(ent + fz));
                if (nn > 4 && lane >= APP_SHALLOW - 1)
#pragma unroll
                    for (int u = 0; u < 7; ++u)
                        if ((u + 1) * step <= nn) asm volatile("prefetch.global.L2 [%0];" ::"l"(ent + fz + (u + 1) * step - 1));
            }
        } else { new_cb = 0; new_w = 0; }
        if (needs) {
            const unsigned room = lane == 0 ? 0u : (pw >> ROOM_SHIFT) & ROOM_MASK;
            const unsigned rw = pw & ~(ROOM_MASK << ROOM_SHIFT);
            const bool leaf = need && n == 0;                    // first child of a leaf, or a new depth-1 node
            int asz = 0;                                         // fresh entries this lane needs
            if (leaf) asz = room > 0u ? 0 : D - lane;            // continue the chain block behind the parent, or start one
            else if (need && (uint32_t)n == sd_run_capacity(rw)) asz = (int)sd_pow2ceil((uint32_t)n + 1u);
            int fresh = parent + 1;
            if (__any_sync(FULL, asz > 0)) {
                int inc = asz;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int y = __shfl_up_sync(FULL, inc, o);
                    if (lane >= o) inc += y;
                }
                const int total = __shfl_sync(FULL, inc, 31);
                if ((long long)used + total > (long long)sv.spn) {
                    // nothing of this token stays: the counts raised above go back
                    if (found >= 0) *word(&ent[found], 1) = fy;
                    status |= SD_STATUS_POOL_FULL;
                    return;
                }
                if (asz > 0) fresh = used + inc - asz;
                used += total;
            }
            if (leaf) new_w = (asz > 0 ? (unsigned)(asz - 1) : room - 1u) << ROOM_SHIFT;
            // (the nodes of suffixes of one another: leaves are the deepest lanes' parents)
            if (leaf) {
                ent[fresh] = make_int4(x, 1, 0, 0);
                if (lane == 0) root[x] = fresh;
                else *reinterpret_cast<int2*>(&ent[parent].z) = make_int2(fresh, 1);
                new_act = fresh;
            }
            unsigned runs = __ballot_sync(FULL, need && !leaf);
            if (runs) {
                // A tail that repeats one token is the only case in which a run to be edited holds the parent of the next
                // lane: the deeper lane goes first.
                const bool moves = asz > 0;
                const unsigned clash = __ballot_sync(FULL, need && next_parent >= pcb && next_parent < pcb + n);
                // A run of one or two children, most of those that grow: its lane lays it down with the new child.  (Through the warp as
                // the others: steps of 512 requests of text without repeats 3 % longer, of one agent 1 %.  Runs of up to four by their lanes: 1 %.)
                const bool own = need && !leaf && n <= 2 && !((clash >> lane) & 1u);
                if (own) {
                    const int4 e0 = ent[pcb], e1 = n > 1 ? ent[pcb + 1] : e0;             // (such a run is always full: it moves)
                    ent[fresh + (place == 0 ? 1 : 0)] = e0;
                    if (n > 1) ent[fresh + (place <= 1 ? 2 : 1)] = e1;
                    ent[fresh + place] = make_int4(x, 1, 0, 0);
                    *word(&ent[parent], 2) = fresh;
                    *word(&ent[parent], 3) = n + 1;
                    new_act = fresh + place;
                }
                runs = __ballot_sync(FULL, need && !leaf && !own);
                const unsigned big = __ballot_sync(FULL, need && (moves ? n : n - place) > APP_BIG);
                __syncwarp();
                while (runs) {
                    const int top = 31 - __clz((int)runs);
                    unsigned batch = 0;
                    int mine = -1, took = 0;
                    while (runs && took < 4) {
                        const int src = 31 - __clz((int)runs);
                        if (took > 0 && ((((clash >> src) & 1u) && ((batch >> (src + 1)) & 1u)) || ((big >> src) & 1u))) break;
                        if ((lane >> 3) == took) mine = src;
                        batch |= 1u << src;
                        runs &= ~(1u << src);
                        ++took;
                        if ((big >> src) & 1u) break;
                    }
                    if (took == 1) {
                        const int idx = insert_child_warp(ent, __shfl_sync(FULL, parent, top), __shfl_sync(FULL, pcb, top), __shfl_sync(FULL, n, top),
                                                          __shfl_sync(FULL, place, top), x, __shfl_sync(FULL, fresh, top),
                                                          __shfl_sync(FULL, moves ? 1 : 0, top) != 0, lane);
                        if (lane == top) new_act = idx;
                    } else {
                        const int idx = insert_child_groups(ent, mine, parent, pcb, n, place, x, fresh, moves, lane);
                        // the lanes of the batch take theirs, the deepest from the first group
                        const int at = __shfl_sync(FULL, idx, 8 * (__popc(batch >> 1 >> lane) & 3));
                        if ((batch >> lane) & 1u) new_act = at;
                    }
                }
            }
            live += __popc(needs);
        }
        __syncwarp();
        act = valid ? new_act : -1;
        cb = valid ? new_cb : 0;
        w = valid ? new_w : 0u;
        if (lane == 0) text[len] = x;
        ++len;
        x2 = x1; x1 = x; x = xn; xn = xnn;
        r = rn; re = ren; rn = rnn;
    }
}

// SlotState's fields to and from the registers of append_tokens.
__device__ __forceinline__ unsigned append_pack(unsigned run_w, int room) { return run_w == RUN_UNKNOWN ? run_w : run_w | ((unsigned)room << ROOM_SHIFT); }
__device__ __forceinline__ void append_store(SlotState* ss, int lane, int act, int cb, unsigned w) {
    ss->active[lane] = act; ss->run_cb[lane] = cb;
    ss->room[lane] = w == RUN_UNKNOWN ? 0 : (int)((w >> ROOM_SHIFT) & ROOM_MASK);
    ss->run_w[lane] = w == RUN_UNKNOWN ? w : w & ~(ROOM_MASK << ROOM_SHIFT);
}

}  // namespace
