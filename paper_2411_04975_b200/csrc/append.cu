// sd_append: the batched append kernel for the per-request trees (see append_core.cuh for how one
// token is appended) and the insert of whole sequences into the global tree.
#include <atomic>

#include <cooperative_groups.h>

#include "append_core.cuh"
#include "device_memory.h"
#include "global_insert.cuh"
#include "suffix_order.cuh"

namespace cg = cooperative_groups;

namespace {

// ---------------------------------------------------------------------------------------------
// Global online insert (a finished request's output goes into the global tree).
//
// Inserting a sequence adds one occurrence to every string of at most D tokens that starts at one
// of its positions: one root-to-depth-D PATH per start position.  Up to 2,016 positions are taken at once, in one
// launch:
//   1. every path goes down the tree as far as it exists, eight lanes each, and raises the counts on its way (no path
//      waits for another: nothing moves yet).  Meanwhile one block sorts the positions' suffixes;
//   2. the sorted suffixes and their common prefixes are a trie of the whole batch.  Its nodes deeper than the walk
//      came are new.  They are laid down in pre-order in one stretch of the pool, by the sweeps that build
//      a tree offline (see build.cu: a lane per depth), with the depth the walk reached taking the place of the root:
//      counts, children and places follow from running state per depth.  EVENTS are the new nodes whose parent
//      exists;
//   3. events are grouped by parent, and every parent's run is merged once with all its new children (in place, or
//      into a roomier run), while the rest of the new nodes is written;
//   4. every parent's entry gets its new run, in the place it has now if its own run was merged, too.
// Six barriers and no rounds: the time is that of the walk (dependent loads) or of the sort, whichever is
// longer, and of the sweeps over the tiles.  (Level by level with an election per parent and round, by a cluster of 8
// blocks: 150 us for 352 paths, 58 for 91; now 56 and 42, of which the walk 16 and 12, grouping 8 and 6.)
// The nodes that a batch adds need the pool to hold them all: a batch that does not fit raises counts only.
// A cluster of 16 blocks, which meet at the hardware's barrier, where the device has room for one; else 24 blocks that meet at a grid
// barrier (1.5 us each).  Services of 16 / 32 requests 2,651 / 1,975 us with the grid, 2,482 / 1,847 with the cluster; of 256, whose
// batches its 960 walks at a time often take two rounds for, 11,725 either way.
constexpr int GI_CLUSTER = 16, GI_GRID = 24;
constexpr int GI_THREADS = 512;               // (1,024 leave 64 registers: the sweeps spill)
constexpr int GI_ITEMS = 256;
constexpr int GI_CELLS = 2 * GI_MAX;
constexpr int GI_BIG = 256;                   // runs longer than this are merged by a whole block

struct GiItems {
    int item[GI_ITEMS];
    long long begin[GI_ITEMS], end[GI_ITEMS], pref[GI_ITEMS + 1];
    int n_items;
};

struct GiSort {                               // block 0, while it sorts
    unsigned char order[block_order_smem<GI_THREADS, GI_MAX / GI_THREADS>()];
    int tok[GI_MAX];
    unsigned short begin[GI_MAX], end[GI_MAX], sa[GI_MAX];
};
struct GiTable {                              // block 0, while it groups
    int key[GI_CELLS];                        // parent + 2, 0 = free
    int cnt[GI_CELLS];                        // events
    int at[GI_CELLS];                         // first place | group << 16
    int tok[GI_MAX], ev[GI_MAX];
    int n_big;
};
__host__ __device__ constexpr int gi_warp_tiles(int blocks) { return ((GI_REAL + GI_TILE - 1) / GI_TILE + blocks - 2) / (blocks - 1); }  // tiles per block
static_assert(gi_warp_tiles(GI_CLUSTER) <= GI_THREADS / 32 && gi_warp_tiles(GI_GRID) <= GI_THREADS / 32, "a warp per tile");
template <int BLOCKS>
struct GiSweep {                              // the other blocks
    int2 state[gi_warp_tiles(BLOCKS)][GI_TILE][32];   // state from behind, by suffix of a tile and depth
    int f[GI_TILES][32], e[GI_TILES][32];     // of all tiles; f then r
    int s[GI_TILES], ev[GI_TILES];
};
template <int BLOCKS>
union GiShared {
    GiSort sort;
    GiTable table;
    GiSweep<BLOCKS> sweep;
};

// exclusive sum over the block's threads, the total in `all`
__device__ __forceinline__ int gi_block_scan(int v, int* wsum, int tid, int& all) {
    const unsigned FULL = 0xffffffffu;
    const int lane = tid & 31, wib = tid >> 5;
    int inc = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(FULL, inc, o);
        if (lane >= o) inc += y;
    }
    if (lane == 31) wsum[wib] = inc;
    __syncthreads();
    const int c = lane < GI_THREADS / 32 ? wsum[lane] : 0;
    const int before = (int)__reduce_add_sync(FULL, lane < wib ? (unsigned)c : 0u);
    all = (int)__reduce_add_sync(FULL, (unsigned)c);
    __syncthreads();
    return before + inc - v;
}

__device__ __forceinline__ int gi_item_of(const GiItems& I, long long p) {
    int lo = 0, hi = I.n_items - 1;                              // last item whose prefix is <= p
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (I.pref[mid] <= p) lo = mid; else hi = mid - 1;
    }
    return lo;
}

// 1. the paths from positions [0, m) of the pass that starts at c0
__device__ void gi_walk(const sd_store& sv, GiScratch* X, const GiItems& I, const int32_t* d_tokens, long long c0, int m, int group,
                        int groups, int lane) {
    const unsigned FULL = 0xffffffffu;
    const int l = lane & (APP_LANES - 1), gb = lane & ~(APP_LANES - 1), D = sv.D;
    int4* const ent = sv.g_ent;
    for (int p0 = 0; p0 < m; p0 += groups) {                     // (uniform for the warp)
        const int p = p0 + group;
        const bool mine = p < m;
        const int32_t* tp = d_tokens;
        int len = 0;
        if (mine) {
            const int it = gi_item_of(I, c0 + p);
            const long long k = I.begin[it] + (c0 + p - I.pref[it]);
            tp = d_tokens + k;
            len = (int)min((long long)D, I.end[it] - k);
        }
        int node = -1, prev = -1, v = 0, wb = -64;
        int2 zw = make_int2(0, 0);
        int4 e = make_int4(-1, 0, 0, 0);
        if (mine) {
            node = sv.g_root[tp[0]];
            if (node >= 0) {
                zw = *reinterpret_cast<const int2*>(&ent[node].z);
                v = 1;
                if (l == 0) atomicAdd(word(&ent[node], 1), 1);
            }
        }
        bool alive = node >= 0;
        while (true) {
            const bool on = alive && v < len;
            if (!__any_sync(FULL, on)) break;
            const int x = on ? tp[v] : -1;
            const int n = on ? (int)((unsigned)zw.y & RUN_COUNT_MASK) : 0;
            const bool far = n > APP_LANES;
            int at = -1;
            int2 next = make_int2(0, 0);
            if (__any_sync(FULL, far)) {
                int place;
                int2 fz;
                const int q = group_lookup(RunSearch{ent + zw.x, 0, far ? n : 0}, x, lane, place, fz);
                if (far && q >= 0) { at = zw.x + q; next = fz; }
            }
            const bool near = on && !far;
            if (__any_sync(FULL, near)) {
                if (near && (zw.x < wb || zw.x + n > wb + APP_LANES)) {
                    wb = zw.x;
                    if (wb + l < (int)sv.g_cap) e = ent[wb + l];
                }
                const int off = zw.x - wb;
                const unsigned eq = (__ballot_sync(FULL, near && l >= off && l < off + n && e.x == x) >> gb) & 0xffu;
                const int q = eq ? __ffs(eq) - 1 : 0;
                const int nz = __shfl_sync(FULL, e.z, q, APP_LANES), nw = __shfl_sync(FULL, e.w, q, APP_LANES);
                if (near && eq) { at = wb + q; next = make_int2(nz, nw); }
            }
            if (on) {
                if (at < 0) alive = false;
                else {
                    if (l == 0) {
                        atomicAdd(word(&ent[at], 1), 1);
                        // a count changes: the copies in the run's top block (if any) are stale from now on
                        if ((unsigned)zw.y & RUN_HAS_TOP) atomicAnd(word(&ent[node], 3), (int)~RUN_HAS_TOP);
                    }
                    prev = node; node = at; zw = next;
                    ++v;
                }
            }
        }
        if (mine && l == 0) { X->v[p] = v; X->p[p] = node; X->q[p] = prev; }
    }
}

// 2. The sweeps: a warp per tile of GI_TILE suffixes, a lane per depth.  A lane also looks after the tile's suffix of its number.
// What a sweep waits for are reads of what other blocks have just written (about 1,500 cycles behind a grid barrier), so
// everything about a tile's suffixes is read once and kept in registers, and what the tiles leave for one another comes
// into shared memory in one go.
struct GiOwn {
    int lnv;                                  // common prefix, length, levels that exist: packed
    int at;                                   // start position
    int below, event;                         // new nodes whose parent is new, whose parent exists
    int p, q, ptok, xtok;                     // of the event: the parent, the node above it, the parent's token and its own
    int tok[GI_TILE];                         // token of this lane's depth, by suffix of the tile
};

__device__ __forceinline__ void gi_own(GiOwn& o, const GiScratch* X, int j0, int mm, int lane) {
    const unsigned FULL = 0xffffffffu;
    o.lnv = 0; o.at = 0; o.below = 0; o.event = 0; o.p = -1; o.q = -1; o.ptok = -1; o.xtok = 0;
    if (lane < mm) {
        o.at = X->sa[j0 + lane];
        const int l = X->lcp[j0 + lane], n = X->len[j0 + lane], v = X->v[o.at];
        o.p = X->p[o.at]; o.q = X->q[o.at];
        o.lnv = l | (n << 8) | (v << 16);
        o.below = max(0, n - max(l, v + 1));
        o.event = l <= v && v < n ? 1 : 0;
    }
#pragma unroll
    for (int i = 0; i < GI_TILE; ++i) {
        const int at = __shfl_sync(FULL, o.at, i), x = __shfl_sync(FULL, o.lnv, i);
        o.tok[i] = lane < ((x >> 8) & 255) ? X->tok[at + lane] : 0;
        const int v = x >> 16, t1 = __shfl_sync(FULL, o.tok[i], min(v, 31)), t0 = __shfl_sync(FULL, o.tok[i], max(v - 1, 0));
        if (lane == i) { o.xtok = t1; o.ptok = v > 0 ? t0 : -1; }
    }
}

// what the tile does to the state from behind: children counted up to the first reset, and where that is
__device__ __forceinline__ void gi_sweep_tile(GiScratch* X, const GiOwn& o, int t, int m, int lane) {
    const unsigned FULL = 0xffffffffu;
    const int j0 = t * GI_TILE, mm = min(GI_TILE, m - j0), d = lane + 1;
    int cnt = 0, first = m;
    bool seen = false;
#pragma unroll 1
    for (int i = 0; i < mm; ++i) {
        const int x = __shfl_sync(FULL, o.lnv, i), l = x & 255, len = (x >> 8) & 255;
        if (!seen) {
            cnt += l == d && len > l ? 1 : 0;
            if (l < d) { seen = true; first = j0 + i; }
        }
    }
    X->f[t][lane] = cnt | (seen ? (int)0x80000000 : 0);
    X->e[t][lane] = first;
    const int sb = (int)__reduce_add_sync(FULL, (unsigned)o.below), se = (int)__reduce_add_sync(FULL, (unsigned)o.event);
    if (lane == 0) { X->s[t] = sb; X->ev[t] = se; }
}

// sums over the first t tiles
__device__ __forceinline__ void gi_sums(const int* s, const int* ev, int t, int lane, int& a, int& b) {
    a = 0; b = 0;
    for (int q = lane; q < t; q += 32) { a += s[q]; b += ev[q]; }
    a = (int)__reduce_add_sync(0xffffffffu, (unsigned)a);
    b = (int)__reduce_add_sync(0xffffffffu, (unsigned)b);
}

// from behind: the events, the end of the last run opened per depth, and the state at every suffix.  s_own: new nodes with a
// new parent in front of the lane's suffix.
template <class Sweep>
__device__ __forceinline__ void gi_sweep_runs(GiScratch* X, Sweep& sw, const GiOwn& o, int wib, int t, int tiles, int m, int lane,
                                              int& s_own) {
    const unsigned FULL = 0xffffffffu;
    const int j0 = t * GI_TILE, mm = min(GI_TILE, m - j0), d = lane + 1;
    int s_at, ev_at;
    gi_sums(sw.s, sw.ev, t, lane, s_at, ev_at);
    int is = o.below, ie = o.event;
#pragma unroll
    for (int k = 1; k < GI_TILE; k <<= 1) {
        const int a = __shfl_up_sync(FULL, is, k), b = __shfl_up_sync(FULL, ie, k);
        if (lane >= k) { is += a; ie += b; }
    }
    s_own = s_at + is - o.below;
    const int ev_own = ev_at + ie - o.event;
    if (o.event) { X->ev_p[ev_own] = o.p; X->ev_q[ev_own] = o.q; X->ev_ptok[ev_own] = o.ptok; X->ev_tok[ev_own] = o.xtok; }
    int F = 0, e = m;
    for (int q = t + 1; q < tiles; ++q) {
        const int fq = sw.f[q][lane];
        F += fq & 0x7fffffff;
        if (fq < 0) { e = sw.e[q][lane]; break; }
    }
    __syncwarp();
    int g = F;
#pragma unroll
    for (int k = 1; k < 32; k <<= 1) {
        const int y = __shfl_up_sync(FULL, g, k);
        if (lane >= k) g += y;
    }
    g -= F;                                                      // G: children of the levels above
    int R = -1;
#pragma unroll 1
    for (int i = mm - 1; i >= 0; --i) {
        const int x = __shfl_sync(FULL, o.lnv, i), l = x & 255, len = (x >> 8) & 255, v = x >> 16;
        const int si = __shfl_sync(FULL, s_own, i), ei = __shfl_sync(FULL, ev_own, i);
        sw.state[wib][i][lane] = make_int2(g, e);
        const int up = __shfl_down_sync(FULL, g, 1), gv = __shfl_sync(FULL, g, min(v, 31));
        const int kids = (lane == 31 ? 0 : up - g) + (d < len ? 1 : 0);
        const int run = si + d - max(l, v + 1) + g - gv;
        const bool opens = d > max(l, v) && d <= len;
        if (opens && R < 0) R = run + kids;
        if (opens && l <= v && d == v + 1) { X->ev_cnt[ei] = e - (j0 + i); X->ev_run[ei] = run; X->ev_kids[ei] = kids; }
        const int step = __shfl_sync(FULL, g, min(l, 31)) + (len > l ? 1 : 0);
        if (d > l) { g = l == 0 ? 0 : step; e = j0 + i; }
    }
    X->r[t][lane] = R;
}

// from the front: the new nodes below the events, from entry `used` on (sw.f holds what the tiles left in r)
template <class Sweep>
__device__ __forceinline__ void gi_sweep_emit(const Sweep& sw, const GiOwn& o, int4* ent, int used, int wib, int t, int m, int lane,
                                              int s_own) {
    const unsigned FULL = 0xffffffffu;
    const int j0 = t * GI_TILE, mm = min(GI_TILE, m - j0), d = lane + 1;
    int R = -1;
    for (int q = t - 1; q >= 0 && R < 0; --q) R = sw.f[q][lane];
    __syncwarp();
#pragma unroll
    for (int i = 0; i < GI_TILE; ++i) {
        if (i >= mm) break;
        const int x = __shfl_sync(FULL, o.lnv, i), l = x & 255, len = (x >> 8) & 255, v = x >> 16;
        const int si = __shfl_sync(FULL, s_own, i);
        const int2 ge = sw.state[wib][i][lane];
        const int up = __shfl_down_sync(FULL, ge.x, 1), gv = __shfl_sync(FULL, ge.x, min(v, 31));
        const int later = lane == 31 ? 0 : up - ge.x, kids = later + (d < len ? 1 : 0);
        const int run = si + d - max(l, v + 1) + ge.x - gv;
        const bool opens = d > max(l, v) && d <= len;
        // the entry of the next depth's node: this node's first child, or the next of its other children
        const int place = __shfl_up_sync(FULL, opens ? run : R - 1 - later, 1);
        if (opens) R = run + kids;
        if (opens && !(l <= v && d == v + 1))
            ent[used + place] = make_int4(o.tok[i], ge.y - (j0 + i), kids > 0 ? used + run : 0, kids > 0 ? (int)((unsigned)kids | RUN_STATIC) : 0);
    }
}

// 3. the events by parent (one block): every parent's new children by token, its run's new place
__device__ __forceinline__ void gi_group(const sd_store& sv, GiScratch* X, GiTable& tb, int* wsum, int used, int s_all, int ev_all, int tid) {
    int4* const ent = sv.g_ent;
    for (int i = tid; i < GI_CELLS; i += GI_THREADS) { tb.key[i] = 0; tb.cnt[i] = 0; }
    if (tid == 0) tb.n_big = 0;
    __syncthreads();
    auto cell_of = [&](int key, bool insert) {
        int c = (int)(((unsigned)key * 2654435761u) >> 20) & (GI_CELLS - 1);
        for (int probe = 0; probe < GI_CELLS; ++probe) {
            const int old = insert ? atomicCAS(&tb.key[c], 0, key) : tb.key[c];
            if (old == key || (insert && old == 0)) return c;
            if (old == 0) return -1;
            c = (c + 1) & (GI_CELLS - 1);
        }
        return -1;
    };
    constexpr int PER = GI_MAX / GI_THREADS;
    int cell[PER], at[PER], x[PER];
#pragma unroll
    for (int u = 0; u < PER; ++u) {
        const int e = tid + u * GI_THREADS;
        cell[u] = -1; at[u] = 0; x[u] = 0;
        if (e < ev_all) {
            x[u] = X->ev_tok[e];
            cell[u] = cell_of(X->ev_p[e] + 2, true);
            at[u] = atomicAdd(&tb.cnt[cell[u]], 1);
        }
    }
    __syncthreads();
    constexpr int CELLS = GI_CELLS / GI_THREADS;
    int sum = 0, groups = 0, all, n_groups;
#pragma unroll
    for (int u = 0; u < CELLS; ++u) { const int c = tb.cnt[tid * CELLS + u]; sum += c; groups += c > 0 ? 1 : 0; }
    int first = gi_block_scan(sum, wsum, tid, all), id = gi_block_scan(groups, wsum, tid, n_groups);
#pragma unroll
    for (int u = 0; u < CELLS; ++u) {
        const int c = tb.cnt[tid * CELLS + u];
        tb.at[tid * CELLS + u] = first | (id << 16);
        first += c; id += c > 0 ? 1 : 0;
    }
    __syncthreads();
#pragma unroll
    for (int u = 0; u < PER; ++u)
        if (cell[u] >= 0) { const int p = (tb.at[cell[u]] & 0xffff) + at[u]; tb.tok[p] = x[u]; tb.ev[p] = tid + u * GI_THREADS; }
    __syncthreads();
#pragma unroll
    for (int u = 0; u < PER; ++u)
        if (cell[u] >= 0) {                          // tokens of one parent's events are distinct
            const int p = tb.at[cell[u]] & 0xffff, k = tb.cnt[cell[u]];
            int rank = 0;
            for (int q = 0; q < k; ++q) rank += tb.tok[p + q] < x[u] ? 1 : 0;
            X->m_tok[p + rank] = x[u]; X->m_ev[p + rank] = tid + u * GI_THREADS;
        }
    __syncthreads();                                             // (the counts have been read: they become sizes)
    int mine_size = 0;
#pragma unroll 1
    for (int u = 0; u < CELLS; ++u) {
        const int c = tid * CELLS + u, k = tb.cnt[c];
        if (k == 0) continue;
        GiGroup G;
        const int id = tb.at[c] >> 16;
        G.first = tb.at[c] & 0xffff; G.k = k;
        const int e = tb.ev[G.first], q = X->ev_q[e];
        G.parent = tb.key[c] - 2; G.parent_tok = X->ev_ptok[e];
        G.cb = 0; G.n = 0; G.above = -1; G.base = 0;
        int size = 0;
        if (G.parent >= 0) {
            const int4 pe = __ldcg(ent + G.parent);
            G.cb = pe.z; G.n = (int)((unsigned)pe.w & RUN_COUNT_MASK);
            if ((uint32_t)(G.n + k) > sd_run_capacity((uint32_t)pe.w)) size = (int)sd_pow2ceil((uint32_t)(G.n + k));
            if (q >= 0) { const int qc = cell_of(q + 2, false); if (qc >= 0) G.above = tb.at[qc] >> 16; }
        } else size = k;
        if (G.n > GI_BIG || k > GI_BIG) X->big[atomicAdd(&tb.n_big, 1)] = id;
        X->group[id] = G;
        tb.cnt[c] = size;                                        // (only this thread looks at this cell's count)
        mine_size += size;
    }
    int entries, place = used + s_all + gi_block_scan(mine_size, wsum, tid, entries);
#pragma unroll 1
    for (int u = 0; u < CELLS; ++u) {
        const int c = tid * CELLS + u, size = tb.cnt[c];
        if (tb.key[c] == 0) continue;
        GiGroup* const G = &X->group[tb.at[c] >> 16];
        G->base = size > 0 ? place : G->cb;
        place += size;
    }
    if (tid == 0) {
        X->n_groups = n_groups; X->n_big = tb.n_big; X->entries = entries;
        X->fits = (long long)used + s_all + entries <= sv.g_cap ? 1 : 0;
    }
}

// 3. one parent's run with its new children, by a team of T threads (a warp or a block)
template <int T, class Sync>
__device__ __forceinline__ void gi_merge(const sd_store& sv, const GiScratch* X, int* m_pos, const GiGroup& g, int base0, int t, Sync sync) {
    constexpr int U = 4;
    int4* const ent = sv.g_ent;
    const int* const tok = X->m_tok + g.first;
    int* const pos = m_pos + g.first;
    // where the new children belong
    for (int r = t; r < g.k; r += T) {
        int lo = 0, hi = g.n;
        while (lo < hi) { const int mid = (lo + hi) >> 1; if (__ldcg(&ent[g.cb + mid].x) < tok[r]) lo = mid + 1; else hi = mid; }
        pos[r] = lo;
    }
    sync();
    auto before = [&](int x) {                                   // new children in front of token x
        int lo = 0, hi = g.k;
        while (lo < hi) { const int mid = (lo + hi) >> 1; if (tok[mid] < x) lo = mid + 1; else hi = mid; }
        return lo;
    };
    if (g.parent >= 0 && g.base != g.cb) {
        for (int i0 = t; i0 < g.n; i0 += T * U) {
            int4 e[U];
#pragma unroll
            for (int u = 0; u < U; ++u) if (i0 + u * T < g.n) e[u] = __ldcg(ent + g.cb + i0 + u * T);
#pragma unroll
            for (int u = 0; u < U; ++u) if (i0 + u * T < g.n) ent[g.base + i0 + u * T + before(e[u].x)] = e[u];
        }
    } else if (g.parent >= 0) {
        const int stop = pos[0];
        for (int hi = g.n; hi > stop; hi -= T * U) {             // from the top down, a chunk at a time
            const int lo = max(stop, hi - T * U);
            int4 e[U];
#pragma unroll
            for (int u = 0; u < U; ++u) if (lo + t + u * T < hi) e[u] = __ldcg(ent + g.cb + lo + t + u * T);
            sync();
#pragma unroll
            for (int u = 0; u < U; ++u) if (lo + t + u * T < hi) ent[g.cb + lo + t + u * T + before(e[u].x)] = e[u];
            sync();
        }
    }
    for (int r = t; r < g.k; r += T) {
        const int ev = X->m_ev[g.first + r], kids = X->ev_kids[ev], at = g.base + pos[r] + r;
        ent[at] = make_int4(tok[r], X->ev_cnt[ev], kids > 0 ? base0 + X->ev_run[ev] : 0, kids > 0 ? (int)((unsigned)kids | RUN_STATIC) : 0);
        if (g.parent < 0) sv.g_root[tok[r]] = at;
    }
    sync();
}

template <int GI_BLOCKS>
__global__ void __launch_bounds__(GI_THREADS, 1)
global_insert_kernel(sd_store sv, int n, const int32_t* d_slot, const int64_t* d_offsets, const int32_t* d_tokens, int tok_bits) {
    extern __shared__ __align__(16) unsigned char gi_smem[];
    __shared__ GiItems I;
    __shared__ int wsum[GI_THREADS / 32];
    const unsigned FULL = 0xffffffffu;
    const int tid = threadIdx.x, lane = tid & 31, wib = tid >> 5, blk = (int)blockIdx.x;
    const int D = sv.D;
    int4* const ent = sv.g_ent;
    GiScratch* const X = sv.gi;
    GiShared<GI_BLOCKS>& sh = *reinterpret_cast<GiShared<GI_BLOCKS>*>(gi_smem);
    auto meet = [] { if constexpr (GI_BLOCKS == GI_CLUSTER) cluster_sync(); else cg::this_grid().sync(); };

    // (every block looks at all items: all blocks take the same way)
    bool mine = false;
    for (int i = tid; i < n; i += GI_THREADS) mine |= d_slot[i] == -1;
    if (!__syncthreads_or(mine)) return;                         // the usual decode step: nothing for the global tree
    bool full = (sv.g_state->status & SD_STATUS_GLOBAL_FULL) != 0, bad = false, again = false;
    int used = sv.g_state->used, live = 0;
    long long tokens_done = 0;

    for (int base = 0; base < n && !full; base += GI_ITEMS) {
        // the sequences among items [base, base + GI_ITEMS), in item order
        __syncthreads();
        if (tid == 0) I.n_items = 0;
        __syncthreads();
        if (tid < 32) {
            for (int i0 = 0; i0 < GI_ITEMS; i0 += 32) {
                const int i = base + i0 + lane;
                const bool is = i < n && d_slot[i] == -1;
                const unsigned m = __ballot_sync(FULL, is);
                if (is) I.item[I.n_items + __popc(m & ((1u << lane) - 1u))] = i;
                __syncwarp();
                if (lane == 0) I.n_items += __popc(m);
                __syncwarp();
            }
        }
        __syncthreads();
        const int n_items = I.n_items;
        if (n_items == 0) continue;
        for (int j = tid; j < n_items; j += GI_THREADS) { I.begin[j] = d_offsets[I.item[j]]; I.end[j] = d_offsets[I.item[j] + 1]; }
        __syncthreads();
        // a token outside the vocabulary ends its sequence there
        for (int j = 0; j < n_items; ++j) {
            const long long b = I.begin[j], e = d_offsets[I.item[j] + 1];
            for (long long k = b + tid; k < e; k += GI_THREADS) {
                const int x = d_tokens[k];
                if (x < 0 || x >= sv.V) { atomicMin(&I.end[j], k); bad = true; }
            }
        }
        __syncthreads();
        if (tid == 0) {
            long long acc = 0;
            for (int j = 0; j < n_items; ++j) { I.pref[j] = acc; acc += max(I.end[j] - I.begin[j], 0ll); }
            I.pref[n_items] = acc;
        }
        __syncthreads();
        const long long total = I.pref[n_items];

        for (long long c0 = 0; c0 < total && !full; c0 += GI_REAL) {
            if (again) meet();                                   // the pass before is over
            again = true;
            const int m = (int)min((long long)GI_REAL, total - c0);
            // ---------------- 1. walk, and sort
            if (blk == 0) {
                // (the last sequence's next tokens, as far as the paths reach)
                const int M = m + (int)min((long long)(D - 1), I.pref[gi_item_of(I, c0 + m - 1) + 1] - (c0 + m));
                GiSort& so = sh.sort;
                for (int i = tid; i < M; i += GI_THREADS) {
                    const int it = gi_item_of(I, c0 + i);
                    const int x = d_tokens[I.begin[it] + (c0 + i - I.pref[it])];
                    so.tok[i] = x; X->tok[i] = x;
                    so.begin[i] = (unsigned short)max(I.pref[it] - c0, 0ll);
                    so.end[i] = (unsigned short)min(I.pref[it + 1] - c0, (long long)M);
                }
                __syncthreads();
                auto token = [&](int i) { return so.tok[i]; };
                auto begin = [&](int i) { return (int)so.begin[i]; };
                auto end = [&](int i) { return (int)so.end[i]; };
                const unsigned short* order;
                if (M <= GI_THREADS) order = block_suffix_order<GI_THREADS, 1>(so.order, wsum, M, tok_bits, D, token, begin, end);
                else order = block_suffix_order<GI_THREADS, GI_MAX / GI_THREADS>(so.order, wsum, M, tok_bits, D, token, begin, end);
                // start positions only
                int at = 0;
                for (int i0 = 0; i0 < M; i0 += GI_THREADS) {
                    const int i = i0 + tid;
                    const int q = i < M ? order[i] : GI_MAX;
                    int all;
                    const int k = at + gi_block_scan(q < m ? 1 : 0, wsum, tid, all);
                    if (q < m) { so.sa[k] = (unsigned short)q; X->sa[k] = q; }
                    at += all;
                }
                __syncthreads();
                for (int j = tid; j < m; j += GI_THREADS) {
                    const int q = so.sa[j], len = min(D, so.end[q] - q);
                    int l = 0;
                    if (j > 0) {
                        const int h = so.sa[j - 1], most = min(len, min(D, so.end[h] - h));
                        while (l < most && so.tok[q + l] == so.tok[h + l]) ++l;
                    }
                    X->lcp[j] = l; X->len[j] = len;
                }
            } else {
                gi_walk(sv, X, I, d_tokens, c0, m, tid / APP_LANES * (GI_BLOCKS - 1) + blk - 1,
                        (GI_BLOCKS - 1) * GI_THREADS / APP_LANES, lane);
            }
            meet();
            // ---------------- 2. the sweeps, a warp per tile
            const int tiles = (m + GI_TILE - 1) / GI_TILE, t = (blk - 1) + wib * (GI_BLOCKS - 1);
            const bool sweeps = blk > 0 && t < tiles;
            GiOwn own;
            int s_own = 0;
            if (sweeps) {
                gi_own(own, X, t * GI_TILE, min(GI_TILE, m - t * GI_TILE), lane);
                gi_sweep_tile(X, own, t, m, lane);
            }
            meet();
            int s_all, ev_all;
            if (blk == 0) gi_sums(X->s, X->ev, tiles, lane, s_all, ev_all);
            else {
                auto& sw = sh.sweep;
                for (int i = tid; i < tiles * 8; i += GI_THREADS) {                 // (four depths at a time)
                    reinterpret_cast<int4*>(sw.f)[i] = reinterpret_cast<const int4*>(X->f)[i];
                    reinterpret_cast<int4*>(sw.e)[i] = reinterpret_cast<const int4*>(X->e)[i];
                }
                for (int i = tid; i < tiles; i += GI_THREADS) { sw.s[i] = X->s[i]; sw.ev[i] = X->ev[i]; }
                __syncthreads();
                gi_sums(sw.s, sw.ev, tiles, lane, s_all, ev_all);
                if (sweeps) gi_sweep_runs(X, sw, own, wib, t, tiles, m, lane, s_own);
            }
            meet();
            // ---------------- 3. grouping (block 0) while the others write the new nodes below the events
            if (blk == 0) gi_group(sv, X, sh.table, wsum, used, s_all, ev_all, tid);
            else {
                auto& sw = sh.sweep;
                for (int i = tid; i < tiles * 8; i += GI_THREADS) reinterpret_cast<int4*>(sw.f)[i] = reinterpret_cast<const int4*>(X->r)[i];
                __syncthreads();
                if (sweeps && (long long)used + s_all <= sv.g_cap) gi_sweep_emit(sw, own, ent, used, wib, t, m, lane, s_own);
            }
            meet();
            // ---------------- merges: a warp per parent, a block per parent with a long run
            const int n_groups = X->n_groups;
            full = X->fits == 0;
            if (!full) {
                for (int gi = wib * GI_BLOCKS + blk; gi < n_groups; gi += GI_BLOCKS * (GI_THREADS / 32)) {
                    const GiGroup g = X->group[gi];
                    if (g.n <= GI_BIG && g.k <= GI_BIG) gi_merge<32>(sv, X, X->m_pos, g, used, lane, [] { __syncwarp(); });
                }
                const int n_big = X->n_big;
                for (int b = blk; b < n_big; b += GI_BLOCKS) {
                    const GiGroup g = X->group[X->big[b]];
                    gi_merge<GI_THREADS>(sv, X, X->m_pos, g, used, tid, [] { __syncthreads(); });
                }
            }
            meet();
            // ---------------- 4. the parents' entries
            if (!full) {
                for (int gi = blk * GI_THREADS + tid; gi < n_groups; gi += GI_BLOCKS * GI_THREADS) {
                    const GiGroup g = X->group[gi];
                    if (g.parent < 0) continue;
                    int at = g.parent;
                    if (g.above >= 0) {
                        const GiGroup a = X->group[g.above];
                        int lo = 0, hi = a.k;
                        while (lo < hi) { const int mid = (lo + hi) >> 1; if (X->m_tok[a.first + mid] < g.parent_tok) lo = mid + 1; else hi = mid; }
                        at = a.base + (g.parent - a.cb) + lo;
                    }
                    *reinterpret_cast<int2*>(&ent[at].z) = make_int2(g.base, g.n + g.k);
                }
                live += s_all + ev_all;
                used += s_all + X->entries;
            }
            tokens_done += m;
        }
    }
    bad = __syncthreads_or(bad) != 0;
    if (again) meet();                               // (who sees the new epoch sees the whole of the new tree; 1 us of an append of 256 requests)
    if (tid == 0 && blk == 0) {
        GlobalState* gs = sv.g_state;
        sd_release(&gs->epoch, gs->epoch + 1);       // cached match nodes of every slot are stale now
        gs->used = used;
        gs->live += live;
        gs->status |= (full ? SD_STATUS_GLOBAL_FULL : 0) | (bad ? SD_STATUS_BAD_TOKEN : 0);
        gs->tokens += tokens_done;
    }
}

// Block i appends item i to its request slot (items for the global tree are taken by
// global_insert_kernel): APP_AHEAD tokens at a time, looked up ahead by all warps and appended by the first.
constexpr int APPEND_THREADS = 256;

__global__ void __launch_bounds__(APPEND_THREADS)
append_kernel(sd_store sv, const int32_t* d_slot, const int64_t* d_offsets, const int32_t* d_tokens, const uint8_t* d_reset) {
    __shared__ AppendShared sh;
    __shared__ int sh_len, sh_status;
    const int i = blockIdx.x, tid = threadIdx.x, lane = tid & 31, wib = tid >> 5;
    const int slot = d_slot[i];
    if (slot < 0 || slot >= sv.R) return;
    SlotState* ss = sv.s_state + slot;
    int32_t* const text = sv.s_text + (long long)slot * sv.T;
    int32_t* const root = sv.s_root + (long long)slot * sv.V;
    int len = ss->len, used = ss->used, live = ss->live, status = ss->status;
    int act = ss->active[lane], cb = ss->run_cb[lane];
    unsigned w = append_pack(ss->run_w[lane], ss->room[lane]);
    if (d_reset && d_reset[i]) {
        // forget the old tree: only root-table cells of tokens that occur can be set
        for (int k = tid; k < len; k += APPEND_THREADS) root[text[k]] = -1;
        len = 0; used = 0; live = 0; status = 0; act = -1; cb = 0; w = 0;
        __syncthreads();
        if (tid == 0) ss->gen += 1;
    }
    const int32_t* const tok = d_tokens + d_offsets[i];
    const int n_new = (int)(d_offsets[i + 1] - d_offsets[i]);
    for (int k = 0; k < n_new && !(status & (SD_STATUS_POOL_FULL | SD_STATUS_BAD_TOKEN)); k += APP_AHEAD) {
        const int m = min(APP_AHEAD, n_new - k);
        append_stage_tokens(sh, text, len, tok + k, n_new - k, tid, APPEND_THREADS);
        if (tid == 0) sh.ahead = m >= 3 ? 1 : 0;
        __syncthreads();
        if (m >= 3) {                                            // (one or two tokens are as soon searched for in their turn)
            search_ahead(sh, sv, sv.s_ent + (long long)slot * sv.spn, root, len, m, tid / APP_LANES, APPEND_THREADS / APP_LANES, lane);
            __syncthreads();
        }
        if (wib == 0) {
            append_tokens<true>(sh, sv, slot, tok + k, m, 1, lane, act, cb, w, len, used, live, status);
            if (lane == 0) { sh_len = len; sh_status = status; }
        }
        __syncthreads();
        len = sh_len; status = sh_status;
    }
    if (wib == 0) {
        append_store(ss, lane, act, cb, w);
        if (lane == 0) { ss->len = len; ss->used = used; ss->live = live; ss->status = status; }
    }
}

}  // namespace

namespace {

// Whether the device has room for the cluster (asked once), and the limits of the kernel that will be launched, at every call: they are
// gone after a cudaDeviceReset.
int insert_setup(int dev, bool* cluster) {
    constexpr int MAX_DEVICES = 64;
    static std::atomic<int> known[MAX_DEVICES];                  // 1: a grid, 2: a cluster
    const bool kept = dev >= 0 && dev < MAX_DEVICES;
    int k = sd_small_clusters() ? 1 : (kept ? known[dev].load() : 0);
    if (k != 1) {
        constexpr size_t smem = sizeof(GiShared<GI_CLUSTER>);
        const bool set = cudaFuncSetAttribute(global_insert_kernel<GI_CLUSTER>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) == cudaSuccess &&
                         cudaFuncSetAttribute(global_insert_kernel<GI_CLUSTER>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess;
        if (k == 0) {
            cudaLaunchAttribute attr;
            attr.id = cudaLaunchAttributeClusterDimension;
            attr.val.clusterDim.x = GI_CLUSTER; attr.val.clusterDim.y = 1; attr.val.clusterDim.z = 1;
            cudaLaunchConfig_t cfg = {};
            cfg.gridDim = dim3(GI_CLUSTER); cfg.blockDim = dim3(GI_THREADS); cfg.dynamicSmemBytes = smem;
            cfg.attrs = &attr; cfg.numAttrs = 1;
            int n = 0;
            k = set && cudaOccupancyMaxActiveClusters(&n, global_insert_kernel<GI_CLUSTER>, &cfg) == cudaSuccess && n > 0 ? 2 : 1;
            cudaGetLastError();
            if (kept) known[dev].store(k);
        } else if (!set) return SD_ERR_CUDA;
    }
    if (k == 1)
        SD_CUDA_OK(cudaFuncSetAttribute(global_insert_kernel<GI_GRID>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(GiShared<GI_GRID>)));
    *cluster = k == 2;
    return SD_OK;
}

}  // namespace

extern "C" int sd_append(sd_store* s, int32_t n, const int32_t* d_slot, const int64_t* d_offsets,
                         const int32_t* d_tokens, const uint8_t* d_reset, void* stream) {
    if (!s || n < 0) return SD_ERR_INVALID_ARG;
    SD_CHECK_DEVICE(s);
    if (n == 0) return SD_OK;
    if (!d_slot || !d_offsets) return SD_ERR_INVALID_ARG;
    // The global tree and the request trees share nothing: the insert into the global tree runs
    // beside the appends, on the store's own stream, which starts behind everything the caller's
    // stream holds so far and which the caller's stream waits for before it goes on.
    cudaStream_t st = (cudaStream_t)stream;
    s->appended = 1;
    SD_CUDA_OK(cudaEventRecord(s->ev_fork, st));
    SD_CUDA_OK(cudaStreamWaitEvent(s->aux, s->ev_fork, 0));
    int tok_bits = 1;
    while (tok_bits < 31 && (1 << tok_bits) < s->V) ++tok_bits;
    void* args[] = {(void*)s, (void*)&n, (void*)&d_slot, (void*)&d_offsets, (void*)&d_tokens, (void*)&tok_bits};
    bool cluster = false;
    const int rc = insert_setup(s->device, &cluster);
    if (rc != SD_OK) return rc;
    const int gi_blocks = cluster ? GI_CLUSTER : GI_GRID;
    const void* const gi_kernel = cluster ? (const void*)global_insert_kernel<GI_CLUSTER> : (const void*)global_insert_kernel<GI_GRID>;
    cudaLaunchAttribute attr;
    if (cluster) {
        attr.id = cudaLaunchAttributeClusterDimension;
        attr.val.clusterDim.x = GI_CLUSTER; attr.val.clusterDim.y = 1; attr.val.clusterDim.z = 1;
    } else {
        attr.id = cudaLaunchAttributeCooperative;
        attr.val.cooperative = 1;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)gi_blocks); cfg.blockDim = dim3(GI_THREADS); cfg.stream = s->aux; cfg.attrs = &attr; cfg.numAttrs = 1;
    cfg.dynamicSmemBytes = cluster ? sizeof(GiShared<GI_CLUSTER>) : sizeof(GiShared<GI_GRID>);
    SD_CUDA_OK(cudaLaunchKernelExC(&cfg, gi_kernel, args));
    // (joined whatever becomes of the launch: the insert reads buffers that the caller may free behind this call on its stream)
    const cudaError_t record = cudaEventRecord(s->ev_join, s->aux);
    append_kernel<<<(unsigned)n, APPEND_THREADS, 0, st>>>(*s, d_slot, d_offsets, d_tokens, d_reset);
    const cudaError_t launch = cudaGetLastError(), join = cudaStreamWaitEvent(st, s->ev_join, 0);
    return record == cudaSuccess && launch == cudaSuccess && join == cudaSuccess ? SD_OK : SD_ERR_CUDA;
}
