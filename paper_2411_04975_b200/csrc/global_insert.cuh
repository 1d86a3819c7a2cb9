// Working memory of the online insert into the global tree (append.cu), kept by the store.
#pragma once

#include "common.cuh"

constexpr int GI_MAX = 2048;                  // positions of a pass, the tokens looked ahead at included
// Start positions of a pass (a lot).  What is in the tree when the pool runs full depends on it: the same for every kernel that inserts.
constexpr int GI_REAL = GI_MAX - SD_MAX_DEPTH;
// Suffixes per tile: a tile is a warp's, and the 15 x 16 warps that sweep in a cluster of 16 blocks take 2,016 positions by nines.
// (By eights, 1,920 a pass, 2,010 positions took two passes: 146 - 148 us, now 116 - 121.  300 sequences of 100 tokens: 1,667 us and, on
// other text, 1,964; now 1,816 and 1,908, since 960 walks at a time go three times for a full pass.)
constexpr int GI_TILE = 9;
constexpr int GI_TILES = (GI_MAX + GI_TILE - 1) / GI_TILE;

// The new children of one node of the tree.
struct GiGroup {
    int parent, parent_tok;                   // the node (-1: the root) and its token
    int above;                                // group of the node above it, if that gets new children, too (else -1)
    int first, k;                             // its new children: m_tok / m_ev [first, first + k)
    int cb, n;                                // its child run
    int base;                                 // where the run goes (cb: it stays)
};

struct __align__(16) GiScratch {
    int tok[GI_MAX];                          // by position
    int v[GI_MAX], p[GI_MAX], q[GI_MAX];      // by start position: levels that exist, the node there, the node above that
    int sa[GI_MAX], lcp[GI_MAX], len[GI_MAX]; // by place in the suffix order
    int f[GI_TILES][32], e[GI_TILES][32], r[GI_TILES][32], s[GI_TILES], ev[GI_TILES];        // by tile
    // by event (first new node below an existing one), in suffix order
    int ev_p[GI_MAX], ev_q[GI_MAX], ev_ptok[GI_MAX], ev_tok[GI_MAX], ev_cnt[GI_MAX], ev_run[GI_MAX], ev_kids[GI_MAX];
    int m_tok[GI_MAX], m_ev[GI_MAX], m_pos[GI_MAX];             // by group, tokens ascending: event, place in the old run
    GiGroup group[GI_MAX];
    int big[GI_MAX];
    int n_groups, n_big, fits, entries;
};
