// How large a tree may be: its entries are found by 32-bit indices.
#pragma once

// Tokens of a corpus, or of the prompts of one sd_build_requests.  (The kernels go through positions with an int, up to 32,768 of
// them beyond the last one.)
constexpr long long SD_MAX_TOKENS = (1ll << 31) - (1 << 16);
constexpr long long SD_MAX_ENTRIES = (1ll << 31) - 3;

// What an offline build counts before it lays anything down.
struct TreeTotals {
    long long below, top;                         // nodes below depth 1, of depth 1
    long long wide;                               // entries that the long runs take with their top blocks, behind the others
    int n_wide;                                   // long runs
    int listed, placed;                           // of these, while they are listed and given their places
};

// Entries of the global pool: the tree's (a long run leaves its first place empty) and head-room for online inserts (extra
// < 0: as many nodes again, 4 M at least).  -1: more than there are indices for.
inline long long sd_pool_entries(const TreeTotals& t, long long extra) {
    if (t.below > SD_MAX_ENTRIES || t.top > SD_MAX_ENTRIES || t.wide > SD_MAX_ENTRIES || extra > SD_MAX_ENTRIES) return -1;
    const long long nodes = t.below + t.top;
    if (extra < 0) extra = nodes > (1ll << 22) ? nodes : 1ll << 22;
    const long long entries = nodes + t.wide + extra;
    return entries > SD_MAX_ENTRIES ? -1 : entries;
}
