// The device memory of the library, kept from store to store, and the release of a store.  Host code only.
#include <pthread.h>
#include <signal.h>
#include <stdlib.h>
#include <string.h>
#include <unistd.h>

#include <algorithm>
#include <atomic>
#include <chrono>
#include <condition_variable>
#include <mutex>
#include <new>
#include <thread>
#include <unordered_map>
#include <vector>

#include "device_memory.h"

// Blocks that stores and builds have given back are kept for the next ones, up to 1/32 of the device's memory (5.7 GB
// of a B200's).  The oldest go first when there are more, all of them when an allocation fails (which is then tried once
// more) or sd_trim is called, and a thread of the library's own gives back what nobody has wanted for half a minute, so
// that a process that only ever frees its last store does not sit on it (1 GB given back beside a loop of drafts held up one
// of its calls, by 2 ms).  Getting and returning memory is what a build or a short-lived store would otherwise spend its time on: 20
// cudaMalloc / cudaFree calls took 2.7 ms of the 3.7 ms of a 32,768-token build and up to 70 ms of a
// 4 M-token one.  (CUDA's own stream-ordered pools cost 6.2 ms per GB whenever they grow or shrink, cudaMalloc
// 0.3 - 0.8 ms at any of these sizes.)  A block is given back when the work on it has ended, so the next owner may be
// on any stream or thread.  Streams, events and pinned memory of freed stores are kept in the same way.
//
// Test hook: the k-th device allocation from now on fails (k = 1: the next one); 0 switches it off.
// Only the allocation-failure tests use it.  While it is on nothing is kept.
#ifndef SD_KEEP_SECONDS
#define SD_KEEP_SECONDS 30.0
#endif

namespace {

constexpr int CACHE_DEVICES = 64;
constexpr int CACHE_FRACTION = 32;
constexpr int KEPT_STREAMS = 8;

typedef std::chrono::steady_clock Clock;
const Clock::duration KEEP = std::chrono::duration_cast<Clock::duration>(std::chrono::duration<double>(SD_KEEP_SECONDS));

struct FreeBlock { void* p; size_t bytes; Clock::time_point since; };
struct FreeStreams { StreamSet set; Clock::time_point since; };
struct DeviceCache {
    std::vector<FreeBlock> idle;                      // oldest first
    size_t bytes = 0, most = 0;
    FreeStreams streams[KEPT_STREAMS];                // of freed stores, for the next ones; oldest first
    int n_streams = 0;
};
struct OwnedBlock { size_t bytes; int dev; };
struct Memory {
    DeviceCache cache[CACHE_DEVICES];
    std::unordered_map<void*, OwnedBlock> owned;      // blocks in use
    std::mutex mutex;                                 // of everything here
    std::condition_variable wake;                     // something is kept where nothing was
    bool keeper = false, asleep = false, ending = false;         // the thread below runs, waits for `wake`, is to end
};
Memory& g = *new Memory;                              // (never destroyed: the keeper and late sd_free calls outlive main)
long long g_fail_alloc_in = 0;
bool g_fail_alloc_on = false;

void drop_streams(const StreamSet& s) {
    for (cudaEvent_t e : {s.ev_fork, s.ev_join, s.ev_check}) if (e) cudaEventDestroy(e);
    if (s.aux) cudaStreamDestroy(s.aux);
    if (s.stage) cudaFreeHost(s.stage);
}

// gives back the oldest blocks until at most `bytes` are kept (the mutex is held)
void cache_trim(DeviceCache& c, size_t bytes) {
    size_t n = 0;
    while (n < c.idle.size() && c.bytes > bytes) { cudaFree(c.idle[n].p); c.bytes -= c.idle[n].bytes; ++n; }
    c.idle.erase(c.idle.begin(), c.idle.begin() + n);
}

// gives back what has been kept since `until` or longer, with its device current (the mutex is held)
void cache_expire(int dev, DeviceCache& c, Clock::time_point until) {
    size_t n = 0, bytes = 0;
    while (n < c.idle.size() && c.idle[n].since <= until) bytes += c.idle[n++].bytes;
    int k = 0;
    while (k < c.n_streams && c.streams[k].since <= until) ++k;
    if (n == 0 && k == 0) return;
    int current = -1;
    const bool away = cudaGetDevice(&current) == cudaSuccess && current != dev;
    if (away) cudaSetDevice(dev);
    cache_trim(c, c.bytes - bytes);
    for (int q = 0; q < k; ++q) drop_streams(c.streams[q].set);
    std::copy(c.streams + k, c.streams + c.n_streams, c.streams);
    c.n_streams -= k;
    if (away) cudaSetDevice(current);
}

// The keeper: sleeps until the oldest of what is kept has been kept for long enough, or, while nothing is, until something is.
void keep_watch() {
    bool first = true;
    std::unique_lock<std::mutex> lock(g.mutex);
    while (!g.ending) {
        const Clock::time_point now = Clock::now();
        Clock::time_point next = Clock::time_point::max();
        for (int dev = 0; dev < CACHE_DEVICES; ++dev) {
            DeviceCache& c = g.cache[dev];
            if (c.idle.empty() && c.n_streams == 0) continue;
            if (first) {
                // another thread may be capturing a stream, which giving memory back on this one does not concern
                cudaSetDevice(dev);
                cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
                cudaThreadExchangeStreamCaptureMode(&mode);
                first = false;
            }
            cache_expire(dev, c, now - KEEP);
            if (!c.idle.empty()) next = std::min(next, c.idle[0].since + KEEP);
            if (c.n_streams > 0) next = std::min(next, c.streams[0].since + KEEP);
        }
        g.asleep = next == Clock::time_point::max();
        if (g.asleep) g.wake.wait(lock);
        else g.wake.wait_until(lock, next);
    }
}

// At the process's end: behind this the keeper makes no call.  (A forked child has no keeper, and the mutex may have been
// held when it was forked.  The library is linked not to be unloaded.)
pid_t g_keeper_of;
void end_watch() {
    if (getpid() != g_keeper_of) return;
    std::lock_guard<std::mutex> lock(g.mutex);
    g.ending = true;
    g.wake.notify_all();
}

// Called before something is kept (the mutex is held): whether somebody will give it back.
bool watched() {
    if (!g.keeper) {
        try {
            // (the process's signals are not for this thread)
            sigset_t all, old;
            sigfillset(&all);
            const bool masked = pthread_sigmask(SIG_SETMASK, &all, &old) == 0;
            try { std::thread(keep_watch).detach(); g.keeper = true; } catch (...) {}
            if (masked) pthread_sigmask(SIG_SETMASK, &old, nullptr);
        } catch (...) {}
        if (!g.keeper) return false;
        g_keeper_of = getpid();
        std::atexit(end_watch);
    }
    if (g.asleep) { g.asleep = false; g.wake.notify_one(); }
    return !g.ending;
}

// a block in use (the mutex is held); false: no host memory for it
bool take_down(void* p, size_t bytes, int dev) {
    try {
        g.owned[p] = OwnedBlock{bytes, dev};
    } catch (const std::bad_alloc&) {
        return false;
    }
    return true;
}

void give_streams(int dev, const StreamSet& s) {
    {
        std::lock_guard<std::mutex> lock(g.mutex);
        if (dev >= 0 && dev < CACHE_DEVICES && g.cache[dev].n_streams < KEPT_STREAMS && watched()) {
            DeviceCache& d = g.cache[dev];
            d.streams[d.n_streams++] = FreeStreams{s, Clock::now()};
            return;
        }
    }
    drop_streams(s);
}

}  // namespace

bool sd_take_streams(int dev, size_t stage_bytes, StreamSet* out) {
    if (dev >= 0 && dev < CACHE_DEVICES) {
        std::lock_guard<std::mutex> lock(g.mutex);
        DeviceCache& d = g.cache[dev];
        for (int k = d.n_streams - 1; k >= 0; --k)
            if (d.streams[k].set.stage_bytes >= stage_bytes) {
                *out = d.streams[k].set;
                std::copy(d.streams + k + 1, d.streams + d.n_streams, d.streams + k);
                --d.n_streams;
                return true;
            }
    }
    memset(out, 0, sizeof(*out));
    out->stage_bytes = std::max<size_t>(stage_bytes, 16384);
    if (cudaStreamCreateWithFlags(&out->aux, cudaStreamNonBlocking) == cudaSuccess &&
        cudaEventCreateWithFlags(&out->ev_fork, cudaEventDisableTiming) == cudaSuccess &&
        cudaEventCreateWithFlags(&out->ev_join, cudaEventDisableTiming) == cudaSuccess &&
        cudaEventCreateWithFlags(&out->ev_check, cudaEventDisableTiming) == cudaSuccess &&
        cudaHostAlloc(&out->stage, out->stage_bytes, cudaHostAllocPortable | cudaHostAllocMapped) == cudaSuccess)
        return true;
    cudaGetLastError();
    drop_streams(*out);
    return false;
}

cudaError_t sd_device_malloc(void** p, size_t bytes) {
    *p = nullptr;
    if (g_fail_alloc_in > 0 && --g_fail_alloc_in == 0) return cudaErrorMemoryAllocation;
    int dev = -1;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= CACHE_DEVICES) return cudaErrorInvalidDevice;
    // (up to a multiple of an eighth of the next lower power of two, 32 MB at most, so that sizes that differ a little share blocks)
    size_t unit = 512;
    while (unit * 16 <= bytes && unit < (32u << 20)) unit *= 2;
    bytes = (bytes + unit - 1) / unit * unit;
    std::lock_guard<std::mutex> lock(g.mutex);
    DeviceCache& c = g.cache[dev];
    if (!g_fail_alloc_on) {
        // the smallest kept block that is not much too large
        size_t best = c.idle.size();
        for (size_t k = 0; k < c.idle.size(); ++k)
            if (c.idle[k].bytes >= bytes && c.idle[k].bytes <= bytes + bytes / 4 && (best == c.idle.size() || c.idle[k].bytes < c.idle[best].bytes))
                best = k;
        if (best < c.idle.size()) {
            if (!take_down(c.idle[best].p, c.idle[best].bytes, dev)) return cudaErrorMemoryAllocation;
            *p = c.idle[best].p;
            c.bytes -= c.idle[best].bytes;
            c.idle.erase(c.idle.begin() + best);
            return cudaSuccess;
        }
    }
    e = cudaMalloc(p, bytes);
    if (e != cudaSuccess && !c.idle.empty()) {
        cudaGetLastError();
        cache_trim(c, 0);
        e = cudaMalloc(p, bytes);
    }
    if (e != cudaSuccess) { *p = nullptr; return e; }
    if (!take_down(*p, bytes, dev)) { cudaFree(*p); *p = nullptr; return cudaErrorMemoryAllocation; }
    return cudaSuccess;
}

void sd_device_free(void* p) {
    if (!p) return;
    std::lock_guard<std::mutex> lock(g.mutex);
    auto it = g.owned.find(p);
    if (it == g.owned.end()) return;
    const OwnedBlock b = it->second;
    g.owned.erase(it);
    DeviceCache& c = g.cache[b.dev];
    if (c.most == 0) {
        size_t free_bytes = 0, total = 0;
        if (cudaMemGetInfo(&free_bytes, &total) == cudaSuccess) c.most = total / CACHE_FRACTION;
    }
    if (g_fail_alloc_on || b.bytes > c.most || !watched()) { cudaFree(p); return; }
    cache_trim(c, c.most - b.bytes);
    try {
        c.idle.push_back(FreeBlock{p, b.bytes, Clock::now()});
    } catch (const std::bad_alloc&) {
        cudaFree(p);
        return;
    }
    c.bytes += b.bytes;
}

static std::atomic<int> g_trims{0};

int sd_trims() { return g_trims.load(); }

extern "C" void sd_trim(void) {
    ++g_trims;
    std::lock_guard<std::mutex> lock(g.mutex);
    for (int dev = 0; dev < CACHE_DEVICES; ++dev) cache_expire(dev, g.cache[dev], Clock::time_point::max());
}

static std::atomic<bool> g_small_clusters{false};

bool sd_small_clusters() { return g_small_clusters.load(); }

extern "C" void sd_debug_small_clusters(int32_t on) { g_small_clusters = on != 0; }

extern "C" void sd_debug_fail_alloc(int64_t k) { g_fail_alloc_in = k; g_fail_alloc_on = k > 0; }

void sd_store_release(sd_store* s, cudaStream_t st) {
    if (!s) return;
    cudaStreamSynchronize(st);
    void* const own[] = {s->g_ent, s->g_root, s->g_state, s->gi, s->s_ent, s->s_root, s->s_text, s->s_state};
    for (void* p : own) sd_device_free(p);
    if (s->ws) {
        for (int k = 0; k < 48; ++k) sd_device_free(s->ws->ptr[k]);
        delete s->ws;
    }
    if (s->aux) give_streams(s->device, StreamSet{s->aux, s->ev_fork, s->ev_join, s->ev_check, s->stage, s->stage_bytes});
    delete s;
}

extern "C" void sd_free(sd_store* s) {
    if (!s) return;
    // What may still use the store runs on the device that owns it, whichever is current here (a garbage collector frees
    // where it happens to run), and its memory goes on to the next store of that device as soon as it is released.
    int current = -1;
    const bool away = cudaGetDevice(&current) == cudaSuccess && current != s->device;
    if (away) cudaSetDevice(s->device);
    cudaDeviceSynchronize();
    sd_store_release(s, s->aux);
    if (away) cudaSetDevice(current);
}
