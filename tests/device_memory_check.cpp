// Checks of csrc/device_memory.cpp on the CPU, linked with the stand-in for the CUDA runtime below: what is kept between stores, when
// it is given back, and what a store's release waits for.  `device_memory_check NAME` runs one check; 0 = it holds.
#include <stdio.h>
#include <stdlib.h>
#include <string.h>
#include <sys/wait.h>
#include <unistd.h>

#include <atomic>
#include <chrono>
#include <map>
#include <mutex>
#include <new>
#include <thread>
#include <vector>

#include "device_memory.h"

static thread_local bool no_host_memory = false;
void* operator new(size_t n) {
    void* p = no_host_memory ? nullptr : malloc(n ? n : 1);
    if (!p) throw std::bad_alloc();
    return p;
}
void operator delete(void* p) noexcept { free(p); }
void operator delete(void* p, size_t) noexcept { free(p); }

struct HostMemory {                                   // the stand-in itself has some
    const bool was = no_host_memory;
    HostMemory() { no_host_memory = false; }
    ~HostMemory() { no_host_memory = was; }
};

// ---- the stand-in: devices of 32 GB, work that is queued on a device until something waits for that device
namespace fake {
constexpr int DEVICES = 4;
constexpr size_t TOTAL = 32ull << 30;
struct Block { int dev; size_t bytes; };
std::mutex mutex;
std::map<void*, Block> blocks;
bool busy[DEVICES];                                   // kernels of a caller's stream are still at work
size_t used[DEVICES];
int streams;                                          // in existence
bool touched[DEVICES];                                // some thread made a call with this device current: it has a context
std::atomic<bool> capturing{false}, spoilt{false};    // some thread captures a stream; a call of another thread broke that
thread_local int current = 0;
thread_local cudaStreamCaptureMode mode = cudaStreamCaptureModeGlobal;

size_t all_used() {
    std::lock_guard<std::mutex> l(mutex);
    size_t n = 0;
    for (size_t u : used) n += u;
    return n + (size_t)streams;
}
}  // namespace fake

extern "C" {
cudaError_t cudaGetDevice(int* d) { *d = fake::current; return cudaSuccess; }
cudaError_t cudaSetDevice(int d) { if (d < 0 || d >= fake::DEVICES) return cudaErrorInvalidDevice; fake::current = d; fake::touched[d] = true; return cudaSuccess; }
cudaError_t cudaDeviceSynchronize() { std::lock_guard<std::mutex> l(fake::mutex); fake::busy[fake::current] = false; return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaMalloc(void** p, size_t n) {
    HostMemory m;
    std::lock_guard<std::mutex> l(fake::mutex);
    if (fake::used[fake::current] + n > fake::TOTAL) return cudaErrorMemoryAllocation;
    *p = malloc(1);
    fake::touched[fake::current] = true;
    fake::blocks[*p] = fake::Block{fake::current, n};
    fake::used[fake::current] += n;
    return cudaSuccess;
}
cudaError_t cudaFree(void* p) {
    std::lock_guard<std::mutex> l(fake::mutex);
    fake::touched[fake::current] = true;
    if (fake::capturing && fake::mode == cudaStreamCaptureModeGlobal) fake::spoilt = true;
    auto it = fake::blocks.find(p);
    if (it == fake::blocks.end()) return cudaErrorInvalidValue;
    fake::busy[it->second.dev] = false;               // (it waits for the device that owns the memory)
    fake::used[it->second.dev] -= it->second.bytes;
    fake::blocks.erase(it);
    free(p);
    return cudaSuccess;
}
cudaError_t cudaMemGetInfo(size_t* f, size_t* t) { *t = fake::TOTAL; *f = fake::TOTAL - fake::used[fake::current]; return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaThreadExchangeStreamCaptureMode(cudaStreamCaptureMode* m) { std::swap(*m, fake::mode); return cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) {
    std::lock_guard<std::mutex> l(fake::mutex);
    ++fake::streams;
    *s = (cudaStream_t)malloc(1);
    return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t s) {
    std::lock_guard<std::mutex> l(fake::mutex);
    --fake::streams;
    free(s);
    return cudaSuccess;
}
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { *e = (cudaEvent_t)malloc(1); return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t e) { free(e); return cudaSuccess; }
cudaError_t cudaHostAlloc(void** p, size_t n, unsigned) { *p = malloc(n); return cudaSuccess; }
cudaError_t cudaFreeHost(void* p) { free(p); return cudaSuccess; }
}

#define EXPECT(x) do { if (!(x)) { fprintf(stderr, "line %d: %s\n", __LINE__, #x); return 1; } } while (0)

namespace {

// a store on the current device that holds one block of that many bytes
sd_store* make_store(size_t bytes) {
    sd_store* s = new sd_store();
    memset(s, 0, sizeof(*s));
    cudaGetDevice(&s->device);
    StreamSet k;
    if (sd_device_malloc((void**)&s->g_ent, bytes) != cudaSuccess || !sd_take_streams(s->device, 64, &k)) return nullptr;
    s->aux = k.aux; s->ev_fork = k.ev_fork; s->ev_join = k.ev_join; s->ev_check = k.ev_check; s->stage = k.stage; s->stage_bytes = k.stage_bytes;
    return s;
}

// A store that is freed while another device is current: its memory goes on only when its own device has ended its work.
int free_waits_for_the_owner() {
    for (int owner = 0; owner < 2; ++owner)
        for (int current = 0; current < 2; ++current) {
            cudaSetDevice(owner);
            sd_store* s = make_store(1 << 20);
            EXPECT(s);
            void* const p = s->g_ent;
            fake::busy[owner] = true;
            cudaSetDevice(current);
            sd_free(s);
            EXPECT(!fake::busy[owner]);
            EXPECT(fake::current == current);
            cudaSetDevice(owner);
            void* q = nullptr;
            EXPECT(sd_device_malloc(&q, 1 << 20) == cudaSuccess);
            EXPECT(q == p && fake::blocks[q].dev == owner);      // kept, and for its own device
            sd_device_free(q);
        }
    return 0;
}

bool given_back_within(double seconds) {
    for (int k = 0; k < (int)(seconds * 100); ++k) {
        if (fake::all_used() == 0) return true;
        std::this_thread::sleep_for(std::chrono::milliseconds(10));
    }
    return false;
}

// Nothing is called any more after the last store was freed: what was kept of it goes back all the same, once it has been
// kept for as long as that (SD_KEEP_SECONDS, here 0.3), with no context made on a device that had none.
int kept_memory_goes_back_by_itself() {
    for (int round = 0; round < 2; ++round) {
        for (int dev = 1; dev < 3; ++dev) {
            cudaSetDevice(dev);
            sd_store* s = make_store(3 << 20);
            EXPECT(s);
            sd_free(s);
        }
        EXPECT(fake::all_used() > (6u << 20));               // (kept for the next store)
        fake::capturing = true;
        EXPECT(given_back_within(10));
        EXPECT(!fake::spoilt);
        fake::capturing = false;
    }
    EXPECT(!fake::touched[0] && fake::touched[1] && fake::touched[2] && !fake::touched[3]);
    return 0;
}

// What a store has taken out of what was kept stays, however long it is used.
int what_is_in_use_stays() {
    sd_store* s = make_store(1 << 20);
    sd_free(s);
    std::this_thread::sleep_for(std::chrono::milliseconds(100));
    s = make_store(1 << 20);
    std::this_thread::sleep_for(std::chrono::milliseconds(700));
    EXPECT(fake::blocks.count(s->g_ent) == 1 && fake::streams == 1);
    sd_free(s);
    EXPECT(given_back_within(10));
    return 0;
}

int trim_gives_back_at_once() {
    void* p = nullptr;
    cudaSetDevice(2);
    EXPECT(sd_device_malloc(&p, 5000) == cudaSuccess);
    for (int dev = 0; dev < 3; ++dev) { cudaSetDevice(dev); sd_free(make_store(1 << 20)); }
    cudaSetDevice(1);
    const size_t before = fake::all_used();
    sd_trim();
    EXPECT(fake::current == 1);
    EXPECT(before > (3u << 20) && fake::all_used() > 0 && fake::all_used() < 8192);      // (the block in use stays)
    EXPECT(fake::blocks.count(p) == 1);
    sd_device_free(p);
    sd_trim();
    EXPECT(fake::all_used() == 0);
    return 0;
}

int many_threads() {
    std::vector<std::thread> threads;
    std::atomic<int> bad{0};
    for (int t = 0; t < 8; ++t)
        threads.emplace_back([t, &bad] {
            unsigned x = 12345u + 777u * t;
            cudaSetDevice(t & 1);
            for (int k = 0; k < 4000; ++k) {
                x = x * 1664525u + 1013904223u;
                sd_store* s = make_store(1000 + (x >> 12));
                if (!s) { ++bad; continue; }
                if ((x & 1023) == 0) std::this_thread::sleep_for(std::chrono::milliseconds(40));
                { std::lock_guard<std::mutex> l(fake::mutex); if (fake::blocks.count(s->g_ent) != 1 || fake::blocks[s->g_ent].dev != (t & 1)) ++bad; }
                sd_free(s);
                if ((x & 255) == 1) sd_trim();
            }
        });
    for (std::thread& t : threads) t.join();
    EXPECT(bad == 0);
    EXPECT(given_back_within(10));
    return 0;
}

// A forked child has no thread that gives memory back; it must end all the same.
int a_forked_child_ends() {
    sd_free(make_store(1 << 20));
    const pid_t child = fork();
    if (child == 0) exit(0);
    int status = 1;
    EXPECT(waitpid(child, &status, 0) == child && WIFEXITED(status) && WEXITSTATUS(status) == 0);
    EXPECT(given_back_within(10));
    return 0;
}

// 1/32 of a device's 32 GB: the oldest go first, what is larger than that is not kept at all, and what is kept of other devices
// does not count.
int kept_memory_is_bounded() {
    const size_t most = fake::TOTAL / 32, half = most / 2;
    void* p[6];
    cudaSetDevice(1);
    EXPECT(sd_device_malloc(&p[5], half) == cudaSuccess);
    sd_device_free(p[5]);
    cudaSetDevice(0);
    for (int k = 0; k < 5; ++k) EXPECT(sd_device_malloc(&p[k], half - (size_t)k * (80u << 20)) == cudaSuccess);
    for (int k = 0; k < 5; ++k) {
        sd_device_free(p[k]);
        size_t in_use = 0;
        for (int q = k + 1; q < 5; ++q) in_use += fake::blocks[p[q]].bytes;
        EXPECT(fake::used[0] - in_use <= most);
        EXPECT(fake::blocks.count(p[k]) == 1);
    }
    EXPECT(fake::blocks.count(p[0]) == 0 && fake::blocks.count(p[5]) == 1);
    EXPECT(sd_device_malloc(&p[0], most + (64u << 20)) == cudaSuccess);
    sd_device_free(p[0]);
    EXPECT(fake::blocks.count(p[0]) == 0 && fake::blocks.count(p[4]) == 1);
    sd_trim();
    return 0;
}

// The C entry points report a lack of host memory and throw nothing; no block is lost.
int no_host_memory_throws_nothing() {
    void *p = nullptr, *q = nullptr;
    no_host_memory = true;
    const cudaError_t fresh = sd_device_malloc(&p, 4096);
    no_host_memory = false;
    EXPECT(fresh == cudaErrorMemoryAllocation && !p && fake::all_used() == 0);
    EXPECT(sd_device_malloc(&p, 4096) == cudaSuccess);
    no_host_memory = true;
    sd_device_free(p);
    no_host_memory = false;
    EXPECT(fake::all_used() == 0);
    EXPECT(sd_device_malloc(&p, 4096) == cudaSuccess);
    sd_device_free(p);
    no_host_memory = true;
    const cudaError_t kept = sd_device_malloc(&q, 4096);
    no_host_memory = false;
    EXPECT(kept == cudaErrorMemoryAllocation && !q);
    sd_trim();
    EXPECT(fake::all_used() == 0);
    return 0;
}

struct Check { const char* name; int (*run)(); };
const Check checks[] = {
    {"free_waits_for_the_owner", free_waits_for_the_owner},
    {"kept_memory_goes_back_by_itself", kept_memory_goes_back_by_itself},
    {"what_is_in_use_stays", what_is_in_use_stays},
    {"trim_gives_back_at_once", trim_gives_back_at_once},
    {"many_threads", many_threads},
    {"a_forked_child_ends", a_forked_child_ends},
    {"kept_memory_is_bounded", kept_memory_is_bounded},
    {"no_host_memory_throws_nothing", no_host_memory_throws_nothing},
};

}  // namespace

int main(int argc, char** argv) {
    for (const Check& c : checks)
        if (argc > 1 && !strcmp(argv[1], c.name)) return c.run();
    fprintf(stderr, "no such check\n");
    return 2;
}
