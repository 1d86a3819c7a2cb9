// Checks of csrc/memory.cpp on the CPU, linked with the stand-in for the CUDA runtime below: what is kept between stores, when
// it is given back, and what a store's release waits for.  `device_memory_check NAME` runs one check; 0 = it holds.
#include <stdio.h>
#include <stdlib.h>
#include <string.h>

#include <map>
#include <mutex>

#include "memory.h"

// ---- the stand-in: devices of 32 GB, work that is queued on a device until something waits for that device
namespace fake {
constexpr int DEVICES = 4;
constexpr size_t TOTAL = 32ull << 30;
struct Block { int dev; size_t bytes; };
std::mutex mutex;
std::map<void*, Block> blocks;
bool busy[DEVICES];                                   // kernels of a caller's stream are still at work
size_t used[DEVICES];
thread_local int current = 0;
}  // namespace fake

extern "C" {
cudaError_t cudaGetDevice(int* d) { *d = fake::current; return cudaSuccess; }
cudaError_t cudaSetDevice(int d) { if (d < 0 || d >= fake::DEVICES) return cudaErrorInvalidDevice; fake::current = d; return cudaSuccess; }
cudaError_t cudaDeviceSynchronize() { std::lock_guard<std::mutex> l(fake::mutex); fake::busy[fake::current] = false; return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaMalloc(void** p, size_t n) {
    std::lock_guard<std::mutex> l(fake::mutex);
    if (fake::used[fake::current] + n > fake::TOTAL) return cudaErrorMemoryAllocation;
    *p = malloc(1);
    fake::blocks[*p] = fake::Block{fake::current, n};
    fake::used[fake::current] += n;
    return cudaSuccess;
}
cudaError_t cudaFree(void* p) {
    std::lock_guard<std::mutex> l(fake::mutex);
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
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { *s = (cudaStream_t)malloc(1); return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t s) { free(s); return cudaSuccess; }
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

struct Check { const char* name; int (*run)(); };
const Check checks[] = {
    {"free_waits_for_the_owner", free_waits_for_the_owner},
};

}  // namespace

int main(int argc, char** argv) {
    for (const Check& c : checks)
        if (argc > 1 && !strcmp(argv[1], c.name)) return c.run();
    fprintf(stderr, "no such check\n");
    return 2;
}
