// Device memory, streams and pinned memory of the library (device_memory.cpp): kept from store to store.
#pragma once

#include "common.cuh"

// What a store holds besides device memory: a stream and events, and pinned memory for the arguments of sd_build_requests.
struct StreamSet { cudaStream_t aux; cudaEvent_t ev_fork, ev_join, ev_check; void* stage; size_t stage_bytes; };

// For a store on the current device, with at least `stage_bytes` of pinned memory.
bool sd_take_streams(int dev, size_t stage_bytes, StreamSet* out);

// Calls of sd_trim so far.  What is set up once per device is set up anew behind one: a cudaDeviceReset may have followed.
int sd_trims();

// sd_debug_small_clusters is on.
bool sd_small_clusters();

// Releases what a store holds, behind the work on `st`: the caller has waited for every other stream that used the store.
void sd_store_release(sd_store* s, cudaStream_t st);
