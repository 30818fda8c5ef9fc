// Device results into the caller's ordinary (pageable) memory.  A copy to pageable memory goes through the driver's own
// staging buffer on one host thread, and a freshly allocated destination has each of its pages mapped inside that copy: 16 MB of
// logits took 0.93 ms of copying and another millisecond of page faults.  Here the pages are touched by several threads
// while the GPU still computes, and the copy runs through a ring of pinned slots: while the GPU fills some over PCIe, several threads
// each move one to its place (all threads on one slot at a time, a fork and a join per slot, took 0.75 ms for those 16 MB; this way 0.53).
#include <omp.h>

#include <algorithm>
#include <atomic>
#include <cstring>
#include <mutex>
#include <vector>

#include "gad_internal.h"

namespace gad {

namespace {

constexpr size_t kSlotBytes = 512u << 10;   // 10 us over PCIe, 50 to 100 us of one thread's copying
constexpr int kSlots = 16, kMaxThreads = 8;
constexpr size_t kTouchBytes = 1u << 20;  // destinations below this are not worth waking threads for
constexpr size_t kPage = 4096;
constexpr size_t kSmallPinned = 16384;

int copy_threads(size_t bytes) {
    return (int)std::max<size_t>(1, std::min<size_t>({(size_t)kMaxThreads, (size_t)omp_get_num_procs() / 2, bytes / (128u << 10)}));
}

// Pinned buffers of kSlots slots, shared by all contexts of the process: at most two are kept while a context exists, none
// after the last one has gone.
struct Pool {
    std::mutex lock;
    int users = 0;
    std::vector<char*> idle, idle_small;
} g_pool;

// One buffer of `bytes` from the idle ones, or a new one (null if there is none to be had).
char* take_from(std::vector<char*>& idle, size_t bytes) {
    {
        std::lock_guard<std::mutex> g(g_pool.lock);
        if (!idle.empty()) { char* b = idle.back(); idle.pop_back(); return b; }
    }
    void* b = nullptr;
    if (cudaHostAlloc(&b, bytes, cudaHostAllocPortable) != cudaSuccess) { cudaGetLastError(); return nullptr; }
    return (char*)b;
}
void give_to(std::vector<char*>& idle, size_t most, char* b) {
    {
        std::lock_guard<std::mutex> g(g_pool.lock);
        if (g_pool.users > 0 && idle.size() < most) { idle.push_back(b); return; }
    }
    cudaFreeHost(b);
}
char* take_buffer() {
    {
        std::lock_guard<std::mutex> g(g_pool.lock);
        if (g_pool.users <= 0) return nullptr;   // no context to keep the buffer for: pinning one for a single copy costs more than it saves
    }
    return take_from(g_pool.idle, kSlots * kSlotBytes);
}
void give_buffer(char* b) { give_to(g_pool.idle, 2, b); }

bool is_pageable(const void* p) {
    cudaPointerAttributes a;
    if (cudaPointerGetAttributes(&a, p) != cudaSuccess) { cudaGetLastError(); return true; }
    return a.type == cudaMemoryTypeUnregistered;
}

struct Events {
    cudaEvent_t ev[kSlots] = {};
    ~Events() { for (cudaEvent_t e : ev) if (e) cudaEventDestroy(e); }
};

}  // namespace

void host_copy_user(int delta) {
    std::vector<char*> drop;
    {
        std::lock_guard<std::mutex> g(g_pool.lock);
        g_pool.users += delta;
        if (g_pool.users <= 0) {
            drop.swap(g_pool.idle);
            drop.insert(drop.end(), g_pool.idle_small.begin(), g_pool.idle_small.end());
            g_pool.idle_small.clear();
        }
    }
    for (char* b : drop) cudaFreeHost(b);
}

// Pinned memory for a context's small results.  Allocating pinned memory costs about a millisecond and waits for the device, so
// blocks of the common size are kept (at most 16) for the next context.
char* take_small_pinned(size_t bytes) {
    if (bytes <= kSmallPinned) return take_from(g_pool.idle_small, kSmallPinned);
    void* b = nullptr;
    if (cudaHostAlloc(&b, bytes, cudaHostAllocPortable) != cudaSuccess) { cudaGetLastError(); return nullptr; }
    return (char*)b;
}
void give_small_pinned(char* b, size_t bytes) {
    if (bytes <= kSmallPinned) give_to(g_pool.idle_small, 16, b);
    else cudaFreeHost(b);
}

void host_prefault(void* dst, size_t bytes) {
    if (bytes < kTouchBytes || !is_pageable(dst)) return;
    char* d = (char*)dst;
    const int64_t n = (int64_t)(bytes / kPage);
#pragma omp parallel for num_threads(copy_threads(bytes)) schedule(static)
    for (int64_t i = 0; i < n; ++i) *(volatile char*)(d + (size_t)i * kPage) = 0;
}

cudaError_t copy_to_host(void* dst, const void* src, size_t bytes, cudaStream_t s) {
    cudaError_t e;
    char* buf = bytes > 0 && is_pageable(dst) ? take_buffer() : nullptr;
    if (!buf) {   // pinned destination, or no ring: one plain copy
        e = cudaMemcpyAsync(dst, src, bytes, cudaMemcpyDeviceToHost, s);
        return e != cudaSuccess ? e : cudaStreamSynchronize(s);
    }
    Events evs;
    const int64_t n = (int64_t)((bytes + kSlotBytes - 1) / kSlotBytes);
    // a power of two, so that one thread handles every use of a slot and slots need no hand-over between threads
    int nt = 1;
    while (2 * nt <= copy_threads(bytes)) nt *= 2;
    int dev = 0;
    e = cudaGetDevice(&dev);
    for (int64_t q = 0; q < std::min<int64_t>(n, kSlots) && e == cudaSuccess; ++q) e = cudaEventCreateWithFlags(&evs.ev[q], cudaEventDisableTiming);
    auto length = [&](int64_t i) { return std::min(kSlotBytes, bytes - (size_t)i * kSlotBytes); };
    auto fill = [&](int64_t i) {
        const int q = (int)(i % kSlots);
        const cudaError_t r = cudaMemcpyAsync(buf + q * kSlotBytes, (const char*)src + (size_t)i * kSlotBytes, length(i), cudaMemcpyDeviceToHost, s);
        return r == cudaSuccess ? cudaEventRecord(evs.ev[q], s) : r;
    };
    for (int64_t i = 0; i < std::min<int64_t>(n, kSlots) && e == cudaSuccess; ++i) e = fill(i);
    if (e == cudaSuccess) {
        std::atomic<int> bad{0};
#pragma omp parallel for num_threads(nt) schedule(static, 1)
        for (int t = 0; t < nt; ++t) {
            cudaError_t r = cudaSetDevice(dev);
            for (int64_t i = t; i < n && r == cudaSuccess && !bad.load(); i += nt) {
                r = cudaEventSynchronize(evs.ev[i % kSlots]);
                if (r != cudaSuccess) break;
                std::memcpy((char*)dst + (size_t)i * kSlotBytes, buf + (i % kSlots) * kSlotBytes, length(i));
                if (i + kSlots < n) r = fill(i + kSlots);
            }
            if (r != cudaSuccess) bad.store((int)r);
        }
        e = (cudaError_t)bad.load();
    }
    if (e != cudaSuccess) cudaStreamSynchronize(s);   // nothing may still be writing into the buffer when it goes back
    give_buffer(buf);
    return e;
}

}  // namespace gad
