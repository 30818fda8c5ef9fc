// Device results into the caller's ordinary (pageable) memory.  A copy to pageable memory goes through the driver's own
// staging buffer on one host thread, and a freshly allocated destination has each of its pages mapped inside that copy: 16 MB of
// logits took 0.93 ms of copying and another millisecond of page faults.  Here the pages are touched by several threads
// while the GPU still computes, and the copy runs through a ring of pinned slots: while the GPU fills some over PCIe, several threads
// move another to its place, a share each.  A copy over PCIe costs 9 us and then 55 bytes a nanosecond (512 KB: 28 GB/s, 2 MB: 46), so
// slots are large where there is much to copy; sharing a slot keeps what is left after the last of them short, and counters instead of a
// fork and a join per slot keep it cheap.  (16 MB: 0.75 ms with a join per 512 KB slot, 0.55 ms with a thread to every slot, 0.45 ms now;
// the bare copy of 16 MB takes 0.30.)
#include <omp.h>

#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstring>
#include <mutex>
#include <thread>
#include <vector>

#include "gad_internal.h"

namespace gad {

namespace {

constexpr size_t kRingBytes = 8u << 20, kMinSlot = 256u << 10, kMaxSlot = 2u << 20;
constexpr int kSlots = 32, kMaxThreads = 8;   // most slots of a ring; most threads that copy
constexpr size_t kTouchBytes = 1u << 20;  // destinations below this are not worth waking threads for
constexpr size_t kPage = 4096;
constexpr size_t kSmallPinned = 16384;

// Threads that take part.  They belong to the team of all host loops of the library (gad_internal.h); the others of it leave at once.
int copy_threads(size_t bytes) {
    return (int)std::max<size_t>(1, std::min<size_t>({(size_t)kMaxThreads, (size_t)omp_get_num_procs() / 2, bytes / (128u << 10)}));
}

// Pinned buffers of kRingBytes, shared by all contexts of the process: at most two are kept while a context exists, none
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
    return take_from(g_pool.idle, kRingBytes);
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
    const int nt = copy_threads(bytes);
#pragma omp parallel if (nt > 1)
    {
        const int team = std::min(nt, omp_get_num_threads()), t = omp_get_thread_num();
        // adding nothing is a write as far as the page is concerned, and leaves what is there: the copy may never come
        for (int64_t i = n * t / team; t < team && i < n * (t + 1) / team; ++i) __atomic_fetch_add(d + (size_t)i * kPage, 0, __ATOMIC_RELAXED);
    }
}

cudaError_t copy_to_host(void* dst, const void* src, size_t bytes, cudaStream_t s) {
    cudaError_t e;
    char* buf = bytes > 0 && is_pageable(dst) ? take_buffer() : nullptr;
    if (!buf) {   // pinned destination, or no ring: one plain copy
        e = cudaMemcpyAsync(dst, src, bytes, cudaMemcpyDeviceToHost, s);
        return e != cudaSuccess ? e : cudaStreamSynchronize(s);
    }
    // n slots cost 9 us each on the way, and the last one's copying (about as fast as PCIe) comes after the last transfer: together least at
    // slots of sqrt(bytes x 512 KB)
    const size_t slot = std::min(kMaxSlot, std::max(kMinSlot, (size_t)round_up((int64_t)std::sqrt((double)bytes * (512 << 10)), 64 << 10)));
    const int64_t n = (int64_t)((bytes + slot - 1) / slot), ring = std::min<int64_t>(n, (int64_t)(kRingBytes / slot));
    const int nt = copy_threads(bytes);
    Events evs;
    int dev = 0;
    e = cudaGetDevice(&dev);
    for (int64_t q = 0; q < ring && e == cudaSuccess; ++q) e = cudaEventCreateWithFlags(&evs.ev[q], cudaEventDisableTiming);
    auto length = [&](int64_t i) { return std::min(slot, bytes - (size_t)i * slot); };
    std::atomic<int64_t> filled[kSlots];          // what a slot holds, or is being filled with
    for (std::atomic<int64_t>& f : filled) f.store(-1);
    auto fill = [&](int64_t i) {
        const int64_t q = i % ring;
        const cudaError_t r = cudaMemcpyAsync(buf + q * slot, (const char*)src + (size_t)i * slot, length(i), cudaMemcpyDeviceToHost, s);
        if (r != cudaSuccess) return r;
        const cudaError_t v = cudaEventRecord(evs.ev[q], s);
        if (v == cudaSuccess) filled[q].store(i, std::memory_order_release);
        return v;
    };
    for (int64_t i = 0; i < ring && e == cudaSuccess; ++i) e = fill(i);
    if (e == cudaSuccess) {
        std::atomic<int> bad{0};
        std::atomic<int64_t> arrived{0};          // slots known to have arrived
        std::atomic<bool> waiting{false};         // a thread waits for the next one (for all of them)
        std::atomic<int> moved[kSlots] = {};      // shares of a slot's contents that have been moved
        auto wait_for_slot = [&](int64_t i) {
            while (arrived.load(std::memory_order_acquire) <= i && !bad.load()) {
                if (waiting.exchange(true)) { std::this_thread::yield(); continue; }
                const int64_t a = arrived.load(std::memory_order_acquire);
                if (filled[a % ring].load(std::memory_order_acquire) != a) std::this_thread::yield();   // others are still at its last contents
                else if (a <= i) {
                    const cudaError_t r = cudaEventSynchronize(evs.ev[a % ring]);
                    if (r != cudaSuccess) bad.store((int)r);
                    else arrived.store(a + 1, std::memory_order_release);
                }
                waiting.store(false);
            }
        };
#pragma omp parallel if (nt > 1)
        {
            const int team = std::min(nt, omp_get_num_threads()), t = omp_get_thread_num();
            const cudaError_t r = t < team ? cudaSetDevice(dev) : cudaSuccess;
            if (r != cudaSuccess) bad.store((int)r);
            for (int64_t i = 0; t < team && i < n && !bad.load(); ++i) {
                wait_for_slot(i);
                if (bad.load()) break;
                const size_t len = length(i), lo = len * (size_t)t / team / 64 * 64, hi = t + 1 == team ? len : len * (size_t)(t + 1) / team / 64 * 64;
                std::memcpy((char*)dst + (size_t)i * slot + lo, buf + (i % ring) * slot + lo, hi - lo);
                if (moved[i % ring].fetch_add(1) + 1 == team) {
                    moved[i % ring].store(0);
                    if (i + ring < n) {
                        const cudaError_t f = fill(i + ring);
                        if (f != cudaSuccess) bad.store((int)f);
                    }
                }
            }
        }
        e = (cudaError_t)bad.load();
    }
    if (e != cudaSuccess) cudaStreamSynchronize(s);   // nothing may still be writing into the buffer when it goes back
    give_buffer(buf);
    return e;
}

}  // namespace gad
