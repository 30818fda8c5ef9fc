// Device results into the caller's ordinary (pageable) memory.  A copy to pageable memory goes through the driver's own
// staging buffer on one host thread, and a freshly allocated destination has each of its pages mapped inside that copy: 16 MB of
// logits took 0.93 ms of copying and another millisecond of page faults.  Here the pages are touched by several threads
// while the GPU still computes, and the copy runs through a ring of pinned slots: while the GPU fills some over PCIe, several threads
// move another to its place, a share each.  A copy over PCIe costs 9 us and then 55 bytes a nanosecond (512 KB: 28 GB/s, 2 MB: 46), so
// slots are large where there is much to copy; sharing a slot keeps what is left after the last of them short, and counters instead of a
// fork and a join per slot keep it cheap.  (16 MB: 0.75 ms with a join per 512 KB slot, 0.55 ms with a thread to every slot, 0.45 ms now;
// the bare copy of 16 MB takes 0.30.)
#include <cuda.h>
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

// Pinned memory that lies idle, for all contexts of the process: at most two rings and sixteen small blocks.  It stays when the last
// context goes (pinning 16 KB took 1.0 to 2.3 ms and 8 MB 4 to 6, freeing them 0.4 and 1.3, each wait for the device included: a program
// with one context at a time paid that in every one) until gad_release_pinned or the end of the process.
struct Block { char* p; unsigned long long id; };   // id: the driver's of this very allocation
struct Pool {
    std::mutex lock;
    int users = 0;
    std::vector<Block> idle, idle_small;
} g_pool;

// The driver's identifier of the allocation at p, which no other one ever gets; 0 if there is none.
unsigned long long allocation_id(const void* p) {
    typedef CUresult (*GetAttributeFn)(void*, CUpointer_attribute, CUdeviceptr);
    static const GetAttributeFn get = [] {
        void* f = nullptr;
        cudaDriverEntryPointQueryResult q;
        const bool ok = cudaGetDriverEntryPoint("cuPointerGetAttribute", &f, cudaEnableDefault, &q) == cudaSuccess && q == cudaDriverEntryPointSuccess;
        if (!ok) cudaGetLastError();
        return ok ? (GetAttributeFn)f : nullptr;
    }();
    unsigned long long id = 0;
    return get && get(&id, CU_POINTER_ATTRIBUTE_BUFFER_ID, (CUdeviceptr)p) == CUDA_SUCCESS ? id : 0;
}

// One block of `bytes` from the idle ones, or a new one (null if there is none to be had).  An idle block that is no longer what it was
// (the device has been reset since) is forgotten, not freed.
Block take_from(std::vector<Block>& idle, size_t bytes) {
    for (;;) {
        Block b{nullptr, 0};
        {
            std::lock_guard<std::mutex> g(g_pool.lock);
            if (idle.empty()) break;
            b = idle.back();
            idle.pop_back();
        }
        if (allocation_id(b.p) == b.id) return b;
    }
    void* p = nullptr;
    if (cudaHostAlloc(&p, bytes, cudaHostAllocPortable) != cudaSuccess) { cudaGetLastError(); return {nullptr, 0}; }
    return {(char*)p, allocation_id(p)};
}
void give_to(std::vector<Block>& idle, size_t most, Block b) {
    if (b.id) {
        std::lock_guard<std::mutex> g(g_pool.lock);
        if (idle.size() < most) { idle.push_back(b); return; }
    }
    cudaFreeHost(b.p);
}
Block take_buffer() {
    {
        std::lock_guard<std::mutex> g(g_pool.lock);
        if (g_pool.users <= 0 && g_pool.idle.empty()) return {nullptr, 0};   // no context: pinning a ring for a single copy costs more than it saves
    }
    return take_from(g_pool.idle, kRingBytes);
}
void give_buffer(Block b) { give_to(g_pool.idle, 2, b); }

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
    std::lock_guard<std::mutex> g(g_pool.lock);
    g_pool.users += delta;
}

void release_pinned() {
    std::vector<Block> drop;
    {
        std::lock_guard<std::mutex> g(g_pool.lock);
        drop.swap(g_pool.idle);
        drop.insert(drop.end(), g_pool.idle_small.begin(), g_pool.idle_small.end());
        g_pool.idle_small.clear();
    }
    for (const Block& b : drop)
        if (allocation_id(b.p) == b.id) cudaFreeHost(b.p);
}

// Pinned memory for a context's small results.
Pinned take_small_pinned(size_t bytes) {
    if (bytes <= kSmallPinned) { const Block b = take_from(g_pool.idle_small, kSmallPinned); return {b.p, bytes, b.id}; }
    void* p = nullptr;
    if (cudaHostAlloc(&p, bytes, cudaHostAllocPortable) != cudaSuccess) { cudaGetLastError(); p = nullptr; }
    return {(char*)p, bytes, 0};
}
void give_small_pinned(const Pinned& m) {
    if (m.bytes <= kSmallPinned) give_to(g_pool.idle_small, 16, {m.p, m.id});
    else cudaFreeHost(m.p);
}

void host_prefault(void* dst, size_t bytes) {
    if (bytes < kTouchBytes || !is_pageable(dst)) return;
    char* d = (char*)dst;
    const int64_t n = (int64_t)(bytes / kPage);
#pragma omp parallel if (copy_threads(bytes) > 1)
    {
        const int team = omp_get_num_threads(), t = omp_get_thread_num();
        // adding nothing is a write as far as the page is concerned, and leaves what is there: the copy may never come
        for (int64_t i = n * t / team; i < n * (t + 1) / team; ++i) __atomic_fetch_add(d + (size_t)i * kPage, 0, __ATOMIC_RELAXED);
    }
}

cudaError_t copy_to_host(void* dst, const void* src, size_t bytes, cudaStream_t s) {
    cudaError_t e;
    const Block ring_block = bytes > 0 && is_pageable(dst) ? take_buffer() : Block{nullptr, 0};
    char* buf = ring_block.p;
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
    give_buffer(ring_block);
    return e;
}

}  // namespace gad
