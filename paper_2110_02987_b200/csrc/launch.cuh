// Launches of the main sequence of an epoch.  Each kernel may start before the one in front of it has finished (programmatic dependent
// launch): its blocks come up, set up barriers and tensor memory and read what no kernel writes while the last blocks in front still
// run, and wait (pdl_wait) before they touch anything else.  pdl_next lets the next kernel start; it is called first of all, because the
// blocks of that kernel are only placed where no block of this one is waiting for room.  Without it the gaps and set-up between the
// kernels of a 2000-node epoch were a third of its time.
#pragma once

#include <cuda_runtime.h>

#include <utility>

namespace gad {

__device__ __forceinline__ void pdl_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
// Everything the kernels in front have written is visible after this.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
// The compiler may move a load through a pointer it knows to be read-only ahead of the wait: a pointer that has passed through here after
// it cannot have been used before.
template <class P> __device__ __forceinline__ void after_wait(P& p) {
    unsigned long long a = (unsigned long long)p;
    asm volatile("" : "+l"(a));
    p = (P)a;
}

// Set while an epoch is enqueued: the stream of the main sequence, whether all its kernels overlap or the finishing ones only, and whether
// the next kernel on it directly follows a kernel.
struct PdlState { cudaStream_t stream = nullptr; bool on = false, direct = false, tails = false; };   // tails: those of launch_tail only
PdlState& pdl_state();   // of this thread

// How much shared memory an SM sets aside while it runs a kernel (the rest of its 256 KB is L1) is changed only when the SM is empty, and a
// kernel that does not ask runs with what the SM has been cut for.  Where blocks of a small kernel beside the aggregation had come up on
// SMs still cut for a transform (227 KB), the whole aggregation behind them ran with the L1 that leaves, which holds fewer operand rows
// in flight than its warps ask for (8 x 7800 rows of 265 entries, 256 wide: 807 us beside the importance statistics, 609 on its own, now 633).
// So these kernels ask: the aggregation for what its blocks need (16 of 2 KB), the importance statistics for four blocks of 17 KB.
// Not where the kernels of the main sequence overlap: each change then waits for an SM that the overlap keeps busy (2708 rows: 163 -> 166 us an epoch).
constexpr unsigned kGatherSharedKB = 32, kZetaSharedKB = 100;

// When a kernel may come up ahead of the end of the one in front: never, where the whole main sequence overlaps, or as a finishing kernel too.
enum class Early { kNever, kOverlap, kTail };

template <class... P, class... Args>
cudaError_t launch_cluster(void (*kernel)(P...), dim3 grid, unsigned block, size_t smem, unsigned cluster, Early early, unsigned shared_kb, cudaStream_t s,
                           Args&&... args) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid; cfg.blockDim = dim3(block); cfg.dynamicSmemBytes = smem; cfg.stream = s;
    cudaLaunchAttribute attr[3];
    cfg.attrs = attr;
    if (cluster > 1) {
        attr[cfg.numAttrs].id = cudaLaunchAttributeClusterDimension;
        attr[cfg.numAttrs].val.clusterDim.x = cluster; attr[cfg.numAttrs].val.clusterDim.y = 1; attr[cfg.numAttrs].val.clusterDim.z = 1;
        ++cfg.numAttrs;
    }
    PdlState& st = pdl_state();
    if ((st.on || st.tails) && s == st.stream && early != Early::kNever) {
        if (st.direct && (st.on || early == Early::kTail)) {
            attr[cfg.numAttrs].id = cudaLaunchAttributeProgrammaticStreamSerialization;
            attr[cfg.numAttrs].val.programmaticStreamSerializationAllowed = 1;
            ++cfg.numAttrs;
        }
        st.direct = true;
    }
    if (shared_kb && !st.on) {
        attr[cfg.numAttrs].id = cudaLaunchAttributePreferredSharedMemoryCarveout;
        attr[cfg.numAttrs].val.sharedMemCarveout = 100 * shared_kb / 228;   // percent; rounded up to a size there is
        ++cfg.numAttrs;
    }
    return cudaLaunchKernelEx(&cfg, kernel, P(std::forward<Args>(args))...);
}
template <class... P, class... Args>
cudaError_t launch(void (*kernel)(P...), dim3 grid, unsigned block, size_t smem, cudaStream_t s, Args&&... args) {
    return launch_cluster(kernel, grid, block, smem, 1, Early::kOverlap, 0, s, std::forward<Args>(args)...);
}
// The same for a kernel that asks for a share of the SM's memory (kGatherSharedKB, kZetaSharedKB).
template <class... P, class... Args>
cudaError_t launch_share(void (*kernel)(P...), dim3 grid, unsigned block, unsigned shared_kb, cudaStream_t s, Args&&... args) {
    return launch_cluster(kernel, grid, block, 0, 1, Early::kOverlap, shared_kb, s, std::forward<Args>(args)...);
}
// The same for a kernel of the side work.  It does not wait for the one in front (pdl_wait), so it never comes up early, on whatever stream: a pointer that
// has passed through after_wait is no longer known to be read-only, and the importance statistics of 1200 features took 64 us that way instead of 44.
template <class... P, class... Args>
cudaError_t launch_beside(void (*kernel)(P...), dim3 grid, unsigned block, unsigned shared_kb, cudaStream_t s, Args&&... args) {
    return launch_cluster(kernel, grid, block, 0, 1, Early::kNever, shared_kb, s, std::forward<Args>(args)...);
}
// A small kernel that only finishes what the one in front has left (rows cut into parts, sums of chunks): its blocks find room beside the
// last ones in front on a store of any size (89 250 rows in 50 subgraphs: 912 -> 903 us an epoch; 70 000 of 60-60-60-5: 362 -> 356).
template <class... P, class... Args>
cudaError_t launch_tail(void (*kernel)(P...), dim3 grid, unsigned block, size_t smem, cudaStream_t s, Args&&... args) {
    return launch_cluster(kernel, grid, block, smem, 1, Early::kTail, 0, s, std::forward<Args>(args)...);
}

// A kernel of one or two blocks for every SM, each with work for several microseconds, does not come up early: its blocks would go where
// the kernel in front leaves room first, eight to sixteen on an SM, and the other SMs would have none (weight gradient of 20 x 6 over
// 47 250 rows: 17 us, spread over all SMs 6).
template <class... P, class... Args>
cudaError_t launch_spread(void (*kernel)(P...), dim3 grid, unsigned block, size_t smem, cudaStream_t s, Args&&... args) {
    if (s == pdl_state().stream) pdl_state().direct = false;
    return launch(kernel, grid, block, smem, s, std::forward<Args>(args)...);
}

}  // namespace gad
