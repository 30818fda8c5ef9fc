// What the tensor-core transforms (gemm_rows.cu, gemm_tn.cu) are given: the TF32 split of the weights and the TMA descriptors; and their
// bounded wait made to run out.
#include <cuda.h>

#include "epilogue.cuh"
#include "gad_internal.h"
#include "tc_common.cuh"

namespace gad {

namespace {

constexpr int BK = 32;   // values of an operand row per TMA box (128 bytes)

// W_k^(l) [fi x ldw] -> the K-major operand copies the tensor-core kernels read, for every layer in one launch:
//   w_hi / w_lo   [K][fi][ldw]    (B of mode 1: rows n = input feature, Kd = output feature; only layers l >= 1 have a dH)
//   wt_hi / wt_lo [K][fo][ldkt]   (B of mode 0: rows n = output feature, Kd = input feature)
// A 32 x 32 block per CTA, turned through shared memory so that both layouts are written in whole rows (written straight from
// the plain layout, a 500 x 128 layer of 50 replicas took 39 us, bound by its 4-byte column writes).
__global__ void __launch_bounds__(256) split_weights_kernel(const float* __restrict__ params, long long pstride, const SplitLayers ls) {
    __shared__ float th[32][33], tl[32][33];
    pdl_next();
    const SplitLayer& y = ls.y[blockIdx.z];
    const int ntj = (y.ldw + 31) / 32, ntiles = ((y.fi + 31) / 32) * ntj;
    if ((int)blockIdx.x >= ntiles) return;
    const int i0 = ((int)blockIdx.x / ntj) * 32, j0 = ((int)blockIdx.x % ntj) * 32, k = blockIdx.y;
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    pdl_wait();
    after_wait(params);
    const float* W = params + (long long)k * pstride + y.w_int;
#pragma unroll
    for (int r = 0; r < 32; r += 8) {
        const int i = i0 + ty + r, j = j0 + tx;
        if (i < y.fi && j < y.ldw) {
            const long long idx = (long long)i * y.ldw + j;
            const float w = W[idx], h = tf32_hi(w), l = tf32_round(w - h);
            if (y.w_hi) { y.w_hi[(long long)k * y.fi * y.ldw + idx] = h; y.w_lo[(long long)k * y.fi * y.ldw + idx] = l; }
            th[ty + r][tx] = h; tl[ty + r][tx] = l;
        }
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < 32; r += 8) {
        const int j = j0 + ty + r, i = i0 + tx;
        if (j < y.fo && i < y.fi) {
            const long long at = ((long long)k * y.fo + j) * y.ldkt + i;
            y.wt_hi[at] = th[tx][ty + r]; y.wt_lo[at] = tl[tx][ty + r];
        }
    }
}

// The bounded wait of the tensor-core kernels, made to run out: one thread polls a barrier that nothing ever arrives at.
__global__ void expire_wait_kernel(int32_t* err, uint32_t polls) {
    __shared__ __align__(8) uint64_t bar;
    __shared__ uint32_t abort_flag;
    if (threadIdx.x == 0) {
        mbar_init(smem_u32(&bar), 1);
        abort_flag = 0u;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        mbar_wait(smem_u32(&bar), 0u, &abort_flag, err, 99, polls);
    }
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                                  const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn() {
    static EncodeTiledFn fn = nullptr;
    if (!fn) {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) == cudaSuccess && q == cudaDriverEntryPointSuccess)
            fn = (EncodeTiledFn)p;
    }
    return fn;
}

}  // namespace

// fp32 tensor [outer (z)] x [rows (y)] x [inner (x)], box = 32 floats (`half`: 64 fp16 values) x box_rows x 1, zero fill outside.  K-major
// operand tiles use the 128-byte swizzle of 16-byte units; MN-major TF32 tiles need the 128-byte swizzle of
// 32-byte units (the only MN-major layout the tensor cores accept for 32-bit operands).
bool tc_make_map(void* out_map, const void* base, uint64_t inner, uint64_t rows, uint64_t outer, uint64_t row_stride_bytes,
                 uint64_t outer_stride_bytes, uint32_t box_rows, bool mn_major, bool half) {
    EncodeTiledFn fn = encode_fn();
    if (!fn) return false;
    const bool three = outer > 0;
    cuuint64_t dims[3] = {inner, rows, three ? outer : 1};
    cuuint64_t strides[2] = {row_stride_bytes, outer_stride_bytes};
    cuuint32_t box[3] = {(cuuint32_t)(half ? 2 * BK : BK), box_rows, 1};
    cuuint32_t estr[3] = {1, 1, 1};
    CUresult r = fn(reinterpret_cast<CUtensorMap*>(out_map), half ? CU_TENSOR_MAP_DATA_TYPE_FLOAT16 : CU_TENSOR_MAP_DATA_TYPE_FLOAT32, three ? 3 : 2, const_cast<void*>(base), dims,
                    strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                    mn_major ? CU_TENSOR_MAP_SWIZZLE_128B_ATOM_32B : CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS;
}

cudaError_t launch_expire_wait(int32_t* err, uint32_t polls, cudaStream_t s) {
    expire_wait_kernel<<<1, 32, 0, s>>>(err, polls);
    ++g_kernel_launches;
    return cudaGetLastError();
}

cudaError_t launch_split_weights(const float* params, int64_t pstride, int K, const SplitLayer* layers, int L, cudaStream_t s) {
    for (int l0 = 0; l0 < L; l0 += SplitLayers::MAX) {
        SplitLayers ls{};
        const int n = L - l0 < SplitLayers::MAX ? L - l0 : SplitLayers::MAX;
        int tiles = 0;
        for (int l = 0; l < n; ++l) {
            ls.y[l] = layers[l0 + l];
            const int t = ((ls.y[l].fi + 31) / 32) * ((ls.y[l].ldw + 31) / 32);
            tiles = tiles > t ? tiles : t;
        }
        launch(split_weights_kernel, dim3((unsigned)tiles, (unsigned)K, (unsigned)n), 256, 0, s, params, pstride, ls);
        ++g_kernel_launches;
    }
    return cudaGetLastError();
}

}  // namespace gad
