// Memory-bound kernels of the epoch other than the SpMM: fused softmax cross-entropy with its gradient,
// chunked column sums, the statistics of the variance-based importance weight, the fused SGD step +
// weighted global consensus, and the create-time / accessor gathers.  Every reduction runs in a fixed order
// (rows of a chunk in order, chunks of a subgraph in order, replicas in ascending k), so a run is bitwise
// reproducible.
#include <math.h>

#include "epilogue.cuh"
#include "gad_internal.h"

namespace gad {

// ---------------------------------------------------------------------------------------------
// "The last CTA finishes the reduction": every CTA writes its partial result, then counts itself in; the CTA
// whose arrival completes the group adds the partial results in their fixed order.  Which CTA that is varies
// from run to run, the order of the additions does not, so the results stay bitwise reproducible.  Counters only
// grow (a group is complete at every multiple of its size), so they never need resetting.
// ---------------------------------------------------------------------------------------------
__device__ __forceinline__ bool cta_arrive_last(unsigned* counter, unsigned expected) {
    __shared__ unsigned last_flag;
    __threadfence();                  // this CTA's partial results are visible before its arrival is counted
    __syncthreads();
    if (threadIdx.x == 0) last_flag = (atomicAdd(counter, 1u) + 1u) % expected == 0u ? 1u : 0u;
    __syncthreads();
    const bool last = last_flag != 0u;
    if (last) __threadfence();        // the other CTAs published their results before they arrived
    return last;
}

// Sum over the chunks [c0, c1) of src[c * stride + j], for one column j, as the finishing CTA does it: the chunk
// range is cut into `nseg` equal segments, segment `seg` is added in chunk order by the calling thread (up to
// eight loads in flight), and the caller then adds the segment sums in segment order.  The order of the additions
// depends only on (c0, c1, nseg).
template <class T>
__device__ __forceinline__ T segment_sum(const T* src, long long stride, long long j, int c0, int c1, int seg, int nseg) {
    const int len = (c1 - c0 + nseg - 1) / nseg;
    int c = c0 + seg * len;
    const int e = min(c1, c + len);
    T s = (T)0;
    for (; c + 8 <= e; c += 8) {
        T v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) v[u] = __ldcg(src + (long long)(c + u) * stride + j);
#pragma unroll
        for (int u = 0; u < 8; ++u) s += v[u];
    }
    for (; c < e; ++c) s += __ldcg(src + (long long)c * stride + j);
    return s;
}
// Columns are handled T / nseg at a time by T threads; nseg = T / (columns rounded up to a power of two), at least 1.
__device__ __forceinline__ int segments_for(int cols, int T = 256) {
    int p = 1;
    while (p < cols && p < T) p <<= 1;
    return T / p;
}

// What follows the loss kernel, beside the backward pass: the CTA of subgraph k adds up the column sums of its chunks' d logits
// (the bias gradient of the last layer; bias_ld == 0: none were taken), the last CTA the losses.  The chunk losses are first
// brought into shared memory by the whole CTA (4096 at a time); one thread per subgraph then adds its subgraph's sums in chunk order,
// and thread 0 adds the K subgraph sums in ascending k for the global loss sum_k |T_k| L_k / sum_k |T_k|.
__global__ void __launch_bounds__(256) loss_finish_kernel(const float* __restrict__ loss_partial, const float* __restrict__ inv_ntrain,
                                                          const int32_t* __restrict__ chunk_ptr, int K, float inv_total, float* __restrict__ loss,
                                                          int32_t* __restrict__ nonfinite, const float* __restrict__ bias_partial,
                                                          long long pstride_chunk, int bias_ld, float* __restrict__ out, long long ostride,
                                                          long long off) {
    if ((int)blockIdx.x < K && bias_ld > 0) {
        __shared__ float seg_sm[256];
        const int k = blockIdx.x, c0 = chunk_ptr[k], c1 = chunk_ptr[k + 1];
        const int nseg = segments_for(bias_ld), per = 256 / nseg;
        const int jl = threadIdx.x % per, seg = threadIdx.x / per;
        for (int j0 = 0; j0 < bias_ld; j0 += per) {
            const int j = j0 + jl;
            seg_sm[threadIdx.x] = j < bias_ld ? segment_sum(bias_partial, pstride_chunk, j, c0, c1, seg, nseg) : 0.f;
            __syncthreads();
            if (seg == 0 && j < bias_ld) {
                float t = seg_sm[jl];
                for (int q = 1; q < nseg; ++q) t += seg_sm[q * per + jl];
                out[(long long)k * ostride + off + j] = t;
            }
            __syncthreads();
        }
        return;
    }
    __shared__ float stage[4096];
    __shared__ float sums[1024];
    const int nchunks = chunk_ptr[K];
    const bool staged = nchunks <= 4096;
    if (staged)
        for (int c = threadIdx.x; c < nchunks; c += blockDim.x) stage[c] = loss_partial[c];
    __syncthreads();
    for (int k = threadIdx.x; k < K; k += blockDim.x) {
        float s = 0.f;
        for (int c = chunk_ptr[k]; c < chunk_ptr[k + 1]; ++c) s += staged ? stage[c] : loss_partial[c];
        if (k < 1024) sums[k] = s;
        loss[k] = s * inv_ntrain[k];
        if (!isfinite(s)) atomicExch(nonfinite, 1);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        float s = 0.f;
        for (int k = 0; k < K; ++k) {
            if (k < 1024) { s += sums[k]; continue; }
            float sk = 0.f;
            for (int c = chunk_ptr[k]; c < chunk_ptr[k + 1]; ++c) sk += staged ? stage[c] : loss_partial[c];
            s += sk;
        }
        loss[K] = s * inv_total;
    }
}
cudaError_t launch_loss_finish(const float* loss_partial, const float* inv_ntrain, const int32_t* chunk_ptr, int K, float inv_total, float* loss,
                               int32_t* nonfinite, const float* bias_partial, int64_t pstride_chunk, int bias_ld, float* out, int64_t ostride,
                               int64_t off, cudaStream_t s) {
    loss_finish_kernel<<<(unsigned)(bias_ld > 0 ? K + 1 : 1), 256, 0, s>>>(loss_partial, inv_ntrain, chunk_ptr, K, inv_total, loss, nonfinite, bias_partial,
                                                                          pstride_chunk, bias_ld, out, ostride, off);
    ++g_kernel_launches;
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------------------------
// Softmax cross-entropy over the core training rows and d(loss)/d(logits)  (loss equation, Section 3.3, read
// as multi-class cross-entropy averaged over the subgraph's training nodes).  One CTA per row chunk, one warp
// per row; lanes stride over the classes.
// ---------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(256) softmax_xent_kernel(const float* __restrict__ logits, int ld, int C,
                                                           const int32_t* __restrict__ label,
                                                           const uint8_t* __restrict__ train,
                                                           const RowSpan* __restrict__ chunks,
                                                           const float* __restrict__ inv_ntrain,
                                                           float* __restrict__ dlogits, float* __restrict__ loss_partial) {
    __shared__ float wsum[8];
    pdl_next();
    const RowSpan c = chunks[blockIdx.x];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const float inv = inv_ntrain[c.k];
    pdl_wait();
    after_wait(logits);
    float acc = 0.f;
    for (int r = warp; r < c.nrows; r += 8) {
        const long long row = c.row0 + r;
        const float* z = logits + row * ld;
        float* g = dlogits + row * ld;
        if (!train[row]) {
            for (int j = lane; j < ld; j += 32) g[j] = 0.f;
            continue;
        }
        float mx = -INFINITY;
        for (int j = lane; j < C; j += 32) mx = fmaxf(mx, z[j]);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        float se = 0.f;
        for (int j = lane; j < C; j += 32) se += expf(z[j] - mx);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) se += __shfl_xor_sync(0xffffffffu, se, o);
        const float lse = mx + logf(se);
        const int y = label[row];
        acc += lse - z[y];
        for (int j = lane; j < ld; j += 32) {
            float v = 0.f;
            if (j < C) v = (expf(z[j] - lse) - (j == y ? 1.f : 0.f)) * inv;
            g[j] = v;
        }
    }
    if (lane == 0) wsum[warp] = acc;  // every lane holds the same acc
    __syncthreads();
    if (threadIdx.x == 0) {
        float s = 0.f;
        for (int w = 0; w < 8; ++w) s += wsum[w];
        loss_partial[blockIdx.x] = s;
    }
}

// Up to 128 classes: L lanes hold one row (a float4 each), 32/L rows per warp step, the row stays in registers.  The column sums of
// d logits (the bias gradient of the last layer) come out of the same pass: per chunk into cs_partial.  dlogits_bf (may be null): d logits
// go there in bfloat16 instead, the operand copy of the reduced-precision aggregation.
template <int L>
__global__ void __launch_bounds__(256) softmax_xent_small_kernel(const float* __restrict__ logits, int ld, int C,
                                                                 const int32_t* __restrict__ label,
                                                                 const uint8_t* __restrict__ train,
                                                                 const RowSpan* __restrict__ chunks,
                                                                 const float* __restrict__ inv_ntrain,
                                                                 float* __restrict__ dlogits, float* __restrict__ loss_partial,
                                                                 float* __restrict__ cs_partial, long long pstride_chunk,
                                                                 uint2* __restrict__ dlogits_bf) {
    constexpr int RPW = 32 / L;
    __shared__ float wsum[8];
    __shared__ float4 csum[8][L];
    float4 cs = make_float4(0.f, 0.f, 0.f, 0.f);
    const RowSpan c = chunks[blockIdx.x];
    pdl_next();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int g = lane / L, gl = lane & (L - 1);
    const unsigned gmask = L == 32 ? 0xffffffffu : (((1u << L) - 1u) << (lane & ~(L - 1)));
    const int ld4 = ld >> 2;
    const float inv = inv_ntrain[c.k];
    float acc = 0.f;
    pdl_wait();
    after_wait(logits);
    after_wait(label);
    // the loads of a row (loss mask, label, logits) do not wait for one another, and the next row's are requested
    // before this row's are used
    struct RowIn { bool train; int y; float4 v; };
    auto fetch = [&](int r) {
        RowIn in{false, 0, make_float4(0.f, 0.f, 0.f, 0.f)};
        if (r < c.nrows) {
            const long long row = c.row0 + r;
            in.train = train[row] != 0;
            in.y = label[row];
            if (gl < ld4) in.v = reinterpret_cast<const float4*>(logits + row * ld)[gl];
        }
        return in;
    };
    auto finish = [&](int r, const RowIn& cur) {
        const long long row = c.row0 + r;
        float4* gout = reinterpret_cast<float4*>(dlogits + row * ld);
        if (!cur.train) {
            if (gl < ld4) {
                if (dlogits_bf) dlogits_bf[row * ld4 + gl] = make_uint2(0u, 0u);
                else gout[gl] = make_float4(0.f, 0.f, 0.f, 0.f);
            }
            return;
        }
        float z[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
        if (gl < ld4) {
            const float4 v = cur.v;
            if (4 * gl + 0 < C) z[0] = v.x;
            if (4 * gl + 1 < C) z[1] = v.y;
            if (4 * gl + 2 < C) z[2] = v.z;
            if (4 * gl + 3 < C) z[3] = v.w;
        }
        float mx = fmaxf(fmaxf(z[0], z[1]), fmaxf(z[2], z[3]));
#pragma unroll
        for (int o = L / 2; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(gmask, mx, o, L));
        float se = 0.f, ex[4];
#pragma unroll
        for (int t = 0; t < 4; ++t) { ex[t] = 4 * gl + t < C ? expf(z[t] - mx) : 0.f; se += ex[t]; }
#pragma unroll
        for (int o = L / 2; o > 0; o >>= 1) se += __shfl_xor_sync(gmask, se, o, L);
        const float lse = mx + logf(se), inv_se = 1.f / se;
        const int y = cur.y;
        const int yt = y & 3;
        const float mine = yt == 0 ? z[0] : (yt == 1 ? z[1] : (yt == 2 ? z[2] : z[3]));
        const float zy = __shfl_sync(gmask, mine, y >> 2, L);
        if (gl == 0) acc += lse - zy;
        if (gl < ld4) {
            float o4[4];
#pragma unroll
            for (int t = 0; t < 4; ++t) {
                const int j = 4 * gl + t;
                o4[t] = j < C ? (ex[t] * inv_se - (j == y ? 1.f : 0.f)) * inv : 0.f;
            }
            if (dlogits_bf) dlogits_bf[row * ld4 + gl] = bf16_pack4(make_float4(o4[0], o4[1], o4[2], o4[3]));
            else gout[gl] = make_float4(o4[0], o4[1], o4[2], o4[3]);
            cs.x += o4[0]; cs.y += o4[1]; cs.z += o4[2]; cs.w += o4[3];
        }
    };
    // Two rows per lane group at a time, and the next two on their way.
    int r = warp * RPW + g;
    RowIn a0 = fetch(r), a1 = fetch(r + 8 * RPW);
    for (; r < c.nrows; r += 16 * RPW) {
        const RowIn n0 = fetch(r + 16 * RPW), n1 = fetch(r + 24 * RPW);
        finish(r, a0);
        if (r + 8 * RPW < c.nrows) finish(r + 8 * RPW, a1);
        a0 = n0; a1 = n1;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
#pragma unroll
    for (int o = 16; o >= L; o >>= 1) {   // the row groups of the warp
        cs.x += __shfl_xor_sync(0xffffffffu, cs.x, o); cs.y += __shfl_xor_sync(0xffffffffu, cs.y, o);
        cs.z += __shfl_xor_sync(0xffffffffu, cs.z, o); cs.w += __shfl_xor_sync(0xffffffffu, cs.w, o);
    }
    if (lane == 0) wsum[warp] = acc;
    if (lane < L) csum[warp][lane] = cs;
    __syncthreads();
    if (threadIdx.x == 0) {
        float s = 0.f;
        for (int w = 0; w < 8; ++w) s += wsum[w];
        loss_partial[blockIdx.x] = s;
    }
    if ((int)threadIdx.x < ld4) {
        float4 t = csum[0][threadIdx.x];
        for (int w = 1; w < 8; ++w) { const float4 u = csum[w][threadIdx.x]; t.x += u.x; t.y += u.y; t.z += u.z; t.w += u.w; }
        reinterpret_cast<float4*>(cs_partial + (long long)blockIdx.x * pstride_chunk)[threadIdx.x] = t;
    }
}

bool softmax_sums_columns(int ld) { return ld <= 128; }
cudaError_t launch_softmax_xent(const float* logits, int ld, int C, const int32_t* label, const uint8_t* train,
                                const RowSpan* chunks, int nchunks, const float* inv_ntrain, float* dlogits,
                                float* loss_partial, float* cs_partial, int64_t pstride_chunk, void* dlogits_bf16, cudaStream_t s) {
    if (nchunks > 0) {
        const int ld4 = ld >> 2;
#define GAD_SMALL(L) launch(softmax_xent_small_kernel<L>, dim3((unsigned)nchunks), 256, 0, s, logits, ld, C, label, train, chunks, inv_ntrain, dlogits, loss_partial, cs_partial, pstride_chunk, reinterpret_cast<uint2*>(dlogits_bf16))
        if (ld4 <= 1) GAD_SMALL(1);
        else if (ld4 <= 2) GAD_SMALL(2);
        else if (ld4 <= 4) GAD_SMALL(4);
        else if (ld4 <= 8) GAD_SMALL(8);
        else if (ld4 <= 16) GAD_SMALL(16);
        else if (ld4 <= 32) GAD_SMALL(32);
        else launch(softmax_xent_kernel, dim3((unsigned)nchunks), 256, 0, s, logits, ld, C, label, train, chunks, inv_ntrain, dlogits, loss_partial);
#undef GAD_SMALL
        ++g_kernel_launches;
    }
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------------------------
// Column sums of a row chunk (bias gradient db = column sums of dPre over the subgraph's rows).
// ---------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(256) colsum_chunks_kernel(const float* __restrict__ G, int ld,
                                                            const RowSpan* __restrict__ chunks, float* partial,
                                                            long long pstride_chunk, const int32_t* __restrict__ chunk_ptr,
                                                            unsigned* counters, float* __restrict__ out, long long ostride,
                                                            long long off) {
    // threads = 8 row lanes x 32 column lanes of one float4 each; a block of 128 columns is summed over the
    // rows ry, ry+8, ... by every row lane and the 8 row lanes are then added in order
    __shared__ float4 sm[8][32];
    const RowSpan c = chunks[blockIdx.x];
    const int cx = threadIdx.x & 31, ry = threadIdx.x >> 5;
    const int ld4 = ld >> 2;
    for (int v0 = 0; v0 < ld4; v0 += 32) {
        const int v = v0 + cx;
        float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
        if (v < ld4) {
            const float4* g = reinterpret_cast<const float4*>(G + (long long)c.row0 * ld) + v;
            int r = ry;
            for (; r + 24 < c.nrows; r += 32) {
                float4 a0 = g[(long long)r * ld4], a1 = g[(long long)(r + 8) * ld4];
                float4 a2 = g[(long long)(r + 16) * ld4], a3 = g[(long long)(r + 24) * ld4];
                s.x += a0.x; s.y += a0.y; s.z += a0.z; s.w += a0.w;
                s.x += a1.x; s.y += a1.y; s.z += a1.z; s.w += a1.w;
                s.x += a2.x; s.y += a2.y; s.z += a2.z; s.w += a2.w;
                s.x += a3.x; s.y += a3.y; s.z += a3.z; s.w += a3.w;
            }
            for (; r < c.nrows; r += 8) {
                float4 a0 = g[(long long)r * ld4];
                s.x += a0.x; s.y += a0.y; s.z += a0.z; s.w += a0.w;
            }
        }
        sm[ry][cx] = s;
        __syncthreads();
        if (ry == 0 && v < ld4) {
            float4 t = sm[0][cx];
            for (int w = 1; w < 8; ++w) { t.x += sm[w][cx].x; t.y += sm[w][cx].y; t.z += sm[w][cx].z; t.w += sm[w][cx].w; }
            reinterpret_cast<float4*>(partial + (long long)blockIdx.x * pstride_chunk)[v] = t;
        }
        __syncthreads();
    }
    // the last CTA of this subgraph adds the subgraph's chunk sums: segments of the chunk range in parallel, then
    // the segment sums in order
    const int c0 = chunk_ptr[c.k], c1 = chunk_ptr[c.k + 1];
    if (!cta_arrive_last(counters + c.k, (unsigned)(c1 - c0))) return;
    float* seg_sm = reinterpret_cast<float*>(sm);   // 256 floats of the 4 KiB tile above
    const int nseg = segments_for(ld), per = 256 / nseg;
    const int jl = threadIdx.x % per, seg = threadIdx.x / per;
    for (int j0 = 0; j0 < ld; j0 += per) {
        const int j = j0 + jl;
        seg_sm[threadIdx.x] = j < ld ? segment_sum(partial, pstride_chunk, j, c0, c1, seg, nseg) : 0.f;
        __syncthreads();
        if (seg == 0 && j < ld) {
            float t = seg_sm[jl];
            for (int q = 1; q < nseg; ++q) t += seg_sm[q * per + jl];
            out[(long long)c.k * ostride + off + j] = t;
        }
        __syncthreads();
    }
}
// Column sums of G over every subgraph's rows: out[k][off + j] = sum over the rows of subgraph k of G[row][j], j < ld.
cudaError_t launch_colsum_chunks(const float* G, int ld, const RowSpan* chunks, int nchunks, float* partial,
                                 int64_t pstride_chunk, const int32_t* chunk_ptr, unsigned* counters, float* out,
                                 int64_t ostride, int64_t off, cudaStream_t s) {
    if (nchunks > 0) {
        colsum_chunks_kernel<<<(unsigned)nchunks, 256, 0, s>>>(G, ld, chunks, partial, pstride_chunk, chunk_ptr, counters, out, ostride, off);
        ++g_kernel_launches;
    }
    return cudaGetLastError();
}

__global__ void __launch_bounds__(256) colsum_finish_kernel(const float* __restrict__ colsum, int ld, const int2* __restrict__ clusters,
                                                            float* __restrict__ out, long long ostride, long long off) {
    __shared__ float seg_sm[256];
    const int k = blockIdx.x;
    const int2 r = clusters[k];
    const int c0 = (r.x + k) * 8, c1 = (r.y + k + 1) * 8;   // rows of the partial sums
    const int nseg = segments_for(ld), per = 256 / nseg;
    const int jl = threadIdx.x % per, seg = threadIdx.x / per;
    for (int j0 = 0; j0 < ld; j0 += per) {
        const int j = j0 + jl;
        seg_sm[threadIdx.x] = j < ld ? segment_sum(colsum, ld, j, c0, c1, seg, nseg) : 0.f;
        __syncthreads();
        if (seg == 0 && j < ld) {
            float t = seg_sm[jl];
            for (int q = 1; q < nseg; ++q) t += seg_sm[q * per + jl];
            out[(long long)k * ostride + off + j] = t;
        }
        __syncthreads();
    }
}
cudaError_t launch_colsum_finish(const float* colsum, int ld, const int2* clusters, int K, float* out, int64_t ostride, int64_t off, cudaStream_t s) {
    launch_beside(colsum_finish_kernel, dim3((unsigned)K), 256, kGatherSharedKB, s, colsum, ld, clusters, out, ostride, off);
    ++g_kernel_launches;
    return cudaGetLastError();
}

__global__ void reduce_chunks_kernel(const float* __restrict__ partial, long long pstride_chunk,
                                     const int32_t* __restrict__ chunk_ptr, float* __restrict__ out, long long ostride,
                                     long long off, long long len) {
    pdl_next();
    const int k = blockIdx.y;
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= len) return;
    pdl_wait();
    after_wait(partial);
    float s = 0.f;
    const int c1 = chunk_ptr[k + 1];
    int c = chunk_ptr[k];
    for (; c + 8 <= c1; c += 8) {   // eight chunks' values requested together, added in chunk order
        float v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) v[u] = partial[(long long)(c + u) * pstride_chunk + i];
#pragma unroll
        for (int u = 0; u < 8; ++u) s += v[u];
    }
    for (; c < c1; ++c) s += partial[(long long)c * pstride_chunk + i];
    out[(long long)k * ostride + off + i] = s;
}
cudaError_t launch_reduce_chunks(const float* partial, int64_t pstride_chunk, const int32_t* chunk_ptr, int K, float* out,
                                 int64_t ostride, int64_t off, int64_t len, cudaStream_t s) {
    if (len > 0 && K > 0) {
        launch_tail(reduce_chunks_kernel, dim3((unsigned)((len + 255) / 256), (unsigned)K), 256, 0, s, partial, pstride_chunk, chunk_ptr, out,
                                                                                               ostride, off, len); ++g_kernel_launches; }
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------------------------
// Variance-based importance (Section 3.4.1).  With p_i = deg_i / D (D = sum of local degrees; weight 1 and
// D = n' when the subgraph has no edges) the distance statistic splits by feature dimension:
//   sum_{i<j} p_i p_j |x_i - x_j|^2 = sum_f ( sum_i p_i (x_if - c_f)^2 - (sum_i p_i (x_if - c_f))^2 )
// for any shift c_f; c_f = the subgraph's first row keeps the two sums small.  This kernel accumulates the
// two weighted sums per chunk and per feature in double precision.
// ---------------------------------------------------------------------------------------------
// zeta_k = S_k / (D_k + beta) from the chunk sums of subgraph k, chunks added in order; one CTA per subgraph.
// `phase` spreads one zeta over several matrices (the layers' inputs, zeta_mode 2): 0 = this matrix alone; 1 = the first
// of several (its distance sum goes to q_acc[k]); 2 = a further one (added to q_acc[k]); 3 = the last one (added, then zeta).
__global__ void __launch_bounds__(1024) zeta_finish_kernel(const double* __restrict__ partial, int F, int ld, const int32_t* __restrict__ chunk_ptr,
                                              const int32_t* __restrict__ sub_off, const int64_t* __restrict__ deg_sum,
                                              const int64_t* __restrict__ deg_sq, float beta, double* __restrict__ zeta,
                                              double* __restrict__ q_acc, int phase) {
    __shared__ double seg_a[1024], seg_b[1024];
    const int k = blockIdx.x;
    const long long n = sub_off[k + 1] - sub_off[k];
    if (n == 0) return;   // zero since creation
    const bool uniform = deg_sum[k] == 0;
    const double D = uniform ? (double)n : (double)deg_sum[k];
    double q = 0.0;
    if (n > 0) {
        // segments of the chunk range in parallel, the segment sums then added in order, per feature
        const int c0 = chunk_ptr[k], c1 = chunk_ptr[k + 1];
        const int nseg = segments_for(F, 1024), per = 1024 / nseg;
        const int fl = threadIdx.x % per, seg = threadIdx.x / per;
        for (int f0 = 0; f0 < F; f0 += per) {
            const int f = f0 + fl;
            seg_a[threadIdx.x] = f < F ? segment_sum(partial, 2ll * ld, f, c0, c1, seg, nseg) : 0.0;
            seg_b[threadIdx.x] = f < F ? segment_sum(partial, 2ll * ld, (long long)ld + f, c0, c1, seg, nseg) : 0.0;
            __syncthreads();
            if (seg == 0 && f < F) {
                double a = seg_a[fl], b = seg_b[fl];
                for (int t = 1; t < nseg; ++t) { a += seg_a[t * per + fl]; b += seg_b[t * per + fl]; }
                const double m1 = a / D;
                q += b / D - m1 * m1;
            }
            __syncthreads();
        }
    }
    double* red = seg_a;
    red[threadIdx.x] = q;
    __syncthreads();
    for (int o = 512; o > 0; o >>= 1) {
        if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        double Q = red[0] > 0.0 ? red[0] : 0.0;
        if (phase == 2 || phase == 3) Q += q_acc[k];
        if (phase == 1 || phase == 2) {
            q_acc[k] = Q;
        } else {
            double z = 0.0;
            if (n > 0) {
                const double sq = uniform ? 1.0 / (double)n : (double)deg_sq[k] / (D * D);
                const double S = 0.5 * (1.0 - sq);
                if (S > 0.0) z = S / (sqrt(Q / S) + (double)beta);
            }
            zeta[k] = z;
        }
    }
}

// Grid: (row chunks, blocks of 128 columns); threads = 8 row lanes x 32 column lanes of one float4 each (as in the column sums above).
// The columns are spread over CTAs because the chunks of a small graph are few: with one CTA per chunk 2843 rows of 1433 features
// took 58 us on 24 CTAs.
__global__ void __launch_bounds__(256) zeta_partial_kernel(const float* __restrict__ X, int ld, const int32_t* __restrict__ deg,
                                                           const RowSpan* __restrict__ chunks, const int32_t* __restrict__ sub_off,
                                                           const int64_t* __restrict__ deg_sum, double* __restrict__ partial) {
    __shared__ double sm[8][32][8];
    const RowSpan c = chunks[blockIdx.x];
    const bool uniform = deg_sum[c.k] == 0;
    const int cx = threadIdx.x & 31, ry = threadIdx.x >> 5;
    const int ld4 = ld >> 2, v = (int)blockIdx.y * 32 + cx;
    double* P = partial + (long long)blockIdx.x * 2 * ld;
    double a[4] = {0.0, 0.0, 0.0, 0.0}, b[4] = {0.0, 0.0, 0.0, 0.0};
    if (v < ld4) {
        const float4 sh = reinterpret_cast<const float4*>(X + (long long)sub_off[c.k] * ld)[v];
        const float4* g = reinterpret_cast<const float4*>(X + (long long)c.row0 * ld) + v;
        const int32_t* dg = deg + c.row0;
        auto add = [&](const float4& u, int d) {
            const double w = uniform ? 1.0 : (double)d;
            const double x[4] = {(double)(u.x - sh.x), (double)(u.y - sh.y), (double)(u.z - sh.z), (double)(u.w - sh.w)};
#pragma unroll
            for (int t = 0; t < 4; ++t) { a[t] = fma(w, x[t], a[t]); b[t] = fma(w * x[t], x[t], b[t]); }
        };
        int r = ry;
        for (; r + 24 < c.nrows; r += 32) {   // four rows in flight
            float4 u[4];
            int d[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) { u[q] = g[(long long)(r + 8 * q) * ld4]; d[q] = dg[r + 8 * q]; }
#pragma unroll
            for (int q = 0; q < 4; ++q) add(u[q], d[q]);
        }
        for (; r < c.nrows; r += 8) add(g[(long long)r * ld4], dg[r]);
    }
#pragma unroll
    for (int t = 0; t < 4; ++t) { sm[ry][cx][t] = a[t]; sm[ry][cx][4 + t] = b[t]; }
    __syncthreads();
    if (ry == 0 && v < ld4) {
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            double sa = 0.0, sb = 0.0;
            for (int w = 0; w < 8; ++w) { sa += sm[w][cx][t]; sb += sm[w][cx][4 + t]; }
            P[4 * v + t] = sa;
            P[ld + 4 * v + t] = sb;
        }
    }
}

// zeta[k] for every subgraph that has rows (the entry of an empty subgraph is left as it is: zero since creation).
cudaError_t launch_zeta(const float* X, int ld, int F, const int32_t* deg, const RowSpan* chunks, int nchunks,
                        const int32_t* chunk_ptr, const int32_t* sub_off, int K, const int64_t* deg_sum, const int64_t* deg_sq,
                        float beta, double* partial, double* zeta, double* q_acc, int phase, cudaStream_t s) {
    if (nchunks > 0) {
        launch_beside(zeta_partial_kernel, dim3((unsigned)nchunks, (unsigned)((ld / 4 + 31) / 32)), 256, kZetaSharedKB, s, X, ld, deg, chunks, sub_off, deg_sum, partial);
        launch_beside(zeta_finish_kernel, dim3((unsigned)K), 1024, kZetaSharedKB, s, partial, F, ld, chunk_ptr, sub_off, deg_sum, deg_sq, beta, zeta, q_acc, phase);
        g_kernel_launches += 2;
    }
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------------------------
// Consensus weights w_k = zeta_k / sum_j zeta_j (Section 3.4.2); 1/K for the plain average of Definition 3
// or when every zeta is zero.  Computed by each CTA for itself (K is small).
// ---------------------------------------------------------------------------------------------
__device__ __forceinline__ void consensus_weights(const double* __restrict__ zeta, int K, int weighted, float* w_sm) {
    __shared__ double total;
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int k = 0; k < K; ++k) t += zeta[k];
        total = t;
    }
    __syncthreads();
    for (int k = threadIdx.x; k < K; k += blockDim.x)
        w_sm[k] = (weighted && total > 0.0) ? (float)(zeta[k] / total) : 1.f / (float)K;
    __syncthreads();
}

// sum_k w_k (theta_k - lr grad_k) for the four parameters at float4 index i, k ascending.  The copies are read eight at a time,
// all sixteen loads of a batch issued before the first is used: with many copies of a small model (K = 64 copies of a
// 256-256 layer are 50 MB spread over 65 CTAs) the kernel is a chain of dependent loads otherwise.
__device__ __forceinline__ float4 weighted_sum(const float* params, long long pstride_p, const float* __restrict__ grads, long long pstride,
                                               long long i, int K, float lr, int with_sgd, const float* w_sm) {
    constexpr int B = 8;
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int k0 = 0; k0 < K; k0 += B) {
        float4 p[B], g[B];
#pragma unroll
        for (int t = 0; t < B; ++t) {
            const int k = min(k0 + t, K - 1);   // past the end: the last copy again, with weight 0 below
            p[t] = reinterpret_cast<const float4*>(params + (long long)k * pstride_p)[i];
            g[t] = with_sgd ? reinterpret_cast<const float4*>(grads + (long long)k * pstride)[i] : make_float4(0.f, 0.f, 0.f, 0.f);
        }
#pragma unroll
        for (int t = 0; t < B; ++t) {
            if (k0 + t < K) {
                const float w = w_sm[k0 + t];
                float4 q = p[t];
                if (with_sgd) { q.x = fmaf(-lr, g[t].x, q.x); q.y = fmaf(-lr, g[t].y, q.y); q.z = fmaf(-lr, g[t].z, q.z); q.w = fmaf(-lr, g[t].w, q.w); }
                acc.x = fmaf(w, q.x, acc.x); acc.y = fmaf(w, q.y, acc.y); acc.z = fmaf(w, q.z, acc.z); acc.w = fmaf(w, q.w, acc.w);
            }
        }
    }
    return acc;
}

// What the first block of an update does besides; false: a bounded wait ran out earlier in this epoch, and the parameters stay as they are.
__device__ __forceinline__ bool end_of_epoch(long long pstride_p, int32_t* words, long long* epoch, const float* report, float* report_to, int nreport) {
    const bool timed_out = words[1] != 0;
    if (blockIdx.x == 0) {
        if (threadIdx.x == 0 && pstride_p != 0 && !timed_out) words[2] = 0;
        __syncthreads();
        if (report_to)   // the epoch's losses and error words, final by now, straight into the host's memory
            for (int i = threadIdx.x; i < nreport; i += blockDim.x) report_to[i] = report[i];
    }
    if (epoch && blockIdx.x == 0 && threadIdx.x == 0) *epoch += 1;   // last kernel of an epoch: nothing reads the counter beside it
    return !timed_out;
}

// theta_k <- theta_k - lr * grad_k (each replica's own step, update equation of Section 3.3), then
// theta_k <- sum_j w_j theta_j for every k (weighted global consensus, Section 3.4.2).  One float4 per thread.  All copies come out
// equal, so only copy 0 is written, and while they are equal it is the only one read (pstride_p == 0): K gradient sets and one
// parameter set in, one out, where K of each went both ways (50 copies of a 500-128-128-128-7 net: 13.5 -> 11 us).  words[2] says on
// the device whether the copies differ.
__global__ void __launch_bounds__(256) sgd_consensus_kernel(float* params, long long pstride_p, const float* __restrict__ grads,
                                                            long long pstride, long long len4, int K, float lr,
                                                            const double* __restrict__ zeta, int weighted, int with_sgd,
                                                            int32_t* words, long long* epoch, const float* report, float* report_to,
                                                            int nreport) {
    extern __shared__ float w_sm[];
    pdl_wait();
    after_wait(grads);
    after_wait(zeta);
    if (!end_of_epoch(pstride_p, words, epoch, report, report_to, nreport)) return;
    consensus_weights(zeta, K, weighted, w_sm);
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= len4) return;
    reinterpret_cast<float4*>(params)[i] = weighted_sum(params, pstride_p, grads, pstride, i, K, lr, with_sgd, w_sm);
}
cudaError_t launch_sgd_consensus(float* params, int64_t pstride_p, const float* grads, int64_t pstride, int64_t len, int K, float lr,
                                 const double* zeta, int weighted, int with_sgd, int32_t* words, long long* epoch, const float* report, float* report_to, int nreport, cudaStream_t s) {
    const long long len4 = len / 4;
    if (len4 > 0) {
        const int threads = len4 >= 148 * 256 * 4 ? 256 : 64;   // a small model is spread over more CTAs
        launch(sgd_consensus_kernel, dim3((unsigned)((len4 + threads - 1) / threads)), threads, (size_t)K * sizeof(float), s, 
            params, pstride_p, grads, pstride, len4, K, lr, zeta, weighted, with_sgd, words, epoch, report, report_to, nreport);
        ++g_kernel_launches;
    }
    return cudaGetLastError();
}

// The sum of one float4 over the chunks c0 .. c1 - 1 in order, eight loads at a time: as reduce_chunks_kernel adds them.
__device__ __forceinline__ float4 chunk_sum(const float4* __restrict__ partial, long long stride4, long long i, int c0, int c1) {
    float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int c = c0; c < c1; c += 8) {
        float4 v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) v[u] = c + u < c1 ? partial[(long long)(c + u) * stride4 + i] : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int u = 0; u < 8; ++u)
            if (c + u < c1) { s.x += v[u].x; s.y += v[u].y; s.z += v[u].z; s.w += v[u].w; }
    }
    return s;
}

// The same update where the gradients of the parameters `sums` are still chunk sums: they are added here and written to grads, which saves a short epoch the
// kernel between its last weight gradient and the update (19 717 rows of 500-256-3: 185.6 -> 178.3 us).  A block takes 32 float4: a warp for every replica, up
// to blockDim / 32 of them at a time (the chunks of one replica are a chain of loads), whose stepped values are then added in order by the first warp.
// The barriers and the small blocks cost more than that kernel where there are many parameters (16.8 M of 8 replicas: 0.39 ms, the kernel above 0.11).
__global__ void __launch_bounds__(512) step_sums_consensus_kernel(float* params, long long pstride_p, float* grads, long long pstride, long long len4, int K,
                                                                  float lr, const double* __restrict__ zeta, int weighted, int32_t* words, long long* epoch,
                                                                  const float* report, float* report_to, int nreport, ChunkSums sums) {
    extern __shared__ float4 q_sm[];   // [blockDim / 32][32], then K weights
    const int lane = threadIdx.x & 31, ky = threadIdx.x >> 5, ny = blockDim.x >> 5;
    float* w_sm = reinterpret_cast<float*>(q_sm + blockDim.x);
    pdl_wait();
    after_wait(grads);
    after_wait(zeta);
    after_wait(sums.partial);
    after_wait(sums.chunk_ptr);
    // (after a time-out too the chunks are added up: all the gradients are then those of one epoch, as where a kernel of its own adds them)
    const bool update = end_of_epoch(pstride_p, words, epoch, report, report_to, nreport);
    const long long i = (long long)blockIdx.x * 32 + lane;
    const bool here = i < len4, summed = here && i >= sums.first4 && i < sums.first4 + sums.count4;
    // float4 i of replica k after its step
    auto stepped = [&](int k) {
        if (!here || k >= K) return make_float4(0.f, 0.f, 0.f, 0.f);
        float4 q = reinterpret_cast<const float4*>(params + (long long)k * pstride_p)[i];
        float4* gk = reinterpret_cast<float4*>(grads + (long long)k * pstride) + i;
        float4 g;
        if (summed) *gk = g = chunk_sum(sums.partial, sums.stride4, i - sums.first4, sums.chunk_ptr[k], sums.chunk_ptr[k + 1]);
        else g = *gk;
        q.x = fmaf(-lr, g.x, q.x); q.y = fmaf(-lr, g.y, q.y); q.z = fmaf(-lr, g.z, q.z); q.w = fmaf(-lr, g.w, q.w);
        return q;
    };
    float4 next = stepped(ky);
    consensus_weights(zeta, K, weighted, w_sm);
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int k0 = 0; k0 < K; k0 += ny) {
        q_sm[ky * 32 + lane] = next;
        __syncthreads();
        if (k0 + ny < K) next = stepped(k0 + ny + ky);
        if (ky == 0)
            for (int t = 0; t < min(ny, K - k0); ++t) {
                const float w = w_sm[k0 + t];
                const float4 q = q_sm[t * 32 + lane];
                acc.x = fmaf(w, q.x, acc.x); acc.y = fmaf(w, q.y, acc.y); acc.z = fmaf(w, q.z, acc.z); acc.w = fmaf(w, q.w, acc.w);
            }
        __syncthreads();
    }
    if (update && ky == 0 && here) reinterpret_cast<float4*>(params)[i] = acc;   // (every read of copy 0 at i is this block's, and lies before a barrier)
}
cudaError_t launch_step_sums_consensus(float* params, int64_t pstride_p, float* grads, int64_t pstride, int64_t len, int K, float lr, const double* zeta,
                                       int weighted, int32_t* words, long long* epoch, const float* report, float* report_to, int nreport,
                                       const ChunkSums& sums, cudaStream_t s) {
    const long long len4 = len / 4;
    if (len4 > 0) {
        const int ny = K <= 4 ? 4 : K <= 8 ? 8 : 16;
        launch(step_sums_consensus_kernel, dim3((unsigned)((len4 + 31) / 32)), 32u * ny, (size_t)ny * 32 * sizeof(float4) + (size_t)K * sizeof(float), s,
               params, (long long)pstride_p, grads, (long long)pstride, len4, K, lr, zeta, weighted, words, epoch, report, report_to, nreport, sums);
        ++g_kernel_launches;
    }
    return cudaGetLastError();
}

__global__ void epoch_counter_kernel(long long* epoch, long long set_to, int advance) { *epoch = advance ? *epoch + 1 : set_to; }
cudaError_t launch_epoch_counter(long long* epoch, long long set_to, bool advance, cudaStream_t s) {
    epoch_counter_kernel<<<1, 1, 0, s>>>(epoch, set_to, advance ? 1 : 0); ++g_kernel_launches;
    return cudaGetLastError();
}

// The same sum over the replicas of one context when the subgraphs are spread over several contexts:
//   out = sum_k w_k (theta_k - lr * grad_k),  w_k = zeta_k / total (weighted) or 1 / total,
// with `total` the sum over ALL contexts, so that the contexts' results add up to the consensus.  The parameters
// themselves are left alone; consensus_apply_kernel writes the finished sum (to copy 0: the copies are equal from then on).
__global__ void __launch_bounds__(256) consensus_partial_kernel(const float* __restrict__ params, long long pstride_p, const float* __restrict__ grads,
                                                                long long pstride, long long len4, int K, float lr,
                                                                const double* __restrict__ zeta, int weighted, int with_sgd,
                                                                double total, float* __restrict__ out, const int32_t* __restrict__ err_word) {
    extern __shared__ float w_sm[];
    if (err_word && *err_word) return;
    for (int k = threadIdx.x; k < K; k += blockDim.x) w_sm[k] = (float)((weighted ? zeta[k] : 1.0) / total);
    __syncthreads();
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= len4) return;
    reinterpret_cast<float4*>(out)[i] = weighted_sum(params, pstride_p, grads, pstride, i, K, lr, with_sgd, w_sm);
}
__global__ void __launch_bounds__(256) consensus_apply_kernel(float* __restrict__ params, long long len4, const float* __restrict__ in, int32_t* words) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= len4 || words[1]) return;
    reinterpret_cast<float4*>(params)[i] = reinterpret_cast<const float4*>(in)[i];
    if (i == 0) words[2] = 0;
}
cudaError_t launch_consensus_partial(const float* params, int64_t pstride_p, const float* grads, int64_t pstride, int64_t len, int K, float lr,
                                     const double* zeta, int weighted, int with_sgd, double total, float* out, const int32_t* err_word, cudaStream_t s) {
    const long long len4 = len / 4;
    if (len4 > 0) {
        const int threads = len4 >= 148 * 256 * 4 ? 256 : 64;
        consensus_partial_kernel<<<(unsigned)((len4 + threads - 1) / threads), threads, (size_t)K * sizeof(float), s>>>(params, pstride_p, grads, pstride, len4, K, lr,
                                                                                                       zeta, weighted, with_sgd, total, out, err_word);
        ++g_kernel_launches;
    }
    return cudaGetLastError();
}
cudaError_t launch_consensus_apply(float* params, int64_t len, const float* in, int32_t* words, cudaStream_t s) {
    const long long len4 = len / 4;
    if (len4 > 0) { consensus_apply_kernel<<<(unsigned)((len4 + 255) / 256), 256, 0, s>>>(params, len4, in, words); ++g_kernel_launches; }
    return cudaGetLastError();
}

__global__ void weights_kernel(const double* __restrict__ zeta, int K, int weighted, float* __restrict__ zeta_f,
                               float* __restrict__ w_f) {
    extern __shared__ float w_sm[];
    consensus_weights(zeta, K, weighted, w_sm);
    for (int k = threadIdx.x; k < K; k += blockDim.x) {
        zeta_f[k] = (float)zeta[k];
        w_f[k] = w_sm[k];
    }
}
cudaError_t launch_weights(const double* zeta, int K, int weighted, float* zeta_f, float* w_f, cudaStream_t s) {
    weights_kernel<<<1, 256, (size_t)K * sizeof(float), s>>>(zeta, K, weighted, zeta_f, w_f); ++g_kernel_launches;
    return cudaGetLastError();
}

__global__ void __launch_bounds__(256) relu_mask_kernel(float4* __restrict__ G, const float4* __restrict__ H, long long n4, float scale) {
    pdl_next();
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n4) return;
    pdl_wait();
    after_wait(H);
    float4 g = G[i];
    const float4 h = H[i];
    g.x = h.x > 0.f ? g.x * scale : 0.f; g.y = h.y > 0.f ? g.y * scale : 0.f;
    g.z = h.z > 0.f ? g.z * scale : 0.f; g.w = h.w > 0.f ? g.w * scale : 0.f;
    G[i] = g;
}
cudaError_t launch_relu_mask(float* G, const float* H, int ld, int64_t rows, float scale, cudaStream_t s) {
    const long long n4 = (long long)rows * (ld / 4);
    if (n4 > 0) {
        launch(relu_mask_kernel, dim3((unsigned)((n4 + 255) / 256)), 256, 0, s, reinterpret_cast<float4*>(G), reinterpret_cast<const float4*>(H), n4, scale);
        ++g_kernel_launches;
    }
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------------------------
// Gathers between graph-node order and store-row order.
// ---------------------------------------------------------------------------------------------
// A row per group of up to 256 threads, so that no thread divides by the row length; V = float4 where the rows of Xg are whole 16-byte units,
// float where they start at any 4-byte boundary.  With the bfloat16 copy where the reduced-precision aggregation will gather it.  (A CTA
// per row took 63 us for 110 000 rows of 128; a thread per value of the result, with its division, 30 us more for 22 000 of 789.)
template <class V>
__global__ void __launch_bounds__(256) gather_rows_kernel(const float* __restrict__ Xg, int F, const int32_t* __restrict__ gid, long long rows, int ld,
                                                          int lane_bits, float* __restrict__ H0, uint16_t* __restrict__ bf) {
    constexpr int W = sizeof(V) / 4;
    const long long row = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> lane_bits;
    if (row >= rows) return;
    const float* src = Xg + (long long)gid[row] * F;
    float* dst = H0 + row * ld;
#pragma unroll 4
    for (int j = W * (int)(threadIdx.x & ((1u << lane_bits) - 1u)); j < ld; j += W << lane_bits) {
        V v{};
        if (W == 4 || j < F) v = __ldg(reinterpret_cast<const V*>(src + j));
        *reinterpret_cast<V*>(dst + j) = v;
        if constexpr (W == 4) { if (bf) *reinterpret_cast<uint2*>(bf + row * ld + j) = bf16_pack4(v); }
        else if (bf) bf[row * ld + j] = (uint16_t)bf16_bits(v);
    }
}
cudaError_t launch_gather_rows(const float* Xg, int F, const int32_t* gid, int64_t Np, float* H0, int ld, void* bf16_copy, cudaStream_t s) {
    if (Np > 0 && ld > 0) {
        const bool whole = F % 4 == 0;
        int bits = 0;
        while (bits < 8 && (1 << bits) < (whole ? ld / 4 : ld)) ++bits;
        const unsigned grid = (unsigned)((((long long)Np << bits) + 255) / 256);
        if (whole) gather_rows_kernel<float4><<<grid, 256, 0, s>>>(Xg, F, gid, Np, ld, bits, H0, reinterpret_cast<uint16_t*>(bf16_copy));
        else gather_rows_kernel<float><<<grid, 256, 0, s>>>(Xg, F, gid, Np, ld, bits, H0, reinterpret_cast<uint16_t*>(bf16_copy));
        ++g_kernel_launches;
    }
    return cudaGetLastError();
}
__global__ void gather_labels_kernel(const int32_t* __restrict__ yg, const int32_t* __restrict__ gid, long long Np,
                                     int32_t* __restrict__ label) {
    const long long r = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (r < Np) label[r] = yg[gid[r]];
}
cudaError_t launch_gather_labels(const int32_t* yg, const int32_t* gid, int64_t Np, int32_t* label, cudaStream_t s) {
    if (Np > 0) { gather_labels_kernel<<<(unsigned)((Np + 255) / 256), 256, 0, s>>>(yg, gid, Np, label); ++g_kernel_launches; }
    return cudaGetLastError();
}
// Logits of the core rows back to graph-node order; a quarter of a span of core rows per CTA, a row per group of up to 256 threads (V: as
// in gather_rows_kernel).  (A thread per value, with its division: 25 us for 100 000 rows of 40.)
template <class V>
__global__ void __launch_bounds__(256) scatter_core_kernel(const float* __restrict__ logits, int ld, int C, const int32_t* __restrict__ gid,
                                                           const RowSpan* __restrict__ spans, int lane_bits, float* __restrict__ out) {
    constexpr int W = sizeof(V) / 4;
    const RowSpan sp = spans[blockIdx.x];
    const int r1 = sp.nrows * (int)(blockIdx.y + 1) / 4, lane = threadIdx.x & ((1 << lane_bits) - 1);
#pragma unroll 2
    for (int r = sp.nrows * (int)blockIdx.y / 4 + (threadIdx.x >> lane_bits); r < r1; r += 256 >> lane_bits) {
        const float* src = logits + (long long)(sp.row0 + r) * ld;
        float* dst = out + (long long)gid[sp.row0 + r] * C;
        for (int j = W * lane; j < C; j += W << lane_bits) *reinterpret_cast<V*>(dst + j) = __ldg(reinterpret_cast<const V*>(src + j));
    }
}
cudaError_t launch_scatter_core(const float* logits, int ld, int C, const int32_t* gid, const RowSpan* core_spans, int nspans,
                                float* out, cudaStream_t s) {
    if (nspans > 0) {
        const bool whole = C % 4 == 0;
        int bits = 0;
        while (bits < 8 && (1 << bits) < (whole ? C / 4 : C)) ++bits;
        const dim3 grid((unsigned)nspans, 4);
        if (whole) scatter_core_kernel<float4><<<grid, 256, 0, s>>>(logits, ld, C, gid, core_spans, bits, out);
        else scatter_core_kernel<float><<<grid, 256, 0, s>>>(logits, ld, C, gid, core_spans, bits, out);
        ++g_kernel_launches;
    }
    return cudaGetLastError();
}

}  // namespace gad
