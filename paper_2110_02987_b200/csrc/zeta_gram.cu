// Variance-based importance in its literal pairwise form (Section 3.4.1, the printed equation read as it stands),
//   zeta_k = sum over unordered pairs i < j of subgraph k of  p_i p_j / (|x_i - x_j|_2 + beta),
// with the squared distances taken from a Gram matrix on the tensor cores:
//   |x_i - x_j|^2 = |x_i|^2 + |x_j|^2 - 2 x_i . x_j .
// The pairs of a subgraph are cut into tiles of 256 x 256 (i-block <= j-block).  A tile's inner products are one tcgen05 accumulator of a
// pair of CTAs: each CTA holds 128 rows of the i-block and half of the j-block (rows of the feature matrix, K-major, loaded by TMA with the
// 128-byte swizzle) and receives 128 x 256 products.  The features are split once per call into fp16 hi and lo copies of the row times a power of two (a
// streaming kernel that also takes the squared norms and keeps the scales), and the product is accumulated as hi.hi + hi.lo + lo.hi in fp32 in tensor
// memory.  hi and lo have 11 significant bits each, as TF32 parts have, and the scale keeps them clear of fp16's range: with the largest value of a row at 2^14
// the parts of a value are short of 22 bits only where it is below 2^-16 of that, by no more than 2^-39 of the largest.  fp16 operands are multiplied twice as fast: in three TF32
// passes the MMAs bounded the kernel (8 x 6563 rows of 128: 184 us, split 14).
// The accumulator is added to half as often, and with it goes a third to a half of what the tensor core cuts off.  Relative error of zeta against fp64, TF32 halves
// -> these, over 15 kinds of features (normal, uniform, with an offset, ReLU outputs, counts, sparse ones and zeros with and without weights, heavy tails, scales that
// differ by up to 2^40 between rows or inside one) at 24 to 1433 features: where the sum is long and of one sign it is what is cut off - 1433 uniform features 2.3e-5 -> 1.7e-5,
// 500 6.7e-6 -> 4.8e-6, 128 1.4e-6 -> 9e-7, 1433 ReLU outputs 2.0e-6 -> 1.3e-6 - and else 1e-7 and less, the same or smaller in all 90 combinations (one, heavy tails,
// 5.8e-8 -> 6.0e-8).
// What bounds it now is the drain: 17.7 instructions a pair, the schedulers issuing 65 % of the time, the tensor pipe active 43 % (157 us, split 14).  At the
// 96 registers that 18 warps leave a thread of it spills 28 bytes.
//
// While the MMA warp fills the second accumulator, sixteen warps read the first one back (tcgen05.ld), turn every inner product into a
// distance and add p_j / (d + beta) over the pairs i < j inside the subgraph.  Two pairs share a reciprocal, p / x + q / y = (p y + q x) /
// (x y): with a square root and half a reciprocal per pair the special-function unit (16 a cycle and SM) keeps up.  (Approximate square root and
// reciprocal, relative error 2^-23 each, and the errors of different pairs do not add up
// coherently.)
//
// Cancellation: for two rows that are close compared with their norms the Gram form loses digits, so a pair whose
// squared distance comes out below 5 % of |x_i|^2 + |x_j|^2 is computed from the differences x_if - x_jf
// themselves (plain loads, FP32 ALU).  On generic features that never happens; on features that are all alike it is
// every pair, which then costs what the FP32 tile kernel of zeta_pair.cu costs.
//
// Order of the sum: every cluster takes a contiguous range of tiles (ascending, subgraph by subgraph; the i-block stays in L2); every
// draining warp keeps one fp64 running sum per subgraph and writes it to its own slot; a second kernel adds the slots of the clusters
// whose ranges meet the subgraph in slot order.  For a given number of clusters the result does not depend on scheduling.
#include <cuda_fp16.h>

#include <algorithm>
#include <atomic>

#include "gad_internal.h"
#include "tc_common.cuh"

namespace gad {

namespace {

constexpr int GT = 256;                                   // rows of a tile side
constexpr int GH = 128;                                   // rows of a tile a CTA has of A (M of the pair's MMA is twice that)
constexpr int GBOX = 64;                                  // rows of a TMA box
constexpr int GBK = 64;                                   // features per ring stage
constexpr int G_TILE_BYTES = GH * GBK * 2;                // 16 KiB
constexpr int G_BOX_BYTES = GBOX * GBK * 2;
constexpr int G_STAGE_BYTES = 4 * G_TILE_BYTES;           // A_hi | A_lo | B_hi | B_lo
constexpr int G_STAGES = 3;
constexpr int G_RING_BYTES = G_STAGES * G_STAGE_BYTES;
constexpr int G_EPI_WARPS = 16;                           // four per quarter of the tensor-memory lanes, every fourth block of 32 columns each
constexpr int G_EPI_WARP0 = 2;
constexpr int G_THREADS = 32 * (G_EPI_WARP0 + G_EPI_WARPS);
constexpr int G_COL_BYTES = G_EPI_WARPS * 32 * 16;        // per draining warp: (p_j, |x_j|^2, -2 / scale of x_j) of its 32 columns
constexpr int G_SMEM_BYTES = G_RING_BYTES + 1024 + 256 + G_COL_BYTES;
constexpr int G_TMEM_COLS = 2 * GT;                       // two accumulators of 256 columns: all of it

struct GramArgs {
    const float* X;            // [rows x ld] features in store-row order
    int ld, F;
    const float2* norm2;       // [rows] squared norm, 1 / scale of the fp16 copies
    const int32_t* deg;
    const int32_t* sub_off;
    const int64_t* deg_sum;
    const int64_t* tile_ptr;   // [K+1] first tile of every subgraph
    int K;
    long long ntiles;          // tiles x parts
    int parts;                 // column parts of a tile, each taken on its own: 1, or 2 of 128 columns
    float beta;
    double* partial;           // [gridDim.x][G_EPI_WARPS][K], slots of subgraphs the cluster does not meet unwritten
    int32_t* err;
};

// Contiguous share of cluster c out of n.
__host__ __device__ __forceinline__ long long share(long long ntiles, int c, int n) { return ntiles * c / n; }

// A position in the list of (tile, part): subgraph by subgraph, the upper triangle of its T x T blocks row by row.
struct TilePos {
    int k, r0, n, T, bi, bj, part;
    __device__ __forceinline__ void open(const GramArgs& a, int k_) {
        k = k_;
        r0 = a.sub_off[k];
        n = a.sub_off[k + 1] - r0;
        T = (n + GT - 1) / GT;
    }
    __device__ __forceinline__ TilePos(const GramArgs& a, long long tp) {
        part = (int)(tp % a.parts);
        const long long t = tp / a.parts;
        int lo = 0, hi = a.K;                              // the largest k with tile_ptr[k] <= t
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (a.tile_ptr[mid] <= t) lo = mid; else hi = mid;
        }
        open(a, lo);
        long long q = t - a.tile_ptr[lo];
        bi = 0;
        while (bi + 1 < T && q >= T - bi) { q -= T - bi; ++bi; }
        bj = bi + (int)q;
    }
    __device__ __forceinline__ void next(const GramArgs& a) {
        if (++part < a.parts) return;
        part = 0;
        if (++bj < T) return;
        bj = ++bi;
        if (bi < T) return;
        bi = bj = 0;
        int nk = k + 1;
        while (nk < a.K - 1 && a.tile_ptr[nk + 1] == a.tile_ptr[nk]) ++nk;   // (subgraphs without rows have no tiles)
        if (nk < a.K) open(a, nk);
    }
    __device__ __forceinline__ int i0() const { return bi * GT; }
    __device__ __forceinline__ int j0(const GramArgs& a) const { return bj * GT + part * (GT / a.parts); }
};

// (FTZ: one instruction each; subnormal arguments and results count as zero)
template <bool FTZ>
__device__ __forceinline__ float sqrt_approx(float x) {
    float y;
    if (FTZ) asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    else asm("sqrt.approx.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
template <bool FTZ>
__device__ __forceinline__ float rcp_approx(float x) {
    float y;
    if (FTZ) asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    else asm("rcp.approx.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// Whether a pair has to be taken from the differences (true also where the Gram form has overflowed).
__device__ __forceinline__ bool near_pair(float d2, float s2) { return !(d2 >= 0.05f * s2); }
// Within these bounds of beta and of both squared norms (or with norms of zero) the product of two denominators (distances up to 2^62, plus beta) neither
// overflows nor underflows, and no squared distance of a pair that is not near is subnormal.
constexpr float kLeastBeta = 0x1p-60f, kMostBeta = 0x1p60f, kLeastNorm2 = 0x1p-120f, kMostNorm2 = 0x1p122f;
__device__ __forceinline__ bool plain_norm(float n2) { return n2 == 0.f || (n2 >= kLeastNorm2 && n2 <= kMostNorm2); }

// p_j / (d_ij + beta) summed over 16 columns j of one row i.  EACH: only the columns first .. last - 1, and without the pairs that have to be
// taken from the differences; those are reported in `close` either way.  PAIRED (norms and beta within the bounds above): two pairs share a reciprocal.
// (Two-wide FP32 instructions, 8.5 a pair counted by hand instead of 17.7 as executed, made the kernel spill: 181 us instead of 157.)
template <bool EACH, bool PAIRED>
__device__ __forceinline__ float gram_terms(const uint32_t (&v)[16], const float4* cols, float ni, float si, float beta, int first, int last, bool& close) {
    float part = 0.f, p0 = 0.f, x0 = 0.f;
#pragma unroll
    for (int jj = 0; jj < 16; ++jj) {
        float4 c = cols[jj];                                   // one broadcast load
        const float s2 = ni + c.y;
        float d2 = fmaf(__uint_as_float(v[jj]) * si, c.z, s2);
        bool near = near_pair(d2, s2);
        if (EACH) {
            const bool valid = jj >= first && jj < last;
            const bool counts = valid && !near;
            near = near && valid;
            c.x = counts ? c.x : 0.f;
            d2 = counts ? d2 : 1.f;
        }
        close |= near;
        const float x = sqrt_approx<PAIRED>(d2) + beta;
        if (!PAIRED) part = fmaf(c.x, rcp_approx<false>(x), part);
        else if (jj & 1) part = fmaf(fmaf(p0, x, c.x * x0), rcp_approx<true>(x0 * x), part);
        p0 = c.x; x0 = x;
    }
    return part;
}

__device__ __noinline__ float distance2(const float4* x, const float4* y, int n4) {
    float s = 0.f;
    for (int f = 0; f < n4; ++f) {       // pad columns are zero
        const float4 u = __ldg(x + f), w = __ldg(y + f);
        const float dx = u.x - w.x, dy = u.y - w.y, dz = u.z - w.z, dw = u.w - w.w;
        s = fmaf(dx, dx, s); s = fmaf(dy, dy, s); s = fmaf(dz, dz, s); s = fmaf(dw, dw, s);
    }
    return s;
}

// This warp's 32 tensor-memory lanes x 16 columns, complete on return: lane t receives its own lane's.
__device__ __forceinline__ void tmem_ld16(uint32_t addr, uint32_t (&r)[16]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];\n"
        "tcgen05.wait::ld.sync.aligned;\n"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]),
          "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(addr)
        : "memory");
}

__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(G_THREADS, 1)
zeta_gram_kernel(const __grid_constant__ CUtensorMap tmHi, const __grid_constant__ CUtensorMap tmLo, const GramArgs a) {
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw_addr = smem_u32(smem_raw);
    const uint32_t pad = ((raw_addr + 1023u) & ~1023u) - raw_addr;   // the same in both CTAs (the 128B swizzle repeats every 1024 bytes)
    uint8_t* sm = smem_raw + pad;
    const uint32_t sm_addr = raw_addr + pad;
    const uint32_t rank = cluster_rank();
    const uint32_t bars = sm_addr + G_RING_BYTES;
    auto full = [&](int s) { return bars + 8u * s; };
    auto empty = [&](int s) { return bars + 8u * (G_STAGES + s); };
    auto pfull = [&](int s) { return bars + 8u * (2 * G_STAGES + s); };      // leader: the other CTA's stage is full
    auto tfull = [&](int i) { return bars + 8u * (3 * G_STAGES + i); };
    auto tempty = [&](int i) { return bars + 8u * (3 * G_STAGES + 2 + i); };
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(sm + G_RING_BYTES + 8 * (3 * G_STAGES + 4));
    volatile uint32_t* abort_flag = tmem_slot + 1;
    float4* col_sm = reinterpret_cast<float4*>(sm + G_RING_BYTES + 256);   // [G_EPI_WARPS][32]

    const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int s = 0; s < G_STAGES; ++s) { mbar_init(full(s), 1); mbar_init(empty(s), 1); mbar_init(pfull(s), 1); }
        for (int i = 0; i < 2; ++i) { mbar_init(tfull(i), 1); mbar_init(tempty(i), 2 * G_EPI_WARPS); }
        *abort_flag = 0u;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) tmem_alloc2(smem_u32(tmem_slot), G_TMEM_COLS);
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    cluster_sync();           // the peer's barriers exist before anything arrives at them
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem_base = *tmem_slot;

    const int nkb = (a.F + GBK - 1) / GBK, width = GT / a.parts;
    const int ncl = gridDim.x >> 1, cl = blockIdx.x >> 1;
    const long long t_begin = share(a.ntiles, cl, ncl), t_end = share(a.ntiles, cl + 1, ncl);

    if (warp == 0 && lane == 0) {
        // ---------------- TMA producer: hi and lo of this CTA's rows of the two blocks of the tile, 64 features at a time ----------------
        int stage = 0;
        uint32_t phase = 0;
        bool ok = true;
        TilePos p(a, t_begin);
        for (long long t = t_begin; t < t_end && ok; ++t, p.next(a)) {
            const int ri = p.r0 + p.i0() + (int)rank * GH, rj = p.r0 + p.j0(a) + (int)rank * (width / 2);
            for (int kb = 0; kb < nkb; ++kb) {
                if (!(ok = mbar_wait(empty(stage), phase ^ 1u, abort_flag, a.err, 21))) break;
                mbar_expect_tx(full(stage), 2u * G_TILE_BYTES + 2u * (uint32_t)(width / 2) * (GBK * 2));
                const uint32_t base = sm_addr + stage * G_STAGE_BYTES;
                for (int b = 0; b < GH / GBOX; ++b) {
                    tma_load_2d(base + b * G_BOX_BYTES, &tmHi, kb * GBK, ri + b * GBOX, full(stage));
                    tma_load_2d(base + G_TILE_BYTES + b * G_BOX_BYTES, &tmLo, kb * GBK, ri + b * GBOX, full(stage));
                }
                for (int b = 0; b < width / 2 / GBOX; ++b) {
                    tma_load_2d(base + 2 * G_TILE_BYTES + b * G_BOX_BYTES, &tmHi, kb * GBK, rj + b * GBOX, full(stage));
                    tma_load_2d(base + 3 * G_TILE_BYTES + b * G_BOX_BYTES, &tmLo, kb * GBK, rj + b * GBOX, full(stage));
                }
                if (++stage == G_STAGES) { stage = 0; phase ^= 1u; }
            }
        }
    } else if (warp == 1 && rank == 1) {
        // ---------------- the other CTA's stages: the leader is told of each ----------------
        int stage = 0;
        uint32_t phase = 0;
        for (long long i = (t_end - t_begin) * nkb; i > 0 && lane == 0; --i) {
            if (!mbar_wait(full(stage), phase, abort_flag, a.err, 24)) break;
            mbar_arrive_leader(pfull(stage));
            if (++stage == G_STAGES) { stage = 0; phase ^= 1u; }
        }
    } else if (warp == 1) {
        // ---------------- MMA issuer (leader of the pair): the whole warp runs the loop, one elected lane issues ----------------
        int stage = 0, acc = 0;
        uint32_t phase = 0, acc_phase = 0;
        const uint32_t idesc = instr_desc_f16(width, 2 * GH);
        bool ok = true;
        for (long long t = t_begin; t < t_end && ok; ++t) {
            if (!(ok = __all_sync(0xffffffffu, mbar_wait<true>(tempty(acc), acc_phase ^ 1u, abort_flag, a.err, 22)))) break;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const uint32_t d = tmem_base + (uint32_t)(acc * GT);
            for (int kb = 0; kb < nkb; ++kb) {
                if (!(ok = __all_sync(0xffffffffu, mbar_wait(full(stage), phase, abort_flag, a.err, 23) &&
                                                       mbar_wait<true>(pfull(stage), phase, abort_flag, a.err, 25)))) break;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const uint32_t base = sm_addr + stage * G_STAGE_BYTES;
                const uint64_t a_hi = smem_desc(base), a_lo = smem_desc(base + G_TILE_BYTES);
                const uint64_t b_hi = smem_desc(base + 2 * G_TILE_BYTES), b_lo = smem_desc(base + 3 * G_TILE_BYTES);
                const int nks = min(GBK / 16, (a.F - kb * GBK + 15) / 16);
                if (elect_one()) {
                    // 16 fp16 values = 32 bytes = 2 descriptor units along K
#pragma unroll
                    for (int ks = 0; ks < GBK / 16; ++ks)
                        if (ks < nks) {
                            mma_f16_pair(d, a_hi + 2 * ks, b_hi + 2 * ks, idesc, (kb | ks) != 0 ? 1u : 0u);
                            mma_f16_pair(d, a_hi + 2 * ks, b_lo + 2 * ks, idesc, 1u);
                            mma_f16_pair(d, a_lo + 2 * ks, b_hi + 2 * ks, idesc, 1u);
                        }
                    mma_commit2(empty(stage));                    // in both CTAs
                    if (kb == nkb - 1) mma_commit2(tfull(acc));
                }
                __syncwarp();
                if (++stage == G_STAGES) { stage = 0; phase ^= 1u; }
            }
            if (++acc == 2) { acc = 0; acc_phase ^= 1u; }
        }
    } else if (warp >= G_EPI_WARP0) {
        // ---------------- drain: inner products -> distances -> weighted sum over the pairs i < j ----------------
        // this warp may read tensor-memory lanes 32q .. 32q+31 (this CTA's rows i of the tile); of the four warps of a quarter each takes
        // every fourth block of 32 columns (tile columns j)
        const int ew = warp - G_EPI_WARP0, q = warp & 3;
        float4* cols = col_sm + ew * 32;
        int acc = 0, cur_k = -1;
        uint32_t acc_phase = 0;
        bool ok = true, uniform = false;
        double sum = 0.0;
        float invD = 0.f;
        const bool beta_ok = a.beta >= kLeastBeta && a.beta <= kMostBeta;
        double* slot = a.partial + ((long long)blockIdx.x * G_EPI_WARPS + ew) * a.K;
        auto flush = [&]() {
            if (cur_k < 0) return;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
            if (lane == 0) slot[cur_k] = sum;
            sum = 0.0;
        };
        TilePos p(a, t_begin);
        for (long long t = t_begin; t < t_end; ++t, p.next(a)) {
            if (p.k != cur_k) {
                flush();
                cur_k = p.k;
                uniform = a.deg_sum[p.k] == 0;
                invD = (float)(1.0 / (uniform ? (double)p.n : (double)a.deg_sum[p.k]));
            }
            const int ib = p.i0() + (int)rank * GH + q * 32, i = ib + lane;   // this thread's row of the tile, inside the subgraph
            const bool iv = i < p.n;
            const float pi = iv ? (uniform ? 1.f : (float)a.deg[p.r0 + i]) * invD : 0.f;
            const float2 nsi = iv ? a.norm2[p.r0 + i] : make_float2(0.f, 1.f);
            const float ni = nsi.x, si = nsi.y;
            if (!(ok = __all_sync(0xffffffffu, mbar_wait(tfull(acc), acc_phase, abort_flag, a.err, 26)))) break;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            float part = 0.f;
            for (int c0 = 32 * (ew >> 2); c0 < width; c0 += 128) {
                const int jb = p.j0(a) + c0;
                if (jb + 31 <= ib || jb >= p.n || ib >= p.n) continue;        // no pair i < j of the subgraph in this block
                __syncwarp();                                                // the previous block's columns have been read
                const int jl = jb + lane;                                    // the column this lane looks up for the warp
                const bool jlv = jl < p.n;
                const float2 nsj = jlv ? a.norm2[p.r0 + jl] : make_float2(0.f, 1.f);
                const float4 mine = make_float4(jlv ? (uniform ? 1.f : (float)a.deg[p.r0 + jl]) * invD : 0.f, nsj.x, -2.f * nsj.y, 0.f);
                cols[lane] = mine;
                __syncwarp();
                const bool plain = beta_ok && __all_sync(0xffffffffu, plain_norm(ni) && plain_norm(mine.y));
                const float4* xi = reinterpret_cast<const float4*>(a.X + (long long)(p.r0 + min(i, p.n - 1)) * a.ld);
                for (int h = 0; h < 32; h += 16) {                           // (32 at a time do not fit the registers)
                    uint32_t v[16];
                    tmem_ld16(tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)(acc * GT + c0 + h), v);
                    // every pair of the block counts, or the columns [first, last) of this row do
                    const bool whole = ib + 31 < jb + h && ib + 31 < p.n && jb + h + 15 < p.n;
                    const int first = i + 1 - jb - h, last = iv ? min(16, p.n - jb - h) : 0;
                    bool close = false;
                    float blk = 0.f;
                    if (whole && plain) blk = gram_terms<false, true>(v, cols + h, ni, si, a.beta, 0, 16, close);
                    if (!whole || !plain || __any_sync(0xffffffffu, close)) {
                        close = false;
                        blk = plain ? gram_terms<true, true>(v, cols + h, ni, si, a.beta, first, last, close) : gram_terms<true, false>(v, cols + h, ni, si, a.beta, first, last, close);
                        if (close) {   // rows close to each other compared with their norms: those pairs from the differences themselves
#pragma unroll
                            for (int jj = 0; jj < 16; ++jj) {                // (unrolled: the accumulator block stays in registers)
                                const float4 c = cols[h + jj];
                                const float s2 = ni + c.y;
                                const float d2 = fmaf(__uint_as_float(v[jj]) * si, c.z, s2);
                                if (jj >= first && jj < last && near_pair(d2, s2))
                                    blk += c.x / (sqrtf(distance2(xi, reinterpret_cast<const float4*>(a.X + (long long)(p.r0 + jb + h + jj) * a.ld), a.ld >> 2)) + a.beta);
                            }
                        }
                    }
                    part += blk;
                }
            }
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            __syncwarp();
            if (lane == 0) mbar_arrive_leader_tmem(tempty(acc));
            if (++acc == 2) { acc = 0; acc_phase ^= 1u; }
            sum += (double)(pi * part);
        }
        if (ok) flush();
    }

    // Tear-down.  After a time-out, give loads that may still be in flight a bounded chance to land before the shared memory is
    // released.  Neither CTA leaves while the other may still read its operands or arrive at its barriers.
    __syncthreads();
    if (*abort_flag && threadIdx.x == 0)
        for (int s = 0; s < G_STAGES; ++s)
            for (uint32_t i = 0; i < 4096u; ++i)
                if (mbar_try_wait(full(s), 0) || mbar_try_wait(full(s), 1)) break;
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    cluster_sync();
    if (warp == 0) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        tmem_dealloc2(tmem_base, G_TMEM_COLS);
    }
}

// One pass over the features: every row times the power of two that brings its largest value to 2^14 .. 2^15 (a row of zeros, or with infinities, stays as
// it is), hi = that rounded to fp16, lo = the rest rounded to fp16; |x_r|^2 in fp32 and 1 / scale.  One warp per row, eight values per lane
// (ldh: a multiple of 8; values past the last feature are zero).
__global__ void __launch_bounds__(256) split_rows_kernel(const float* __restrict__ X, int ld, int ldh, long long rows, __half* __restrict__ Xhi,
                                                         __half* __restrict__ Xlo, float2* __restrict__ norm2) {
    const long long r = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (r >= rows) return;
    const float4* x = reinterpret_cast<const float4*>(X + r * ld);
    const int n4 = ld >> 2;
    constexpr float4 zero = {0.f, 0.f, 0.f, 0.f};
    float s = 0.f, most = 0.f;
    for (int f4 = lane; f4 < n4; f4 += 32) {
        const float4 v = __ldg(x + f4);
        s = fmaf(v.x, v.x, s); s = fmaf(v.y, v.y, s); s = fmaf(v.z, v.z, s); s = fmaf(v.w, v.w, s);
        most = fmaxf(fmaxf(fmaxf(most, fabsf(v.x)), fabsf(v.y)), fmaxf(fabsf(v.z), fabsf(v.w)));
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        s += __shfl_xor_sync(0xffffffffu, s, o);
        most = fmaxf(most, __shfl_xor_sync(0xffffffffu, most, o));
    }
    // 2^e <= most < 2^(e + 1) for the biased exponent e + 127 (subnormal rows: as if 2^-126); scale 2^(14 - e), held to what fp32 has
    const int e = max((int)(__float_as_uint(most) >> 23), 1) - 127;
    const bool scaled = most > 0.f && e < 128;
    const int up = scaled ? min(14 - e, 126) : 0;   // (e >= -126, so up <= 140: held to 126; up >= -113)
    const float scale = __uint_as_float((uint32_t)(up + 127) << 23), back = __uint_as_float((uint32_t)(127 - up) << 23);
    for (int f8 = lane; f8 < (ldh >> 3); f8 += 32) {
        const float4 a = __ldg(x + 2 * f8), b = 2 * f8 + 1 < n4 ? __ldg(x + 2 * f8 + 1) : zero;
        const float v[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
        __half2 h[4], l[4];
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            const float u0 = v[2 * t] * scale, u1 = v[2 * t + 1] * scale;
            h[t] = __floats2half2_rn(u0, u1);
            const float2 back2 = __half22float2(h[t]);
            l[t] = __floats2half2_rn(u0 - back2.x, u1 - back2.y);
        }
        *reinterpret_cast<uint4*>(Xhi + r * ldh + 8 * f8) = *reinterpret_cast<const uint4*>(h);
        *reinterpret_cast<uint4*>(Xlo + r * ldh + 8 * f8) = *reinterpret_cast<const uint4*>(l);
    }
    if (lane == 0) norm2[r] = make_float2(s, back);
}

// zeta_k = the slots of the clusters that meet subgraph k added in slot order (one CTA per subgraph; a warp adds every eighth slot).
__global__ void __launch_bounds__(256) zeta_gram_finish_kernel(const double* __restrict__ partial, const int64_t* __restrict__ tile_ptr, long long ntiles,
                                                               int parts, int ncl, int K, double* __restrict__ zeta) {
    __shared__ double warp_sum[8];
    const int k = blockIdx.x, lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const long long t0 = tile_ptr[k] * parts, t1 = tile_ptr[k + 1] * parts;
    double s = 0.0;
    for (int c = w; c < ncl; c += 8)
        if (share(ntiles, c, ncl) < t1 && share(ntiles, c + 1, ncl) > t0) s += partial[((long long)c * 2 * G_EPI_WARPS + lane) * K + k];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) warp_sum[w] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int i = 1; i < 8; ++i) s += warp_sum[i];
        zeta[k] = s;
    }
}
static_assert(2 * G_EPI_WARPS == 32, "a warp reads the slots of a cluster");

int gram_clusters(int num_sms) {
    static std::atomic<int> known{0};
    if (known.load() <= 0) known.store(max_active_pairs(reinterpret_cast<const void*>(zeta_gram_kernel), G_THREADS, G_SMEM_BYTES, num_sms));
    return known.load();
}

}  // namespace

// Tiles of a subgraph of `rows` rows: T (T + 1) / 2 with T = ceil(rows / 256).
int64_t zeta_gram_tiles(int64_t rows) {
    const int64_t T = (rows + GT - 1) / GT;
    return T * (T + 1) / 2;
}
int64_t zeta_gram_partials(int num_sms, int K) { return (int64_t)num_sms * G_EPI_WARPS * K; }
uint32_t zeta_gram_box_rows() { return GBOX; }

cudaError_t launch_zeta_gram(const void* mapHi, const void* mapLo, const float* X, int ld, int F, long long rows, const int32_t* deg,
                             const int32_t* sub_off, const int64_t* deg_sum, const int64_t* tile_ptr, int64_t ntiles, int K, float beta,
                             void* Xhi, void* Xlo, float2* norm2, double* partial, double* zeta, int32_t* err, int num_sms, cudaStream_t s) {
    if (rows <= 0 || K <= 0) return cudaSuccess;
    cudaError_t e = configure_kernel_once(reinterpret_cast<const void*>(zeta_gram_kernel), G_SMEM_BYTES, false);
    if (e != cudaSuccess) return e;
    split_rows_kernel<<<(unsigned)((rows * 32 + 255) / 256), 256, 0, s>>>(X, ld, (int)round_up(F, 8), rows, reinterpret_cast<__half*>(Xhi), reinterpret_cast<__half*>(Xlo), norm2);
    ++g_kernel_launches;
    GramArgs a;
    a.X = X; a.ld = ld; a.F = F; a.norm2 = norm2; a.deg = deg; a.sub_off = sub_off; a.deg_sum = deg_sum; a.tile_ptr = tile_ptr;
    a.K = K; a.beta = beta; a.partial = partial; a.err = err;
    // Tiles of 256 columns keep the tensor pipe busy.  Tiles of 128 read A twice as often and wait for shared memory, a quarter longer
    // per column, but where there are few tiles they share them out better.
    const int64_t most = std::max(1, std::min(gram_clusters(num_sms), num_sms / 2));
    const auto turns = [&](int64_t n) { return (n + most - 1) / most; };
    a.parts = 5 * turns(2 * ntiles) < 8 * turns(ntiles) ? 2 : 1;
    a.ntiles = ntiles * a.parts;
    const int ncl = (int)std::min<int64_t>(a.ntiles, most);
    if (ncl > 0) {
        zeta_gram_kernel<<<2 * ncl, G_THREADS, G_SMEM_BYTES, s>>>(*reinterpret_cast<const CUtensorMap*>(mapHi),
                                                                  *reinterpret_cast<const CUtensorMap*>(mapLo), a);
        ++g_kernel_launches;
    }
    zeta_gram_finish_kernel<<<(unsigned)K, 256, 0, s>>>(partial, tile_ptr, a.ntiles, a.parts, std::max(ncl, 1), K, zeta);
    ++g_kernel_launches;
    return cudaGetLastError();
}

}  // namespace gad
