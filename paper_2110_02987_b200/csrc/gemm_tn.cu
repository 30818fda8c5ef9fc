// Weight gradients dW_k = H_k^T dZ_k on the 5th-generation tensor cores (chain rule through the forward equation, Section 3.3):
// partial[chunk][m][n] = sum over the chunk's rows r of H[r][m] dZ[r][n].  The reduction index is the row.  dZ stays in shared memory
// "MN-major": a tile of 32 rows x 32 values (128 bytes per row, swizzled in 32-byte units) is one block of the canonical
// layout, blocks of 32 values are 4096 bytes apart (leading byte offset), groups of 4 rows 512 bytes apart (stride byte offset),
// and one MMA (K = 8) consumes 8 rows.  H^T goes through tensor memory: a splitting lane reads one of its columns (32 rows, a bank each) and writes
// both parts of it into its tensor-memory lane, which turns the tile on the way.  (In one pass H is read from shared memory as dZ is.)  fp32
// accuracy as in gemm_rows.cu; both operands are activations here: dZ gets a lo tile in shared memory.  Rows past the end of a chunk become zero.
//
// What bounds it is the tensor pipe, and below 256 columns the split (about 1500 cycles a 32-row step of 128 columns and group of warps, two groups taking
// turns, against 768 of MMAs).  With both operands split in shared memory it was shared-memory bandwidth: 192 KB a step of 128 x 128 (1536 cycles at 128 B), 288 KB of
// 128 x 256; now 128 and 224 KB.  CTAs work in pairs (cta_group::2: each has 128 of the H columns and half of the dZ columns) where there are more than 128
// input columns.  The ring of loaded tiles is separate from the split ones, so that three to five stages hold loads in flight; CTAs are persistent and
// have two accumulators where the tensor memory has room for them beside the slots (up to 128 columns), so that a work unit (a chunk of rows and an
// output tile) drains while the next one is multiplied.
// One timeline of an epoch each, both operands split in shared memory and now: 525 000 rows, 256 x 256 259 -> 239 us, 256 x 47 123 -> 117, 100 x 256 216 -> 167;
// 94 000 rows in 50 subgraphs, 128 x 128 35.7 -> 27.9, 500 x 128 94.5 -> 75; 110 000 rows, 128 x 128 34.5 -> 29.2.
// (Single CTAs: a thread spills 4 bytes at the 96 registers that 18 warps leave it.)
#include <cuda.h>

#include <algorithm>

#include "gad_internal.h"
#include "tc_common.cuh"

namespace gad {

namespace {

constexpr int TBK = 32;                                   // rows of the reduction per ring stage
constexpr int BLOCK_BYTES = TBK * 128;                    // one block: TBK rows x 32 values
constexpr int A_BLOCKS = 4;                               // 128 output rows of a CTA
constexpr int MAX_STAGES = 8, MAX_LO = 4;
constexpr int BAR_BYTES = 512;
constexpr int SMEM_BYTES = 232448;
constexpr int DATA_BYTES = SMEM_BYTES - 1024 - BAR_BYTES;
constexpr int SPLIT_WARPS = 8, EPI_WARPS = 8, EPI_WARP0 = 2 + SPLIT_WARPS;
constexpr int THREADS = 32 * (EPI_WARP0 + EPI_WARPS);
constexpr int SLOT_COLS = 2 * TBK;                        // tensor memory of a split step of H: 32 columns of hi, 32 of lo
constexpr uint32_t TMEM_COLS = 512;

struct TnArgs {
    const RowSpan* chunks;
    int nunits, ntm, ntn, BN, M, ldw;   // work units; output tiles per chunk; MMA N; valid output rows; leading dimension of the output
    int nst, nlo;                       // ring stages; steps whose split operands are kept (2 or 4, at most nst)
    int nacc;                           // accumulators: two where the tensor memory has room for them
    float* partial;
    long long pstride_chunk;
    int32_t* err;
};

// MN-major TF32 tile: layout type 1 (128-byte swizzle of 32-byte units, repeating every 4 rows = 512 bytes).
__device__ __forceinline__ uint64_t smem_desc_mn(uint32_t saddr) {
    return (uint64_t)((saddr & 0x3FFFFu) >> 4) | ((uint64_t)(BLOCK_BYTES >> 4) << 16) | ((uint64_t)(512 >> 4) << 32) | ((uint64_t)1 << 46) |
           ((uint64_t)1 << 61);
}

template <int CG>
__device__ __forceinline__ void mma_any(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
    if constexpr (CG == 2) mma_tf32_pair(d, a, b, idesc, acc);
    else mma_tf32(d, a, b, idesc, acc);
}
template <int CG>
__device__ __forceinline__ void mma_any_ts(uint32_t d, uint32_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
    if constexpr (CG == 2) mma_tf32_pair_ts(d, a, b, idesc, acc);
    else mma_tf32_ts(d, a, b, idesc, acc);
}
template <int CG>
__device__ __forceinline__ void commit_any(uint32_t bar) {
    if constexpr (CG == 2) mma_commit2(bar);
    else mma_commit(bar);
}
template <int CG>
__device__ __forceinline__ void arrive_any(uint32_t bar) {
    if constexpr (CG == 2) mbar_arrive_leader(bar);
    else mbar_arrive(bar);
}
template <int CG>
__device__ __forceinline__ void arrive_drained(uint32_t bar) {
    if constexpr (CG == 2) mbar_arrive_leader_tmem(bar);
    else mbar_arrive(bar);
}

// CG: CTAs that work together on a unit (1, or 2 = a cluster).
template <int CG, bool split>
__global__ void __launch_bounds__(THREADS, 1)
gemm_tn_kernel(const __grid_constant__ CUtensorMap tmH, const __grid_constant__ CUtensorMap tmZ, const TnArgs a) {
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw_addr = smem_u32(smem_raw);
    const uint32_t pad = ((raw_addr + 1023u) & ~1023u) - raw_addr;
    uint8_t* sm = smem_raw + pad;
    const uint32_t sm_addr = raw_addr + pad;
    const int rank = CG == 2 ? (int)cluster_rank() : 0;
    const int bcols = a.BN / CG;                               // this CTA's columns of dZ
    const int nbb = (bcols + 31) / 32, nblocks = A_BLOCKS + nbb;
    const uint32_t stage_bytes = (uint32_t)nblocks * BLOCK_BYTES;
    const uint32_t lo_bytes = (uint32_t)nbb * BLOCK_BYTES;     // lo part of a step of dZ
    const uint32_t off_ring = split ? (uint32_t)a.nlo * lo_bytes : 0u;
    const int nst = a.nst;
    const uint32_t bars = sm_addr + DATA_BYTES;
    auto full = [&](int s) { return bars + 8u * s; };
    auto empty = [&](int s) { return bars + 8u * (MAX_STAGES + s); };
    auto xfull = [&](int q) { return bars + 8u * (2 * MAX_STAGES + q); };
    auto loempty = [&](int q) { return bars + 8u * (2 * MAX_STAGES + MAX_LO + q); };
    auto tfull = [&](int i) { return bars + 8u * (2 * MAX_STAGES + 2 * MAX_LO + i); };
    auto tempty = [&](int i) { return bars + 8u * (2 * MAX_STAGES + 2 * MAX_LO + 2 + i); };
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(sm + DATA_BYTES + 8 * (2 * MAX_STAGES + 2 * MAX_LO + 4));
    volatile uint32_t* abort_flag = tmem_slot + 1;
    uint32_t acc_cols = 16;                                    // columns between the accumulators: BN rounded up to a power of two
    while (acc_cols < (uint32_t)a.BN) acc_cols <<= 1;
    const uint32_t tmem_cols = split ? TMEM_COLS : 2 * acc_cols, slot0 = TMEM_COLS - (uint32_t)a.nlo * SLOT_COLS;

    pdl_next();
    const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
    constexpr int groups = split ? SPLIT_WARPS / 4 : 1;        // of splitting warps, taking steps in turn; each has a warp for every quarter of the lanes
    if (threadIdx.x == 0) {
        for (int s = 0; s < MAX_STAGES; ++s) { mbar_init(full(s), 1); mbar_init(empty(s), 1); }
        for (int q = 0; q < MAX_LO; ++q) { mbar_init(xfull(q), CG * SPLIT_WARPS / groups); mbar_init(loempty(q), 1); }
        for (int i = 0; i < 2; ++i) { mbar_init(tfull(i), 1); mbar_init(tempty(i), CG * EPI_WARPS); }
        *abort_flag = 0u;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        if constexpr (CG == 2) tmem_alloc2(smem_u32(tmem_slot), tmem_cols);
        else {
            asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(tmem_cols) : "memory");
            asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if constexpr (CG == 2) cluster_sync();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem_base = *tmem_slot;

    pdl_wait();   // from here on operands are read and results written
    const int tiles = a.ntm * a.ntn, ncl = gridDim.x / CG, cl = blockIdx.x / CG;
    const int u0 = (int)((long long)a.nunits * cl / ncl), u1 = (int)((long long)a.nunits * (cl + 1) / ncl);
    // calls f(chunk number, chunk, first output row of this CTA, first output column of the tile) until it returns false
    auto for_units = [&](auto&& f) {
        for (int u = u0; u < u1; ++u) {
            const int c = u / tiles, tile = u % tiles;
            if (!f(c, a.chunks[c], (tile / a.ntn) * (CG * BM) + rank * BM, (tile % a.ntn) * a.BN)) return;
        }
    };

    if (warp == 0 && lane == 0) {
        // ---------------- TMA producer ----------------
        int stage = 0;
        uint32_t phase = 0;
        for_units([&](int, const RowSpan c, int m0, int n0) {
            const int nkb = (c.nrows + TBK - 1) / TBK, b0 = n0 + rank * bcols;
            for (int kb = 0; kb < nkb; ++kb) {
                if (!mbar_wait(empty(stage), phase ^ 1u, abort_flag, a.err, 11)) return false;
                mbar_expect_tx(full(stage), stage_bytes);
                const uint32_t base = sm_addr + off_ring + (uint32_t)stage * stage_bytes;
                const int r = c.row0 + kb * TBK;
                for (int j = 0; j < A_BLOCKS; ++j) tma_load_2d(base + j * BLOCK_BYTES, &tmH, m0 + 32 * j, r, full(stage));
                for (int j = 0; j < nbb; ++j) tma_load_2d(base + (A_BLOCKS + j) * BLOCK_BYTES, &tmZ, b0 + 32 * j, r, full(stage));
                if (++stage == nst) { stage = 0; phase ^= 1u; }
            }
            return true;
        });
    } else if (warp == 1 && rank == 0) {
        // ---------------- MMA issuer: the warp runs the loop, one elected lane issues ----------------
        int stage = 0, q = 0, acc = 0;
        uint32_t qphase = 0, acc_phase = 0;
        const uint32_t idesc = instr_desc(a.BN, CG * BM) | (split ? 0u : 1u << 15) | (1u << 16);   // A (in shared memory) and B MN-major
        for_units([&](int, const RowSpan c, int, int) {
            const int nkb = (c.nrows + TBK - 1) / TBK;
            if (!__all_sync(0xffffffffu, mbar_wait<CG == 2>(tempty(acc), acc_phase ^ 1u, abort_flag, a.err, 12))) return false;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const uint32_t d = tmem_base + (uint32_t)acc * acc_cols;
            for (int kb = 0; kb < nkb; ++kb) {
                if (!__all_sync(0xffffffffu, mbar_wait<CG == 2>(xfull(q), qphase, abort_flag, a.err, 13))) return false;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const uint32_t base = sm_addr + off_ring + (uint32_t)stage * stage_bytes, a_tm = tmem_base + slot0 + (uint32_t)q * SLOT_COLS;
                const uint64_t a_hi = smem_desc_mn(base), b_hi = smem_desc_mn(base + A_BLOCKS * BLOCK_BYTES), b_lo = smem_desc_mn(sm_addr + (uint32_t)q * lo_bytes);
                const int nks = min(TBK / 8, (c.nrows - kb * TBK + 7) / 8);
                if (elect_one()) {
                    // the next group of 8 rows is 1024 bytes = 64 descriptor units further on
#pragma unroll
                    for (int ks = 0; ks < TBK / 8; ++ks) {
                        if (ks < nks) {
                            if constexpr (split) {
                                mma_any_ts<CG>(d, a_tm + 8 * ks, b_hi + 64 * ks, idesc, (kb | ks) != 0 ? 1u : 0u);
                                mma_any_ts<CG>(d, a_tm + 8 * ks, b_lo + 64 * ks, idesc, 1u);
                                mma_any_ts<CG>(d, a_tm + TBK + 8 * ks, b_hi + 64 * ks, idesc, 1u);
                            } else {
                                mma_any<CG>(d, a_hi + 64 * ks, b_hi + 64 * ks, idesc, (kb | ks) != 0 ? 1u : 0u);
                            }
                        }
                    }
                    commit_any<CG>(empty(stage));
                    commit_any<CG>(loempty(q));
                    if (kb == nkb - 1) commit_any<CG>(tfull(acc));
                }
                __syncwarp();
                if (++stage == nst) stage = 0;
                if (++q == a.nlo) { q = 0; qphase ^= 1u; }
            }
            if (++acc == a.nacc) { acc = 0; acc_phase ^= 1u; }
            return true;
        });
    } else if (warp >= 2 && warp < EPI_WARP0) {
        // ---------------- split of both operands, rows past the end of the chunk zeroed (groups: see gemm_rows.cu) ----------------
        constexpr int gw = SPLIT_WARPS / groups;
        const int group = (warp - 2) / gw, tt = threadIdx.x - 64 - 32 * gw * group;
        const int nf4 = nblocks * (BLOCK_BYTES / 16), nb4 = nbb * (BLOCK_BYTES / 16);   // 16-byte pieces of a step, and of its dZ
        const int piece = lane >> 3;                  // a lane is a column of H: its 32-byte piece of a row, swizzled by the row
        int stage = 0, q = 0;
        uint32_t phase = 0, qphase = 0;
        for_units([&](int, const RowSpan c, int, int) {
            const int nkb = (c.nrows + TBK - 1) / TBK;
            for (int kb = 0; kb < nkb; ++kb) {
                if (groups == 1 || (q & (groups - 1)) == group) {
                    // (the votes keep the warp together: lanes may see a time-out or an abort at different polls)
                    if (!__all_sync(0xffffffffu, mbar_wait(loempty(q), qphase ^ 1u, abort_flag, a.err, 14))) return false;
                    if (!__all_sync(0xffffffffu, mbar_wait(full(stage), phase, abort_flag, a.err, 15))) return false;
                    uint8_t* base = sm + off_ring + (uint32_t)stage * stage_bytes;
                    const int valid = c.nrows - kb * TBK;
                    float4* raw = reinterpret_cast<float4*>(base + (split ? A_BLOCKS * BLOCK_BYTES : 0));   // what the MMAs read as loaded
                    if (valid < TBK)   // 8 float4 per 128-byte row, TBK rows per block
                        for (int i = tt; i < (split ? nb4 : nf4); i += 32 * gw)
                            if (((i >> 3) & (TBK - 1)) >= valid) raw[i] = make_float4(0.f, 0.f, 0.f, 0.f);
                    if constexpr (split) {
                        // H: this warp's 32 columns, one a lane, 32 rows, on their way while dZ is split
                        const uint8_t* src = base + (warp & 3) * BLOCK_BYTES + 4 * (lane & 7);
                        float ahi[TBK], alo[TBK];
#pragma unroll
                        for (int k = 0; k < TBK; ++k) ahi[k] = *reinterpret_cast<const float*>(src + k * 128 + ((piece ^ (k & 3)) << 5));
                        // dZ: loads ahead of the stores, which the compiler cannot tell apart from what is loaded (a piece at a time took 115 cycles)
                        float4* lo = reinterpret_cast<float4*>(sm + (uint32_t)q * lo_bytes);
                        constexpr int STEP = 32 * gw;
                        for (int i = tt; i < nb4; i += 4 * STEP) {   // (nb4: a multiple of 2 STEP)
                            float4 v[4];
                            const bool four = i + 2 * STEP < nb4;
#pragma unroll
                            for (int u = 0; u < 4; ++u)
                                if (u < 2 || four) v[u] = raw[i + u * STEP];   // stays where it is: the MMA reads it as the hi part
#pragma unroll
                            for (int u = 0; u < 4; ++u)
                                if (u < 2 || four) lo[i + u * STEP] = make_float4(tf32_rest(v[u].x), tf32_rest(v[u].y), tf32_rest(v[u].z), tf32_rest(v[u].w));
                        }
                        if (valid < TBK)
#pragma unroll
                            for (int k = 0; k < TBK; ++k) ahi[k] = k < valid ? ahi[k] : 0.f;
#pragma unroll
                        for (int k = 0; k < TBK; ++k) alo[k] = tf32_rest(ahi[k]);
                        const uint32_t dst = tmem_base + ((uint32_t)(32 * (warp & 3)) << 16) + slot0 + (uint32_t)q * SLOT_COLS;
                        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");   // the MMAs that read the slot have completed
                        tmem_st_32x32b_x32(dst, ahi);
                        tmem_st_32x32b_x32(dst + TBK, alo);
                        tmem_wait_st();
                        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                    }
                    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                    __syncwarp();
                    if (lane == 0) arrive_any<CG>(xfull(q));
                }
                if (++q == a.nlo) { q = 0; qphase ^= 1u; }
                if (++stage == nst) { stage = 0; phase ^= 1u; }
            }
            return true;
        });
    } else if (warp >= EPI_WARP0) {
        // ---------------- drain (see gemm_rows.cu for the shape of the reads) ----------------
        const int quarter = warp & 3, half = (warp - EPI_WARP0) >> 2;
        const int sub_c = 2 * (lane & 3);
        int acc = 0;
        uint32_t acc_phase = 0;
        for_units([&](int cn, const RowSpan, int m0, int n0) {
            if (!__all_sync(0xffffffffu, mbar_wait(tfull(acc), acc_phase, abort_flag, a.err, 16))) return false;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const int m = m0 + quarter * 32 + (lane >> 2);           // this lane's output rows: m + 8 i
            float* P = a.partial + (long long)cn * a.pstride_chunk;
            for (int c0 = 32 * half; c0 < a.BN && n0 + c0 < a.ldw; c0 += 64) {
                const int nc = n0 + c0 + sub_c;
                const int ng = min(4, (min(a.BN - c0, a.ldw - n0 - c0) - sub_c + 7) >> 3);
                float2 v[4][4];
                const uint32_t t0 = tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)acc * acc_cols + (uint32_t)c0;
                if (a.BN - c0 > 16) tmem_ld_16x256b_x4(t0, v);
                else tmem_ld_16x256b_x2(t0, v);
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    if (m + 8 * i >= a.M) break;
                    float* o = P + (long long)(m + 8 * i) * a.ldw + nc;
#pragma unroll
                    for (int g = 0; g < 4; ++g)
                        if (g < ng) *reinterpret_cast<float2*>(o + 8 * g) = v[i][g];
                }
            }
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            __syncwarp();
            if (lane == 0) arrive_drained<CG>(tempty(acc));
            if (++acc == a.nacc) { acc = 0; acc_phase ^= 1u; }
            return true;
        });
    }

    __syncthreads();
    if (*abort_flag && threadIdx.x == 0)   // loads that may still be in flight get a bounded chance to land
        for (int s = 0; s < nst; ++s)
            for (uint32_t i = 0; i < 4096u; ++i)
                if (mbar_try_wait(full(s), 0) || mbar_try_wait(full(s), 1)) break;
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if constexpr (CG == 2) cluster_sync();
    if (warp == 0) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        if constexpr (CG == 2) tmem_dealloc2(tmem_base, tmem_cols);
        else asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(tmem_cols) : "memory");
    }
}

}  // namespace

// How a layer's weight gradient is cut up: pairs of CTAs where there is more than one tile of 128 output rows, the columns in tiles of
// equal width (a multiple of 16, at most 256).
TnShape tn_shape(int fi, int ldw) {
    TnShape t;
    t.cg = fi > BM ? 2 : 1;
    t.ntm = (fi + t.cg * BM - 1) / (t.cg * BM);
    t.ntn = (ldw + 255) / 256;
    t.bn = (int)round_up((ldw + t.ntn - 1) / t.ntn, 16 * t.cg);   // (an MMA of a pair with A in tensor memory takes multiples of 32)
    return t;
}

// Rows per chunk.  A unit costs its 32-row steps (about 0.45 us for a tile of 256 columns, less for narrower ones) plus the fill and
// drain of the pipeline where no other unit of its CTA overlaps them, the units are dealt to the CTAs (pairs) in rounds, and every
// chunk's result is written and read again by the sum over the chunks.  The length with the least total is taken; at most 4096 rows,
// so that the CTAs that share a chunk stay close enough to share it in L2.
int64_t tn_chunk_rows(const std::vector<int32_t>& sub_off, const TnShape& t, int fi, int ldw, int num_sms) {
    const int64_t slots = num_sms / t.cg, tiles = (int64_t)t.ntm * t.ntn;
    int64_t longest = 1;
    for (size_t k = 0; k + 1 < sub_off.size(); ++k) longest = std::max<int64_t>(longest, sub_off[k + 1] - sub_off[k]);
    const double step_us = 0.25 + 0.2 * t.bn / 256.0, sum_us = 8.0 * fi * ldw / 2.0e6;
    int64_t best = 4096;
    double least = 1e300;
    int64_t last = -1;
    for (int64_t c = 1; c <= 4 * 148; ++c) {
        const int64_t R = std::min<int64_t>(4096, round_up((longest + c - 1) / c, TBK));
        if (R == last) { if (R <= TBK) break; continue; }
        last = R;
        int64_t chunks = 0;
        for (size_t k = 0; k + 1 < sub_off.size(); ++k) chunks += (sub_off[k + 1] - sub_off[k] + R - 1) / R;
        const int64_t rounds = (chunks * tiles + slots - 1) / slots;
        const double cost = rounds * (double)(R / TBK) * step_us + 4.0 + 0.5 * rounds + chunks * sum_us;
        if (cost < least) { least = cost; best = R; }
    }
    return best;
}

int tc_tn_rows() { return TBK; }

cudaError_t launch_gemm_tn_tc(const void* mapH, const void* mapZ, int passes, int M, int ldw, const RowSpan* chunks, int nchunks, float* partial,
                              int32_t* err, int num_sms, cudaStream_t s) {
    if (nchunks <= 0) return cudaSuccess;
    const TnShape t = tn_shape(M, ldw);
    TnArgs a;
    a.chunks = chunks; a.ntm = t.ntm; a.ntn = t.ntn; a.BN = t.bn; a.M = M; a.ldw = ldw;
    a.nunits = nchunks * t.ntm * t.ntn;
    const int lo = (t.bn / t.cg + 31) / 32 * BLOCK_BYTES, stage = A_BLOCKS * BLOCK_BYTES + lo;
    a.nlo = passes > 1 && (DATA_BYTES - MAX_LO * lo) / stage >= MAX_LO ? MAX_LO : 2;   // (at most as many as stages: see gemm_rows.cu)
    a.nst = std::min(MAX_STAGES, passes > 1 ? (DATA_BYTES - a.nlo * lo) / stage : DATA_BYTES / stage);
    a.nacc = passes > 1 && t.bn > 128 ? 1 : 2;
    a.partial = partial; a.pstride_chunk = (long long)M * ldw; a.err = err;
    const int units = std::min(a.nunits, num_sms / t.cg);
    auto go = [&](auto kernel) {
        cudaError_t e = configure_kernel_once(reinterpret_cast<const void*>(kernel), SMEM_BYTES, false);
        if (e != cudaSuccess) return e;
        e = launch_cluster(kernel, dim3((unsigned)(units * t.cg)), THREADS, SMEM_BYTES, (unsigned)t.cg, Early::kOverlap, 0, s, *reinterpret_cast<const CUtensorMap*>(mapH),
                   *reinterpret_cast<const CUtensorMap*>(mapZ), a);
        ++g_kernel_launches;
        return e;
    };
    if (t.cg == 2) return passes > 1 ? go(gemm_tn_kernel<2, true>) : go(gemm_tn_kernel<2, false>);
    return passes > 1 ? go(gemm_tn_kernel<1, true>) : go(gemm_tn_kernel<1, false>);
}

}  // namespace gad
