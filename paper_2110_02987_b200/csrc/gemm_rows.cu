// Grouped dense transforms on the 5th-generation tensor cores (tcgen05, accumulators in tensor memory):
//   mode 0   Z_l  = H^(l) W_k^(l)                        (the H.W of the forward equation, Section 3.3)
//   mode 1   dPre = (dZ_l W_k^(l)^T) masked by H^(l) > 0  (chain rule through the forward equation; the mask as bits, which mode 0 left
//            behind while it split H^(l): with the activations themselves the drain waited for its mask loads.  525 000 rows, 256 <- 47 276 -> 174 us,
//            256 <- 256 355 -> 281, 256 -> 256 289 -> 296; 94 000 rows in 50 subgraphs, 128 <- 128 38.9 -> 29.6, 128 -> 128 22.2 -> 25)
//   mode 2   H^(l+1) = sigma((A~ H^(l)) W_k^(l) + b_k^(l)) with dropout: mode 0 finished in the epilogue, for a layer
//            that aggregates before it transforms
// All are C[rows x N] = A[rows x Kd] * B_k^T with A row-major (Kd contiguous) and B_k stored as N rows of Kd contiguous
// values, i.e. both operands K-major.  Row tiles never cross a subgraph, so a tile uses one replica's B.
//
// fp32 accuracy from TF32 tensor cores: every operand value x is split into hi, a value with a 10-bit mantissa (exactly
// representable in TF32), and lo = x - hi rounded to TF32, and the product is accumulated as A_hi B_hi + A_hi B_lo + A_lo B_hi
// in fp32 (the dropped A_lo B_lo term and the rounding of lo are ~2^-20 relative).  B is split once per epoch by a small kernel
// (hi = x rounded).  For A the tile as loaded is its own hi part, because the tensor core ignores the low 13 mantissa bits
// of an fp32 operand (hi = x truncated); eight warps write lo: beside the loaded tile in shared memory, or both parts into tensor memory, from
// which the MMAs then read A (tiles of up to 128 columns).  With passes = 1 only A B is issued on the unsplit operands (TF32 operand precision).
//
// What bounds it is the tensor pipe at 256 x 256, the drain for short reductions, the chain TMA -> split -> MMA -> drain on small launches.  Per 32 values of
// the reduction and 256 output columns the tensor pipe needs 1536 cycles; shared memory gives 128 B per clock and SM.  One CTA alone, A split there, moves
// 256 KB meanwhile (operand reads 144, TMA 80, split 32) and another 32 for a drain that turns its tiles through shared memory: 2250 cycles.  Therefore
//   - the CTAs of a cluster of two work as a pair (cta_group::2): each holds 128 rows of A and half of the B rows, and one
//     MMA of M = 256 reads 4 KB of each from either CTA: 96 KB of operand reads and 48 of TMA instead of 144 and 80;
//   - B stays in shared memory for all tiles of a CTA where it fits beside the ring (up to 256 columns x 128 values);
//   - the drain reads tensor memory in the 16 x 256-bit shape, in which four lanes hold 32 consecutive bytes of a row: whole
//     sectors go to global memory straight from the registers;
//   - the ring of loaded tiles is separate from the split ones (two or four lo tiles, or four slots of tensor memory), so that most of the
//     space holds loads in flight (short reductions are a chain of TMA latency, split and MMA).
// Before this kernel (one CTA per tile, B streamed, drain through shared memory) and with it, event times inside an epoch under the power cap,
// 525 000 rows: 100 -> 256 300 -> 168 us, 256 -> 256 346 -> 290, 256 -> 47 181 -> 153; 110 000 rows, 128 -> 128: 48 -> 33 us (27 through tensor memory).
// Roles of a CTA: warp 0 issues TMA loads, warps 2-9 split the A tile and tell the pair's leader, warp 1 of the leader
// issues the MMAs, warps 10-17 drain.  Every mbarrier wait is bounded: on a time-out the CTA raises an error word, stops, meets its
// peer at the cluster barrier, frees its tensor memory and returns.
#include <cuda.h>

#include <algorithm>

#include "epilogue.cuh"
#include "gad_internal.h"
#include "tc_common.cuh"

namespace gad {

namespace {

constexpr int BK = 32;                                    // values of the reduction per ring stage
constexpr int A_BYTES = BM * BK * 4;                      // 16 KiB
constexpr int MAX_STAGES = 8, MAX_LO = 4;
constexpr int BAR_BYTES = 512;
constexpr int COLSUM_BYTES = 4 * 256 * 4;                 // column sums of the mask drain: 4 row quarters x 256 columns
constexpr int DATA_BYTES = 232448 - 1024 - BAR_BYTES - COLSUM_BYTES;   // 227 KiB less alignment, barriers and column sums
constexpr int SMEM_BYTES = 232448;
constexpr int SPLIT_WARPS = 8, EPI_WARPS = 8, EPI_WARP0 = 2 + SPLIT_WARPS;
constexpr int THREADS = 32 * (EPI_WARP0 + EPI_WARPS);

struct RowsArgs {
    const RowSpan* tiles;     // an even number of them; tiles 2 p and 2 p + 1 belong to the same subgraph
    int npairs, ntn, BN, Kd;
    int nst, nlo;             // ring stages; lo tiles (2 or 4, at most nst: see the split)
    int resident;             // B loaded once per (subgraph, column tile) instead of once per stage
    float* C;
    uint32_t* Cbf;            // mode 0: the result as bfloat16 (two values per word) instead of C, or null
    int ldc;
    uint32_t* bits;           // mode 0: receives which values of A are above zero; mode 1: the mask; or null.  Bit c % 32 of word c / 32 of a row
    int bit_words;            // words of a row
    float scale;
    float* colsum;            // masked drains: column sums of what is written (the bias gradient of the layer below), or null:
                              // [(cluster + subgraph) * 8 + rank * 4 + row quarter][ldc] of every (cluster, subgraph) that meet
    int kmul;                 // 1: every subgraph has its own B; 0: one B for all (the replicas' parameters are equal)
    int32_t* err;
    ActEpi act;               // mode 2
};

// What the drain does with a value: nothing (mode 0, or 1 without a mask), bfloat16 (mode 0), the ReLU mask and dropout scale (mode
// 1), bias and ReLU (mode 2), those with dropout.  A template parameter, like the number of passes: as branches inside the unrolled
// drain they made the kernel wait for instructions, 10.7 us per 128 x 256 tile.
enum Drain { kPlain, kBf16, kMask, kMaskBf16, kAct, kActDrop };

// Tile t of the launch: resident, column tile by column tile (B changes rarely); otherwise the column tiles of a row tile
// follow each other (A comes from L2 the second time).
__device__ __forceinline__ void tile_of(const RowsArgs& a, int t, int& pair, int& n) {
    if (a.resident) { n = t / a.npairs; pair = t % a.npairs; }
    else { pair = t / a.ntn; n = t % a.ntn; }
}

// How A reaches the tensor cores: as loaded (one pass); its lo part beside it in shared memory; or both parts through tensor memory.
enum Form { kOnePass, kSharedLo, kTensorMem };
constexpr int ACC_COLS = 128;                   // columns between the accumulators there (the other forms: as many as the tile has)
constexpr int SLOTS = 4, SLOT_COLS = 2 * BK;   // tensor-memory slots of a 128 x 32 step of A: 32 columns of hi, 32 of lo
constexpr uint32_t TMEM_COLS = 512;
constexpr int kRowPairs = 74;                   // pairs of CTAs at work at a time

template <int DRAIN, int FORM>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(THREADS, 1)
gemm_rows_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, const __grid_constant__ CUtensorMap tmBlo,
                 const RowsArgs a) {
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw_addr = smem_u32(smem_raw);
    const uint32_t pad = ((raw_addr + 1023u) & ~1023u) - raw_addr;   // the same in both CTAs (the 128B swizzle repeats every 1024 bytes)
    uint8_t* sm = smem_raw + pad;
    const uint32_t sm_addr = raw_addr + pad;
    const uint32_t rank = cluster_rank();
    const int nkb = (a.Kd + BK - 1) / BK;
    const uint32_t b_bytes = (uint32_t)(a.BN / 2) * (BK * 4);              // this CTA's half of a B tile
    constexpr bool split = FORM != kOnePass;
    constexpr uint32_t nb = split ? 2u : 1u;
    const uint32_t off_lo = a.resident ? (uint32_t)nkb * b_bytes * nb : 0u;
    const uint32_t off_ring = off_lo + (FORM == kSharedLo ? (uint32_t)a.nlo * A_BYTES : 0u);
    const uint32_t stage_bytes = (uint32_t)A_BYTES + (a.resident ? 0u : nb * b_bytes);
    const int nst = a.nst;
    const uint32_t bars = sm_addr + DATA_BYTES;
    auto full = [&](int s) { return bars + 8u * s; };
    auto empty = [&](int s) { return bars + 8u * (MAX_STAGES + s); };
    auto xfull = [&](int q) { return bars + 8u * (2 * MAX_STAGES + q); };              // leader: both CTAs' operands of this step are ready
    auto loempty = [&](int q) { return bars + 8u * (2 * MAX_STAGES + MAX_LO + q); };
    auto tfull = [&](int i) { return bars + 8u * (2 * MAX_STAGES + 2 * MAX_LO + i); };
    auto tempty = [&](int i) { return bars + 8u * (2 * MAX_STAGES + 2 * MAX_LO + 2 + i); };
    const uint32_t bfull = bars + 8u * (2 * MAX_STAGES + 2 * MAX_LO + 4), bempty = bfull + 8u;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(sm + DATA_BYTES + 8 * (2 * MAX_STAGES + 2 * MAX_LO + 6));
    volatile uint32_t* abort_flag = tmem_slot + 1;
    const uint32_t tmem_cols = FORM == kTensorMem ? TMEM_COLS : 2u * (uint32_t)a.BN;
    const int acc_cols = FORM == kTensorMem ? ACC_COLS : a.BN;
    // groups of splitting warps that take steps in turn (kTensorMem: a group has a warp for every quarter of the lanes)
    const int groups = FORM == kTensorMem ? SPLIT_WARPS / 4 : a.nlo == MAX_LO ? MAX_LO : 1;

    pdl_next();
    const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;   // (uniform, and known to be)
    if (threadIdx.x == 0) {
        for (int s = 0; s < MAX_STAGES; ++s) { mbar_init(full(s), 1); mbar_init(empty(s), FORM == kTensorMem && a.resident ? SPLIT_WARPS / groups : 1); }
        for (int q = 0; q < MAX_LO; ++q) { mbar_init(xfull(q), 2 * SPLIT_WARPS / groups); mbar_init(loempty(q), 1); }
        for (int i = 0; i < 2; ++i) { mbar_init(tfull(i), 1); mbar_init(tempty(i), 2 * EPI_WARPS); }
        mbar_init(bfull, 1); mbar_init(bempty, 1);
        *abort_flag = 0u;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) tmem_alloc2(smem_u32(tmem_slot), tmem_cols);
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    cluster_sync();           // the peer's barriers exist before anything arrives at them
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem_base = *tmem_slot;

    // From here on operands are read (the tile list is nobody's output: what follows may have it already).  Every thread waits: each role
    // reads or writes something of its own.
    pdl_wait();
    // contiguous ranges of tiles: B changes as rarely as possible
    const int ntiles = a.npairs * a.ntn, ncl = gridDim.x >> 1, cl = blockIdx.x >> 1;
    const int t_begin = (int)((long long)ntiles * cl / ncl), t_end = (int)((long long)ntiles * (cl + 1) / ncl);
    // calls f(tile, pair, n, B differs from the previous tile's) until it returns false
    auto for_tiles = [&](auto&& f) {
        int last_k = -1, last_n = -1;
        for (int t = t_begin; t < t_end; ++t) {
            int pair, n;
            tile_of(a, t, pair, n);
            const int k = a.kmul ? a.tiles[2 * pair].k : 0;
            if (!f(pair, n, k, k != last_k || n != last_n)) return;
            last_k = k; last_n = n;
        }
    };

    if (warp == 0 && lane == 0) {
        // ---------------- TMA producer ----------------
        int stage = 0;
        uint32_t phase = 0, bphase = 0;
        for_tiles([&](int pair, int n, int k, bool new_b) {
            const int row0 = a.tiles[2 * pair + (int)rank].row0, n0 = n * a.BN + (int)rank * (a.BN / 2);
            if (a.resident && new_b) {
                if (!mbar_wait(bempty, bphase ^ 1u, abort_flag, a.err, 1)) return false;
                bphase ^= 1u;
                mbar_expect_tx(bfull, (uint32_t)nkb * nb * b_bytes);
                for (int kb = 0; kb < nkb; ++kb) {
                    tma_load_3d(sm_addr + (uint32_t)kb * nb * b_bytes, &tmB, kb * BK, n0, k, bfull);
                    if (split) tma_load_3d(sm_addr + ((uint32_t)kb * nb + 1u) * b_bytes, &tmBlo, kb * BK, n0, k, bfull);
                }
            }
            for (int kb = 0; kb < nkb; ++kb) {
                if (!mbar_wait(empty(stage), phase ^ 1u, abort_flag, a.err, 2)) return false;
                mbar_expect_tx(full(stage), stage_bytes);
                const uint32_t base = sm_addr + off_ring + (uint32_t)stage * stage_bytes;
                tma_load_2d(base, &tmA, kb * BK, row0, full(stage));
                if (!a.resident) {
                    tma_load_3d(base + A_BYTES, &tmB, kb * BK, n0, k, full(stage));
                    if (split) tma_load_3d(base + A_BYTES + b_bytes, &tmBlo, kb * BK, n0, k, full(stage));
                }
                if (++stage == nst) { stage = 0; phase ^= 1u; }
            }
            return true;
        });
    } else if (warp == 1 && rank == 0) {
        // ---------------- MMA issuer (leader of the pair) ----------------
        // The whole warp runs the loop and one elected lane issues: everything the MMAs take then stays in uniform registers, where
        // the instruction wants it (with a loop of one lane alone an MMA took 75 cycles to issue).
        int stage = 0, q = 0, acc = 0;
        uint32_t qphase = 0, acc_phase = 0;
        const uint32_t idesc = instr_desc(a.BN, 2 * BM);
        bool first = true;
        for_tiles([&](int, int, int, bool new_b) {
            if (a.resident && new_b && !first && elect_one()) mma_commit2(bempty);   // every MMA on the previous B has been issued
            first = false;
            if (!__all_sync(0xffffffffu, mbar_wait<true>(tempty(acc), acc_phase ^ 1u, abort_flag, a.err, 3))) return false;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const uint32_t d = tmem_base + (uint32_t)(acc * acc_cols);
            for (int kb = 0; kb < nkb; ++kb) {
                if (!__all_sync(0xffffffffu, mbar_wait<true>(xfull(q), qphase, abort_flag, a.err, 4))) return false;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const uint32_t base = sm_addr + off_ring + (uint32_t)stage * stage_bytes;
                const uint32_t bbase = a.resident ? sm_addr + (uint32_t)kb * nb * b_bytes : base + A_BYTES;
                const uint64_t a_hi = smem_desc(base), a_lo = smem_desc(sm_addr + off_lo + (uint32_t)q * A_BYTES);
                const uint32_t a_tm = tmem_base + TMEM_COLS - SLOTS * SLOT_COLS + (uint32_t)(q * SLOT_COLS);
                const uint64_t b_hi = smem_desc(bbase), b_lo = smem_desc(bbase + b_bytes);
                const int nks = min(BK / 8, (a.Kd - kb * BK + 7) / 8);
                if (elect_one()) {
                    // 8 TF32 values = 32 bytes = 2 descriptor units along K
#pragma unroll
                    for (int ks = 0; ks < BK / 8; ++ks) {
                        if (ks < nks) {
                            if constexpr (FORM == kTensorMem) {
                                mma_tf32_pair_ts(d, a_tm + 8 * ks, b_hi + 2 * ks, idesc, (kb | ks) != 0 ? 1u : 0u);
                                mma_tf32_pair_ts(d, a_tm + 8 * ks, b_lo + 2 * ks, idesc, 1u);
                                mma_tf32_pair_ts(d, a_tm + BK + 8 * ks, b_hi + 2 * ks, idesc, 1u);
                                continue;
                            }
                            mma_tf32_pair(d, a_hi + 2 * ks, b_hi + 2 * ks, idesc, (kb | ks) != 0 ? 1u : 0u);
                            if (split) {
                                mma_tf32_pair(d, a_hi + 2 * ks, b_lo + 2 * ks, idesc, 1u);
                                mma_tf32_pair(d, a_lo + 2 * ks, b_hi + 2 * ks, idesc, 1u);
                            }
                        }
                    }
                    // the stage may be refilled, and the lo tile rewritten, in both CTAs once these MMAs have read them
                    if (FORM != kTensorMem || !a.resident) mma_commit2(empty(stage));
                    mma_commit2(loempty(q));
                    if (kb == nkb - 1) mma_commit2(tfull(acc));   // accumulator complete, in both CTAs
                }
                __syncwarp();
                if (++stage == nst) stage = 0;
                if (++q == a.nlo) { q = 0; qphase ^= 1u; }
            }
            if (++acc == 2) { acc = 0; acc_phase ^= 1u; }
            return true;
        });
    } else if (warp >= 2 && warp < EPI_WARP0) {
        // ---------------- A split: lo = x - (x as the tensor core reads it); the pair's leader is told ----------------
        // With two lo tiles (wide outputs: the tensor pipe sets the pace) all warps share a step.  With four they form four groups
        // that take turns: what a step costs is then mostly waiting - for the barriers, the proxy fence and the arrival - so four
        // steps are in hand at a time.  (Through tensor memory a group has a warp for every quarter of the lanes, so that there are two.)  (A group's wait for a ring stage is unambiguous because nlo <= nst: once its own previous
        // step has been multiplied, so has the step before in that stage.)
        const int gw = SPLIT_WARPS / groups, group = (warp - 2) / gw, tt = threadIdx.x - 64 - 32 * gw * group;
        constexpr bool leaves_bits = DRAIN == kPlain || DRAIN == kBf16;
        uint32_t* bits = a.bits;
        after_wait(bits);
        const int row = 32 * (warp & 3) + lane;       // kTensorMem: this thread's row of the tile, in its warp's quarter of the lanes
        int stage = 0, q = 0;
        uint32_t phase = 0, qphase = 0, bphase = 0;
        for_tiles([&](int pair, int n, int, bool new_b) {
            RowSpan sp{0, 0, 0, 0};                       // the rows whose signs are left behind: with the first column tile, where asked for
            if (leaves_bits && a.bits && n == 0) sp = a.tiles[2 * pair + (int)rank];
            // (the votes keep the warp together: lanes may see a time-out or an abort at different polls)
            if (a.resident && new_b) {
                if (!__all_sync(0xffffffffu, mbar_wait(bfull, bphase, abort_flag, a.err, 5))) return false;
                bphase ^= 1u;
            }
            for (int kb = 0; kb < nkb; ++kb) {
                if (groups == 1 || (q & (groups - 1)) == group) {
                    if (!__all_sync(0xffffffffu, mbar_wait(loempty(q), qphase ^ 1u, abort_flag, a.err, 6))) return false;
                    if (!__all_sync(0xffffffffu, mbar_wait(full(stage), phase, abort_flag, a.err, 7))) return false;
                    if constexpr (FORM == kTensorMem) {
                        // (the 16-byte pieces of a row are swizzled by the row; eight neighbouring lanes cover all banks)
                        const uint8_t* src = sm + off_ring + (uint32_t)stage * stage_bytes + row * (4 * BK);
                        float hi[BK], lo[BK];
#pragma unroll
                        for (int j = 0; j < BK / 4; ++j) {
                            const float4 v = *reinterpret_cast<const float4*>(src + ((j ^ (row & 7)) << 4));
                            hi[4 * j] = v.x; hi[4 * j + 1] = v.y; hi[4 * j + 2] = v.z; hi[4 * j + 3] = v.w;
                        }
#pragma unroll
                        for (int i = 0; i < BK; ++i) lo[i] = tf32_rest(hi[i]);
                        const uint32_t dst = tmem_base + ((uint32_t)(32 * (warp & 3)) << 16) + TMEM_COLS - SLOTS * SLOT_COLS + (uint32_t)(q * SLOT_COLS);
                        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");   // the MMAs that read the slot have completed
                        tmem_st_32x32b_x32(dst, hi);
                        tmem_st_32x32b_x32(dst + BK, lo);
                        tmem_wait_st();
                        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                        __syncwarp();
                        if (lane == 0) {
                            if (a.resident) mbar_arrive(empty(stage));   // nobody else reads the stage
                            mbar_arrive_leader_tmem(xfull(q));
                        }
                        if (row < sp.nrows) {
                            uint32_t w = 0;
#pragma unroll
                            for (int i = 0; i < BK; ++i) w |= (hi[i] > 0.f ? 1u : 0u) << i;
                            bits[((long long)sp.row0 + row) * a.bit_words + kb] = w;
                        }
                    } else {
                    if (FORM == kSharedLo || sp.nrows > 0) {
                        // a thread takes half a row at a time (its 16-byte pieces are swizzled by the row: neighbouring lanes cover all banks); a
                        // word of sign bits put together from several lanes made the kernel 37 to 85 % longer
                        const uint8_t* hi = sm + off_ring + (uint32_t)stage * stage_bytes;
                        uint8_t* lo = sm + off_lo + (uint32_t)q * A_BYTES;
                        for (int u = tt; u < 2 * BM; u += 32 * gw) {
                            const int r = u & (BM - 1), h = u >> 7;
                            float4 v[4];
#pragma unroll
                            for (int j = 0; j < 4; ++j) v[j] = *reinterpret_cast<const float4*>(hi + r * (4 * BK) + (((4 * h + j) ^ (r & 7)) << 4));
                            if (FORM == kSharedLo)   // (the tile as loaded stays where it is: the MMA reads it as the hi part)
#pragma unroll
                                for (int j = 0; j < 4; ++j)
                                    *reinterpret_cast<float4*>(lo + r * (4 * BK) + (((4 * h + j) ^ (r & 7)) << 4)) =
                                        make_float4(tf32_rest(v[j].x), tf32_rest(v[j].y), tf32_rest(v[j].z), tf32_rest(v[j].w));
                            if (r < sp.nrows) {
                                uint32_t w = 0;
#pragma unroll
                                for (int j = 0; j < 4; ++j)
                                    w |= ((v[j].x > 0.f ? 1u : 0u) | (v[j].y > 0.f ? 2u : 0u) | (v[j].z > 0.f ? 4u : 0u) | (v[j].w > 0.f ? 8u : 0u)) << (4 * j);
                                reinterpret_cast<uint16_t*>(bits + ((long long)sp.row0 + r) * a.bit_words + kb)[h] = (uint16_t)w;
                            }
                        }
                    }
                    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // generic-proxy writes -> tensor-core reads
                    __syncwarp();
                    if (lane == 0) mbar_arrive_leader(xfull(q));
                    }
                }
                if (++q == a.nlo) { q = 0; qphase ^= 1u; }
                if (++stage == nst) { stage = 0; phase ^= 1u; }
            }
            return true;
        });
    } else if (warp >= EPI_WARP0) {
        // ---------------- epilogue: tensor memory -> registers -> global ----------------
        // This warp may read tensor-memory lanes 32 q .. 32 q + 31; the two warps of a quarter take alternate blocks of 32 columns.
        // In a 16 x 256-bit read lane t gets, of every 8 columns, columns 2 (t % 4) and the next one of rows t / 4 and t / 4 + 8.
        const int quarter = warp & 3, half = (warp - EPI_WARP0) >> 2;
        const int sub_r = lane >> 2, sub_c = 2 * (lane & 3);
        const uint32_t* bits = a.bits;
        ActEpi act = a.act;
        after_wait(bits);
        after_wait(act.params);
        constexpr bool masked = DRAIN == kMask || DRAIN == kMaskBf16, to_bf16 = DRAIN == kBf16 || DRAIN == kMaskBf16;
        // This warp's column sums: the columns of its blocks, of its quarter of the rows; nobody else touches them.  They are written out
        // when the subgraph changes and at the end: the tiles of a cluster are consecutive, so its subgraphs ascend and cluster +
        // subgraph names the pair.
        float* cs = reinterpret_cast<float*>(sm + DATA_BYTES + BAR_BYTES) + quarter * 256;
        int cs_k = -1;
        auto flush_colsum = [&](int next_k) {
            __syncwarp();
            for (int c0 = 32 * half; c0 < a.BN; c0 += 64) {
                const int c = c0 + lane;
                if (cs_k >= 0 && c < a.ldc && c < a.BN) a.colsum[((long long)(cl + cs_k) * 8 + (int)rank * 4 + quarter) * a.ldc + c] = cs[c];
                cs[c] = 0.f;
            }
            __syncwarp();
            cs_k = next_k;
        };
        int acc = 0;
        uint32_t acc_phase = 0;
        for_tiles([&](int pair, int n, int, bool) {
            const RowSpan sp = a.tiles[2 * pair + (int)rank];
            const int n0 = n * a.BN;
            if (masked && a.colsum && sp.k != cs_k) flush_colsum(sp.k);
            const int r0 = quarter * 32 + sub_r;                 // this lane's rows: r0 + 8 i
            // a block's mask bits are asked for one block ahead, the first ones before the wait for the accumulator
            uint32_t next_mb[4];
            auto fetch_bits = [&](int c0) {
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    next_mb[i] = r0 + 8 * i < sp.nrows && c0 < a.BN && n0 + c0 < a.ldc
                                     ? __ldg(bits + ((long long)sp.row0 + r0 + 8 * i) * a.bit_words + ((n0 + c0) >> 5)) >> sub_c : 0u;
            };
            if (masked) fetch_bits(32 * half);
            if (!__all_sync(0xffffffffu, mbar_wait(tfull(acc), acc_phase, abort_flag, a.err, 8))) return false;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            for (int c0 = 32 * half; c0 < a.BN && n0 + c0 < a.ldc; c0 += 64) {
                const int nc = n0 + c0 + sub_c;                  // this lane's columns: nc + 8 g, nc + 8 g + 1
                const int ng = min(4, (min(a.BN - c0, a.ldc - n0 - c0) - sub_c + 7) >> 3);   // groups it has columns in
                const long long at0 = ((long long)sp.row0 + r0) * a.ldc + nc;
                float2 bias[4];
                uint32_t mb[4];
                if (masked) {
#pragma unroll
                    for (int i = 0; i < 4; ++i) mb[i] = next_mb[i];
                    fetch_bits(c0 + 64);
                }
                if (DRAIN == kAct || DRAIN == kActDrop)
#pragma unroll
                    for (int g = 0; g < 4; ++g) bias[g] = g < ng ? load_bias2(act, sp.k, nc + 8 * g) : make_float2(0.f, 0.f);
                float2 v[4][4];                                  // [row r0 + 8 i][columns nc + 8 g]
                const uint32_t t0 = tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(acc * acc_cols + c0);
                tmem_ld_16x256b_x4(t0, v);
                if (masked) {
#pragma unroll
                    for (int i = 0; i < 4; ++i)
#pragma unroll
                        for (int g = 0; g < 4; ++g) {
                            v[i][g].x = mb[i] >> (8 * g) & 1u ? v[i][g].x * a.scale : 0.f;
                            v[i][g].y = mb[i] >> (8 * g + 1) & 1u ? v[i][g].y * a.scale : 0.f;
                        }
                    if (a.colsum) {   // (rows and columns that do not exist are masked to zero)
#pragma unroll
                        for (int g = 0; g < 4; ++g) {
                            float2 t = make_float2((v[0][g].x + v[1][g].x) + (v[2][g].x + v[3][g].x), (v[0][g].y + v[1][g].y) + (v[2][g].y + v[3][g].y));
#pragma unroll
                            for (int o = 4; o < 32; o <<= 1) { t.x += __shfl_xor_sync(0xffffffffu, t.x, o); t.y += __shfl_xor_sync(0xffffffffu, t.y, o); }
                            if (lane < 4 && c0 + 8 * g < a.BN) { cs[c0 + 8 * g + sub_c] += t.x; cs[c0 + 8 * g + sub_c + 1] += t.y; }
                        }
                    }
                }
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    if (r0 + 8 * i >= sp.nrows) break;
                    uint64_t key = 0;
                    if (DRAIN == kActDrop) key = dropout_row_key(a.act, (long long)sp.row0 + r0 + 8 * i);
                    const long long at = at0 + 8 * i * a.ldc;
#pragma unroll
                    for (int g = 0; g < 4; ++g) {
                        float2 o = v[i][g];
                        if (DRAIN == kAct || DRAIN == kActDrop) {
                            o.x = relu_unless(o.x + bias[g].x, a.act.relu);
                            o.y = relu_unless(o.y + bias[g].y, a.act.relu);
                        }
                        if (DRAIN == kActDrop) {
                            o.x = dropout_keep(key, nc + 8 * g, a.act.thr) ? o.x * a.act.scale : 0.f;
                            o.y = dropout_keep(key, nc + 8 * g + 1, a.act.thr) ? o.y * a.act.scale : 0.f;
                        }
                        if (g < ng) {
                            if (to_bf16) a.Cbf[(at + 8 * g) >> 1] = bf16_bits(o.x) | (bf16_bits(o.y) << 16);
                            else *reinterpret_cast<float2*>(a.C + at + 8 * g) = o;
                        }
                    }
                }
            }
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            __syncwarp();
            if (lane == 0) mbar_arrive_leader_tmem(tempty(acc));
            if (++acc == 2) { acc = 0; acc_phase ^= 1u; }
            return true;
        });
        if (masked && a.colsum) flush_colsum(-1);
    }

    // Tear-down.  After a time-out, give loads that may still be in flight a bounded chance to land before the shared memory is
    // released.  Neither CTA leaves while the other may still read its operands or arrive at its barriers.
    __syncthreads();
    if (*abort_flag && threadIdx.x == 0)
        for (int s = 0; s < nst; ++s)
            for (uint32_t i = 0; i < 4096u; ++i)
                if (mbar_try_wait(full(s), 0) || mbar_try_wait(full(s), 1)) break;
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    cluster_sync();
    if (warp == 0) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        tmem_dealloc2(tmem_base, tmem_cols);
    }
}

}  // namespace

namespace {

// Which form a launch takes.  Through tensor memory A costs shared memory one write and one read where a lo tile beside it costs six times its
// size (written and read by the split, read by three MMAs); with 256 columns a tile's two accumulators fill the tensor memory.
int form_for(int BN, int passes) { return passes <= 1 ? kOnePass : BN <= 128 ? kTensorMem : kSharedLo; }

// What a resident B (both parts) leaves for A.
long long room_beside_b(int BN, int Kd) { return (long long)DATA_BYTES - (long long)((Kd + BK - 1) / BK) * 2 * (BN / 2) * (BK * 4); }
// Turns of the CTA pairs that a launch of ntn column tiles takes, and whether a launch is one of few turns (in tiles of 256 columns).
long long turns_of(int npairs, int ntn) { return ((long long)npairs * ntn + kRowPairs - 1) / kRowPairs; }
bool few_turns(int npairs, int n_cols) { return turns_of(npairs, (n_cols + 255) / 256) < 4; }
// Through tensor memory: whether B stays for all row tiles.  With several column tiles that means that A is read from HBM for each of them, where a streamed B
// lets it come from L2 the second time, so that on large launches it pays only for reductions of at most four steps whose rows of A share 32-byte sectors (a
// leading dimension that is no multiple of 8).  525 000 rows, us resident / streamed: 100 -> 256 168 / 231, 33 -> 320 without an epilogue 141 / 170; but 64 -> 256 144 / 145,
// 128 -> 384 193 / 180, without an epilogue 192 -> 192 224 / 209, 129 -> 320 275 / 244 and 300 000 rows of 146 -> 267 246 / 181, with dropout 100 -> 300 455 / 369; and where a tile's
// worth of columns is only just passed 100 -> 257 346 / 255, 24 -> 129 163 / 105.  Of few turns: 21 000 rows, 100 -> 150 19 / 19, 128 -> 256 21 / 20, 129 -> 300 27 / 25.
bool keeps_b(int BN, int Kd, int n_cols, int npairs, bool drop) {
    if (room_beside_b(BN, Kd) < SLOTS * A_BYTES) return false;
    if (n_cols <= BN) return true;
    if (Kd > 4 * BK) return false;
    return few_turns(npairs, n_cols) || (!drop && round_up(Kd, 4) % 8 != 0 && (n_cols - 1) % 128 >= 8);
}

// Where the data of a CTA goes: four lo tiles if at least as many ring stages fit beside them, else two; B resident if at least
// three ring stages fit beside it.
void rows_layout(int BN, int Kd, int n_cols, int form, RowsArgs& a) {
    const int passes = form == kOnePass ? 1 : 3;
    const int nkb = (Kd + BK - 1) / BK, nb = passes > 1 ? 2 : 1;
    const int b_bytes = BN / 2 * (BK * 4);
    if (form == kTensorMem) {   // as many stages as there are slots, at least (see the split)
        a.nlo = SLOTS;
        a.resident = keeps_b(BN, Kd, n_cols, a.npairs, a.act.drop != 0) ? 1 : 0;
        a.nst = (int)std::min<long long>(MAX_STAGES, a.resident ? room_beside_b(BN, Kd) / A_BYTES : DATA_BYTES / (A_BYTES + nb * b_bytes));
        return;
    }
    for (a.nlo = 4;; a.nlo = 2) {
        const long long room = (long long)DATA_BYTES - (passes > 1 ? a.nlo * A_BYTES : 0), room_a = room - (long long)nkb * nb * b_bytes;
        a.resident = room_a >= (a.nlo > 3 ? a.nlo : 3) * A_BYTES ? 1 : 0;
        const long long n = a.resident ? room_a / A_BYTES : room / (A_BYTES + nb * b_bytes);
        a.nst = (int)(n < MAX_STAGES ? n : MAX_STAGES);
        // (a resident B with two lo tiles is worth more than a streamed one with four)
        if (a.nlo == 2 || (a.nst >= 4 && (a.resident || (long long)DATA_BYTES - 2 * A_BYTES - (long long)nkb * nb * b_bytes < 3 * A_BYTES))) return;
    }
}

int max_clusters(int num_sms) {
    static std::atomic<int> known{0};
    if (known.load() <= 0) known.store(max_active_pairs(reinterpret_cast<const void*>(gemm_rows_kernel<kPlain, kSharedLo>), THREADS, SMEM_BYTES, num_sms));
    return known.load();
}

}  // namespace

// Output columns per tile.  Where a launch has so few row tiles that most SMs would idle the columns are spread over more CTAs, down to 32
// (2843 rows x 1433 -> 128: 24 row tiles, 40 us with 128 columns per tile, 27 us with 32).
static int spread_columns(int bn, int n_cols, int npairs) {
    while (bn > 32 && (long long)npairs * ((n_cols + bn - 1) / bn) * 2 <= kRowPairs) bn = (int)round_up(bn / 2, 32);
    return bn;
}
// The transform back through a layer, in one pass or three, and every transform in one pass, whose MMAs cost little beside reading A again (256 -> 256 over
// 210 000 rows 86 us in tiles of 256 columns, 104 of 128): as wide as the layer, up to 256, so that a masked drain can sum the columns.  (So are the ways back
// that sum none, without a mask or of more than 256 columns; narrower tiles have not been measured there.)
int tc_rows_bn_whole(int n_cols, int npairs) {
    return spread_columns(n_cols <= 32 ? 32 : n_cols <= 64 ? 64 : n_cols <= 128 ? 128 : 256, n_cols, npairs);
}
// A forward transform in three passes: equal tiles of at most 128 columns, whose A goes through tensor memory, or on large launches the same as above.
// Such a tile costs about half of one of 256 columns, a little more where the drain is what the kernel waits for (reductions of up to 96 values, dropout) or B is
// streamed beside rows of A that share sectors; there that many turns of the CTA pairs have to come out shorter.  us in tiles of 256 / of up to 128 columns:
// 21 000 rows in 8 subgraphs (two turns or three half ones) 500 -> 256 46 / 38, 100 -> 256 24 / 20, with dropout 100 -> 257 47 / 35; 525 000 rows 24 -> 256 121 / 139, 100 -> 256
// 178 / 168, 24 -> 150 80 / 113, 256 -> 256 280 / 287 and without an epilogue 303 / 291, 64 -> 300 220 / 166; with dropout 128 -> 150 240 / 262, 256 -> 256 381 / 412,
// 100 -> 300 506 / 369.  1500 combinations of 24 to 500 -> 129 to 512, four sizes, with and without an epilogue and dropout: 10 % less than in wide tiles (the best of all
// forms for each: 11), 4 % less than in narrow ones throughout, at most 10 % above the best of the two.
int tc_rows_bn(int n_cols, int npairs, int Kd, bool drop) {
    const int ntn = (n_cols + 127) / 128, bn = (int)round_up((n_cols + ntn - 1) / ntn, 32);
    if (n_cols > 128 && !few_turns(npairs, n_cols)) {
        const bool half = !drop && Kd > 96 && (round_up(Kd, 4) % 8 == 0 || Kd > 160 || keeps_b(bn, Kd, n_cols, npairs, drop));
        if ((double)turns_of(npairs, ntn) * (half ? 0.5 : 0.55) > (double)turns_of(npairs, (n_cols + 255) / 256)) return tc_rows_bn_whole(n_cols, npairs);
    }
    return spread_columns(bn, n_cols, npairs);
}

// The drain can sum columns when a tile holds all of them.
bool tc_rows_sums_columns(int n_cols, int npairs) { return tc_rows_bn_whole(n_cols, npairs) >= n_cols; }
int tc_rows_clusters(long long ntiles, int num_sms) { return (int)std::min<long long>(ntiles, std::min(max_clusters(num_sms), kMaxRowClusters)); }

cudaError_t launch_gemm_rows_tc(const void* mapA, const void* mapB, const void* mapBlo, int mode, int passes, int Kd, int n_cols, int bn,
                                float* C, int ldc, const RowSpan* pair_tiles, int npairs, uint32_t* bits, int bit_words, float scale,
                                const ActEpi* act, int32_t* err, int num_sms, cudaStream_t s, bool one_b, void* Cbf16, float* colsum) {
    if (npairs <= 0) return cudaSuccess;
    if ((mode == 2 && !act) || (Cbf16 && mode == 2) || (Cbf16 && mode == 1 && !bits)) return cudaErrorInvalidValue;
    if (colsum && !(mode == 1 && bits && bn >= n_cols)) return cudaErrorInvalidValue;
    RowsArgs a;
    a.tiles = pair_tiles; a.npairs = npairs; a.BN = bn; a.ntn = (ldc + a.BN - 1) / a.BN; a.Kd = Kd;
    a.act = act ? *act : ActEpi{};
    const int form = form_for(a.BN, passes);
    rows_layout(a.BN, Kd, n_cols, form, a);
    a.C = C; a.Cbf = reinterpret_cast<uint32_t*>(Cbf16); a.ldc = ldc; a.bits = mode == 2 ? nullptr : bits; a.bit_words = bit_words; a.scale = scale; a.colsum = colsum;
    a.kmul = one_b ? 0 : 1; a.err = err;
    const unsigned grid = 2u * (unsigned)tc_rows_clusters((long long)npairs * a.ntn, num_sms);
    const int drain = mode == 2 ? (a.act.drop ? kActDrop : kAct) : mode == 1 && bits ? (Cbf16 ? kMaskBf16 : kMask) : Cbf16 ? kBf16 : kPlain;
    auto go = [&](auto kernel) {
        cudaError_t e = configure_kernel_once(reinterpret_cast<const void*>(kernel), SMEM_BYTES, false);
        if (e != cudaSuccess) return e;
        e = launch(kernel, dim3(grid), THREADS, SMEM_BYTES, s, *reinterpret_cast<const CUtensorMap*>(mapA), *reinterpret_cast<const CUtensorMap*>(mapB),
                                                 *reinterpret_cast<const CUtensorMap*>(mapBlo), a);
        ++g_kernel_launches;
        return e;
    };
#define GAD_DRAIN(D) case D: return form == kTensorMem ? go(gemm_rows_kernel<D, kTensorMem>) : form == kSharedLo ? go(gemm_rows_kernel<D, kSharedLo>) : go(gemm_rows_kernel<D, kOnePass>)
    switch (drain) {
        GAD_DRAIN(kPlain);
        GAD_DRAIN(kMask);
        GAD_DRAIN(kAct);
        GAD_DRAIN(kActDrop);
        case kBf16: if (form == kOnePass) return go(gemm_rows_kernel<kBf16, kOnePass>); break;   // the reduced-precision mode's
        case kMaskBf16: if (form == kOnePass) return go(gemm_rows_kernel<kMaskBf16, kOnePass>); break;
    }
#undef GAD_DRAIN
    return cudaErrorInvalidValue;
}

}  // namespace gad
