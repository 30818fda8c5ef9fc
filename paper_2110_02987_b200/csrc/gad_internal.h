// Internal declarations shared by the translation units of the library (not part of the boundary).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>
#include <cmath>
#include <string>
#include <vector>

#include "../../include/gad.h"
#include "launch.cuh"

namespace gad {

// Host loops run on OpenMP's default team or on the calling thread alone, never on a team of another size: a smaller one takes the threads
// it does not need down, and the next full one sets them up again (16 threads: a region of the same team 2 us, the first full one after
// a region of 2 / 4 / 8 threads 310 / 260 / 150 us).

inline int64_t round_up(int64_t x, int64_t m) { return (x + m - 1) / m * m; }

// Kernels launched by this library in this process (every <<<>>> adds one; contexts on several host threads share it).
extern std::atomic<int64_t> g_kernel_launches;

// Function attributes belong to a device: asks once per (current device, kernel) for `smem_bytes` of dynamic shared
// memory and, with `max_carveout`, for the largest shared-memory share of the SM.  Safe from several host threads.
cudaError_t configure_kernel_once(const void* kernel, int smem_bytes, bool max_carveout);

// Clusters of two CTAs of a kernel that fit the GPU at once (a cluster stays inside a GPC).
int max_active_pairs(const void* kernel, unsigned threads, size_t smem_bytes, int num_sms);

// ---------------------------------------------------------------------------------------------
// Host-side result of building the block-diagonal store (create-time, not on the timed path).
// ---------------------------------------------------------------------------------------------
struct HostStore {
    int32_t K = 0;
    int64_t Np = 0, nnz = 0;
    std::vector<int64_t> rowptr;   // [Np+1]
    std::vector<int32_t> col;      // [nnz] store-row ids, ascending inside a row
    std::vector<float> val;        // [nnz] A~ entries, computed in double and rounded once
    std::vector<int32_t> sub_off;  // [K+1]
    std::vector<int32_t> gid;      // [Np]
    std::vector<int32_t> deg;      // [Np] local degree, self-loop excluded
    std::vector<int64_t> core_count;  // [K]
    bool symmetric = false;        // A~ equals its transpose entry by entry
    std::vector<int64_t> t_rowptr; // transposed store (t_col, t_val empty when symmetric or when values were not asked for)
    std::vector<int32_t> t_col;
    std::vector<float> t_val;
};

// Validates the inputs and fills the store; returns a GAD_* status and a message.
int build_store(const gad_csr* g, const gad_partition* part, bool values, HostStore& out, std::string& err);
// Sizes only (for gad_workspace_bytes): rows, entries, and the SpMM scratch slots of the worse orientation.
int store_sizes(const gad_csr* g, const gad_partition* part, int64_t* Np, int64_t* nnz, int64_t* slots, std::string& err);

// Work lists of the SpMM launch (host side).  A row of at most `part_entries` entries is one item; a longer row is
// cut into parts of `part_entries` entries, each an item with a scratch slot of its own, and gets an entry
// fin = {row, first scratch slot, slots, subgraph of the row}.  The part length starts at kMinPart, or at a quarter of the
// entries an average resident warp gets if that is more, and doubles (up to kMaxPart) until the cut rows need at most one
// scratch slot per two store rows; a row that would still need more than kMaxSlotsPerRow parts gets longer parts of its own.
// items = {row, low 32 bits of the first entry's position in the store, (high bits << 16) | entries, scratch slot
// or -1 for an uncut row}, subgraph by subgraph and inside a subgraph binned by floor(log2(entries)), longest bin
// first, ascending row inside a bin.  `perm` (uncut rows in that order) and `parts` are the intermediate lists the
// items are built from.  runs = the same items, those of some subgraphs binned inside runs of kItemWindow rows (no such subgraph: empty).
constexpr int64_t kMinPart = 64, kMaxPart = 8192, kMaxSlotsPerRow = 32;
// Neighbouring rows of a graph that is numbered by community, time or site gather the same operand rows.  Ordered by length over a whole
// subgraph the resident warps (9472) spread over all of it, and where its operand does not fit the L2 (126 MB) beside what else passes, those rows come
// from HBM again and again; in runs they do not.  Epochs of 4 x 131 000 rows of 34 entries, 256 wide: 6100 us without runs, 5995 with
// runs of 65 536 rows, 5915 of 32 768, 5900 of 16 384, 5900 of 4096.  A run ends on short items beside the long ones of the next, which costs every launch.
// So runs serve launches whose operand takes half of the L2 and more, in subgraphs a good third of whose entries read a row less than a run away (those between
// two replicated nodes aside: their rows are few and stay in the L2 in any order).  us without / with, by rows of a subgraph, columns and that share:
//   both: 131 000, 256 (134 MB), 0.75 1258 / 1171 and 1230 / 1144; 157 000, 0.71, 128 (81 MB) 351 / 335, 192 (121 MB) 581 / 532, 384 and 512 (242, 323 MB)
//     572 / 530; 210 000, 256 (215 MB), 0.42 1596 / 1520 and 1583 / 1496, 100 (84 MB) 737 / 718; 79 000, 256 (81 MB), 0.37 822 / 812 and 823 / 803;
//     bfloat16, 131 000, 256 (67 MB), 0.75 834 / 802 and 764 / 730;
//   smaller operands: 131 000, 0.75, 100 (52 MB) 586 / 602; bfloat16, 131 000, 0.75, 100 (26 MB) 453 / 475, 210 000, 0.42, 100 (42 MB) 377 / 369; and the kernels
//     of up to 64 columns, whose warps have two to eight items each: 157 000, 0.71, 8 101 / 122 and 64 / 74, 64 233 / 237, 131 000, 47 438 / 473 and 222 / 253;
//   fewer near: 16 x 161 000, 256 (165 MB), 0.16 to 0.32 6200 / 6260 and 5990 / 6070; 131 000, 256, 0.25 1300 / 1320 and 1271 / 1290; 157 000, 0.21, 128 356 / 360,
//     192 591 / 595; bfloat16, 131 000, 256, 0.25 833 / 852 and 762 / 767.
constexpr int64_t kItemWindow = 16384, kRunOperandBytes = 63 << 20;
constexpr double kRunNearShare = 0.35;
struct RowWork {
    std::vector<int32_t> perm;
    std::vector<int4> parts, fin, items, runs;
    int64_t slots = 0, part_entries = kMinPart;
};
int64_t part_entries_for(const std::vector<int64_t>& rowptr);
// forced_part > 0: cut rows into parts of that many entries instead of the length part_entries_for would choose.  by_runs [K]: subgraphs of `runs` cut into runs.
void bin_rows(const std::vector<int64_t>& rowptr, const std::vector<int32_t>& sub_off, RowWork& out, int64_t forced_part, const std::vector<uint8_t>& by_runs);
// Scratch slots bin_rows would use, from the row lengths alone.
int64_t count_slots(const std::vector<int64_t>& rowptr);

// ---------------------------------------------------------------------------------------------
// Device views
// ---------------------------------------------------------------------------------------------
struct SparseDev {
    const int64_t* rowptr = nullptr;  // [Np+1] (kept for the accessors; the kernels read the work list)
    const uint2* ecv = nullptr;       // [nnz] packed (column, value bits)
    const int4* fin = nullptr;        // rows made of several parts
    const int4* items = nullptr;      // parts and uncut rows together, longest first inside a subgraph
    const int4* runs = nullptr;       // the same, longest first inside a run of rows where a subgraph gains by it; or null
    int64_t run_rows = 0;             // rows of the smallest of those subgraphs
    float* scratch = nullptr;         // [slots x leading dimension of the output] partial rows
    int32_t nfin = 0, nitems = 0;
    int64_t nrows = 0, nnz = 0;       // rows (and columns) of the store, its entries
};

struct Layer {
    int32_t fi, fo;        // F_l, F_{l+1}
    int32_t ldi, ldo;      // leading dimensions of H^(l), H^(l+1) (multiples of 4 floats)
    int32_t ldw;           // leading dimension of W_l rows inside the padded parameter block
    int64_t w_int, b_int;  // offsets inside one replica's padded parameter block (multiples of 4 floats)
    int64_t w_ext, b_ext;  // offsets inside the caller-visible [P] layout
};

// A run of rows that belongs to one subgraph: {first row, row count, subgraph, unused}.
struct RowSpan { int32_t row0, nrows, k, pad; };

struct Epilogue {            // of the forward SpMM: bias, ReLU, dropout
    const float* params;     // padded parameter blocks
    int64_t pstride;         // floats between replicas
    int64_t b_int;           // bias offset inside a block
    const int32_t* sub_off;  // [K+1]
    int32_t K;
    int32_t relu;            // 0 on the last layer
    float dropout;
    uint64_t seed;
    const long long* epoch;  // device counter that indexes the dropout mask (read only with dropout > 0)
    int32_t layer;
};

// What a finishing kernel gets: where the biases are and how ReLU / dropout apply on this layer and epoch.
struct ActEpi {
    const float* params;   // padded parameter blocks
    long long pstride;     // floats between replicas
    long long b_int;       // bias offset inside a block
    int relu;              // 0 on the last layer
    int drop;              // dropout is applied (rate > 0 on a layer with ReLU)
    uint32_t thr;          // keep an element when the top 24 bits of its hash reach this
    float scale;           // 1 / (1 - rate)
    unsigned long long seed;
    const long long* epoch;   // device counter of the epochs run so far
    int layer;
    int col0;              // column of the operand's first column (column slabs)
};
inline ActEpi make_act(const Epilogue& e, int col0) {
    ActEpi t{};
    t.params = e.params; t.pstride = e.pstride; t.b_int = e.b_int + col0;
    t.relu = e.relu; t.layer = e.layer;
    t.drop = e.dropout > 0.f && e.relu;
    t.thr = t.drop ? (uint32_t)std::floor((double)e.dropout * 16777216.0) : 0u;
    t.scale = t.drop ? 1.f / (1.f - e.dropout) : 1.f;
    t.seed = e.seed; t.epoch = e.epoch; t.col0 = col0;
    return t;
}

// ---------------------------------------------------------------------------------------------
// Kernel launchers (each enqueues on `s` and returns the cudaGetLastError of its launches)
// ---------------------------------------------------------------------------------------------
// bf16_scratch: null, or device room for nrows x ldz bfloat16 values: the operand is then copied there in bfloat16 and
// gathered from the copy (reduced-precision mode); with bf16_ready the copy is there already (written by the producer).
cudaError_t launch_spmm(const SparseDev& A, const float* Z, int ldz, float* out, int ldo, int F,
                        const Epilogue* epi, void* bf16_scratch, bool bf16_ready, cudaStream_t s);

// Tests every index of a device store and its work lists against its range (see check_store_kernel); bad[0] += violations,
// bad[1] = min(bad[1], first offending work-list position + 1).
cudaError_t launch_check_store(const SparseDev& A, long long nnz, long long slots, const int32_t* sub_off, int K, unsigned long long* bad,
                               cudaStream_t s);

// mode 0: C = A * W_k (W row-major [Kd x N], ld ldw); mode 1: C = (A * W_k^T) masked by Hmask > 0, scaled
// (W row-major [N x Kd]); mode 2: C = sigma(A * W_k + b_k) with dropout as `act` says.  Tiles never cross a subgraph.
cudaError_t launch_gemm_rows_simt(int mode, const float* A, int lda, int Kd, const float* params, int64_t pstride,
                                  int64_t w_int, int ldw, int N, float* C, int ldc, const RowSpan* tiles,
                                  int ntiles, const float* Hmask, int ldh, float scale, const ActEpi* act, cudaStream_t s);

// Tensor-core (tcgen05) version of launch_gemm_rows_simt.  The operands come through TMA descriptors made by
// tc_make_map (A: [rows x Kd]; B, B_lo: [K][N][Kd] copies written by launch_split_weights); passes = 3 gives fp32
// accuracy by operand splitting, passes = 1 plain TF32 operands.  err receives a role code if a bounded wait runs out.
int tc_rows_bn(int n_cols, int npairs, int Kd, bool drop);   // columns per tile of a forward transform in three passes (drop: with dropout in its epilogue)
int tc_rows_bn_whole(int n_cols, int npairs);                // of the others
int tc_tn_rows();   // rows of the row-box descriptors the weight-gradient kernel reads (mapH / mapZ of launch_gemm_tn_tc)
bool tc_make_map(void* out_map, const void* base, uint64_t inner, uint64_t rows, uint64_t outer, uint64_t row_stride_bytes,
                 uint64_t outer_stride_bytes, uint32_t box_rows, bool mn_major = false, bool half = false);
struct SplitLayer {
    int fi, fo, ldw, ldkt;
    long long w_int;
    float *w_hi, *w_lo, *wt_hi, *wt_lo;   // w_hi, w_lo: null where no kernel reads the plain copies
};
struct SplitLayers {
    static constexpr int MAX = 8;
    SplitLayer y[MAX];
};
cudaError_t launch_split_weights(const float* params, int64_t pstride, int K, const SplitLayer* layers, int L, cudaStream_t s);
// pair_tiles: 2 npairs row tiles (at most 128 rows, or none), the two of a pair in the same subgraph; bn (tc_rows_bn, tc_rows_bn_whole) columns
// per tile, half of them the rows of B's descriptor box.  bits: with mode 0 (may be null) the transform leaves there which values of A are above
// zero, bit c % 32 of word c / 32 of a row of bit_words words; mode 1 masks with such bits (null: no mask), 1/32 of the bytes of the activations.  one_b: the operand copies of replica 0 serve every subgraph.
// Cbf16 (mode 0, or 1 with a mask; may be null): the result goes there as bfloat16 [rows x ldc] INSTEAD of to C - the operand copy the
// reduced-precision aggregation gathers, written by its producer.  colsum (mode 1 with a mask, where tc_rows_sums_columns): the
// column sums of the result, for launch_colsum_finish.
cudaError_t launch_gemm_rows_tc(const void* mapA, const void* mapB, const void* mapBlo, int mode, int passes, int Kd, int n_cols, int bn,
                                float* C, int ldc, const RowSpan* pair_tiles, int npairs, uint32_t* bits, int bit_words, float scale,
                                const ActEpi* act, int32_t* err, int num_sms, cudaStream_t s, bool one_b, void* Cbf16 = nullptr, float* colsum = nullptr);
inline int32_t bit_words_of(int32_t ld) { return (ld + 31) / 32; }
bool tc_rows_sums_columns(int n_cols, int npairs);
constexpr int kMaxRowClusters = 128;
int tc_rows_clusters(long long ntiles, int num_sms);   // clusters of a launch: cluster c takes tiles [ntiles c / n, ntiles (c + 1) / n)

// Tensor-core version of launch_gemm_tn_simt; mapH / mapZ are row-box descriptors (tc_tn_rows rows) of H^(l) and dZ.
struct TnShape { int cg, ntm, ntn, bn; };   // CTAs per work unit, output tiles (of 128 cg rows and bn columns)
TnShape tn_shape(int fi, int ldw);
int64_t tn_chunk_rows(const std::vector<int32_t>& sub_off, const TnShape& t, int fi, int ldw, int num_sms);
cudaError_t launch_gemm_tn_tc(const void* mapH, const void* mapZ, int passes, int M, int ldw, const RowSpan* chunks, int nchunks, float* partial,
                              int32_t* err, int num_sms, cudaStream_t s);

// Backward transforms of a layer with at most 16 output columns as one stream on the FP32 ALUs (narrow.cu).  `chunks`
// are runs of rows of one subgraph, one CTA each.  In one pass over H and dZ: dPre = (dZ W_k^T) masked by H > 0, times
// `scale`, and partial[chunk] = [column sums of those dPre rows (ldh floats)] [H[chunk rows]^T dZ[chunk rows] (fi x ldw)],
// to be added per subgraph by launch_reduce_chunks (the bias of a layer lies right before the weights of the next).  H and dZ must be contiguous (leading dimension = row length).  err receives 90 if a bounded wait runs out.
bool narrow_supported(int ldi, int ldo);
cudaError_t launch_narrow_bwd(const float* H, int ldh, int fi, const float* dZ, int ldz, const float* params, int64_t pstride,
                              int64_t w_int, int ldw, const RowSpan* chunks, int nchunks, float scale, float* dPre, float* partial,
                              int64_t partial_stride, int32_t* err, cudaStream_t s);

// partial[chunk] = H[chunk rows]^T * dZ[chunk rows]   ([M x ldw] each), one CTA column per chunk.  small_chunks: they are of
// simt_tn_chunk_rows.
int64_t simt_tn_chunk_rows(int64_t rows, int fi, int ldw);
cudaError_t launch_gemm_tn_simt(const float* H, int ldh, int M, const float* dZ, int ldz, int N,
                                const RowSpan* chunks, int nchunks, bool small_chunks, float* partial, int ldw, cudaStream_t s);

// out[k][off + i] = sum over the chunks of subgraph k, in chunk order, of partial[chunk][i], i < len.
cudaError_t launch_reduce_chunks(const float* partial, int64_t pstride_chunk, const int32_t* chunk_ptr, int K,
                                 float* out, int64_t ostride, int64_t off, int64_t len, cudaStream_t s);

// out[k][off + j] = sum over the rows of subgraph k of G[row][j], j < ld.  A single kernel whose last-arriving CTA of a subgraph
// adds the chunk sums in chunk order; counters: one per subgraph, monotonic, zero at creation.
cudaError_t launch_colsum_chunks(const float* G, int ld, const RowSpan* chunks, int nchunks, float* partial,
                                 int64_t pstride_chunk, const int32_t* chunk_ptr, unsigned* counters, float* out,
                                 int64_t ostride, int64_t off, cudaStream_t s);

// out[k][off + j] = sum over the clusters first[k] .. last[k] that had tiles of subgraph k, and their eight row groups, of the column sums
// a transform's drain has left (first > last: no rows).
cudaError_t launch_colsum_finish(const float* colsum, int ld, const int2* clusters, int K, float* out, int64_t ostride, int64_t off, cudaStream_t s);

// dlogits and per chunk the loss, and where softmax_sums_columns(ld) holds the column sums of dlogits (cs_partial); there dlogits_bf16 (may
// be null) receives dlogits in bfloat16 instead.
bool softmax_sums_columns(int ld);
cudaError_t launch_softmax_xent(const float* logits, int ld, int C, const int32_t* label, const uint8_t* train,
                                const RowSpan* chunks, int nchunks, const float* inv_ntrain, float* dlogits,
                                float* loss_partial, float* cs_partial, int64_t pstride_chunk, void* dlogits_bf16, cudaStream_t s);
// loss[0..K-1] = mean loss of each subgraph, loss[K] = mean over all training rows, and with bias_ld > 0 out[k][off + j] = sum of
// the column sums of subgraph k's chunks, j < bias_ld.
cudaError_t launch_loss_finish(const float* loss_partial, const float* inv_ntrain, const int32_t* chunk_ptr, int K, float inv_total, float* loss,
                               int32_t* nonfinite, const float* bias_partial, int64_t pstride_chunk, int bias_ld, float* out, int64_t ostride,
                               int64_t off, cudaStream_t s);

// zeta[k] of every subgraph that has rows.  phase 0: from the matrix X alone; phases 1, 2, 3: X is the first, a further, the last
// of several matrices whose squared distances add up (q_acc: one double per subgraph).
cudaError_t launch_zeta(const float* X, int ld, int F, const int32_t* deg, const RowSpan* chunks, int nchunks,
                        const int32_t* chunk_ptr, const int32_t* sub_off, int K, const int64_t* deg_sum, const int64_t* deg_sq,
                        float beta, double* partial, double* zeta, double* q_acc, int phase, cudaStream_t s);

// zeta_k in the literal pairwise form, sum_{i<j} p_i p_j / (|x_i - x_j| + beta), 64 x 64 tiles of pairs (one CTA each,
// pair_ptr[k] = first tile of subgraph k); counters: one per subgraph; partial: one double per tile.
constexpr int64_t kZetaPairMaxRows = 32768;
int64_t zeta_pair_tiles(int64_t rows);
cudaError_t launch_zeta_pair(const float* X, int ld, int F, const int32_t* deg, const int32_t* sub_off, const int64_t* deg_sum,
                             const int64_t* pair_ptr, int64_t npairs, int K, float beta, double* partial, unsigned* counters,
                             double* zeta, cudaStream_t s);

// `err_word` (may be null): when a kernel of the epoch has reported a bounded wait that ran out, the gradients are not to
// be trusted and the three consensus kernels leave the parameters (and `out`) untouched.
// The same zeta_k with the squared distances from a Gram matrix on the tensor cores (zeta_gram.cu): tiles of 256 x 256 pairs,
// tile_ptr[k] = first tile of subgraph k, any subgraph size.  Xhi, Xlo: [rows x ldh] fp16 values each, ldh = F rounded up to 8 (split of the scaled rows of X, written
// by the call; mapHi / mapLo are their descriptors, boxes of zeta_gram_box_rows rows); norm2: [rows] squared norms and scales; partial: zeta_gram_partials doubles.
constexpr int kGramMaxCtas = 256;
int64_t zeta_gram_tiles(int64_t rows);
int64_t zeta_gram_partials(int num_ctas, int K);
uint32_t zeta_gram_box_rows();
cudaError_t launch_zeta_gram(const void* mapHi, const void* mapLo, const float* X, int ld, int F, long long rows, const int32_t* deg,
                             const int32_t* sub_off, const int64_t* deg_sum, const int64_t* tile_ptr, int64_t ntiles, int K, float beta,
                             void* Xhi, void* Xlo, float2* norm2, double* partial, double* zeta, int32_t* err, int num_sms, cudaStream_t s);

// `epoch` (may be null): the device epoch counter, advanced by one.
// pstride_p: floats between the replicas' parameters, 0 while they are equal (copy 0 then stands for all of them; the result always
// goes to copy 0).  report_to (may be null): pinned host memory that receives the nreport words at `report`.  words: the context's error words {non-finite loss, wait that ran out, copies differ}.
cudaError_t launch_sgd_consensus(float* params, int64_t pstride_p, const float* grads, int64_t pstride, int64_t len, int K, float lr,
                                 const double* zeta, int weighted, int with_sgd, int32_t* words, long long* epoch, const float* report, float* report_to,
                                 int nreport, cudaStream_t s);
// The same with a step where the gradients of the parameters [4 first4, 4 (first4 + count4)) have yet to be added up, chunk by chunk in order; they are written
// to grads.  For at most kStepSumsFloats parameters, kStepSumsReplicas replicas and kStepSumsChunks chunks in each: a warp reads a replica's chunks eight at a
// time, one after the other.  1750 nets of up to 262 144 parameters and 48 000 rows, mean change of an epoch against a kernel of its own by the most chunks
// a replica has: up to 8 -3.8 us, 16 -2.6, 24 -1.4, 32 -2.2, 64 0 (more than 64 000 parameters less: 1509 rows of 225-493-13, 47 chunks, 142 -> 126), 72 +3.4, 100 and more
// +10 (23 700 rows of 27-129-13 in one subgraph: 127 -> 140).  At the limit of parameters (2700 to 42 000 rows, 2 to 50 replicas of 0.23 to 0.26 M) 0 to 10 us less.
struct ChunkSums { long long first4, count4; const float4* partial; long long stride4; const int32_t* chunk_ptr; };
constexpr int64_t kStepSumsFloats = 256 << 10, kStepSumsReplicas = 4096, kStepSumsChunks = 64;
cudaError_t launch_step_sums_consensus(float* params, int64_t pstride_p, float* grads, int64_t pstride, int64_t len, int K, float lr, const double* zeta,
                                       int weighted, int32_t* words, long long* epoch, const float* report, float* report_to, int nreport,
                                       const ChunkSums& sums, cudaStream_t s);
// The device epoch counter on its own: + 1, or set to a value.
cudaError_t launch_epoch_counter(long long* epoch, long long set_to, bool advance, cudaStream_t s);
// One context's share of a consensus over several contexts: out = sum_k w_k (theta_k - lr grad_k) with w_k = zeta_k / total
// (or 1 / total), the parameters unchanged; and the finished sum written to every replica.
cudaError_t launch_consensus_partial(const float* params, int64_t pstride_p, const float* grads, int64_t pstride, int64_t len, int K, float lr,
                                     const double* zeta, int weighted, int with_sgd, double total, float* out, const int32_t* err_word, cudaStream_t s);
cudaError_t launch_consensus_apply(float* params, int64_t len, const float* in, int32_t* words, cudaStream_t s);

// One CTA waits, with the transforms' bounded wait and a limit of `polls` polls, on a barrier that nothing arrives at, and
// reports it in `err` like a transform would (role 99).  For testing the time-out path; returns at once.
cudaError_t launch_expire_wait(int32_t* err, uint32_t polls, cudaStream_t s);
cudaError_t launch_weights(const double* zeta, int K, int weighted, float* zeta_f, float* w_f, cudaStream_t s);

// G[r][c] = H[r][c] > 0 ? G[r][c] * scale : 0 over rows x ld values (the ReLU and dropout scale of the layer below, applied
// to an input gradient that was aggregated after its transform).
cudaError_t launch_relu_mask(float* G, const float* H, int ld, int64_t rows, float scale, cudaStream_t s);

cudaError_t launch_gather_rows(const float* Xg, int F, const int32_t* gid, int64_t Np, float* H0, int ld, void* bf16_copy,
                               cudaStream_t s);
cudaError_t launch_gather_labels(const int32_t* yg, const int32_t* gid, int64_t Np, int32_t* label, cudaStream_t s);
cudaError_t launch_scatter_core(const float* logits, int ld, int C, const int32_t* gid, const RowSpan* core_spans,
                                int nspans, float* out, cudaStream_t s);

// host_copy.cu: `bytes` of device memory into the caller's memory through pinned slots, complete on return; the pages of
// a pageable destination touched ahead of it, their contents kept; contexts that may copy, + 1 / - 1.
cudaError_t copy_to_host(void* dst, const void* src, size_t bytes, cudaStream_t s);
void host_prefault(void* dst, size_t bytes);
void host_copy_user(int delta);
struct Pinned { char* p = nullptr; size_t bytes = 0; unsigned long long id = 0; };
Pinned take_small_pinned(size_t bytes);   // p null: none to be had
void give_small_pinned(const Pinned& m);
void release_pinned();   // frees the pinned memory that lies idle

}  // namespace gad
