// Importance-based subgraph augmentation (Algorithm 1 of the paper, Section 3.2.2): for every subgraph of a
// partition, Monte-Carlo random walks from its boundary nodes estimate how often each outside node is reached
// (importance equation), the number of walks follows the Monte-Carlo error equation, and the replication nodes are
// taken walk by walk in descending order of the walks' summed importance until the density-sized number n(g_i) is
// reached.  Its output (the replication-node lists) is what gad_create takes as `halo_nodes`.
//
// On the GPU, for all subgraphs of a batch at once: the boundary test and list, the walks with their visit counts, the count
// statistics and the number of walks that follows from them, the walk scores and the leading walks in rank order, in integers
// but for the two formulas, whose operations are rounded one by one (the same draws, counts and scores as a CPU evaluation:
// every random number is a pure function mix(seed, subgraph, walk, step) of the splitmix64 output function).  On the host: the selection loop over the leading walks, which is
// sequential by definition.  What bounds it is latency, of launches and of dependent random reads: one subgraph after the
// other with four host waits each took 5.1 ms for 8 subgraphs of 12 500 nodes, one batch with one wait takes 0.43 ms.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <numeric>
#include <string>
#include <vector>

#include "gad_internal.h"

namespace gad {

namespace {

constexpr int kMaxSteps = 8;

__host__ __device__ inline uint64_t aug_mix64(uint64_t z) {
    z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ULL;
    z = (z ^ (z >> 27)) * 0x94d049bb133111ebULL;
    return z ^ (z >> 31);
}
// key of (seed, subgraph, walk); the step is mixed in per draw
__host__ __device__ inline uint64_t walk_key(uint64_t seed, int sub, int64_t walk) {
    const uint64_t G = 0x9e3779b97f4a7c15ULL;
    const uint64_t h = aug_mix64(seed + G * (uint64_t)(1 + sub));
    return aug_mix64(h + G * (uint64_t)(1 + walk));
}
__host__ __device__ inline uint64_t walk_draw(uint64_t key, int step) {
    const uint64_t G = 0x9e3779b97f4a7c15ULL;
    return aug_mix64(key + G * (uint64_t)(1 + step));
}
// A node as a walk wants it: where its row of the graph begins and how long it is (33 and 31 bits), and the reciprocal of that length.
struct __align__(16) WalkNode { unsigned long long row, recip; };
constexpr int kLenBits = 31;
constexpr int64_t kMaxPackedEntries = 1ll << (64 - kLenBits), kMaxPackedRow = 1ll << kLenBits;   // both exclusive
// x mod d by m = floor((2^64 - 1) / d): x m / 2^64 lies less than one below x / d, so that the quotient is right or one too small.
__device__ __forceinline__ unsigned long long reciprocal(unsigned long long d) { return d > 0 ? ~0ull / d : 0ull; }
__device__ __forceinline__ unsigned long long mod_by(unsigned long long x, unsigned long long d, unsigned long long m) {
    const unsigned long long r = x - __umul64hi(x, m) * d;
    return r >= d ? r - d : r;
}
__device__ __forceinline__ WalkNode walk_node(const int64_t* rowptr, int64_t v) {
    const unsigned long long r0 = (unsigned long long)rowptr[v], d = (unsigned long long)rowptr[v + 1] - r0;
    return {r0 << kLenBits | d, reciprocal(d)};
}

// The node sequence of one walk: start at a uniformly drawn boundary node, every step to a uniformly drawn neighbour.
__host__ __device__ inline void make_walk(const int64_t* rowptr, const int32_t* col, const int32_t* B, int64_t nB, uint64_t seed, int sub,
                                          int64_t walk, int steps, int32_t* seq) {
    const uint64_t key = walk_key(seed, sub, walk);
    int32_t cur = B[walk_draw(key, 0) % (uint64_t)nB];
    seq[0] = cur;
    for (int s = 1; s <= steps; ++s) {
        const int64_t r0 = rowptr[cur], d = rowptr[cur + 1] - r0;
        if (d > 0) cur = col[r0 + (int64_t)(walk_draw(key, s) % (uint64_t)d)];
        seq[s] = cur;
    }
}
// v is outside the subgraph and does not occur earlier in the walk
__host__ __device__ inline bool first_outside(const uint8_t* inside, const int32_t* seq, int s) {
    const int32_t v = seq[s];
    if (inside[v]) return false;
    for (int t = 0; t < s; ++t)
        if (seq[t] == v) return false;
    return true;
}

// One subgraph of a batch.  desc: what the host knows before the first kernel; state: what the kernels find out.
struct SubDesc {
    int64_t core0, ncore;   // its part of the batch's core list
    int64_t key0;           // first ranking key
    int64_t top0, top_cap;  // first row, and rows, of the leading walks' sequences; the buffer of gathered keys is kTopSlack times that
    int64_t max_walks;      // there is room for: cap times the core set's degree sum, which no count of walks exceeds on the same graph
    int32_t sub, pad;       // number of the subgraph: its random stream
};
struct SubState {
    unsigned long long inner;                 // directed entries between two different core nodes (2 |e_i| of the density definition)
    unsigned long long n0;                    // walks of the first batch: degree sum of the boundary nodes
    unsigned long long m, s1, s2;             // visited candidates, sum of counts, sum of squared counts
    unsigned long long prefix, mask;          // key selection: digits fixed so far and their mask
    unsigned long long got;                   // keys gathered
    unsigned long long arrived;               // CTAs that have added their histogram
    long long nB, nwalks, n_rep, lead, remaining;
};
constexpr int kTopSlack = 2;


__global__ void __launch_bounds__(256) mark_kernel(const int32_t* __restrict__ core, const SubDesc* __restrict__ desc, uint8_t* __restrict__ inside, int64_t n,
                                                   const int64_t* __restrict__ rowptr, WalkNode* __restrict__ nodes) {
    if (nodes)
        for (int64_t v = ((int64_t)blockIdx.y * gridDim.x + blockIdx.x) * blockDim.x + threadIdx.x; v < n; v += (int64_t)gridDim.x * gridDim.y * blockDim.x) nodes[v] = walk_node(rowptr, v);
    const SubDesc d = desc[blockIdx.y];
    uint8_t* in = inside + (int64_t)blockIdx.y * n;
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < d.ncore; t += (int64_t)gridDim.x * blockDim.x) in[core[d.core0 + t]] = 1;
}

// A core node with a neighbour outside the core set is a boundary node.  One warp per core node; rows of more than kLongRow
// entries are set aside and then read by the whole CTA (one thread per node lasted as long as the longest row).  The flags
// go to a map of their own: set in the map that the other warps are reading, the stores alone took the kernel from 31 to 100 us.
constexpr int kLongRow = 256, kMaxLong = 256;
__global__ void __launch_bounds__(256) boundary_kernel(const int64_t* __restrict__ rowptr, const int32_t* __restrict__ col, const int32_t* __restrict__ core,
                                                       const SubDesc* __restrict__ desc, SubState* __restrict__ state, const uint8_t* __restrict__ inside, uint8_t* __restrict__ boundary, int64_t n) {
    __shared__ unsigned long long sum[8];
    __shared__ int32_t long_node[kMaxLong];
    __shared__ int nlong;
    const SubDesc d = desc[blockIdx.y];
    const uint8_t* in = inside + (int64_t)blockIdx.y * n;
    uint8_t* flag = boundary + (int64_t)blockIdx.y * n;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (threadIdx.x == 0) nlong = 0;
    __syncthreads();
    unsigned long long inner = 0;
    const int64_t step = (int64_t)gridDim.x * 8;
    int32_t next = -1;
    int64_t t = (int64_t)blockIdx.x * 8 + warp;
    if (t < d.ncore) next = core[d.core0 + t];
    for (; t < d.ncore; t += step) {
        const int32_t v = next;
        if (t + step < d.ncore) next = core[d.core0 + t + step];
        const int64_t e0 = rowptr[v];
        const int64_t len = rowptr[v + 1] - e0;
        if (len > kLongRow) {
            int at = kMaxLong;
            if (lane == 0) at = atomicAdd(&nlong, 1);
            at = __shfl_sync(0xffffffffu, at, 0);
            if (at < kMaxLong) {
                if (lane == 0) long_node[at] = v;
                continue;
            }   // no room: read here
        }
        bool out = false;
        int mine = 0;
        for (int64_t o = lane; o < len; o += 32) {
            const int32_t c = col[e0 + o];
            const bool i = in[c] != 0;
            out |= !i;
            mine += i && c != v;
        }
        inner += mine;
        if (__any_sync(0xffffffffu, out) && lane == 0) flag[v] = 1;
    }
    __syncthreads();
    const int nl = min(nlong, kMaxLong);
    for (int w = 0; w < nl; ++w) {
        const int32_t v = long_node[w];
        const int64_t e0 = rowptr[v], e1 = rowptr[v + 1];
        int out = 0, mine = 0;
        for (int64_t e = e0 + threadIdx.x; e < e1; e += 1024) {   // four entries in flight per thread
            int32_t c[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) c[u] = e + 256 * u < e1 ? col[e + 256 * u] : v;   // (v itself: inside, and not counted)
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const bool i = in[c[u]] != 0;
                out |= !i;
                mine += i && c[u] != v;
            }
        }
        inner += mine;
        if (__syncthreads_or(out) && threadIdx.x == 0) flag[v] = 1;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) inner += __shfl_xor_sync(0xffffffffu, inner, o);
    if (lane == 0) sum[warp] = inner;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < 8; ++w) inner += sum[w];
        if (inner) atomicAdd(&state[blockIdx.y].inner, inner);
    }
}

// The boundary nodes in ascending node id: per tile of kTile nodes a count, then every tile adds up the counts before it and
// writes its own.
constexpr int kTile = 2048;
__device__ __forceinline__ unsigned long long boundary_bits(const uint8_t* flag, int64_t v0, int64_t n) {
    unsigned long long bits = 0;   // byte i: node v0 + i is a boundary node
    if (v0 + 8 <= n && ((uintptr_t)(flag + v0) & 7) == 0) bits = *reinterpret_cast<const unsigned long long*>(flag + v0);
    else
        for (int i = 0; i < 8; ++i)
            if (v0 + i < n && flag[v0 + i]) bits |= 1ull << (8 * i);
    return bits;
}
__global__ void __launch_bounds__(256) boundary_count_kernel(const uint8_t* __restrict__ boundary, int64_t n, int ntiles, int32_t* __restrict__ tile_count) {
    __shared__ int total;
    if (threadIdx.x == 0) total = 0;
    __syncthreads();
    const unsigned long long bits = boundary_bits(boundary + (int64_t)blockIdx.y * n, (int64_t)blockIdx.x * kTile + threadIdx.x * 8, n);
    int c = __popcll(bits);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
    if ((threadIdx.x & 31) == 0 && c) atomicAdd(&total, c);
    __syncthreads();
    if (threadIdx.x == 0) tile_count[(int64_t)blockIdx.y * ntiles + blockIdx.x] = total;
}
__global__ void __launch_bounds__(256) boundary_list_kernel(const uint8_t* __restrict__ boundary, int64_t n, int ntiles, const int32_t* __restrict__ tile_count,
                                                            const int64_t* __restrict__ rowptr, const SubDesc* __restrict__ desc,
                                                            SubState* __restrict__ state, int32_t* __restrict__ B, WalkNode* __restrict__ Bnodes) {
    __shared__ int warp_sum[8];
    __shared__ int before;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int32_t* tc = tile_count + (int64_t)blockIdx.y * ntiles;
    if (threadIdx.x == 0) before = 0;
    __syncthreads();
    int c = 0;
    for (int t = threadIdx.x; t < (int)blockIdx.x; t += 256) c += tc[t];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
    if (lane == 0 && c) atomicAdd(&before, c);
    const int64_t v0 = (int64_t)blockIdx.x * kTile + threadIdx.x * 8;
    unsigned long long bits = boundary_bits(boundary + (int64_t)blockIdx.y * n, v0, n);
    const int mine = __popcll(bits);
    int incl = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) { const int u = __shfl_up_sync(0xffffffffu, incl, o); if (lane >= o) incl += u; }
    if (lane == 31) warp_sum[warp] = incl;
    __syncthreads();
    int at = before + incl - mine;
    for (int w = 0; w < warp; ++w) at += warp_sum[w];
    int32_t* out = B + desc[blockIdx.y].core0;
    unsigned long long deg = 0;
    while (bits) {
        const int i = (__ffsll((long long)bits) - 1) >> 3;
        bits &= bits - 1;
        const int64_t v = v0 + i;
        out[at] = (int32_t)v;
        if (Bnodes) Bnodes[desc[blockIdx.y].core0 + at] = walk_node(rowptr, v);
        ++at;
        deg += (unsigned long long)(rowptr[v + 1] - rowptr[v]);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) deg += __shfl_xor_sync(0xffffffffu, deg, o);
    if (lane == 0 && deg) atomicAdd(&state[blockIdx.y].n0, deg);
    if (blockIdx.x == gridDim.x - 1 && threadIdx.x == 255) state[blockIdx.y].nB = at;
}

// Walks [0, n0) (extra == 0) or [n0, nwalks) (extra == 1) of every subgraph of the batch, their candidates counted and kept:
// node[t][walk] is the node of step t, or -1 where it is inside the core set or occurred before.  (The scoring kernel reads them
// back in 10 us where drawing the walks again took it 69.)
// What bounds it is the number of lines that the lanes of a warp touch, each its own: 1.9 M walks of two steps made fourteen such reads each (two
// row ends a node) and three 64-bit remainders by the division routine, 82 us.  PACKED: one 16-byte read gives
// a node's row and the reciprocal for the remainder, for the first node in place of its number; and the first node, one of the core set, is not looked up.
// PACKED: where every row fits a WalkNode (walks_pack).
template <bool PACKED>
__global__ void __launch_bounds__(256) walk_count_kernel(const int64_t* __restrict__ rowptr, const int32_t* __restrict__ col, const int32_t* __restrict__ B,
                                                         const WalkNode* __restrict__ nodes, const WalkNode* __restrict__ Bnodes,
                                                         const uint8_t* __restrict__ inside, int64_t n, const SubDesc* __restrict__ desc,
                                                         const SubState* __restrict__ state, uint64_t seed, int extra, int steps,
                                                         int32_t* __restrict__ count, int32_t* __restrict__ node, int64_t plane) {
    const SubDesc d = desc[blockIdx.y];
    const SubState& s = state[blockIdx.y];
    const int64_t nB = s.nB, j1 = extra ? s.nwalks : min((int64_t)s.n0, d.max_walks);
    const uint8_t* in = inside + (int64_t)blockIdx.y * n;
    int32_t* cnt = count + (int64_t)blockIdx.y * n;
    const unsigned long long rB = reciprocal((unsigned long long)nB);
    int32_t seq[kMaxSteps + 1];
    for (int64_t j = (extra ? (int64_t)s.n0 : 0) + (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < j1; j += (int64_t)gridDim.x * blockDim.x) {
        if constexpr (PACKED) {
            const uint64_t key = walk_key(seed, d.sub, j);
            const int64_t b = d.core0 + (int64_t)mod_by(walk_draw(key, 0), (unsigned long long)nB, rB);
            WalkNode w = Bnodes[b];
            seq[0] = -1;   // (inside, and so is whatever equals it)
            node[d.key0 + j] = -1;
            for (int t = 1; t <= steps; ++t) {
                const unsigned long long deg = w.row & ((1ull << kLenBits) - 1);
                const int32_t v = deg > 0 ? col[(int64_t)(w.row >> kLenBits) + (int64_t)mod_by(walk_draw(key, t), deg, w.recip)] : t == 1 ? B[b] : seq[t - 1];
                seq[t] = v;
                if (t < steps) w = nodes[v];
                bool f = in[v] == 0;
                for (int u = 1; u < t; ++u) f = f && seq[u] != v;
                if (f) atomicAdd(cnt + v, 1);   // integer: the result does not depend on the order
                node[t * plane + d.key0 + j] = f ? v : -1;
            }
        } else {
            make_walk(rowptr, col, B + d.core0, nB, seed, d.sub, j, steps, seq);
            for (int t = 0; t <= steps; ++t) {
                const bool f = first_outside(in, seq, t);
                if (f) atomicAdd(cnt + seq[t], 1);
                node[t * plane + d.key0 + j] = f ? seq[t] : -1;
            }
        }
    }
}
// m, S1, S2 of the counts; with extra only where more walks were drawn.
__global__ void __launch_bounds__(256) count_stats_kernel(const int32_t* __restrict__ count, int64_t n, SubState* __restrict__ state, int extra) {
    SubState& st = state[blockIdx.y];
    if (extra && st.nwalks <= (long long)st.n0) return;
    const int32_t* cnt = count + (int64_t)blockIdx.y * n;
    unsigned long long m = 0, s1 = 0, s2 = 0;
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += (int64_t)gridDim.x * blockDim.x) {
        const unsigned long long c = (unsigned long long)cnt[v];
        if (c) { ++m; s1 += c; s2 += c * c; }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        m += __shfl_xor_sync(0xffffffffu, m, o); s1 += __shfl_xor_sync(0xffffffffu, s1, o); s2 += __shfl_xor_sync(0xffffffffu, s2, o);
    }
    if ((threadIdx.x & 31) == 0 && m) { atomicAdd(&st.m, m); atomicAdd(&st.s1, s1); atomicAdd(&st.s2, s2); }
}
// Number of walks from the Monte-Carlo error equation, sigma / mean of the visit frequencies from the integer sums.  Every
// operation is rounded on its own, as on the host.
__global__ void decide_walks_kernel(SubState* __restrict__ state, const SubDesc* __restrict__ desc, int G, double zc_over_E, int cap) {
    const int g = blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= G) return;
    SubState& s = state[g];
    const long long n0 = min((long long)s.n0, (long long)desc[g].max_walks);
    long long want = 0;
    if (s.m > 0) {
        const double ratio = __dadd_rn(__ddiv_rn(__dmul_rn((double)s.m, (double)s.s2), __dmul_rn((double)s.s1, (double)s.s1)), -1.0);
        if (ratio > 0.0) want = (long long)ceil(__dmul_rn(__dmul_rn(zc_over_E, zc_over_E), ratio));
    }
    const long long most = min((long long)cap * n0, (long long)desc[g].max_walks);
    s.nwalks = max(n0, min(want, most));
    if (s.nwalks > n0) { s.m = 0; s.s1 = 0; s.s2 = 0; }   // counted again over all walks
}
// n(g_i) = alpha (1 + d(g_i)) |v_i|, at most the visited candidates, and how many leading walks are ranked.
__global__ void decide_lead_kernel(SubState* __restrict__ state, const SubDesc* __restrict__ desc, int G, double alpha, int steps) {
    const int g = blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= G) return;
    SubState& s = state[g];
    const SubDesc d = desc[g];
    long long n_rep = 0;
    if (d.ncore >= 2) {
        const double dens = __ddiv_rn((double)(long long)s.inner, __dmul_rn((double)d.ncore, (double)(d.ncore - 1)));
        n_rep = (long long)floor(__dmul_rn(__dmul_rn(alpha, __dadd_rn(1.0, dens)), (double)d.ncore));
    }
    n_rep = min(n_rep, (long long)s.m);
    s.n_rep = n_rep;
    // a walk's score is at most (steps + 1) nwalks (a node counts once per walk): when score and walk index fit 32 bits each,
    // the walks get unique 64-bit ranking keys and the leading ones are selected on the device
    const bool keyed = s.nwalks > 0 && s.nwalks < (1ll << 32) && (long long)(steps + 1) * s.nwalks < (1ll << 31);
    s.lead = keyed && n_rep > 0 ? min(min(s.nwalks, max(1024ll, 8 * n_rep)), (long long)d.top_cap) : 0;
    s.remaining = s.lead;
}
// Ranking keys: a better walk (higher score; equal scores: lower index) has the larger key, and no two walks share one.
__global__ void __launch_bounds__(256) walk_key_kernel(int64_t n, const SubDesc* __restrict__ desc, const SubState* __restrict__ state, int steps,
                                                       const int32_t* __restrict__ count, const int32_t* __restrict__ node, int64_t plane,
                                                       unsigned long long* __restrict__ key, int raw_score) {
    const SubDesc d = desc[blockIdx.y];
    const SubState& s = state[blockIdx.y];
    if (!raw_score && s.lead == 0) return;
    const int64_t nwalks = s.nwalks;
    const int32_t* cnt = count + (int64_t)blockIdx.y * n;
    for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < nwalks; j += (int64_t)gridDim.x * blockDim.x) {
        int64_t sc = 0;
        for (int t = 0; t <= steps; ++t) {
            const int32_t v = node[t * plane + d.key0 + j];
            if (v >= 0) sc += cnt[v];
        }
        key[d.key0 + j] = raw_score ? (unsigned long long)sc : ((unsigned long long)sc << 32) | (unsigned long long)(0xFFFFFFFFu - (uint32_t)j);
    }
}

// Selection of the `lead` largest ranking keys without sorting them all: the keys are unique, so the lead-th largest one is
// found digit by digit (13 bits at a time, from the top), each pass a histogram of the next digit over the keys that share
// the digits fixed so far, until the keys not below the digits fixed so far fit the buffer of gathered keys (after one or two
// passes unless very many walks share a score).  A last pass gathers those; ranking them leaves out the ones past `lead`.
constexpr int kDigitBits = 13, kDigits = 1 << kDigitBits;
// One pass.  The CTA of a subgraph that arrives last fixes the digit in the state - the digit whose bin holds the key of rank
// `remaining`, counted from the largest digit down - and clears the histogram for the next pass; as a kernel of its own that
// step took another 9 us a pass.
__global__ void __launch_bounds__(1024) key_digit_kernel(const unsigned long long* __restrict__ key, const SubDesc* __restrict__ desc,
                                                         SubState* __restrict__ state, int shift, unsigned* __restrict__ hist_all) {
    __shared__ unsigned h[kDigits];
    __shared__ int warp_sum[32];
    __shared__ bool last;
    SubState& st = state[blockIdx.y];
    if (st.lead == 0 || st.remaining == 0) return;
    unsigned* hist = hist_all + (int64_t)blockIdx.y * kDigits;
    const unsigned long long prefix = st.prefix, mask = st.mask;
    const int64_t n = st.nwalks;
    const unsigned long long* k0 = key + desc[blockIdx.y].key0;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    for (int i = t; i < kDigits; i += 1024) h[i] = 0u;
    __syncthreads();
    for (int64_t j = (int64_t)blockIdx.x * 1024 + t; j < n; j += (int64_t)gridDim.x * 1024) {
        const unsigned long long k = k0[j];
        if ((k & mask) == prefix) atomicAdd(&h[(unsigned)(k >> shift) & (kDigits - 1)], 1u);
    }
    __syncthreads();
    for (int i = t; i < kDigits; i += 1024)
        if (h[i]) atomicAdd(hist + i, h[i]);
    __threadfence();
    __syncthreads();
    if (t == 0) last = (atomicAdd(&st.arrived, 1ull) + 1) % gridDim.x == 0;
    __syncthreads();
    if (!last) return;
    __threadfence();
    constexpr int PER = kDigits / 1024;   // thread t owns the bins kDigits-1 - PER t .. kDigits - PER (t + 1), largest first
    const long long remaining = st.remaining;
    unsigned mine[PER];
    int s = 0;   // (a subgraph with keys has fewer than 2^31 walks)
#pragma unroll
    for (int i = 0; i < PER; ++i) { mine[i] = __ldcg(hist + kDigits - 1 - (PER * t + i)); s += (int)mine[i]; }
    int incl = s;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) { const int u = __shfl_up_sync(0xffffffffu, incl, o); if (lane >= o) incl += u; }
    if (lane == 31) warp_sum[warp] = incl;
    __syncthreads();
    int w = warp_sum[lane];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) { const int u = __shfl_up_sync(0xffffffffu, w, o); if (lane >= o) w += u; }
    const int upto = __shfl_sync(0xffffffffu, w, warp > 0 ? warp - 1 : 0);
    const long long before = (long long)incl - s + (warp > 0 ? upto : 0);
    __syncthreads();   // every bin has been read
#pragma unroll
    for (int i = 0; i < PER; ++i) hist[PER * t + i] = 0u;
    if (before < remaining && remaining <= before + s) {   // exactly one thread: the bins are disjoint and ordered
        long long r = remaining - before;
        int i = 0;
        for (; i < PER - 1 && (long long)mine[i] < r; ++i) r -= mine[i];
        st.prefix = prefix | ((unsigned long long)(kDigits - 1 - (PER * t + i)) << shift);
        st.mask = mask | ((unsigned long long)(kDigits - 1) << shift);
        // keys at or above this digit: those ranked before it and its whole bin
        st.remaining = st.lead - r + (long long)mine[i] <= kTopSlack * desc[blockIdx.y].top_cap ? 0 : r;
    }
}
__global__ void __launch_bounds__(256) key_gather_kernel(const unsigned long long* __restrict__ key, const SubDesc* __restrict__ desc,
                                                         SubState* __restrict__ state, unsigned long long* __restrict__ top) {
    const SubDesc d = desc[blockIdx.y];
    SubState& s = state[blockIdx.y];
    if (s.lead == 0) return;
    const unsigned long long least = s.prefix;
    const int64_t n = s.nwalks;
    for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < n; j += (int64_t)gridDim.x * blockDim.x) {
        const unsigned long long k = key[d.key0 + j];
        if (k >= least) {
            const unsigned long long at = atomicAdd(&s.got, 1ull);   // ranked below: the order here is free
            if ((int64_t)at < kTopSlack * d.top_cap) top[kTopSlack * d.top0 + (int64_t)at] = k;
        }
    }
}
// The leading walks in rank order, as their candidate nodes: row r of `seq` is the walk of rank r, its nodes in walk order, -1
// where a node is inside the core set or occurred before.  A key's rank is the number of larger keys; four lanes share a key.
__global__ void __launch_bounds__(256) lead_walks_kernel(const SubDesc* __restrict__ desc, const SubState* __restrict__ state, int steps,
                                                         const int32_t* __restrict__ node, int64_t plane,
                                                         const unsigned long long* __restrict__ top, int32_t* __restrict__ seq_out) {
    __shared__ unsigned long long tile[1024];
    const SubDesc d = desc[blockIdx.y];
    const SubState& s = state[blockIdx.y];
    const int lead = (int)s.lead, got = (int)min((long long)s.got, kTopSlack * (long long)d.top_cap);
    const unsigned long long* keys = top + kTopSlack * d.top0;
    const int q = threadIdx.x & 3;
    for (int i0 = blockIdx.x * 64; i0 < got; i0 += gridDim.x * 64) {
        const int i = i0 + (threadIdx.x >> 2);
        const unsigned long long mine = i < got ? keys[i] : ~0ull;
        int rank = 0;
        for (int t0 = 0; t0 < got; t0 += 1024) {
            __syncthreads();
#pragma unroll
            for (int u = 0; u < 4; ++u) { const int t = t0 + 256 * u + (int)threadIdx.x; tile[256 * u + threadIdx.x] = t < got ? keys[t] : 0ull; }
            __syncthreads();
            const int m = min(1024, got - t0);
#pragma unroll 8
            for (int t = q; t < m; t += 4) rank += tile[t] > mine ? 1 : 0;
        }
        rank += __shfl_xor_sync(0xffffffffu, rank, 1);
        rank += __shfl_xor_sync(0xffffffffu, rank, 2);
        if (i < got && rank < lead) {
            const int64_t j = (int64_t)(0xFFFFFFFFu - (uint32_t)(mine & 0xFFFFFFFFull));
            for (int t = q; t <= steps; t += 4) seq_out[(d.top0 + rank) * (steps + 1) + t] = node[t * plane + d.key0 + j];
        }
    }
}

struct AugPlan {
    size_t o_rowptr, o_col, bytes;
    std::vector<int64_t> max_walks;          // [K] cap times the core set's degree sum: n0 is at most that sum
    std::vector<int32_t> first;              // subgraphs first[b] .. first[b + 1] - 1 form batch b
    bool packed = false;                     // walks_pack
};
// The buffers of one batch of G subgraphs, behind the graph in the workspace.
struct BatchLayout {
    size_t o_desc, o_nodes, o_Bnodes, o_core, o_B, o_tile, o_key, o_node, o_top, o_count, o_inside, o_bound, o_hist, o_state, o_seq, end;
    int64_t ncore, nkeys, ntop;
};
// Leading walks whose order is established first: the selection loop rarely needs more (it then orders all of them).
// n(g_i) <= alpha (1 + d) |v_i| <= 2 alpha |v_i|
inline int64_t leading_walks(int64_t max_walks, double alpha, int64_t ncore) {
    return std::min<int64_t>(max_walks, std::max<int64_t>(1024, 8 * (int64_t)std::floor(alpha * 2.0 * (double)ncore)));
}

size_t take(size_t& cur, size_t bytes) { size_t o = cur; cur += (size_t)round_up((int64_t)std::max<size_t>(bytes, 4), 256); return o; }

int num_tiles(int64_t n) { return (int)std::max<int64_t>(1, (n + kTile - 1) / kTile); }

BatchLayout batch_layout(const AugPlan& p, size_t base, int64_t n, const int64_t* core_ptr, int32_t k0, int32_t k1, double alpha, int steps) {
    BatchLayout b;
    const size_t G = (size_t)(k1 - k0);
    b.ncore = core_ptr[k1] - core_ptr[k0]; b.nkeys = 0; b.ntop = 0;
    for (int32_t k = k0; k < k1; ++k) {
        b.nkeys += p.max_walks[(size_t)k];
        b.ntop += leading_walks(p.max_walks[(size_t)k], alpha, core_ptr[k + 1] - core_ptr[k]);
    }
    size_t cur = base;
    b.o_desc = take(cur, sizeof(SubDesc) * G);
    b.o_nodes = take(cur, sizeof(WalkNode) * (size_t)n); b.o_Bnodes = take(cur, sizeof(WalkNode) * (size_t)b.ncore);
    b.o_core = take(cur, 4 * (size_t)b.ncore); b.o_B = take(cur, 4 * (size_t)b.ncore);
    b.o_tile = take(cur, 4 * G * (size_t)num_tiles(n));
    b.o_key = take(cur, 8 * (size_t)b.nkeys); b.o_node = take(cur, 4 * (size_t)b.nkeys * (size_t)(steps + 1)); b.o_top = take(cur, 8 * kTopSlack * (size_t)b.ntop);
    // cleared together for every batch ...
    b.o_count = take(cur, 4 * G * (size_t)n); b.o_inside = take(cur, G * (size_t)n); b.o_bound = take(cur, G * (size_t)n); b.o_hist = take(cur, 4 * G * (size_t)kDigits);
    b.o_state = take(cur, sizeof(SubState) * G);
    // ... and the state is read back together with the leading walks
    b.o_seq = take(cur, 4 * (size_t)b.ntop * (size_t)(steps + 1));
    b.end = cur;
    return b;
}

// Subgraphs are processed a batch at a time: their kernels share launches and the host waits once per batch.  A batch holds
// as many as fit these bounds (at least one): c2-sized graphs go through in one piece.
constexpr size_t kBatchNodeBytes = 256u << 20;    // visit counts, inside and boundary maps, 6 bytes per node and subgraph
constexpr int64_t kBatchWalkBytes = 1ll << 30;    // a ranking key (8 bytes) and steps + 1 nodes per walk

int check_columns(const gad_csr* g, std::string& err) {
    int bad = 0;
#pragma omp parallel for schedule(static) reduction(| : bad) if (g->nnz > (1 << 16))
    for (int64_t e = 0; e < g->nnz; ++e) bad |= g->col[e] < 0 || g->col[e] >= g->n;
    if (bad) { err = "column out of range"; return GAD_ERR_RANGE; }
    return GAD_OK;
}

// rowptr must not decrease.  lengths: the bits that occur in the rows' lengths (a negative one would bring the sign).
int check_rows(const gad_csr* g, int64_t& lengths, std::string& err) {
    int64_t bits = 0;
#pragma omp parallel for schedule(static) reduction(| : bits) if (g->n > (1 << 16))
    for (int32_t v = 0; v < g->n; ++v) bits |= g->rowptr[v + 1] - g->rowptr[v];
    lengths = bits;
    if (bits < 0) { err = "rowptr decreases"; return GAD_ERR_UNSORTED; }
    return GAD_OK;
}
// Every row's start and length fit a WalkNode.  (Columns may repeat, so that a row can be longer than there are nodes.)
bool walks_pack(int64_t nnz, int64_t lengths) { return nnz < kMaxPackedEntries && lengths < kMaxPackedRow; }

// `columns`: check them here; else the caller does (check_columns).
int plan_augment(const gad_csr* g, int32_t K, const int64_t* core_ptr, const int32_t* core_nodes, const gad_augment_config* cfg, AugPlan& p,
                 std::string& err, bool columns) {
    if (!g || !g->rowptr || (g->nnz > 0 && !g->col) || g->n < 0 || K < 1 || !core_ptr || !cfg) { err = "bad arguments"; return GAD_ERR_ARG; }
    if (cfg->steps < 1 || cfg->steps > kMaxSteps) { err = "steps must be 1 .. 8"; return GAD_ERR_ARG; }
    if (!(cfg->alpha >= 0.0) || !(cfg->E > 0.0) || !(cfg->zc > 0.0) || cfg->cap < 1) { err = "alpha >= 0, E > 0, zc > 0, cap >= 1"; return GAD_ERR_ARG; }
    // the kernels index rowptr, col and the per-node arrays with the caller's values: check the whole CSR here, on the host
    if (g->nnz < 0 || g->rowptr[0] != 0) { err = "rowptr must start at 0 and nnz must not be negative"; return GAD_ERR_ARG; }
    int64_t lengths = 0;
    if (int rc = check_rows(g, lengths, err)) return rc;
    p.packed = walks_pack(g->nnz, lengths);
    if (g->rowptr[g->n] != g->nnz) { err = "rowptr[n] differs from nnz"; return GAD_ERR_ARG; }
    if (columns) { int rc = check_columns(g, err); if (rc != GAD_OK) return rc; }
    for (int32_t k = 0; k < K; ++k)
        if (core_ptr[k + 1] < core_ptr[k]) { err = "core_ptr decreases"; return GAD_ERR_UNSORTED; }
    p.max_walks.assign((size_t)K, 0);
    int bad = 0;
#pragma omp parallel for schedule(dynamic) reduction(| : bad) if (core_ptr[K] - core_ptr[0] > (1 << 15))
    for (int32_t k = 0; k < K; ++k) {
        int64_t deg = 0;
        for (int64_t t = core_ptr[k]; t < core_ptr[k + 1]; ++t) {
            const int32_t v = core_nodes[t];
            if (v < 0 || v >= g->n) { bad = 1; break; }
            deg += g->rowptr[v + 1] - g->rowptr[v];
        }
        p.max_walks[(size_t)k] = deg * (int64_t)cfg->cap;
    }
    if (bad) { err = "core node out of range"; return GAD_ERR_RANGE; }
    size_t cur = 0;
    p.o_rowptr = take(cur, 8 * (size_t)(g->n + 1)); p.o_col = take(cur, 4 * (size_t)g->nnz);
    p.first.assign(1, 0);
    p.bytes = cur;
    for (int32_t k0 = 0; k0 < K;) {
        int32_t k1 = k0 + 1;
        int64_t keys = p.max_walks[(size_t)k0];
        while (k1 < K && k1 - k0 < 1024 && 6 * (size_t)(k1 + 1 - k0) * (size_t)g->n <= kBatchNodeBytes && (keys + p.max_walks[(size_t)k1]) * (8 + 4 * (cfg->steps + 1)) <= kBatchWalkBytes)
            keys += p.max_walks[(size_t)k1++];
        p.bytes = std::max(p.bytes, batch_layout(p, cur, g->n, core_ptr, k0, k1, cfg->alpha, cfg->steps).end);
        p.first.push_back(k1);
        k0 = k1;
    }
    return GAD_OK;
}

thread_local std::string g_aug_error;
int aug_fail(int code, const std::string& msg) { g_aug_error = msg; return code; }

#define AUG_CK(call)                                                                      \
    do {                                                                                  \
        cudaError_t e_ = (call);                                                          \
        if (e_ != cudaSuccess) return aug_fail(GAD_ERR_CUDA, cudaGetErrorString(e_));     \
    } while (0)
#define AUG_LAUNCH(kernel, grid, block, ...)           \
    do {                                               \
        kernel<<<grid, block, 0, s>>>(__VA_ARGS__);    \
        ++g_kernel_launches;                           \
    } while (0)

}  // namespace

const char* augment_last_error() { return g_aug_error.c_str(); }

// gad_augment; `general`: the walks in the form that takes rows of any length, whatever this graph's are (for tests).
int augment_in_form(bool general, const gad_csr* g, int32_t K, const int64_t* core_ptr, const int32_t* core_nodes, const gad_augment_config* cfg,
                    void* workspace, size_t workspace_bytes, void* stream_, int64_t* halo_ptr, int32_t* halo_nodes, int64_t halo_capacity,
                    int64_t* walks_out) {
    if (!workspace || !halo_ptr || (halo_capacity > 0 && !halo_nodes) || ((uintptr_t)workspace & 255) != 0) return aug_fail(GAD_ERR_ARG, "bad arguments");
    AugPlan p;
    std::string err;
    // A graph that is on the device already had its columns checked on the way there; the kernels read that copy, so the caller's columns, which
    // the host reads after them, are checked while they run.
    bool unchecked = cfg && cfg->graph_resident != 0;
    int rc = plan_augment(g, K, core_ptr, core_nodes, cfg, p, err, !unchecked);
    if (rc != GAD_OK) return aug_fail(rc, err);
    if (workspace_bytes < p.bytes) return aug_fail(GAD_ERR_OOM, "workspace smaller than gad_augment_workspace_bytes");
    cudaStream_t s = (cudaStream_t)stream_;
    char* ws = (char*)workspace;
    int64_t* d_rowptr = (int64_t*)(ws + p.o_rowptr);
    int32_t* d_col = (int32_t*)(ws + p.o_col);
    const int64_t n = g->n;
    const int steps = cfg->steps;
    if (!cfg->graph_resident) {   // else: an earlier call left this very graph at the start of this workspace
        AUG_CK(cudaMemcpyAsync(d_rowptr, g->rowptr, 8 * (size_t)(n + 1), cudaMemcpyHostToDevice, s));
        if (g->nnz > 0) AUG_CK(cudaMemcpyAsync(d_col, g->col, 4 * (size_t)g->nnz, cudaMemcpyHostToDevice, s));
    }
    const size_t graph_end = (size_t)p.o_col + (size_t)round_up((int64_t)std::max<size_t>(4 * (size_t)g->nnz, 4), 256);
    std::vector<uint8_t> taken((size_t)n, 0);
    std::vector<SubDesc> desc;
    std::vector<char> back;
    int64_t out = 0;
    halo_ptr[0] = 0;
    for (size_t b = 0; b + 1 < p.first.size(); ++b) {
        const int32_t k0 = p.first[b], k1 = p.first[b + 1];
        const int G = k1 - k0;
        const BatchLayout L = batch_layout(p, graph_end, n, core_ptr, k0, k1, cfg->alpha, steps);
        desc.resize((size_t)G);
        int64_t key0 = 0, top0 = 0, most_walks = 0;
        for (int32_t k = k0; k < k1; ++k) {
            SubDesc& d = desc[(size_t)(k - k0)];
            d.core0 = core_ptr[k] - core_ptr[k0]; d.ncore = core_ptr[k + 1] - core_ptr[k];
            d.key0 = key0; d.top0 = top0; d.top_cap = leading_walks(p.max_walks[(size_t)k], cfg->alpha, d.ncore); d.max_walks = p.max_walks[(size_t)k]; d.sub = k; d.pad = 0;
            key0 += p.max_walks[(size_t)k]; top0 += d.top_cap;
            most_walks = std::max(most_walks, p.max_walks[(size_t)k]);
        }
        SubDesc* d_desc = (SubDesc*)(ws + L.o_desc);
        SubState* d_state = (SubState*)(ws + L.o_state);
        int32_t *d_core = (int32_t*)(ws + L.o_core), *d_B = (int32_t*)(ws + L.o_B), *d_tile = (int32_t*)(ws + L.o_tile), *d_count = (int32_t*)(ws + L.o_count);
        int32_t *d_seq = (int32_t*)(ws + L.o_seq), *d_node = (int32_t*)(ws + L.o_node);
        uint8_t *d_inside = (uint8_t*)(ws + L.o_inside), *d_bound = (uint8_t*)(ws + L.o_bound);
        unsigned long long *d_key = (unsigned long long*)(ws + L.o_key), *d_top = (unsigned long long*)(ws + L.o_top);
        WalkNode *d_nodes = (WalkNode*)(ws + L.o_nodes), *d_Bnodes = (WalkNode*)(ws + L.o_Bnodes);
        const bool packed = p.packed && !general;
        unsigned* d_hist = (unsigned*)(ws + L.o_hist);
        const int ntiles = num_tiles(n);
        // about `waves` CTAs per SM over all subgraphs of the batch, at least one each
        auto grid = [&](int64_t work_per_block, int64_t work, int waves) {
            const int64_t want = std::max<int64_t>(1, (work + work_per_block - 1) / work_per_block), most = std::max<int64_t>(1, 148 * waves / G);
            return dim3((unsigned)std::min(want, most), (unsigned)G);
        };
        AUG_CK(cudaMemcpyAsync(d_desc, desc.data(), sizeof(SubDesc) * (size_t)G, cudaMemcpyHostToDevice, s));
        if (L.ncore > 0) AUG_CK(cudaMemcpyAsync(d_core, core_nodes + core_ptr[k0], 4 * (size_t)L.ncore, cudaMemcpyHostToDevice, s));
        AUG_CK(cudaMemsetAsync(ws + L.o_count, 0, L.o_seq - L.o_count, s));
        const dim3 node_grid = grid(1024, n, 8), walk_grid = grid(256, most_walks, 8), tile_grid((unsigned)ntiles, (unsigned)G);
        AUG_LAUNCH(mark_kernel, node_grid, 256, d_core, d_desc, d_inside, n, d_rowptr, packed ? d_nodes : nullptr);
        AUG_LAUNCH(boundary_kernel, grid(16, L.ncore / G, 8), 256, d_rowptr, d_col, d_core, d_desc, d_state, d_inside, d_bound, n);
        AUG_LAUNCH(boundary_count_kernel, tile_grid, 256, d_bound, n, ntiles, d_tile);
        AUG_LAUNCH(boundary_list_kernel, tile_grid, 256, d_bound, n, ntiles, d_tile, d_rowptr, d_desc, d_state, d_B, packed ? d_Bnodes : nullptr);
        for (int extra = 0; extra < 2; ++extra) {   // the first batch of walks, then what the error equation asks for on top
            if (packed) AUG_LAUNCH(walk_count_kernel<true>, walk_grid, 256, d_rowptr, d_col, d_B, d_nodes, d_Bnodes, d_inside, n, d_desc, d_state, cfg->seed, extra, steps, d_count, d_node, L.nkeys);
            else AUG_LAUNCH(walk_count_kernel<false>, walk_grid, 256, d_rowptr, d_col, d_B, d_nodes, d_Bnodes, d_inside, n, d_desc, d_state, cfg->seed, extra, steps, d_count, d_node, L.nkeys);
            AUG_LAUNCH(count_stats_kernel, node_grid, 256, d_count, n, d_state, extra);
            if (!extra) AUG_LAUNCH(decide_walks_kernel, (unsigned)((G + 127) / 128), 128, d_state, d_desc, G, cfg->zc / cfg->E, cfg->cap);
        }
        AUG_LAUNCH(decide_lead_kernel, (unsigned)((G + 127) / 128), 128, d_state, d_desc, G, cfg->alpha, steps);
        AUG_LAUNCH(walk_key_kernel, walk_grid, 256, n, d_desc, d_state, steps, d_count, d_node, L.nkeys, d_key, 0);
        int top_bit = 32;
        while (top_bit < 63 && (((int64_t)(steps + 1) * most_walks) >> (top_bit - 32)) > 0) ++top_bit;
        const dim3 hist_grid = grid(8192, most_walks, 2);
        for (int shift = top_bit; shift > 0;) {   // (the last digit may overlap the one before: its upper bits are fixed then)
            shift = std::max(0, shift - kDigitBits);
            AUG_LAUNCH(key_digit_kernel, hist_grid, 1024, d_key, d_desc, d_state, shift, d_hist);
        }
        AUG_LAUNCH(key_gather_kernel, walk_grid, 256, d_key, d_desc, d_state, d_top);
        AUG_LAUNCH(lead_walks_kernel, grid(64, std::max<int64_t>(1, kTopSlack * L.ntop / G), 16), 256, d_desc, d_state, steps, d_node, L.nkeys, d_top, d_seq);
        AUG_CK(cudaGetLastError());
        if (unchecked && (rc = check_columns(g, err)) != GAD_OK) {
            cudaStreamSynchronize(s);   // the kernels are done with the workspace when the call returns
            return aug_fail(rc, err);
        }
        unchecked = false;
        back.resize(L.o_seq - L.o_state + 4 * (size_t)L.ntop * (size_t)(steps + 1));
        AUG_CK(copy_to_host(back.data(), ws + L.o_state, back.size(), s));
        const SubState* state = (const SubState*)back.data();
        const int32_t* leads = (const int32_t*)(back.data() + (L.o_seq - L.o_state));
        for (int32_t k = k0; k < k1; ++k) {
            const int gi = k - k0;
            const SubState& st = state[gi];
            if (walks_out) walks_out[k] = st.nwalks;
            if ((int64_t)st.n0 > p.max_walks[(size_t)k] / cfg->cap) return aug_fail(GAD_ERR_ARG, "the graph on the device is not the caller's (graph_resident)");
            if ((int64_t)st.got < st.lead || (int64_t)st.got > kTopSlack * desc[(size_t)gi].top_cap) return aug_fail(GAD_ERR_CUDA, "selection of the leading walks came out with the wrong count");
            const int64_t first = out;
            auto offer = [&](int32_t v) {   // false: the caller's list is full
                if (taken[(size_t)v]) return true;
                if (out >= halo_capacity) return false;
                taken[(size_t)v] = 1;
                halo_nodes[out++] = v;
                return true;
            };
            const int32_t* row = leads + desc[(size_t)gi].top0 * (steps + 1);
            for (int64_t a = 0; a < st.lead && out - first < st.n_rep; ++a, row += steps + 1)
                for (int t = 0; t <= steps && out - first < st.n_rep; ++t)
                    if (row[t] >= 0 && !offer(row[t])) return aug_fail(GAD_ERR_OOM, "halo_nodes too small");
            if (out - first < st.n_rep && st.lead < st.nwalks) {
                // the leading stretch is used up: every score to the host, every walk ranked there (the leading ones come out first
                // again and offer nothing new)
                AUG_LAUNCH(walk_key_kernel, dim3(148 * 8), 256, n, d_desc + gi, d_state + gi, steps, d_count + (int64_t)gi * n, d_node, L.nkeys, d_key, 1);
                std::vector<int64_t> score((size_t)st.nwalks), order((size_t)st.nwalks);
                std::vector<int32_t> B((size_t)st.nB), seq((size_t)steps + 1);
                AUG_CK(copy_to_host(score.data(), d_key + desc[(size_t)gi].key0, 8 * score.size(), s));
                AUG_CK(copy_to_host(B.data(), d_B + desc[(size_t)gi].core0, 4 * B.size(), s));
                std::iota(order.begin(), order.end(), (int64_t)0);
                std::sort(order.begin(), order.end(), [&](int64_t x, int64_t y) {
                    return score[(size_t)x] != score[(size_t)y] ? score[(size_t)x] > score[(size_t)y] : x < y;
                });
                std::vector<uint8_t> inside((size_t)n, 0);
                for (int64_t t = core_ptr[k]; t < core_ptr[k + 1]; ++t) inside[(size_t)core_nodes[t]] = 1;
                for (int64_t a = 0; a < st.nwalks && out - first < st.n_rep; ++a) {
                    make_walk(g->rowptr, g->col, B.data(), st.nB, cfg->seed, k, order[(size_t)a], steps, seq.data());
                    for (int t = 0; t <= steps && out - first < st.n_rep; ++t)
                        if (!inside[(size_t)seq[(size_t)t]] && !offer(seq[(size_t)t])) return aug_fail(GAD_ERR_OOM, "halo_nodes too small");
                }
            }
            for (int64_t t = first; t < out; ++t) taken[(size_t)halo_nodes[t]] = 0;
            halo_ptr[k + 1] = out;
        }
    }
    AUG_CK(cudaGetLastError());
    return GAD_OK;
}

// For tests: which form the walks of a graph take, from its row pointers.
bool augment_packs(const gad_csr* g) {
    int64_t lengths = 0;
    std::string err;
    return check_rows(g, lengths, err) == GAD_OK && walks_pack(g->nnz, lengths);
}

}  // namespace gad

using namespace gad;

extern "C" {

int gad_augment_workspace_bytes(const gad_csr* g, int32_t K, const int64_t* core_ptr, const int32_t* core_nodes,
                                const gad_augment_config* cfg, size_t* bytes) {
    if (!bytes) return GAD_ERR_ARG;
    AugPlan p;
    std::string err;
    int rc = plan_augment(g, K, core_ptr, core_nodes, cfg, p, err, true);
    if (rc != GAD_OK) return aug_fail(rc, err);
    *bytes = p.bytes;
    return GAD_OK;
}

int gad_augment(const gad_csr* g, int32_t K, const int64_t* core_ptr, const int32_t* core_nodes, const gad_augment_config* cfg,
                void* workspace, size_t workspace_bytes, void* stream_, int64_t* halo_ptr, int32_t* halo_nodes, int64_t halo_capacity,
                int64_t* walks_out) {
    return augment_in_form(false, g, K, core_ptr, core_nodes, cfg, workspace, workspace_bytes, stream_, halo_ptr, halo_nodes, halo_capacity, walks_out);
}

const char* gad_augment_last_error(void) { return augment_last_error(); }

}  // extern "C"
