// Max-IDF summary selection (Section 3.1, Eq. 2-4; Algorithm 1 lines 3 and 6).
//
// Up to 16 blocks of ordinary length are one launch, a cluster with a CTA per block (select_cluster_kernel).  Other problems take
// four launches on one stream, no host synchronisation:
//   presence_kernel   one CTA per block: a V-bit presence set of the block's token ids, built
//                     with shared-memory atomicOr and written to the workspace
//   df_idf_kernel     one thread per vocabulary entry: df(t) = number of blocks whose set holds
//                     t, IDF(t) = ln(B / max(df, 1))   (Eq. 3)
//   chunk_level_kernel one warp per chunk: the minimum df of its tokens (the chunk with the largest
//                     IDF is the one with the smallest df, Eq. 2)
//   topk_kernel       one CTA per block: a counting select of the k best chunks with ties to the
//                     lower index, then the block's part of the prefix list (Eq. 4)
// Ranking uses the integer df only, so the selection is exact.
//
// pulsar_chunk_select runs the same first two launches (one for up to 16 blocks), then chunk_score_kernel (a float64 score
// per chunk under TF-IDF, BM25, the type-token ratio or Max-IDF, Appendix C Eq. 6-9) and
// topk_score_kernel (rank by score, ties to the lower index).
#include <atomic>
#include <cmath>
#include <mutex>
#include <type_traits>

#include <math_constants.h>

#include "common.cuh"

namespace pulsar {
namespace {

constexpr int kPresenceThreads = 1024;
constexpr int kTopkThreads = 256;
constexpr size_t kMaxDynSmem = 227 * 1024;

// Dynamic shared memory above 48 KB has to be allowed, and what is allowed belongs to the kernel on its device, not to the
// launch: it is always set to all there is beside the kernel's own, because another thread may set it for its call between
// here and the launch.
template <typename Kernel>
cudaError_t allow_smem(Kernel* kernel, size_t bytes) {
    if (bytes <= 48 * 1024) return cudaSuccess;
    cudaFuncAttributes own;
    const cudaError_t e = cudaFuncGetAttributes(&own, kernel);
    return e != cudaSuccess ? e
                            : cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                   static_cast<int>(kMaxDynSmem - own.sharedSizeBytes));
}

__global__ void __launch_bounds__(kPresenceThreads)
presence_kernel(const uint32_t* __restrict__ ids, int64_t L, int block_size, int vocab_size, int words,
                uint32_t* __restrict__ bitmaps, int32_t* status) {
    extern __shared__ uint32_t bits[];
    const int b = blockIdx.x;
    for (int w = threadIdx.x; w < words; w += blockDim.x) bits[w] = 0u;
    grid_dependency_wait();            // the token ids, and the workspace, may be in use by the launch before this one
    grid_launch_dependents();          // the next launch of the chain may be placed; it waits for this grid itself
    __syncthreads();
    const uint32_t* blk = ids + static_cast<size_t>(b) * block_size;
    const int len = static_cast<int>(min(static_cast<int64_t>(block_size), L - static_cast<int64_t>(b) * block_size));
    for (int i = threadIdx.x; i < len; i += blockDim.x) {
        const uint32_t t = blk[i];
        if (t < static_cast<uint32_t>(vocab_size)) atomicOr(&bits[t >> 5], 1u << (t & 31));
        else report(status, PULSAR_DEV_BAD_TOKEN);
    }
    __syncthreads();
    uint32_t* out = bitmaps + static_cast<size_t>(b) * words;
    for (int w = threadIdx.x; w < words; w += blockDim.x) out[w] = bits[w];
}

__global__ void df_idf_kernel(const uint32_t* __restrict__ bitmaps, int n_blocks, int words, int vocab_size,
                              uint16_t* __restrict__ df_table, uint32_t* __restrict__ df_out,
                              float* __restrict__ idf_out) {
    grid_launch_dependents();
    grid_dependency_wait();            // the presence sets are complete
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= vocab_size) return;
    const int w = t >> 5, bit = t & 31;
    uint32_t df = 0;
    for (int b = 0; b < n_blocks; ++b) df += (bitmaps[static_cast<size_t>(b) * words + w] >> bit) & 1u;
    df_table[t] = static_cast<uint16_t>(df);
    if (df_out) df_out[t] = df;
    if (idf_out) idf_out[t] = logf(static_cast<float>(n_blocks) / static_cast<float>(df > 0 ? df : 1));
}

// Exclusive block-wide prefix sum of one int per thread; returns the thread's offset and the
// block total through `total`.  warp_sums: kTopkThreads/32 ints of shared scratch.
__device__ __forceinline__ int block_exclusive_scan(int v, int* warp_sums, int& total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int incl = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        int n = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += n;
    }
    if (lane == 31) warp_sums[warp] = incl;
    __syncthreads();
    int base = 0;
    total = 0;
    for (int i = 0; i < kTopkThreads / 32; ++i) {
        int s = warp_sums[i];
        if (i < warp) base += s;
        total += s;
    }
    __syncthreads();
    return base + incl - v;
}

// level[b*C + c] = min over the chunk's tokens of df.  Slot c of block b covers the tokens
// [b*block_size + c*chunk, +chunk) that lie inside the block and the sequence: the last chunk of
// a block may be shorter, and a slot past the end of a short last block holds no chunk at all.
// Ranks: a chunk whose ids all lie outside the vocabulary gets `worst` (after every real df), a
// slot without a chunk worst + 1 (never selected).
__global__ void __launch_bounds__(256)
chunk_level_kernel(const uint32_t* __restrict__ ids, const uint16_t* __restrict__ df_table, int64_t L,
                   int block_size, int chunks_per_block, int n_slots_total, int chunk, int vocab_size, int worst,
                   uint16_t* __restrict__ level) {
    grid_launch_dependents();
    grid_dependency_wait();            // the df table is complete
    const int lane = threadIdx.x & 31;
    const int slot = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (slot >= n_slots_total) return;
    const int b = slot / chunks_per_block, c = slot - b * chunks_per_block;
    const int64_t lo = static_cast<int64_t>(b) * block_size;
    const int64_t block_end = min(lo + block_size, L);
    const int64_t start = lo + static_cast<int64_t>(c) * chunk;
    const int len = static_cast<int>(max(static_cast<int64_t>(0), min(static_cast<int64_t>(chunk), block_end - start)));
    int mn = len > 0 ? worst : worst + 1;
    for (int p = lane; p < len; p += 32) {
        const uint32_t t = ids[start + p];
        if (t < static_cast<uint32_t>(vocab_size)) mn = min(mn, static_cast<int>(df_table[t]));
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mn = min(mn, __shfl_xor_sync(0xffffffffu, mn, o));
    if (lane == 0) level[slot] = static_cast<uint16_t>(mn);
}

// Where a block's part of the prefix list goes and how long it is when lengths do not divide.
struct PrefixGeometry {
    int k_b;          // chunks this block contributes: min(k, chunks it has)
    int sink_eff;     // min(sink, tokens of block 0)
    int tail;         // tokens of the last chunk slot of a full block (= chunk when chunk divides block_size)
    int cap;          // entries of prefix_idx: sink + (n_blocks - 1) * k * chunk
};

__device__ __forceinline__ PrefixGeometry prefix_geometry(int b, int n_blocks, int64_t L, int block_size, int chunk,
                                                          int k, int sink) {
    PrefixGeometry g;
    const int64_t lo = static_cast<int64_t>(b) * block_size;
    const int len_b = static_cast<int>(min(static_cast<int64_t>(block_size), L - lo));
    const int chunks_b = (len_b + chunk - 1) / chunk;
    g.k_b = min(k, chunks_b);
    g.sink_eff = static_cast<int>(min(static_cast<int64_t>(sink), min(static_cast<int64_t>(block_size), L)));
    const int C = (block_size + chunk - 1) / chunk;
    g.tail = block_size - (C - 1) * chunk;
    g.cap = sink + (n_blocks - 1) * k * chunk;
    return g;
}

// Block b's part of the prefix list (Eq. 4): its chosen chunks (ascending, in shared memory) as
// global token positions starting at entry `offset`, the sink entries (written by block 0), the
// unused entries at the end (-1, written by the last block) and prefix_len[b] = offset (0 for
// block 0).  Only the last chosen chunk can be a short one (the last slot of the block), so the
// block's entries are the leading ones of k_b * chunk: those whose position lies inside the block.
__device__ __forceinline__ void write_block_prefix(int b, int n_blocks, int block_size, int chunk, int k,
                                                   const PrefixGeometry& g, int offset, const int* chosen,
                                                   int32_t* __restrict__ sel_chunks, int32_t* __restrict__ prefix_idx,
                                                   int32_t* __restrict__ prefix_len) {
    for (int j = g.k_b + threadIdx.x; j < k; j += blockDim.x) sel_chunks[static_cast<size_t>(b) * k + j] = -1;
    if (b < n_blocks - 1) {
        int32_t* dst = prefix_idx + offset;
        const int n = g.k_b * chunk;
        for (int i = threadIdx.x; i < n; i += blockDim.x) {
            const int j = i / chunk, p = i - j * chunk;
            const int pos = chosen[j] * chunk + p;
            if (pos < block_size) dst[i] = b * block_size + pos;
        }
    } else {
        for (int i = offset + threadIdx.x; i < g.cap; i += blockDim.x) prefix_idx[i] = -1;
    }
    if (b == 0)
        for (int i = threadIdx.x; i < g.sink_eff; i += blockDim.x) prefix_idx[i] = i;
    if (threadIdx.x == 0) prefix_len[b] = b == 0 ? 0 : offset;
}

// Entry of prefix_idx at which block b's summary starts: the sink plus the tokens of the
// summaries of blocks 0..b-1.  Those blocks are full ones; each contributes k chunks of `chunk`
// tokens, except that a block which selected its last chunk slot contributes only that slot's
// `tail` tokens for it.  The last slot (index C-1) is selected iff fewer than k of the other slots
// rank at or before it, i.e. have a level <= its own (they all have a lower index).  Only needed
// when chunk does not divide block_size; one warp per earlier block.
__device__ __forceinline__ int prefix_offset(int b, const uint16_t* __restrict__ level_all, int C, int chunk, int k,
                                             const PrefixGeometry& g, int* s_short) {
    if (g.tail == chunk || k == 0 || b == 0) return g.sink_eff + b * k * chunk;
    if (threadIdx.x == 0) *s_short = 0;
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, n_warps = blockDim.x >> 5;
    for (int j = warp; j < b; j += n_warps) {
        const uint16_t* lv = level_all + static_cast<size_t>(j) * C;
        const int last = lv[C - 1];
        int before = 0;
        for (int c = lane; c < C - 1; c += 32) before += (lv[c] <= last) ? 1 : 0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) before += __shfl_xor_sync(0xffffffffu, before, o);
        if (lane == 0 && before < k) atomicAdd(s_short, 1);
    }
    __syncthreads();
    return g.sink_eff + b * k * chunk - *s_short * (chunk - g.tail);
}

__global__ void __launch_bounds__(kTopkThreads)
topk_kernel(const uint16_t* __restrict__ level_all, int n_blocks, int64_t L, int block_size, int chunk, int k_all,
            int sink, int32_t* __restrict__ sel_chunks, int32_t* __restrict__ prefix_idx,
            int32_t* __restrict__ prefix_len) {
    extern __shared__ int smem[];
    const int C = (block_size + chunk - 1) / chunk;
    int* level = smem;                       // [C]   min df of the chunk
    int* hist = level + C;                   // [n_blocks + 3]
    int* chosen = hist + n_blocks + 3;       // [k]   selected chunk ids, ascending
    __shared__ int warp_sums[kTopkThreads / 32];
    __shared__ int s_threshold, s_need, s_short;

    const int b = blockIdx.x;
    const PrefixGeometry geo = prefix_geometry(b, n_blocks, L, block_size, chunk, k_all, sink);
    const int k = geo.k_b;                   // a short last block may have fewer than k_all chunks

    for (int i = threadIdx.x; i < n_blocks + 3; i += blockDim.x) hist[i] = 0;
    grid_dependency_wait();                  // the chunk levels are complete
    grid_launch_dependents();
    __syncthreads();
    for (int c = threadIdx.x; c < C; c += blockDim.x) {
        const int lv = level_all[static_cast<size_t>(b) * C + c];
        level[c] = lv;
        atomicAdd(&hist[lv], 1);
    }
    __syncthreads();

    // threshold level T: all chunks below T are taken, `need` more at T (lowest indices first)
    if (threadIdx.x == 0) {
        int cum = 0, T = 0;
        for (; T <= n_blocks + 1; ++T) {
            if (cum + hist[T] >= k) break;
            cum += hist[T];
        }
        s_threshold = T;
        s_need = k - cum;
    }
    __syncthreads();
    const int T = s_threshold, need = s_need;

    // ordered compaction over the chunks, a tile of blockDim chunks at a time
    int at_T_before = 0, taken_before = 0;
    for (int c0 = 0; c0 < C; c0 += kTopkThreads) {
        const int c = c0 + threadIdx.x;
        const int lv = c < C ? level[c] : n_blocks + 3;
        const int is_T = (lv == T) ? 1 : 0;
        int tot_T;
        const int rank_T = at_T_before + block_exclusive_scan(is_T, warp_sums, tot_T);
        const int take = (lv < T || (is_T && rank_T < need)) ? 1 : 0;
        int tot_take;
        const int pos = taken_before + block_exclusive_scan(take, warp_sums, tot_take);
        if (take && pos < k) {
            chosen[pos] = c;
            sel_chunks[static_cast<size_t>(b) * k_all + pos] = c;
        }
        at_T_before += tot_T;
        taken_before += tot_take;
    }
    __syncthreads();

    const int offset = prefix_offset(b, level_all, C, chunk, k_all, geo, &s_short);
    write_block_prefix(b, n_blocks, block_size, chunk, k_all, geo, offset, chosen, sel_chunks, prefix_idx, prefix_len);
}

// ---------------------------------------------------------------------------------------------
// Selection under the other chunk scores of Appendix C (Eq. 6-8) and Max-IDF as a score (Eq. 9).
// Scores are float64 and every operation is an explicitly rounded add, multiply or divide in
// the order the equations are written (positions left to right, types by first occurrence), so
// two chunks tie exactly when their scores are the same double.  The logarithms are a table over
// df = 0..B that the host fills (B + 1 values) and passes as a kernel parameter.  |C| is the number
// of tokens the chunk has (the last chunk of a block may be short), the mean chunk length of the
// BM25 normaliser is L over the number of chunks of the sequence.
// ---------------------------------------------------------------------------------------------
constexpr int kMaxScoreBlocks = 1024;
constexpr int kMaxScoreChunk = 1024;
constexpr int kMaxScoreChunksPerBlock = 4096;
// kBlocks: room for df = 0 .. kBlocks.  A kernel parameter costs the host about 1.2 us a kilobyte at every launch (20.6
// against 18.1 us for the whole BM25 selection over 16 blocks), so there are two sizes.
constexpr int kFewScoreBlocks = 64;
template <int kBlocks>
struct ScoreTable {
    double by_df[kBlocks + 1];           // Eq. 5 (TF-IDF, Max-IDF) or the BM25 IDF of Eq. 7, per df
    double k1_plus_1, k1, b, one_minus_b, mean_len;   // BM25: D(C) = (1 - b) + b * (|C| / mean chunk length)
};

// The terms of a chunk's sum under TF-IDF and BM25, formed by a warp side by side, one per position; a position that carries no
// term holds 0.0, which leaves the sum's bits as they are.  Under BM25 and the type-token ratio each position is compared with all
// others of the chunk, for a chunk of at most 32 tokens in one warp match.  Returns the number of types (type-token ratio).
// df_of(p, first): the df of the token at position p, kNoDf where its id lies outside the vocabulary; tok: the ids, read only
// where positions are compared.
template <int kMode, uint32_t kNoDf, int kBlocks, typename DfOf>
__device__ __forceinline__ int chunk_terms(const uint32_t* tok, int len, const ScoreTable<kBlocks>& tab, DfOf df_of, double* term) {
    const int lane = threadIdx.x & 31;
    double k1_times_D = 0.0;
    if (kMode == PULSAR_SCORE_BM25)
        // D(C) = (1 - b) + b * (|C| / mean chunk length), then k1 * D(C): one rounding per operation
        k1_times_D =
            __dmul_rn(tab.k1, __dadd_rn(tab.one_minus_b, __dmul_rn(tab.b, __ddiv_rn(static_cast<double>(len), tab.mean_len))));
    int distinct = 0;
    for (int p0 = 0; p0 < len; p0 += 32) {
        const int p = p0 + lane;
        const bool in = p < len;
        bool first = in;
        int tf = 0;
        if (kMode != PULSAR_SCORE_TF_IDF) {
            const uint32_t t = in ? tok[p] : ~0u;
            if (len <= 32) {
                // (an id of ~0 meets the lanes past the end, which come after it: its count, unused, is too large)
                const uint32_t same = __match_any_sync(0xffffffffu, t);
                first = in && lane == __ffs(same) - 1;
                tf = __popc(same);
            } else {
                int before = 0;
#pragma unroll 16                                    // 1024 positions 256 us, with the compiler's four at a time 314
                for (int q = 0; q < len; ++q) {
                    const int eq = tok[q] == t ? 1 : 0;
                    tf += eq;
                    before += q < p ? eq : 0;
                }
                first = in && before == 0;
            }
        }
        if (kMode == PULSAR_SCORE_TYPE_TOKEN) {
            distinct += __popc(__ballot_sync(0xffffffffu, first));
        } else if (in) {
            const uint32_t df = df_of(p, first);
            double x = 0.0;
            if (first && df != kNoDf) {
                x = tab.by_df[df];
                if (kMode == PULSAR_SCORE_BM25) {
                    const double tfd = static_cast<double>(tf);
                    x = __ddiv_rn(__dmul_rn(x, __dmul_rn(tfd, tab.k1_plus_1)), __dadd_rn(tfd, k1_times_D));
                }
            }
            term[p] = x;
        }
    }
    return distinct;
}

// One warp per chunk slot.  Slot c of block b covers the tokens [b*block_size + c*chunk, +chunk)
// that lie inside the block and the sequence (|C| = len); a slot without a chunk scores -inf.
// The lanes form the terms (chunk_terms), and lane 0 adds them up in the order of the equations.
// Latency-bound: one thread per chunk, walking the chunk's pairs
// of positions serially, took 92 us for 4096 chunks of 32 tokens under BM25 (the whole call 115 us, 16 us with
// this form and its launches, three or four, chained as programmatic dependents).
constexpr int kScoreWarps = 4;

template <int kMode, int kBlocks>
__global__ void __launch_bounds__(kScoreWarps * 32)
chunk_score_kernel(const uint32_t* __restrict__ ids, const uint16_t* __restrict__ df_table, int64_t L,
                   int block_size, int chunks_per_block, int n_slots_total, int chunk, int vocab_size,
                   const __grid_constant__ ScoreTable<kBlocks> tab, double* __restrict__ score) {
    extern __shared__ double smem_d[];                     // per warp: a term and a token per position
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    double* term = smem_d + warp * chunk;
    uint32_t* tok = reinterpret_cast<uint32_t*>(smem_d + kScoreWarps * chunk) + warp * chunk;
    const int slot = blockIdx.x * kScoreWarps + warp;
    if (slot >= n_slots_total) return;
    const int b = slot / chunks_per_block, c = slot - b * chunks_per_block;
    const int64_t lo = static_cast<int64_t>(b) * block_size;
    const int64_t start = lo + static_cast<int64_t>(c) * chunk;
    const int len = static_cast<int>(max(static_cast<int64_t>(0),
                                         min(static_cast<int64_t>(chunk), min(lo + block_size, L) - start)));
    const uint32_t V = static_cast<uint32_t>(vocab_size);
    // The ids may be read before the wait: the presence launch of this call, which let its dependents in only after its own
    // wait, has found them complete.
    for (int p = lane; p < len; p += 32) tok[p] = ids[start + p];
    __syncwarp();
    grid_dependency_wait();                                // the df table is complete
    if (kMode == PULSAR_SCORE_MAX_IDF || len == 0) {
        double best = -CUDART_INF;
        for (int p = lane; p < len; p += 32)
            if (tok[p] < V) best = fmax(best, tab.by_df[df_table[tok[p]]]);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) best = fmax(best, __shfl_xor_sync(0xffffffffu, best, o));
        if (lane == 0) score[slot] = best;
        return;
    }
    const int distinct = chunk_terms<kMode, ~0u>(
        tok, len, tab, [&](int p, bool first) { return first && tok[p] < V ? df_table[tok[p]] : ~0u; }, term);
    __syncwarp();
    // The selection's CTAs, one per block and bound by float64 compares, are placed where there is room.  Let in while this grid
    // still fills the chip they were put several to an SM: 16 blocks of 2048 chunks of 4 tokens under BM25 took 829 us, 190 us
    // with the dependents let in here.
    grid_launch_dependents();
    if (lane != 0) return;
    double s = 0.0;
    if (kMode == PULSAR_SCORE_TYPE_TOKEN) {
        s = static_cast<double>(distinct);
    } else {
#pragma unroll 8
        for (int p = 0; p < len; ++p) s = __dadd_rn(s, term[p]);
    }
    score[slot] = kMode == PULSAR_SCORE_BM25 ? s : __ddiv_rn(s, static_cast<double>(len));
}

// Very many short chunks: one thread per chunk slot walks its tokens, the positions of a type counted where it first occurs.
// A warp per chunk leaves most of its lanes idle there and needs a warp's start for each.  us of the whole call under BM25,
// warp / thread form: 262,144 chunks of 4 256 / 197, 131,072 of 8 97 / 67, 125,000 of 4 in 500 blocks 75 / 53, 42,000 of 12
// in 500 blocks 94 / 89; from 16 tokens on (65,536: 55 against 73 with one thread each) and with few chunks, where one
// warp each is still all at once, the warp is the better form.
constexpr int kThreadFormChunk = 12;
constexpr int kThreadFormSlots = 40000;

template <int kMode, int kBlocks>
__global__ void __launch_bounds__(128)
chunk_score_thread_kernel(const uint32_t* __restrict__ ids, const uint16_t* __restrict__ df_table, int64_t L,
                          int block_size, int chunks_per_block, int n_slots_total, int chunk, int vocab_size,
                          const __grid_constant__ ScoreTable<kBlocks> tab, double* __restrict__ score) {
    const int slot = blockIdx.x * blockDim.x + threadIdx.x;
    const int b = slot / chunks_per_block, c = slot - b * chunks_per_block;
    const int64_t lo = static_cast<int64_t>(b) * block_size;
    const int64_t start = lo + static_cast<int64_t>(c) * chunk;
    const int len = slot < n_slots_total
                        ? static_cast<int>(max(static_cast<int64_t>(0), min(static_cast<int64_t>(chunk), min(lo + block_size, L) - start)))
                        : 0;
    const uint32_t V = static_cast<uint32_t>(vocab_size);
    uint32_t tok[kThreadFormChunk];
#pragma unroll
    for (int p = 0; p < kThreadFormChunk; ++p) tok[p] = p < len ? ids[start + p] : 0u;    // complete: see the warp form
    grid_dependency_wait();                                // the df table is complete
    double s = 0.0;
    if (kMode == PULSAR_SCORE_MAX_IDF || len == 0) {
        s = -CUDART_INF;
#pragma unroll
        for (int p = 0; p < kThreadFormChunk; ++p)
            if (p < len && tok[p] < V) s = fmax(s, tab.by_df[df_table[tok[p]]]);
    } else if (kMode == PULSAR_SCORE_TF_IDF) {
#pragma unroll
        for (int p = 0; p < kThreadFormChunk; ++p)
            if (p < len && tok[p] < V) s = __dadd_rn(s, tab.by_df[df_table[tok[p]]]);
        s = __ddiv_rn(s, static_cast<double>(len));
    } else {
        const double k1_times_D =
            __dmul_rn(tab.k1, __dadd_rn(tab.one_minus_b, __dmul_rn(tab.b, __ddiv_rn(static_cast<double>(len), tab.mean_len))));
        int distinct = 0;
#pragma unroll
        for (int p = 0; p < kThreadFormChunk; ++p) {
            int before = 0, tf = 0;
#pragma unroll
            for (int q = 0; q < kThreadFormChunk; ++q) {
                const int eq = q < len && tok[q] == tok[p] ? 1 : 0;
                tf += eq;
                before += q < p ? eq : 0;
            }
            if (p >= len || before > 0) continue;
            ++distinct;
            if (kMode == PULSAR_SCORE_BM25 && tok[p] < V) {
                const double tfd = static_cast<double>(tf);
                const double num = __dmul_rn(tab.by_df[df_table[tok[p]]], __dmul_rn(tfd, tab.k1_plus_1));
                s = __dadd_rn(s, __ddiv_rn(num, __dadd_rn(tfd, k1_times_D)));
            }
        }
        if (kMode == PULSAR_SCORE_TYPE_TOKEN) s = __ddiv_rn(static_cast<double>(distinct), static_cast<double>(len));
    }
    grid_launch_dependents();
    if (slot < n_slots_total) score[slot] = s;
}

// One CTA per block: chunk c is taken when fewer than k chunks beat it (a larger score, or the
// same score at a lower index); the taken chunks are compacted in index order.
__global__ void __launch_bounds__(kTopkThreads)
topk_score_kernel(const double* __restrict__ score_all, int n_blocks, int64_t L, int block_size, int chunk, int k_all,
                  int sink, int32_t* __restrict__ sel_chunks, int32_t* __restrict__ prefix_idx,
                  int32_t* __restrict__ prefix_len) {
    extern __shared__ double smem_d[];
    const int C = (block_size + chunk - 1) / chunk;
    double* sc = smem_d;                                   // [C]
    int* chosen = reinterpret_cast<int*>(sc + C);          // [k]
    __shared__ int warp_sums[kTopkThreads / 32];
    __shared__ int s_short;
    const int b = blockIdx.x;
    const PrefixGeometry geo = prefix_geometry(b, n_blocks, L, block_size, chunk, k_all, sink);
    const int k = geo.k_b;                                 // a short last block may have fewer than k_all chunks
    const int64_t lo = static_cast<int64_t>(b) * block_size;
    const int Cb = static_cast<int>((min(static_cast<int64_t>(block_size), L - lo) + chunk - 1) / chunk);
    grid_dependency_wait();                                // the scores are complete
    grid_launch_dependents();
    for (int c = threadIdx.x; c < C; c += blockDim.x) sc[c] = score_all[static_cast<size_t>(b) * C + c];
    __syncthreads();
    int taken_before = 0;
    for (int c0 = 0; c0 < C; c0 += kTopkThreads) {
        const int c = c0 + threadIdx.x;
        int take = 0;
        if (c < Cb) {
            const double mine = sc[c];
            int better = 0;
            for (int o = 0; o < Cb; ++o) {
                const double v = sc[o];
                better += (v > mine || (v == mine && o < c)) ? 1 : 0;
            }
            take = better < k ? 1 : 0;
        }
        int tot;
        const int pos = taken_before + block_exclusive_scan(take, warp_sums, tot);
        if (take && pos < k) {
            chosen[pos] = c;
            sel_chunks[static_cast<size_t>(b) * k_all + pos] = c;
        }
        taken_before += tot;
    }
    __syncthreads();
    // Entry of prefix_idx at which this block's summary starts: as in prefix_offset, with the scores
    // deciding whether an earlier (full) block selected its short last chunk -- it did iff fewer
    // than k of its other chunks, which all have a lower index, score at least as much.
    int offset = geo.sink_eff + b * k_all * chunk;
    if (geo.tail != chunk && k_all > 0 && b > 0) {
        if (threadIdx.x == 0) s_short = 0;
        __syncthreads();
        const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, n_warps = blockDim.x >> 5;
        for (int j = warp; j < b; j += n_warps) {
            const double* sj = score_all + static_cast<size_t>(j) * C;
            const double last = sj[C - 1];
            int before = 0;
            for (int c = lane; c < C - 1; c += 32) before += (sj[c] >= last) ? 1 : 0;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) before += __shfl_xor_sync(0xffffffffu, before, o);
            if (lane == 0 && before < k_all) atomicAdd(&s_short, 1);
        }
        __syncthreads();
        offset -= s_short * (chunk - geo.tail);
    }
    write_block_prefix(b, n_blocks, block_size, chunk, k_all, geo, offset, chosen, sel_chunks, prefix_idx, prefix_len);
}

struct SelectPlan {
    int n_blocks, words, C;
    size_t bitmap_bytes, df_bytes, level_bytes, total;
    size_t presence_smem, topk_smem;
};

int32_t plan_select(int64_t L, int32_t vocab_size, int32_t block_size, int32_t chunk, int32_t k, int32_t sink,
                    SelectPlan& p) {
    if (L <= 0 || vocab_size <= 0 || block_size <= 0 || chunk <= 0 || k < 0 || sink < 0) return PULSAR_ERR_INVALID_ARG;
    if (L >= (1ll << 31)) return PULSAR_ERR_SHAPE;
    const int64_t B = (L + block_size - 1) / block_size;
    p.C = (block_size + chunk - 1) / chunk;
    // chunk levels are 16-bit: the real df values 0..B and the two ranks after them, B + 1 and B + 2
    if (B > 65533 || k > p.C || sink > block_size || p.C > 32768) return PULSAR_ERR_SHAPE;
    if (sink + (B - 1) * static_cast<int64_t>(k) * chunk >= (1ll << 31)) return PULSAR_ERR_SHAPE;
    p.n_blocks = static_cast<int>(B);
    p.words = (vocab_size + 31) / 32;
    p.presence_smem = static_cast<size_t>(p.words) * 4;
    p.topk_smem = (static_cast<size_t>(p.C) + p.n_blocks + 3 + k) * 4;
    if (p.presence_smem > kMaxDynSmem || p.topk_smem > kMaxDynSmem) return PULSAR_ERR_SHAPE;
    p.bitmap_bytes = round_up(static_cast<size_t>(p.n_blocks) * p.words * 4, 256);
    p.df_bytes = round_up(static_cast<size_t>(vocab_size) * 2, 256);
    p.level_bytes = round_up(static_cast<size_t>(p.n_blocks) * p.C * 2, 256);
    p.total = p.bitmap_bytes + p.df_bytes + p.level_bytes;
    return PULSAR_OK;
}

// ---------------------------------------------------------------------------------------------
// The whole selection in one launch, for sequences of at most 16 blocks: a CTA per block, in a cluster of 8 or 16.
// The presence sets stay in shared memory and are read there by the CTAs, those without a block too, that form the df of a slice
// of the vocabulary each; the df of the block's tokens, the chunks' ranks and the selected chunks are the CTA's own.  What crosses
// CTAs are two cluster barriers instead of three launches, and the df table (a byte per entry, in L2).  Bound by a chain of
// latencies: each thread's loads are issued together (one at a time: 45,011 tokens 10.2 us, 8.0 like this and with a look at
// the presence bit before the atomic).
// kModeTable ends with the df table.
// ---------------------------------------------------------------------------------------------
constexpr int kClusterThreads = 1024;
constexpr int kClusterBlocks = 16;              // CTAs of the largest cluster
constexpr int kClusterTokens = 8192;            // of a block: its ids, and a term per id, are kept in shared memory
constexpr int kClusterChunks = 1024;            // of a block: a thread each in the selection
constexpr int kModeLevels = -1;                 // chunks ranked by their least df (pulsar_maxidf_select), without scores
constexpr int kModeTable = -2;                  // the df table alone, 16 bits an entry, for score launches of their own

struct ClusterShape {
    size_t bits, tokens, dfs, ranks, chosen, terms, total;       // offsets in shared memory
    __host__ __device__ ClusterShape(int words, int block_size, int C, int chunk, int k, int mode) {
        const auto up = [](size_t x) { return (x + 15) / 16 * 16; };
        const bool scores = mode >= 0, ids = mode == PULSAR_SCORE_BM25 || mode == PULSAR_SCORE_TYPE_TOKEN;
        bits = 0;
        tokens = up(static_cast<size_t>(words) * 4);
        dfs = tokens + (ids ? up(static_cast<size_t>(block_size) * 4) : 0);
        ranks = dfs + up(block_size);
        chosen = ranks + up(static_cast<size_t>(C) * (scores ? 8 : 4));
        terms = chosen + up(static_cast<size_t>(k) * 4);
        // a term per position; chunks an odd number of terms apart, so that the threads that add them up meet in no bank
        total = terms + (scores ? static_cast<size_t>(C) * (chunk | 1) * 8 : 0);
    }
};

__device__ __forceinline__ void cluster_sync() {
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ uint32_t ld_cluster_u32(uint32_t addr, int rank) {
    uint32_t v;
    asm volatile("{\n\t.reg .u32 a;\n\tmapa.shared::cluster.u32 a, %1, %2;\n\tld.shared::cluster.u32 %0, [a];\n\t}"
                 : "=r"(v) : "r"(addr), "r"(rank) : "memory");
    return v;
}
__device__ __forceinline__ void st_cluster_u32(uint32_t addr, int rank, uint32_t v) {
    asm volatile("{\n\t.reg .u32 a;\n\tmapa.shared::cluster.u32 a, %0, %1;\n\tst.shared::cluster.u32 [a], %2;\n\t}"
                 ::"r"(addr), "r"(rank), "r"(v) : "memory");
}

// The position of the calling thread's chunk among those taken (one bit a thread, in thread order).
__device__ __forceinline__ int taken_before(bool take, int* warp_sums) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t mine = __ballot_sync(0xffffffffu, take);
    if (lane == 0) warp_sums[warp] = __popc(mine);
    __syncthreads();
    const int base = __reduce_add_sync(0xffffffffu, lane < warp ? warp_sums[lane] : 0);
    __syncthreads();
    return base + __popc(mine & ((1u << lane) - 1));
}

struct ClusterArgs {
    const uint32_t* ids;
    int64_t L;
    int n_blocks, block_size, chunk, k, sink, vocab_size, words;
    uint8_t* df_table;                          // [vocab_size rounded up to 32], of uint16 with kModeTable
    int32_t *sel_chunks, *prefix_idx, *prefix_len;
    uint32_t* df_out;
    float* idf_out;
    double* score;                              // [blocks, C] or null
    int32_t* status;
};

template <int kMode>
__global__ void __launch_bounds__(kClusterThreads, 1)
select_cluster_kernel(const __grid_constant__ ClusterArgs a,
                      const __grid_constant__ std::conditional_t<kMode < 0, int, ScoreTable<kClusterBlocks>> tab) {
    constexpr bool kScores = kMode >= 0;
    extern __shared__ __align__(16) uint8_t smem_c[];
    __shared__ int s_warp[32], s_hist[32], s_short[kClusterBlocks], s_threshold, s_need;
    __shared__ float s_idf[kClusterBlocks + 1];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int b = blockIdx.x, n_blocks = a.n_blocks;            // CTAs from n_blocks on have a slice of the vocabulary only
    const int C = (a.block_size + a.chunk - 1) / a.chunk;
    const ClusterShape at(a.words, a.block_size, C, a.chunk, a.k, kMode);
    uint32_t* bits = reinterpret_cast<uint32_t*>(smem_c + at.bits);
    uint32_t* tok = reinterpret_cast<uint32_t*>(smem_c + at.tokens);
    uint8_t* dfs = smem_c + at.dfs;
    int* chosen = reinterpret_cast<int*>(smem_c + at.chosen);
    const uint32_t V = static_cast<uint32_t>(a.vocab_size);
    const PrefixGeometry geo = prefix_geometry(b, n_blocks, a.L, a.block_size, a.chunk, a.k, a.sink);
    const int64_t lo = static_cast<int64_t>(b) * a.block_size;
    const int len_b = b < n_blocks ? static_cast<int>(min(static_cast<int64_t>(a.block_size), a.L - lo)) : 0;

    if (b < n_blocks)
        for (int w = tid; w < a.words; w += kClusterThreads) bits[w] = 0u;
    if (tid < 32) s_hist[tid] = 0;
    grid_dependency_wait();            // the token ids, and the workspace, may be in use by the launch before this one
    grid_launch_dependents();
    __syncthreads();
    constexpr int kPerThread = kClusterTokens / kClusterThreads;       // all of a thread's loads are under way at once
    uint32_t mine_t[kPerThread];
#pragma unroll
    for (int j = 0; j < kPerThread; ++j) mine_t[j] = tid + j * kClusterThreads < len_b ? a.ids[lo + tid + j * kClusterThreads] : 0u;
#pragma unroll
    for (int j = 0; j < kPerThread; ++j) {
        const int i = tid + j * kClusterThreads;
        if (i >= len_b) break;
        if (kMode == PULSAR_SCORE_BM25 || kMode == PULSAR_SCORE_TYPE_TOKEN) tok[i] = mine_t[j];
        if (mine_t[j] < V) {
            // (most tokens of a block repeat, and an atomic on a word that many lanes want is done lane by lane)
            const uint32_t bit = 1u << (mine_t[j] & 31);
            if ((*const_cast<volatile uint32_t*>(bits + (mine_t[j] >> 5)) & bit) == 0u) atomicOr(&bits[mine_t[j] >> 5], bit);
        } else {
            report(a.status, PULSAR_DEV_BAD_TOKEN);
        }
    }
    cluster_sync();                    // every block's set is complete

    // ---- df of this CTA's slice of the vocabulary: the sets' words added up bit by bit, 32 entries a thread ----
    const int n_ctas = gridDim.x, per_cta = (a.words + n_ctas - 1) / n_ctas, w_end = min(a.words, (b + 1) * per_cta);
    for (int w = b * per_cta + tid; w < w_end; w += kClusterThreads) {
        uint32_t x[kClusterBlocks], plane[5] = {0u, 0u, 0u, 0u, 0u};
        const uint32_t addr = smem_u32(bits + w);
#pragma unroll
        for (int j = 0; j < kClusterBlocks; ++j) x[j] = j < n_blocks ? ld_cluster_u32(addr, j) : 0u;
#pragma unroll
        for (int j = 0; j < kClusterBlocks; ++j) {
            uint32_t carry = x[j];
#pragma unroll
            for (int p = 0; p < 5; ++p) {
                const uint32_t next = plane[p] & carry;
                plane[p] ^= carry;
                carry = next;
            }
        }
        uint32_t out[8];
#pragma unroll
        for (int n = 0; n < 8; ++n) {                          // four entries: bit i of a plane's nibble to byte i
            out[n] = 0u;
#pragma unroll
            for (int p = 0; p < 5; ++p) out[n] |= ((((plane[p] >> (4 * n)) & 15u) * 0x00204081u) & 0x01010101u) << p;
        }
        uint4* dst = reinterpret_cast<uint4*>(a.df_table + static_cast<size_t>(w) * (kMode == kModeTable ? 64 : 32));
        if (kMode == kModeTable) {
#pragma unroll
            for (int n = 0; n < 4; ++n)
                dst[n] = make_uint4(__byte_perm(out[2 * n], 0u, 0x4140), __byte_perm(out[2 * n], 0u, 0x4342),
                                    __byte_perm(out[2 * n + 1], 0u, 0x4140), __byte_perm(out[2 * n + 1], 0u, 0x4342));
        } else {
            dst[0] = make_uint4(out[0], out[1], out[2], out[3]);
            dst[1] = make_uint4(out[4], out[5], out[6], out[7]);
        }
    }
    cluster_sync();                    // the table is complete, and no CTA reads another's set any more
    if constexpr (kMode == kModeTable) return;
    // The caller's tables, from this CTA's slice of the byte table: neighbouring threads write neighbouring entries, and the
    // logarithms are one per df.  (A thread that wrote its 32 entries out of the bit planes touched a sector per store: 128,256
    // entries of one block 207 us a call, 31 like this; of four blocks 54 and 12.)
    if (a.df_out != nullptr || a.idf_out != nullptr) {
        if (tid <= n_blocks) s_idf[tid] = logf(static_cast<float>(n_blocks) / static_cast<float>(tid > 0 ? tid : 1));
        __syncthreads();
        const int end = min(a.vocab_size, w_end * 32);
        constexpr int kBatch = 8;
        for (int i0 = b * per_cta * 32 + tid; i0 < end; i0 += kBatch * kClusterThreads) {
            uint32_t df[kBatch];
#pragma unroll
            for (int j = 0; j < kBatch; ++j) df[j] = i0 + j * kClusterThreads < end ? a.df_table[i0 + j * kClusterThreads] : 0u;
#pragma unroll
            for (int j = 0; j < kBatch; ++j) {
                const int i = i0 + j * kClusterThreads;
                if (i >= end) break;
                if (a.df_out != nullptr) a.df_out[i] = df[j];
                if (a.idf_out != nullptr) a.idf_out[i] = s_idf[df[j]];
            }
        }
    }
    const bool shifted = geo.tail != a.chunk && a.k > 0 && n_blocks > 1;       // a third barrier at the end, the same for all CTAs
    if (b >= n_blocks) {
        if (shifted) cluster_sync();
        return;
    }
    constexpr uint32_t kNoToken = 255;
    uint32_t mine_df[kPerThread];
#pragma unroll
    for (int j = 0; j < kPerThread; ++j)
        mine_df[j] = tid + j * kClusterThreads < len_b && mine_t[j] < V ? a.df_table[mine_t[j]] : kNoToken;
#pragma unroll
    for (int j = 0; j < kPerThread; ++j)
        if (tid + j * kClusterThreads < len_b) dfs[tid + j * kClusterThreads] = static_cast<uint8_t>(mine_df[j]);
    __syncthreads();

    // ---- a rank per chunk slot: its least df, or its score; see chunk_level_kernel and chunk_score_kernel ----
    const int k = geo.k_b;
    int* level = reinterpret_cast<int*>(smem_c + at.ranks);
    double* score = reinterpret_cast<double*>(smem_c + at.ranks);
    bool take;
    if constexpr (!kScores) {
        for (int c = warp; c < C; c += kClusterThreads / 32) {
            const int len = max(0, min(a.chunk, len_b - c * a.chunk));
            uint32_t least = static_cast<uint32_t>(len > 0 ? n_blocks + 1 : n_blocks + 2);
            for (int p = lane; p < len; p += 32) {
                const uint32_t df = dfs[c * a.chunk + p];
                if (df != kNoToken) least = min(least, df);
            }
            least = __reduce_min_sync(0xffffffffu, least);
            if (lane == 0) level[c] = static_cast<int>(least);
        }
        __syncthreads();
        for (int c0 = warp * 32; c0 < C; c0 += kClusterThreads) {                              // at most once
            const int own = c0 + lane < C ? level[c0 + lane] : -1;
            const uint32_t same = __match_any_sync(0xffffffffu, own);
            if (own >= 0 && lane == __ffs(same) - 1) atomicAdd(&s_hist[own], __popc(same));
        }
        __syncthreads();
        // threshold level: all chunks below it are taken, s_need more at it (lowest indices first)
        if (warp == 0) {
            int cum = s_hist[lane];
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int n = __shfl_up_sync(0xffffffffu, cum, o);
                if (lane >= o) cum += n;
            }
            const uint32_t enough = __ballot_sync(0xffffffffu, cum >= k);
            if (lane == __ffs(enough) - 1) {
                s_threshold = lane;
                s_need = k - (cum - s_hist[lane]);
            }
        }
        __syncthreads();
        const int mine = tid < C ? level[tid] : n_blocks + 3, T = s_threshold;
        const int rank_T = taken_before(mine == T, s_warp);
        take = mine < T || (mine == T && rank_T < s_need);
    } else {
        double* term = reinterpret_cast<double*>(smem_c + at.terms);
        const int stride = a.chunk | 1;
        for (int c = warp; c < C; c += kClusterThreads / 32) {
            const int len = max(0, min(a.chunk, len_b - c * a.chunk));
            const uint32_t* ct = tok + c * a.chunk;
            const uint8_t* cd = dfs + c * a.chunk;
            double* terms = term + c * stride;
            if (kMode == PULSAR_SCORE_MAX_IDF) {               // the largest IDF is that of the least df
                uint32_t least = kNoToken;
                for (int p = lane; p < len; p += 32) least = min(least, static_cast<uint32_t>(cd[p]));
                least = __reduce_min_sync(0xffffffffu, least);
                if (lane == 0) score[c] = least == kNoToken ? -CUDART_INF : tab.by_df[least];
                continue;
            }
            const int distinct = chunk_terms<kMode, kNoToken>(ct, len, tab, [&](int p, bool) { return cd[p]; }, terms);
            if (kMode == PULSAR_SCORE_TYPE_TOKEN && lane == 0) score[c] = static_cast<double>(distinct);
        }
        __syncthreads();
        if (kMode != PULSAR_SCORE_MAX_IDF && tid < C) {
            const int len = max(0, min(a.chunk, len_b - tid * a.chunk));
            double sum = kMode == PULSAR_SCORE_TYPE_TOKEN ? score[tid] : 0.0;
            if (kMode != PULSAR_SCORE_TYPE_TOKEN) {            // in the order of the equations
#pragma unroll 8
                for (int p = 0; p < len; ++p) sum = __dadd_rn(sum, term[tid * stride + p]);
            }
            score[tid] = len == 0 ? -CUDART_INF : kMode == PULSAR_SCORE_BM25 ? sum : __ddiv_rn(sum, static_cast<double>(len));
        }
        // How many chunks beat each (a larger score, or the same at a lower index), counted by as many threads as there are to a chunk.
        int* better = reinterpret_cast<int*>(term);            // [C]; the terms are used up
        __syncthreads();
        for (int c = tid; c < C; c += kClusterThreads) better[c] = 0;
        __syncthreads();
        const int Cb = (len_b + a.chunk - 1) / a.chunk, span = (C + 31) / 32 * 32, parts = kClusterThreads / span;
        const int part = tid / span, c = tid - part * span;
        if (part < parts && c < Cb) {
            const double mine = score[c];
            const int end = Cb * (part + 1) / parts, c_warp = c & ~31;
            int n = 0, o = Cb * part / parts;
#pragma unroll 4
            for (; o < min(end, c_warp); ++o) n += score[o] >= mine ? 1 : 0;                       // before every lane's own
            for (; o < min(end, c_warp + 32); ++o) n += (score[o] > mine || (score[o] == mine && o < c)) ? 1 : 0;
#pragma unroll 4
            for (; o < end; ++o) n += score[o] > mine ? 1 : 0;
            atomicAdd(&better[c], n);
        }
        if (a.score != nullptr)
            for (int i = tid; i < C; i += kClusterThreads) a.score[static_cast<size_t>(b) * C + i] = score[i];
        __syncthreads();
        take = tid < Cb && better[tid] < k;
    }
    const int pos = taken_before(take, s_warp);
    if (take && pos < k) {
        chosen[pos] = tid;
        a.sel_chunks[static_cast<size_t>(b) * a.k + pos] = tid;
    }
    // ---- the prefix list; its entries are shifted by earlier blocks that selected their short last chunk ----
    int offset = geo.sink_eff + b * a.k * a.chunk;
    if (shifted) {
        const uint32_t is_short = tid == C - 1 && take && len_b == a.block_size ? 1u : 0u;
        if (tid == C - 1)
            for (int j = 0; j < n_blocks; ++j) st_cluster_u32(smem_u32(s_short + b), j, is_short);
        cluster_sync();
        int n_short = 0;
        for (int j = 0; j < b; ++j) n_short += s_short[j];
        offset -= n_short * (a.chunk - geo.tail);
    }
    __syncthreads();
    write_block_prefix(b, n_blocks, a.block_size, a.chunk, a.k, geo, offset, chosen, a.sel_chunks, a.prefix_idx, a.prefix_len);
}

// Whether a cluster of that many CTAs can be resident on the current device, whatever its mode and shared memory (an SM holds one
// CTA of any).  A process that sees a part of the GPU, or a GPU with smaller clusters of SMs, takes the four launches.
bool cluster_fits(int ctas) {
    static std::atomic<signed char> known[64][kClusterBlocks + 1];     // per device; 0: not asked yet, else 1 or -1
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) {
        (void)cudaGetLastError();
        return false;
    }
    const signed char seen = known[dev][ctas].load(std::memory_order_relaxed);
    if (seen != 0) return seen > 0;
    auto kernel = select_cluster_kernel<kModeLevels>;
    const size_t smem = kMaxDynSmem - 2048;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(ctas);
    cfg.blockDim = dim3(kClusterThreads);
    cfg.dynamicSmemBytes = smem;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = static_cast<unsigned>(ctas);
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int n = 0;
    if (allow_smem(kernel, smem) != cudaSuccess ||
        cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess ||
        cudaOccupancyMaxActiveClusters(&n, kernel, &cfg) != cudaSuccess) {
        (void)cudaGetLastError();
        return false;
    }
    known[dev][ctas].store(n > 0 ? 1 : -1, std::memory_order_relaxed);
    return n > 0;
}

constexpr int kClusterDfWords = 4096, kClusterTableWords = 16384;       // of 32 entries: see the rules below
// CTAs of the cluster; 0 where none fits.  More than blocks where these are few, since the vocabulary is shared out among all: with a
// CTA per block one block took 13.4 us with 128,256 entries and 71 with a million (the four launches 5.8 and 10.5 on the device), with
// eight CTAs 5.7 and 13.3, with sixteen 5.4 and 9.5.  Up to 131,072 entries, unless the caller wants their tables as well (8.3 us
// with eight, 6.9 with sixteen), eight do: sixteen have to find an SM each in one GPC at the end of the launch before them, and
// a step of 4062 tokens in seven blocks takes 54.8 us instead of 54.3.
// shared: another launch wants the SMs meanwhile (pulsar_encode_step).  Then it is a CTA per block as long as each has 1024
// words of the vocabulary at most: 136 work items of Phase 2 beside the selection of 12 blocks found no SM for four of them beside
// sixteen CTAs, and the step took 37.5 us instead of 33.8.
int cluster_ctas(const SelectPlan& p, bool tables, bool shared) {
    if (p.n_blocks > kClusterBlocks) return 0;
    if (shared && p.words <= 1024 * p.n_blocks && cluster_fits(p.n_blocks)) return p.n_blocks;
    const bool eight = p.n_blocks <= 8 && p.words <= kClusterDfWords && !tables;
    if (!eight && cluster_fits(kClusterBlocks)) return kClusterBlocks;
    return p.n_blocks <= 8 && cluster_fits(8) ? 8 : 0;
}

// Whether a selection of this shape is the cluster's: at most 16 blocks that their CTAs get through in less time than the host
// takes for three launches more.  us a call in a row of them from Python, one launch / four, with the time on the device in brackets:
// levels, blocks of 128 to 6144 tokens, up to 500,000 entries 9.6-12.5 (5-12) / 16.8 (5-12); the caller's tables of 128,256 entries as
// well 13.9 (6.9-9.1) / 21.1 (5.8-8.5), of a million 31 (20) / 21.3 (12).  Scores, 16 blocks, one launch / three (see below): BM25,
// blocks of 1024 11.4 (8.0) / 17.6 (7.0), of 2048 11.4 (9.6) / 17.8 (7.5); the divisions of a block's terms are one SM's in one launch, as are
// the comparisons of a long chunk's positions: chunks of 64 in blocks of 2048 13.8 / 17.9, of 100 21.4 / 18.0, in blocks of
// 1024 16.2 / 17.7, of 512 in blocks of 1024 87 / 93; type-token ratio, chunks of 128 14.3 / 17.5, of 256 29.7 / 23.6.  (Where the
// host's launches cost nothing, in a graph, four launches are up to 4 us faster: 1024 chunks of two tokens a block 8.5 against 12.1.)
// Blocks and chunks above that share the df table's launch and have the scores formed by the whole chip, three launches instead of
// four: BM25 over blocks of 8192, 128,256 entries, 1 block 17.1 (9.9) / 19.5 (10.7), 16 blocks 17.3 (13.2) / 19.7 (14.7); with more
// entries the table costs the few CTAs more than the launch does: 500,000 18.3 (12.8) / 20.2 (12.6), a million 24.3 (17.4) / 19.8 (15.8).
constexpr int kClusterLevelTokens = 6144, kClusterScoreTokens = 2048;
bool cluster_table_takes(const SelectPlan& p, int32_t block_size) {
    return p.n_blocks <= kClusterBlocks && block_size <= kClusterTokens && p.words <= kClusterTableWords &&
           static_cast<size_t>(p.words) * 64 <= p.df_bytes &&
           ClusterShape(p.words, block_size, p.C, 1, 0, kModeTable).tokens <= kMaxDynSmem - 2048 && cluster_ctas(p, false, false) > 0;
}
// mode: a score or kModeLevels.  tables: the caller wants df or IDF.
bool cluster_takes(const SelectPlan& p, int32_t block_size, int32_t chunk, int32_t k, int mode, bool tables) {
    const bool scores = mode != kModeLevels;
    if (p.n_blocks > kClusterBlocks || block_size > (scores ? kClusterScoreTokens : kClusterLevelTokens) || p.C > kClusterChunks) return false;
    if (tables && p.words > kClusterDfWords) return false;
    if (mode == PULSAR_SCORE_BM25 && chunk > 64 && block_size > 1024) return false;
    if (mode == PULSAR_SCORE_TYPE_TOKEN && chunk > 128) return false;
    return ClusterShape(p.words, block_size, p.C, chunk, k, mode).total <= kMaxDynSmem - 2048 &&
           static_cast<size_t>(p.words) * 32 <= p.df_bytes && cluster_ctas(p, tables, false) > 0;
}

template <int kMode, typename Table>
cudaError_t launch_cluster(const SelectPlan& p, const ClusterArgs& args, const Table& tab, cudaStream_t stream, bool shared = false) {
    const ClusterShape shape(p.words, args.block_size, p.C, args.chunk, args.k, kMode);
    const size_t smem = kMode == kModeTable ? shape.tokens : shape.total;
    auto kernel = select_cluster_kernel<kMode>;
    cudaError_t e = allow_smem(kernel, smem);
    const int ctas = cluster_ctas(p, args.df_out != nullptr || args.idf_out != nullptr, shared);
    if (e == cudaSuccess && ctas > 8) e = cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(ctas);
    cfg.blockDim = dim3(kClusterThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = static_cast<unsigned>(ctas);
    attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    return cudaLaunchKernelEx(&cfg, kernel, args, tab);
}

}  // namespace
}  // namespace pulsar

using namespace pulsar;

extern "C" size_t pulsar_maxidf_select_workspace_bytes(int64_t L, int32_t vocab_size, int32_t block_size,
                                                       int32_t chunk, int32_t k, int32_t sink) {
    SelectPlan p;
    if (plan_select(L, vocab_size, block_size, chunk, k, sink, p) != PULSAR_OK) return 0;
    return p.total;
}

int32_t pulsar::launch_maxidf_select(const uint32_t* token_ids, int64_t L, int32_t vocab_size, int32_t block_size, int32_t chunk,
                                     int32_t k, int32_t sink, int32_t* sel_chunks, int32_t* prefix_idx, int32_t* prefix_len,
                                     uint32_t* df_out, float* idf_out, void* workspace, size_t workspace_bytes,
                                     int32_t* device_status, void* stream_, bool shared) {
    SelectPlan p;
    int32_t rc = plan_select(L, vocab_size, block_size, chunk, k, sink, p);
    if (rc != PULSAR_OK) return rc;
    if (!token_ids || !sel_chunks || !prefix_idx || !prefix_len || !workspace) return PULSAR_ERR_INVALID_ARG;
    if (!aligned(token_ids, 16) || !aligned(sel_chunks, 16) || !aligned(prefix_idx, 16) || !aligned(prefix_len, 16) ||
        (df_out && !aligned(df_out, 16)) || (idf_out && !aligned(idf_out, 16)) || !aligned(workspace, 256))
        return PULSAR_ERR_ALIGNMENT;
    if (workspace_bytes < p.total) return PULSAR_ERR_WORKSPACE;
    rc = check_device();
    if (rc != PULSAR_OK) return rc;
    cudaStream_t stream = static_cast<cudaStream_t>(stream_);

    if (cluster_takes(p, block_size, chunk, k, kModeLevels, df_out != nullptr || idf_out != nullptr)) {
        const ClusterArgs args{token_ids, L, p.n_blocks, block_size, chunk, k, sink, vocab_size, p.words,
                               static_cast<uint8_t*>(workspace) + p.bitmap_bytes, sel_chunks, prefix_idx, prefix_len, df_out, idf_out,
                               nullptr, device_status};
        PULSAR_CUDA_OK(launch_cluster<kModeLevels>(p, args, 0, stream, shared));
        count_launch();
        return PULSAR_OK;
    }
    uint32_t* bitmaps = static_cast<uint32_t*>(workspace);
    uint16_t* df_table = reinterpret_cast<uint16_t*>(static_cast<char*>(workspace) + p.bitmap_bytes);
    uint16_t* level = reinterpret_cast<uint16_t*>(static_cast<char*>(workspace) + p.bitmap_bytes + p.df_bytes);

    PULSAR_CUDA_OK(allow_smem(presence_kernel, p.presence_smem));
    PULSAR_CUDA_OK(allow_smem(topk_kernel, p.topk_smem));
    PULSAR_CUDA_OK(launch_kernel(presence_kernel, dim3(p.n_blocks), dim3(kPresenceThreads), p.presence_smem, stream, true,
                                 token_ids, L, block_size, vocab_size, p.words, bitmaps, device_status));
    count_launch();
    // The three launches that follow are programmatic dependents of the one before them: they are placed
    // while it runs and wait for it on the device, which takes the launch gaps out of the chain.
    PULSAR_CUDA_OK(launch_kernel(df_idf_kernel, dim3((vocab_size + 255) / 256), dim3(256), 0, stream, true, bitmaps,
                                 p.n_blocks, p.words, vocab_size, df_table, df_out, idf_out));
    count_launch();
    const int n_chunks_total = p.n_blocks * p.C;
    PULSAR_CUDA_OK(launch_kernel(chunk_level_kernel, dim3((n_chunks_total + 7) / 8), dim3(256), 0, stream, true, token_ids,
                                 df_table, L, block_size, p.C, n_chunks_total, chunk, vocab_size, p.n_blocks + 1, level));
    count_launch();
    PULSAR_CUDA_OK(launch_kernel(topk_kernel, dim3(p.n_blocks), dim3(kTopkThreads), p.topk_smem, stream, true, level,
                                 p.n_blocks, L, block_size, chunk, k, sink, sel_chunks, prefix_idx, prefix_len));
    count_launch();
    return PULSAR_OK;
}

extern "C" int32_t pulsar_maxidf_select(const uint32_t* token_ids, int64_t L, int32_t vocab_size,
                                        int32_t block_size, int32_t chunk, int32_t k, int32_t sink,
                                        int32_t* sel_chunks, int32_t* prefix_idx, int32_t* prefix_len,
                                        uint32_t* df_out, float* idf_out, void* workspace,
                                        size_t workspace_bytes, int32_t* device_status, void* stream) {
    return launch_maxidf_select(token_ids, L, vocab_size, block_size, chunk, k, sink, sel_chunks, prefix_idx, prefix_len, df_out, idf_out,
                                workspace, workspace_bytes, device_status, stream, false);
}

// =============================================================================================
// Selection under a chosen chunk score
// =============================================================================================
namespace {
struct ScorePlan {
    SelectPlan base;
    size_t score_bytes, total, topk_smem;
};
int32_t plan_score(int64_t L, int32_t vocab_size, int32_t block_size, int32_t chunk, int32_t k, int32_t sink,
                   int32_t mode, ScorePlan& p) {
    if (mode < PULSAR_SCORE_MAX_IDF || mode > PULSAR_SCORE_TYPE_TOKEN) return PULSAR_ERR_INVALID_ARG;
    int32_t rc = plan_select(L, vocab_size, block_size, chunk, k, sink, p.base);
    if (rc != PULSAR_OK) return rc;
    if (p.base.n_blocks > kMaxScoreBlocks || chunk > kMaxScoreChunk || p.base.C > kMaxScoreChunksPerBlock)
        return PULSAR_ERR_SHAPE;
    p.score_bytes = round_up(static_cast<size_t>(p.base.n_blocks) * p.base.C * 8, 256);
    p.total = p.base.bitmap_bytes + p.base.df_bytes + p.score_bytes;
    p.topk_smem = static_cast<size_t>(p.base.C) * 8 + static_cast<size_t>(k) * 4;
    return PULSAR_OK;
}

template <int kBlocks>
ScoreTable<kBlocks> score_table(const SelectPlan& b, int32_t score_mode, int64_t L, int32_t block_size, int32_t chunk) {
    // The logarithms of Eq. 5 / Eq. 7 for every possible df, in float64 from the host's libm.
    ScoreTable<kBlocks> tab;
    const double N = static_cast<double>(b.n_blocks);
    for (int f = 0; f <= b.n_blocks; ++f) {
        const double fd = static_cast<double>(f);
        tab.by_df[f] = score_mode == PULSAR_SCORE_BM25 ? std::log((N - fd + 0.5) / (fd + 0.5) + 1.0)
                                                       : std::log(N / static_cast<double>(f > 1 ? f : 1));
    }
    const double k1 = 1.2, bb = 0.75;
    // mean chunk length over the sequence: full blocks have C chunks, a short last block what it needs
    const int64_t last_len = L - static_cast<int64_t>(b.n_blocks - 1) * block_size;
    const int64_t n_chunks = static_cast<int64_t>(b.n_blocks - 1) * b.C + (last_len + chunk - 1) / chunk;
    tab.k1_plus_1 = k1 + 1.0;
    tab.k1 = k1;
    tab.b = bb;
    tab.one_minus_b = 1.0 - bb;
    tab.mean_len = static_cast<double>(L) / static_cast<double>(n_chunks);
    return tab;
}

template <int kBlocks>
cudaError_t launch_scores(const SelectPlan& b, int32_t score_mode, const uint32_t* token_ids, const uint16_t* df_table, int64_t L,
                          int32_t block_size, int32_t chunk, int32_t vocab_size, double* score, cudaStream_t stream) {
    const ScoreTable<kBlocks> tab = score_table<kBlocks>(b, score_mode, L, block_size, chunk);
    const int n_chunks_total = b.n_blocks * b.C;
    if (chunk <= kThreadFormChunk && n_chunks_total >= kThreadFormSlots) {
        auto kernel = score_mode == PULSAR_SCORE_MAX_IDF ? chunk_score_thread_kernel<PULSAR_SCORE_MAX_IDF, kBlocks>
                    : score_mode == PULSAR_SCORE_TF_IDF  ? chunk_score_thread_kernel<PULSAR_SCORE_TF_IDF, kBlocks>
                    : score_mode == PULSAR_SCORE_BM25    ? chunk_score_thread_kernel<PULSAR_SCORE_BM25, kBlocks>
                                                         : chunk_score_thread_kernel<PULSAR_SCORE_TYPE_TOKEN, kBlocks>;
        return launch_kernel(kernel, dim3((n_chunks_total + 127) / 128), dim3(128), 0, stream, true, token_ids, df_table, L,
                             block_size, b.C, n_chunks_total, chunk, vocab_size, tab, score);
    }
    auto kernel = score_mode == PULSAR_SCORE_MAX_IDF ? chunk_score_kernel<PULSAR_SCORE_MAX_IDF, kBlocks>
                : score_mode == PULSAR_SCORE_TF_IDF  ? chunk_score_kernel<PULSAR_SCORE_TF_IDF, kBlocks>
                : score_mode == PULSAR_SCORE_BM25    ? chunk_score_kernel<PULSAR_SCORE_BM25, kBlocks>
                                                     : chunk_score_kernel<PULSAR_SCORE_TYPE_TOKEN, kBlocks>;
    const size_t smem = static_cast<size_t>(kScoreWarps) * chunk * (sizeof(double) + sizeof(uint32_t));
    return launch_kernel(kernel, dim3((n_chunks_total + kScoreWarps - 1) / kScoreWarps), dim3(kScoreWarps * 32), smem, stream,
                         true, token_ids, df_table, L, block_size, b.C, n_chunks_total, chunk, vocab_size, tab, score);
}
}  // namespace

extern "C" size_t pulsar_chunk_select_workspace_bytes(int64_t L, int32_t vocab_size, int32_t block_size,
                                                      int32_t chunk, int32_t k, int32_t sink, int32_t score_mode) {
    ScorePlan p;
    if (plan_score(L, vocab_size, block_size, chunk, k, sink, score_mode, p) != PULSAR_OK) return 0;
    return p.total;
}

extern "C" int32_t pulsar_chunk_select(const uint32_t* token_ids, int64_t L, int32_t vocab_size, int32_t block_size,
                                       int32_t chunk, int32_t k, int32_t sink, int32_t score_mode,
                                       int32_t* sel_chunks, int32_t* prefix_idx, int32_t* prefix_len,
                                       double* score_out, void* workspace, size_t workspace_bytes,
                                       int32_t* device_status, void* stream_) {
    ScorePlan p;
    int32_t rc = plan_score(L, vocab_size, block_size, chunk, k, sink, score_mode, p);
    if (rc != PULSAR_OK) return rc;
    if (!token_ids || !sel_chunks || !prefix_idx || !prefix_len || !workspace) return PULSAR_ERR_INVALID_ARG;
    if (!aligned(token_ids, 16) || !aligned(sel_chunks, 16) || !aligned(prefix_idx, 16) || !aligned(prefix_len, 16) ||
        (score_out && !aligned(score_out, 16)) || !aligned(workspace, 256))
        return PULSAR_ERR_ALIGNMENT;
    if (workspace_bytes < p.total) return PULSAR_ERR_WORKSPACE;
    rc = check_device();
    if (rc != PULSAR_OK) return rc;
    cudaStream_t stream = static_cast<cudaStream_t>(stream_);
    const SelectPlan& b = p.base;

    if (cluster_takes(b, block_size, chunk, k, score_mode, false)) {
        const ClusterArgs args{token_ids, L, b.n_blocks, block_size, chunk, k, sink, vocab_size, b.words,
                               static_cast<uint8_t*>(workspace) + b.bitmap_bytes, sel_chunks, prefix_idx, prefix_len, nullptr, nullptr,
                               score_out, device_status};
        const auto tab = score_table<kClusterBlocks>(b, score_mode, L, block_size, chunk);
        PULSAR_CUDA_OK(score_mode == PULSAR_SCORE_MAX_IDF ? launch_cluster<PULSAR_SCORE_MAX_IDF>(b, args, tab, stream)
                       : score_mode == PULSAR_SCORE_TF_IDF ? launch_cluster<PULSAR_SCORE_TF_IDF>(b, args, tab, stream)
                       : score_mode == PULSAR_SCORE_BM25   ? launch_cluster<PULSAR_SCORE_BM25>(b, args, tab, stream)
                                                           : launch_cluster<PULSAR_SCORE_TYPE_TOKEN>(b, args, tab, stream));
        count_launch();
        return PULSAR_OK;
    }
    uint32_t* bitmaps = static_cast<uint32_t*>(workspace);
    uint16_t* df_table = reinterpret_cast<uint16_t*>(static_cast<char*>(workspace) + b.bitmap_bytes);
    double* score = score_out ? score_out
                              : reinterpret_cast<double*>(static_cast<char*>(workspace) + b.bitmap_bytes + b.df_bytes);

    if (cluster_table_takes(b, block_size)) {
        const ClusterArgs args{token_ids, L, b.n_blocks, block_size, chunk, k, sink, vocab_size, b.words, reinterpret_cast<uint8_t*>(df_table),
                               nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, device_status};
        PULSAR_CUDA_OK(launch_cluster<kModeTable>(b, args, 0, stream));
        count_launch();
    } else {
        PULSAR_CUDA_OK(allow_smem(presence_kernel, b.presence_smem));
        PULSAR_CUDA_OK(launch_kernel(presence_kernel, dim3(b.n_blocks), dim3(kPresenceThreads), b.presence_smem, stream, true,
                                     token_ids, L, block_size, vocab_size, b.words, bitmaps, device_status));
        count_launch();
        PULSAR_CUDA_OK(launch_kernel(df_idf_kernel, dim3((vocab_size + 255) / 256), dim3(256), 0, stream, true, bitmaps,
                                     b.n_blocks, b.words, vocab_size, df_table, nullptr, nullptr));
        count_launch();
    }
    // Programmatic dependents of the launch before them, as in pulsar_maxidf_select.
    PULSAR_CUDA_OK(b.n_blocks <= kFewScoreBlocks
                       ? launch_scores<kFewScoreBlocks>(b, score_mode, token_ids, df_table, L, block_size, chunk, vocab_size, score, stream)
                       : launch_scores<kMaxScoreBlocks>(b, score_mode, token_ids, df_table, L, block_size, chunk, vocab_size, score, stream));
    count_launch();
    PULSAR_CUDA_OK(launch_kernel(topk_score_kernel, dim3(b.n_blocks), dim3(kTopkThreads), p.topk_smem, stream, true, score,
                                 b.n_blocks, L, block_size, chunk, k, sink, sel_chunks, prefix_idx, prefix_len));
    count_launch();
    return PULSAR_OK;
}

// =============================================================================================
// Selection without a caller workspace
// =============================================================================================
namespace {

// Scratch shared by every pulsar_maxidf_select_noalloc call on a device.  It is part of the
// library image: each GPU that loads the library holds these bytes until the process exits.
constexpr size_t kStaticScratchBytes = 4u << 20;
static __device__ __align__(256) unsigned char g_select_scratch[kStaticScratchBytes];

constexpr int kMaxDevices = 64;
std::mutex g_scratch_mutex;
void* g_scratch_ptr[kMaxDevices] = {};

// Device address of g_select_scratch on the current device.  In host code the symbol's name is
// only a stand-in; the address a kernel can use comes from cudaGetSymbolAddress, looked up once
// per device with that device current and remembered for the life of the process.  (A device
// reset, or a primary context torn down and created again, would leave the remembered address
// stale: the header tells callers not to use this entry point across one.)
int32_t static_scratch(void** out) {
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) {
        (void)cudaGetLastError();
        return PULSAR_ERR_CUDA;
    }
    std::lock_guard<std::mutex> lock(g_scratch_mutex);
    if (g_scratch_ptr[dev] == nullptr) {
        void* p = nullptr;
        if (cudaGetSymbolAddress(&p, g_select_scratch) != cudaSuccess || p == nullptr) {
            (void)cudaGetLastError();
            return PULSAR_ERR_CUDA;
        }
        g_scratch_ptr[dev] = p;
    }
    *out = g_scratch_ptr[dev];
    return PULSAR_OK;
}

}  // namespace

extern "C" size_t pulsar_maxidf_select_noalloc_max_scratch(void) { return kStaticScratchBytes; }

extern "C" int32_t pulsar_maxidf_select_noalloc(const uint32_t* token_ids, int64_t L, int32_t vocab_size,
                                                int32_t block_size, int32_t chunk, int32_t k, int32_t sink,
                                                int32_t* sel_chunks, int32_t* prefix_idx, int32_t* prefix_len,
                                                uint32_t* df_out, float* idf_out, int32_t* device_status,
                                                void* stream) {
    SelectPlan p;
    int32_t rc = plan_select(L, vocab_size, block_size, chunk, k, sink, p);
    if (rc != PULSAR_OK) return rc;
    if (p.total > kStaticScratchBytes) return PULSAR_ERR_WORKSPACE;      // problem too large for the built-in scratch
    rc = check_device();
    if (rc != PULSAR_OK) return rc;
    void* scratch = nullptr;
    rc = static_scratch(&scratch);
    if (rc != PULSAR_OK) return rc;
    // Same kernels, same order as pulsar_maxidf_select; every scratch region is fully written
    // before it is read, so nothing needs clearing between calls.
    return pulsar_maxidf_select(token_ids, L, vocab_size, block_size, chunk, k, sink, sel_chunks, prefix_idx,
                                prefix_len, df_out, idf_out, scratch, kStaticScratchBytes, device_status, stream);
}
