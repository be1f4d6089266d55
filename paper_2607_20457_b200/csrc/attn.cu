// Phase-1 prefix-block attention and Phase-2 split-KV attention (Eq. 1 over Eq. 4; Section 3.2).
//
// One FlashAttention-form kernel serves both phases.  A CTA owns a tile of 128 query rows and
// walks a list of 128-key tiles: S = Q K^T and O += P V run on the tensor cores (tcgen05.mma,
// accumulators in TMEM), operands are staged by TMA into 128-byte-swizzled shared memory, the
// softmax runs one thread per query row straight out of TMEM, and the probabilities go back to
// TMEM as the bf16 A operand of the PV product.
//
//   Phase 1: rows = 128 consecutive tokens of one block and one query head.  Key tiles: first
//            the gathered prefix rows [0, P_i) (fully visible, last tile possibly partial), then
//            the block's own rows up to the diagonal tile (causal mask on that tile only).
//   Phase 2: rows = (128/g tokens) x (the g query heads of one KV head); key tiles = one
//            contiguous part of the retained KV, no mask; output is the fp32 partial (A_j, l_j)
//            or, with a single part, the final bf16 result.  With at most 32 such rows (decode; up to
//            eight against a long context are decode.cu's) the rows are replicated into the four lane quarters of the tile and each softmax
//            warp takes a quarter of the keys; the generation shard of Algorithm 1 l.11-16, causal by
//            token, is one more part or stands in front of the last part's context keys.
//   Assembled inputs (Algorithm 1 l.8 as the paper runs it): sequences of any lengths packed back
//            to back, every token a query, plain causal attention inside each.
#include <algorithm>
#include <functional>
#include <type_traits>

#include <cuda.h>

#include "common.cuh"
#include "decode.cuh"

namespace pulsar {

namespace {

constexpr int kTileM = 128;   // query rows per CTA
constexpr int kTileN = 128;   // keys per tile
constexpr int kPanelBytes = kTileN * 128;   // one 64-column panel of a 128-row bf16 tile (128-byte lines)

enum : int { kModePhase1 = 0, kModePhase2 = 1, kModeVarlen = 2 };

// Sequence table of the variable-length causal mode (passed by value with the launch).
constexpr int kMaxVarlenSeqs = 64;
struct VarlenTable {
    int start[kMaxVarlenSeqs + 1];      // first row of sequence j; start[n] = total rows
    int pair_cum[kMaxVarlenSeqs + 1];   // work items per head of the sequences n-1, n-2, ... j summed (scheduling order)
    int n_seq;
};

// Stands in for the table in the decode-shaped instance, which has no sequences (a kilobyte of parameters costs a
// launch about 1.2 us on the host).
struct NoTable {
    int start[1], pair_cum[1], n_seq;
};

struct AttnArgs {
    int mode;
    int n_tokens;          // L (phase 1) or nq (phase 2): tokens that exist, for the store guard
    int Hq, g;             // query heads, heads per KV head
    int pack_shift;        // log2 of the rows a token has in a tile (1, or the g heads of one KV head)
    int block_size;        // phase 1: tokens per block
    int prefix_total;      // phase 1: rows in the gathered prefix buffers
    const int32_t* prefix_len;
    int split_len;         // phase 2: keys per KV part (the last part may be shorter)
    int kv_len;            // phase 2: context keys in total
    int ctx_part0;         // phase 2: the first part with context keys (1 where part 0 is the generation shard)
    int gen_part;          // phase 2: the part that has the generation shard in front of its context keys (if any)
    int gen_len;           // phase 2: rows of the generation shard that precede the new tokens
    int gen_total;         // phase 2: gen_len + new tokens (0 = no generation shard)
    const uint4* Knew;     // phase 2, one query tile per KV head and few new tokens: their KV(q), appended to the generation
    const uint4* Vnew;     // shard by the CTA that reads the head's part of it (null: appended by a launch of its own)
    uint4* Kgen;
    uint4* Vgen;
    int quad;              // phase 2, at most 32 query rows per KV head: the rows are replicated into the four
                           // lane quarters of the tile and each softmax warp takes one quarter of the keys
    int tile_max;          // phase 2: P of a key tile is formed with that tile's own maximum (see cut_generate, next_max)
    int single;            // work items of one query tile: the tile's logits alternate between the two S buffers so
                           // that S of the next key tile is formed during the softmax of this one.  Phase 2 with
                           // one query tile per KV head (set with quad as well), causal attention with few items
    int Hkv;
    int pairs;             // phase 1: work items (query-tile pairs, or tiles if single) per full block and head;
                           // phase 2: per KV head and part
    int last_len;          // phase 1: tokens of the last block (block_size unless the sequence ends inside it)
    int pairs_last;        // phase 1: the same for the last block
    int n_items;           // work items in total
    int n_blocks;          // phase 1
    int32_t* counter;      // work counter (zeroed before the launch): items are drawn in index order as CTAs
                           // become free; null = fixed round order
    float scale_log2;      // softmax scale * log2(e)
    uint16_t* O;           // bf16 [tokens, Hq, d]   (final output mode)
    float* LSE;            // f32  [tokens, Hq] or null
    float* part_O;         // f32  [parts, tokens, Hq, d] (partial output mode) or null
    float* part_LSE;       // f32  [parts, tokens, Hq]
    int beside;            // phase 2: see launch_lse_merge
    int out_wide;          // the base of O (or part_O) is 32-byte aligned
    int32_t* status;
};

// ---------------------------------------------------------------------------------------------
// Gather of the prefix rows: Kp[j] = K[prefix_idx[j]], Vp[j] = V[prefix_idx[j]] for j < total.
// One CTA per prefix row; also checks that the row lies before the first block that uses it.  CTA 0 clears the
// attention launch's work counter (a memset between the two launches would cost a launch of its own).
// ---------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(128)
gather_prefix_kernel(const uint4* __restrict__ K, const uint4* __restrict__ V, const int32_t* __restrict__ prefix_idx,
                     const int32_t* __restrict__ prefix_len, int n_blocks, int block_size, int64_t L,
                     int row_vecs, uint4* __restrict__ Kp, uint4* __restrict__ Vp, int32_t* counter, int32_t* status) {
    const int j = blockIdx.x;
    __shared__ int s_src;
    grid_dependency_wait();                 // the prefix list may come from the launch before this one
    grid_launch_dependents();
    if (threadIdx.x < 32) {
        if (threadIdx.x == 0 && j == 0) *counter = 0;
        const int entry = prefix_idx[j];
        int64_t limit = -1;                 // stays -1 when no block uses entry j (the list may be shorter than its buffer)
        for (int i0 = 0; i0 < n_blocks && limit < 0; i0 += 32) {               // the first block that does, 32 at a time
            const int i = i0 + static_cast<int>(threadIdx.x);
            const uint32_t uses = __ballot_sync(0xffffffffu, i < n_blocks && prefix_len[i] > j);
            if (uses != 0u) limit = static_cast<int64_t>(i0 + __ffs(uses) - 1) * block_size;
        }
        if (threadIdx.x == 0) {
            int src = -1;
            if (limit >= 0) {
                src = entry;
                if (src < 0 || src >= limit) {
                    report(status, PULSAR_DEV_BAD_PREFIX);
                    src = 0;
                }
            }
            s_src = src;
        }
    }
    __syncthreads();
    const size_t dst = static_cast<size_t>(j) * row_vecs;
    if (s_src < 0) {
        // An entry no block uses still shares a key tile with used ones: the attention kernel masks
        // its logits, but the PV product multiplies whatever the row holds by zero, and 0 * NaN
        // is NaN.  The workspace is the caller's and may hold anything, so the row is cleared.
        for (int v = threadIdx.x; v < row_vecs; v += blockDim.x) {
            Kp[dst + v] = make_uint4(0u, 0u, 0u, 0u);
            Vp[dst + v] = make_uint4(0u, 0u, 0u, 0u);
        }
        return;
    }
    const size_t src = static_cast<size_t>(s_src) * row_vecs;
    for (int v = threadIdx.x; v < row_vecs; v += blockDim.x) {
        Kp[dst + v] = K[src + v];
        Vp[dst + v] = V[src + v];
    }
}

// The work counter of an attention launch, cleared by a launch before it.  A memset there takes the chain apart: an assembled
// input of 22,080 rows of 8 heads, d = 64, 127.1 -> 125.0 us, one of two GPUs' 19,264 tokens 101.6 -> 99.2.  (Dependents are let in
// after the wait: attention CTAs that take their SMs before the launch before this one is done cost 1-5 %.)
__global__ void clear_counter_kernel(int32_t* counter) {
    grid_dependency_wait();
    grid_launch_dependents();
    *counter = 0;
}

// KV(q) of the new tokens appended to the generation shard: one launch for both tensors, for calls with more than
// one query tile per KV head or with many new tokens (otherwise the attention kernel appends: append_head).
__global__ void __launch_bounds__(256)
append_kv_kernel(const uint4* __restrict__ Knew, const uint4* __restrict__ Vnew, uint4* __restrict__ Kdst,
                 uint4* __restrict__ Vdst, int vecs) {
    grid_dependency_wait();
    grid_launch_dependents();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < vecs) {
        Kdst[i] = Knew[i];
        Vdst[i] = Vnew[i];
    }
}

// KV discard (Section 3.1, Appendix F): of every assembled input only the last block_size rows -- the
// block's own keys and values -- are kept.  first[j] = first kept row of input j.  What is kept of an input is one run of
// memory, copied as such, four vectors of K and of V under way per thread.  HBM-bound; a CTA of 128 threads per row left seven
// in eight idle where a row has 16 vectors (us: 53,504 rows of 2 x 64 30.8 -> 5.9, 20,736 of 2 x 64 14.4 -> 5.5, 20,480 of 8 x 128 28.7 -> 26.8, in cache).
struct RetainTable {
    int first[kMaxVarlenSeqs];
};
constexpr int kCopyThreads = 256, kCopyUnroll = 4;
constexpr int64_t kCopyVecs = kCopyThreads * kCopyUnroll;                    // of a CTA
__global__ void __launch_bounds__(kCopyThreads)
retain_block_kv_kernel(const uint4* __restrict__ K, const uint4* __restrict__ V, const __grid_constant__ RetainTable tab,
                       int block_size, int row_vecs, uint4* __restrict__ Kret, uint4* __restrict__ Vret) {
    grid_dependency_wait();
    grid_launch_dependents();
    const int j = blockIdx.y;
    const int64_t n = static_cast<int64_t>(block_size) * row_vecs;           // vectors of an input that are kept
    const int64_t src = static_cast<int64_t>(tab.first[j]) * row_vecs, dst = j * n;
    const int64_t i0 = blockIdx.x * kCopyVecs + threadIdx.x;
    uint4 k[kCopyUnroll], v[kCopyUnroll];
#pragma unroll
    for (int u = 0; u < kCopyUnroll; ++u)
        if (i0 + u * kCopyThreads < n) {
            k[u] = K[src + i0 + u * kCopyThreads];
            v[u] = V[src + i0 + u * kCopyThreads];
        }
#pragma unroll
    for (int u = 0; u < kCopyUnroll; ++u)
        if (i0 + u * kCopyThreads < n) {
            Kret[dst + i0 + u * kCopyThreads] = k[u];
            Vret[dst + i0 + u * kCopyThreads] = v[u];
        }
}

// Rows of K and V copied to consecutive ones of Kout and Vout: a thread moves four vectors of each, so that a CTA covers the
// rows that its vectors come to and waits for the launch before it once for all of them.  (A CTA of 128 threads per row, as dependents
// of the launch before them: 13,235 rows of 8 x 64 14.6 us, 10.3 as plain launches, 6.4 like this.)
// row_of(j): the source row of row j, found once for each of the CTA's rows (for every vector, packing few rows 3.5 us instead of 2.9).
template <typename RowOf>
__device__ __forceinline__ void copy_rows(const uint4* __restrict__ K, const uint4* __restrict__ V, uint4* __restrict__ Kout,
                                          uint4* __restrict__ Vout, int64_t n_rows, int row_vecs, RowOf row_of) {
    __shared__ int s_src[kCopyVecs + 1];                                     // (a vector per row, and a row begun before)
    const int64_t base = blockIdx.x * kCopyVecs, j0 = base / row_vecs, left = n_rows * row_vecs - base;
    const uint32_t r0 = static_cast<uint32_t>(base - j0 * row_vecs), n = static_cast<uint32_t>(min(left, kCopyVecs));    // vectors from base on
    for (uint32_t j = threadIdx.x; j * row_vecs < r0 + n; j += kCopyThreads) s_src[j] = row_of(j0 + j);
    __syncthreads();
    uint4 k[kCopyUnroll], v[kCopyUnroll];
#pragma unroll
    for (int u = 0; u < kCopyUnroll; ++u) {
        const uint32_t i = threadIdx.x + u * kCopyThreads, j = (r0 + i) / row_vecs;
        if (i < n) {
            const int64_t src = static_cast<int64_t>(s_src[j]) * row_vecs + (r0 + i - j * row_vecs);
            k[u] = K[src];
            v[u] = V[src];
        }
    }
#pragma unroll
    for (int u = 0; u < kCopyUnroll; ++u) {
        const uint32_t i = threadIdx.x + u * kCopyThreads;
        if (i < n) {
            Kout[base + i] = k[u];
            Vout[base + i] = v[u];
        }
    }
}
unsigned copy_ctas(int64_t n_rows, int row_vecs) { return static_cast<unsigned>((n_rows * row_vecs + kCopyVecs - 1) / kCopyVecs); }

// Row gather without the prefix check: Kout[j] = K[idx[j]], Vout[j] = V[idx[j]].  An index outside
// [0, rows_in) is reported and row 0 used.
__global__ void __launch_bounds__(kCopyThreads)
gather_rows_kernel(const uint4* __restrict__ K, const uint4* __restrict__ V, const int32_t* __restrict__ idx, int n_idx,
                   int64_t rows_in, int row_vecs, uint4* __restrict__ Kout, uint4* __restrict__ Vout,
                   int32_t* status) {
    grid_dependency_wait();
    grid_launch_dependents();
    copy_rows(K, V, Kout, Vout, n_idx, row_vecs, [&](int64_t j) {
        const int src_row = idx[j];
        if (src_row >= 0 && src_row < rows_in) return src_row;
        report(status, PULSAR_DEV_BAD_PREFIX);
        return 0;
    });
}

// What one GPU contributes to the prefix exchange: row j < sink is row j of its first local block
// (meaningful only on the GPU that holds logical block 0); row sink + (s*k + c)*chunk + p is token
// p of the c-th selected chunk of local block s (logical block block_ids[s]).
__global__ void __launch_bounds__(kCopyThreads)
pack_summary_kernel(const uint4* __restrict__ K, const uint4* __restrict__ V, const int32_t* __restrict__ sel_chunks,
                    const int32_t* __restrict__ block_ids, int n_local, int n_blocks, int block_size, int chunk,
                    int k, int sink, int row_vecs, uint4* __restrict__ Kout, uint4* __restrict__ Vout,
                    int32_t* status) {
    grid_dependency_wait();
    grid_launch_dependents();
    copy_rows(K, V, Kout, Vout, sink + static_cast<int64_t>(n_local) * k * chunk, row_vecs, [&](int64_t row) {
        const int j = static_cast<int>(row);
        if (j < sink) return j;
        const int t = j - sink, sigma = k * chunk;
        const int s = t / sigma, r = t - s * sigma;
        const int c = r / chunk, p = r - c * chunk;
        const int blk = block_ids[s];
        int ch = 0;
        if (blk < 0 || blk >= n_blocks) {
            report(status, PULSAR_DEV_BAD_PREFIX);
        } else {
            ch = sel_chunks[static_cast<size_t>(blk) * k + c];
            if (ch < 0 || (ch + 1) * chunk > block_size) {
                report(status, PULSAR_DEV_BAD_PREFIX);
                ch = 0;
            }
        }
        return s * block_size + ch * chunk + p;
    });
}

// ---------------------------------------------------------------------------------------------
// Attention kernel: persistent, warp-specialised.
//
//   warps 0-3   softmax of query tile 0 (one thread per query row, TMEM lane = row)
//   warps 4-7   softmax of query tile 1 (of the other half of the keys where an item has one tile: kHalves)
//   warp  8     MMA issuer (one elected lane): S_s = Q_s K^T, O_s += P_s V
//   warp  9     TMA loader (one elected lane): Q tiles and the K/V ring
//
// A work item is two 128-row query tiles sharing one list of 128-key tiles.  The two tiles
// ping-pong on the tensor pipe: while the softmax warpgroup of one tile works on S, the pipe
// runs the other tile's PV and next S.  TMEM: S0 [0,128) S1 [128,256) O0 [256,384) O1 [384,512);
// P_s (bf16 pairs) overwrites the first 64 columns of S_s.  The running maximum is only moved
// when a logit exceeds it by more than 2^8, in the first 96 keys of a tile when their probabilities sum to more than
// 96 * 2^8 (kPieceSumBound: one of them may reach 2^14.6).  The stale maximum is used consistently for P, O and the row
// sum, so the result is unchanged; the rare rescale of O is done by the softmax warpgroup.
// P goes to the issuer in two pieces (96 and 32 keys, two barriers), so the first piece of PV runs while
// the second half of the row is exponentiated.  The loader publishes the CTA's work items through
// a small shared-memory queue; all device waits are bounded (see mbar_wait).
// ---------------------------------------------------------------------------------------------
// Stages of the key/value ring (one K or V tile each).  For the decode-shaped launches, which stream K and V
// from HBM, 4 and 5 stages measure the same (93 / 99 us for 1 / 8 query tokens at the 128K key/value set), 3
// stages 120 / 126 us, and a sixth stage in the unused second query tile's memory 95 / 101 us: more loads in
// flight than the latency needs only add contention in the memory system.
constexpr int kStages = 5;
constexpr int kItemQueue = 4;     // work items the loader may publish ahead of the slowest consumer
constexpr int kAttnThreads = 384;             // warps 10 and 11 only take part in the register hand-back
// Keys of the first of the two pieces in which P is handed over: PV of the first piece runs while the second is exponentiated,
// and the shorter the second, the sooner the next S follows it (64 keys: 16K +0.1..2 %, 32 or 128: 1.5..3 % slower).
constexpr int kFirstKeys = 96;
constexpr int kMmaWarp = 8;
constexpr int kLoadWarp = 9;
constexpr float kRescaleThreshold = 8.0f;      // in log2 units
constexpr float kPieceSumBound = 256.f * kFirstKeys;   // of a piece formed with an old maximum, all at the threshold
// Measured and not kept: a polynomial exponential on the FMA pipe for part of the columns (2.5-4 % slower with d = 128, no
// difference with d = 64), the two softmax warps of a scheduler taking turns at a key tile's exponentials (8.5 %
// slower: one warp alone does not fill the MUFU pipe), reading S from TMEM in two halves (2 % slower).
// Registers per thread: the kernel is compiled for 168 (twelve warps).  setmaxnreg moves
// registers inside the CTA's own pool of 12 * 168 per lane slot and acts on whole warpgroups:
// warpgroup 2 (MMA issuer, TMA loader and two spare warps) hands back all but kRegsIssuer,
// the eight softmax warps grow to kRegsSoftmax:  4 * 88 + 8 * 208 = 2016 = 12 * 168.
constexpr int kRegsIssuer = 88;
constexpr int kRegsSoftmax = 208;

// What one work item covers.  The loader decodes it and hands it to the issuer and the softmax warps through a queue in
// shared memory; they read what they need rarely where they need it, which leaves the registers to the logits.
struct __align__(16) Item {
    int valid;                   // 0: no further work items

    int token0_a, token0_b;      // first token of each query tile
    int head0, kvh, part;
    int has1;                    // second query tile exists
    int n_tiles_a, n_tiles_b;    // key tiles each query tile walks
    int n_load;                  // key tiles to stage = max of the two
    int n_pref_tiles, pref_len;
    int main_row0, main_len;
    int row0_a, row0_b;          // first row of each query tile within its block (phase 1)
    int bad_length;              // phase 1: prefix_len of the block was outside [0, prefix_total] (clamped)
    int gen_base;                // >= 0: generation shard, token u sees its rows [0, gen_base + u]; -1 otherwise
    int pad_;
};
static_assert(sizeof(Item) == 80, "whole 16-byte words");

template <int D>
struct SmemLayout {
    static constexpr int kPanels = D / 64;
    static constexpr int kTileBytes = kPanels * kPanelBytes;
    static constexpr int kQ = 0;                                   // 2 query tiles
    static constexpr int kKV = 2 * kTileBytes;                     // kStages key/value tiles
    static constexpr int kBars = kKV + kStages * kTileBytes;
    // barrier indices
    static constexpr int bQFull = 0, bQEmpty = 2, bSFull = 4, bPFull = 6, bOFull = 8, bOEmpty = 10, bPFull2 = 12;
    static constexpr int bKvFull = 14, bKvEmpty = 14 + kStages;
    static constexpr int bItemFull = 14 + 2 * kStages, bItemEmpty = bItemFull + kItemQueue;
    static constexpr int kNumBars = bItemEmpty + kItemQueue;
    static constexpr int kTmemPtr = kBars + kNumBars * 8;
    static constexpr int kAbort = kTmemPtr + 4;
    static constexpr int kItemQ = (kAbort + 4 + 15) / 16 * 16;     // Item [kItemQueue]: published work items
    static constexpr int kTotal = kItemQ + static_cast<int>(sizeof(Item)) * kItemQueue;
    static constexpr int kDynBytes = kTotal;
};

// Work item of this CTA in a given round.  Items are sorted costliest first; rounds alternate
// direction (boustrophedon) so that no CTA always draws the costlier end of a round.  -1: none.
__device__ __forceinline__ int item_of_round(int round, int n_items) {
    const int G = static_cast<int>(gridDim.x), c = static_cast<int>(blockIdx.x);
    const int idx = round * G + ((round & 1) ? G - 1 - c : c);
    return idx < n_items ? idx : -1;
}

// (Table: the sequence table, or NoTable where the launch has no sequences.)
template <typename Table>
__device__ __forceinline__ void decode_item(const AttnArgs& a, const Table& vt, int idx, Item& it) {
    it.valid = 1;
    it.bad_length = 0;
    it.part = 0;
    it.gen_base = -1;
    const int tpt = kTileM >> a.pack_shift;                    // tokens per query tile
    if (a.mode != kModePhase2) {
        const int per_item = a.single ? 1 : 2;                 // query tiles per work item
        const int heads = a.pack_shift ? a.Hkv : a.Hq;         // work items per run of tokens
        const int rank = idx / heads, h = idx - rank * heads;
        it.head0 = a.pack_shift ? h * a.g : h;
        it.kvh = a.pack_shift ? h : h / a.g;
        int pair, len, start;
        if (a.mode == kModeVarlen) {
            // Independent sequences of different lengths, plain causal attention inside each.
            // Items run from the last sequence down and, inside a sequence, from its last tokens
            // down (for assembled Pulsar inputs the later blocks are the longer ones).
            int k = 0;                                             // k-th sequence from the end
            while (k + 1 < vt.n_seq && vt.pair_cum[k + 1] <= rank) ++k;
            const int seq = vt.n_seq - 1 - k;
            start = vt.start[seq];
            len = vt.start[seq + 1] - start;
            pair = (len + per_item * tpt - 1) / (per_item * tpt) - 1 - (rank - vt.pair_cum[k]);
            it.pref_len = 0;
        } else {
            // Items run block-major from the last block (longest prefix) down and, within a block,
            // from the last tokens (most causal tiles) down; the heads of one run of tokens are
            // adjacent.  CTAs that run at the same time therefore read the same K/V rows (L2 hits),
            // and the costliest items are handed out first.
            // The last block may be shorter than the others: it then has fewer items.
            int blk;
            if (rank < a.pairs_last) {
                blk = a.n_blocks - 1;
                pair = a.pairs_last - 1 - rank;
                len = a.last_len;
            } else {
                const int r2 = rank - a.pairs_last;
                blk = a.n_blocks - 2 - r2 / a.pairs;
                pair = a.pairs - 1 - r2 % a.pairs;
                len = a.block_size;
            }
            start = blk * a.block_size;
            int pl = a.prefix_len[blk];
            it.bad_length = (pl < 0 || pl > a.prefix_total) ? 1 : 0;
            it.pref_len = max(0, min(pl, a.prefix_total));
        }
        it.n_pref_tiles = (it.pref_len + kTileN - 1) / kTileN;
        it.row0_a = per_item * pair * tpt;
        it.row0_b = it.row0_a + tpt;
        it.has1 = (per_item == 2 && it.row0_b < len) ? 1 : 0;
        it.token0_a = start + it.row0_a;
        it.token0_b = start + it.row0_b;
        it.main_row0 = start;
        it.main_len = len;
        // key tiles up to the one with the tile's last row
        it.n_tiles_a = it.n_pref_tiles + (min(it.row0_a + tpt, len) + kTileN - 1) / kTileN;
        it.n_tiles_b = it.has1 ? it.n_pref_tiles + (min(it.row0_b + tpt, len) + kTileN - 1) / kTileN : 0;
    } else {
        const int rp = idx % a.pairs;
        const int rest = idx / a.pairs;
        it.kvh = rest % a.Hkv;
        it.part = rest / a.Hkv;
        it.head0 = it.kvh * a.g;
        it.token0_a = (2 * rp) * tpt;
        it.token0_b = (2 * rp + 1) * tpt;
        it.has1 = (it.token0_b < a.n_tokens) ? 1 : 0;
        it.row0_a = it.row0_b = 0;
        // the generation shard: read through the second pair of tensor maps, causal by token
        const bool shard = a.gen_total > 0 && it.part == a.gen_part;
        it.pref_len = shard ? a.gen_total : 0;
        it.n_pref_tiles = (it.pref_len + kTileN - 1) / kTileN;
        if (shard) it.gen_base = a.gen_len;
        it.main_row0 = (it.part - a.ctx_part0) * a.split_len;
        it.main_len = it.main_row0 < 0 ? 0 : min(a.split_len, a.kv_len - it.main_row0);
        const int n = it.n_pref_tiles + (it.main_len + kTileN - 1) / kTileN;
        it.n_tiles_a = n;
        it.n_tiles_b = it.has1 ? n : 0;
    }
    it.n_load = max(it.n_tiles_a, it.n_tiles_b);
}

// KV(q) of the new tokens of one KV head appended to the generation shard by the warp that is about to load the
// head's shard rows through TMA: written with plain stores, made visible to the async proxy, then loaded.  No other CTA
// of the launch touches the head's rows.  (As a launch of its own the append cost 2.8 us on the host and 2-3 us on the
// device of every decoding step.)  The warp's loads are latency, about 0.8 us a round: four vectors of K and of V are
// under way per lane, and rows that take more than four such rounds (kAppendVecs) come from a launch of their own (64
// tokens of 8 heads with d = 128 at 65,536: 83 us with one vector at a time, 50 us with that launch; 32 tokens 19.8 -> 15.0).
constexpr int kAppendVecs = 512;                              // 16-byte vectors of a head's new rows: 32 tokens with d = 128

__device__ __forceinline__ void append_head(const AttnArgs& a, int kvh, int d, int lane) {
    const int vecs = d / 8;                                   // 16-byte vectors of a head's row
    const int n = (a.gen_total - a.gen_len) * vecs;
    const auto at = [&](int i, int row0) {
        const int u = i / vecs;
        return (static_cast<size_t>(row0 + u) * a.Hkv + kvh) * vecs + (i - u * vecs);
    };
    int i0 = lane;
    for (; n > 32 && i0 < n; i0 += 128) {
        uint4 k[4], v[4];
#pragma unroll
        for (int j = 0; j < 4; ++j)
            if (i0 + 32 * j < n) {
                k[j] = a.Knew[at(i0 + 32 * j, 0)];
                v[j] = a.Vnew[at(i0 + 32 * j, 0)];
            }
#pragma unroll
        for (int j = 0; j < 4; ++j)
            if (i0 + 32 * j < n) {
                a.Kgen[at(i0 + 32 * j, a.gen_len)] = k[j];
                a.Vgen[at(i0 + 32 * j, a.gen_len)] = v[j];
            }
    }
    if (i0 < n) {                                             // a row or two: nothing to overlap
        const uint4 k = a.Knew[at(i0, 0)], v = a.Vnew[at(i0, 0)];
        a.Kgen[at(i0, a.gen_len)] = k;
        a.Vgen[at(i0, a.gen_len)] = v;
    }
    fence_proxy_async_global();
    __syncwarp();
}

// The maximum that the P of a key tile is formed with.  It moves up when the tile's maximum is more than the threshold
// above it, always on the first tile.  With tile_max it follows the tile's maximum down as well (by at most the
// threshold at a time, and only while the row sum shows that no earlier probability is far above 1), so that the
// largest probability of every tile is 1 and has no rounding error.
__device__ __forceinline__ float next_max(float m_tile, float m_used, float l_run, bool tile_max) {
    if (tile_max && (m_tile > m_used || l_run < 256.f)) return fmaxf(m_tile, m_used - kRescaleThreshold);
    return m_tile > m_used + kRescaleThreshold ? m_tile : m_used;
}

// Row maximum of N raw logits (3-input max, four independent chains).
template <int N>
__device__ __forceinline__ float row_max(const uint32_t (&r)[N]) {
    float m0 = -INFINITY, m1 = -INFINITY, m2 = -INFINITY, m3 = -INFINITY;
#pragma unroll
    for (int c = 0; c < N; c += 8) {
        m0 = max3(m0, __uint_as_float(r[c]), __uint_as_float(r[c + 1]));
        m1 = max3(m1, __uint_as_float(r[c + 2]), __uint_as_float(r[c + 3]));
        m2 = max3(m2, __uint_as_float(r[c + 4]), __uint_as_float(r[c + 5]));
        m3 = max3(m3, __uint_as_float(r[c + 6]), __uint_as_float(r[c + 7]));
    }
    return fmaxf(fmaxf(m0, m1), fmaxf(m2, m3));
}

// p_c = 2^(s_c * scale + neg_m) for logits [kBegin, kEnd) of a row, rounded to bf16 pairs and written
// to TMEM as the A operand of the PV product; returns the fp32 row sum.
template <int kBegin, int kEnd, int N>
__device__ __forceinline__ float exp_row(const uint32_t (&r)[N], float scale, float neg_m, uint32_t tP) {
    float2 acc0 = make_float2(0.f, 0.f), acc1 = make_float2(0.f, 0.f);
    const float2 sc = make_float2(scale, scale), nm = make_float2(neg_m, neg_m);
#pragma unroll
    for (int c0 = kBegin; c0 < kEnd; c0 += 32) {
        uint32_t pk[16];
#pragma unroll
        for (int c = 0; c < 32; c += 2) {
            const float2 x =
                __ffma2_rn(make_float2(__uint_as_float(r[c0 + c]), __uint_as_float(r[c0 + c + 1])), sc, nm);
            float2 pv;
            pv.x = ex2(x.x);
            pv.y = ex2(x.y);
            if ((c >> 1) & 1) acc1 = __fadd2_rn(acc1, pv);
            else acc0 = __fadd2_rn(acc0, pv);
            pk[c >> 1] = pack_bf16x2(pv.x, pv.y);
        }
        tmem_st16(tP + (c0 >> 1), pk);                           // P column c/2 holds keys c, c+1
    }
    return (acc0.x + acc0.y) + (acc1.x + acc1.y);
}

// kQuad: the decode-shaped instance (AttnArgs::quad); a separate instantiation keeps its code out
// of the Phase-1 kernel's register allocation.
// kSingle: every work item of the launch has one query tile (AttnArgs::single).  With a second tile the
// tensor pipe forms one tile's products while the other tile is in its softmax; with one tile it would
// idle during the softmax and the softmax during the products (S_t -> softmax_t -> PV_t -> S_t+1 in a
// chain).  Here the logits of successive key tiles alternate between the S buffers of the two tiles
// (buffer = key-tile count of the CTA, parity), the issuer forms S_t+1 before it waits for P_t, and
// softmax warpgroup 0 walks all key tiles with both sets of barriers.  A rescale of O at key tile t
// needs PV_t-1 complete, which the completion of S_t no longer implies (it implies PV_t-2): the issuer
// commits every PV to the O barrier of the absent second tile, and a softmax warp that has to rescale
// waits for it first.  Measured against the 128K key/value set (131,072 keys, 18 parts, L2 flushed clean
// before each call): 9 to 32 query tokens of 4 heads per KV head 120-124 us -> 99-103 us (0.69 -> 0.83 of
// the HBM bandwidth), the 8-token decode shape 101.3 -> 99.4 us.
// kHalves (kSingle without kQuad): the two warpgroups share the key tile, 64 keys of every row each, with a maximum, a sum
// and an accumulator of their own (the absent second tile's), and bring them together when the item ends.  The exponentials of
// a key tile take the SM's special functions 1024 cycles whoever forms them, but the reads of S, the stores of P and the
// barriers around them are now under way in two warps per scheduler.  us per key tile of a part, d = 64 0.87 -> 0.80, d = 128
// 0.88 -> 0.82 (64 key tiles of 64 rows 60.1 -> 55.7 and 61.1 -> 57.4; 4096 causal rows of one head 36.4 -> 34.3 and
// 36.9 -> 36.0); launches that stream from HBM take what they took.
// kTileMax: see next_max; generation steps whose parts were made longer.  An instance of its own, since the test alone
// costs Phase 1 0.4 % (16K 658 -> 661 us).
// kBeside: see launch_lse_merge (an instance of its own: the test alone cost calls of 20-40 us 0.1-0.2 us).
template <int D, bool kQuad, bool kSingle, bool kTileMax, bool kBeside>
__global__ void __launch_bounds__(kAttnThreads, 1)
attn_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK,
            const __grid_constant__ CUtensorMap tmV, const __grid_constant__ CUtensorMap tmKp,
            const __grid_constant__ CUtensorMap tmVp, const AttnArgs a,
            const __grid_constant__ std::conditional_t<kQuad, NoTable, VarlenTable> vt) {
    using SL = SmemLayout<D>;
    constexpr bool kHalves = kSingle && !kQuad;
    constexpr int kCols = kHalves ? kTileN / 2 : kTileN;      // logits of a softmax thread per key tile
    constexpr int kFirst = kHalves ? kCols : kFirstKeys;      // of which it hands over first
    static_assert(kSingle || !kQuad, "the decode-shaped instance has one query tile per item");
    // The swizzled tiles want 1024-byte alignment.  Declared, not computed: tile addresses and descriptors are constants
    // then, which takes them out of the registers of the issuer.
    extern __shared__ __align__(1024) uint8_t smem[];
    uint8_t* sQ = smem + SL::kQ;
    uint8_t* sKV = smem + SL::kKV;
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem + SL::kBars);
    uint32_t* tmem_ptr = reinterpret_cast<uint32_t*>(smem + SL::kTmemPtr);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + SL::kAbort);

    const int tid = threadIdx.x, lane = tid & 31;
    // Broadcast, so that the compiler knows the branches into the roles to be warp-uniform.
    const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);

    if (tid == 0) {
        *abort_flag = 0;
        for (int s = 0; s < 2; ++s) {
            mbar_init(bars + SL::bQFull + s, 1);
            mbar_init(bars + SL::bQEmpty + s, 1);
            mbar_init(bars + SL::bSFull + s, 1);
            mbar_init(bars + SL::bPFull + s, 4);        // first half of P: one arrival per softmax warp
            mbar_init(bars + SL::bPFull2 + s, 4);       // second half of P
            mbar_init(bars + SL::bOFull + s, 1);
            mbar_init(bars + SL::bOEmpty + s, kHalves ? 8 : 4);
        }
        for (int i = 0; i < kItemQueue; ++i) {
            mbar_init(bars + SL::bItemFull + i, 1);
            mbar_init(bars + SL::bItemEmpty + i, 9);        // MMA issuer + one lane of each softmax warp
        }
        for (int i = 0; i < kStages; ++i) {
            mbar_init(bars + SL::bKvFull + i, 1);
            mbar_init(bars + SL::bKvEmpty + i, 1);
        }
        mbar_fence_init();
    }
    if (warp == kLoadWarp && lane == 0) {
        tma_prefetch_desc(&tmQ);
        tma_prefetch_desc(&tmK);
        tma_prefetch_desc(&tmV);
        tma_prefetch_desc(&tmKp);
        tma_prefetch_desc(&tmVp);
    }
    if (warp == kMmaWarp) {
        tmem_alloc(tmem_ptr, 512);
        tmem_relinquish();
    }
    // The CTAs of this launch may have been placed while the launch before it was still running; everything above
    // (barriers, tensor maps, TMEM) overlaps its end, nothing below may.
    if (!kBeside) grid_dependency_wait();
    // The launch that follows (the merge of this launch's partials, or another call's) may be placed as
    // SMs become free; it waits for this grid to finish before it reads anything.
    grid_launch_dependents();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_ptr;

    if (warp >= 8) reg_dealloc<kRegsIssuer>();
    // Ring bookkeeping shared by the two issuer roles: `stage` walks 0..kStages-1, `phase`
    // flips at every wrap.  Barrier i lives at bar0 + 8 * i.
    const uint32_t bar0 = smem_u32(bars);
    Item* item_q = reinterpret_cast<Item*>(smem + SL::kItemQ);
#define PULSAR_RING_NEXT(stage, phase) \
    do { if (++(stage) == kStages) { (stage) = 0; (phase) ^= 1u; } } while (0)

    if (warp == kLoadWarp) {
        // =============================== TMA loader ===============================
        // The whole warp walks the loops so that addresses, coordinates and barrier numbers stay
        // warp-uniform (the copy and barrier instructions take uniform operands); one elected
        // lane issues.
        {
            const bool leader = elect_one();
            const uint32_t q_smem = smem_u32(sQ), kv_smem = smem_u32(sKV);
            uint32_t stage = 0, phase = 0;           // next ring slot to fill
            uint32_t q_use0 = 0, q_use1 = 0;
            bool ok = true;
            for (uint32_t seq = 0; ok; ++seq) {
                // Reconverge once per iteration: every barrier is waited on at most once per
                // iteration, so a lane that is still polling can never be more than one phase behind
                // the lanes that went ahead (two phases behind, its parity test would read "not yet"
                // again and it would stall until the bound expires).
                __syncwarp();
                // Next work item: drawn from the global counter (items differ in cost or outnumber the
                // CTAs, so they are handed out as CTAs become free) or the fixed round order.
                // It is published through a small queue for the MMA issuer and the softmax warps.
                const uint32_t slot = seq % kItemQueue;
                ok = mbar_wait_a(bar0 + 8 * (SL::bItemEmpty + slot), ((seq / kItemQueue) & 1) ^ 1, abort_flag, a.status);
                if (!ok) break;
                int idx;
                if (a.counter != nullptr) {
                    int v = 0;
                    if (lane == 0) v = atomicAdd(a.counter, 1);
                    idx = __shfl_sync(0xffffffffu, v, 0);
                    if (idx >= a.n_items) idx = -1;
                } else {
                    idx = static_cast<int>(seq) * static_cast<int>(gridDim.x) < a.n_items
                              ? item_of_round(static_cast<int>(seq), a.n_items) : -1;
                }
                Item it;
                it.valid = 0;
                if (idx >= 0) decode_item(a, vt, idx, it);
                if (lane == 0) {
                    item_q[slot] = it;
                    mbar_arrive(bars + SL::bItemFull + slot);
                }
                if (idx < 0) break;
                if (it.bad_length && lane == 0) report(a.status, PULSAR_DEV_BAD_LENGTH);
                if (kSingle && it.gen_base >= 0 && a.Knew != nullptr) append_head(a, it.kvh, D, lane);
                const int x = it.kvh * D;
                // query tile 0
                ok = mbar_wait_a(bar0 + 8 * (SL::bQEmpty + 0), (q_use0 & 1) ^ 1, abort_flag, a.status);
                ++q_use0;
                if (!ok) break;
                if (leader) mbar_expect_tx_a(bar0 + 8 * (SL::bQFull + 0), SL::kTileBytes);
                if (kQuad) {
                    // the same 32 rows four times, at rows 0, 32, 64, 96 of the tile (the box of the
                    // tensor map is 32 rows here; 32 rows of a panel are 4096 bytes)
#pragma unroll
                    for (int c = 0; c < 4; ++c)
#pragma unroll
                        for (int p = 0; p < SL::kPanels; ++p)
                            if (leader) tma_load_3d_a(q_smem + p * kPanelBytes + c * 4096, &tmQ, bar0 + 8 * (SL::bQFull + 0),
                                          p * 64, it.head0, it.token0_a);
                } else {
#pragma unroll
                    for (int p = 0; p < SL::kPanels; ++p)
                        if (leader) tma_load_3d_a(q_smem + p * kPanelBytes, &tmQ, bar0 + 8 * (SL::bQFull + 0), p * 64, it.head0,
                                      it.token0_a);
                }
                for (int t = 0; t < it.n_load && ok; ++t) {
                    __syncwarp();
                    const bool pref = t < it.n_pref_tiles;
                    const int row = pref ? t * kTileN : it.main_row0 + (t - it.n_pref_tiles) * kTileN;
                    // K_t
                    ok = mbar_wait_a(bar0 + 8 * (SL::bKvEmpty + stage), phase ^ 1, abort_flag, a.status);
                    if (!ok) break;
                    {
                        const uint32_t full = bar0 + 8 * (SL::bKvFull + stage), dst = kv_smem + stage * SL::kTileBytes;
                        if (leader) mbar_expect_tx_a(full, SL::kTileBytes);
#pragma unroll
                        for (int p = 0; p < SL::kPanels; ++p)
                            if (leader) tma_load_2d_a(dst + p * kPanelBytes, pref ? &tmKp : &tmK, full, x + p * 64, row);
                    }
                    PULSAR_RING_NEXT(stage, phase);
                    if (t == 0 && it.has1) {
                        ok = mbar_wait_a(bar0 + 8 * (SL::bQEmpty + 1), (q_use1 & 1) ^ 1, abort_flag, a.status);
                        ++q_use1;
                        if (!ok) break;
                        if (leader) mbar_expect_tx_a(bar0 + 8 * (SL::bQFull + 1), SL::kTileBytes);
#pragma unroll
                        for (int p = 0; p < SL::kPanels; ++p)
                            if (leader) tma_load_3d_a(q_smem + SL::kTileBytes + p * kPanelBytes, &tmQ, bar0 + 8 * (SL::bQFull + 1),
                                          p * 64, it.head0, it.token0_b);
                    }
                    // V_t
                    ok = mbar_wait_a(bar0 + 8 * (SL::bKvEmpty + stage), phase ^ 1, abort_flag, a.status);
                    if (!ok) break;
                    {
                        const uint32_t full = bar0 + 8 * (SL::bKvFull + stage), dst = kv_smem + stage * SL::kTileBytes;
                        if (leader) mbar_expect_tx_a(full, SL::kTileBytes);
#pragma unroll
                        for (int p = 0; p < SL::kPanels; ++p)
                            if (leader) tma_load_2d_a(dst + p * kPanelBytes, pref ? &tmVp : &tmV, full, x + p * 64, row);
                    }
                    PULSAR_RING_NEXT(stage, phase);
                }
            }
        }
        __syncwarp();
    } else if (warp == kMmaWarp) {
        // =============================== MMA issuer ===============================
        // Per key tile t the issue order is PV_0(t), S_0(t+1), PV_1(t), S_1(t+1): tile 0 gets its
        // next S about one PV + S ahead of tile 1, which keeps the two softmax warpgroups half a
        // period apart (one exponentiates while the tensor pipe works for the other).
        // Warp-uniform control flow, one elected lane issues: descriptors, TMEM addresses and
        // barrier numbers then live in uniform registers, which the MMA instructions read.
        {
            const bool leader = elect_one();
            constexpr uint32_t kIdescQK = umma_idesc_bf16(kTileM, kTileN, false, false);
            constexpr uint32_t kIdescPV = umma_idesc_bf16(kTileM, D, false, true);
            constexpr uint32_t kStageStep = SL::kTileBytes >> 4;         // descriptor address units (16 bytes)
            // Descriptors of stage 0 / query tile 0; other tiles add a multiple of kStageStep to the
            // address field (shared memory is below 256 KB, so the 14-bit field never carries).
            const uint64_t descQ0 = umma_smem_desc_sw128(smem_u32(sQ), 16, 1024);
            const uint64_t descQ1 = descQ0 + kStageStep;
            const uint64_t descK = umma_smem_desc_sw128(smem_u32(sKV), 16, 1024);
            const uint64_t descV = umma_smem_desc_sw128(smem_u32(sKV), kPanelBytes, 1024);
            const uint32_t tS0 = tmem_base, tS1 = tmem_base + 128, tO0 = tmem_base + 256, tO1 = tmem_base + 384;
            uint32_t stage = 0, phase = 0;           // next ring slot to consume
            uint32_t q_use0 = 0, q_use1 = 0, p_cnt0 = 0, p_cnt1 = 0, o_use0 = 0, o_use1 = 0;
            uint32_t g_tile = 0;                     // kSingle: key tiles this CTA has walked
            bool ok = true;

#define PULSAR_ISSUE_S(tS, dq, dk, s_)                                                                    \
    do {                                                                                                  \
        _Pragma("unroll") for (int kk = 0; kk < D / 16; ++kk) {                                           \
            const uint64_t off = static_cast<uint64_t>(((kk >> 2) * kPanelBytes + (kk & 3) * 32) >> 4);    \
            if (leader) umma_ss(tS, (dq) + off, (dk) + off, kIdescQK, kk > 0 ? 1u : 0u);                  \
        }                                                                                                 \
        if (leader) umma_commit_a(bar0 + 8 * (SL::bSFull + (s_)));                                        \
    } while (0)
// P arrives in two pieces (kFirstKeys keys, then the rest), each with its own barrier.
// With kHalves they are the two warpgroups': P of keys [64, 128) stands at column 64, and its product goes to the
// accumulator of the absent second tile.
#define PULSAR_ISSUE_PV(tO, tP, dv, acc, s_, par)                                                         \
    do {                                                                                                  \
        _Pragma("unroll") for (int half = 0; half < 2; ++half) {                                          \
            ok = ok && mbar_wait_a(bar0 + 8 * ((half ? SL::bPFull2 : SL::bPFull) + (s_)), par, abort_flag, \
                                   a.status);                                                             \
            tc_fence_after();                                                                             \
            _Pragma("unroll") for (int kk = half ? kFirst / 16 : 0; kk < (half ? kTileN : kFirst) / 16; ++kk) \
                if (leader && ok)                                                                         \
                    umma_ts((tO) + (kHalves && half ? 128 : 0), (tP) + kk * 8 + (kHalves && half ? 32 : 0), \
                            (dv) + static_cast<uint64_t>(kk * 128), kIdescPV,                             \
                            ((acc) || kk > (kHalves && half ? kFirst / 16 : 0)) ? 1u : 0u);               \
        }                                                                                                 \
    } while (0)

            for (uint32_t seq = 0; ok; ++seq) {
                __syncwarp();              // see the loader: lanes stay within one barrier phase of each other
                const uint32_t slot = seq % kItemQueue;
                ok = mbar_wait_a(bar0 + 8 * (SL::bItemFull + slot), (seq / kItemQueue) & 1, abort_flag, a.status);
                if (!ok) break;
                const int valid = item_q[slot].valid, n0 = item_q[slot].n_tiles_a, n1 = item_q[slot].n_tiles_b;
                __syncwarp();
                if (leader) mbar_arrive(bars + SL::bItemEmpty + slot);
                if (!valid) break;
                const int n_load = max(n0, n1);
                if (kSingle) {
                    // Ring slots: K_t at position 2t of the item, V_t at 2t + 1 (the loader's order); the
                    // issuer consumes K_t+1 before V_t.
                    uint32_t kst = stage, kph = phase, vst = stage, vph = phase;
                    PULSAR_RING_NEXT(vst, vph);
                    ok = mbar_wait_a(bar0 + 8 * (SL::bQFull + 0), q_use0 & 1, abort_flag, a.status) &&
                         mbar_wait_a(bar0 + 8 * (SL::bKvFull + kst), kph, abort_flag, a.status);
                    ++q_use0;
                    if (!ok) break;
                    tc_fence_after();
                    {
                        const uint32_t b = g_tile & 1u;
                        PULSAR_ISSUE_S(tS0 + b * 128, descQ0, descK + static_cast<uint64_t>(kst * kStageStep), b);
                    }
                    if (leader) umma_commit_a(bar0 + 8 * (SL::bKvEmpty + kst));
                    if (n0 == 1 && leader) umma_commit_a(bar0 + 8 * (SL::bQEmpty + 0));
                    PULSAR_RING_NEXT(kst, kph);
                    PULSAR_RING_NEXT(kst, kph);
                    for (int t = 0; t < n0; ++t) {
                        __syncwarp();
                        const uint32_t b = g_tile & 1u, par = (g_tile >> 1) & 1u;
                        if (t + 1 < n0) {                                  // S_t+1 into the other buffer
                            ok = mbar_wait_a(bar0 + 8 * (SL::bKvFull + kst), kph, abort_flag, a.status);
                            if (!ok) break;
                            tc_fence_after();
                            PULSAR_ISSUE_S(tS0 + (b ^ 1u) * 128, descQ0, descK + static_cast<uint64_t>(kst * kStageStep), b ^ 1u);
                            if (leader) umma_commit_a(bar0 + 8 * (SL::bKvEmpty + kst));
                            if (t + 2 == n0 && leader) umma_commit_a(bar0 + 8 * (SL::bQEmpty + 0));
                            PULSAR_RING_NEXT(kst, kph);
                            PULSAR_RING_NEXT(kst, kph);
                        }
                        ok = mbar_wait_a(bar0 + 8 * (SL::bKvFull + vst), vph, abort_flag, a.status);
                        if (!ok) break;
                        if (t == 0) {
                            ok = mbar_wait_a(bar0 + 8 * (SL::bOEmpty + 0), (o_use0 & 1) ^ 1, abort_flag, a.status);
                            ++o_use0;
                        }
                        const uint64_t dv = descV + static_cast<uint64_t>(vst * kStageStep);
                        PULSAR_ISSUE_PV(tO0, tS0 + b * 128, dv, t > 0, b, par);
                        if (!ok) break;
                        if (leader) {
                            umma_commit_a(bar0 + 8 * (SL::bKvEmpty + vst));
                            umma_commit_a(bar0 + 8 * (SL::bOFull + 1));            // PV_t complete
                            if (t == n0 - 1) umma_commit_a(bar0 + 8 * (SL::bOFull + 0));
                        }
                        PULSAR_RING_NEXT(vst, vph);
                        PULSAR_RING_NEXT(vst, vph);
                        ++g_tile;
                    }
                    stage = kst;
                    phase = kph;
                    continue;
                }
                // K_0
                uint32_t ks = stage, kp = phase;
                PULSAR_RING_NEXT(stage, phase);
                ok = mbar_wait_a(bar0 + 8 * (SL::bQFull + 0), q_use0 & 1, abort_flag, a.status) &&
                     mbar_wait_a(bar0 + 8 * (SL::bKvFull + ks), kp, abort_flag, a.status);
                ++q_use0;
                if (!ok) break;
                tc_fence_after();
                PULSAR_ISSUE_S(tS0, descQ0, descK + static_cast<uint64_t>(ks * kStageStep), 0);
                if (n0 == 1 && leader) umma_commit_a(bar0 + 8 * (SL::bQEmpty + 0));
                if (n1 > 0) {
                    ok = mbar_wait_a(bar0 + 8 * (SL::bQFull + 1), q_use1 & 1, abort_flag, a.status);
                    ++q_use1;
                    if (!ok) break;
                    tc_fence_after();
                    PULSAR_ISSUE_S(tS1, descQ1, descK + static_cast<uint64_t>(ks * kStageStep), 1);
                    if (n1 == 1 && leader) umma_commit_a(bar0 + 8 * (SL::bQEmpty + 1));
                }
                if (leader) umma_commit_a(bar0 + 8 * (SL::bKvEmpty + ks));
                // Key tile t: PV_0(t), S_0(t+1), PV_1(t), S_1(t+1).  The issuer's own time is part of the chain that sets
                // the pace (a barrier test takes 100-300 cycles while the softmax warps of its scheduler keep the
                // queue that special functions and shared memory share full), so everything that can be waited for
                // early is waited for before PV_0, and the key tiles in the middle of an item, for which none of the
                // conditions below can fail, run without them (kMid).  With the constants and the uniform role branch
                // above, and no register spilled any more: Phase 1 at 64K 5.94 -> 5.53 ms (4.82 before the power
                // limit bites), at 16K 0.685 -> 0.638 ms, 45K ragged with d = 64 1.04 -> 0.96 ms.
                const auto key_tile = [&](auto mid, int t) {
                    constexpr bool kMid = decltype(mid)::value;
                    __syncwarp();
                    const uint32_t vs = stage, vp = phase;                 // V_t
                    PULSAR_RING_NEXT(stage, phase);
                    const bool more = kMid || t + 1 < n_load;
                    if (more) {                                            // K_{t+1}
                        ks = stage;
                        kp = phase;
                        PULSAR_RING_NEXT(stage, phase);
                    }
                    const uint64_t dv = descV + static_cast<uint64_t>(vs * kStageStep);
                    const uint64_t dk = descK + static_cast<uint64_t>(ks * kStageStep);
                    ok = mbar_wait_a(bar0 + 8 * (SL::bKvFull + vs), vp, abort_flag, a.status);
                    if (!ok) return;
                    if (more) {
                        ok = mbar_wait_a(bar0 + 8 * (SL::bKvFull + ks), kp, abort_flag, a.status);
                        if (!ok) return;
                    }
                    if (kMid || t < n0) {
                        if (!kMid && t == 0) {
                            ok = mbar_wait_a(bar0 + 8 * (SL::bOEmpty + 0), (o_use0 & 1) ^ 1, abort_flag, a.status);
                            ++o_use0;
                        }
                        PULSAR_ISSUE_PV(tO0, tS0, dv, kMid || t > 0, 0, p_cnt0 & 1);
                        ++p_cnt0;
                        if (!ok) return;
                        if (!kMid && t == n0 - 1 && leader) umma_commit_a(bar0 + 8 * (SL::bOFull + 0));
                    }
                    if (kMid || t + 1 < n0) {
                        PULSAR_ISSUE_S(tS0, descQ0, dk, 0);
                        // the tile's last S: nothing reads its Q any more
                        if (!kMid && t + 2 == n0 && leader) umma_commit_a(bar0 + 8 * (SL::bQEmpty + 0));
                    }
                    if (kMid || t < n1) {
                        if (!kMid && t == 0) {
                            ok = mbar_wait_a(bar0 + 8 * (SL::bOEmpty + 1), (o_use1 & 1) ^ 1, abort_flag, a.status);
                            ++o_use1;
                        }
                        PULSAR_ISSUE_PV(tO1, tS1, dv, kMid || t > 0, 1, p_cnt1 & 1);
                        ++p_cnt1;
                        if (!ok) return;
                        if (!kMid && t == n1 - 1 && leader) umma_commit_a(bar0 + 8 * (SL::bOFull + 1));
                    }
                    if (leader) umma_commit_a(bar0 + 8 * (SL::bKvEmpty + vs));
                    if (more) {
                        if (kMid || t + 1 < n1) {
                            PULSAR_ISSUE_S(tS1, descQ1, dk, 1);
                            if (!kMid && t + 2 == n1 && leader) umma_commit_a(bar0 + 8 * (SL::bQEmpty + 1));
                        }
                        if (leader) umma_commit_a(bar0 + 8 * (SL::bKvEmpty + ks));
                    }
                };
                int t = 0;
                key_tile(std::false_type{}, t++);
                for (const int t_mid = min(n0, n1) - 2; ok && t < t_mid; ++t) key_tile(std::true_type{}, t);
                for (; ok && t < n_load; ++t) key_tile(std::false_type{}, t);
            }
#undef PULSAR_ISSUE_S
#undef PULSAR_ISSUE_PV
        }
        __syncwarp();
    } else if (warp < 8) {
        // =============================== softmax warpgroups ===============================
        reg_alloc<kRegsSoftmax>();
        const int s = warp >> 2;
        const int row = (warp & 3) * 32 + lane;                // row of the tile = TMEM lane
        const uint32_t lane_sel = static_cast<uint32_t>((warp & 3) * 32) << 16;
        const int tile = kHalves ? 0 : s;                      // query tile of this warpgroup
        const int key0 = kHalves ? s * kCols : 0;              // its first key of a key tile
        const uint32_t tS_own = tmem_base + (kHalves ? key0 : s * 128) + lane_sel;
        const uint32_t tO = tmem_base + 256 + s * 128 + lane_sel;
        const uint32_t tO_other = tmem_base + 256 + (s ^ 1) * 128 + lane_sel;
        uint64_t* bar_of = bars + SL::bOFull + tile;
        uint64_t* bar_pv = bars + SL::bOFull + 1;              // kSingle: one completion per PV product
        uint32_t g_tile = 0;                                   // kSingle: key tiles this CTA has walked
        uint64_t* bar_oe = bars + SL::bOEmpty + tile;
        // kHalves: maximum and sum of each half of a row [2][2][128], where the second query tile would be, behind a barrier of
        // their own.  Items take the two places in turn: an item of one or two key tiles can end before a warp of the other
        // warpgroup has read what the item before it left, because S of its key tiles waits for no epilogue.  The
        // barrier of the item between orders those reads before the next writes to the same place.
        float2* half_all = reinterpret_cast<float2*>(sQ + SL::kTileBytes);
        uint64_t* bar_half = bars + SL::bOEmpty + 1;
        static_assert(!kHalves || 2 * 2 * kTileM * sizeof(float2) <= SL::kTileBytes, "the halves' sums take a tile's place");
        uint32_t s_cnt = 0, o_cnt = 0;
        bool ok = true;

        for (uint32_t seq = 0; ok; ++seq) {
            const uint32_t slot = seq % kItemQueue;
            ok = __all_sync(0xffffffffu, mbar_wait(bars + SL::bItemFull + slot, (seq / kItemQueue) & 1, abort_flag, a.status));
            if (!ok) break;
            const volatile Item& it = item_q[slot];            // handed back at the end of the item
            if (!it.valid) break;
            const int n = tile ? it.n_tiles_b : it.n_tiles_a;
            const int pref_len = it.pref_len;
            const bool tile_max = kTileMax && it.main_len > 0;
            float m_used = -INFINITY, l_run = 0.f;
            const int row_t = kQuad ? lane : row;             // row as far as token and head are concerned

            for (int t = 0; t < n; ++t) {
                // visible key columns of this tile for this row: [0, n_vis)
                int n_vis = kTileN;
                bool masked = false;
                const int pref_left = pref_len - t * kTileN;
                if (pref_left > 0) {
                    if (pref_left < kTileN) { n_vis = pref_left; masked = true; }
                    if (it.gen_base >= 0) {                   // generation shard: causal by token
                        const int token = (tile ? it.token0_b : it.token0_a) + (row_t >> a.pack_shift);
                        n_vis = min(n_vis, it.gen_base + token + 1 - t * kTileN);
                        masked = true;
                    }
                } else {
                    const int j = t - (pref_len + kTileN - 1) / kTileN;
                    const int valid = it.main_len - j * kTileN;
                    if (valid < kTileN) { n_vis = valid; masked = true; }
                    if (a.mode != kModePhase2 && t == n - 1) {
                        n_vis = min(n_vis, (tile ? it.row0_b : it.row0_a) + (row_t >> a.pack_shift) - j * kTileN + 1);
                        masked = true;
                    }
                }

                // kSingle: buffer and barriers alternate with the CTA's key-tile count
                const uint32_t gb = kSingle ? (g_tile & 1u) : 0u;
                const uint32_t tS = tS_own + gb * 128;
                uint64_t* bar_s = bars + SL::bSFull + tile + gb;
                uint64_t* bar_p = bars + (kHalves && s ? SL::bPFull2 : SL::bPFull) + tile + gb;
                uint64_t* bar_p2 = bars + SL::bPFull2 + tile + gb;
                ok = __all_sync(0xffffffffu,
                                ok && mbar_wait(bar_s, kSingle ? ((g_tile >> 1) & 1u) : (s_cnt & 1u), abort_flag, a.status));
                ++s_cnt;
                ++g_tile;
                if (!ok) break;
                tc_fence_after();

                if (kQuad) {
                    // Few query rows (decode): this warp's lane quarter holds a copy of the rows and
                    // the warp takes keys [32q, 32q+32) of the tile only; the other keys get P = 0 in
                    // its copy.  Each copy ends as a partial of its own, merged with the KV parts.
                    const int q4 = warp & 3;
                    uint32_t rq[32];
                    tmem_ld32(tS + 32 * q4, rq);
                    tmem_wait_ld();
                    if (masked) {
#pragma unroll
                        for (int c = 0; c < 32; ++c)
                            if (32 * q4 + c >= n_vis) rq[c] = 0xff800000u;          // -inf
                    }
                    float mq = -INFINITY;
#pragma unroll
                    for (int c = 0; c < 32; c += 2) mq = max3(mq, __uint_as_float(rq[c]), __uint_as_float(rq[c + 1]));
                    const float m_tile = mq * a.scale_log2;
                    const float m_new = next_max(m_tile, m_used, l_run, tile_max);
                    if (__any_sync(0xffffffffu, m_new != m_used)) {
                        if (kSingle && t > 0) {
                            // O may be rescaled once the PV product of the previous key tile is complete.
                            // This is key tile g_tile - 1 of the CTA; completions 0 .. g_tile - 3 are certain
                            // (this tile's S was issued after them), so the barrier is in phase g_tile - 2
                            // or g_tile - 1 and the parity of g_tile - 2 tells the two apart.
                            ok = __all_sync(0xffffffffu, mbar_wait(bar_pv, g_tile & 1u, abort_flag, a.status));
                            if (!ok) break;
                            tc_fence_after();
                        }
                        const float alpha = (m_new == -INFINITY) ? 1.f : ex2(m_used - m_new);
                        l_run *= alpha;
                        m_used = m_new;
                        if (t > 0) {
#pragma unroll
                            for (int c0 = 0; c0 < D; c0 += 32) {
                                uint32_t o[32];
                                tmem_ld32(tO + c0, o);
                                tmem_wait_ld();
#pragma unroll
                                for (int c = 0; c < 32; ++c) o[c] = __float_as_uint(__uint_as_float(o[c]) * alpha);
                                tmem_st32(tO + c0, o);
                            }
                        }
                    }
                    const float neg_m = (m_used == -INFINITY) ? 0.f : -m_used;
                    uint32_t pk[16];
                    float2 acc = make_float2(0.f, 0.f);
                    const float2 sc = make_float2(a.scale_log2, a.scale_log2), nm = make_float2(neg_m, neg_m);
#pragma unroll
                    for (int c = 0; c < 32; c += 2) {
                        const float2 x = __ffma2_rn(make_float2(__uint_as_float(rq[c]), __uint_as_float(rq[c + 1])), sc, nm);
                        float2 pv;
                        pv.x = ex2(x.x);
                        pv.y = ex2(x.y);
                        acc = __fadd2_rn(acc, pv);
                        pk[c >> 1] = pack_bf16x2(pv.x, pv.y);
                    }
                    l_run += acc.x + acc.y;
                    uint32_t zero[16];
#pragma unroll
                    for (int c = 0; c < 16; ++c) zero[c] = 0u;
#pragma unroll
                    for (int qq = 0; qq < 4; ++qq) {
                        if (qq == q4) tmem_st16(tS + 16 * qq, pk);          // P column c/2 holds keys c, c+1
                        else tmem_st16(tS + 16 * qq, zero);
                    }
                    tmem_wait_st();
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) {
                        mbar_arrive(bar_p);
                        mbar_arrive(bar_p2);
                    }
                    continue;
                }

                uint32_t r[kCols];
                PULSAR_TMEM_LD32_AT(tS + 0, r, 0);
                PULSAR_TMEM_LD32_AT(tS + 32, r, 32);
                if constexpr (!kHalves) {
                    PULSAR_TMEM_LD32_AT(tS + 64, r, 64);
                    PULSAR_TMEM_LD32_AT(tS + 96, r, 96);
                }
                tmem_wait_ld();

                if (masked) {
#pragma unroll
                    for (int c = 0; c < kCols; ++c)
                        if (key0 + c >= n_vis) r[c] = 0xff800000u;   // -inf
                }
                // After the first key tile the running maximum is nearly always good enough, so the first piece of P is
                // formed with it at once, and whether it was is seen afterwards: its own sum bounds every one of its
                // probabilities, the logits of the second piece are compared.  If it was not (or the tile is masked),
                // the row maximum is taken over the whole tile, O is rescaled and the piece is formed again.  The
                // maximum and the vote took 520 of the 3250 cycles of a key tile before anything could be
                // exponentiated: Phase 1 at 64K 5.46 -> 5.37 ms, d = 64 0.944 -> 0.918 ms.
                float s1 = 0.f, neg_m = -m_used;
                bool fast = !masked && t > 0 && !tile_max;
                if (fast) {
                    s1 = exp_row<0, kFirst>(r, a.scale_log2, neg_m, tS);
                    float m2 = -INFINITY;
                    if constexpr (!kHalves) {
#pragma unroll
                        for (int c = kFirst; c < kCols; c += 2) m2 = max3(m2, __uint_as_float(r[c]), __uint_as_float(r[c + 1]));
                    }
                    fast = !__any_sync(0xffffffffu, !(s1 <= kPieceSumBound) || m2 * a.scale_log2 > m_used + kRescaleThreshold);
                }
                if (!fast) {
                    tmem_wait_st();          // stores to the same columns have no order among themselves
                    const float m_tile = row_max(r) * a.scale_log2;
                    const float m_new = next_max(m_tile, m_used, l_run, tile_max);
                    if (__any_sync(0xffffffffu, m_new != m_used)) {
                        if (kSingle && t > 0) {
                            // O may be rescaled once the PV product of the previous key tile is complete.
                            // This is key tile g_tile - 1 of the CTA; completions 0 .. g_tile - 3 are certain
                            // (this tile's S was issued after them), so the barrier is in phase g_tile - 2
                            // or g_tile - 1 and the parity of g_tile - 2 tells the two apart.
                            ok = __all_sync(0xffffffffu, mbar_wait(bar_pv, g_tile & 1u, abort_flag, a.status));
                            if (!ok) break;
                            tc_fence_after();
                        }
                        const float alpha = (m_new == -INFINITY) ? 1.f : ex2(m_used - m_new);
                        l_run *= alpha;
                        m_used = m_new;
                        if (t > 0) {
#pragma unroll
                            for (int c0 = 0; c0 < D; c0 += 32) {
                                uint32_t o[32];
                                tmem_ld32(tO + c0, o);
                                tmem_wait_ld();
#pragma unroll
                                for (int c = 0; c < 32; ++c) o[c] = __float_as_uint(__uint_as_float(o[c]) * alpha);
                                tmem_st32(tO + c0, o);
                            }
                        }
                    }
                    neg_m = (m_used == -INFINITY) ? 0.f : -m_used;
                    s1 = exp_row<0, kFirst>(r, a.scale_log2, neg_m, tS);
                }
                l_run += s1;
                // P goes to the MMA issuer in two pieces, so that the first piece of the PV product runs while the
                // rest of the row is exponentiated.  (A rescale has stored its O columns before the first hand-over.)
                tmem_wait_st();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(bar_p);
                if constexpr (!kHalves) {                            // otherwise the rest of the row is the other warpgroup's
                    l_run += exp_row<kFirst, kCols>(r, a.scale_log2, neg_m, tS);

                    tmem_wait_st();
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(bar_p2);
                }
            }
            if (!ok) break;

            // ---- epilogue: normalise and store this thread's row ----
            if (n > 0) {
                float2* half_ml = half_all + (o_cnt & 1) * (2 * kTileM);
                if (kHalves) {
                    half_ml[s * kTileM + row] = make_float2(m_used, l_run);
                    __syncwarp();
                    if (lane == 0) mbar_arrive(bar_half);
                    ok = mbar_wait(bar_half, o_cnt & 1, abort_flag, a.status);
                }
                ok = __all_sync(0xffffffffu, ok && mbar_wait(bar_of, o_cnt & 1, abort_flag, a.status));
                ++o_cnt;
                if (!ok) break;
                tc_fence_after();
                float w_own = 1.f, w_other = 0.f;
                if (kHalves) {
                    const float2 other = half_ml[(s ^ 1) * kTileM + row];
                    const float m_row = fmaxf(m_used, other.x);
                    w_own = m_used == -INFINITY ? 0.f : ex2(m_used - m_row);
                    w_other = other.x == -INFINITY ? 0.f : ex2(other.x - m_row);
                    l_run = w_own * l_run + w_other * other.y;
                    m_used = m_row;
                }
                const int in_tile = row_t >> a.pack_shift, token = (tile ? it.token0_b : it.token0_a) + in_tile;
                const int head = it.head0 + (row_t & ((1 << a.pack_shift) - 1));
                const int part = kQuad ? it.part * 4 + (warp & 3) : it.part;
                bool store = token < a.n_tokens;
                if (a.mode != kModePhase2) store = store && (tile ? it.row0_b : it.row0_a) + in_tile < it.main_len;
                const float inv_l = l_run > 0.f ? 1.f / l_run : 0.f;
                const float lse = (l_run > 0.f) ? (m_used + log2f(l_run)) * 0.6931471805599453f : -INFINITY;
                const size_t orow = static_cast<size_t>(token) * a.Hq + head;
                // The whole accumulator row goes to registers first (the logits' registers are free by
                // now), so that the accumulator can be handed back before the row is scaled and stored.
                constexpr int kOut = kHalves ? D / 2 : D;          // of the row's outputs, this thread's
                const int out0 = kHalves ? s * kOut : 0;
                uint32_t o[kOut];
#pragma unroll
                for (int c0 = 0; c0 < kOut; c0 += 32) PULSAR_TMEM_LD32_AT(tO + out0 + c0, o, c0);
                if (kHalves) {
                    uint32_t x[kOut];
#pragma unroll
                    for (int c0 = 0; c0 < kOut; c0 += 32) PULSAR_TMEM_LD32_AT(tO_other + out0 + c0, x, c0);
                    tmem_wait_ld();
#pragma unroll
                    for (int c = 0; c < kOut; ++c)
                        o[c] = __float_as_uint(__uint_as_float(o[c]) * w_own + __uint_as_float(x[c]) * w_other);
                }
                tmem_wait_ld();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(bar_oe);
                if (store) {
                    // A row per lane: every store instruction touches 32 rows.  With 16-byte stores each sector went
                    // out in two halves and an item's rows took about 5000 cycles; whole 32-byte sectors per store:
                    // Phase 1 at 16K 0.714 -> 0.701 ms, at 64K 6.05 -> 6.02 ms.
                    if (a.part_O != nullptr) {
                        float* dst = a.part_O + (static_cast<size_t>(part) * a.n_tokens * a.Hq + orow) * D + out0;
#pragma unroll
                        for (int c = 0; c < kOut; c += 8) {
                            uint32_t v[8];
#pragma unroll
                            for (int k = 0; k < 8; ++k) v[k] = __float_as_uint(__uint_as_float(o[c + k]) * inv_l);
                            store_32b(dst + c, v, a.out_wide);
                        }
                        if (out0 == 0) a.part_LSE[static_cast<size_t>(part) * a.n_tokens * a.Hq + orow] = lse;
                    } else {
                        uint16_t* dst = a.O + orow * D + out0;
#pragma unroll
                        for (int c = 0; c < kOut; c += 16) {
                            uint32_t v[8];
#pragma unroll
                            for (int k = 0; k < 8; ++k)
                                v[k] = pack_bf16x2(__uint_as_float(o[c + 2 * k]) * inv_l, __uint_as_float(o[c + 2 * k + 1]) * inv_l);
                            store_32b(dst + c, v, a.out_wide);
                        }
                        if (out0 == 0 && a.LSE != nullptr) a.LSE[orow] = lse;
                    }
                }
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(bars + SL::bItemEmpty + slot);
        }
    }

    tc_fence_before();
    __syncthreads();
    if (warp == kMmaWarp) tmem_dealloc(tmem_base, 512);
    if (kBeside) grid_dependency_wait();
}

// ---------------------------------------------------------------------------------------------
// Host side: tensor maps, planning, launches
// ---------------------------------------------------------------------------------------------
using EncodeTiledFn = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                   const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                   CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn() {
    static EncodeTiledFn fn = nullptr;
    if (fn == nullptr) {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) != cudaSuccess ||
            q != cudaDriverEntryPointSuccess) {
            (void)cudaGetLastError();
            return nullptr;
        }
        fn = reinterpret_cast<EncodeTiledFn>(p);
    }
    return fn;
}

// [rows, heads, d] bf16 viewed as (d, heads, rows); box = (64, box_heads, box_rows), 128-byte swizzle.
bool make_map_3d(CUtensorMap* m, const void* base, int64_t rows, int heads, int d, int box_heads, int box_rows) {
    EncodeTiledFn fn = encode_fn();
    if (!fn) return false;
    cuuint64_t dims[3] = {static_cast<cuuint64_t>(d), static_cast<cuuint64_t>(heads), static_cast<cuuint64_t>(rows)};
    cuuint64_t strides[2] = {static_cast<cuuint64_t>(d) * 2, static_cast<cuuint64_t>(heads) * d * 2};
    cuuint32_t box[3] = {64, static_cast<cuuint32_t>(box_heads), static_cast<cuuint32_t>(box_rows)};
    cuuint32_t estr[3] = {1, 1, 1};
    return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims, strides, box, estr,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// [rows, width] bf16; box = (64, 128), 128-byte swizzle.
bool make_map_2d(CUtensorMap* m, const void* base, int64_t rows, int64_t width) {
    EncodeTiledFn fn = encode_fn();
    if (!fn) return false;
    cuuint64_t dims[2] = {static_cast<cuuint64_t>(width), static_cast<cuuint64_t>(rows)};
    cuuint64_t strides[1] = {static_cast<cuuint64_t>(width) * 2};
    cuuint32_t box[2] = {64, kTileN};
    cuuint32_t estr[2] = {1, 1};
    return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, estr,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Launched with programmatic stream serialization: the CTAs may be placed while the launch before it on the stream
// drains, and wait for that launch before they touch global memory.
template <int D>
int32_t launch_attn(const CUtensorMap& q, const CUtensorMap& k, const CUtensorMap& v, const CUtensorMap& kp,
                    const CUtensorMap& vp, AttnArgs a, cudaStream_t stream,
                    const VarlenTable* table = nullptr) {
    constexpr int smem = SmemLayout<D>::kDynBytes;
    // The opt-in to more than 48 KB of dynamic shared memory is a per-device function attribute;
    // setting it on every launch keeps multi-device processes correct and costs well under a microsecond.
    const int grid = a.n_items < sm_count() ? a.n_items : sm_count();     // one persistent CTA per SM
    if (grid <= 0) return PULSAR_OK;
    a.out_wide = aligned(a.part_O != nullptr ? static_cast<const void*>(a.part_O) : a.O, 32) ? 1 : 0;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(static_cast<unsigned>(grid));
    cfg.blockDim = dim3(kAttnThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    const auto launch = [&](auto kernel, const auto& tab) -> cudaError_t {
        const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        return e != cudaSuccess ? e : cudaLaunchKernelEx(&cfg, kernel, q, k, v, kp, vp, a, tab);
    };
    static const VarlenTable kNoSequences{};
    const VarlenTable& tab = table ? *table : kNoSequences;
    const auto pick = [&](auto tile_max, auto beside) -> cudaError_t {
        constexpr bool kTileMax = decltype(tile_max)::value, kBeside = decltype(beside)::value;
        return a.quad     ? launch(attn_kernel<D, true, true, kTileMax, kBeside>, NoTable{})
               : a.single ? launch(attn_kernel<D, false, true, kTileMax, kBeside>, tab)
                          : launch(attn_kernel<D, false, false, kTileMax, kBeside>, tab);
    };
    PULSAR_CUDA_OK(a.beside     ? pick(std::false_type{}, std::true_type{})        // (tile_max is the generation step's)
                   : a.tile_max ? pick(std::true_type{}, std::false_type{})
                                : pick(std::false_type{}, std::false_type{}));
    count_launch();
    return PULSAR_OK;
}

// The work counter of a launch of n_items work items, cleared: null where every item has a CTA of its own.
int32_t clear_counter(int32_t*& counter, int64_t n_items, cudaStream_t stream) {
    if (n_items <= sm_count()) {
        counter = nullptr;
        return PULSAR_OK;
    }
    PULSAR_CUDA_OK(launch_kernel(clear_counter_kernel, dim3(1), dim3(1), 0, stream, true, counter));
    count_launch();
    return PULSAR_OK;
}

struct Phase1Plan {
    int n_blocks;
    int last_len;                             // tokens of the last block
    int pack_shift;                           // log2 of the query rows a token has in a tile
    int single, items_block, items_last;      // one query tile per work item; items per head (group) of a full and of the last block
    int n_items;
    size_t pref_rows, pref_bytes, total;
};

// log2 of a power of two
int log2_of(int g) {
    int s = 0;
    while ((1 << s) < g) ++s;
    return s;
}

// Causal attention with few items takes work items of one query tile instead of two: twice the items, and a key tile costs
// the chain of one tile (0.79 us with d = 64, 0.84 with d = 128; an item 2.5 and 2.8 us more) instead of two interleaved
// ones (1.39 and 1.51 us, 3.0 and 3.4 us).  While every tile has an SM of its own that is the shorter time, and with more pairs than
// SMs the pair is the better unit.  Between the two, tiles that cost alike are walked two after the other and lose
// (one block of 1024 of 32 heads, d = 64, behind 8192 prefix rows: 130 us against 110), tiles that differ are dealt out
// evenly and win (8 blocks of 512 of 8 heads, prefix growing to 7168 rows: 61 us against 95).  So both are laid out on the
// SMs in the order in which the items are drawn, and the shorter time decides.  Over 270 shapes that is the better
// form, or within 4 % of it.
// A run is a block or a sequence: its prefix rows and its own; in the order in which the items are drawn.
struct CausalRun {
    int64_t prefix;
    int len;
};
constexpr int kMaxCausalRuns = 512;             // more runs than that are more pairs than SMs
struct CausalCost {
    int64_t tile, item;                         // ns
};
CausalCost causal_cost(int per_item, int32_t d) {
    return per_item == 1 ? CausalCost{d == 64 ? 785 : 840, d == 64 ? 2500 : 2760} : CausalCost{d == 64 ? 1392 : 1513, d == 64 ? 2986 : 3390};
}

bool causal_single(const CausalRun* runs, int n_runs, int64_t heads, int tile_tokens, int32_t d) {
    const int sms = sm_count();
    const CausalCost cost[2] = {causal_cost(1, d), causal_cost(2, d)};
    const auto items = [&](int64_t tokens) {
        int64_t n = 0;
        for (int r = 0; r < n_runs; ++r) n += (runs[r].len + tokens - 1) / tokens * heads;
        return n;
    };
    if (items(tile_tokens) <= sms) return true;
    if (items(2 * tile_tokens) > sms || sms > 1024) return false;
    int64_t time[2];
    for (int per_item = 1; per_item <= 2; ++per_item) {
        const int tokens = per_item * tile_tokens;
        int64_t done[1024];                     // when each SM is free again, the earliest first (a heap)
        int n = 0;
        for (int r = 0; r < n_runs; ++r)
            for (int i = (runs[r].len + tokens - 1) / tokens - 1; i >= 0; --i) {
                const int rows = std::min(runs[r].len, (i + 1) * tokens);
                const int64_t t = ((runs[r].prefix + kTileN - 1) / kTileN + (rows + kTileN - 1) / kTileN) * cost[per_item - 1].tile +
                                  cost[per_item - 1].item;
                for (int64_t h = 0; h < heads; ++h) {
                    if (n < sms) {
                        done[n++] = t;
                        if (n == sms) std::make_heap(done, done + n, std::greater<int64_t>());
                        continue;
                    }
                    std::pop_heap(done, done + n, std::greater<int64_t>());
                    done[n - 1] += t;
                    std::push_heap(done, done + n, std::greater<int64_t>());
                }
            }
        time[per_item - 1] = *std::max_element(done, done + n);
    }
    return time[0] < time[1];
}

// log2 of the heads of a KV head that share a query tile of causal attention.  With all g heads of 128/g tokens in a tile,
// both tiles of a work item end in the same key tile; with 128 tokens of one head the second needs one more, which
// it walks alone, and a run's last pair of tiles is the emptier the fewer of its 256 rows the run has left.  Against that, the
// items that run at the same time cover g times as many tokens and no longer read the same K/V tiles in step.  With d = 64, where a
// tile is half as large and the GPU is below its power limit, packing gains 3.5 % (45K ragged 0.916 -> 0.884 ms); with
// d = 128 it costs 0.7-1 % from 32K on (64K 5.33 -> 5.37 ms, 128K 14.12 -> 14.27 ms; 16K the same), so there the items have
// to take kPackGain per cent of their time at most.  Causal attention alone, 32 heads of 8 KV heads, us, apart / together: 14
// blocks of 186 tokens 28.7 / 22.3, 16 of 300 53.5 / 38.2, 11 of 512 51.0 / 47.8, 13 of 767 93.6 / 89.3, 16 of 1000 (93 % of
// the time by the rule) 175 / 173, 16 of 1500 (95 %) 313 / 317; 60 of 130, 16 heads of 4, 51.2 / 36.8.  The group must be a power
// of two up to 16.
constexpr int kPackGain = 94;
int causal_pack_shift(const CausalRun* runs, int n_runs, int32_t Hq, int32_t Hkv, int32_t d) {
    const int g = Hq / Hkv;
    if (g > 16 || (g & (g - 1)) != 0) return 0;
    if (d == 64 || g == 1) return log2_of(g);
    const CausalCost cost = causal_cost(2, d);
    const auto time = [&](int64_t heads, int tile_tokens) {
        int64_t t = 0;
        for (int r = 0; r < n_runs; ++r) {
            const int64_t n_pref = (runs[r].prefix + kTileN - 1) / kTileN;
            for (int row = 0; row < runs[r].len; row += 2 * tile_tokens)
                t += (n_pref + (std::min(row + 2 * tile_tokens, runs[r].len) + kTileN - 1) / kTileN) * cost.tile + cost.item;
        }
        return t * heads;
    };
    return time(Hkv, kTileM / g) * 100 < time(Hq, kTileM) * kPackGain ? log2_of(g) : 0;
}

// whole_only: the entry point takes only sequences made of whole blocks.
int32_t plan_phase1(int64_t L, int32_t Hq, int32_t Hkv, int32_t d, int32_t block_size, int32_t prefix_total,
                    Phase1Plan& p, bool whole_only = false) {
    if (L <= 0 || Hq <= 0 || Hkv <= 0 || block_size <= 0 || prefix_total < 0) return PULSAR_ERR_INVALID_ARG;
    if ((d != 64 && d != 128) || Hq % Hkv != 0 || L >= (1ll << 31)) return PULSAR_ERR_SHAPE;
    if (whole_only && L % block_size != 0) return PULSAR_ERR_SHAPE;
    const int64_t B = (L + block_size - 1) / block_size;       // the last block holds the tokens that remain
    if (B > 65535 || Hq > 65535) return PULSAR_ERR_SHAPE;
    if (prefix_total > (1 << 30)) return PULSAR_ERR_SHAPE;
    p.n_blocks = static_cast<int>(B);
    p.pref_rows = static_cast<size_t>(prefix_total > 0 ? prefix_total : 1);
    p.last_len = static_cast<int>(L - (B - 1) * block_size);
    p.pref_bytes = round_up(p.pref_rows * Hkv * d * 2, 256);
    p.total = 2 * p.pref_bytes + 256;                        // gathered prefix K, V and the work counter
    // How long each block's prefix is stands on the device.  It is taken to grow evenly to prefix_total, as in a whole
    // context and as blocks are dealt to GPUs in turn or in zigzag; a single block is taken to see all of it.  (Several
    // blocks that all see a long prefix, the last GPU of a context cut into runs of blocks, would do 1.1-1.2 times
    // better with pairs; pairs would cost the others up to 1.6 times.)
    CausalRun runs[kMaxCausalRuns];
    const int n_runs = static_cast<int>(std::min<int64_t>(B, kMaxCausalRuns));
    for (int64_t i = 0; i < n_runs; ++i)
        runs[i] = {B > 1 ? prefix_total * (B - 1 - i) / (B - 1) : prefix_total, i == 0 ? p.last_len : block_size};
    p.pack_shift = causal_pack_shift(runs, n_runs, Hq, Hkv, d);
    const int64_t heads = p.pack_shift ? Hkv : Hq;
    const int tile_tokens = kTileM >> p.pack_shift;
    p.single = B <= kMaxCausalRuns && causal_single(runs, static_cast<int>(B), heads, tile_tokens, d) ? 1 : 0;
    const int64_t tokens = static_cast<int64_t>(p.single ? 1 : 2) * tile_tokens;
    p.items_block = static_cast<int>((block_size + tokens - 1) / tokens);
    p.items_last = static_cast<int>((p.last_len + tokens - 1) / tokens);
    const int64_t items = ((B - 1) * p.items_block + p.items_last) * heads;
    if (items >= (1ll << 31)) return PULSAR_ERR_SHAPE;
    p.n_items = static_cast<int>(items);
    return PULSAR_OK;
}

// Number of KV parts for Phase 2 when the caller leaves the choice to the library: the J that
// minimises a simple time model --
//   rounds(J) * (tiles per part * t_tile + t_item)  +  partial traffic(J) / HBM bandwidth,
// rounds = ceil(items / CTAs).  More parts fill the last round better and shorten it, but every
// part writes and re-reads fp32 partials.  The constants are those of a pair of query tiles against 128-key tiles that come from
// HBM (about 2 us a tile; per-item prologue and epilogue about 6 us) and stand for every call: items of one query tile take
// about 0.8 and 2.8 us from L2 (causal_cost), so against their partials' traffic
// the model cuts them somewhat finer than these costs would.  Few rows against long contexts are cut by plan_decode, which takes only the room for partials from here.
int32_t choose_splits(int32_t nq, int64_t L, int32_t Hq, int32_t Hkv, int32_t d) {
    const int g = Hq / Hkv;
    const int64_t row_tiles = (static_cast<int64_t>(nq) * g + kTileM - 1) / kTileM;
    const int64_t items = (row_tiles + 1) / 2 * Hkv;               // a work item is a pair of row tiles
    const int64_t kv_tiles = (L + kTileN - 1) / kTileN;
    const double ctas = sm_count(), t_tile_us = 2.0, t_item_us = 6.0, hbm_bytes_per_us = 6.0e6;
    double best_t = 0;
    int64_t best = 1;
    // Only the j without an empty part, ceil(tiles / ceil(tiles / j)) == j, are worth a look: at most twice the square
    // root of the tiles.  After j comes the part count of the next smaller part size.  (Walking all j took 6.5 us of
    // every call at 1024 tiles.)
    for (int64_t j = 1, tiles_per_part; j <= kv_tiles && j <= 1024;
         j = tiles_per_part > 1 ? (kv_tiles + tiles_per_part - 2) / (tiles_per_part - 1) : kv_tiles + 1) {
        tiles_per_part = (kv_tiles + j - 1) / j;
        const double rounds = static_cast<double>((items * j + static_cast<int64_t>(ctas) - 1) / static_cast<int64_t>(ctas));
        const double partial = j > 1 ? 2.0 * j * nq * Hq * (d + 1) * 4.0 / hbm_bytes_per_us : 0.0;
        const double t = rounds * (static_cast<double>(tiles_per_part) * t_tile_us + t_item_us) + partial;
        if (best_t == 0 || t < best_t) { best_t = t; best = j; }
    }
    return static_cast<int32_t>(best);
}

// Decode shapes: all query rows of a KV head (tokens x heads per KV head) fit one quarter of a
// tile, so the kernel works on four copies of them, one key quarter each; every copy is a partial
// of its own (four times the partials, merged with the KV parts).
inline bool phase2_quad(int32_t nq, int32_t g) { return nq * g <= 32; }

// Keys per KV part: L / n_splits when that divides; otherwise the parts are whole 128-key tiles,
// ceil(tiles / n_splits) each, the last one shorter.  0 if some part would be empty.
int64_t phase2_split_len(int64_t L, int32_t n_splits) {
    if (n_splits <= 0) return 0;
    if (L % n_splits == 0) return L / n_splits;
    const int64_t kv_tiles = (L + kTileN - 1) / kTileN;
    const int64_t tiles_per_part = (kv_tiles + n_splits - 1) / n_splits;
    if ((kv_tiles + tiles_per_part - 1) / tiles_per_part != n_splits) return 0;
    return tiles_per_part * kTileN;
}

// How a generation step cuts context and shard.
struct GenerateCut {
    int n_parts;
    int64_t split_len;        // context keys per part
    bool shard_apart;         // the shard is part 0; otherwise it stands in front of the last part's context keys
    bool lengthened;          // parts of fewer than four key tiles became longer than n_splits parts of the context are: P
                              // is then formed with every tile's own maximum, as it is in parts of one tile (with a
                              // maximum that lags it is 8-10 % further from float64 in decode shapes, 3-5 % in others;
                              // from four tiles on one tile more is worth 1 % and less, and the rescaling of O would cost 7 %)
};

// Either the context in n_splits parts and the shard as one more (J + 1 parts), or context and shard together in parts of
// equally many key tiles, at most n_splits of them, with the shard in front of the last part's context keys where
// it fits there.  The second form has fewer partials and keeps the work items at one per SM where the first opens
// another round (1024 key tiles, 8 KV heads: 152 items on 148 SMs, 97 us against 92; 72 tiles, 4 KV heads: 11.8 against
// 10.6 us), so it is taken unless its longest chain of key tiles is clearly the longer one (n_splits = 1 with 32
// tiles on each side: 53 us against 37).  An item beyond the first of a CTA costs about three tiles more.
GenerateCut cut_generate(int64_t L_ctx, int64_t gen_rows, int64_t items_per_part, int32_t n_splits) {
    const int64_t ctx = (L_ctx + kTileN - 1) / kTileN, gen = (gen_rows + kTileN - 1) / kTileN;      // key tiles
    const int64_t J = n_splits, sms = sm_count();
    const auto chain = [&](int64_t parts, int64_t tiles, int64_t shard_tiles) {
        const int64_t rounds = (parts * items_per_part + sms - 1) / sms;
        return std::max(rounds * (tiles + 3) - 3, shard_tiles);
    };
    const int64_t own = (ctx + J - 1) / J, own_chain = chain(J + 1, own, gen);
    const int64_t joint = (ctx + gen + J - 1) / J, parts = (ctx + joint - 1) / joint;
    const bool fits = ctx - (parts - 1) * joint + gen <= joint;
    const int64_t joint_chain = fits ? chain(parts, joint, 0) : chain(parts + 1, joint, gen);
    if (joint_chain > own_chain + std::max<int64_t>(2, own_chain / 8))
        return {static_cast<int>(J + 1), phase2_split_len(L_ctx, n_splits), true, false};
    return {static_cast<int>(fits ? parts : parts + 1), joint * kTileN, !fits, joint > own && own < 4};
}

}  // namespace
}  // namespace pulsar

using namespace pulsar;

// =============================================================================================
// Phase 1
// =============================================================================================
extern "C" size_t pulsar_phase1_workspace_bytes(int64_t L, int32_t Hq, int32_t Hkv, int32_t d, int32_t block_size,
                                                int32_t prefix_total) {
    Phase1Plan p;
    if (plan_phase1(L, Hq, Hkv, d, block_size, prefix_total, p) != PULSAR_OK) return 0;
    return p.total;
}

extern "C" int32_t pulsar_phase1_attn(const uint16_t* Q, const uint16_t* K, const uint16_t* V, int64_t L, int32_t Hq,
                                      int32_t Hkv, int32_t d, int32_t block_size, const int32_t* prefix_idx,
                                      const int32_t* prefix_len, int32_t prefix_total, float softmax_scale,
                                      uint16_t* O, float* LSE, uint16_t* K_ret, uint16_t* V_ret, void* workspace,
                                      size_t workspace_bytes, int32_t* device_status, void* stream_) {
    Phase1Plan p;
    int32_t rc = plan_phase1(L, Hq, Hkv, d, block_size, prefix_total, p);
    if (rc != PULSAR_OK) return rc;
    if (!Q || !K || !V || !O || !prefix_len || !workspace || (prefix_total > 0 && !prefix_idx))
        return PULSAR_ERR_INVALID_ARG;
    if ((K_ret == nullptr) != (V_ret == nullptr)) return PULSAR_ERR_INVALID_ARG;
    if (!aligned(Q, 16) || !aligned(K, 16) || !aligned(V, 16) || !aligned(O, 16) || !aligned(prefix_len, 4) ||
        !aligned(prefix_idx, 4) || (LSE && !aligned(LSE, 4)) || (K_ret && !aligned(K_ret, 16)) ||
        (V_ret && !aligned(V_ret, 16)) || !aligned(workspace, 256))
        return PULSAR_ERR_ALIGNMENT;
    if (workspace_bytes < p.total) return PULSAR_ERR_WORKSPACE;
    rc = check_device();
    if (rc != PULSAR_OK) return rc;
    cudaStream_t stream = static_cast<cudaStream_t>(stream_);

    uint16_t* Kp = static_cast<uint16_t*>(workspace);
    uint16_t* Vp = reinterpret_cast<uint16_t*>(static_cast<char*>(workspace) + p.pref_bytes);
    int32_t* counter = reinterpret_cast<int32_t*>(static_cast<char*>(workspace) + 2 * p.pref_bytes);

    CUtensorMap tmQ, tmK, tmV, tmKp, tmVp;
    if (!make_map_3d(&tmQ, Q, L, Hq, d, 1 << p.pack_shift, kTileM >> p.pack_shift) || !make_map_2d(&tmK, K, L, static_cast<int64_t>(Hkv) * d) ||
        !make_map_2d(&tmV, V, L, static_cast<int64_t>(Hkv) * d) ||
        !make_map_2d(&tmKp, Kp, static_cast<int64_t>(p.pref_rows), static_cast<int64_t>(Hkv) * d) ||
        !make_map_2d(&tmVp, Vp, static_cast<int64_t>(p.pref_rows), static_cast<int64_t>(Hkv) * d))
        return PULSAR_ERR_CUDA;

    if (prefix_total > 0) {
        PULSAR_CUDA_OK(launch_kernel(gather_prefix_kernel, dim3(prefix_total), dim3(128), 0, stream, true,
                                     reinterpret_cast<const uint4*>(K), reinterpret_cast<const uint4*>(V), prefix_idx,
                                     prefix_len, p.n_blocks, block_size, L, Hkv * d * 2 / 16, reinterpret_cast<uint4*>(Kp),
                                     reinterpret_cast<uint4*>(Vp), counter, device_status));
        count_launch();
    } else {
        rc = clear_counter(counter, p.n_items, stream);
        if (rc != PULSAR_OK) return rc;
    }

    AttnArgs a{};
    a.mode = kModePhase1;
    a.Hkv = Hkv;
    a.single = p.single;
    a.pairs = p.items_block;
    a.last_len = p.last_len;
    a.pairs_last = p.items_last;
    a.n_items = p.n_items;
    a.n_blocks = p.n_blocks;
    a.counter = counter;
    a.n_tokens = static_cast<int>(L);
    a.Hq = Hq;
    a.g = Hq / Hkv;
    a.pack_shift = p.pack_shift;
    a.block_size = block_size;
    a.prefix_total = prefix_total;
    a.prefix_len = prefix_len;
    a.scale_log2 = (softmax_scale > 0.f ? softmax_scale : 1.0f / sqrtf(static_cast<float>(d))) * 1.4426950408889634f;
    a.O = O;
    a.LSE = LSE;
    a.status = device_status;
    rc = d == 128 ? launch_attn<128>(tmQ, tmK, tmV, tmKp, tmVp, a, stream)
                  : launch_attn<64>(tmQ, tmK, tmV, tmKp, tmVp, a, stream);
    if (rc != PULSAR_OK) return rc;

    if (K_ret) {
        const size_t bytes = static_cast<size_t>(L) * Hkv * d * 2;
        PULSAR_CUDA_OK(cudaMemcpyAsync(K_ret, K, bytes, cudaMemcpyDeviceToDevice, stream));
        PULSAR_CUDA_OK(cudaMemcpyAsync(V_ret, V, bytes, cudaMemcpyDeviceToDevice, stream));
    }
    return PULSAR_OK;
}

// =============================================================================================
// Phase 1 with the logical blocks spread over several GPUs (block-to-host mapping, Section 3 and
// Appendix J): what one GPU runs before and after the exchange of summary K/V rows.
// =============================================================================================
extern "C" int32_t pulsar_pack_summary_kv(const uint16_t* K, const uint16_t* V, int32_t n_local, int32_t block_size,
                                          int32_t Hkv, int32_t d, const int32_t* sel_chunks,
                                          const int32_t* block_ids, int32_t n_blocks, int32_t chunk, int32_t k,
                                          int32_t sink, uint16_t* K_send, uint16_t* V_send, int32_t* device_status,
                                          void* stream) {
    if (n_local <= 0 || block_size <= 0 || Hkv <= 0 || d <= 0 || n_blocks <= 0 || chunk <= 0 || k < 0 || sink < 0)
        return PULSAR_ERR_INVALID_ARG;
    if ((static_cast<int64_t>(Hkv) * d * 2) % 16 != 0 || block_size % chunk != 0 || k > block_size / chunk ||
        sink > block_size || n_local > n_blocks || static_cast<int64_t>(n_local) * block_size >= (1ll << 31))
        return PULSAR_ERR_SHAPE;
    if (!K || !V || !sel_chunks || !block_ids || !K_send || !V_send) return PULSAR_ERR_INVALID_ARG;
    if (!aligned(K, 16) || !aligned(V, 16) || !aligned(K_send, 16) || !aligned(V_send, 16) ||
        !aligned(sel_chunks, 4) || !aligned(block_ids, 4))
        return PULSAR_ERR_ALIGNMENT;
    int32_t rc = check_device();
    if (rc != PULSAR_OK) return rc;
    const int64_t rows = sink + static_cast<int64_t>(n_local) * k * chunk;
    if (rows == 0) return PULSAR_OK;
    if (rows > 0x7fffffffll) return PULSAR_ERR_SHAPE;
    PULSAR_CUDA_OK(launch_kernel(pack_summary_kernel, dim3(copy_ctas(rows, Hkv * d * 2 / 16)), dim3(kCopyThreads), 0, static_cast<cudaStream_t>(stream),
                                 true, reinterpret_cast<const uint4*>(K), reinterpret_cast<const uint4*>(V), sel_chunks, block_ids,
                                 n_local, n_blocks, block_size, chunk, k, sink, Hkv * d * 2 / 16, reinterpret_cast<uint4*>(K_send),
                                 reinterpret_cast<uint4*>(V_send), device_status));
    count_launch();
    return PULSAR_OK;
}

extern "C" int32_t pulsar_gather_kv_rows(const uint16_t* K, const uint16_t* V, int64_t rows_in, int32_t Hkv, int32_t d,
                                         const int32_t* idx, int32_t n_idx, uint16_t* K_out, uint16_t* V_out,
                                         int32_t* device_status, void* stream) {
    if (rows_in <= 0 || Hkv <= 0 || d <= 0 || n_idx < 0) return PULSAR_ERR_INVALID_ARG;
    if ((static_cast<int64_t>(Hkv) * d * 2) % 16 != 0 || rows_in >= (1ll << 31)) return PULSAR_ERR_SHAPE;
    if (n_idx == 0) return PULSAR_OK;
    if (!K || !V || !idx || !K_out || !V_out) return PULSAR_ERR_INVALID_ARG;
    if (!aligned(K, 16) || !aligned(V, 16) || !aligned(K_out, 16) || !aligned(V_out, 16) || !aligned(idx, 4))
        return PULSAR_ERR_ALIGNMENT;
    int32_t rc = check_device();
    if (rc != PULSAR_OK) return rc;
    PULSAR_CUDA_OK(launch_kernel(gather_rows_kernel, dim3(copy_ctas(n_idx, Hkv * d * 2 / 16)), dim3(kCopyThreads), 0,
                                 static_cast<cudaStream_t>(stream), true, reinterpret_cast<const uint4*>(K),
                                 reinterpret_cast<const uint4*>(V), idx, n_idx, rows_in,
                                 Hkv * d * 2 / 16, reinterpret_cast<uint4*>(K_out), reinterpret_cast<uint4*>(V_out), device_status));
    count_launch();
    return PULSAR_OK;
}

extern "C" int32_t pulsar_phase1_attn_sharded(const uint16_t* Q, const uint16_t* K, const uint16_t* V, int64_t L_local,
                                              int32_t Hq, int32_t Hkv, int32_t d, int32_t block_size,
                                              const uint16_t* K_prefix, const uint16_t* V_prefix,
                                              int32_t prefix_total, const int32_t* prefix_len_local,
                                              float softmax_scale, uint16_t* O, float* LSE, void* workspace,
                                              size_t workspace_bytes, int32_t* device_status, void* stream_) {
    Phase1Plan p;
    int32_t rc = plan_phase1(L_local, Hq, Hkv, d, block_size, prefix_total, p, /*whole_only=*/true);
    if (rc != PULSAR_OK) return rc;
    if (!Q || !K || !V || !O || !prefix_len_local || !workspace || (prefix_total > 0 && (!K_prefix || !V_prefix)))
        return PULSAR_ERR_INVALID_ARG;
    if (!aligned(Q, 16) || !aligned(K, 16) || !aligned(V, 16) || !aligned(O, 16) || !aligned(prefix_len_local, 4) ||
        !aligned(K_prefix, 16) || !aligned(V_prefix, 16) || (LSE && !aligned(LSE, 4)) || !aligned(workspace, 256))
        return PULSAR_ERR_ALIGNMENT;
    if (workspace_bytes < 256) return PULSAR_ERR_WORKSPACE;
    rc = check_device();
    if (rc != PULSAR_OK) return rc;
    cudaStream_t stream = static_cast<cudaStream_t>(stream_);
    int32_t* counter = static_cast<int32_t*>(workspace);

    // With no prefix at all the two prefix maps still have to describe valid memory: use K, V.
    const uint16_t* Kp = prefix_total > 0 ? K_prefix : K;
    const uint16_t* Vp = prefix_total > 0 ? V_prefix : V;
    CUtensorMap tmQ, tmK, tmV, tmKp, tmVp;
    if (!make_map_3d(&tmQ, Q, L_local, Hq, d, 1 << p.pack_shift, kTileM >> p.pack_shift) ||
        !make_map_2d(&tmK, K, L_local, static_cast<int64_t>(Hkv) * d) ||
        !make_map_2d(&tmV, V, L_local, static_cast<int64_t>(Hkv) * d) ||
        !make_map_2d(&tmKp, Kp, static_cast<int64_t>(p.pref_rows), static_cast<int64_t>(Hkv) * d) ||
        !make_map_2d(&tmVp, Vp, static_cast<int64_t>(p.pref_rows), static_cast<int64_t>(Hkv) * d))
        return PULSAR_ERR_CUDA;

    rc = clear_counter(counter, p.n_items, stream);
    if (rc != PULSAR_OK) return rc;

    AttnArgs a{};
    a.mode = kModePhase1;
    a.Hkv = Hkv;
    a.single = p.single;
    a.pairs = p.items_block;
    a.last_len = p.last_len;
    a.pairs_last = p.items_last;
    a.n_items = p.n_items;
    a.n_blocks = p.n_blocks;
    a.counter = counter;
    a.n_tokens = static_cast<int>(L_local);
    a.Hq = Hq;
    a.g = Hq / Hkv;
    a.pack_shift = p.pack_shift;
    a.block_size = block_size;
    a.prefix_total = prefix_total;
    a.prefix_len = prefix_len_local;
    a.scale_log2 = (softmax_scale > 0.f ? softmax_scale : 1.0f / sqrtf(static_cast<float>(d))) * 1.4426950408889634f;
    a.O = O;
    a.LSE = LSE;
    a.status = device_status;
    return d == 128 ? launch_attn<128>(tmQ, tmK, tmV, tmKp, tmVp, a, stream)
                    : launch_attn<64>(tmQ, tmK, tmV, tmKp, tmVp, a, stream);
}

// =============================================================================================
// Phase 2
// =============================================================================================
namespace {
int32_t plan_phase2(int32_t nq, int32_t B, int32_t block_size, int32_t Hq, int32_t Hkv, int32_t d, int32_t& n_splits,
                    size_t& part_o_bytes, size_t& part_l_bytes) {
    if (nq <= 0 || B <= 0 || block_size <= 0 || Hq <= 0 || Hkv <= 0 || n_splits < 0) return PULSAR_ERR_INVALID_ARG;
    if ((d != 64 && d != 128) || Hq % Hkv != 0) return PULSAR_ERR_SHAPE;
    const int g = Hq / Hkv;
    if (g != 1 && g != 2 && g != 4 && g != 8 && g != 16) return PULSAR_ERR_SHAPE;
    const int64_t L = static_cast<int64_t>(B) * block_size;
    if (L >= (1ll << 31) || Hkv > 65535) return PULSAR_ERR_SHAPE;
    if (n_splits == 0) n_splits = choose_splits(nq, L, Hq, Hkv, d);
    if (n_splits > 65535 || phase2_split_len(L, n_splits) == 0) return PULSAR_ERR_SHAPE;
    part_o_bytes = round_up(static_cast<size_t>(n_splits) * nq * Hq * d * 4, 256);
    part_l_bytes = round_up(static_cast<size_t>(n_splits) * nq * Hq * 4, 256);
    return PULSAR_OK;
}
}  // namespace

extern "C" int32_t pulsar_phase2_choose_splits(int32_t nq, int32_t B, int32_t block_size, int32_t Hq, int32_t Hkv,
                                               int32_t d) {
    int32_t n = 0;
    size_t a, b;
    if (plan_phase2(nq, B, block_size, Hq, Hkv, d, n, a, b) != PULSAR_OK) return 0;
    return n;
}

extern "C" size_t pulsar_phase2_workspace_bytes(int32_t nq, int32_t B, int32_t block_size, int32_t Hq, int32_t Hkv,
                                                int32_t d, int32_t n_splits) {
    size_t a, b;
    if (plan_phase2(nq, B, block_size, Hq, Hkv, d, n_splits, a, b) != PULSAR_OK) return 0;
    if (phase2_quad(nq, Hq / Hkv)) return 4 * (a + b);
    return n_splits == 1 ? 256 : a + b + 256;              // partials and the work counter
}

namespace {
// pulsar_phase2_attn up to the merge, which is left to the caller (todo).
int32_t phase2_launch(const uint16_t* Qq, int32_t nq, const uint16_t* Kb, const uint16_t* Vb, int32_t B, int32_t block_size,
                      int32_t Hq, int32_t Hkv, int32_t d, float softmax_scale, int32_t n_splits, uint16_t* O, float* LSE,
                      float* part_O, float* part_LSE, void* workspace, size_t workspace_bytes, int32_t* device_status,
                      bool beside, MergeTodo& todo, void* stream_) {
    todo = {};
    size_t po_bytes, pl_bytes;
    const bool user_parts = part_O != nullptr;
    if ((part_O == nullptr) != (part_LSE == nullptr)) return PULSAR_ERR_INVALID_ARG;
    if (user_parts && n_splits <= 0) return PULSAR_ERR_INVALID_ARG;
    int32_t rc = plan_phase2(nq, B, block_size, Hq, Hkv, d, n_splits, po_bytes, pl_bytes);
    if (rc != PULSAR_OK) return rc;
    if (!Qq || !Kb || !Vb || !O) return PULSAR_ERR_INVALID_ARG;
    if (!aligned(Qq, 16) || !aligned(Kb, 16) || !aligned(Vb, 16) || !aligned(O, 16) || (LSE && !aligned(LSE, 4)) ||
        (part_O && !aligned(part_O, 16)) || (part_LSE && !aligned(part_LSE, 4)) ||
        (workspace && !aligned(workspace, 256)))
        return PULSAR_ERR_ALIGNMENT;
    const bool quad = !user_parts && phase2_quad(nq, Hq / Hkv);
    const int copies = quad ? 4 : 1;
    po_bytes *= copies;                                        // both stay multiples of 256
    pl_bytes *= copies;
    const bool need_ws = (n_splits > 1 || quad) && !user_parts;
    if (need_ws && (!workspace || workspace_bytes < po_bytes + pl_bytes + (quad ? 0 : 256))) return PULSAR_ERR_WORKSPACE;
    rc = check_device();
    if (rc != PULSAR_OK) return rc;
    cudaStream_t stream = static_cast<cudaStream_t>(stream_);

    const int64_t L = static_cast<int64_t>(B) * block_size;
    const int g = Hq / Hkv;
    const float scale_log2 = (softmax_scale > 0.f ? softmax_scale : 1.0f / sqrtf(static_cast<float>(d))) * 1.4426950408889634f;
    if (!user_parts && decode_takes(nq, Hq, Hkv, L)) {
        DecodeCall c{};
        c.Q = Qq;
        c.n = nq;
        c.Hq = Hq;
        c.Hkv = Hkv;
        c.d = d;
        c.K = Kb;
        c.V = Vb;
        c.ctx_len = L;
        c.scale_log2 = scale_log2;
        c.O = O;
        c.LSE = LSE;
        c.workspace = workspace;
        c.max_parts = need_ws ? static_cast<int64_t>(n_splits) * copies : 0;
        c.beside = beside;
        return launch_decode(c, todo, stream);
    }
    CUtensorMap tmQ, tmK, tmV;
    if (!make_map_3d(&tmQ, Qq, nq, Hq, d, g, (quad ? 32 : kTileM) / g) ||
        !make_map_2d(&tmK, Kb, L, static_cast<int64_t>(Hkv) * d) ||
        !make_map_2d(&tmV, Vb, L, static_cast<int64_t>(Hkv) * d))
        return PULSAR_ERR_CUDA;

    const bool partial_out = n_splits > 1 || user_parts || quad;
    float* pO = user_parts ? part_O : (need_ws ? static_cast<float*>(workspace) : nullptr);
    float* pL = user_parts ? part_LSE
                           : (need_ws ? reinterpret_cast<float*>(static_cast<char*>(workspace) + po_bytes) : nullptr);

    AttnArgs a{};
    a.mode = kModePhase2;
    a.n_tokens = nq;
    a.Hq = Hq;
    a.g = g;
    a.pack_shift = log2_of(g);
    a.split_len = static_cast<int>(phase2_split_len(L, n_splits));
    a.kv_len = static_cast<int>(L);
    a.quad = quad ? 1 : 0;
    a.beside = beside ? 1 : 0;
    a.scale_log2 = scale_log2;
    a.O = O;
    a.LSE = LSE;
    a.part_O = partial_out ? pO : nullptr;
    a.part_LSE = partial_out ? pL : nullptr;
    a.status = device_status;
    const int tokens_per_tile = kTileM / g;
    const int row_tiles = (nq + tokens_per_tile - 1) / tokens_per_tile;
    a.Hkv = Hkv;
    a.single = row_tiles == 1 ? 1 : 0;               // includes every decode shape (quad)
    a.pairs = (row_tiles + 1) / 2;
    a.n_items = a.pairs * Hkv * n_splits;
    if (a.n_items > sm_count() && need_ws && !quad && workspace_bytes >= po_bytes + pl_bytes + 256) {
        // More items than CTAs: hand them out as CTAs become free (the last part is shorter, and the
        // last round would otherwise leave CTAs idle behind the slowest one).  The result of an
        // item does not depend on which CTA computes it.
        a.counter = reinterpret_cast<int32_t*>(static_cast<char*>(workspace) + po_bytes + pl_bytes);
        rc = clear_counter(a.counter, a.n_items, stream);
        if (rc != PULSAR_OK) return rc;
        a.beside = 0;                                // the cleared counter has to be waited for
    }
    rc = d == 128 ? launch_attn<128>(tmQ, tmK, tmV, tmK, tmV, a, stream)
                  : launch_attn<64>(tmQ, tmK, tmV, tmK, tmV, a, stream);
    if (rc == PULSAR_OK && partial_out) todo = {pO, pL, n_splits * copies};
    return rc;
}

int32_t merge_launch(const MergeTodo& todo, int32_t nq, int32_t Hq, int32_t d, uint16_t* O, float* LSE, void* stream, bool beside = false) {
    if (todo.n_parts == 0) return PULSAR_OK;
    return launch_lse_merge(todo.part_O, todo.part_LSE, todo.n_parts, static_cast<int64_t>(nq) * Hq, d, O, LSE,
                            static_cast<cudaStream_t>(stream), beside);
}
}  // namespace

extern "C" int32_t pulsar_phase2_attn(const uint16_t* Qq, int32_t nq, const uint16_t* Kb, const uint16_t* Vb,
                                      int32_t B, int32_t block_size, int32_t Hq, int32_t Hkv, int32_t d,
                                      float softmax_scale, int32_t n_splits, uint16_t* O, float* LSE, float* part_O,
                                      float* part_LSE, void* workspace, size_t workspace_bytes,
                                      int32_t* device_status, void* stream) {
    MergeTodo todo;
    const int32_t rc = phase2_launch(Qq, nq, Kb, Vb, B, block_size, Hq, Hkv, d, softmax_scale, n_splits, O, LSE, part_O, part_LSE,
                                     workspace, workspace_bytes, device_status, false, todo, stream);
    return rc != PULSAR_OK ? rc : merge_launch(todo, nq, Hq, d, O, LSE, stream);
}

// =============================================================================================
// One layer of a context: selection, Phase 1 and the Phase-2 attention of its query
// =============================================================================================
// Phase 2 needs nothing of Phase 1 but the keys and values that both read, so its attention is launched beside the
// selection, which is a chain of latencies on 16 SMs, and its merge beside Phase 1 (4096 tokens 32.6 -> 24.6 us with the
// selection's one launch).  With more work items than SMs, whose counter has to be cleared before it, it follows Phase 1.
// So it does where it shares memory with the other two, which the three calls may, one after the other.
namespace {
struct Span {
    const void* p;
    uint64_t bytes;
};
bool meet(const Span& a, const Span& b) {
    const auto begin = [](const Span& s) { return static_cast<uint64_t>(reinterpret_cast<uintptr_t>(s.p)); };
    const auto end = [&](const Span& s) { return begin(s) + std::min<uint64_t>(s.bytes, UINT64_MAX - begin(s)); };      // (a size may be "all there is")
    return a.p != nullptr && b.p != nullptr && begin(a) < end(b) && begin(b) < end(a);
}
template <int N, int M>
bool meet(const Span (&a)[N], const Span (&b)[M]) {
    return std::any_of(a, a + N, [&](const Span& x) { return std::any_of(b, b + M, [&](const Span& y) { return meet(x, y); }); });
}
}  // namespace

extern "C" int32_t pulsar_encode_step(const uint32_t* token_ids, int64_t L, int32_t vocab_size, int32_t block_size, int32_t chunk,
                                      int32_t k, int32_t sink, int32_t* sel_chunks, int32_t* prefix_idx, int32_t* prefix_len,
                                      void* select_workspace, size_t select_workspace_bytes, const uint16_t* Q, const uint16_t* K,
                                      const uint16_t* V, int32_t Hq, int32_t Hkv, int32_t d, int32_t prefix_total,
                                      float softmax_scale, uint16_t* O, float* LSE, void* phase1_workspace,
                                      size_t phase1_workspace_bytes, const uint16_t* Qq, int32_t nq, int32_t n_splits,
                                      uint16_t* O2, float* LSE2, void* phase2_workspace, size_t phase2_workspace_bytes,
                                      int32_t* device_status, void* stream) {
    int32_t rc = launch_maxidf_select(token_ids, L, vocab_size, block_size, chunk, k, sink, sel_chunks, prefix_idx, prefix_len, nullptr,
                                      nullptr, select_workspace, select_workspace_bytes, device_status, stream, true);
    if (rc != PULSAR_OK) return rc;
    MergeTodo todo;
    const auto phase1 = [&] {
        return pulsar_phase1_attn(Q, K, V, L, Hq, Hkv, d, block_size, prefix_total > 0 ? prefix_idx : nullptr, prefix_len, prefix_total,
                                  softmax_scale, O, LSE, nullptr, nullptr, phase1_workspace, phase1_workspace_bytes, device_status, stream);
    };
    const auto phase2 = [&](bool beside) {
        return phase2_launch(Qq, nq, K, V, 1, static_cast<int32_t>(L), Hq, Hkv, d, softmax_scale, n_splits, O2, LSE2, nullptr, nullptr,
                             phase2_workspace, phase2_workspace_bytes, device_status, beside, todo, stream);
    };
    int32_t parts = n_splits;
    size_t unused_a, unused_b;
    rc = plan_phase2(nq, 1, static_cast<int32_t>(L), Hq, Hkv, d, parts, unused_a, unused_b);
    if (rc != PULSAR_OK) return rc;
    const int64_t pairs = (static_cast<int64_t>(nq) * (Hq / Hkv) + 2 * kTileM - 1) / (2 * kTileM);
    const uint64_t n = static_cast<uint64_t>(L), B = (n + block_size - 1) / block_size;
    const uint64_t entries = std::max<uint64_t>(prefix_total, sink + (B - 1) * k * chunk), row_q = 2ull * Hq * d, row_kv = 2ull * Hkv * d;
    const Span written2[] = {{O2, nq * row_q}, {LSE2, 4ull * nq * Hq}, {phase2_workspace, phase2_workspace_bytes}};
    const Span written1[] = {{O, n * row_q}, {LSE, 4 * n * Hq}, {phase1_workspace, phase1_workspace_bytes},
                             {select_workspace, select_workspace_bytes}, {sel_chunks, 4 * B * k}, {prefix_idx, 4 * entries},
                             {prefix_len, 4 * B}};
    const Span read1[] = {{token_ids, 4 * n}, {Q, n * row_q}, {K, n * row_kv}, {V, n * row_kv}}, read2[] = {{Qq, nq * row_q}};
    const bool beside = pairs * Hkv * parts <= sm_count() && !meet(written2, written1) && !meet(written2, read1) && !meet(written1, read2);
    rc = beside ? phase2(true) : phase1();
    if (rc != PULSAR_OK) return rc;
    rc = beside ? phase1() : phase2(false);
    return rc != PULSAR_OK ? rc : merge_launch(todo, nq, Hq, d, O2, LSE2, stream, beside);
}

// =============================================================================================
// Phase 2, generation step (Algorithm 1 lines 11-16): context parts + the generation shard
// =============================================================================================
extern "C" size_t pulsar_phase2_generate_workspace_bytes(int32_t n_new, int32_t B, int32_t block_size, int32_t Hq,
                                                         int32_t Hkv, int32_t d, int32_t n_splits) {
    size_t a, b;
    if (plan_phase2(n_new, B, block_size, Hq, Hkv, d, n_splits, a, b) != PULSAR_OK) return 0;
    // one more part than the context has: the generation shard; four partials per part for decode shapes
    const size_t parts = static_cast<size_t>(n_splits + 1) * (phase2_quad(n_new, Hq / Hkv) ? 4 : 1);
    return round_up(parts * n_new * Hq * d * 4, 256) + round_up(parts * n_new * Hq * 4, 256);
}

extern "C" int32_t pulsar_phase2_generate_step(const uint16_t* Qnew, const uint16_t* Knew, const uint16_t* Vnew,
                                               int32_t n_new, const uint16_t* Kb, const uint16_t* Vb, int32_t B,
                                               int32_t block_size, uint16_t* Kgen, uint16_t* Vgen, int32_t gen_len,
                                               int32_t gen_capacity, int32_t Hq, int32_t Hkv, int32_t d,
                                               float softmax_scale, int32_t n_splits, uint16_t* O, float* LSE,
                                               void* workspace, size_t workspace_bytes, int32_t* device_status,
                                               void* stream_) {
    size_t unused_a, unused_b;
    if (gen_len < 0 || gen_capacity <= 0) return PULSAR_ERR_INVALID_ARG;
    int32_t rc = plan_phase2(n_new, B, block_size, Hq, Hkv, d, n_splits, unused_a, unused_b);
    if (rc != PULSAR_OK) return rc;
    if (static_cast<int64_t>(gen_len) + n_new > gen_capacity) return PULSAR_ERR_SHAPE;
    if (!Qnew || !Knew || !Vnew || !Kb || !Vb || !Kgen || !Vgen || !O || !workspace) return PULSAR_ERR_INVALID_ARG;
    if (!aligned(Qnew, 16) || !aligned(Knew, 16) || !aligned(Vnew, 16) || !aligned(Kb, 16) || !aligned(Vb, 16) ||
        !aligned(Kgen, 16) || !aligned(Vgen, 16) || !aligned(O, 16) || (LSE && !aligned(LSE, 4)) ||
        !aligned(workspace, 256))
        return PULSAR_ERR_ALIGNMENT;
    const int64_t L_ctx = static_cast<int64_t>(B) * block_size;
    const GenerateCut cut = cut_generate(L_ctx, static_cast<int64_t>(gen_len) + n_new,
                                         (static_cast<int64_t>(n_new) * (Hq / Hkv) + 2 * kTileM - 1) / (2 * kTileM) * Hkv, n_splits);
    const int n_parts = cut.n_parts;
    const bool quad = phase2_quad(n_new, Hq / Hkv);
    const int copies = quad ? 4 : 1;
    const size_t po_bytes = round_up(static_cast<size_t>(n_parts) * copies * n_new * Hq * d * 4, 256);
    const size_t pl_bytes = round_up(static_cast<size_t>(n_parts) * copies * n_new * Hq * 4, 256);
    // The stated size is asked for however the call is cut: what fits must not depend on the length of the shard.
    if (workspace_bytes < pulsar_phase2_generate_workspace_bytes(n_new, B, block_size, Hq, Hkv, d, n_splits)) return PULSAR_ERR_WORKSPACE;
    rc = check_device();
    if (rc != PULSAR_OK) return rc;
    cudaStream_t stream = static_cast<cudaStream_t>(stream_);

    const int64_t L = static_cast<int64_t>(B) * block_size;
    const int g = Hq / Hkv;
    const float scale_log2 = (softmax_scale > 0.f ? softmax_scale : 1.0f / sqrtf(static_cast<float>(d))) * 1.4426950408889634f;
    if (decode_takes(n_new, Hq, Hkv, L)) {
        DecodeCall c{};
        c.Q = Qnew;
        c.n = n_new;
        c.Hq = Hq;
        c.Hkv = Hkv;
        c.d = d;
        c.K = Kb;
        c.V = Vb;
        c.ctx_len = L;
        c.Kgen = Kgen;
        c.Vgen = Vgen;
        c.Knew = Knew;
        c.Vnew = Vnew;
        c.gen_len = gen_len;
        c.scale_log2 = scale_log2;
        c.O = O;
        c.LSE = LSE;
        c.workspace = workspace;
        c.max_parts = static_cast<int64_t>(n_splits + 1) * copies;
        MergeTodo todo;
        rc = launch_decode(c, todo, stream);
        return rc != PULSAR_OK ? rc : merge_launch(todo, n_new, Hq, d, O, LSE, stream);
    }
    const size_t row_bytes = static_cast<size_t>(Hkv) * d * 2;
    CUtensorMap tmQ, tmK, tmV, tmKg, tmVg;
    if (!make_map_3d(&tmQ, Qnew, n_new, Hq, d, g, (quad ? 32 : kTileM) / g) ||
        !make_map_2d(&tmK, Kb, L, static_cast<int64_t>(Hkv) * d) ||
        !make_map_2d(&tmV, Vb, L, static_cast<int64_t>(Hkv) * d) ||
        // The shard's maps end at its live rows: TMA zero-fills the rest of the last key tile, so
        // whatever the unwritten rows [gen_len + n_new, gen_capacity) hold (NaN patterns of an
        // uninitialised cache included) never reaches the PV product as 0 * NaN.
        !make_map_2d(&tmKg, Kgen, static_cast<int64_t>(gen_len) + n_new, static_cast<int64_t>(Hkv) * d) ||
        !make_map_2d(&tmVg, Vgen, static_cast<int64_t>(gen_len) + n_new, static_cast<int64_t>(Hkv) * d))
        return PULSAR_ERR_CUDA;

    float* pO = static_cast<float*>(workspace);
    float* pL = reinterpret_cast<float*>(static_cast<char*>(workspace) + po_bytes);
    AttnArgs a{};
    a.mode = kModePhase2;
    a.n_tokens = n_new;
    a.Hq = Hq;
    a.g = g;
    a.pack_shift = log2_of(g);
    a.split_len = static_cast<int>(cut.split_len);
    a.ctx_part0 = cut.shard_apart ? 1 : 0;
    a.kv_len = static_cast<int>(L);
    a.gen_part = cut.shard_apart ? 0 : n_parts - 1;
    a.tile_max = cut.lengthened ? 1 : 0;
    a.gen_len = gen_len;
    a.gen_total = gen_len + n_new;
    a.quad = quad ? 1 : 0;
    a.scale_log2 = scale_log2;
    a.O = O;
    a.LSE = LSE;
    a.part_O = pO;
    a.part_LSE = pL;
    a.status = device_status;
    const int tokens_per_tile = kTileM / g;
    const int row_tiles = (n_new + tokens_per_tile - 1) / tokens_per_tile;
    a.Hkv = Hkv;
    a.single = row_tiles == 1 ? 1 : 0;               // includes every decode shape (quad)
    // KV(q) is appended to the generation shard first (Algorithm 1 line 15)
    if (a.single && n_new * (d / 8) <= kAppendVecs) {
        a.Knew = reinterpret_cast<const uint4*>(Knew);
        a.Vnew = reinterpret_cast<const uint4*>(Vnew);
        a.Kgen = reinterpret_cast<uint4*>(Kgen);
        a.Vgen = reinterpret_cast<uint4*>(Vgen);
    } else {
        const int vecs = static_cast<int>(n_new * row_bytes / 16);
        PULSAR_CUDA_OK(launch_kernel(append_kv_kernel, dim3((vecs + 255) / 256), dim3(256), 0, stream, true,
                                     reinterpret_cast<const uint4*>(Knew), reinterpret_cast<const uint4*>(Vnew),
                                     reinterpret_cast<uint4*>(reinterpret_cast<char*>(Kgen) + gen_len * row_bytes),
                                     reinterpret_cast<uint4*>(reinterpret_cast<char*>(Vgen) + gen_len * row_bytes), vecs));
        count_launch();
    }
    a.pairs = (row_tiles + 1) / 2;
    a.n_items = a.pairs * Hkv * n_parts;
    rc = d == 128 ? launch_attn<128>(tmQ, tmK, tmV, tmKg, tmVg, a, stream)
                  : launch_attn<64>(tmQ, tmK, tmV, tmKg, tmVg, a, stream);
    if (rc != PULSAR_OK) return rc;
    return launch_lse_merge(pO, pL, n_parts * copies, static_cast<int64_t>(n_new) * Hq, d, O, LSE, stream);
}

// =============================================================================================
// Causal attention over assembled inputs of different lengths (Algorithm 1 line 8 as the paper
// runs it: every token of Input_i is a query, the keys and values are those of Input_i itself)
// =============================================================================================
extern "C" int32_t pulsar_causal_varlen_attn(const uint16_t* Q, const uint16_t* K, const uint16_t* V,
                                             int64_t total_rows, const int32_t* cu_seqlens_host, int32_t n_seq,
                                             int32_t Hq, int32_t Hkv, int32_t d, float softmax_scale, uint16_t* O,
                                             float* LSE, void* workspace, size_t workspace_bytes,
                                             int32_t* device_status, void* stream_) {
    if (total_rows <= 0 || n_seq <= 0 || Hq <= 0 || Hkv <= 0 || !cu_seqlens_host) return PULSAR_ERR_INVALID_ARG;
    if ((d != 64 && d != 128) || Hq % Hkv != 0 || total_rows >= (1ll << 31) || n_seq > kMaxVarlenSeqs || Hq > 65535)
        return PULSAR_ERR_SHAPE;
    if (cu_seqlens_host[0] != 0 || cu_seqlens_host[n_seq] != total_rows) return PULSAR_ERR_SHAPE;
    for (int j = 0; j < n_seq; ++j)
        if (cu_seqlens_host[j + 1] <= cu_seqlens_host[j]) return PULSAR_ERR_SHAPE;       // empty or descending
    if (!Q || !K || !V || !O || !workspace) return PULSAR_ERR_INVALID_ARG;
    if (!aligned(Q, 16) || !aligned(K, 16) || !aligned(V, 16) || !aligned(O, 16) || (LSE && !aligned(LSE, 4)) ||
        !aligned(workspace, 256))
        return PULSAR_ERR_ALIGNMENT;
    if (workspace_bytes < 256) return PULSAR_ERR_WORKSPACE;
    int32_t rc = check_device();
    if (rc != PULSAR_OK) return rc;
    cudaStream_t stream = static_cast<cudaStream_t>(stream_);

    VarlenTable vt{};
    vt.n_seq = n_seq;
    for (int j = 0; j <= n_seq; ++j) vt.start[j] = cu_seqlens_host[j];
    CausalRun runs[kMaxVarlenSeqs];
    for (int k = 0; k < n_seq; ++k) runs[k] = {0, vt.start[n_seq - k] - vt.start[n_seq - 1 - k]};
    const int pack_shift = causal_pack_shift(runs, n_seq, Hq, Hkv, d), heads = pack_shift ? Hkv : Hq;
    const int tile_tokens = kTileM >> pack_shift;
    const int single = causal_single(runs, n_seq, heads, tile_tokens, d) ? 1 : 0, tokens = (single ? 1 : 2) * tile_tokens;
    int64_t pairs_total = 0;
    for (int k = 0; k < n_seq; ++k) {
        vt.pair_cum[k] = static_cast<int>(pairs_total);
        pairs_total += (static_cast<int64_t>(runs[k].len) + tokens - 1) / tokens;
    }
    vt.pair_cum[n_seq] = static_cast<int>(pairs_total);
    if (pairs_total * heads >= (1ll << 31)) return PULSAR_ERR_SHAPE;

    CUtensorMap tmQ, tmK, tmV;
    if (!make_map_3d(&tmQ, Q, total_rows, Hq, d, 1 << pack_shift, kTileM >> pack_shift) ||
        !make_map_2d(&tmK, K, total_rows, static_cast<int64_t>(Hkv) * d) ||
        !make_map_2d(&tmV, V, total_rows, static_cast<int64_t>(Hkv) * d))
        return PULSAR_ERR_CUDA;

    int32_t* counter = static_cast<int32_t*>(workspace);
    rc = clear_counter(counter, pairs_total * heads, stream);
    if (rc != PULSAR_OK) return rc;

    AttnArgs a{};
    a.mode = kModeVarlen;
    a.n_tokens = static_cast<int>(total_rows);
    a.Hq = Hq;
    a.g = Hq / Hkv;
    a.pack_shift = pack_shift;
    a.Hkv = Hkv;
    a.single = single;
    a.n_items = static_cast<int>(pairs_total) * heads;
    a.counter = counter;
    a.scale_log2 = (softmax_scale > 0.f ? softmax_scale : 1.0f / sqrtf(static_cast<float>(d))) * 1.4426950408889634f;
    a.O = O;
    a.LSE = LSE;
    a.status = device_status;
    return d == 128 ? launch_attn<128>(tmQ, tmK, tmV, tmK, tmV, a, stream, &vt)
                    : launch_attn<64>(tmQ, tmK, tmV, tmK, tmV, a, stream, &vt);
}

extern "C" int32_t pulsar_retain_block_kv(const uint16_t* K, const uint16_t* V, int64_t total_rows,
                                          const int32_t* cu_seqlens_host, int32_t n_seq, int32_t block_size,
                                          int32_t Hkv, int32_t d, uint16_t* K_ret, uint16_t* V_ret, void* stream) {
    if (total_rows <= 0 || n_seq <= 0 || block_size <= 0 || Hkv <= 0 || d <= 0 || !cu_seqlens_host)
        return PULSAR_ERR_INVALID_ARG;
    if (n_seq > kMaxVarlenSeqs || total_rows >= (1ll << 31) || (static_cast<int64_t>(Hkv) * d * 2) % 16 != 0 ||
        static_cast<int64_t>(n_seq) * block_size >= (1ll << 31))
        return PULSAR_ERR_SHAPE;
    if (cu_seqlens_host[0] != 0 || cu_seqlens_host[n_seq] != total_rows) return PULSAR_ERR_SHAPE;
    RetainTable tab{};
    for (int j = 0; j < n_seq; ++j) {
        if (cu_seqlens_host[j + 1] - cu_seqlens_host[j] < block_size) return PULSAR_ERR_SHAPE;   // shorter than a block
        tab.first[j] = cu_seqlens_host[j + 1] - block_size;
    }
    if (!K || !V || !K_ret || !V_ret) return PULSAR_ERR_INVALID_ARG;
    if (!aligned(K, 16) || !aligned(V, 16) || !aligned(K_ret, 16) || !aligned(V_ret, 16)) return PULSAR_ERR_ALIGNMENT;
    int32_t rc = check_device();
    if (rc != PULSAR_OK) return rc;
    const int64_t ctas = (static_cast<int64_t>(block_size) * (Hkv * d * 2 / 16) + kCopyVecs - 1) / kCopyVecs;
    if (ctas > 0x7fffffffll) return PULSAR_ERR_SHAPE;
    PULSAR_CUDA_OK(launch_kernel(retain_block_kv_kernel, dim3(static_cast<unsigned>(ctas), static_cast<unsigned>(n_seq)),
                                 dim3(kCopyThreads), 0, static_cast<cudaStream_t>(stream), true,
                                 reinterpret_cast<const uint4*>(K), reinterpret_cast<const uint4*>(V), tab, block_size,
                                 Hkv * d * 2 / 16, reinterpret_cast<uint4*>(K_ret), reinterpret_cast<uint4*>(V_ret)));
    count_launch();
    return PULSAR_OK;
}
