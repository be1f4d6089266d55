// Phase-2 attention of few query rows against a long context: the generation step and short queries (Section 3.2,
// Algorithm 1 lines 11-16), one launch from Q, K, V to the merged output.
//
// A call reads every key and value of the context once for at most eight query rows per KV head, so the memory system is the
// bound and the path from the first byte to the output is what a short context pays for.  Every warp is a pipeline of its own:
// it copies 4 KB units of K and V (16 keys with d = 128) into its ring with cp.async, forms S^T = K Q^T and O^T += V^T P^T on them
// with register-level matrix instructions -- keys, then outputs, in the 16 rows, the query rows in the eight columns -- and keeps
// its own running maximum, so no warp waits for another until its keys are used up.  Then the warps of a CTA merge in shared
// memory, and the CTAs of a KV head, which are a thread-block cluster, through distributed shared memory.
// tcgen05 would want 128 rows (4 of them used by a single token of 4 heads) and a round trip through TMEM, four
// barriers and a second launch for the merge on the way of every key tile.
// One token, us, that form / this one: 6001 keys of 2 heads 10.0 / 7.5, 22,842 of 8 (d = 64) 16.8 / 13.4, 55,734 of 2
// 20.6 / 15.2, 131,072 of 8 91.8 / 84.4 (0.99 of the measured copy rate).  A key costs an SM about 8 cycles (shared memory written
// and read once), HBM delivers one in 23 when all SMs read.
#include <algorithm>
#include <atomic>

#include "common.cuh"
#include "decode.cuh"

namespace pulsar {

namespace {

constexpr int kWarps = 8;
constexpr int kThreads = 32 * kWarps;
constexpr int kRows = 8;                        // query rows of a KV head: the columns of a matrix fragment
constexpr int kUnitBytes = 4096;
constexpr int kMaxClusterShift = 4;
constexpr int kMaxCluster = 1 << kMaxClusterShift;      // CTAs of a KV head that merge through distributed shared memory
constexpr int kMaxChunks = kRows * 4 + kMaxCluster;      // of 32 outputs, rounded up to a multiple of the cluster
constexpr int kUnits = 3;                       // of a warp's ring: one in use, two on their way
constexpr int kRingBytes = kWarps * kUnits * kUnitBytes;
constexpr int kSmemBytes = kRingBytes + kRows * kWarps * 8 + kMaxChunks * (8 + 32 * 4);

struct DecodeArgs {
    const uint16_t* Q;           // [n, Hq, D]
    const uint16_t *K, *V;       // context [ctx_len, Hkv, D]
    uint16_t *Kgen, *Vgen;       // generation shard: its first gen_len rows are read, the new ones appended
    const uint16_t *Knew, *Vnew; // KV of the new tokens [gen_total - gen_len, Hkv, D]
    int ctx_len, gen_len, gen_total;
    int Hq, Hkv, g_shift, n_rows;                // n_rows = n * g query rows of a KV head
    int cluster_shift, clusters;                 // log2 of the CTAs per cluster, clusters per KV head
    float scale_log2;
    uint16_t* O;
    float* LSE;
    float *part_O, *part_LSE;                    // clusters > 1: [clusters, n, Hq, D] and [clusters, n, Hq]
    int64_t part_rows;                           // n * Hq
};

__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src, uint32_t bytes) {
    asm volatile("cp.async.cg.shared.global.L2::128B [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }
__device__ __forceinline__ void ldmatrix4(uint32_t addr, uint32_t (&r)[4]) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void ldmatrix4_trans(uint32_t addr, uint32_t (&r)[4]) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void mma_bf16(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ uint32_t cluster_ctarank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_arrive_release() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ uint32_t map_to_rank(uint32_t addr, int rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
__device__ __forceinline__ void st_cluster2(uint32_t addr, float2 v) {
    asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};" ::"r"(addr), "f"(v.x), "f"(v.y) : "memory");
}
__device__ __forceinline__ void st_cluster1(uint32_t addr, float v) {
    asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(addr), "f"(v) : "memory");
}
__device__ __forceinline__ uint32_t movmatrix(uint32_t x) {
    uint32_t y;
    asm volatile("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(y) : "r"(x));
    return y;
}
__device__ __forceinline__ float warp_max(float x) {            // of the lanes' values that are numbers
    float y;
    asm volatile("redux.sync.max.f32 %0, %1, 0xffffffff;" : "=f"(y) : "f"(x));
    return y;
}
template <int N>                                               // of the first N lanes, in every one of them
__device__ __forceinline__ float low_lanes_sum(float x) {
#pragma unroll
    for (int d = N / 2; d > 0; d >>= 1) x += __shfl_xor_sync(0xffffffffu, x, d);
    return __shfl_sync(0xffffffffu, x, 0);
}
// 2^(m - M) for a maximum M over values of which m is one; 0 where m stands for no keys.
__device__ __forceinline__ float weight(float m, float M) { return m == -INFINITY ? 0.f : ex2(m - M); }

// Two CTAs per SM: while the keys of one are on their way, the other computes, and the next launch's CTAs find room
// beside the last of this one's.
// kBeside: see launch_lse_merge.
template <int D, bool kBeside>
__global__ void __launch_bounds__(kThreads, 2)
decode_kernel(const __grid_constant__ DecodeArgs a) {
    constexpr int kKeys = kUnitBytes / (2 * D);                // keys of a unit: 16 (d = 128), 32 (d = 64)
    constexpr int kVecs = D / 8;                               // 16-byte vectors of a row
    constexpr int kRowsPerCopy = 32 / kVecs;                   // rows a warp copies with one instruction
    constexpr int kCopies = kKeys / kRowsPerCopy;
    constexpr int kPitch = D + 4;                              // floats of a partial row: 2 * kPitch = 8 modulo the banks
    static_assert(kWarps * kRows * kPitch * 4 <= kRingBytes, "the warps' partials take the ring's place");
    extern __shared__ __align__(1024) uint8_t smem[];

    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int gid = lane >> 2, tig = lane & 3;
    const int kvh = blockIdx.y;
    const int C = 1 << a.cluster_shift;

    if (C > 1) cluster_arrive();                               // waited for before another CTA's memory is written
    if (!kBeside) grid_dependency_wait();
    else __threadfence();                                      // (the query rows are read through L1: nothing it holds of the last step)
    grid_launch_dependents();

    // ---- this CTA's pieces of kKeys keys: the context's first, then the shard's ----
    const int ctx_pieces = (a.ctx_len + kKeys - 1) / kKeys, gen_pieces = (a.gen_total + kKeys - 1) / kKeys;
    const int64_t pieces = ctx_pieces + gen_pieces;
    const int n_ctas = C * a.clusters;
    const int p_begin = static_cast<int>(pieces * blockIdx.x / n_ctas), p_end = static_cast<int>(pieces * (blockIdx.x + 1) / n_ctas);

    const uint32_t ring = smem_u32(smem) + warp * (kUnits * kUnitBytes);
    const int copy_row = lane / kVecs, copy_vec = lane % kVecs;
    const int64_t pitch = static_cast<int64_t>(a.Hkv) * D;     // elements between the rows of a head
    const int head_at = kvh * D + copy_vec * 8;
    const int64_t lane_at = copy_row * pitch + head_at;
    const int64_t copy_step = kRowsPerCopy * pitch;

    // A unit is K or V of a piece.  Row r goes to line r, its vector v to place v ^ (r & 7), so that the eight rows of a
    // matrix fragment lie in different banks.
    const auto load = [&](const uint16_t* ctx, const uint16_t* gen, const uint16_t* fresh, int p, int slot) {
        if (p < p_end) {
            const uint32_t dst = ring + slot * kUnitBytes + copy_row * (D * 2);
            if (p < ctx_pieces) {
                const int row0 = p * kKeys, n = a.ctx_len - row0;
                const uint16_t* src = ctx + row0 * pitch + lane_at;
#pragma unroll
                for (int i = 0; i < kCopies; ++i, src += copy_step) {
                    const int r = i * kRowsPerCopy + copy_row;
                    const uint32_t to = dst + i * (kRowsPerCopy * D * 2) + ((copy_vec ^ (r & 7)) << 4);
                    if (n >= kKeys) cp_async16(to, src, 16);
                    else cp_async16(to, r < n ? src : ctx, r < n ? 16 : 0);
                }
            } else {
                const int row0 = (p - ctx_pieces) * kKeys;
#pragma unroll
                for (int i = 0; i < kCopies; ++i) {
                    const int r = i * kRowsPerCopy + copy_row, row = row0 + r;
                    const uint32_t to = dst + i * (kRowsPerCopy * D * 2) + ((copy_vec ^ (r & 7)) << 4);
                    const uint16_t* src = (row < a.gen_len ? gen + row * pitch : fresh + (row - a.gen_len) * pitch) + head_at;
                    cp_async16(to, row < a.gen_total ? src : ctx, row < a.gen_total ? 16 : 0);
                }
            }
        }
        cp_async_commit();                                     // an empty group past the end keeps the count
    };

    const int p_first = p_begin + warp;
    load(a.K, a.Kgen, a.Knew, p_first, 0);
    load(a.V, a.Vgen, a.Vnew, p_first, 1);

    // ---- the query rows (row = token * g + head of the group) as B fragments ----
    uint32_t q[D / 16][2];
    {
        const int token = gid >> a.g_shift, head = (kvh << a.g_shift) + (gid & ((1 << a.g_shift) - 1));
        const uint32_t* src = reinterpret_cast<const uint32_t*>(a.Q + (static_cast<int64_t>(token) * a.Hq + head) * D) + tig;
#pragma unroll
        for (int kk = 0; kk < D / 16; ++kk) {
            q[kk][0] = gid < a.n_rows ? src[kk * 8] : 0u;
            q[kk][1] = gid < a.n_rows ? src[kk * 8 + 4] : 0u;
        }
    }
    // rows 2 tig and 2 tig + 1; o[c]: outputs 16 c + gid and 16 c + 8 + gid of both
    float o[D / 16][4], m[2] = {-INFINITY, -INFINITY}, l[2] = {0.f, 0.f};
#pragma unroll
    for (int c = 0; c < D / 16; ++c)
#pragma unroll
        for (int k = 0; k < 4; ++k) o[c][k] = 0.f;
    const int mi = lane >> 3, l8 = lane & 7;
    const uint32_t k_lane = ring + ((mi & 1) * 8 + l8) * (D * 2), k_x = ((mi >> 1) ^ l8) << 4;     // K: rows are keys
    const uint32_t v_lane = ring + ((mi >> 1) * 8 + l8) * (D * 2), v_x = ((mi & 1) ^ l8) << 4;     // V: read transposed

    // Units are consumed in the order K, V, K, V, ... and refilled in that order, each where the unit before it was.
    int slot = 0, free_slot = kUnits - 1;
    const auto next_unit = [&](const uint16_t* ctx, const uint16_t* gen, const uint16_t* fresh, int p) {
        cp_async_wait<kUnits - 2>();
        __syncwarp();
        load(ctx, gen, fresh, p, free_slot);
        const int now = slot;
        free_slot = now;
        slot = now + 1 == kUnits ? 0 : now + 1;
        return now * kUnitBytes;
    };
    for (int p = p_first; p < p_end; p += kWarps) {
        const int at_k = next_unit(a.K, a.Kgen, a.Knew, p + kWarps);
        // ---- S^T = K Q^T: keys gid and gid + 8 of each 16, rows 2 tig and 2 tig + 1 ----
        float s[kKeys / 16][4];
#pragma unroll
        for (int j = 0; j < kKeys / 16; ++j) {
            float t[2][4] = {};                                // two chains of products
#pragma unroll
            for (int kk = 0; kk < D / 16; ++kk) {
                uint32_t f[4];
                ldmatrix4(k_lane + at_k + j * (16 * D * 2) + ((kk * 32) ^ k_x), f);
                mma_bf16(t[kk & 1], f, q[kk][0], q[kk][1]);
            }
#pragma unroll
            for (int k = 0; k < 4; ++k) s[j][k] = t[0][k] + t[1][k];
        }
        // keys that do not exist, or that the token of a row must not see yet
        const bool shard = p >= ctx_pieces;
        if (shard || a.ctx_len - p * kKeys < kKeys) {
            const int row0 = (shard ? p - ctx_pieces : p) * kKeys;
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                const int token = (2 * tig + k) >> a.g_shift;
                const int n_vis = (shard ? min(a.gen_len + token + 1, a.gen_total) : a.ctx_len) - row0;
#pragma unroll
                for (int j = 0; j < kKeys / 16; ++j) {
                    if (16 * j + gid >= n_vis) s[j][k] = -INFINITY;
                    if (16 * j + gid + 8 >= n_vis) s[j][k + 2] = -INFINITY;
                }
            }
        }
        float x[2], alpha[2], neg[2];
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            x[k] = fmaxf(s[0][k], s[0][k + 2]);
#pragma unroll
            for (int j = 1; j < kKeys / 16; ++j) x[k] = max3(x[k], s[j][k], s[j][k + 2]);
        }
#pragma unroll
        for (int d = 4; d < 32; d <<= 1) {
            x[0] = fmaxf(x[0], __shfl_xor_sync(0xffffffffu, x[0], d));
            x[1] = fmaxf(x[1], __shfl_xor_sync(0xffffffffu, x[1], d));
        }
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            const float m_new = fmaxf(m[k], x[k] * a.scale_log2);
            alpha[k] = m_new == -INFINITY ? 1.f : ex2(m[k] - m_new);
            neg[k] = m_new == -INFINITY ? 0.f : -m_new;
            m[k] = m_new;
        }
        uint32_t pb[kKeys / 16][2];
        l[0] *= alpha[0];
        l[1] *= alpha[1];
#pragma unroll
        for (int j = 0; j < kKeys / 16; ++j) {
#pragma unroll
            for (int k = 0; k < 4; ++k) s[j][k] = ex2(fmaf(s[j][k], a.scale_log2, neg[k & 1]));
            l[0] += s[j][0] + s[j][2];
            l[1] += s[j][1] + s[j][3];
            pb[j][0] = movmatrix(pack_bf16x2(s[j][0], s[j][1]));      // [key][row] -> [row][key]
            pb[j][1] = movmatrix(pack_bf16x2(s[j][2], s[j][3]));
        }
        if (__any_sync(0xffffffffu, alpha[0] != 1.f || alpha[1] != 1.f)) {
#pragma unroll
            for (int c = 0; c < D / 16; ++c)
#pragma unroll
                for (int k = 0; k < 4; ++k) o[c][k] *= alpha[k & 1];
        }
        // ---- O^T += V^T P^T ----
        const int at_v = next_unit(a.V, a.Vgen, a.Vnew, p + kWarps);
#pragma unroll
        for (int j = 0; j < kKeys / 16; ++j)
#pragma unroll
            for (int c = 0; c < D / 16; ++c) {
                uint32_t f[4];
                ldmatrix4_trans(v_lane + at_v + j * (16 * D * 2) + ((c * 32) ^ v_x), f);
                mma_bf16(o[c], f, pb[j][0], pb[j][1]);
            }
        // The new tokens' rows go to the shard from the warp that has just read them (from Knew, so nothing waits for it).  Only the
        // last pieces have any: walked over every piece of the shard, this took half the time of calls with a long one (two tokens of
        // 32 heads, 20,000 keys and 1000 generated ones 21.5 us, 16.7 like this).  Reading the shard's whole pieces without
        // choosing each row's source gave another 0.2-1.8 us to such calls and cost the others 0.1-0.2.
        if (const int row0 = (p - ctx_pieces) * kKeys; shard && row0 + kKeys > a.gen_len) {
#pragma unroll 1
            for (int i = 0; i < kCopies; ++i) {
                const int row = row0 + i * kRowsPerCopy + copy_row;
                if (row >= a.gen_len && row < a.gen_total) {
                    const int64_t from = (row - a.gen_len) * pitch + head_at, to = row * pitch + head_at;
                    *reinterpret_cast<uint4*>(a.Kgen + to) = *reinterpret_cast<const uint4*>(a.Knew + from);
                    *reinterpret_cast<uint4*>(a.Vgen + to) = *reinterpret_cast<const uint4*>(a.Vnew + from);
                }
            }
        }
    }
#pragma unroll
    for (int d = 4; d < 32; d <<= 1) {
        l[0] += __shfl_xor_sync(0xffffffffu, l[0], d);
        l[1] += __shfl_xor_sync(0xffffffffu, l[1], d);
    }

    // ---- the warps' partials, brought to the CTA's maximum ----
    float2* w_ml = reinterpret_cast<float2*>(smem + kRingBytes);       // [kRows][kWarps]
    float2* c_ml = w_ml + kRows * kWarps;                                      // [cluster][slots], written by the peers
    float* c_o = reinterpret_cast<float*>(c_ml + kMaxChunks);                  // [cluster][slots][32], written by the peers
    float* w_o = reinterpret_cast<float*>(smem);                               // [kWarps][kRows][kPitch], where the rings were
    if (gid == 0) {
        w_ml[(2 * tig) * kWarps + warp] = make_float2(m[0], l[0]);
        w_ml[(2 * tig + 1) * kWarps + warp] = make_float2(m[1], l[1]);
    }
    __syncthreads();
    float f[2];
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        f[k] = -INFINITY;
#pragma unroll
        for (int w = gid; w < kWarps; w += 8) f[k] = fmaxf(f[k], w_ml[(2 * tig + k) * kWarps + w].x);
    }
#pragma unroll
    for (int d = 4; d < 32; d <<= 1) {
        f[0] = fmaxf(f[0], __shfl_xor_sync(0xffffffffu, f[0], d));
        f[1] = fmaxf(f[1], __shfl_xor_sync(0xffffffffu, f[1], d));
    }
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        f[k] = weight(m[k], f[k]);
        if (2 * tig + k < a.n_rows) {
            float* dst = w_o + (warp * kRows + 2 * tig + k) * kPitch + gid;
#pragma unroll
            for (int c = 0; c < D / 16; ++c) {
                dst[16 * c] = o[c][k] * f[k];
                dst[16 * c + 8] = o[c][k + 2] * f[k];
            }
        }
    }
    __syncthreads();

    // ---- one partial per CTA: a warp adds up 32 outputs of a row and hands them to the CTA of the cluster that finishes them ----
    const int chunks = a.n_rows * (D / 32), slots = (chunks + C - 1) >> a.cluster_shift;
    const int rank = C > 1 ? static_cast<int>(cluster_ctarank()) : 0;
    if (C > 1) cluster_wait();
    for (int c = warp; c < chunks; c += kWarps) {
        const int r = c / (D / 32);
        const float* src = w_o + r * kPitch + (c % (D / 32)) * 32 + lane;
        float y[2] = {0.f, 0.f};
#pragma unroll
        for (int w = 0; w < kWarps; ++w) y[w & 1] += src[w * (kRows * kPitch)];
        const float2 ml = lane < kWarps ? w_ml[r * kWarps + lane] : make_float2(-INFINITY, 0.f);
        const float M = warp_max(ml.x), sum = low_lanes_sum<kWarps>(weight(ml.x, M) * ml.y);
        const int at = rank * slots + (c >> a.cluster_shift), owner = c & (C - 1);
        st_cluster1(map_to_rank(smem_u32(c_o + at * 32 + lane), owner), y[0] + y[1]);
        if (lane == 0) st_cluster2(map_to_rank(smem_u32(c_ml + at), owner), make_float2(M, sum));
    }
    __syncwarp();
    if (C > 1) {
        cluster_arrive_release();
        cluster_wait();
    } else {
        __syncthreads();
    }

    // ---- and one per cluster ----
    for (int c = warp * C + rank; c < chunks; c += kWarps * C) {
        const int r = c / (D / 32), at_d = (c % (D / 32)) * 32 + lane, at = c >> a.cluster_shift;
        const float2 ml = lane < C ? c_ml[lane * slots + at] : make_float2(-INFINITY, 0.f);
        float x[kMaxCluster];
#pragma unroll
        for (int k = 0; k < kMaxCluster; ++k) x[k] = k < C ? c_o[(k * slots + at) * 32 + lane] : 0.f;
        const float M = warp_max(ml.x), w = weight(ml.x, M), sum = low_lanes_sum<kMaxCluster>(w * ml.y);
        float y[2] = {0.f, 0.f};
#pragma unroll
        for (int k = 0; k < kMaxCluster; ++k) y[k & 1] += __shfl_sync(0xffffffffu, w, k) * x[k];
        y[0] = (y[0] + y[1]) * (sum == 0.f ? 0.f : 1.f / sum);
        const float lse = sum == 0.f ? -INFINITY : (M + log2f(sum)) * 0.6931471805599453f;
        const int token = r >> a.g_shift, head = (kvh << a.g_shift) + (r & ((1 << a.g_shift) - 1));
        const int64_t row = static_cast<int64_t>(token) * a.Hq + head;
        if (a.clusters > 1) {
            const int64_t to = (blockIdx.x >> a.cluster_shift) * a.part_rows + row;
            a.part_O[to * D + at_d] = y[0];
            if (at_d == 0) a.part_LSE[to] = lse;
        } else {
            const float z = __shfl_xor_sync(0xffffffffu, y[0], 1);
            if ((lane & 1) == 0) *reinterpret_cast<uint32_t*>(a.O + row * D + at_d) = pack_bf16x2(y[0], z);
            if (at_d == 0 && a.LSE != nullptr) a.LSE[row] = lse;
        }
    }
    if (kBeside) grid_dependency_wait();
}

// ---------------------------------------------------------------------------------------------
// Host side
// ---------------------------------------------------------------------------------------------
using DecodeKernel = void (*)(DecodeArgs);

// Clusters of 2^shift CTAs that fit the current device at the same time.  The GPCs have different numbers of SMs, so that is
// less than two CTAs per SM give (B200: 148, 71, 33, 14 of 2, 4, 8, 16 CTAs).
int active_clusters(int shift) {
    static std::atomic<int> known[64][kMaxClusterShift + 1];   // per device; 0: not asked yet
    int dev = 0, n = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) {
        (void)cudaGetLastError();
        return 0;
    }
    n = known[dev][shift].load(std::memory_order_relaxed);
    if (n != 0) return n;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(1u << shift);
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = kSmemBytes;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 1u << shift;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    DecodeKernel kernel = decode_kernel<128, false>;
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes) != cudaSuccess ||
        cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess ||
        cudaOccupancyMaxActiveClusters(&n, kernel, &cfg) != cudaSuccess) {
        (void)cudaGetLastError();
        return 0;
    }
    known[dev][shift].store(n, std::memory_order_relaxed);
    return n;
}

// The calls taken: the rows fit a fragment's columns (with two, four or more tiles of eight rows per warp this form loses to the
// tensor cores': 16 rows against 6001 keys of 8 heads 13.1 us, 10.9 there; 32 rows against 32,768 44, 32 there), and the context is
// one whose keys a cluster can share.  (Shorter contexts are a few key tiles; what they launch is counted by their callers.)
constexpr int64_t kLeastKeys = 1024;

// How a call is spread: CTAs per cluster (2^shift) and clusters per KV head.
struct DecodePlan {
    int shift, clusters;
};

// One cluster per KV head, as large as fits for all heads at once, merges on chip.  More of them per head share the keys
// better but leave a merge to a second launch.  Measured, one / several, us: 6001 keys of 2 heads 7.5 / 7.6, 20,000 13.1 / 8.9,
// 55,734 27.5 / 14.8; 16,384 of 8 heads 16.6 / 16.7, 32,768 27.7 / 27.7, 131,072 86.4 / 83.5; 22,842 of 8 heads, d = 64,
// 13.0 / 12.7.  Of several, at least five per head: 131,072 keys of 8 heads 83.5 in 8 clusters of 4, 84.4 in 4 of 8.  Clusters of
// four from two per head on: of two CTAs they leave the launch with twice the clusters and partials, and 103,998 keys
// of 16 heads take 129.8 us, in 4 clusters of four 125.4 (the tensor cores' form 123.6), of 24 heads 183.5, 180.1 in two of four (180.8).
// What a call takes besides the data is 5.1 us with one cluster and 6.5 with a second launch.  The data goes at its CTAs' rate, 85
// kilobytes per us, 60 where two share an SM -- more CTAs than SMs, and clusters of eight or sixteen even of half as many, since a
// cluster keeps to few SMs -- or at the chip's: L2 where it holds the keys, else HBM, which CTAs packed that way do not use up.
// 1.5 us go to the form that needs no second launch: the host takes about one for it, and keys that are not in L2 make the two more
// alike (40 MB of 16 heads, d = 64, 9.4 and 9.4 us from L2, 10.9 and 12.0 from HBM).  Fitted to calls in a row of 141 shapes
// (1 to 48 KV heads, 4 to 400 MB of keys): the choice takes 1.00 times the better form's time in the middle, more than 1.1 in five, and
// 1.012 of the tensor cores' form at most, 0.75 in the middle (20,020 keys of 8 heads 12.9, one cluster 16.2, tensor cores 15.4).
DecodePlan plan_decode(const DecodeCall& c) {
    constexpr double kOne = 5.1, kMore = 6.5, kMargin = 1.5;                                       // us
    constexpr double kAlone = 85e3, kShared = 60e3, kL2 = 12.8e6, kHbm = 6.8e6, kHbmPacked = 5.8e6, kL2Bytes = 126e6;   // bytes (per us)
    const double bytes = 4.0 * (c.ctx_len + c.gen_len + c.n) * c.Hkv * c.d;
    const int sms = sm_count();
    const auto time = [&](const DecodePlan& p) {
        const int64_t ctas = static_cast<int64_t>(p.clusters) * c.Hkv << p.shift;
        const bool packed = p.shift >= 3 && ctas > sms / 2 && ctas <= sms, shared = packed || ctas > sms;
        return std::max(bytes / (ctas * (shared ? kShared : kAlone)), bytes / (bytes < kL2Bytes ? kL2 : packed ? kHbmPacked : kHbm));
    };
    DecodePlan one{0, 1}, more{0, 1};
    for (int shift = 1; shift <= kMaxClusterShift; ++shift) {
        const int heads_fit = active_clusters(shift) / c.Hkv;
        if (heads_fit >= 1) one.shift = shift;
        if (heads_fit >= (shift == 2 ? 2 : 5)) more = {shift, static_cast<int>(std::min<int64_t>(heads_fit, c.max_parts))};
    }
    return more.clusters > 1 && kMore + time(more) + kMargin < kOne + time(one) ? more : one;
}

int32_t launch_decode_as(const DecodeCall& c, const DecodePlan& p, MergeTodo& todo, cudaStream_t stream) {
    const int g = c.Hq / c.Hkv;
    DecodeArgs a{};
    a.Q = c.Q;
    a.K = c.K;
    a.V = c.V;
    a.Kgen = c.Kgen;
    a.Vgen = c.Vgen;
    a.Knew = c.Knew;
    a.Vnew = c.Vnew;
    a.ctx_len = static_cast<int>(c.ctx_len);
    a.gen_len = c.gen_len;
    a.gen_total = c.Kgen != nullptr ? c.gen_len + c.n : 0;
    a.Hq = c.Hq;
    a.Hkv = c.Hkv;
    while ((1 << a.g_shift) < g) ++a.g_shift;
    a.n_rows = c.n * g;
    a.cluster_shift = p.shift;
    a.clusters = p.clusters;
    a.scale_log2 = c.scale_log2;
    a.O = c.O;
    a.LSE = c.LSE;
    a.part_rows = static_cast<int64_t>(c.n) * c.Hq;
    if (p.clusters > 1) {
        a.part_O = static_cast<float*>(c.workspace);
        a.part_LSE = a.part_O + p.clusters * a.part_rows * c.d;
    }
    const DecodeKernel kernel = c.d == 128 ? (c.beside ? decode_kernel<128, true> : decode_kernel<128, false>)
                                           : (c.beside ? decode_kernel<64, true> : decode_kernel<64, false>);
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(static_cast<unsigned>(p.clusters << p.shift), static_cast<unsigned>(c.Hkv));
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = kSmemBytes;
    cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = 1u << p.shift;
    attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = p.shift > 0 ? 2 : 1;
    PULSAR_CUDA_OK(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes));
    if (p.shift > 3) PULSAR_CUDA_OK(cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
    PULSAR_CUDA_OK(cudaLaunchKernelEx(&cfg, kernel, a));
    count_launch();
    todo = {a.part_O, a.part_LSE, p.clusters > 1 ? p.clusters : 0};
    return PULSAR_OK;
}

}  // namespace

bool decode_takes(int32_t n, int32_t Hq, int32_t Hkv, int64_t ctx_len) {
    return static_cast<int64_t>(n) * (Hq / Hkv) <= kRows && ctx_len >= kLeastKeys;
}

int32_t launch_decode(const DecodeCall& c, MergeTodo& todo, cudaStream_t stream) {
    return launch_decode_as(c, plan_decode(c), todo, stream);
}

}  // namespace pulsar
