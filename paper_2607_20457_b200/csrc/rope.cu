// Position ids of the assembled Phase-1 inputs and the rotary embedding they feed (Appendix E).
//
//   assemble_positions_kernel  one CTA column per assembled input: the prefix entries keep their
//                              global positions (sparse) or everything is renumbered (contiguous)
//   rope_kernel                a thread owns one 16-byte vector position of one row, holds its eight
//                              (cos, sin) pairs in registers -- angle in float64, reduced to [-pi, pi],
//                              then sincosf, each formed once -- and walks the heads.  A pure stream
//                              over the rows: HBM-bound.
#include <cmath>

#include "common.cuh"

namespace pulsar {
namespace {

constexpr int kMaxHalf = 128;                       // d <= 256
struct RopeFreq {
    double inv_freq[kMaxHalf];                      // theta^(-2j/d), from the host's libm
};

__global__ void __launch_bounds__(256)
assemble_positions_kernel(const int32_t* __restrict__ prefix_idx, const int32_t* __restrict__ prefix_len,
                          int prefix_total, int n_blocks, int block_size, int mode, int32_t* __restrict__ pos_out,
                          int64_t capacity, int32_t* status) {
    const int i = blockIdx.y;
    __shared__ int64_t s_base;
    __shared__ int s_len;
    if (threadIdx.x == 0) {
        int64_t base = 0;
        bool bad = false;
        for (int b = 0; b <= i; ++b) {
            int pl = prefix_len[b];
            if (pl < 0 || pl > prefix_total) { bad = true; pl = max(0, min(pl, prefix_total)); }
            if (b < i) base += pl + block_size;
            else s_len = pl;
        }
        if (bad && blockIdx.x == 0) report(status, PULSAR_DEV_BAD_LENGTH);
        s_base = base;
    }
    __syncthreads();
    const int P = s_len, n = P + block_size;
    for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < n; j += gridDim.x * blockDim.x) {
        const int64_t at = s_base + j;
        if (at >= capacity) break;
        int v;
        if (mode == PULSAR_POS_CONTIGUOUS) v = j;
        else v = j < P ? prefix_idx[j] : i * block_size + (j - P);
        pos_out[at] = v;
    }
}

__device__ __forceinline__ float bf16_lo(uint32_t w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float bf16_hi(uint32_t w) { return __uint_as_float(w & 0xffff0000u); }

// Measured on B200 against a persistent kernel that took eight rows between two barriers and read the pairs from shared
// memory for every vector (us, Q + K heads x d): 80,320 rows of 32 + 8 x 128 260 -> 258; 37,003 of 16 + 4 x 64 46 -> 39;
// 50,000 of 4 + 1 x 32 16.9 -> 11.4; 65 of 32 + 8 x 128 8.7 -> 4.6.  Six heads in flight 1.5 %, four 2-4 % slower with 40
// heads; loads issued ahead of the barrier of the shared form 15-50 % slower.
constexpr int kRopeThreads = 128;
constexpr int kRopeUnroll = 8;                      // heads (2 x 16-byte loads each) in flight per thread
constexpr int kRopePairs = kRopeThreads * 8;        // a vector holds eight pairs' first or second halves

// X2/Y2/H2 describe an optional second tensor with the same rows and head size (K beside Q): it
// shares the rows' cosines and sines; H2 = 0 when there is none.  `groups` threads share a vector position of a row and
// take every groups-th head.
// kShared: the CTA's threads form the pairs together; one thread's eight in a row take 2 us, most of a small call.
template <bool kShared>
__global__ void __launch_bounds__(kRopeThreads)
rope_kernel(const uint4* __restrict__ X1, uint4* __restrict__ Y1, int H1, const uint4* __restrict__ X2,
            uint4* __restrict__ Y2, int H2, int64_t rows, int d, int groups, const int32_t* __restrict__ positions,
            const __grid_constant__ RopeFreq f, int32_t* status) {
    const int half = d >> 1;
    const int vec_half = half >> 3;                 // 16-byte vectors per half row of a head
    const int head_vecs = d >> 3;
    const int rows_cta = kRopeThreads / vec_half / groups;
    const int64_t row0 = static_cast<int64_t>(blockIdx.x) * rows_cta;
    const int nr = static_cast<int>(min(static_cast<int64_t>(rows_cta), rows - row0));
    const int slot = threadIdx.x / vec_half, v = threadIdx.x - slot * vec_half;
    const int r = slot / groups;
    const bool active = r < nr;
    const int heads = active ? H1 + H2 : 0;
    const int64_t at1 = (row0 + r) * H1 * head_vecs + v, at2 = (row0 + r) * H2 * head_vecs + v;

    uint4 a[kRopeUnroll], b[kRopeUnroll];
    auto load = [&](int h0) {
#pragma unroll
        for (int u = 0; u < kRopeUnroll; ++u) {
            const int h = h0 + u * groups;
            if (h < heads) {
                const uint4* src = h < H1 ? X1 + at1 + h * head_vecs : X2 + at2 + (h - H1) * head_vecs;
                a[u] = src[0];
                b[u] = src[vec_half];
            }
        }
    };
    int h0 = slot - r * groups;
    float cs[8], sn[8];
    auto pair = [&](int64_t row, int j, float* sine, float* cosine) {
        int p = positions[row];
        if (p < 0) {
            report(status, PULSAR_DEV_BAD_POSITION);
            p = 0;
        }
        // angle / 2pi in float64, reduced to [-1/2, 1/2] turns, then float32 sincos of at most pi
        const double turns = static_cast<double>(p) * f.inv_freq[j] * 0.15915494309189535;
        const double frac = turns - rint(turns);
        sincosf(static_cast<float>(frac * 6.283185307179586), sine, cosine);
    };
    if constexpr (kShared) {
        __shared__ __align__(16) float s_cos[kRopePairs], s_sin[kRopePairs];
        for (int e = threadIdx.x; e < nr * half; e += kRopeThreads) {
            const int er = e / half;
            pair(row0 + er, e - er * half, &s_sin[e], &s_cos[e]);
        }
        __syncthreads();
        if (!active) return;
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            cs[k] = s_cos[r * half + v * 8 + k];
            sn[k] = s_sin[r * half + v * 8 + k];
        }
    } else {
        if (!active) return;
#pragma unroll
        for (int k = 0; k < 8; ++k) pair(row0 + r, v * 8 + k, &sn[k], &cs[k]);
    }
    for (; h0 < heads; h0 += kRopeUnroll * groups) {
        load(h0);
#pragma unroll
        for (int u = 0; u < kRopeUnroll; ++u) {
            const int h = h0 + u * groups;
            if (h < heads) {
                uint4* dst = h < H1 ? Y1 + at1 + h * head_vecs : Y2 + at2 + (h - H1) * head_vecs;
                const uint32_t aw[4] = {a[u].x, a[u].y, a[u].z, a[u].w}, bw[4] = {b[u].x, b[u].y, b[u].z, b[u].w};
                uint32_t ya[4], yb[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const float c0 = cs[2 * k], s0 = sn[2 * k], c1 = cs[2 * k + 1], s1 = sn[2 * k + 1];
                    const float a0 = bf16_lo(aw[k]), a1 = bf16_hi(aw[k]), b0 = bf16_lo(bw[k]), b1 = bf16_hi(bw[k]);
                    ya[k] = pack_bf16x2(a0 * c0 - b0 * s0, a1 * c1 - b1 * s1);
                    yb[k] = pack_bf16x2(b0 * c0 + a0 * s0, b1 * c1 + a1 * s1);
                }
                dst[0] = make_uint4(ya[0], ya[1], ya[2], ya[3]);
                dst[vec_half] = make_uint4(yb[0], yb[1], yb[2], yb[3]);
            }
        }
    }
}

int32_t launch_rope(const uint16_t* X1, uint16_t* Y1, int32_t H1, const uint16_t* X2, uint16_t* Y2, int32_t H2,
                    int64_t rows, int32_t d, const int32_t* positions, double theta, int32_t* device_status,
                    void* stream) {
    if (rows < 0 || H1 <= 0 || H2 < 0 || d <= 0 || !(theta > 0.0)) return PULSAR_ERR_INVALID_ARG;
    if (d % 16 != 0 || d > 2 * kMaxHalf || H1 > 65535 || H2 > 65535) return PULSAR_ERR_SHAPE;
    if (rows == 0) return PULSAR_OK;
    if (!X1 || !Y1 || !positions || (H2 > 0 && (!X2 || !Y2))) return PULSAR_ERR_INVALID_ARG;
    if (!aligned(X1, 16) || !aligned(Y1, 16) || !aligned(X2, 16) || !aligned(Y2, 16) || !aligned(positions, 4))
        return PULSAR_ERR_ALIGNMENT;
    int32_t rc = check_device();
    if (rc != PULSAR_OK) return rc;
    RopeFreq f;
    for (int j = 0; j < d / 2; ++j) f.inv_freq[j] = std::pow(theta, -2.0 * static_cast<double>(j) / static_cast<double>(d));
    // Few rows: the threads of a CTA split the heads instead of taking more rows, as long as the chip then has no more than
    // the four CTAs per SM that fit (113 registers); a power of two leaves no slot idle.  32 + 8 heads x 128, us with a
    // target of one / two / four / eight CTAs per SM: 1500 rows 12.8 / 10.7 / 8.7 / 8.9, 4000 rows 16.9 / 16.9 / 14.8 / 16.8.
    const int slots = kRopeThreads / (d / 16);       // vector positions of whole rows per CTA, at least 8
    const int64_t want = static_cast<int64_t>(sm_count()) * 4 * slots / rows;
    int groups = 1;
    while (2 * groups <= std::min<int64_t>(want, std::min(slots, H1 + H2))) groups *= 2;
    // Many heads: a thread that walks all of them leaves a warp's rows a whole row apart, and the CTA's threads would come back
    // to a line long after its other half.  Four threads a row keep the lines together: 16 heads x 16 or 32 heads with
    // d < 64, and 32 heads of any size once the tensors no longer fit the L2, unless more than a tenth of the slots
    // would idle (d = 192).  us, 32 + 8 heads unless noted, one / four threads: d = 16, 100,000 rows 89 / 49 (the persistent kernel
    // 60), d = 32, 50,000 60 / 47 (53), d = 64, 20,000 47 / 41 (42), 64 + 8 x 64, 50,000 155 / 144 (148); below that size
    // one is better: d = 64, 6000 rows 12.4 / 14.3.
    const int heads = H1 + H2;
    const bool past_l2 = 4 * rows * heads * d > 128000000;
    if ((d == 16 && heads >= 16) || (heads >= 32 && (d < 64 || past_l2) && slots / 4 * 4 * 10 >= slots * 9))
        groups = std::max(groups, 4);
    const int64_t ctas = (rows + slots / groups - 1) / (slots / groups);
    if (ctas > INT32_MAX) return PULSAR_ERR_SHAPE;
    auto kernel = groups > 1 ? rope_kernel<true> : rope_kernel<false>;
    kernel<<<static_cast<unsigned>(ctas), kRopeThreads, 0, static_cast<cudaStream_t>(stream)>>>(
        reinterpret_cast<const uint4*>(X1), reinterpret_cast<uint4*>(Y1), H1, reinterpret_cast<const uint4*>(X2),
        reinterpret_cast<uint4*>(Y2), H2, rows, d, groups, positions, f, device_status);
    PULSAR_CUDA_OK(cudaGetLastError());
    count_launch();
    return PULSAR_OK;
}

}  // namespace
}  // namespace pulsar

using namespace pulsar;

extern "C" int32_t pulsar_assemble_positions(const int32_t* prefix_idx, const int32_t* prefix_len,
                                             int32_t prefix_total, int32_t n_blocks, int32_t block_size,
                                             int32_t mode, int32_t* pos_out, int64_t pos_capacity,
                                             int32_t* device_status, void* stream) {
    if (n_blocks <= 0 || block_size <= 0 || prefix_total < 0 || pos_capacity < 0) return PULSAR_ERR_INVALID_ARG;
    if (mode != PULSAR_POS_SPARSE && mode != PULSAR_POS_CONTIGUOUS) return PULSAR_ERR_INVALID_ARG;
    if (n_blocks > 65535) return PULSAR_ERR_SHAPE;
    if (!prefix_len || !pos_out || (prefix_total > 0 && !prefix_idx)) return PULSAR_ERR_INVALID_ARG;
    if (!aligned(prefix_len, 4) || !aligned(pos_out, 4) || !aligned(prefix_idx, 4)) return PULSAR_ERR_ALIGNMENT;
    int32_t rc = check_device();
    if (rc != PULSAR_OK) return rc;
    const int64_t longest = static_cast<int64_t>(prefix_total) + block_size;
    const unsigned gx = static_cast<unsigned>(std::min<int64_t>((longest + 255) / 256, 64));
    assemble_positions_kernel<<<dim3(gx, n_blocks), 256, 0, static_cast<cudaStream_t>(stream)>>>(
        prefix_idx, prefix_len, prefix_total, n_blocks, block_size, mode, pos_out, pos_capacity, device_status);
    PULSAR_CUDA_OK(cudaGetLastError());
    count_launch();
    return PULSAR_OK;
}

extern "C" int32_t pulsar_rope_apply(const uint16_t* X, uint16_t* Y, int64_t rows, int32_t H, int32_t d,
                                     const int32_t* positions, double theta, int32_t* device_status,
                                     void* stream) {
    return launch_rope(X, Y, H, nullptr, nullptr, 0, rows, d, positions, theta, device_status, stream);
}

extern "C" int32_t pulsar_rope_apply_qk(const uint16_t* Q, uint16_t* Q_out, int32_t Hq, const uint16_t* K,
                                        uint16_t* K_out, int32_t Hkv, int64_t rows, int32_t d,
                                        const int32_t* positions, double theta, int32_t* device_status,
                                        void* stream) {
    if (Hkv <= 0) return PULSAR_ERR_INVALID_ARG;
    return launch_rope(Q, Q_out, Hq, K, K_out, Hkv, rows, d, positions, theta, device_status, stream);
}
