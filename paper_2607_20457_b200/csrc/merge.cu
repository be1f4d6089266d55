// Online-softmax merge of attention partials (Appendix H, Eq. 12-13) in closed form:
//   l = m + ln sum_j exp(l_j - m),  O = sum_j exp(l_j - l) A_j,  m = max_j l_j.
// For the head sizes of the attention kernels and few rows a warp owns an output row and its parts are spread over
// the warps of a CTA; otherwise one thread takes four consecutive output elements (merge_warps).
#include "common.cuh"

namespace pulsar {

// stride_O / stride_L: floats between consecutive parts of part_O / part_LSE.  kF32: the merged
// output stays float32 (a partial for a later merge) instead of being rounded to bf16.
template <bool kF32>
__global__ void __launch_bounds__(256)
lse_merge_kernel(const float* __restrict__ part_O, const float* __restrict__ part_LSE, int n_parts,
                 int64_t stride_O, int64_t stride_L, int64_t rows, int d, void* __restrict__ O_,
                 float* __restrict__ LSE) {
    grid_dependency_wait();        // launched beside the attention kernel that writes the partials: wait for it
    grid_launch_dependents();
    const int vec_per_row = d >> 2;
    const int64_t idx = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
    if (idx >= rows * vec_per_row) return;
    const int64_t row = idx / vec_per_row;
    const int v = static_cast<int>(idx - row * vec_per_row);

    // The loads of a group of parts are independent: issue them together (a decode-shaped merge is
    // a few CTAs whose run time is a chain of load latencies).
    float m = -INFINITY;
#pragma unroll 8
    for (int j = 0; j < n_parts; ++j) m = fmaxf(m, part_LSE[static_cast<size_t>(j) * stride_L + row]);

    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    float denom = 0.f;
    if (m > -INFINITY) {
#pragma unroll 8
        for (int j = 0; j < n_parts; ++j) {
            const float w = __expf(part_LSE[static_cast<size_t>(j) * stride_L + row] - m);
            const float4 o = *reinterpret_cast<const float4*>(part_O + static_cast<size_t>(j) * stride_O + row * d + v * 4);
            denom += w;
            acc.x += w * o.x; acc.y += w * o.y; acc.z += w * o.z; acc.w += w * o.w;
        }
        const float inv = 1.f / denom;
        acc.x *= inv; acc.y *= inv; acc.z *= inv; acc.w *= inv;
    }
    if (kF32) {
        *reinterpret_cast<float4*>(static_cast<float*>(O_) + row * d + v * 4) = acc;
    } else {
        uint2 packed;
        packed.x = pack_bf16x2(acc.x, acc.y);
        packed.y = pack_bf16x2(acc.z, acc.w);
        *reinterpret_cast<uint2*>(static_cast<uint16_t*>(O_) + row * d + v * 4) = packed;
    }
    if (LSE != nullptr && v == 0) LSE[row] = (m > -INFINITY) ? m + logf(denom) : -INFINITY;
}

// The same merge for rows of 32 * kVec floats (d = 64, 128): a warp loads a part's row as one contiguous run,
// kWarps warps share a row, warp w taking parts w, w + kWarps, ...  The merge after an attention launch is latency-bound
// -- a few hundred rows, tens of parts, everything in L2 -- so each warp issues the loads of eight parts (the l_j and
// the row pieces, which do not depend on them) before it uses any, and there are enough warps per row that one or
// two such rounds cover all parts.  The order of the sums is fixed, so the result is reproducible.
// Measured tail from the end of the attention launch to the end of the merge: 384 rows of 19 parts
// 8.5 us with one thread per four outputs, 3.4 us with this form.
// kBeside: see launch_lse_merge (an instance of its own: the test alone cost 0.2 us of a 20 us query).
template <bool kF32, int kVec, int kWarps, int kRows, bool kBeside>
__global__ void __launch_bounds__(32 * kWarps * kRows)
lse_merge_rows_kernel(const float* __restrict__ part_O, const float* __restrict__ part_LSE, int n_parts,
                      int64_t stride_O, int64_t stride_L, int64_t rows, void* __restrict__ O_,
                      float* __restrict__ LSE) {
    static_assert(kRows == 1 || kWarps == 1, "a CTA has one row, or one warp per row");
    if (!kBeside) grid_dependency_wait();        // launched beside the attention kernel that writes the partials: wait for it
    grid_launch_dependents();
    constexpr int kD = 32 * kVec, kInFlight = 8;
    // Beside another launch the partials are read from L2, where the launch that wrote them has left them: no wait stands
    // between an SM's L1, which may hold the last call's, and these loads.
    const auto load = [](const auto* p) { return kBeside ? __ldcg(p) : *p; };
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t row = static_cast<int64_t>(blockIdx.x) * kRows + (kWarps == 1 ? warp : 0);
    if (row >= rows) return;                                     // kRows > 1 only: no barrier follows
    const float* src = part_O + row * kD + lane * kVec;

    float m = -INFINITY, denom = 0.f, acc[kVec];
#pragma unroll
    for (int k = 0; k < kVec; ++k) acc[k] = 0.f;
    for (int j0 = kWarps == 1 ? 0 : warp; j0 < n_parts; j0 += kWarps * kInFlight) {
        float l[kInFlight], o[kInFlight][kVec];
#pragma unroll
        for (int i = 0; i < kInFlight; ++i) {
            const int j = j0 + i * kWarps;
            l[i] = -INFINITY;
            if (j < n_parts) {
                l[i] = load(part_LSE + static_cast<size_t>(j) * stride_L + row);
                const float* p = src + static_cast<size_t>(j) * stride_O;
                if (kVec == 4) {
                    const float4 v = load(reinterpret_cast<const float4*>(p));
                    o[i][0] = v.x; o[i][1] = v.y; o[i][kVec - 2] = v.z; o[i][kVec - 1] = v.w;
                } else {
                    const float2 v = load(reinterpret_cast<const float2*>(p));
                    o[i][0] = v.x; o[i][1] = v.y;
                }
            } else {
#pragma unroll
                for (int k = 0; k < kVec; ++k) o[i][k] = 0.f;
            }
        }
        float m_new = m;
#pragma unroll
        for (int i = 0; i < kInFlight; ++i) m_new = fmaxf(m_new, l[i]);
        if (m_new > -INFINITY) {
            const float keep = (m == -INFINITY) ? 0.f : __expf(m - m_new);
            denom *= keep;
#pragma unroll
            for (int k = 0; k < kVec; ++k) acc[k] *= keep;
#pragma unroll
            for (int i = 0; i < kInFlight; ++i) {
                const float w = (l[i] == -INFINITY) ? 0.f : __expf(l[i] - m_new);
                denom += w;
#pragma unroll
                for (int k = 0; k < kVec; ++k) acc[k] += w * o[i][k];
            }
            m = m_new;
        } else {
            // Parts without keys weigh nothing, but an undefined row in one stays undefined in the result.  (A branch of its
            // own: the step at 2500 tokens takes 10.6 us with the sums above formed in any case, 9.9 like this.)
#pragma unroll
            for (int i = 0; i < kInFlight; ++i) {
                denom += 0.f * (l[i] == -INFINITY ? 0.f : l[i]);
#pragma unroll
                for (int k = 0; k < kVec; ++k) acc[k] += 0.f * o[i][k];
            }
        }
    }
    if (kWarps > 1) {
        __shared__ float s_m[kWarps], s_denom[kWarps], s_acc[kWarps][kD];
        if (lane == 0) {
            s_m[warp] = m;
            s_denom[warp] = denom;
        }
#pragma unroll
        for (int k = 0; k < kVec; ++k) s_acc[warp][k * 32 + lane] = acc[k];
        __syncthreads();
        if (warp != 0) return;
#pragma unroll
        for (int w = 0; w < kWarps; ++w) m = fmaxf(m, s_m[w]);
        denom = 0.f;
#pragma unroll
        for (int k = 0; k < kVec; ++k) acc[k] = 0.f;
        if (m > -INFINITY) {
#pragma unroll
            for (int w = 0; w < kWarps; ++w) {
                const float f = (s_m[w] == -INFINITY) ? 0.f : __expf(s_m[w] - m);
                denom += f * s_denom[w];
#pragma unroll
                for (int k = 0; k < kVec; ++k) acc[k] += f * s_acc[w][k * 32 + lane];
            }
        }
    }
    if (m > -INFINITY) {
        const float inv = 1.f / denom;
#pragma unroll
        for (int k = 0; k < kVec; ++k) acc[k] *= inv;
    } else {
#pragma unroll
        for (int k = 0; k < kVec; ++k) acc[k] = 0.f;
    }
    const int64_t at = row * kD + lane * kVec;
    if (kF32) {
        float* dst = static_cast<float*>(O_) + at;
        if (kVec == 4) *reinterpret_cast<float4*>(dst) = make_float4(acc[0], acc[1], acc[kVec - 2], acc[kVec - 1]);
        else *reinterpret_cast<float2*>(dst) = make_float2(acc[0], acc[1]);
    } else {
        uint16_t* dst = static_cast<uint16_t*>(O_) + at;
        if (kVec == 4)
            *reinterpret_cast<uint2*>(dst) = make_uint2(pack_bf16x2(acc[0], acc[1]), pack_bf16x2(acc[kVec - 2], acc[kVec - 1]));
        else *reinterpret_cast<uint32_t*>(dst) = pack_bf16x2(acc[0], acc[1]);
    }
    if (LSE != nullptr && lane == 0) LSE[row] = (m > -INFINITY) ? m + logf(denom) : -INFINITY;
    if (kBeside) grid_dependency_wait();
}

// The merge with every part at its own address: part j is the buffer parts[j], laid out
// [rows_total * d outputs | rows_total LSE] like the Phase-2 exchange buffer of a GPU, and only rows
// [row0, row0 + rows) are merged.  The addresses may be peer-mapped memory of other GPUs: the kernel
// then pulls its slice of every GPU's partial over NVLink with plain loads while it merges (no copy
// engine, no TMA) -- the all-gather and the merge in one pass, each GPU reducing 1/H of
// the rows.
constexpr int kMaxMergePeers = 64;
struct PartTable {
    const float* base[kMaxMergePeers];
};

template <bool kF32>
__global__ void __launch_bounds__(256)
lse_merge_table_kernel(const __grid_constant__ PartTable parts, int n_parts, int64_t rows_total, int64_t row0,
                       int64_t rows, int d, void* __restrict__ O_, float* __restrict__ LSE) {
    const int vec_per_row = d >> 2;
    const int64_t idx = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
    if (idx >= rows * vec_per_row) return;
    const int64_t r = idx / vec_per_row;
    const int v = static_cast<int>(idx - r * vec_per_row);
    const int64_t row = row0 + r;
    const int64_t lse_at = rows_total * d + row;

    float m = -INFINITY;
#pragma unroll 8
    for (int j = 0; j < n_parts; ++j) m = fmaxf(m, parts.base[j][lse_at]);
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    float denom = 0.f;
    if (m > -INFINITY) {
#pragma unroll 8
        for (int j = 0; j < n_parts; ++j) {
            const float w = __expf(parts.base[j][lse_at] - m);
            const float4 o = *reinterpret_cast<const float4*>(parts.base[j] + row * d + v * 4);
            denom += w;
            acc.x += w * o.x; acc.y += w * o.y; acc.z += w * o.z; acc.w += w * o.w;
        }
        const float inv = 1.f / denom;
        acc.x *= inv; acc.y *= inv; acc.z *= inv; acc.w *= inv;
    }
    if (kF32) {
        *reinterpret_cast<float4*>(static_cast<float*>(O_) + r * d + v * 4) = acc;
    } else {
        uint2 packed;
        packed.x = pack_bf16x2(acc.x, acc.y);
        packed.y = pack_bf16x2(acc.z, acc.w);
        *reinterpret_cast<uint2*>(static_cast<uint16_t*>(O_) + r * d + v * 4) = packed;
    }
    if (LSE != nullptr && v == 0) LSE[r] = (m > -INFINITY) ? m + logf(denom) : -INFINITY;
}

namespace {
template <bool kF32, int kVec, bool kBeside>
auto merge_rows_kernel(int warps) {
    return warps == 16  ? lse_merge_rows_kernel<kF32, kVec, 16, 1, kBeside>
           : warps == 8 ? lse_merge_rows_kernel<kF32, kVec, 8, 1, kBeside>
           : warps == 4 ? lse_merge_rows_kernel<kF32, kVec, 4, 1, kBeside>
           : warps == 2 ? lse_merge_rows_kernel<kF32, kVec, 2, 1, kBeside>
                        : lse_merge_rows_kernel<kF32, kVec, 1, 8, kBeside>;
}

// Warps that share an output row; 0: one thread per four outputs (lse_merge_kernel).  That form reads the l_j before
// it can use an output row, and eight parts at a time: 6 us of latency for 18 parts fresh from another kernel, 10 for 48 (a
// remainder of the eights part by part).  Rows over warps take a third of that, but every row costs its warps: with several
// a row up to 3200 warps in all, with one up to 3200 rows; from 48 parts on one warp a row is the better form for any
// number of rows (more than two if there are more than 64 parts and few rows).  Measured behind a kernel that writes the parts, us, rows
// form / thread form, d = 128: 18 parts of 512 rows 3.1 / 5.7, of 1600 4.8 / 6.0, of 2048 6.0 / 6.1, of 4096 8.0 / 7.1;
// 33 of 512 4.0 / 8.4, of 4096 14.7 / 15.9; 4 of 1024 2.9 / 3.6, of 8192 5.5 / 6.2; d = 64: 9 of 4096 4.5 / 3.8, of 16384
// 13.4 / 8.4; 96 of 4096 19 / 40; alone and in cache the thread form gains earlier (9 of 4096 4.3 / 3.2).
int merge_warps(int32_t n_parts, int64_t rows, int32_t d) {
    constexpr int64_t kMost = 3200;
    if (n_parts > 4 && n_parts < 8 && (d == 128 || rows <= 8192)) return 1;     // the thread form's eights are all remainder
    if (n_parts == 1 || (n_parts < 48 && rows > kMost)) return 0;
    if (rows > kMost) return 1;
    int warps = n_parts > 64 ? 16 : n_parts > 32 ? 8 : n_parts > 16 ? 4 : n_parts > 8 ? 2 : 1;
    while (warps > (n_parts > 64 ? 2 : 1) && rows * warps > kMost) warps /= 2;
    return warps;
}

int32_t launch_merge(const float* part_O, const float* part_LSE, int32_t n_parts, int64_t stride_O, int64_t stride_L,
                     int64_t rows, int32_t d, void* O, bool f32, float* LSE, cudaStream_t stream, bool beside = false) {
    // (beside is honoured where f32 is not asked for; the thread form always waits at its start, which is right as well)
    if (rows == 0) return PULSAR_OK;
    const int warps = (d == 64 || d == 128) ? merge_warps(n_parts, rows, d) : 0;
    if (warps > 0) {
        const int64_t blocks = warps == 1 ? (rows + 7) / 8 : rows;
        if (blocks > 0x7fffffffll) return PULSAR_ERR_SHAPE;
        auto kernel = d == 128 ? (f32      ? merge_rows_kernel<true, 4, false>(warps)
                                  : beside ? merge_rows_kernel<false, 4, true>(warps)
                                           : merge_rows_kernel<false, 4, false>(warps))
                               : (f32      ? merge_rows_kernel<true, 2, false>(warps)
                                  : beside ? merge_rows_kernel<false, 2, true>(warps)
                                           : merge_rows_kernel<false, 2, false>(warps));
        PULSAR_CUDA_OK(launch_kernel(kernel, dim3(static_cast<unsigned>(blocks)), dim3(warps == 1 ? 256 : 32 * warps), 0, stream,
                                     true, part_O, part_LSE, n_parts, stride_O, stride_L, rows, O, LSE));
        count_launch();
        return PULSAR_OK;
    }
    const int64_t threads = rows * (d >> 2);
    const int64_t blocks = (threads + 255) / 256;
    if (blocks > 0x7fffffffll) return PULSAR_ERR_SHAPE;
    auto kernel = f32 ? lse_merge_kernel<true> : lse_merge_kernel<false>;
    PULSAR_CUDA_OK(launch_kernel(kernel, dim3(static_cast<unsigned>(blocks)), dim3(256), 0, stream, true, part_O, part_LSE,
                                 n_parts, stride_O, stride_L, rows, d, O, LSE));
    count_launch();
    return PULSAR_OK;
}
}  // namespace

// Placed as the CTAs of the launch before it leave (programmatic stream serialization), waits until that has finished
// (grid_dependency_wait): no launch gap separates the merge from the attention launch that writes the partials.
// beside: see common.cuh.
int32_t launch_lse_merge(const float* part_O, const float* part_LSE, int32_t n_parts, int64_t rows, int32_t d,
                         uint16_t* O, float* LSE, cudaStream_t stream, bool beside) {
    return launch_merge(part_O, part_LSE, n_parts, rows * d, rows, rows, d, O, false, LSE, stream, beside);
}

}  // namespace pulsar

using namespace pulsar;

extern "C" int32_t pulsar_lse_merge(const float* part_O, const float* part_LSE, int32_t n_parts, int64_t rows,
                                    int32_t d, uint16_t* O, float* LSE, void* stream) {
    if (n_parts < 1 || rows < 0 || d <= 0) return PULSAR_ERR_INVALID_ARG;
    if (d % 4 != 0 || d > 1024) return PULSAR_ERR_SHAPE;
    if (rows > 0 && (!part_O || !part_LSE || !O)) return PULSAR_ERR_INVALID_ARG;
    if (!aligned(part_O, 16) || !aligned(part_LSE, 4) || !aligned(O, 8)) return PULSAR_ERR_ALIGNMENT;
    int32_t rc = check_device();
    if (rc != PULSAR_OK) return rc;
    return launch_lse_merge(part_O, part_LSE, n_parts, rows, d, O, LSE, static_cast<cudaStream_t>(stream));
}

extern "C" int32_t pulsar_lse_merge_strided(const float* part_O, const float* part_LSE, int32_t n_parts,
                                            int64_t part_stride_O, int64_t part_stride_LSE, int64_t rows, int32_t d,
                                            void* O, int32_t out_is_f32, float* LSE, void* stream) {
    if (n_parts < 1 || rows < 0 || d <= 0) return PULSAR_ERR_INVALID_ARG;
    if (d % 4 != 0 || d > 1024) return PULSAR_ERR_SHAPE;
    if (part_stride_O < rows * d || part_stride_LSE < rows || part_stride_O % 4 != 0) return PULSAR_ERR_SHAPE;
    if (rows > 0 && (!part_O || !part_LSE || !O)) return PULSAR_ERR_INVALID_ARG;
    if (!aligned(part_O, 16) || !aligned(part_LSE, 4) || !aligned(O, out_is_f32 ? 16 : 8)) return PULSAR_ERR_ALIGNMENT;
    int32_t rc = check_device();
    if (rc != PULSAR_OK) return rc;
    return launch_merge(part_O, part_LSE, n_parts, part_stride_O, part_stride_LSE, rows, d, O, out_is_f32 != 0, LSE,
                        static_cast<cudaStream_t>(stream));
}

extern "C" int32_t pulsar_lse_merge_peers(const float* const* part_bases_host, int32_t n_parts, int64_t rows_total,
                                          int64_t row_begin, int64_t rows, int32_t d, void* O, int32_t out_is_f32,
                                          float* LSE, void* stream) {
    if (n_parts < 1 || n_parts > kMaxMergePeers || rows_total < 0 || row_begin < 0 || rows < 0 || d <= 0 ||
        !part_bases_host)
        return PULSAR_ERR_INVALID_ARG;
    if (d % 4 != 0 || d > 1024 || row_begin + rows > rows_total) return PULSAR_ERR_SHAPE;
    if (rows == 0) return PULSAR_OK;
    if (!O) return PULSAR_ERR_INVALID_ARG;
    PartTable t{};
    for (int j = 0; j < n_parts; ++j) {
        if (!part_bases_host[j]) return PULSAR_ERR_INVALID_ARG;
        if (!aligned(part_bases_host[j], 16)) return PULSAR_ERR_ALIGNMENT;
        t.base[j] = part_bases_host[j];
    }
    if (!aligned(O, out_is_f32 ? 16 : 8) || !aligned(LSE, 4)) return PULSAR_ERR_ALIGNMENT;
    int32_t rc = check_device();
    if (rc != PULSAR_OK) return rc;
    const int64_t blocks = (rows * (d >> 2) + 255) / 256;
    if (blocks > 0x7fffffffll) return PULSAR_ERR_SHAPE;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (out_is_f32)
        lse_merge_table_kernel<true><<<static_cast<unsigned>(blocks), 256, 0, st>>>(t, n_parts, rows_total, row_begin, rows,
                                                                                   d, O, LSE);
    else
        lse_merge_table_kernel<false><<<static_cast<unsigned>(blocks), 256, 0, st>>>(t, n_parts, rows_total, row_begin,
                                                                                    rows, d, O, LSE);
    PULSAR_CUDA_OK(cudaGetLastError());
    count_launch();
    return PULSAR_OK;
}
