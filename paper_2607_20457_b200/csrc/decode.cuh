// Attention of few query rows against a long context: what the Phase-2 entry points hand to decode.cu.
#pragma once

#include "common.cuh"

namespace pulsar {

struct DecodeCall {
    const uint16_t* Q;                           // [n, Hq, d]
    int32_t n, Hq, Hkv, d;
    const uint16_t *K, *V;                       // context [ctx_len, Hkv, d]
    int64_t ctx_len;
    uint16_t *Kgen, *Vgen;                       // generation shard, or null
    const uint16_t *Knew, *Vnew;                 // the new tokens' KV, appended at row gen_len
    int32_t gen_len;
    float scale_log2;
    uint16_t* O;
    float* LSE;
    void* workspace;                             // for partials; max_parts of them fit (0: none)
    int64_t max_parts;
    bool beside;                                 // see launch_lse_merge
};

// What is left of a Phase-2 call when its attention has been launched: the merge of n_parts partials (0: nothing).
struct MergeTodo {
    const float *part_O, *part_LSE;
    int32_t n_parts;
};

// Whether the call is one of few rows and many keys (d and Hq / Hkv have been checked by the caller).
bool decode_takes(int32_t n, int32_t Hq, int32_t Hkv, int64_t ctx_len);
int32_t launch_decode(const DecodeCall& call, MergeTodo& todo, cudaStream_t stream);

}  // namespace pulsar
