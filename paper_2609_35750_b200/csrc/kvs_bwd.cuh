// What the two main kernels of the backward share.
#pragma once

#include "kvs_common.cuh"

namespace kvs {

constexpr int BWD_THREADS = 512;

struct BwdParams {
    int batch, total_tokens, max_seqlen;   // what the caller says meta_buf was built for
    int Hq, Hkv;
    float scale, scale_log2;
    const float* lse;
    const float* dvec;
    void* dk;
    void* dv;
    long long dkv_ts;       // elements between consecutive tokens of dk and dv
    int grad_fp32;
    int32_t* status;
};

// head_dim 128 by CTA pairs (kvs_bwd_pair.cu).  k, v: tensor maps with 128-row boxes; q64, do64, dq64: with 64-row boxes
int launch_bwd_pair(const CUtensorMap& q64, const CUtensorMap& k, const CUtensorMap& v, const CUtensorMap& do64, const CUtensorMap& dq64,
                    const MetaView& mv, const BwdParams& p, int nb_cap, cudaStream_t st);

#ifdef __CUDACC__
// rows of zeros for a key block that no query sees (its gradients are zero)
template <int D>
__device__ __forceinline__ void bwd_zero_rows(const BwdParams& p, int tok, int rows, int g) {
    const int per_row = D * (p.grad_fp32 ? 4 : 2) / 16;          // 16-byte words of one (token, head) row
    for (int i = threadIdx.x; i < rows * per_row; i += BWD_THREADS) {
        const size_t off = (size_t)(tok + i / per_row) * (size_t)(p.dkv_ts / D) * per_row + (size_t)g * per_row + i % per_row;
        reinterpret_cast<uint4*>(p.dk)[off] = make_uint4(0, 0, 0, 0);
        reinterpret_cast<uint4*>(p.dv)[off] = make_uint4(0, 0, 0, 0);
    }
}

// 32 fp32 columns of a dK or dV row from registers to memory, as fp32 or bf16
__device__ __forceinline__ void bwd_store_cols(void* base, size_t elem, const uint32_t (&r)[32], int grad_fp32) {
    if (grad_fp32) {
        float4* dst = reinterpret_cast<float4*>(reinterpret_cast<float*>(base) + elem);
#pragma unroll
        for (int e = 0; e < 8; ++e)
            dst[e] = make_float4(__uint_as_float(r[e * 4]), __uint_as_float(r[e * 4 + 1]), __uint_as_float(r[e * 4 + 2]), __uint_as_float(r[e * 4 + 3]));
    } else {
        uint4* dst = reinterpret_cast<uint4*>(reinterpret_cast<__nv_bfloat16*>(base) + elem);
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            uint4 w;
            w.x = pack_bf16(__uint_as_float(r[e * 8 + 0]), __uint_as_float(r[e * 8 + 1]));
            w.y = pack_bf16(__uint_as_float(r[e * 8 + 2]), __uint_as_float(r[e * 8 + 3]));
            w.z = pack_bf16(__uint_as_float(r[e * 8 + 4]), __uint_as_float(r[e * 8 + 5]));
            w.w = pack_bf16(__uint_as_float(r[e * 8 + 6]), __uint_as_float(r[e * 8 + 7]));
            dst[e] = w;
        }
    }
}
#endif

}  // namespace kvs
