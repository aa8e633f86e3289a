// What the two main kernels of the backward share.
#pragma once

#include "kvs_common.cuh"

namespace kvs {

constexpr int BWD_THREADS = 512;

// The work of the main kernel, per KV head: units of consecutive tiles of one item (a key block, or a pair of them).  An item
// is cut into several units where whole items would leave SMs idle (the prompt of a long trace is seen by every query of it,
// by all heads of the group: on one rollout of 32768 tokens with G = 7 its key blocks take 1792 tiles each, more than an
// SM's share of the whole work).  The units of an item write their dK and dV to slots of the workspace, and the last of
// them to finish adds the slots up in their order, so the sums do not depend on which it was.
struct BwdUnit {
    int32_t block;          // (first) key block of the item
    int32_t tile0, tile1;   // tiles [tile0, tile1) of its (head of the group, query block) list
    int32_t cut;            // 0: the whole item; else first slot << 18 | index of the unit << 9 | units of the item
};
// What the roles of a CTA need of its unit.  They read it from shared memory once they have parted: kept in registers from
// before, it was spilled around their loops.
struct BwdWork {
    int n, tok0, T;                 // key block, first token and length of its trace
    int m_first, m_last;            // query blocks of the item's list
    int h_start, m_start, n_iter;   // first (head, query block) tile of the unit, number of tiles
    int g, cut, general, pad;
};
struct BwdPlan {
    int32_t n_units;
    int32_t slots;          // slots used per KV head
    // Which unit a CTA takes: the first n_heavy units of ALL heads start first; then, of the next n_apart, one head's, the next
    // head's, ...; then what is left, again of all heads together.
    int32_t n_heavy, n_apart;
};
constexpr int BWD_MAX_CUT = 511;          // units of an item, and the unit's index, are 9 bits each

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
    const BwdPlan* plan;    // nullptr: whole items in the metadata's order
    const BwdUnit* units;
    int32_t* arrived;       // [Hkv][slots][2] units of an item that have written their slot (entry of the item's first slot)
    float4* part;           // [Hkv][slots] of 2 x rows of the item x D / 4
};

// head_dim 128 by CTA pairs (kvs_bwd_pair.cu).  k, v: tensor maps with 128-row boxes; q64, do64, dq64: with 64-row boxes
int launch_bwd_pair(const CUtensorMap& q64, const CUtensorMap& k, const CUtensorMap& v, const CUtensorMap& do64, const CUtensorMap& dq64,
                    const MetaView& mv, const BwdParams& p, unsigned units, cudaStream_t st);

// The batch a backward over a part of it is planned for (the chunks of the host path cut their items as one call over the
// whole batch does, so that both give the same sums), and the room for its plan and slots, which chunks that follow one
// another on a stream share.
struct BwdWhole {
    const void* meta_buf;
    int batch, total_tokens, max_seqlen, Hkv;
    void* cut_buf;
    bool cut_less;          // which of the two sizes of bwd_cut_bytes it has
};
int bwd_of_chunk(const BwdWhole& whole, const void* dout, const void* q, const void* k, const void* v, const void* out, const float* lse,
                 const void* meta_buf, int batch, int total_tokens, int max_seqlen, int Hq, int Hkv, int head_dim, float softmax_scale,
                 int grad_dtype, void* dq, void* dk, void* dv, void* workspace, size_t workspace_bytes, kvs_stream_t stream);
// workspace bytes of a backward: what it needs without cutting items (status, row sums, fp32 dQ accumulator), and the rest (`less`:
// with the fewer slots of longer units)
size_t bwd_base_bytes(int total_tokens, int Hq, int head_dim, int grad_dtype);
size_t bwd_cut_bytes(int total_tokens, int Hq, int head_dim, bool less);

#ifdef __CUDACC__
// The unit and KV head of CTA (or pair) x of a one-dimensional grid; false: there is none.  The CTAs without work come last.
// A whole item has tile1 = -1: all of its list.
__device__ __forceinline__ bool bwd_unit_of(const BwdParams& p, const int32_t* order, int n_items, int x, BwdUnit& unit, int& g) {
    const int n = p.plan ? p.plan->n_units : n_items, heavy = p.plan ? p.plan->n_heavy : 0, apart = p.plan ? p.plan->n_apart : n;
    if (x >= n * p.Hkv) return false;
    int u;
    if (x < heavy * p.Hkv || x >= (heavy + apart) * p.Hkv) {
        u = x / p.Hkv;
        g = x % p.Hkv;
    } else {
        x -= heavy * p.Hkv;
        u = heavy + x % apart;
        g = x / apart;
    }
    unit = p.plan ? p.units[u] : BwdUnit{order[u], 0, -1, 0};
    return true;
}

__device__ __forceinline__ bool bwd_has_unit(const BwdParams& p, int n_items, int x) { return x < (p.plan ? p.plan->n_units : n_items) * p.Hkv; }

// bits [lo, hi) of a 32-bit word (either end may lie outside it)
__device__ __forceinline__ uint32_t bit_range(int lo, int hi) {
    const int l = min(max(lo, 0), 32), h = min(max(hi, 0), 32);
    return (h >= 32 ? 0xffffffffu : (1u << h) - 1u) & (l >= 32 ? 0u : ~((1u << l) - 1u));
}

// rows of zeros for a key block that no query sees (its gradients are zero)
template <int D>
__device__ __forceinline__ void bwd_zero_rows(const BwdParams& p, int tok, int rows, int g, int threads = BWD_THREADS) {
    const int per_row = D * (p.grad_fp32 ? 4 : 2) / 16;          // 16-byte words of one (token, head) row
    for (int i = threadIdx.x; i < rows * per_row; i += threads) {
        const size_t off = (size_t)(tok + i / per_row) * (size_t)(p.dkv_ts / D) * per_row + (size_t)g * per_row + i % per_row;
        reinterpret_cast<uint4*>(p.dk)[off] = make_uint4(0, 0, 0, 0);
        reinterpret_cast<uint4*>(p.dv)[off] = make_uint4(0, 0, 0, 0);
    }
}

// Epilogue of the 256 compute threads: thread (row, half) has the columns [half * D/2, +D/2) of its row of dK and dV in
// tensor memory.  A whole item goes straight to memory (`tok`: first token of this warp's 32 rows, `rows`: how many of them the
// trace has; `stage`: 4 KB of shared memory of this warp's own).  A unit of a cut item writes them to its slot; the item's last unit
// adds the slots up in order.  `ctas`: CTAs per item, `cta`: this one's index; `meet`: a barrier of the 256 threads.
template <int D, typename Meet>
__device__ __forceinline__ void bwd_epilogue(const BwdParams& p, int cut, int g, int ctas, int cta, uint32_t tmem_dk, uint32_t tmem_dv, int row,
                                             int half, int tok, int rows, uint8_t* stage, volatile int* s_last, Meet meet) {
    constexpr int CH = D / 64;              // 32-column pieces per thread and tensor
    const int lane = threadIdx.x & 31;
    const size_t elem = (size_t)tok * (size_t)p.dkv_ts + (size_t)g * D + half * (D / 2);
    // piece i (32 columns) of this thread's row of dK, then dV: fp32 leaves piece by piece, bf16 with the whole half row
    auto put = [&](int i, const uint32_t (&r)[32]) {
        void* base = i < CH ? p.dk : p.dv;
        if (p.grad_fp32) {
            RowStage<32>::put_f32(stage, lane, r);
            RowStage<32>::template flush<4>(stage, lane, reinterpret_cast<char*>(base) + (elem + (i % CH) * 32) * 4, (size_t)p.dkv_ts, rows);
        } else {
            RowStage<D / 2>::put_bf16(stage, lane, i % CH, r);
            if (i % CH == CH - 1)
                RowStage<D / 2>::template flush<2>(stage, lane, reinterpret_cast<char*>(base) + elem * 2, (size_t)p.dkv_ts, rows);
        }
    };
    if (cut == 0) {
#pragma unroll
        for (int i = 0; i < 2 * CH; ++i) {
            uint32_t r[32];
            tmem_ld32((i < CH ? tmem_dk : tmem_dv) + (i % CH) * 32, r);
            tmem_wait_ld();
            put(i, r);
        }
        return;
    }
    const int first = cut >> 18, index = (cut >> 9) & BWD_MAX_CUT, count = cut & BWD_MAX_CUT;
    constexpr size_t SLOT = 2 * TILE * D / 4;               // float4s of one CTA's slot: [piece][half][8][128 rows]
    const size_t slot0 = (size_t)g * p.plan->slots + first;
    float4* base = p.part + (slot0 * ctas + cta) * SLOT + (size_t)half * 8 * TILE + row;
    {
        float4* dst = base + (size_t)index * ctas * SLOT;
#pragma unroll
        for (int i = 0; i < 2 * CH; ++i) {
            uint32_t r[32];
            tmem_ld32((i < CH ? tmem_dk : tmem_dv) + (i % CH) * 32, r);
            tmem_wait_ld();
#pragma unroll
            for (int e = 0; e < 8; ++e)
                dst[(size_t)(i * 16 + e) * TILE] = make_float4(__uint_as_float(r[e * 4]), __uint_as_float(r[e * 4 + 1]), __uint_as_float(r[e * 4 + 2]),
                                                               __uint_as_float(r[e * 4 + 3]));
        }
    }
    __threadfence();
    meet();
    if (threadIdx.x == 0) *s_last = atomicAdd(&p.arrived[slot0 * 2 + cta], 1) == count - 1;
    meet();
    if (!*s_last) return;
    __threadfence();
#pragma unroll
    for (int i = 0; i < 2 * CH; ++i) {
        float4 a[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) a[e] = __ldcg(base + (size_t)(i * 16 + e) * TILE);
        for (int c = 1; c < count; ++c) {
            const float4* src = base + (size_t)c * ctas * SLOT;
            float4 b[8];
#pragma unroll
            for (int e = 0; e < 8; ++e) b[e] = __ldcg(src + (size_t)(i * 16 + e) * TILE);
#pragma unroll
            for (int e = 0; e < 8; ++e) a[e] = make_float4(a[e].x + b[e].x, a[e].y + b[e].y, a[e].z + b[e].z, a[e].w + b[e].w);
        }
        uint32_t r[32];
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            r[e * 4] = __float_as_uint(a[e].x);
            r[e * 4 + 1] = __float_as_uint(a[e].y);
            r[e * 4 + 2] = __float_as_uint(a[e].z);
            r[e * 4 + 3] = __float_as_uint(a[e].w);
        }
        put(i, r);
    }
}

#endif

}  // namespace kvs
