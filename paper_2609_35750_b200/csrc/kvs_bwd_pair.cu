// Backward main kernel for head_dim 128 by CTA pairs: dQ, dK, dV with cta_group::2 MMAs.
//
// The single-CTA kernel (kvs_bwd.cu) is bound by shared memory: a 128x128x16 MMA with both operands there reads 8 KB in
// its 64 clocks, the whole bandwidth of an SM, and fills, dS and the dQ staging come on top (4216 bank cycles per tile
// against 2560 clocks of MMA work).  Here two CTAs of a cluster take two neighbouring key blocks 2p, 2p+1 of a trace and
// walk the same (head, query block) list.  An MMA spans both: each CTA supplies its own 128 key rows of A and HALF of B.
//   S^T, dP^T   A = own K, V [128 keys x d]          B = 64 of the 128 query rows of Q, dO       48 instead of 64 KB
//   dV, dK      A = P^T, dS^T in tensor memory        B = 64 of the 128 columns of dO, Q          16 instead of 32, 64 KB
//   dQ          M = 128 queries, K = 256 keys: each CTA has 64 query rows of dS against all 256 keys and 64 columns of K;
//               the half of its dS^T that belongs to the other CTA's queries is copied there (bulk copy, 16 KB)
// so a tile reads 192 KB of operands instead of 288, stages half a dQ tile instead of a whole one, and the global
// reduce-adds are halved (two key blocks are summed in the tensor core before they leave).
//
// Q and dO are needed in two cuts, 64 rows x d (B of S^T, dP^T) and 128 rows x 64 columns (B of dK, dV), in single buffers
// of 16 KB each: a buffer is refilled as soon as the one product that reads it is complete and is needed again a whole
// tile later.  Only the even CTA's warp 13 issues MMAs; whatever they wait for is signalled on the even CTA's barriers
// by both CTAs (TMA bytes and remote arrivals), and their completions are committed to the barriers of both.
// dS goes over by bulk copy and not by remote stores, and no arrival carries a cluster-scope release: 16-byte remote stores
// with a fence and a releasing arrival behind them took 2700 clocks of a tile.
//
// Warps (16, as in the single-CTA kernel): 0-7 compute, 8-11 drain dQ, 12 TMA producer, 13 MMA issuer (even CTA) or relay
// of the dS copies (odd CTA), 14 lse / D loader.
// Tensor memory:  [0,128)   S^T fp32, then P^T bf16 in [0,32) and [96,128) and the PREVIOUS tile's dQ fp32 in [32,96) (M = 128
//                           over two CTAs: lanes 0-63 hold columns 0-63 of the 64 query rows, lanes 64-127 columns 64-127)
//                 [128,256) dP^T fp32, then dS^T bf16 in [128,160) and [192,224)
//                 [256,384) dV     [384,512) dK
// Per tile j the tensor pipe runs  dK(j-1), dP^T(j), dQ(j-1), dV(j), S^T(j+1).  dQ runs one tile late, in columns that are free
// from the moment the compute warps have S^T(j) in registers: its wait for the other CTA's dS and its drain then lie beside
// P(j) and not in the chain dP -> dS -> dK -> dP (4630 -> 3900 clocks per tile).
#include "kvs_bwd.cuh"

namespace kvs {

namespace {

constexpr int D = 128;
constexpr int TB = TILE * D * 2;             // a 128 x 128 bf16 tile
constexpr int BOX = TILE * 128;              // 128 rows x 64 columns
constexpr int HBOX = BOX / 2;                // 64 rows x 64 columns

struct PairSmem {
    static constexpr int OFF_K = 0;                       // own key block, two 64-column boxes
    static constexpr int OFF_V = OFF_K + TB;
    static constexpr int OFF_KC = OFF_V + TB;             // 64 columns (this CTA's half) of both key blocks, [256 x 64]
    static constexpr int OFF_QR = OFF_KC + TB;            // 64 query rows (this CTA's half) x 128
    static constexpr int OFF_QC = OFF_QR + TB / 2;        // 128 query rows x 64 columns (this CTA's half)
    static constexpr int OFF_DOR = OFF_QC + TB / 2;
    static constexpr int OFF_DOC = OFF_DOR + TB / 2;
    static constexpr int OFF_DS = OFF_DOC + TB / 2;       // dS^T of both key blocks for this CTA's 64 queries, [256 keys x 64]
    static constexpr int OFF_OUT = OFF_DS + TB;           // dS^T of the own key block for the other CTA's queries, on its way there
    static constexpr int OFF_STG = OFF_OUT + TB / 2;      // dQ: two [64 queries x 32] fp32 boxes
    static constexpr int OFF_LSE = OFF_STG + TB / 2;      // 2 stages x 128 fp32: -lse * log2 e
    static constexpr int OFF_DVEC = OFF_LSE + 2 * TILE * 4;   // 2 stages x 128 fp32: -D * scale
    static constexpr int OFF_BAR = OFF_DVEC + 2 * TILE * 4;
    static constexpr int OFF_MISC = OFF_BAR + 20 * 8;     // tmem base, abort flag
    static constexpr int OFF_WORK = OFF_MISC + 16;
    static constexpr int TOTAL = OFF_WORK + (int)sizeof(BwdWork);
    static constexpr int MAX_DYN = 232448;                // 227 KB
    static constexpr int DYN_BYTES = (TOTAL + 1024 > MAX_DYN) ? MAX_DYN : TOTAL + 1024;
};

// ---- PTX wrappers: cluster, cta_group::2 -----------------------------------------------------------
__device__ __forceinline__ uint32_t cluster_rank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ uint32_t map_to(uint32_t addr, uint32_t rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}
__device__ __forceinline__ void arrive_cluster(uint32_t bar) {       // bar: a cluster address (map_to)
    asm volatile("mbarrier.arrive.shared::cluster.b64 _, [%0];" ::"r"(bar) : "memory");
}
// TMA load into this CTA's shared memory whose bytes are counted on a barrier of either CTA of the pair (no multicast)
__device__ __forceinline__ void tma_load_pair(uint32_t dst, const CUtensorMap* map, int c0, int c1, int c2, uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes.cta_group::2 [%0], [%1, {%2, %3, %4}], [%5];"
        ::"r"(dst), "l"(map), "r"(c0), "r"(c1), "r"(c2), "r"(bar)
        : "memory");
}
__device__ __forceinline__ void tmem_alloc_pair(uint32_t smem_result, uint32_t ncols) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_result), "r"(ncols) : "memory");
}
__device__ __forceinline__ void tmem_relinquish_pair() {
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc_pair(uint32_t taddr, uint32_t ncols) {
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
__device__ __forceinline__ void mma_ss_pair(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(d_tmem), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
}
__device__ __forceinline__ void mma_ts_pair(uint32_t d_tmem, uint32_t a_tmem, uint64_t bdesc, uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::2.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
        ::"r"(d_tmem), "r"(a_tmem), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
}
// the barrier at this offset of BOTH CTAs arrives once every MMA issued so far by this thread has completed
__device__ __forceinline__ void mma_commit_pair(uint32_t bar) {
    asm volatile(
        "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;"
        ::"r"(bar), "h"((unsigned short)3)
        : "memory");
}
// bytes from this CTA's shared memory to the other's, counted on a barrier there (dst, bar: cluster addresses)
__device__ __forceinline__ void bulk_to_peer(uint32_t dst, uint32_t src, uint32_t bytes, uint32_t bar) {
    asm volatile("cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(dst), "r"(src), "r"(bytes), "r"(bar)
                 : "memory");
}
// instruction descriptor: bf16 x bf16 -> fp32, M rows over both CTAs
__host__ __device__ constexpr uint32_t pair_idesc(int m, int n, int a_mn_major, int b_mn_major) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)a_mn_major << 15) | ((uint32_t)b_mn_major << 16) | ((uint32_t)(n >> 3) << 17) |
           ((uint32_t)(m >> 4) << 24);
}

__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(BWD_THREADS, 1)
bwd_pair_kernel(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_k,
                const __grid_constant__ CUtensorMap tm_v, const __grid_constant__ CUtensorMap tm_do,
                const __grid_constant__ CUtensorMap tm_dq, const __grid_constant__ MetaView mv,
                const __grid_constant__ BwdParams p) {
    using L = PairSmem;
    constexpr uint32_t TMEM_COLS = 512;
    constexpr uint32_t IDESC_ST = pair_idesc(256, 128, 0, 0);    // K-major x K-major, N = 128 queries
    constexpr uint32_t IDESC_KV = pair_idesc(256, D, 0, 1);      // A from tensor memory, B MN-major, N = d
    constexpr uint32_t IDESC_DQ = pair_idesc(128, D, 1, 1);      // A, B MN-major, 64 query rows per CTA, N = d

    extern __shared__ uint8_t smem_raw[];

    const int tid = threadIdx.x;
    const int warp = tid >> 5;
    const int lane = tid & 31;
    const uint32_t rank = cluster_rank();
    pdl_wait();
    // The returns below are taken by both CTAs of a pair alike.
    if (!meta_matches(mv.hdr, p.batch, p.total_tokens, p.max_seqlen)) {
        if (tid == 0 && blockIdx.x == 0) set_status(p.status, KVS_ERR_BAD_META);
        return;
    }
    BwdWork w;
    {
        BwdUnit unit;
        if (!bwd_unit_of(p, mv.pair_order, mv.hdr->npair_total, blockIdx.x >> 1, unit, w.g)) return;
        const int4 me = block_info(mv, unit.block);
        const int G = p.Hq / p.Hkv, n0 = me.z;
        w.n = n0 + (int)rank;                           // this CTA's key block; past the trace when its block count is odd
        w.tok0 = me.x;
        w.T = me.y;
        pair_range(mv.col_first, mv.col_last, unit.block, (n0 + 1) * TILE < w.T, w.m_first, w.m_last);
        w.general = mv.hdr->general != 0;
        const int nm = w.m_last - w.m_first + 1;        // query blocks m_first .. m_last can see one of the two key blocks
        if (nm <= 0) {
            if (w.n * TILE < w.T) bwd_zero_rows<D>(p, w.tok0 + w.n * TILE, min(TILE, w.T - w.n * TILE), w.g);
            return;
        }
        w.n_iter = (unit.tile1 < 0 ? G * nm : unit.tile1) - unit.tile0;     // of the G * nm (head, query block) tiles of the pair
        w.h_start = w.g * G + unit.tile0 / nm;
        w.m_start = w.m_first + unit.tile0 % nm;
        w.cut = unit.cut;
    }
    int32_t* status = p.status;

    const uint32_t sraw = smem_u32(smem_raw);
    const uint32_t sbase = (sraw + 1023u) & ~1023u;
    if ((sbase - sraw) + L::TOTAL > (uint32_t)L::DYN_BYTES) {      // shared window not aligned as expected (the same in both CTAs)
        if (tid == 0) set_status(status, KVS_ERR_CUDA);
        return;
    }
    uint8_t* sgen = smem_raw + (sbase - sraw);
    const uint32_t sK = sbase + L::OFF_K, sV = sbase + L::OFF_V, sKC = sbase + L::OFF_KC, sQR = sbase + L::OFF_QR, sQC = sbase + L::OFF_QC,
                   sDOR = sbase + L::OFF_DOR, sDOC = sbase + L::OFF_DOC, sDS = sbase + L::OFF_DS, sOUT = sbase + L::OFF_OUT,
                   sSTG = sbase + L::OFF_STG;
    uint32_t* s_tmem_base = reinterpret_cast<uint32_t*>(sgen + L::OFF_MISC);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(sgen + L::OFF_MISC + 4);
    const uint32_t bars = sbase + L::OFF_BAR;
    // Waited for by the issuer, in the even CTA: TMA bytes of both CTAs, arrivals of both CTAs' warps
    const uint32_t bar_kv = bars, bar_qr = bars + 8, bar_qc = bars + 16, bar_dor = bars + 24, bar_doc = bars + 32, bar_p = bars + 40,
                   bar_dst = bars + 48, bar_dss = bars + 56, bar_drained = bars + 64, bar_sl = bars + 152;
    // Committed by the issuer, in both CTAs: a product is complete (and the buffer that only it reads is free: S^T the Q
    // rows, dP^T the dO rows, dV the dO columns, dK the Q columns)
    const uint32_t bar_s = bars + 72, bar_dp = bars + 80, bar_dv = bars + 88, bar_dk = bars + 96, bar_dq = bars + 104, bar_done = bars + 112;
    // Within a CTA
    auto bar_ldfull = [&](int s) { return bars + 120 + 8 * s; };
    auto bar_ldfree = [&](int s) { return bars + 136 + 8 * s; };

    if (tid == 0) {
        *abort_flag = 0;
        mbar_init(bar_kv, 1);
        mbar_init(bar_qr, 1);
        mbar_init(bar_qc, 1);
        mbar_init(bar_dor, 1);
        mbar_init(bar_doc, 1);
        mbar_init(bar_sl, 16);
        mbar_init(bar_p, 16);
        mbar_init(bar_dst, 16);
        // even CTA: 4 + 4 warps that write their dS^T rows in place, the odd CTA's relay, and the bytes from the odd CTA;
        // odd CTA: the bytes from the even CTA
        mbar_init(bar_dss, rank == 0 ? 10 : 1);
        mbar_init(bar_drained, 8);
        mbar_init(bar_s, 1);
        mbar_init(bar_dp, 1);
        mbar_init(bar_dv, 1);
        mbar_init(bar_dk, 1);
        mbar_init(bar_dq, 1);
        mbar_init(bar_done, 1);
        for (int s = 0; s < 2; ++s) {
            mbar_init(bar_ldfull(s), 32);
            mbar_init(bar_ldfree(s), 8);
        }
        fence_mbar_init();
    }
    if (warp == 13) {
        tmem_alloc_pair(smem_u32(s_tmem_base), TMEM_COLS);
        tmem_relinquish_pair();
    }
    if (tid == 0) *reinterpret_cast<BwdWork*>(sgen + L::OFF_WORK) = w;
    tc_fence_before();
    __syncthreads();
    cluster_sync();                   // the other CTA's barriers and tensor memory are set up too
    tc_fence_after();
    const uint32_t tmem = *s_tmem_base;
    const volatile BwdWork* work = reinterpret_cast<const volatile BwdWork*>(sgen + L::OFF_WORK);
    const int n = work->n, tok0 = work->tok0, T = work->T, m_first = work->m_first, m_last = work->m_last;
    const int h_start = work->h_start, m_start = work->m_start, n_iter = work->n_iter, g = work->g;
    const uint32_t tmem_S = tmem;
    const uint32_t tmem_dQ = tmem + 32;
    const uint32_t tmem_P = tmem + 128;
    const uint32_t tmem_dV = tmem + 256;
    const uint32_t tmem_dK = tmem + 384;

    if (warp >= 12) {
        reg_dec<88>();
        if (warp == 12) {
            // ================= producer: this CTA's operands, counted on the even CTA's barriers =================
            const uint32_t l_kv = map_to(bar_kv, 0), l_qr = map_to(bar_qr, 0), l_qc = map_to(bar_qc, 0), l_dor = map_to(bar_dor, 0),
                           l_doc = map_to(bar_doc, 0);
            const bool expects = rank == 0 && lane == 0;
            const int row0 = (int)rank * 64;            // first of this CTA's query rows of a tile / columns of d
            auto rows_of = [&](uint32_t dst, const CUtensorMap* map, int h, int m, uint32_t full, uint32_t l_full) {
                if (expects) mbar_expect_tx(full, TB);
                if (lane == 0)
                    for (int c = 0; c < 2; ++c) tma_load_pair(dst + c * HBOX, map, c * 64, h, tok0 + m * TILE + row0, l_full);
            };
            auto cols_of = [&](uint32_t dst, const CUtensorMap* map, int h, int m, uint32_t full, uint32_t l_full) {
                if (expects) mbar_expect_tx(full, TB);
                if (lane == 0)
                    for (int c = 0; c < 2; ++c) tma_load_pair(dst + c * HBOX, map, row0, h, tok0 + m * TILE + c * 64, l_full);
            };
            int h = h_start, m = m_start;
            if (expects) mbar_expect_tx(bar_kv, 6 * TB);
            if (lane == 0) {
                // a key block past the end of the trace is read as zeros (a start past the last token is filled)
                const int tok_own = n * TILE < T ? tok0 + n * TILE : p.total_tokens;
                for (int c = 0; c < 2; ++c) tma_load_pair(sK + c * BOX, &tm_k, c * 64, g, tok_own, l_kv);
            }
            rows_of(sQR, &tm_q, h, m, bar_qr, l_qr);
            if (lane == 0) {
                const int tok_own = n * TILE < T ? tok0 + n * TILE : p.total_tokens;
                for (int c = 0; c < 2; ++c) tma_load_pair(sV + c * BOX, &tm_v, c * 64, g, tok_own, l_kv);
                const int n0 = n - (int)rank;
                for (int c = 0; c < 2; ++c)
                    tma_load_pair(sKC + c * BOX, &tm_k, row0, g, (n0 + c) * TILE < T ? tok0 + (n0 + c) * TILE : p.total_tokens, l_kv);
            }
            rows_of(sDOR, &tm_do, h, m, bar_dor, l_dor);
            cols_of(sDOC, &tm_do, h, m, bar_doc, l_doc);
            for (int j = 0; j < n_iter; ++j) {
                const uint32_t ph = j & 1;
                int h1 = h, m1 = m + 1;                   // tile j + 1
                if (m1 > m_last) {
                    m1 = m_first;
                    ++h1;
                }
                const bool more = j + 1 < n_iter;
                if (more) {
                    mbar_wait(bar_s, ph, abort_flag, status);
                    rows_of(sQR, &tm_q, h1, m1, bar_qr, l_qr);
                }
                if (j > 0) mbar_wait(bar_dk, ph ^ 1, abort_flag, status);
                cols_of(sQC, &tm_q, h, m, bar_qc, l_qc);
                if (more) {
                    mbar_wait(bar_dp, ph, abort_flag, status);
                    rows_of(sDOR, &tm_do, h1, m1, bar_dor, l_dor);
                    mbar_wait(bar_dv, ph, abort_flag, status);
                    cols_of(sDOC, &tm_do, h1, m1, bar_doc, l_doc);
                }
                h = h1;
                m = m1;
                if (*abort_flag) {                        // a wait gave up: let the copies in flight land, then leave
                    const long long t0 = clock64();
                    while (clock64() - t0 < 2000000) {}
                    break;
                }
            }
        } else if (warp == 13) {
            if (rank == 0) {
                // ================= MMA issuer (all lanes walk the loop, one elected lane issues) =================
                const bool leader = elect_one();
                const uint64_t dK_k = smem_desc(sK, 16, 1024), dV_k = smem_desc(sV, 16, 1024);
                const uint64_t dQR = smem_desc(sQR, 16, 1024), dDOR = smem_desc(sDOR, 16, 1024);
                const uint64_t dQC = smem_desc(sQC, BOX, 1024), dDOC = smem_desc(sDOC, BOX, 1024);
                const uint64_t dDS = smem_desc(sDS, BOX, 1024), dKC = smem_desc(sKC, BOX, 1024);
                auto issue_rows = [&](uint32_t d_tmem, uint64_t a, uint64_t bq) {       // S^T, dP^T: over d
#pragma unroll
                    for (int kk = 0; kk < D / 16; ++kk) {
                        const uint64_t offa = (uint64_t)(((kk >> 2) * BOX + (kk & 3) * 32) >> 4);
                        const uint64_t offb = (uint64_t)(((kk >> 2) * HBOX + (kk & 3) * 32) >> 4);
                        if (leader) mma_ss_pair(d_tmem, a + offa, bq + offb, IDESC_ST, kk > 0);
                    }
                };
                // dK(j) += dS^T Q, A from tensor memory
                auto issue_dk = [&](int j) {
                    const uint32_t ph = j & 1;
                    mbar_wait(bar_qc, ph, abort_flag, status);
                    mbar_wait(bar_dst, ph, abort_flag, status);
                    tc_fence_after();
#pragma unroll
                    for (int kk = 0; kk < TILE / 16; ++kk)
                        if (leader)
                            mma_ts_pair(tmem_dK, tmem_P + (kk >> 2) * 64 + (kk & 3) * 8, dQC + (uint64_t)(kk * 128), IDESC_KV, (j > 0) || (kk > 0));
                    if (leader) mma_commit_pair(bar_dk);
                };
                // dQ(j) = dS K over both key blocks
                auto issue_dq = [&](int j) {
                    mbar_wait(bar_dss, j & 1, abort_flag, status);
                    tc_fence_after();
#pragma unroll
                    for (int kk = 0; kk < 2 * TILE / 16; ++kk)
                        if (leader) mma_ss_pair(tmem_dQ, dDS + (uint64_t)(kk * 128), dKC + (uint64_t)(kk * 128), IDESC_DQ, kk > 0);
                    if (leader) mma_commit_pair(bar_dq);
                };
                mbar_wait(bar_kv, 0, abort_flag, status);
                mbar_wait(bar_qr, 0, abort_flag, status);
                tc_fence_after();
                issue_rows(tmem_S, dK_k, dQR);
                if (leader) mma_commit_pair(bar_s);
                for (int j = 0; j < n_iter; ++j) {
                    const uint32_t ph = j & 1;
                    if (j > 0) issue_dk(j - 1);
                    // dP^T(j) = V dO^T, over the columns of dS(j-1), which dK(j-1) has read
                    mbar_wait(bar_dor, ph, abort_flag, status);
                    tc_fence_after();
                    issue_rows(tmem_P, dV_k, dDOR);
                    if (leader) mma_commit_pair(bar_dp);
                    if (j > 0) {
                        mbar_wait(bar_sl, ph, abort_flag, status);         // S^T(j) has left the columns
                        issue_dq(j - 1);
                    }
                    // dV(j) += P^T dO
                    mbar_wait(bar_doc, ph, abort_flag, status);
                    mbar_wait(bar_p, ph, abort_flag, status);
                    tc_fence_after();
#pragma unroll
                    for (int kk = 0; kk < TILE / 16; ++kk)
                        if (leader)
                            mma_ts_pair(tmem_dV, tmem_S + (kk >> 2) * 96 + (kk & 3) * 8, dDOC + (uint64_t)(kk * 128), IDESC_KV, (j > 0) || (kk > 0));
                    if (leader) mma_commit_pair(bar_dv);
                    // S^T(j+1) = K Q^T, over P(j), which dV(j) has read, and dQ(j-1), once it is drained
                    if (j + 1 < n_iter) {
                        mbar_wait(bar_qr, ph ^ 1, abort_flag, status);
                        if (j > 0) mbar_wait(bar_drained, ph ^ 1, abort_flag, status);
                        tc_fence_after();
                        issue_rows(tmem_S, dK_k, dQR);
                        if (leader) mma_commit_pair(bar_s);
                    }
                }
                issue_dk(n_iter - 1);
                if (n_iter > 1) mbar_wait(bar_drained, n_iter & 1, abort_flag, status);
                issue_dq(n_iter - 1);
                if (leader) mma_commit_pair(bar_done);
            } else {
                // ================= odd CTA: dS^T from the even CTA has arrived -> the issuer =================
                const uint32_t l_dss = map_to(bar_dss, 0);
                for (int j = 0; j < n_iter; ++j) {
                    mbar_wait(bar_dss, j & 1, abort_flag, status);
                    if (lane == 0) arrive_cluster(l_dss);
                }
            }
        } else if (warp == 14) {
            // ================= lse and D of the tile's queries =================
            float* sLse = reinterpret_cast<float*>(sgen + L::OFF_LSE);
            float* sDv = reinterpret_cast<float*>(sgen + L::OFF_DVEC);
            int h = h_start, m = m_start;
            for (int j = 0; j < n_iter; ++j) {
                const int s = j & 1;
                const size_t rowbase = (size_t)h * p.total_tokens + tok0 + m * TILE;
                float l[4], dv[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int i = u * 32 + lane;
                    const bool qv = (m * TILE + i) < T;
                    // stored negated (they are subtracted with one fused multiply-add); -inf makes P vanish
                    // for the rows past the end of the trace
                    l[u] = qv ? p.lse[rowbase + i] * -1.4426950408889634f : -INFINITY;
                    dv[u] = qv ? p.dvec[rowbase + i] * -p.scale : 0.f;
                }
                if (j >= 2) mbar_wait(bar_ldfree(s), ((j >> 1) + 1) & 1, abort_flag, status);
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    sLse[s * TILE + u * 32 + lane] = l[u];
                    sDv[s * TILE + u * 32 + lane] = dv[u];
                }
                mbar_arrive(bar_ldfull(s));
                if (++m > m_last) {
                    m = m_first;
                    ++h;
                }
            }
        }
    } else if (warp >= 8) {
        // ================= drain warps: dQ(j), this CTA's 64 query rows =================
        reg_dec<104>();
        const int quad = warp & 3;
        const int row = (quad & 1) * 32 + lane;            // query row of this CTA's half
        const uint32_t lane_sel = (uint32_t)(quad * 32) << 16;
        const int chalf = quad >> 1;                       // columns 64 chalf .. + 63 of d
        uint8_t* stg_row = sgen + L::OFF_STG + chalf * (64 * 128) + row * 128;
        const uint32_t l_drained = map_to(bar_drained, 0);
        int h = h_start, m = m_start;
        for (int j = 0; j < n_iter; ++j) {
            mbar_wait(bar_dq, j & 1, abort_flag, status);
            tc_fence_after();
            uint32_t r0[32], r1[32];
            tmem_ld32(tmem_dQ + lane_sel, r0);
            tmem_ld32(tmem_dQ + lane_sel + 32, r1);
            tmem_wait_ld();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) arrive_cluster(l_drained);     // the columns may be overwritten from here on
            // 32 of each lane group's 64 columns at a time through the staging buffers
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                if (tid == 256) bulk_wait_read<0>();      // the reduces that last read the buffers have finished reading
                named_bar_sync(1, 128);
#pragma unroll
                for (int c = 0; c < 8; ++c) {
                    const uint32_t(&r)[32] = u == 0 ? r0 : r1;
                    *reinterpret_cast<uint4*>(stg_row + ((c ^ (row & 7)) << 4)) = make_uint4(r[c * 4], r[c * 4 + 1], r[c * 4 + 2], r[c * 4 + 3]);
                }
                fence_proxy_async();
                named_bar_sync(1, 128);
                // 64 rows that all lie past the end of the trace are zero and may lie past the tensor: nothing to add
                if (tid == 256 && m * TILE + (int)rank * 64 < T) {
#pragma unroll
                    for (int c = 0; c < 2; ++c)
                        tma_reduce_add_3d(&tm_dq, c * 64 + u * 32, h, tok0 + m * TILE + (int)rank * 64, sSTG + c * (64 * 128));
                    bulk_commit();
                }
            }
            if (++m > m_last) {
                m = m_first;
                ++h;
            }
        }
        if (tid == 256) bulk_wait<0>();
    } else {
        // ================= compute warps: one key row per thread, 64 of the tile's 128 queries =================
        reg_inc<160>();
        const int quad = warp & 3;
        const int half = warp >> 2;
        const int row = quad * 32 + lane;                  // TMEM lane: key row of S^T, dP^T
        const uint32_t lane_sel = (uint32_t)(quad * 32) << 16;
        const int col0 = half * 64;                        // this thread's 64 query columns
        const int kj = n * TILE + row;
        // queries [my_first, my_end) of the trace see this key; nobody sees a slot past the trace
        const int my_end = (kj < T) ? min(mv.evict[tok0 + kj], T) : 0;
        const int my_first = (work->general && kj < T) ? mv.kfirst[tok0 + kj] : kj;
        const float* sLse = reinterpret_cast<const float*>(sgen + L::OFF_LSE);
        const float* sDv = reinterpret_cast<const float*>(sgen + L::OFF_DVEC);
        // dS^T of this key for queries col0 .. col0+63, a 128-byte row: in place, or on its way to the CTA that owns these queries
        const bool local = half == (int)rank;
        uint8_t* sDS_row = sgen + (local ? L::OFF_DS + (int)rank * BOX : L::OFF_OUT) + row * 128;
        const uint32_t peer = map_to(sbase, rank ^ 1), even = map_to(sbase, 0);      // the other's, the issuer's shared memory
        const uint32_t peer_ds = peer + L::OFF_DS + rank * BOX + quad * 4096, peer_dss = peer + (bar_dss - sbase);
        const uint32_t l_sl = even + (bar_sl - sbase), l_p = even + (bar_p - sbase), l_dst = even + (bar_dst - sbase),
                       l_dss = even + (bar_dss - sbase);
        float pv[64];
        int m = m_start;                                   // query block of the tile of the next phase_p

        auto phase_p = [&](int j) {        // P^T(j) = exp2(S^T * c - lse), masked
            const int s = j & 1;
            const int lo = my_first - (m * TILE + col0), hi = my_end - (m * TILE + col0);     // columns [lo, hi) see the key
            m = (m == m_last) ? m_first : m + 1;
            mbar_wait(bar_ldfull(s), (j >> 1) & 1, abort_flag, status);
            mbar_wait(bar_s, j & 1, abort_flag, status);
            tc_fence_after();
            const float4* l4 = reinterpret_cast<const float4*>(sLse + s * TILE + col0);
            uint32_t r0[32], r1[32];
            tmem_ld32(tmem_S + lane_sel + col0, r0);
            tmem_ld32(tmem_S + lane_sel + col0 + 32, r1);
            tmem_wait_ld();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) arrive_cluster(l_sl);
            const float2 c2 = make_float2(p.scale_log2, p.scale_log2);
#pragma unroll
            for (int e4 = 0; e4 < 16; ++e4) {          // packed fp32x2 multiply-adds, then one ex2 per element
                const float4 l = l4[e4];
                const uint32_t* r = (e4 < 8) ? &r0[e4 * 4] : &r1[(e4 - 8) * 4];
                const float2 x01 = __ffma2_rn(make_float2(__uint_as_float(r[0]), __uint_as_float(r[1])), c2, make_float2(l.x, l.y));
                const float2 x23 = __ffma2_rn(make_float2(__uint_as_float(r[2]), __uint_as_float(r[3])), c2, make_float2(l.z, l.w));
                pv[e4 * 4 + 0] = fast_exp2(x01.x);
                pv[e4 * 4 + 1] = fast_exp2(x01.y);
                pv[e4 * 4 + 2] = fast_exp2(x23.x);
                pv[e4 * 4 + 3] = fast_exp2(x23.y);
            }
            // Only the warps that hold a hidden pair pay for the mask, whatever the class of the tile (a loop of at most one
            // pass: as an if, its 64 selects are predicated and issued for every tile)
            const int masked = __any_sync(0xffffffffu, lo > 0 || hi < 64) ? 1 : 0;
#pragma unroll 1
            for (int pass = 0; pass < masked; ++pass) {
                const uint32_t seen0 = bit_range(lo, hi), seen1 = bit_range(lo - 32, hi - 32);
#pragma unroll
                for (int e = 0; e < 64; ++e) pv[e] = ((e < 32 ? seen0 : seen1) >> (e & 31) & 1u) ? pv[e] : 0.f;
            }
            uint32_t pk[32];
#pragma unroll
            for (int e = 0; e < 32; ++e) pk[e] = pack_bf16(pv[2 * e], pv[2 * e + 1]);
            tmem_st32(tmem_S + lane_sel + half * 96, pk);  // 64 queries -> 32 packed columns, clear of dQ(j-1)
            tmem_wait_st();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) arrive_cluster(l_p);
        };

        auto phase_ds = [&](int j) {       // dS^T(j) = P^T (scale dP^T - scale D)
            const int s = j & 1;
            mbar_wait(bar_dp, j & 1, abort_flag, status);
            tc_fence_after();
            const float4* d4 = reinterpret_cast<const float4*>(sDv + s * TILE + col0);
            uint32_t r0[32], r1[32];
            tmem_ld32(tmem_P + lane_sel + col0, r0);
            tmem_ld32(tmem_P + lane_sel + col0 + 32, r1);
            tmem_wait_ld();
            uint32_t dk_[32];
            const float2 sc2 = make_float2(p.scale, p.scale);
#pragma unroll
            for (int e4 = 0; e4 < 16; ++e4) {          // dS = P * (scale dP - scale D), two elements per instruction
                const float4 dd = d4[e4];
                const uint32_t* r = (e4 < 8) ? &r0[e4 * 4] : &r1[(e4 - 8) * 4];
                const float2 t01 = __ffma2_rn(make_float2(__uint_as_float(r[0]), __uint_as_float(r[1])), sc2, make_float2(dd.x, dd.y));
                const float2 t23 = __ffma2_rn(make_float2(__uint_as_float(r[2]), __uint_as_float(r[3])), sc2, make_float2(dd.z, dd.w));
                const float2 d01 = __fmul2_rn(make_float2(pv[e4 * 4 + 0], pv[e4 * 4 + 1]), t01);
                const float2 d23 = __fmul2_rn(make_float2(pv[e4 * 4 + 2], pv[e4 * 4 + 3]), t23);
                dk_[e4 * 2 + 0] = pack_bf16(d01.x, d01.y);
                dk_[e4 * 2 + 1] = pack_bf16(d23.x, d23.y);
            }
            auto to_tmem = [&] {
                // dS^T for dK: columns of this half's own dP^T (its first 32)
                tmem_st32(tmem_P + lane_sel + col0, dk_);
                tmem_wait_st();
                tc_fence_before();                   // also orders this thread's reads of dP^T before the products that overwrite it
                __syncwarp();
                if (lane == 0) {
                    arrive_cluster(l_dst);
                    mbar_arrive(bar_ldfree(s));
                }
            };
            auto to_smem = [&] {
                // dS^T for dQ: MN-major rows of 64 queries, 128-byte swizzle (16-byte chunk c sits at c ^ (row % 8)), once the
                // previous tile's dQ has read both buffers (or their copy)
                if (j > 0) mbar_wait(bar_dq, (j - 1) & 1, abort_flag, status);
#pragma unroll
                for (int c = 0; c < 8; ++c)
                    *reinterpret_cast<uint4*>(sDS_row + ((c ^ (row & 7)) << 4)) =
                        make_uint4(dk_[c * 4], dk_[c * 4 + 1], dk_[c * 4 + 2], dk_[c * 4 + 3]);
                fence_proxy_async();                 // visible to the tensor core's reads and to the copy
                __syncwarp();
            };
            if (local) {
                to_tmem();
                to_smem();
                if (lane == 0) arrive_cluster(l_dss);
            } else {                                 // what has the longer way first
                to_smem();
                if (lane == 0) bulk_to_peer(peer_ds, sOUT + quad * 4096, 4096, peer_dss);
                if (tid == ((int)rank ^ 1) * 128) mbar_expect_tx(bar_dss, TB / 2);       // what this CTA receives for the tile
                to_tmem();
            }
        };

        phase_p(0);
        for (int j = 0; j < n_iter; ++j) {
            phase_ds(j);
            if (j + 1 < n_iter) phase_p(j + 1);
        }

        // ---- epilogue: dK, dV of this key block, once every MMA has completed ----
        mbar_wait(bar_done, 0, abort_flag, status);
        tc_fence_after();
        // through the memory of K and V, which nothing reads any more
        bwd_epilogue<D>(p, work->cut, g, 2, (int)rank, tmem_dK + lane_sel + half * 64, tmem_dV + lane_sel + half * 64, row, half,
                        tok0 + n * TILE + quad * 32, T - n * TILE - quad * 32, sgen + L::OFF_K + warp * 4096,
                        reinterpret_cast<volatile int*>(sgen + L::OFF_MISC + 8), [] { named_bar_sync(2, 256); });
    }
    tc_fence_before();
    __syncthreads();
    cluster_sync();                   // neither CTA leaves while the other's copies, arrivals or MMAs may still reach it
    if (warp == 13) {
        __syncwarp();
        tmem_dealloc_pair(tmem, TMEM_COLS);
    }
}

}  // namespace

int launch_bwd_pair(const CUtensorMap& q64, const CUtensorMap& k, const CUtensorMap& v, const CUtensorMap& do64, const CUtensorMap& dq64,
                    const MetaView& mv, const BwdParams& p, unsigned units, cudaStream_t st) {
    if (cudaFuncSetAttribute(bwd_pair_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, PairSmem::DYN_BYTES) != cudaSuccess)
        return cuda_refused();
    return launch_after(bwd_pair_kernel, 2 * units, BWD_THREADS, PairSmem::DYN_BYTES, st, q64, k, v, do64, dq64, mv, p);
}

}  // namespace kvs
