// Forward: eviction-masked causal attention.
//
// One item per (query block, pair of query heads of one GQA group), and a CTA per item or a chain of
// items.  The two heads share every K/V tile (identical key-block list and element mask), so each tile
// is fetched once for two 128-row query tiles.  The last head of an odd group (and every head when there is no grouping) gets an item
// of its own, in which the two softmax groups take alternate key blocks of that one head as two
// independent streams, merged at the end.  384 threads in three warp groups:
//   warps 0-3   softmax of tile 0 (one query row per thread)        } registers re-balanced with
//   warps 4-7   softmax of tile 1                                    } setmaxnreg (208 / 208 / 88)
//   warp 8      producer: TMA for Q0, Q1 and the K and V rings (2 stages each; K runs one key
//               block ahead of V, its slot being released a whole iteration earlier); plain loads
//               for evict_at
//   warp 9      MMA issuer: all 32 lanes walk the loop and one elected lane issues, so descriptor
//               arithmetic stays in uniform registers and an MMA costs a few issue slots even while
//               the softmax warps of the same scheduler are busy
//   warp 10     the list of items, where they are chained;  warp 11 idle
// Tensor memory: S0 [0,128)  S1 [128,256)  O0 [256,256+D)  O1 [384,384+D); P (bf16) overwrites S.
// Per key block i the tensor pipe runs  O0 += P0 V, S0(i+1) = Q0 K^T, O1 += P1 V, S1(i+1) = Q1 K^T
// while the two softmax groups alternate, so the exponentials of one tile overlap the MMAs of the
// other.  A row's probabilities are handed over in two parts (the first P_SPLIT keys, then the
// rest), so most of P V overlaps the last exponentials of the row.  EMPTY tiles are never visited (the
// CTA walks the row's non-empty list); the element mask is evaluated on PARTIAL or ragged tiles only,
// and there only by the warps and for the 32 keys that need it.  O is rescaled lazily: a row keeps its reference
// maximum until the running maximum exceeds it by more than 8 (base-2), so exp2 arguments stay
// below 2^8 and the rescale of O in tensor memory is rare.
#include "kvs_common.cuh"
#include <type_traits>

namespace kvs {

constexpr int FWD_THREADS = 384;
constexpr float RESCALE_THRESHOLD = 8.0f;
// Chained: key blocks left of an item when the CTA asks for the next one.  Forward, us, with 1, 2, 4: 131 traces of 500 tokens, 32 heads
// on 8, 524.5, 524.5, 530; 96 of 480, 16 on 2, 204.1, 204.5, 206.4; 32 of 2000 708, 709, 702.
constexpr int FWD_LATE = 2;
constexpr int P_SPLIT = 96;     // keys of a tile whose probabilities are handed to the MMA warp early

// an item of work: a query block of a pair of heads (or of a single one)
struct FwdItem {
    int nlist;          // key blocks to walk; -1: no more items
    int m, T, tok0;     // query block, length and first token of its trace
    int g, h0, ntile;   // KV head, first query head, number of query heads
    int pad;
    long long at;       // the row's entries in row_list and tile_class
};

template <int D>
struct FwdSmem {
    static constexpr int TB = TILE * D * 2;
    static constexpr int OFF_Q = 0;                      // 2 query tiles
    static constexpr int OFF_KV = 2 * TB;                // 2 stages x (K, V)
    static constexpr int OFF_STG = OFF_KV + 4 * TB;      // chained: 32 rows x 32 columns of out per softmax warp
    static constexpr int OFF_EV = OFF_STG + 8 * 2048;    // 2 stages x 128 int32: eviction step of the stage's key slots
    static constexpr int OFF_KF = OFF_EV + 2 * TILE * 4; // 2 stages x 128 int32: first query that may see the slot
    static constexpr int OFF_FLAG = OFF_KF + 2 * TILE * 4;   // 2 stages x (compare, hidden)
    static constexpr int OFF_BAR = OFF_FLAG + 16;
    static constexpr int OFF_ITEM = OFF_BAR + 32 * 8;    // 2 slots x FwdItem
    static constexpr int OFF_ASK = OFF_ITEM + 2 * 48;    // the answer of the launch control
    static constexpr int OFF_MISC = OFF_ASK + 16;
    static constexpr int TOTAL = OFF_MISC + 16;
    static constexpr int DYN_BYTES = TOTAL + 1024;          // slack for the 1024-byte alignment
};

struct FwdParams {
    int batch, total_tokens, max_seqlen;   // what the caller says meta_buf was built for
    int Hq, Hkv;
    int heads;          // pairs of heads, and single ones: Hkv * ceil(G / 2)
    float scale_log2;   // softmax_scale * log2(e)
    __nv_bfloat16* out;
    float* lse;
    const __nv_bfloat16* first_out;     // MERGE: the result over the other keys of the same queries, in the layout of out and lse
    const float* first_lse;
};


// CHAIN: a CTA takes over items of CTAs of the grid that have not started (cluster launch control) and starts an item's
// loads and products while the softmax groups still write out the one before.  With a CTA per item the launch, the chain of
// metadata loads, the set-up, the first loads and the write-out stand beside the tiles of the row, which counts where rows are
// short; the loop over items costs registers that the long rows' tiles are faster with (see launch_fwd for the line).
// MERGE: out and lse are those of attention over these keys and the ones that first_out and first_lse stand for (the teacher's of
// self-distillation): the rows meet here, in fp32 and on their way out.  As a pass of its own the merge was bound by memory and
// rounded this part to bf16 first: 3 traces of 9000 to 17000 tokens, 32 heads on 8, both forwards 4282 -> 4125 us.
// The parameters are passed by value and not read in place (__grid_constant__): that costs the tile loop registers, 1 to 5 % of long
// rows (24576 tokens of token-level eviction 5085 -> 5330 us).
template <int D, bool CHAIN, bool MERGE>
__global__ void __launch_bounds__(FWD_THREADS, 1)
fwd_kernel(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_k,
           const __grid_constant__ CUtensorMap tm_v, MetaView mv, FwdParams p) {
    using L = FwdSmem<D>;
    constexpr int NBOX = D / 64;             // 64-column TMA boxes per tile row
    constexpr int BOX_BYTES = TILE * 128;    // 128 rows x 128 bytes
    constexpr uint32_t TMEM_COLS = 512;
    constexpr uint32_t IDESC_S = make_idesc(TILE, 0, 0);
    constexpr uint32_t IDESC_O = make_idesc(D, 0, 1);

    extern __shared__ uint8_t smem_raw[];

    const int tid = threadIdx.x;
    const int warp = tid >> 5;
    const int lane = tid & 31;
    pdl_wait();
    // meta_buf must be the one kvs_mask_meta wrote for these sizes: every index below comes out of it
    if (!meta_matches(mv.hdr, p.batch, p.total_tokens, p.max_seqlen)) {
        if (tid == 0 && blockIdx.x == 0 && blockIdx.y == 0) set_status(&mv.hdr->status, KVS_ERR_BAD_META);
        return;
    }
    const int nblk = mv.hdr->nblk_total;
    if (!CHAIN && (int)blockIdx.x >= nblk) return;
    const int G = p.Hq / p.Hkv;
    const int pairs_per_group = (G + 1) >> 1;
    auto item_of = [&](int x, int y) {
        FwdItem it;
        const int gb = mv.fwd_order[x];
        const int4 me = block_info(mv, gb);
        it.nlist = mv.row_cnt[gb];
        it.tok0 = me.x;
        it.T = me.y;
        it.m = me.z;
        it.at = (long long)(uint32_t)me.w;
        it.g = y / pairs_per_group;
        it.h0 = it.g * G + 2 * (y % pairs_per_group);
        // An odd group ends with a single head.  Its item still runs both softmax groups: they take alternate key blocks of
        // that head as two independent streams (own S, O, running maximum and sum), merged at the end like the splits of a
        // split-KV decode.
        it.ntile = (it.h0 + 1 < (it.g + 1) * G) ? 2 : 1;
        return it;
    };
    int32_t* status = &mv.hdr->status;

    const uint32_t sraw = smem_u32(smem_raw);
    const uint32_t sbase = (sraw + 1023u) & ~1023u;
    uint8_t* sgen = smem_raw + (sbase - sraw);
    const uint32_t sQ = sbase + L::OFF_Q, sKV = sbase + L::OFF_KV;
    int32_t* sEv = reinterpret_cast<int32_t*>(sgen + L::OFF_EV);
    int32_t* sKf = reinterpret_cast<int32_t*>(sgen + L::OFF_KF);
    const bool general = mv.hdr->general != 0;       // key slots carry their own first visible query (re-ordered keys)
    volatile int32_t* sFlag = reinterpret_cast<volatile int32_t*>(sgen + L::OFF_FLAG);
    volatile FwdItem* s_item = reinterpret_cast<volatile FwdItem*>(sgen + L::OFF_ITEM);
    uint32_t* s_tmem_base = reinterpret_cast<uint32_t*>(sgen + L::OFF_MISC);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(sgen + L::OFF_MISC + 4);
    const uint32_t bars = sbase + L::OFF_BAR;
    const uint32_t bar_q = bars;
    auto bar_vfull = [&](int s) { return bars + 8 * (1 + s); };     // TMA bytes of V
    auto bar_kfull = [&](int s) { return bars + 8 * (16 + s); };    // TMA bytes of K
    auto bar_evfull = [&](int s) { return bars + 8 * (3 + s); };    // evict_at tile + need_mask flag (32 arrivals)
    auto bar_vfree = [&](int s) { return bars + 8 * (5 + s); };     // every P V product reading the stage's V has completed
    auto bar_kfree = [&](int s) { return bars + 8 * (18 + s); };    // every Q K^T product reading the stage's K has completed
    auto bar_s = [&](int t) { return bars + 8 * (7 + t); };         // S_t ready
    auto bar_p = [&](int t) { return bars + 8 * (9 + t); };         // all of P_t written (4 arrivals)
    auto bar_p0 = [&](int t) { return bars + 8 * (14 + t); };       // first P_SPLIT keys of P_t written (4 arrivals)
    auto bar_evfree = [&](int s) { return bars + 8 * (11 + s); };   // softmax groups done with the evict_at tile
    const uint32_t bar_done = bars + 8 * 13;                         // every MMA of the item complete
    const uint32_t bar_qfree = bars + 8 * 20;                        // every Q K^T product of the item complete
    const uint32_t bar_ofree = bars + 8 * 21;                        // O read out by both softmax groups (8 arrivals)
    const uint32_t bar_xfree = bars + 8 * 22;                        // a single head's streams are merged: the K/V ring is free again (4)
    const uint32_t bar_x = bars + 8 * 27;                            // stream 1 of a single head is in the exchange buffer (4)
    // CHAIN
    auto bar_item = [&](int s) { return bars + 8 * (23 + s); };      // item written
    auto bar_itemfree = [&](int s) { return bars + 8 * (25 + s); };  // item read by the producer, MMA and 8 softmax warps
    const uint32_t bar_ask = bars + 8 * 28;                          // the launch control has answered
    const uint32_t bar_late = bars + 8 * 29;                      // the MMA warp is near the end of an item
    auto put = [&](int slot, const FwdItem& it) {
        volatile FwdItem* dst = s_item + slot;
        dst->nlist = it.nlist;
        dst->m = it.m;
        dst->T = it.T;
        dst->tok0 = it.tok0;
        dst->g = it.g;
        dst->h0 = it.h0;
        dst->ntile = it.ntile;
        dst->at = it.at;
    };
    // the r-th item of the CTA
    auto take = [&](int r, int& nlist, int& m, int& T, int& tok0, int& h0, int& ntile) {
        if (CHAIN) mbar_wait(bar_item(r & 1), (r >> 1) & 1, abort_flag, status);
        volatile FwdItem* it = s_item + (r & 1);
        nlist = it->nlist;
        m = it->m;
        T = it->T;
        tok0 = it->tok0;
        h0 = it->h0;
        ntile = it->ntile;
    };
    auto taken = [&](int r) {
        if (CHAIN) {
            __syncwarp();
            if (lane == 0) mbar_arrive(bar_itemfree(r & 1));
        }
    };

    if (tid == 0) {
        *abort_flag = 0;
        mbar_init(bar_q, 1);
        for (int s = 0; s < 2; ++s) {
            mbar_init(bar_vfull(s), 1);
            mbar_init(bar_kfull(s), 1);
            mbar_init(bar_evfull(s), 32);
            mbar_init(bar_vfree(s), 1);
            mbar_init(bar_kfree(s), 1);
            mbar_init(bar_evfree(s), 8);
            mbar_init(bar_item(s), 1);
            mbar_init(bar_itemfree(s), 10);
            mbar_init(bar_s(s), 1);
            mbar_init(bar_p(s), 4);
            mbar_init(bar_p0(s), 4);
        }
        mbar_init(bar_done, 1);
        mbar_init(bar_qfree, 1);
        mbar_init(bar_ofree, 8);
        mbar_init(bar_xfree, 4);
        mbar_init(bar_x, 4);
        mbar_init(bar_ask, 1);
        mbar_init(bar_late, 1);
        fence_mbar_init();
    }
    if (!CHAIN && tid == 256) put(0, item_of(blockIdx.x, blockIdx.y));
    if (warp == 9) {
        tmem_alloc(smem_u32(s_tmem_base), TMEM_COLS);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *s_tmem_base;

    if (warp >= 8) {
        reg_dec<88>();
        if (warp == 8) {
            // ================= producer =================
            uint32_t ring = 0, q_items = 0, singles = 0;       // key blocks, items with a Q load, single-head items so far
            bool single_before = false;
            for (int r = 0; CHAIN || r == 0; ++r) {
                int nlist, m, T, tok0, h0, ntile;
                take(r, nlist, m, T, tok0, h0, ntile);
                const int g = s_item[r & 1].g;
                const long long at = s_item[r & 1].at;
                taken(r);
                if (nlist < 0) break;
                if (*abort_flag) {                        // a wait gave up: let the copies in flight land, then leave
                    const long long t0 = clock64();
                    while (clock64() - t0 < 2000000) {}
                    break;
                }
                const uint16_t* list = mv.row_list + at;
                const uint8_t* cls = mv.tile_class + at;
                if (nlist > 0) {
                    if (q_items > 0) mbar_wait(bar_qfree, (q_items - 1) & 1, abort_flag, status);
                    if (lane == 0) {
                        mbar_expect_tx(bar_q, ntile * L::TB);
                        for (int t = 0; t < ntile; ++t)
                            for (int c = 0; c < NBOX; ++c)
                                tma_load_3d(sQ + t * L::TB + c * BOX_BYTES, &tm_q, c * 64, h0 + t, tok0 + m * TILE, bar_q);
                    }
                    ++q_items;
                    // the streams of a single head are merged through the ring's memory
                    if (single_before) mbar_wait(bar_xfree, (singles - 1) & 1, abort_flag, status);
                }
                // K runs one key block ahead of V: the slot of K(i+1) is released by the Q K^T products of
                // block i-1, which are issued a whole iteration before the P V products that release V's slot.
                auto load_k = [&](int i) {
                    const uint32_t R = ring + i;
                    const int s = R & 1;
                    if (R >= 2) mbar_wait(bar_kfree(s), ((R >> 1) + 1) & 1, abort_flag, status);
                    if (lane == 0) {
                        mbar_expect_tx(bar_kfull(s), L::TB);
                        const uint32_t dst = sKV + s * 2 * L::TB;
                        for (int c = 0; c < NBOX; ++c) tma_load_3d(dst + c * BOX_BYTES, &tm_k, c * 64, g, tok0 + list[i] * TILE, bar_kfull(s));
                    }
                };
                if (nlist > 0) load_k(0);
                for (int i = 0; i < nlist; ++i) {
                    const uint32_t R = ring + i;
                    const int s = R & 1;
                    const int n = list[i];
                    const bool need_mask = (cls[n] != KVS_CLASS_FULL) || (n * TILE + TILE > T);
                    // What the mask needs comes first: the softmax groups are done with the stage's last one well before its V is
                    // free, and must not wait for that.
                    int ev[4] = {0, 0, 0, 0}, kf[4] = {0, 0, 0, 0};       // the intervals of the tile's key slots
                    if (need_mask) {
#pragma unroll
                        for (int u = 0; u < 4; ++u) {
                            const int j = n * TILE + lane * 4 + u;
                            ev[u] = (j < T) ? mv.evict[tok0 + j] : 0;                       // 0: visible to nobody
                            kf[u] = (general && j < T) ? mv.kfirst[tok0 + j] : j;
                        }
                    }
                    // What a softmax warp (32 rows, quadrant q) has to do for the keys 32 c .. 32 c + 31: bit 8 c + q of `hidden`:
                    // none of its rows sees any of them; else bit 8 c + q of `compare`: some key is evicted before the last row,
                    // bit 8 c + 4 + q: some key is not there yet for the first row.  Found here, beside the loads: votes by the
                    // softmax warps, with both comparisons where a group was mixed, took 13 % of a forward whose tiles all are
                    // (24576 tokens, token-level eviction: 11.1 -> 9.2 ms).
                    uint32_t compare = 0, hidden = 0;
                    if (need_mask) {
                        int ev0 = min(min(ev[0], ev[1]), min(ev[2], ev[3])), ev1 = max(max(ev[0], ev[1]), max(ev[2], ev[3]));
                        int kf0 = min(min(kf[0], kf[1]), min(kf[2], kf[3])), kf1 = max(max(kf[0], kf[1]), max(kf[2], kf[3]));
#pragma unroll
                        for (int o = 1; o < 8; o <<= 1) {                 // over the 8 lanes with the group's keys
                            ev0 = min(ev0, __shfl_xor_sync(0xffffffffu, ev0, o));
                            ev1 = max(ev1, __shfl_xor_sync(0xffffffffu, ev1, o));
                            kf0 = min(kf0, __shfl_xor_sync(0xffffffffu, kf0, o));
                            kf1 = max(kf1, __shfl_xor_sync(0xffffffffu, kf1, o));
                        }
                        const int q_lo = m * TILE + (lane & 3) * 32, q_hi = q_lo + 31;
                        const bool none = kf0 > q_hi || ev1 <= q_lo;
                        hidden = __ballot_sync(0xffffffffu, none);
                        compare = __ballot_sync(0xffffffffu, !none && ((lane & 4) ? kf1 > q_lo : ev0 <= q_hi));
                    }
                    if (R >= 2) mbar_wait(bar_evfree(s), ((R >> 1) + 1) & 1, abort_flag, status);
                    if (need_mask) {
                        *reinterpret_cast<int4*>(sEv + s * TILE + lane * 4) = make_int4(ev[0], ev[1], ev[2], ev[3]);
                        *reinterpret_cast<int4*>(sKf + s * TILE + lane * 4) = make_int4(kf[0], kf[1], kf[2], kf[3]);
                    }
                    if (lane == 0) {
                        sFlag[2 * s] = (int32_t)compare;
                        sFlag[2 * s + 1] = (int32_t)hidden;
                    }
                    mbar_arrive(bar_evfull(s));
                    if (R >= 2) mbar_wait(bar_vfree(s), ((R >> 1) + 1) & 1, abort_flag, status);
                    if (lane == 0) {
                        mbar_expect_tx(bar_vfull(s), L::TB);
                        const uint32_t dst = sKV + s * 2 * L::TB;
                        for (int c = 0; c < NBOX; ++c) tma_load_3d(dst + L::TB + c * BOX_BYTES, &tm_v, c * 64, g, tok0 + n * TILE, bar_vfull(s));
                    }
                    if (i + 1 < nlist) load_k(i + 1);
                }
                if (nlist > 0) {
                    ring += nlist;
                    single_before = ntile == 1;
                    if (ntile == 1) ++singles;
                }
            }
        } else if (CHAIN && warp == 10) {
            // ================= work list =================
            // The first item is the CTA's own; after it the CTAs that have not started yet, one at a time and only near the end of
            // the item before, so that the last items still go to whoever is free (20 traces of 500 to 2000: 274 -> 271 us against
            // asking at its start).  The chain of metadata loads of an item lies beside the one before.
            int x = blockIdx.x, y = blockIdx.y;
            bool ok = true;
            for (int r = 0, asked = 0;;) {
                while (ok && x >= nblk) {                             // also a CTA without work: the grid has room for any batch of these sizes
                    if (lane == 0) {
                        mbar_expect_tx(bar_ask, 16);
                        ask_for_cta(sbase + L::OFF_ASK, bar_ask);
                    }
                    mbar_wait(bar_ask, asked & 1, abort_flag, status);
                    ok = cta_answer(sbase + L::OFF_ASK, x, y) && !*abort_flag;
                    fence_proxy_async();                              // the answer is read before the next one comes over it
                    __syncwarp();
                    ++asked;
                }
                const int slot = r & 1;
                FwdItem it;
                it.nlist = -1;
                it.m = it.T = it.tok0 = it.g = it.h0 = it.ntile = 0;
                it.at = 0;
                if (ok) it = item_of(x, y);
                if (r >= 2) mbar_wait(bar_itemfree(slot), ((r >> 1) + 1) & 1, abort_flag, status);
                if (lane == 0) {
                    put(slot, it);
                    mbar_arrive(bar_item(slot));
                }
                __syncwarp();
                if (!ok || *abort_flag) break;
                mbar_wait(bar_late, r & 1, abort_flag, status);
                ++r;
                x = nblk;                                             // ask
            }
        } else if (warp == 9) {
            // ================= MMA issuer (all lanes walk the loop, one elected lane issues) =================
            const bool leader = elect_one();
            const uint64_t dQ0 = smem_desc(sQ, 16, 1024);
            const uint64_t dK0 = smem_desc(sKV, 16, 1024);
            const uint64_t dV0 = smem_desc(sKV + L::TB, BOX_BYTES, 1024);
            constexpr uint64_t TBU = (uint64_t)(L::TB >> 4);
            auto issue_s_q = [&](int t, int s, int qt) {      // S_t = Q_qt K(stage s)^T
#pragma unroll
                for (int kk = 0; kk < D / 16; ++kk) {
                    const uint64_t off = (uint64_t)(((kk >> 2) * BOX_BYTES + (kk & 3) * 32) >> 4);
                    if (leader) mma_ss(tmem + t * 128, dQ0 + qt * TBU + off, dK0 + s * 2 * TBU + off, IDESC_S, kk > 0);
                }
                if (leader) mma_commit(bar_s(t));
            };
            uint32_t ring = 0, q_items = 0, p_phase = 0;               // bit t of p_phase: phase of group t's next P
            int items = 0;                                             // items with key blocks
            for (int r = 0; CHAIN || r == 0; ++r) {
                int nlist, m, T, tok0, h0, ntile;
                take(r, nlist, m, T, tok0, h0, ntile);
                taken(r);
                if (CHAIN && (nlist < 0 || *abort_flag)) break;
                // the next item is asked for when this one has FWD_LATE key blocks left
                auto near_end = [&](int i) {
                    if (CHAIN && lane == 0 && (i + FWD_LATE == nlist || (i == 0 && nlist < FWD_LATE))) mbar_arrive(bar_late);
                };
                if (nlist == 0) {
                    near_end(0);
                    continue;
                }
                const uint32_t r0 = ring;
                ring += nlist;
                mbar_wait(bar_q, q_items & 1, abort_flag, status);
                ++q_items;
                // O_t += P_t V in two parts, once P's rows are there:  A = P rows from tensor memory (16 keys = 8 packed columns
                // per step), B = V, MN-major, 16 key rows per step.  The first P_SPLIT keys of P arrive while the row's last
                // exponentials are still being taken, so most of this product overlaps the tail of the softmax.
                auto issue_pv = [&](int t, uint32_t R, bool first, bool wait_v) {
                    const int s = R & 1;
                    const uint32_t pph = (p_phase >> t) & 1;
                    p_phase ^= 1u << t;
                    mbar_wait(bar_p0(t), pph, abort_flag, status);
                    if (wait_v) mbar_wait(bar_vfull(s), (R >> 1) & 1, abort_flag, status);
                    tc_fence_after();
#pragma unroll
                    for (int kk = 0; kk < P_SPLIT / 16; ++kk)
                        if (leader) mma_ts(tmem + 256 + t * 128, tmem + t * 128 + kk * 8, dV0 + s * 2 * TBU + (uint64_t)(kk * 128), IDESC_O,
                               !first || (kk > 0));
                    mbar_wait(bar_p(t), pph, abort_flag, status);
                    tc_fence_after();
#pragma unroll
                    for (int kk = P_SPLIT / 16; kk < TILE / 16; ++kk)
                        if (leader) mma_ts(tmem + 256 + t * 128, tmem + t * 128 + kk * 8, dV0 + s * 2 * TBU + (uint64_t)(kk * 128), IDESC_O, true);
                };
                auto wait_k = [&](uint32_t R) {
                    mbar_wait(bar_kfull(R & 1), (R >> 1) & 1, abort_flag, status);
                    tc_fence_after();
                };
                if (ntile == 1) {
                    // One head, two streams: stream t = key blocks i with i % 2 == t, on S_t / O_t.
                    for (int t = 0; t < 2 && t < nlist; ++t) {
                        wait_k(r0 + t);
                        issue_s_q(t, (r0 + t) & 1, 0);
                        if (leader) mma_commit(bar_kfree((r0 + t) & 1));
                    }
                    if (leader && nlist <= 2) mma_commit(bar_qfree);
                    if (items > 0) mbar_wait(bar_ofree, (items - 1) & 1, abort_flag, status);
#pragma unroll 1
                    for (int i = 0; i < nlist; ++i) {
                        const int t = i & 1;
                        const uint32_t R = r0 + i;
                        near_end(i);
                        issue_pv(t, R, i < 2, true);
                        if (leader) mma_commit(bar_vfree(R & 1));
                        if (i + 2 < nlist) {
                            wait_k(R + 2);
                            issue_s_q(t, R & 1, 0);
                            if (leader) mma_commit(bar_kfree(R & 1));
                            if (leader && i + 3 == nlist) mma_commit(bar_qfree);
                        }
                    }
                } else {
                    wait_k(r0);
                    for (int t = 0; t < 2; ++t) issue_s_q(t, r0 & 1, t);
                    if (leader) mma_commit(bar_kfree(r0 & 1));
                    if (leader && nlist == 1) mma_commit(bar_qfree);
                    if (items > 0) mbar_wait(bar_ofree, (items - 1) & 1, abort_flag, status);
#pragma unroll 1
                    for (int i = 0; i < nlist; ++i) {
                        const uint32_t R = r0 + i;
                        near_end(i);
#pragma unroll 1
                        for (int t = 0; t < 2; ++t) {
                            issue_pv(t, R, i == 0, t == 0);
                            if (leader && t == 1) mma_commit(bar_vfree(R & 1));       // V(i) is not read by anything issued later
                            if (i + 1 < nlist) {
                                if (t == 0) wait_k(R + 1);
                                issue_s_q(t, (R + 1) & 1, t);
                                if (leader && t == 1) mma_commit(bar_kfree((R + 1) & 1));
                                if (leader && t == 1 && i + 2 == nlist) mma_commit(bar_qfree);
                            }
                        }
                    }
                }
                if (leader) mma_commit(bar_done);
                ++items;
            }
        }
    } else {
        // ================= softmax groups =================
        reg_inc<208>();
        const int t = warp >> 2;                                  // which query tile / head (or stream of the single head)
        const int quad = warp & 3;
        const int row = quad * 32 + lane;                         // query row of the tile == TMEM lane
        const uint32_t lane_sel = (uint32_t)(quad * 32) << 16;
        const uint32_t tmem_S = tmem + t * 128 + lane_sel;
        const uint32_t tmem_O = tmem + 256 + t * 128 + lane_sel;
        uint32_t ring = 0, s_count = 0;                           // key blocks of the CTA, S tiles of this group so far
        int items = 0, singles = 0;                               // items with key blocks, those of a single head
        for (int r = 0; CHAIN || r == 0; ++r) {
            int nlist, m, T, tok0, h0, ntile;
            take(r, nlist, m, T, tok0, h0, ntile);
            taken(r);
            if (CHAIN && (nlist < 0 || *abort_flag)) break;
            const bool dual = ntile == 1;
            const int h = dual ? h0 : h0 + t;
            const int qi = m * TILE + row;                        // trace-local query index
            float ref_max = -INFINITY;                            // base-2 domain; the exponent's reference
            float run_sum = 0.f;

            const uint32_t first = ring + (dual ? t : 0), stride = dual ? 2 : 1;
            // The phase of this group's S follows from the key block's number, up to a constant of the item.  As a bit that every
            // tile flips it cost 1 % of a long row (3 traces of 9000 to 17000 tokens, nothing evicted: 3.39 -> 3.35 ms).
            const uint32_t s_shift = dual ? 1 : 0, s_off = CHAIN ? s_count - (first >> s_shift) : 0;
            ring += nlist;
            if (CHAIN && ring > first) s_count += (ring - first + stride - 1) >> s_shift;
            for (uint32_t R = first; R < ring; R += stride) {
                const int s = R & 1;
                mbar_wait(bar_evfull(s), (R >> 1) & 1, abort_flag, status);
                const uint32_t compare = (uint32_t)sFlag[2 * s] >> quad, hidden = (uint32_t)sFlag[2 * s + 1] >> quad;
                mbar_wait(bar_s(t), ((R >> s_shift) + s_off) & 1, abort_flag, status);
                tc_fence_after();
                // raw logits of this row (the softmax scale is positive, so the maximum can be taken before it)
                float sv[TILE];
                {
                    uint32_t r0[32], r1[32], r2[32], r3[32];
                    tmem_ld32(tmem_S, r0);
                    tmem_ld32(tmem_S + 32, r1);
                    tmem_ld32(tmem_S + 64, r2);
                    tmem_ld32(tmem_S + 96, r3);
                    tmem_wait_ld();
#pragma unroll
                    for (int e = 0; e < 32; ++e) {
                        sv[e] = __uint_as_float(r0[e]);
                        sv[32 + e] = __uint_as_float(r1[e]);
                        sv[64 + e] = __uint_as_float(r2[e]);
                        sv[96 + e] = __uint_as_float(r3[e]);
                    }
                }
                if (((compare | hidden) & 0x11111111u) != 0) {
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        if (hidden >> (8 * c) & 1u) {
#pragma unroll
                            for (int e = 0; e < 32; ++e) sv[c * 32 + e] = -INFINITY;
                        }
                        const int by_end = compare >> (8 * c) & 1u, by_start = compare >> (8 * c + 4) & 1u;
#pragma unroll 1
                        for (int pass = 0; pass < by_end; ++pass) {          // loops of at most one pass: not predicated
                            const int4* ev4 = reinterpret_cast<const int4*>(sEv + s * TILE + c * 32);
#pragma unroll
                            for (int e4 = 0; e4 < 8; ++e4) {
                                const int4 ev = ev4[e4];
                                float* x = sv + c * 32 + e4 * 4;
                                x[0] = (qi < ev.x) ? x[0] : -INFINITY;
                                x[1] = (qi < ev.y) ? x[1] : -INFINITY;
                                x[2] = (qi < ev.z) ? x[2] : -INFINITY;
                                x[3] = (qi < ev.w) ? x[3] : -INFINITY;
                            }
                        }
#pragma unroll 1
                        for (int pass = 0; pass < by_start; ++pass) {
                            const int4* kf4 = reinterpret_cast<const int4*>(sKf + s * TILE + c * 32);
#pragma unroll
                            for (int e4 = 0; e4 < 8; ++e4) {
                                const int4 kf = kf4[e4];
                                float* x = sv + c * 32 + e4 * 4;
                                x[0] = (kf.x <= qi) ? x[0] : -INFINITY;
                                x[1] = (kf.y <= qi) ? x[1] : -INFINITY;
                                x[2] = (kf.z <= qi) ? x[2] : -INFINITY;
                                x[3] = (kf.w <= qi) ? x[3] : -INFINITY;
                            }
                        }
                    }
                }
                __syncwarp();
                if (lane == 0) mbar_arrive_n(bar_evfree(s), stride);
                // eight independent partial maxima (three-input max), then a short tree
                float mx[8];
#pragma unroll
                for (int u = 0; u < 8; ++u) mx[u] = fmaxf(sv[u], sv[8 + u]);
#pragma unroll
                for (int e = 16; e < TILE; e += 16) {
#pragma unroll
                    for (int u = 0; u < 8; ++u) mx[u] = fmax3(mx[u], sv[e + u], sv[e + 8 + u]);
                }
                const float tile_max =
                    fmaxf(fmax3(mx[0], mx[1], mx[2]), fmaxf(fmax3(mx[3], mx[4], mx[5]), fmaxf(mx[6], mx[7]))) * p.scale_log2;
                // lazy rescale: move the reference only when the maximum ran away from it
                const bool grow = (tile_max > ref_max + RESCALE_THRESHOLD) || (ref_max == -INFINITY && tile_max > -INFINITY);
                if (__any_sync(0xffffffffu, grow)) {
                    const float new_ref = grow ? tile_max : ref_max;
                    const float alpha = (new_ref == -INFINITY) ? 1.f : fast_exp2(ref_max - new_ref);   // ref_max = -inf -> 0
                    run_sum *= alpha;
                    ref_max = new_ref;
                    if (R != first) {
#pragma unroll
                        for (int c = 0; c < D / 32; ++c) {
                            uint32_t r[32];
                            tmem_ld32(tmem_O + c * 32, r);
                            tmem_wait_ld();
#pragma unroll
                            for (int e = 0; e < 32; ++e) r[e] = __float_as_uint(__uint_as_float(r[e]) * alpha);
                            tmem_st32(tmem_O + c * 32, r);
                        }
                    }
                }
                const float neg_ref = (ref_max == -INFINITY) ? 0.f : -ref_max;
                // packed fp32x2: one multiply-add forms two exponents, one add accumulates two terms
                const float2 c2 = make_float2(p.scale_log2, p.scale_log2);
                const float2 nr2 = make_float2(neg_ref, neg_ref);
                float2 ts[4] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f), make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
                uint32_t pk[TILE / 2];
#pragma unroll
                for (int e = 0; e < TILE; e += 8) {
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const float2 x = __ffma2_rn(make_float2(sv[e + 2 * u], sv[e + 2 * u + 1]), c2, nr2);
                        const float2 pp = make_float2(fast_exp2(x.x), fast_exp2(x.y));
                        ts[u] = __fadd2_rn(ts[u], pp);
                        pk[(e >> 1) + u] = pack_bf16(pp.x, pp.y);
                    }
                    if (e + 8 == P_SPLIT) {
                        // P (bf16, packed two per column) goes over the S columns already read; the first
                        // P_SPLIT keys are handed to the MMA warp before the rest of the row is done
                        uint32_t r[32], r2[16];
#pragma unroll
                        for (int c = 0; c < 32; ++c) r[c] = pk[c];
#pragma unroll
                        for (int c = 0; c < 16; ++c) r2[c] = pk[32 + c];
                        tmem_st32(tmem_S, r);
                        tmem_st16(tmem_S + 32, r2);
                        tmem_wait_st();
                        tc_fence_before();
                        __syncwarp();
                        if (lane == 0) mbar_arrive(bar_p0(t));
                    }
                }
                const float2 t01 = __fadd2_rn(ts[0], ts[1]), t23 = __fadd2_rn(ts[2], ts[3]);
                const float tile_sum = (t01.x + t01.y) + (t23.x + t23.y);
                run_sum += tile_sum;
                {
                    uint32_t r2[16];
#pragma unroll
                    for (int c = 0; c < 16; ++c) r2[c] = pk[48 + c];
                    tmem_st16(tmem_S + 48, r2);
                }
                tmem_wait_st();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(bar_p(t));
            }

            // ---- epilogue: O / l -> bf16, LSE -> fp32 ----
            if (nlist > 0) mbar_wait(bar_done, items & 1, abort_flag, status);
            tc_fence_after();
            const bool valid = qi < T;
            // single head: stream 1 hands its partial result (O1 column by column, reference, sum) to stream 0
            // through the K/V ring's shared memory, which nothing uses any more
            float* x_o = reinterpret_cast<float*>(sgen + L::OFF_KV);           // [D][128 rows]
            float* x_ms = x_o + D * TILE;                                     // [2][128 rows]
            const bool has1 = dual && nlist > 1;
            float a0 = 1.f, a1 = 0.f;
            if (dual && nlist > 0) {
                if (t == 1) {
                    if (has1) {
#pragma unroll
                        for (int c = 0; c < D / 32; ++c) {
                            uint32_t r[32];
                            tmem_ld32(tmem_O + c * 32, r);
                            tmem_wait_ld();
#pragma unroll
                            for (int e = 0; e < 32; ++e) x_o[(c * 32 + e) * TILE + row] = __uint_as_float(r[e]);
                        }
                    }
                    x_ms[row] = ref_max;
                    x_ms[TILE + row] = run_sum;
                    fence_proxy_async();                          // the ring's next tile comes over these by TMA
                    __syncwarp();
                    if (lane == 0) mbar_arrive(bar_x);
                } else {
                    mbar_wait(bar_x, singles & 1, abort_flag, status);
                    const float ref1 = has1 ? x_ms[row] : -INFINITY, sum1 = has1 ? x_ms[TILE + row] : 0.f;
                    const float mm = fmaxf(ref_max, ref1);
                    a0 = (ref_max == -INFINITY) ? 0.f : fast_exp2(ref_max - mm);
                    a1 = (ref1 == -INFINITY) ? 0.f : fast_exp2(ref1 - mm);
                    run_sum = run_sum * a0 + sum1 * a1;
                    ref_max = mm;
                }
                ++singles;
            }
            if (!dual || t == 0) {
                float inv = (run_sum > 0.f && nlist > 0) ? 1.f / run_sum : 0.f;
                float lse = ref_max * 0.6931471805599453f + logf(run_sum), w_first = 0.f;
                if (MERGE) {
                    // this part's is -inf where it saw no key and NaN where a score was one, and stays so
                    const float other = valid ? p.first_lse[(size_t)h * p.total_tokens + tok0 + qi] : -INFINITY, mine = lse;
                    const float top = fmaxf(other, mine);
                    lse = -INFINITY;
                    if (top > -INFINITY) {
                        const float ea = __expf(other - top), eb = __expf(mine - top), sum = ea + eb;      // exp(-inf) = 0 for a part that saw no key
                        w_first = ea / sum;
                        inv *= eb / sum;
                        lse = top + logf(sum);
                    }
                }
                // Through shared memory to memory as whole rows: the whole row through the query tile, which no product reads any
                // more, or, where the next item's comes there, in pieces of 64 bytes through memory of its own.
                constexpr int COLS = CHAIN ? 32 : D;
                using Rows = RowStage<COLS>;
                uint8_t* stage = sgen + (CHAIN ? L::OFF_STG + warp * 2048 : L::OFF_Q + warp * (L::TB / 4));
                __nv_bfloat16* orow = p.out + ((size_t)(tok0 + m * TILE + quad * 32) * p.Hq + h) * D;
                const int rows = T - m * TILE - quad * 32;
#pragma unroll
                for (int c = 0; c < D / 32; ++c) {
                    uint32_t r[32];
                    tmem_ld32(tmem_O + c * 32, r);
                    tmem_wait_ld();
                    if (nlist == 0) {      // a bad evict_at (already reported by the metadata pass), or nothing evicted yet
#pragma unroll
                        for (int e = 0; e < 32; ++e) r[e] = 0u;
                    }
                    if (dual && nlist > 0) {
#pragma unroll
                        for (int e = 0; e < 32; ++e) {
                            float o = __uint_as_float(r[e]) * a0;
                            if (a1 > 0.f) o = fmaf(x_o[(c * 32 + e) * TILE + row], a1, o);
                            r[e] = __float_as_uint(o);
                        }
                    }
                    if (MERGE) {
                        if (c % (COLS / 32) == 0)
                            Rows::template fetch<2>(stage, lane, reinterpret_cast<const char*>(p.first_out + (orow - p.out) + (CHAIN ? c * 32 : 0)),
                                                    (size_t)p.Hq * D, rows);
                        uint32_t x[16];
                        Rows::get_bf16(stage, lane, c % (COLS / 32), x);
#pragma unroll
                        for (int e = 0; e < 16; ++e) {
                            r[2 * e] = __float_as_uint(fmaf(__uint_as_float(x[e] << 16), w_first, __uint_as_float(r[2 * e]) * inv));
                            r[2 * e + 1] = __float_as_uint(fmaf(__uint_as_float(x[e] & 0xffff0000u), w_first, __uint_as_float(r[2 * e + 1]) * inv));
                        }
                    } else {
#pragma unroll
                        for (int e = 0; e < 32; ++e) r[e] = __float_as_uint(__uint_as_float(r[e]) * inv);
                    }
                    Rows::put_bf16(stage, lane, c % (COLS / 32), r);
                    if ((c + 1) % (COLS / 32) == 0)
                        Rows::template flush<2>(stage, lane, reinterpret_cast<char*>(orow + (CHAIN ? c * 32 : 0)), (size_t)p.Hq * D, rows);
                }
                if (valid) p.lse[(size_t)h * p.total_tokens + tok0 + qi] = lse;
            }
            if (nlist > 0) {
                tc_fence_before();
                __syncwarp();
                if (CHAIN && lane == 0) {
                    mbar_arrive(bar_ofree);                       // the next item's P V products may overwrite O
                    if (dual && t == 0) mbar_arrive(bar_xfree);
                }
                ++items;
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 9) {
        __syncwarp();
        tmem_dealloc(tmem, TMEM_COLS);
    }
}

template <int D, bool CHAIN, bool MERGE>
static int launch_fwd(const CUtensorMap& tq, const CUtensorMap& tk, const CUtensorMap& tv, const MetaView& mv, const FwdParams& p,
                      int nb_cap, cudaStream_t st) {
    auto kern = fwd_kernel<D, CHAIN, MERGE>;
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, FwdSmem<D>::DYN_BYTES) != cudaSuccess) return cuda_refused();
    return launch_after(kern, dim3(nb_cap, p.heads, 1), FWD_THREADS, FwdSmem<D>::DYN_BYTES, st, tq, tk, tv, mv, p);
}

// Items are chained where rows are short and the grid is a few waves of CTAs.  A chained CTA saves the start and the end of an
// item; its loop over items costs 2 to 4 % of a tile.  Forward, a CTA per item -> chained, us (32 heads on 8; of the same batch
// with last-4-turns eviction and with none): 131 x 500 tokens 751 -> 615, 725 -> 589; 32 x 2000 946 -> 841, 1260 -> 1167;
// 14 x 4500 1333 -> 1272, 2123 -> 2111; 9 x 7000 1639 -> 1597, 2955 -> 2987; 5 x 12000 2210 -> 2209, 4519 -> 4637: with nothing
// evicted they meet at 5000 tokens.  Longer traces need more waves, or a CTA has an item in hand while others have nothing left:
// 4 x 1000 (3.8 waves) 64.5 -> 62.7, but 1 x 3000 (2.6) 72.2 -> 75.8, 2 x 3000 (5.2) 117 -> 118; 1 x 1000 (0.9) 22.5 -> 24.3.
// The mean length is what is known here that a caller cannot overstate.  A long trace among many short ones is chained with them
// (32768 + 60 x 300: 2938 -> 2984; 16000 + 100 x 300: 1118 -> 1098).
static bool chain_items(int batch, int total_tokens, int nb_cap, int heads) {
    const long long ctas = (long long)nb_cap * heads;
    const int mean = total_tokens / batch;
    return (mean <= 2048 && ctas > 2 * 148) || (mean <= 4096 && ctas > 6 * 148);
}

}  // namespace kvs

using namespace kvs;

namespace {
// q_ts / kv_ts: elements between consecutive tokens of q and of k, v (0: tensors of their own)
int fwd_impl(const void* q, const void* k, const void* v, long long q_ts, long long kv_ts, const void* meta_buf, int batch,
             int total_tokens, int max_seqlen, int Hq, int Hkv, int head_dim, float softmax_scale, void* out, float* lse,
             kvs_stream_t stream, const void* first_out = nullptr, const float* first_lse = nullptr) {
    if (batch < 0 || total_tokens < 0 || max_seqlen < 0 || Hq <= 0 || Hkv <= 0) return KVS_ERR_INVALID_ARG;
    if (head_dim != 64 && head_dim != 128) return KVS_ERR_UNSUPPORTED;
    if (Hq % Hkv != 0 || Hq > 65535) return KVS_ERR_UNSUPPORTED;
    if (total_tokens == 0 || batch == 0) return KVS_OK;
    if (!q || !k || !v || !meta_buf || !out || !lse) return KVS_ERR_INVALID_ARG;
    if ((((uintptr_t)q | (uintptr_t)k | (uintptr_t)v | (uintptr_t)out) & 15) != 0 || ((uintptr_t)lse & 3) != 0) return KVS_ERR_ALIGNMENT;
    if (((uintptr_t)meta_buf & 255) != 0) return KVS_ERR_ALIGNMENT;
    if (softmax_scale < 0.f || softmax_scale != softmax_scale) return KVS_ERR_INVALID_ARG;
    int rc = check_device_sm100();
    if (rc != KVS_OK) return rc;
    const MetaLayout L = meta_layout(batch, total_tokens, max_seqlen);
    const MetaView mv = meta_view(meta_buf, L);
    CUtensorMap tq, tk, tv;
    if ((rc = make_tmap_thd(&tq, q, total_tokens, Hq, head_dim, TILE, q_ts)) != KVS_OK) return rc;
    if ((rc = make_tmap_thd(&tk, k, total_tokens, Hkv, head_dim, TILE, kv_ts)) != KVS_OK) return rc;
    if ((rc = make_tmap_thd(&tv, v, total_tokens, Hkv, head_dim, TILE, kv_ts)) != KVS_OK) return rc;
    FwdParams p;
    p.batch = batch;
    p.total_tokens = total_tokens;
    p.max_seqlen = max_seqlen < total_tokens ? max_seqlen : total_tokens;
    p.Hq = Hq;
    p.Hkv = Hkv;
    p.heads = Hkv * ((Hq / Hkv + 1) / 2);
    const float s = softmax_scale == 0.f ? 1.0f / sqrtf((float)head_dim) : softmax_scale;
    p.scale_log2 = s * 1.4426950408889634f;
    p.out = (__nv_bfloat16*)out;
    p.lse = lse;
    p.first_out = (const __nv_bfloat16*)first_out;
    p.first_lse = first_lse;
    cudaStream_t st = (cudaStream_t)stream;
    const bool chain = chain_items(batch, total_tokens, L.nb_cap, p.heads);
    auto launch = [&](auto dim) {
        constexpr int D = decltype(dim)::value;
        if (first_out) return chain ? launch_fwd<D, true, true>(tq, tk, tv, mv, p, L.nb_cap, st) : launch_fwd<D, false, true>(tq, tk, tv, mv, p, L.nb_cap, st);
        return chain ? launch_fwd<D, true, false>(tq, tk, tv, mv, p, L.nb_cap, st) : launch_fwd<D, false, false>(tq, tk, tv, mv, p, L.nb_cap, st);
    };
    return head_dim == 64 ? launch(std::integral_constant<int, 64>()) : launch(std::integral_constant<int, 128>());
}
}  // namespace

extern "C" int kvs_attn_fwd(const void* q, const void* k, const void* v, const void* meta_buf, int batch, int total_tokens,
                            int max_seqlen, int Hq, int Hkv, int head_dim, float softmax_scale, void* out, float* lse,
                            kvs_stream_t stream) {
    return fwd_impl(q, k, v, 0, 0, meta_buf, batch, total_tokens, max_seqlen, Hq, Hkv, head_dim, softmax_scale, out, lse, stream);
}

extern "C" int kvs_attn_fwd_packed(const void* qkv, const void* meta_buf, int batch, int total_tokens, int max_seqlen, int Hq,
                                   int Hkv, int head_dim, float softmax_scale, void* out, float* lse, kvs_stream_t stream) {
    if (Hq <= 0 || Hkv <= 0 || head_dim <= 0) return KVS_ERR_INVALID_ARG;
    if (total_tokens > 0 && batch > 0 && !qkv) return KVS_ERR_INVALID_ARG;
    const long long ts = (long long)(Hq + 2 * Hkv) * head_dim;
    const char* base = (const char*)qkv;
    return fwd_impl(base, base + (size_t)Hq * head_dim * 2, base + (size_t)(Hq + Hkv) * head_dim * 2, ts, ts, meta_buf, batch,
                    total_tokens, max_seqlen, Hq, Hkv, head_dim, softmax_scale, out, lse, stream);
}

int kvs::attn_fwd_merged(const void* q, const void* k, const void* v, const void* meta_buf, int batch, int total_tokens, int max_seqlen, int Hq,
                         int Hkv, int head_dim, float softmax_scale, const void* first_out, const float* first_lse, void* out, float* lse,
                         kvs_stream_t stream) {
    return fwd_impl(q, k, v, 0, 0, meta_buf, batch, total_tokens, max_seqlen, Hq, Hkv, head_dim, softmax_scale, out, lse, stream, first_out,
                    first_lse);
}
