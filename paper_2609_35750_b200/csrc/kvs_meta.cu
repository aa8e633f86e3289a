// Mask metadata: per key block min/max of evict_at, per-tile class, per-row lists, launch orders.
// Integer work only, bound by latency: two kernels on the caller's stream, or one for small batches, no host synchronisation.
#include "kvs_common.cuh"

namespace kvs {

constexpr int META_THREADS = 256;
constexpr int META_WARPS = META_THREADS / 32;

// ---- parts of the kernels ---------------------------------------------------------------------------------------
// What a key block's slots say, found by a warp; lane 0 has `first`, `last`: the query blocks that can see the block.
struct BlockStat {
    int mn, mx, fmn, fmx, first, last;
    bool invalid;
};
__device__ __forceinline__ BlockStat meta_block_stat(const int32_t* evict_at, const int32_t* key_first, int complement, int n, int tok0, int T,
                                                     int32_t* evict_copy, int32_t* first_copy) {
    const int lane = threadIdx.x & 31, nb = (T + TILE - 1) / TILE;
    BlockStat r = {INT32_MAX, INT32_MIN, INT32_MAX, INT32_MIN, 0, 0, false};
    const bool general = complement || key_first;
#pragma unroll
    for (int t = 0; t < TILE / 32; ++t) {
        const int j = n * TILE + t * 32 + lane;
        if (j < T) {
            const int e = complement ? INT32_MAX : evict_at[tok0 + j];
            const int f = complement ? evict_at[tok0 + j] : (key_first ? key_first[tok0 + j] : j);
            evict_copy[tok0 + j] = e;
            if (general) first_copy[tok0 + j] = f;
            r.invalid |= general ? (f < 0) : (e <= j);
            r.mn = min(r.mn, e);
            r.mx = max(r.mx, e);
            r.fmn = min(r.fmn, f);
            r.fmx = max(r.fmx, f);
        }
    }
    r.mn = __reduce_min_sync(0xffffffffu, r.mn);
    r.mx = __reduce_max_sync(0xffffffffu, r.mx);
    r.fmn = __reduce_min_sync(0xffffffffu, r.fmn);
    r.fmx = __reduce_max_sync(0xffffffffu, r.fmx);
    r.invalid = __any_sync(0xffffffffu, r.invalid);
    // last query block whose first row q0 = 128 m is still below kmax; first one whose last row reaches fmin
    long long last = ((long long)r.mx - 1) / TILE;
    if (last > nb - 1) last = nb - 1;
    long long first = r.fmn / TILE;
    if (first > nb) first = nb;
    if (first < 0) first = 0;                  // a negative key_first is reported; never an index
    if (!general && last < n) last = n;
    r.first = (int)first;
    r.last = (r.mx <= 0) ? -1 : (int)last;
    return r;
}

// A warp's query block row m of a trace of T tokens: the classes of its tiles and the list of the non-empty ones, whose number
// is returned.  kmin .. fmax: of the trace's key blocks.
__device__ __forceinline__ int meta_classify_row(int m, int T, const int32_t* kmin, const int32_t* kmax, const int32_t* fmin, const int32_t* fmax,
                                                 uint8_t* cls_row, uint16_t* list_row) {
    const int lane = threadIdx.x & 31, nb = (T + TILE - 1) / TILE;
    const int q0 = m * TILE, q1 = min(q0 + TILE - 1, T - 1);
    int count = 0;
    for (int n0 = 0; n0 < nb; n0 += 32) {
        const int n = n0 + lane;
        int c = KVS_CLASS_EMPTY;
        if (n < nb) {
            // f0, f1: the earliest / latest "first query that may see the slot" of the block; for plain
            // metadata these are the block's first and last valid key, k0 and k1
            const int f0 = fmin[n], f1 = fmax[n];
            const int mn = kmin[n], mx = kmax[n];
            if (f0 > q1 || q0 >= mx) c = KVS_CLASS_EMPTY;
            else if (f1 <= q0 && q1 < mn) c = KVS_CLASS_FULL;
            else c = KVS_CLASS_PARTIAL;
            cls_row[n] = (uint8_t)c;
        }
        const unsigned live = __ballot_sync(0xffffffffu, c != KVS_CLASS_EMPTY);
        if (c != KVS_CLASS_EMPTY) list_row[count + __popc(live & ((1u << lane) - 1u))] = (uint16_t)n;
        count += __popc(live);
    }
    return count;
}

// The bucket of a length in a launch order (see meta_order), of nbins
__device__ __forceinline__ bool meta_exact(int max_seqlen) { return max_seqlen <= 16 * TILE; }
__device__ __forceinline__ int meta_bins(int max_seqlen, int most) { return meta_exact(max_seqlen) ? 17 : min((max_seqlen / TILE >> 4) + 2, most); }
__device__ __forceinline__ int meta_bin(int len, bool exact, int nbins) { return nbins - 1 - min(exact ? len : len >> 4, nbins - 1); }   // the longest first

// ---- kernel 1: offsets, and per key block (one warp each) min / max over its key slots, validity ---------------
// Every CTA goes through the traces itself, 256 at a time (a scan of their block counts), and keeps what its eight blocks
// need; the first CTA writes the tables.  A kernel of its own for the offsets, with one thread walking the traces, took 24 us
// for 96 of them, and another launch.
//
// Slot j of a trace holds a key that query i may read iff first[j] <= i < evict[j].  Plain metadata
// (key_first == nullptr): first[j] = j and evict[j] > j is required.  General metadata: both arrays come
// from the caller (keys re-ordered, or another visibility rule) and a slot may be visible to nobody.
// complement != 0: the slots of the EVICTED keys: slot j becomes visible at evict_at[j] and stays (first = evict_at,
// evict = never), i.e. the causal key set minus what the eviction mask still shows.
__global__ void __launch_bounds__(META_THREADS)
meta_blocks_kernel(const int32_t* __restrict__ evict_at, const int32_t* __restrict__ key_first, int complement,
                   const int32_t* __restrict__ cu_seqlens, int batch, int total_tokens, int max_seqlen, MetaHeader* hdr, int32_t* blk_off,
                   uint32_t* cls_off, int32_t* seq_start, int32_t* blk_trace, int4* info, int nb_cap, unsigned long long cls_cap, int32_t* kmin,
                   int32_t* kmax, int32_t* fmin, int32_t* fmax, int32_t* col_first, int32_t* col_last, int32_t* row_cnt,
                   int32_t* evict_copy, int32_t* first_copy) {
    __shared__ unsigned long long s_cls[META_WARPS];
    __shared__ long long s_blk[META_WARPS];
    __shared__ int s_trace[META_WARPS];
    __shared__ int4 s_mine[META_WARPS];              // the block's info
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    pdl_wait();
    const long long blk0 = (long long)blockIdx.x * META_WARPS;
    const bool writer = blockIdx.x == 0;
    if (tid < META_WARPS) s_trace[tid] = -1;
    bool bad = cu_seqlens[0] != 0 || cu_seqlens[batch] != total_tokens;
    long long nblk = 0;
    unsigned long long ncls = 0;
    for (int b0 = 0; b0 < batch; b0 += META_THREADS) {
        const int b = b0 + tid;
        long long a = 0, T = 0;
        if (b < batch) {
            a = cu_seqlens[b];
            T = cu_seqlens[b + 1] - a;
            if (T < 0 || T > max_seqlen || a < 0 || a + T > total_tokens) {
                bad = true;
                T = 0;
            }
        }
        const long long nb = (T + TILE - 1) / TILE;
        long long ib = nb;
        unsigned long long ic = (unsigned long long)(nb * nb);
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const long long tb = __shfl_up_sync(0xffffffffu, ib, o);
            const unsigned long long tc = __shfl_up_sync(0xffffffffu, ic, o);
            if (lane >= o) {
                ib += tb;
                ic += tc;
            }
        }
        __syncthreads();                                  // the previous round's totals have been read
        if (lane == 31) {
            s_blk[warp] = ib;
            s_cls[warp] = ic;
        }
        __syncthreads();
        long long first = nblk + ib - nb;
        unsigned long long first_cls = ncls + ic - (unsigned long long)(nb * nb);
#pragma unroll
        for (int w = 0; w < META_WARPS; ++w) {
            if (w < warp) {
                first += s_blk[w];
                first_cls += s_cls[w];
            }
            nblk += s_blk[w];
            ncls += s_cls[w];
        }
        if (b < batch) {
            const long long lo = max(first, blk0), hi = min(first + nb, blk0 + META_WARPS);
            for (long long i = lo; i < hi; ++i) {
                s_trace[i - blk0] = b;
                s_mine[i - blk0] = make_int4((int)a, (int)T, (int)(i - first), (int)(uint32_t)(first_cls + (i - first) * nb));
            }
            if (writer) {
                blk_off[b] = (int32_t)first;
                cls_off[b] = (uint32_t)first_cls;
                seq_start[b] = (int32_t)a;
            }
        }
    }
    if (__syncthreads_or(bad) || nblk > nb_cap || ncls > cls_cap) {
        bad = true;
        nblk = 0;
        ncls = 0;
    }
    if (writer && tid == 0) {
        blk_off[batch] = (int32_t)nblk;
        cls_off[batch] = (uint32_t)ncls;
        seq_start[batch] = total_tokens;
        hdr->magic = META_MAGIC;
        hdr->status = bad ? KVS_ERR_BAD_EVICT : KVS_OK;         // invalid keys are reported by the next kernel
        hdr->batch = batch;
        hdr->total_tokens = total_tokens;
        hdr->max_seqlen = max_seqlen;
        hdr->nblk_total = (int32_t)nblk;
        hdr->ncls_total = (uint32_t)ncls;
        hdr->general = (key_first || complement) ? 1 : 0;
        hdr->npair_total = 0;
        hdr->rows_done = 0;
        hdr->has_info = info != nullptr;
    }
    const int4 mine = s_mine[warp];
    if (blk0 + warp >= nblk || s_trace[warp] < 0) return;
    const int blk = (int)blk0 + warp;
    const int n = mine.z, tok0 = mine.x, T = mine.y;
    const BlockStat st = meta_block_stat(evict_at, key_first, complement, n, tok0, T, evict_copy, first_copy);
    if (lane == 0) {
        blk_trace[blk] = s_trace[warp];
        if (info) info[blk] = mine;
        kmin[blk] = st.mn;
        kmax[blk] = st.mx;
        fmin[blk] = st.fmn;
        fmax[blk] = st.fmx;
        col_first[blk] = st.first;
        col_last[blk] = st.last;
        row_cnt[blk] = st.invalid ? -1 : 0;        // for the next kernel, which puts the count here
    }
}

// ---- launch orders, heaviest first -----------------------------------------------------------------------------
// One CTA sorts n items into buckets by length, longest bucket first; items of a bucket keep their order in the batch, so
// CTAs launched together work on neighbouring blocks and share tiles in L2.
//   ORDER_ROWS   query blocks by their number of non-empty key blocks (forward)
//   ORDER_COLS   key blocks by the length of their query-block range (backward)
//   ORDER_PAIRS  pairs (2p, 2p+1) of a trace's key blocks by the length of their joint range (backward by CTA pairs)
// Coarse buckets (16 tiles): exact lengths would interleave blocks from all over the batch, coarse ones keep runs of
// neighbouring blocks together while still starting the long ones first.  Where no trace has more than 16 tiles they
// would all fall into one bucket and the longest might start last: there the lengths are exact (96 traces of 60 to
// 900 tokens: step 955 -> 894 us; 12 traces of 1500 to 12000 tokens with exact short lengths: 8274 -> 8678 us).
enum { ORDER_ROWS, ORDER_COLS, ORDER_PAIRS };
constexpr int ORDER_BINS = 4096;
constexpr int ORDER_CACHED = 12288;        // lengths kept in shared memory between the passes
// A kept length has 16 bits.  Two of its values stand for something else: a block that is not an item, and a length that they
// leave no room for (65534 and 65535 blocks, the longest traces there are), which is looked up again.
constexpr int ORDER_NONE = 0xffff, ORDER_LONG = 0xfffe;

__device__ void meta_order(int what, MetaHeader* hdr, const int32_t* blk_off, const int32_t* blk_trace, const int32_t* row_cnt,
                           const int32_t* col_first, const int32_t* col_last, int32_t* order, int32_t* len_out) {
    __shared__ int bins[ORDER_BINS];
    __shared__ uint16_t cached[ORDER_CACHED];
    __shared__ unsigned int s_sum;
    __shared__ int s_most, s_items;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int n = hdr->nblk_total;
    const bool exact = meta_exact(hdr->max_seqlen);
    const int nbins = meta_bins(hdr->max_seqlen, ORDER_BINS);
    auto length = [&](int i) {              // -1: not an item of its own
        if (what == ORDER_ROWS) return __ldcg(row_cnt + i);
        if (what == ORDER_COLS) return max(col_last[i] - col_first[i] + 1, 0);
        const int b = blk_trace[i], lo = blk_off[b], hi = blk_off[b + 1];
        int first, last;
        pair_range(col_first, col_last, i, i + 1 < hi, first, last);
        return ((i - lo) & 1) ? -1 : max(last - first + 1, 0);
    };
    auto bin = [&](int len) { return meta_bin(len, exact, nbins); };
    // Every warp has a run of the items and a column of the bins, so that all of them can scatter: by one warp alone the
    // metadata of 128 traces of 32768 tokens took 493 us, 172 like this.  Fewer columns where the bins have no room for eight
    // (traces of a million tokens), one for the few items of a small batch, whose sort is a matter of latency.
    int cols = n > 64 ? META_WARPS : 1;
    while (nbins * cols > ORDER_BINS) cols >>= 1;
    const int run_len = (n + 32 * cols - 1) / (32 * cols) * 32;
    for (int i = tid; i < nbins * cols; i += META_THREADS) bins[i] = 0;
    if (tid == 0) {
        s_sum = 0;
        s_most = 0;
    }
    __syncthreads();
    unsigned int sum = 0;
    int most = 0;
    for (int i = tid; i < n; i += META_THREADS) {
        const int len = length(i);
        if (i < ORDER_CACHED) cached[i] = (uint16_t)(len < 0 ? ORDER_NONE : min(len, ORDER_LONG));
        if (len < 0) continue;
        atomicAdd(&bins[bin(len) * cols + (cols == 1 ? 0 : i / run_len)], 1);
        sum += len;
        most = max(most, len);
    }
    sum = __reduce_add_sync(0xffffffffu, sum);
    most = __reduce_max_sync(0xffffffffu, most);
    if (lane == 0) {
        atomicAdd(&s_sum, sum);
        atomicMax(&s_most, most);
    }
    __syncthreads();
    if (warp == 0) {
        // exclusive scan over the bins, and in a bin over the columns
        int run = 0;
        for (int i0 = 0; i0 < nbins * cols; i0 += 32) {
            const int c = i0 + lane < nbins * cols ? bins[i0 + lane] : 0;
            int incl = c;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int t = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += t;
            }
            if (i0 + lane < nbins * cols) bins[i0 + lane] = run + incl - c;
            run += __shfl_sync(0xffffffffu, incl, 31);
        }
        if (lane == 0) s_items = run;
    }
    __syncthreads();
    if (warp >= cols) return;
    // the stable scatter of the warp's run, 32 blocks at a time in index order
    const int end = min(n, (warp + 1) * run_len);
    for (int i0 = warp * run_len; i0 < end; i0 += 32) {
        const int i = i0 + lane;
        int len = -1;
        if (i < end) {
            len = i < ORDER_CACHED ? (int)cached[i] : ORDER_LONG;
            len = len == ORDER_NONE ? -1 : len == ORDER_LONG ? length(i) : len;
        }
        const int k = len < 0 ? -1 : bin(len) * cols + warp;
        const unsigned same = __match_any_sync(0xffffffffu, k);
        if (k >= 0) {
            const int at = bins[k] + __popc(same & ((1u << lane) - 1u));
            order[at] = i;
            if (len_out) len_out[at] = len;
        }
        __syncwarp();
        if (k >= 0 && lane == (__ffs(same) - 1)) bins[k] += __popc(same);
        __syncwarp();
    }
    if (warp != 0) return;
    if (lane == 0 && what == ORDER_COLS) {
        hdr->blk_most = s_most;
        hdr->blk_tiles = s_sum;
    }
    if (lane == 0 && what == ORDER_PAIRS) {
        hdr->npair_total = s_items;
        hdr->pair_most = s_most;
        hdr->pair_tiles = s_sum;
    }
}

// ---- kernel 2: one warp per query block row: classes and the compact non-empty list; the orders ----------------------
// The first two CTAs sort the key blocks and the pairs, the others classify, and the last of those to finish sorts the rows.
__global__ void __launch_bounds__(META_THREADS)
meta_classify_kernel(MetaHeader* hdr, MetaView mv, const int32_t* __restrict__ blk_off, const int32_t* __restrict__ blk_trace,
                     const int32_t* __restrict__ kmin, const int32_t* __restrict__ kmax,
                     const int32_t* __restrict__ fmin, const int32_t* __restrict__ fmax, const int32_t* __restrict__ col_first,
                     const int32_t* __restrict__ col_last, uint8_t* tile_class, uint16_t* row_list, int32_t* row_cnt, int32_t* fwd_order,
                     int32_t* bwd_order, int32_t* pair_order, int32_t* bwd_len, int32_t* pair_len) {
    pdl_wait();
    if (blockIdx.x < 2) {
        const bool pairs = blockIdx.x == 1;
        meta_order(pairs ? ORDER_PAIRS : ORDER_COLS, hdr, blk_off, blk_trace, row_cnt, col_first, col_last, pairs ? pair_order : bwd_order,
                   pairs ? pair_len : bwd_len);
        return;
    }
    __shared__ int s_last;
    const int row = (blockIdx.x - 2) * META_WARPS + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    if (row < hdr->nblk_total) {
        const int4 me = block_info(mv, row);
        const int base = row - me.z;
        const size_t at = (uint32_t)me.w;
        const int count = meta_classify_row(me.z, me.y, kmin + base, kmax + base, fmin + base, fmax + base, tile_class + at, row_list + at);
        if (lane == 0) {
            if (row_cnt[row] < 0) set_status(&hdr->status, KVS_ERR_BAD_EVICT);       // the block's keys, seen by kernel 1
            row_cnt[row] = count;
            __threadfence();
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) s_last = atomicAdd(&hdr->rows_done, 1u) == gridDim.x - 3;
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    meta_order(ORDER_ROWS, hdr, blk_off, blk_trace, row_cnt, col_first, col_last, fwd_order, nullptr);
}

// ---- small batches: all of it by one CTA ---------------------------------------------------------------------------
// The two kernels above are latency: a launch, two chains of loads and a sort each.  For up to META_SMALL blocks of few tokens everything
// between the input and the tables stays in shared memory of one CTA of 32 warps, and an item's place in an order is counted,
// not sorted for (the same order: by bucket, then by index).  It is slower where the one CTA
// has much to read and write: see launch_mask_meta.
constexpr int META_SMALL = 64, META_SMALL_TOKENS = 5120, META_SMALL_THREADS = 1024;
__global__ void __launch_bounds__(META_SMALL_THREADS)
meta_small_kernel(const int32_t* __restrict__ evict_at, const int32_t* __restrict__ key_first, int complement,
                  const int32_t* __restrict__ cu_seqlens, int batch, int total_tokens, int max_seqlen, MetaView v, int has_info, int nb_cap,
                  unsigned long long cls_cap) {
    // per block: trace, block of the trace, first token and length of the trace, first tile of the row
    __shared__ int s_trace[META_SMALL], s_n[META_SMALL], s_tok0[META_SMALL], s_T[META_SMALL], s_at[META_SMALL];
    __shared__ int s_kmin[META_SMALL], s_kmax[META_SMALL], s_fmin[META_SMALL], s_fmax[META_SMALL], s_first[META_SMALL], s_last[META_SMALL];
    __shared__ int s_len[3][META_SMALL];               // the items' lengths in the three orders, -1: not an item
    __shared__ int s_nblk, s_ncls, s_bad;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (tid < META_SMALL) s_len[0][tid] = s_len[1][tid] = s_len[2][tid] = -1;
    if (tid == 0) s_bad = 0;
    pdl_wait();
    if (warp == 0) {                                   // the offsets: the traces, 32 at a time
        bool bad = cu_seqlens[0] != 0 || cu_seqlens[batch] != total_tokens;
        long long nblk = 0, ncls = 0;
        for (int b0 = 0; b0 < batch; b0 += 32) {
            const int b = b0 + lane;
            long long a = 0, T = 0;
            if (b < batch) {
                a = cu_seqlens[b];
                T = cu_seqlens[b + 1] - a;
                if (T < 0 || T > max_seqlen || a < 0 || a + T > total_tokens) {
                    bad = true;
                    T = 0;
                }
            }
            const long long nb = (T + TILE - 1) / TILE;
            long long ib = nb, ic = nb * nb;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const long long tb = __shfl_up_sync(0xffffffffu, ib, o), tc = __shfl_up_sync(0xffffffffu, ic, o);
                if (lane >= o) {
                    ib += tb;
                    ic += tc;
                }
            }
            const long long first = nblk + ib - nb, cls = ncls + ic - nb * nb;
            nblk += __shfl_sync(0xffffffffu, ib, 31);
            ncls += __shfl_sync(0xffffffffu, ic, 31);
            if (b < batch) {
                ((int32_t*)v.blk_off)[b] = (int32_t)first;
                ((uint32_t*)v.cls_off)[b] = (uint32_t)cls;
                ((int32_t*)v.seq_start)[b] = (int32_t)a;
                for (long long i = 0; i < nb && first + i < META_SMALL; ++i) {
                    s_trace[first + i] = b;
                    s_n[first + i] = (int)i;
                    s_tok0[first + i] = (int)a;
                    s_T[first + i] = (int)T;
                    s_at[first + i] = (int)(cls + i * nb);
                }
            }
        }
        bad = __any_sync(0xffffffffu, bad) || nblk > nb_cap || (unsigned long long)ncls > cls_cap;
        if (lane == 0) {
            s_nblk = bad ? 0 : (int)nblk;
            s_ncls = bad ? 0 : (int)ncls;
            if (bad) s_bad = 1;
            ((int32_t*)v.blk_off)[batch] = s_nblk;
            ((uint32_t*)v.cls_off)[batch] = (uint32_t)s_ncls;
            ((int32_t*)v.seq_start)[batch] = total_tokens;
        }
    }
    __syncthreads();
    const int nblk = s_nblk;
    for (int i = warp; i < nblk; i += META_SMALL_THREADS / 32) {
        const BlockStat st = meta_block_stat(evict_at, key_first, complement, s_n[i], s_tok0[i], s_T[i], (int32_t*)v.evict, (int32_t*)v.kfirst);
        if (lane == 0) {
            ((int32_t*)v.blk_trace)[i] = s_trace[i];
            if (has_info) ((int4*)v.info)[i] = make_int4(s_tok0[i], s_T[i], s_n[i], s_at[i]);
            ((int32_t*)v.kmin)[i] = s_kmin[i] = st.mn;
            ((int32_t*)v.kmax)[i] = s_kmax[i] = st.mx;
            ((int32_t*)v.fmin)[i] = s_fmin[i] = st.fmn;
            ((int32_t*)v.fmax)[i] = s_fmax[i] = st.fmx;
            ((int32_t*)v.col_first)[i] = s_first[i] = st.first;
            ((int32_t*)v.col_last)[i] = s_last[i] = st.last;
            s_len[ORDER_COLS][i] = max(st.last - st.first + 1, 0);
            if (st.invalid) s_bad = 1;
        }
    }
    __syncthreads();
    for (int i = warp; i < nblk; i += META_SMALL_THREADS / 32) {
        const int base = i - s_n[i];
        const int count = meta_classify_row(s_n[i], s_T[i], s_kmin + base, s_kmax + base, s_fmin + base, s_fmax + base,
                                            (uint8_t*)v.tile_class + s_at[i], (uint16_t*)v.row_list + s_at[i]);
        if (lane == 0) {
            ((int32_t*)v.row_cnt)[i] = s_len[ORDER_ROWS][i] = count;
            if (s_n[i] % 2 == 0) {
                int first, last;
                pair_range(s_first, s_last, i, (s_n[i] + 1) * TILE < s_T[i], first, last);
                s_len[ORDER_PAIRS][i] = max(last - first + 1, 0);
            }
        }
    }
    __syncthreads();
    // A quarter warp per item: its place is the number of items before it
    const bool exact = meta_exact(max_seqlen);
    const int nbins = meta_bins(max_seqlen, 1 << 30);
    for (int x = tid >> 3; x < 3 * META_SMALL; x += META_SMALL_THREADS / 8) {
        const int what = x / META_SMALL, i = x % META_SMALL, len = s_len[what][i];
        const int mine = meta_bin(max(len, 0), exact, nbins);
        int before = 0;
        if (len >= 0)
            for (int j = lane & 7; j < nblk; j += 8) {
                const int other = s_len[what][j], k = meta_bin(max(other, 0), exact, nbins);
                if (other >= 0 && (k < mine || (k == mine && j < i))) ++before;
            }
#pragma unroll
        for (int o = 1; o < 8; o <<= 1) before += __shfl_xor_sync(0xffffffffu, before, o);
        if (len >= 0 && (lane & 7) == 0) {
            int32_t* order = (int32_t*)(what == ORDER_ROWS ? v.fwd_order : what == ORDER_COLS ? v.bwd_order : v.pair_order);
            order[before] = i;
            if (what == ORDER_COLS) ((int32_t*)v.bwd_len)[before] = len;
            if (what == ORDER_PAIRS) ((int32_t*)v.pair_len)[before] = len;
        }
    }
    if (warp == 0) {
        MetaHeader h;
        int most[3], items[3];
        unsigned int sum[3];
#pragma unroll
        for (int what = 0; what < 3; ++what) {
            const int a = s_len[what][lane], b = s_len[what][lane + 32];
            most[what] = max(__reduce_max_sync(0xffffffffu, max(a, b)), 0);
            sum[what] = __reduce_add_sync(0xffffffffu, (unsigned)(max(a, 0) + max(b, 0)));
            items[what] = __popc(__ballot_sync(0xffffffffu, a >= 0)) + __popc(__ballot_sync(0xffffffffu, b >= 0));
        }
        h.magic = META_MAGIC;
        h.status = s_bad ? KVS_ERR_BAD_EVICT : KVS_OK;
        h.batch = batch;
        h.total_tokens = total_tokens;
        h.max_seqlen = max_seqlen;
        h.nblk_total = nblk;
        h.ncls_total = (uint32_t)s_ncls;
        h.general = (key_first || complement) ? 1 : 0;
        h.npair_total = items[ORDER_PAIRS];
        h.rows_done = 0;
        h.has_info = has_info;
        h.blk_most = most[ORDER_COLS];
        h.pair_most = most[ORDER_PAIRS];
        h.blk_tiles = sum[ORDER_COLS];
        h.pair_tiles = sum[ORDER_PAIRS];
        if (lane == 0) *v.hdr = h;
    }
}

// ---- compaction event log -> evict_at ---------------------------------------------------------
__global__ void evict_fill_kernel(int32_t* evict_at, int total_tokens) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < total_tokens) evict_at[i] = INT32_MAX;
}

// one CTA per event: the earliest `when` wins for every key of the span
__global__ void evict_events_kernel(const int32_t* __restrict__ events, int n_events, const int32_t* __restrict__ cu_seqlens,
                                    int batch, int32_t* evict_at) {
    const int e = blockIdx.x;
    if (e >= n_events) return;
    const int b = events[4 * e + 0], when = events[4 * e + 1];
    if (b < 0 || b >= batch) return;
    const int tok0 = cu_seqlens[b];
    const int T = cu_seqlens[b + 1] - tok0;
    const int a = max(events[4 * e + 2], 0), z = min(events[4 * e + 3], T);
    for (int j = a + threadIdx.x; j < z; j += blockDim.x) atomicMin(&evict_at[tok0 + j], when);
}

}  // namespace kvs

using namespace kvs;

extern "C" int kvs_evict_at_from_events(const int32_t* events, int n_events, const int32_t* cu_seqlens, int batch, int total_tokens,
                                        int32_t* evict_at, kvs_stream_t stream) {
    if (n_events < 0 || batch < 0 || total_tokens < 0) return KVS_ERR_INVALID_ARG;
    if (total_tokens == 0) return KVS_OK;
    if (!evict_at || !cu_seqlens || (n_events > 0 && !events)) return KVS_ERR_INVALID_ARG;
    cudaStream_t st = (cudaStream_t)stream;
    evict_fill_kernel<<<(total_tokens + 255) / 256, 256, 0, st>>>(evict_at, total_tokens);
    if (n_events > 0) evict_events_kernel<<<n_events, 256, 0, st>>>(events, n_events, cu_seqlens, batch, evict_at);
    return cudaGetLastError() == cudaSuccess ? KVS_OK : KVS_ERR_CUDA;
}

extern "C" size_t kvs_mask_meta_bytes(int batch, int total_tokens, int max_seqlen) {
    if (batch < 0 || total_tokens < 0 || max_seqlen < 0) return 0;
    return meta_layout(batch, total_tokens, max_seqlen).total;
}

namespace {
int launch_mask_meta(const int32_t* key_evict, const int32_t* key_first, int complement, const int32_t* cu_seqlens, int batch,
                     int total_tokens, int max_seqlen, void* meta_buf, size_t meta_bytes, kvs_stream_t stream) {
    if (!cu_seqlens || !meta_buf || batch < 0 || total_tokens < 0 || max_seqlen < 0) return KVS_ERR_INVALID_ARG;
    if (total_tokens > 0 && !key_evict) return KVS_ERR_INVALID_ARG;
    if (max_seqlen > total_tokens) max_seqlen = total_tokens;
    if (((uintptr_t)meta_buf & 255) != 0) return KVS_ERR_ALIGNMENT;
    if (((uintptr_t)key_evict & 3) != 0 || ((uintptr_t)key_first & 3) != 0 || ((uintptr_t)cu_seqlens & 3) != 0) return KVS_ERR_ALIGNMENT;
    if ((long long)((max_seqlen + TILE - 1) / TILE) > 65535) return KVS_ERR_UNSUPPORTED;
    const MetaLayout L = meta_layout(batch, total_tokens, max_seqlen);
    if (L.cls_cap > 0xFFFFFFF0ull) return KVS_ERR_UNSUPPORTED;
    if (meta_bytes < L.least) return KVS_ERR_WORKSPACE;
    const int has_info = meta_bytes >= L.total;
    cudaStream_t st = (cudaStream_t)stream;
    MetaView v = meta_view(meta_buf, L);
    // Two kernels -> one, us: 1 x 1024 tokens 7.8 -> 4.6, 6 of 120 to 627 6.3 -> 5.1, 20 of 50 to 380 8.8 -> 7.2, 1 x 4096 7.9 -> 6.9;
    // 20 x 380 8.7 -> 8.6, 60 x 128 8.3 -> 8.9, 2 x 4000 8.2 -> 9.3, 1 x 8192 8.5 -> 11.4: the tokens decide.
    if (L.nb_cap <= META_SMALL && total_tokens <= META_SMALL_TOKENS)
        return launch_after(meta_small_kernel, 1, META_SMALL_THREADS, 0, st, key_evict, key_first, complement, cu_seqlens, batch, total_tokens,
                            max_seqlen, v, has_info, L.nb_cap, (unsigned long long)L.cls_cap);
    const int grid = (L.nb_cap + META_WARPS - 1) / META_WARPS;
    const int rc = launch_after(meta_blocks_kernel, grid, META_THREADS, 0, st, key_evict, key_first, complement, cu_seqlens, batch, total_tokens,
                                max_seqlen, v.hdr, (int32_t*)v.blk_off, (uint32_t*)v.cls_off, (int32_t*)v.seq_start, (int32_t*)v.blk_trace,
                                has_info ? (int4*)v.info : nullptr, L.nb_cap, (unsigned long long)L.cls_cap, (int32_t*)v.kmin, (int32_t*)v.kmax, (int32_t*)v.fmin,
                                (int32_t*)v.fmax, (int32_t*)v.col_first, (int32_t*)v.col_last, (int32_t*)v.row_cnt, (int32_t*)v.evict,
                                (int32_t*)v.kfirst);
    if (rc != KVS_OK) return rc;
    return launch_after(meta_classify_kernel, grid + 2, META_THREADS, 0, st, v.hdr, v, v.blk_off, v.blk_trace, v.kmin,
                        v.kmax, v.fmin, v.fmax, v.col_first, v.col_last, (uint8_t*)v.tile_class, (uint16_t*)v.row_list, (int32_t*)v.row_cnt,
                        (int32_t*)v.fwd_order, (int32_t*)v.bwd_order, (int32_t*)v.pair_order, (int32_t*)v.bwd_len, (int32_t*)v.pair_len);
}
}  // namespace

extern "C" int kvs_mask_meta(const int32_t* evict_at, const int32_t* cu_seqlens, int batch, int total_tokens, int max_seqlen,
                             void* meta_buf, size_t meta_bytes, kvs_stream_t stream) {
    return launch_mask_meta(evict_at, nullptr, 0, cu_seqlens, batch, total_tokens, max_seqlen, meta_buf, meta_bytes, stream);
}

extern "C" int kvs_mask_meta_keys(const int32_t* key_first, const int32_t* key_evict, const int32_t* cu_seqlens, int batch,
                                  int total_tokens, int max_seqlen, void* meta_buf, size_t meta_bytes, kvs_stream_t stream) {
    if (total_tokens > 0 && !key_first) return KVS_ERR_INVALID_ARG;
    return launch_mask_meta(key_evict, key_first, 0, cu_seqlens, batch, total_tokens, max_seqlen, meta_buf, meta_bytes, stream);
}

extern "C" int kvs_mask_meta_evicted(const int32_t* key_evict, const int32_t* cu_seqlens, int batch, int total_tokens, int max_seqlen,
                                     void* meta_buf, size_t meta_bytes, kvs_stream_t stream) {
    return launch_mask_meta(key_evict, nullptr, 1, cu_seqlens, batch, total_tokens, max_seqlen, meta_buf, meta_bytes, stream);
}

// ---- key re-ordering for token-level eviction ------------------------------------------------------
namespace kvs {
constexpr int REORDER_MAX_WINDOW = 4096;
constexpr int REORDER_COUNTED = 512;
// One CTA per (window, trace): the window's keys sorted by (eviction step, index).  Up to REORDER_COUNTED keys a key's place is
// counted, by 1024 / n threads; above, the counting grows with the square of n and a bitonic network in shared memory takes
// over, whose steps are a synchronisation each (step of 2 traces of 300 tokens in sorted slots, 28 heads on 4: 74.6 -> 72.1 us).
__global__ void __launch_bounds__(1024)
reorder_sort_kernel(const int32_t* __restrict__ evict_at, const int32_t* __restrict__ cu_seqlens, int window, int32_t* perm,
                    int32_t* key_first, int32_t* key_evict) {
    __shared__ unsigned long long keys[REORDER_MAX_WINDOW];
    pdl_wait();
    const int b = blockIdx.y;
    const int tok0 = cu_seqlens[b];
    const int T = cu_seqlens[b + 1] - tok0;
    const int w0 = blockIdx.x * window;
    if (w0 >= T) return;
    const int n = min(window, T - w0);
    int cap = 1;
    while (cap < n) cap <<= 1;
    for (int i = threadIdx.x; i < cap; i += blockDim.x)
        keys[i] = (i < n) ? (((unsigned long long)(uint32_t)evict_at[tok0 + w0 + i] << 32) | (uint32_t)i) : ~0ull;
    __syncthreads();
    if (cap <= REORDER_COUNTED) {
        const int per = min((int)blockDim.x / cap, 32);        // threads of a warp for each key
        const int i = threadIdx.x / per;
        const unsigned long long mine = i < n ? keys[i] : 0;
        int before = 0;
        if (i < n)
            for (int j = threadIdx.x % per; j < n; j += per) before += keys[j] < mine;
        for (int o = 1; o < per; o <<= 1) before += __shfl_xor_sync(0xffffffffu, before, o);
        if (i < n && threadIdx.x % per == 0) {
            const int at = tok0 + w0 + before;
            perm[at] = tok0 + w0 + i;
            key_first[at] = w0 + i;
            key_evict[at] = (int32_t)(mine >> 32);
        }
        return;
    }
    for (int k = 2; k <= cap; k <<= 1) {
        for (int j = k >> 1; j > 0; j >>= 1) {
            for (int i = threadIdx.x; i < cap; i += blockDim.x) {
                const int l = i ^ j;
                if (l > i) {
                    const unsigned long long a = keys[i], c = keys[l];
                    const bool up = (i & k) == 0;
                    if ((a > c) == up) {
                        keys[i] = c;
                        keys[l] = a;
                    }
                }
            }
            __syncthreads();
        }
    }
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        const int src = w0 + (int)(uint32_t)keys[i];           // trace-local index of the key that lands in slot w0 + i
        perm[tok0 + w0 + i] = tok0 + src;
        key_first[tok0 + w0 + i] = src;
        key_evict[tok0 + w0 + i] = (int32_t)(keys[i] >> 32);
    }
}

// dst row r = src row perm[r] (inverse == 0) or dst row perm[r] = src row r (inverse != 0); 16 bytes per lane
__global__ void permute_rows_kernel(const uint4* __restrict__ src, const int32_t* __restrict__ perm, uint4* __restrict__ dst,
                                    long long n_rows, int row_vec, int inverse) {
    pdl_wait();
    const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const long long r = idx / row_vec;
    const int c = (int)(idx % row_vec);
    if (r >= n_rows) return;
    const long long p = perm[r];
    if (inverse) dst[p * row_vec + c] = src[r * row_vec + c];
    else dst[r * row_vec + c] = src[p * row_vec + c];
}
}  // namespace kvs

extern "C" int kvs_reorder_keys(const int32_t* evict_at, const int32_t* cu_seqlens, int batch, int total_tokens, int max_seqlen,
                                int window, int32_t* perm, int32_t* key_first, int32_t* key_evict, kvs_stream_t stream) {
    if (batch < 0 || total_tokens < 0 || max_seqlen < 0) return KVS_ERR_INVALID_ARG;
    if (window < 1 || window > REORDER_MAX_WINDOW) return KVS_ERR_UNSUPPORTED;
    if (total_tokens == 0 || batch == 0) return KVS_OK;
    if (!evict_at || !cu_seqlens || !perm || !key_first || !key_evict) return KVS_ERR_INVALID_ARG;
    if (batch > 65535) return KVS_ERR_UNSUPPORTED;
    if (max_seqlen > total_tokens) max_seqlen = total_tokens;
    const int nwin = (max_seqlen + window - 1) / window;
    dim3 grid(nwin > 0 ? nwin : 1, batch, 1);
    return launch_after(reorder_sort_kernel, grid, 1024, 0, (cudaStream_t)stream, evict_at, cu_seqlens, window, perm, key_first, key_evict);
}

extern "C" int kvs_permute_rows(const void* src, const int32_t* perm, void* dst, long long n_rows, long long row_bytes, int inverse,
                                kvs_stream_t stream) {
    if (n_rows < 0 || row_bytes <= 0 || row_bytes % 16 != 0 || row_bytes / 16 > 0x7fffffffLL) return KVS_ERR_INVALID_ARG;
    if (n_rows == 0) return KVS_OK;
    if (!src || !perm || !dst || src == dst) return KVS_ERR_INVALID_ARG;
    if ((((uintptr_t)src | (uintptr_t)dst) & 15) != 0 || ((uintptr_t)perm & 3) != 0) return KVS_ERR_ALIGNMENT;
    const int row_vec = (int)(row_bytes / 16);
    const long long total = n_rows * row_vec;
    const long long blocks = (total + 255) / 256;
    if (blocks > 0x7fffffffLL) return KVS_ERR_UNSUPPORTED;
    return launch_after(permute_rows_kernel, (unsigned)blocks, 256, 0, (cudaStream_t)stream, (const uint4*)src, perm, (uint4*)dst, n_rows, row_vec,
                        inverse);
}

extern "C" int kvs_mask_meta_export(const void* meta_buf, int batch, const int32_t* cu_seqlens_host, int total_tokens,
                                    int max_seqlen, uint8_t* tile_class_host, int32_t* kmin_host, int32_t* kmax_host,
                                    kvs_stream_t stream) {
    if (!meta_buf || !cu_seqlens_host || batch < 0) return KVS_ERR_INVALID_ARG;
    if (max_seqlen > total_tokens) max_seqlen = total_tokens;
    const MetaLayout L = meta_layout(batch, total_tokens, max_seqlen);
    cudaStream_t st = (cudaStream_t)stream;
    size_t nblk = 0, ncls = 0;
    for (int b = 0; b < batch; ++b) {
        long long T = (long long)cu_seqlens_host[b + 1] - cu_seqlens_host[b];
        if (T < 0 || T > max_seqlen) return KVS_ERR_INVALID_ARG;
        size_t nb = (size_t)((T + TILE - 1) / TILE);
        nblk += nb;
        ncls += nb * nb;
    }
    if (nblk > (size_t)L.nb_cap || ncls > L.cls_cap) return KVS_ERR_INVALID_ARG;
    MetaHeader h;
    const char* p = (const char*)meta_buf;
    if (cudaMemcpyAsync(&h, p, sizeof(h), cudaMemcpyDeviceToHost, st) != cudaSuccess) return KVS_ERR_CUDA;
    if (tile_class_host && ncls)
        if (cudaMemcpyAsync(tile_class_host, p + L.tile_class, ncls, cudaMemcpyDeviceToHost, st) != cudaSuccess) return KVS_ERR_CUDA;
    if (kmin_host && nblk)
        if (cudaMemcpyAsync(kmin_host, p + L.kmin, nblk * 4, cudaMemcpyDeviceToHost, st) != cudaSuccess) return KVS_ERR_CUDA;
    if (kmax_host && nblk)
        if (cudaMemcpyAsync(kmax_host, p + L.kmax, nblk * 4, cudaMemcpyDeviceToHost, st) != cudaSuccess) return KVS_ERR_CUDA;
    if (cudaStreamSynchronize(st) != cudaSuccess) return KVS_ERR_CUDA;
    if (h.magic != META_MAGIC || h.batch != batch || h.total_tokens != total_tokens || h.max_seqlen != max_seqlen) return KVS_ERR_BAD_META;
    if (h.status != KVS_OK) return h.status;
    if ((size_t)h.nblk_total != nblk || (size_t)h.ncls_total != ncls) return KVS_ERR_BAD_META;
    return KVS_OK;
}
