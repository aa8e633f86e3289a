// Backward: dQ, dK, dV of eviction-masked causal attention.
//
//   pre-pass   D_i = dout_i . out_i                         (one warp per (token, head))
//   main       one CTA per unit of (key block n, KV head g), longest first; K and V tiles stay in
//              shared memory; the CTA loops over the G query heads of the group and over the
//              contiguous range of query blocks n .. col_last[n] that can see the key block, or over
//              a part of that list (see BwdUnit and bwd_plan; the comment above bwd_kernel for the
//              pipeline).  Long traces at head_dim 128: CTA pairs, kvs_bwd_pair.cu
//   post-pass  fp32 dQ accumulator -> bf16 (bf16 gradients only)
#include "kvs_bwd.cuh"
#include <cstring>

namespace kvs {

constexpr int BWD_SMS = 148;
// A batch whose Q, dO and fp32 dQ are larger than this is listed by trace (see bwd_plan): sorted by length throughout, a trace's
// key blocks run far apart and its tiles come from memory again for each (96 traces of 60 to 900 tokens, 16 heads on 2: 2.7 GB
// moved at 5.7 TB/s, 1.9 GB by trace).  Main kernel, by length -> by trace, us, 32 heads on 8: 200 traces of 300 tokens 1219 ->
// 977, 96 of 60 to 900 (16 on 2) 480 -> 434, 60 of 100 to 2000 (28 on 4) 1409 -> 1302, 12 of 1500 to 12000 5216 -> 5126, 8 of
// 8000 4771 -> 4712, 9 of 14000 with nothing evicted (16 on 2) 18.1 -> 17.6 ms.  Of fewer traces than eight an eighth is not to
// be had for the end (3 of 14000: 11.5 -> 11.8 ms; 4 of 20000 without groups 6.9 -> 7.0 ms).
constexpr long long BWD_L2_BYTES = 96ll << 20;
constexpr int BWD_MANY_TRACES = 8, BWD_MOST_LATE = 6;
// Tiles left of a unit when the CTA asks for the next one.  Main kernel, us, with 1, 2, 3, 5, 8 (32 heads on 8): 200 traces of 300 tokens
// 953, 945, 945, 947, 970; 20 of 500 to 2000 552, 548, 548, 548, 550; 123 of 270, 16 on 4, head_dim 64 199.7, 197.6, 197.6, 197.6,
// 201.7: earlier takes units from CTAs that are free before, with 1 they are waited for.
constexpr uint32_t BWD_LATE = 3;
// Tiles of the shortest unit: 2 (1 x 1024 tokens, 4 heads, head_dim 64: main kernel 21.5 us with 4, 19.5 with 2), but as many as make
// four units of the longest item, up to 4: an item's last unit reads the slots of all, 1.6 us each at head_dim 128 (16 heads on 2,
// 1 x 600 tokens 35.8 us with 4, 44.0 with 2; 1 x 1000 43.0, 50.1).  The shorter the unit, the more slots a small batch asks for; a
// buffer that was sized for units of four is accepted and keeps to them.
constexpr int BWD_MIN_UNIT = 2, BWD_MIN_UNIT_LESS = 4;
constexpr int BWD_MAX_SLOTS = 2 * BWD_SMS;  // slots of one CTA each for the dK and dV of cut items, over all KV heads

struct BwdWsLayout {
    size_t dvec, dq_acc, base;              // base: what is needed without cutting items
    size_t plan, units, arrived, part;      // offsets from there
    size_t total;
    int slots, unit_cap;                    // slots of one CTA; entries of the unit list
};

inline BwdWsLayout bwd_ws_layout(int total_tokens, int Hq, int head_dim, int grad_dtype, int min_unit = BWD_MIN_UNIT) {
    BwdWsLayout L;
    size_t o = align_up(sizeof(WsHeader), 256);
    L.dvec = o;
    o = align_up(o + sizeof(float) * (size_t)total_tokens * Hq, 256);
    L.dq_acc = o;
    if (grad_dtype == KVS_GRAD_BF16) o = align_up(o + sizeof(float) * (size_t)total_tokens * Hq * head_dim, 256);
    L.base = o;
    // An item of t tiles cut into units of at least min_unit tiles has at most 2 t / min_unit of them, and all items
    // of a batch have at most Hq nb (nb + 1) / 2 tiles (one trace, nothing evicted).
    const long long nb = ((long long)total_tokens + TILE - 1) / TILE;
    const long long most = Hq * nb * (nb + 1) / min_unit;
    L.slots = (int)(most < BWD_MAX_SLOTS ? most : BWD_MAX_SLOTS);
    // key blocks of a batch: short traces have more than total / 128; beyond 4096 more the items are not cut
    L.unit_cap = (int)((total_tokens < nb + 4096 ? total_tokens : nb + 4096) + L.slots);
    o = 0;
    L.plan = o;    o = align_up(o + sizeof(BwdPlan), 256);
    L.units = o;   o = align_up(o + sizeof(BwdUnit) * (size_t)L.unit_cap, 256);
    L.arrived = o; o = align_up(o + sizeof(int32_t) * 2 * (size_t)L.slots, 256);
    L.part = o;    o = align_up(o + sizeof(float) * 2 * TILE * (size_t)head_dim * L.slots, 256);
    L.total = L.base + o;
    return L;
}

// ---- plan ---------------------------------------------------------------------------------------
struct BwdPlanArgs {
    MetaView all, mv;                       // the batch the cut is chosen for; the (part of the) batch whose units are listed
    int all_batch, all_tokens, all_maxlen, batch, tokens, maxlen;
    int all_cap, cap;                       // key blocks that the two have room for
    int by_trace;                           // the batch does not fit in L2: see BWD_L2_BYTES
    int pairs;                              // items are pairs of key blocks
    int G, all_Hkv, Hkv;
    int all_slots, slots;                   // slots there are, of an item's CTAs, over all KV heads
    int min_unit;                           // tiles of the shortest unit
    BwdPlan* plan;                          // nullptr: none is wanted
    BwdUnit* units;
    int32_t* arrived;
    int arrived_n;
};

// One CTA of 256 threads, beside the pre-pass.  Chooses the longest unit L among eight candidates (fractions of an SM's, or
// pair's, share of all tiles, and "no cut") by an estimate of the makespan in tiles, then lists the units.  An item of t
// tiles becomes ceil(t / L) units of equal length.  The estimate: a unit costs BWD_UNIT_COST tiles beside its own (loads
// before the first product, the pipeline's first and last tile, the stores), a unit of a cut item BWD_CUT_COST more (slot
// written and read again); no unit is longer than the makespan; where the longest is over one and a half times what a head
// has for an SM, those above that start first, over all heads, so what is left over at the end is half of it at most (always
// doing so costs L2 hits, 2 x 65536 tokens 41.4 -> 42.6 ms, but not on traces of at most 16 tiles: 96 of 60 to 900
// 472 -> 454 us); and up to three waves take that many average units.
// Main kernel, whole items -> cut, us: 1 trace of 1000 tokens with 16 heads on 2 154 -> 42; 4000 with 32 on 8 355 -> 180; 16000,
// head_dim 64 1199 -> 748; 20 of 100 to 2000, head_dim 64 229 -> 161; 32768 with 28 on 4 (pairs) 5500 -> 4400.  Where nothing is
// cut, the list and the registers of the slots cost 1 % at head_dim 64 and 9 % at 128 (96 of 60 to 900: 316 -> 319, 447 -> 494;
// before units were chained).  BWD_UNIT_COST of 2, 4, 6 with chained units, us: 96 of 60 to 900 401, 401, 427; 20 of 500 to 2000, 1 x 1000
// (16 on 2), 1 x 4000, 20 x 550 at head_dim 64 the same.
constexpr float BWD_UNIT_COST = 4.f, BWD_CUT_COST = 3.f;
__device__ void bwd_plan(const BwdPlanArgs& a) {
    constexpr int NC = 8;
    __shared__ int s_units[NC], s_cut[NC], s_longest[NC], s_len;
    __shared__ float s_heavy_from;
    __shared__ int s_scan[2][8], s_run[2], s_heavy;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const MetaHeader* all = a.all.hdr;
    const MetaHeader* part = a.mv.hdr;
    const int32_t* all_len = a.pairs ? a.all.pair_len : a.all.bwd_len;
    const int32_t* len = a.pairs ? a.mv.pair_len : a.mv.bwd_len;
    const int32_t* order = a.pairs ? a.mv.pair_order : a.mv.bwd_order;
    if (!meta_matches(all, a.all_batch, a.all_tokens, a.all_maxlen) || !meta_matches(part, a.batch, a.tokens, a.maxlen)) {
        if (tid == 0) a.plan->n_units = a.plan->n_heavy = a.plan->n_apart = 0;
        return;
    }
    // this thread's first item, on its way while the candidates are set up (the arrays have room for `cap` entries, with or
    // without a value yet)
    const int all_len0 = tid < a.all_cap ? all_len[tid] : 0;
    const int len0 = tid < a.cap ? len[tid] : 0, order0 = tid < a.cap ? order[tid] : 0;
    const int n_all = a.pairs ? all->npair_total : all->nblk_total, n = a.pairs ? part->npair_total : part->nblk_total;
    const int most = max(a.G * (a.pairs ? all->pair_most : all->blk_most), 1);
    const int sms = a.pairs ? BWD_SMS / 2 : BWD_SMS;
    const float share = (float)(a.pairs ? all->pair_tiles : all->blk_tiles) * a.G * a.all_Hkv / sms;          // tiles per SM or pair
    for (int i = tid; i < a.arrived_n; i += 256) a.arrived[i] = 0;
    const int min_unit = max(a.min_unit, min(most / 4, BWD_MIN_UNIT_LESS));
    int cand[NC];
    const float frac[NC] = {0.25f, 0.5f, 0.75f, 1.0f, 1.25f, 1.6f, 2.2f, 0.f};
#pragma unroll
    for (int k = 0; k < NC; ++k) {
        const float l = fmaxf(ceilf(share * frac[k]), (float)max(min_unit, (most + BWD_MAX_CUT - 1) / BWD_MAX_CUT));
        cand[k] = (k == NC - 1 || l > (float)most) ? most : (int)l;
    }
    // What a warp makes of the candidates' numbers (lane k: those of candidate k): the longest unit, and from which length on
    // units of all heads start first.
    auto choose = [&](int n_units, int n_cut, int n_longest, int& length, float& heavy) {
        const int k = lane & (NC - 1);
        const float units = (float)n_units * a.all_Hkv, longest = (float)n_longest, head = share / a.all_Hkv;
        const float waves = ceilf(units / sms);
        float est = longest + BWD_UNIT_COST;
        if (waves > 1.f) {
            est = share + (BWD_UNIT_COST * units + BWD_CUT_COST * n_cut * a.all_Hkv) / sms + 0.5f * fminf(longest, head);
            est = fmaxf(est, longest + BWD_UNIT_COST);
            if (waves <= 3.f) est = fmaxf(est, waves * (share * sms / units + BWD_UNIT_COST));
        }
        if (n_cut > 0) est += BWD_CUT_COST;
        if (k < NC - 1 && (long long)n_cut * a.all_Hkv > a.all_slots) est = INFINITY;          // "no cut" always fits
        float best = est;
        int at = k;
#pragma unroll
        for (int o = 1; o < NC; o <<= 1) {
            const float e = __shfl_xor_sync(0xffffffffu, best, o);
            const int x = __shfl_xor_sync(0xffffffffu, at, o);
            if (e < best || (e == best && x > at)) {
                best = e;
                at = x;
            }
        }
        length = cand[0];
#pragma unroll
        for (int c = 1; c < NC; ++c) length = c == at ? cand[c] : length;
        heavy = part->max_seqlen <= 16 * TILE ? 0.125f * share : __shfl_sync(0xffffffffu, longest, at) > 1.5f * head ? head : INFINITY;
    };
    auto unit_of = [&](int block, int t, int c, int i, int slot0) {      // the i-th of an item's c units
        return BwdUnit{block, (int)((long long)t * i / c), (int)((long long)t * (i + 1) / c), c > 1 ? (slot0 << 18 | i << 9 | c) : 0};
    };
    if (n_all <= 32 && part == all) {       // a few items: one warp, an item a lane, no synchronisation of the CTA
        if (warp != 0) return;
        const int t = lane < n_all ? a.G * all_len0 : 0;
        int my_units = 0, my_cut = 0, my_longest = 0;
#pragma unroll
        for (int k = 0; k < NC; ++k) {
            const int c = lane >= n_all ? 0 : t > cand[k] ? (t + cand[k] - 1) / cand[k] : 1;
            const int units = __reduce_add_sync(0xffffffffu, c), cut = __reduce_add_sync(0xffffffffu, c > 1 ? c : 0);
            const int longest = __reduce_max_sync(0xffffffffu, c > 1 ? (t + c - 1) / c : t);
            if ((lane & (NC - 1)) == k) {
                my_units = units;
                my_cut = cut;
                my_longest = longest;
            }
        }
        int longest;
        float heavy_from;
        choose(my_units, my_cut, my_longest, longest, heavy_from);
        const int c = lane < n_all ? max((t + longest - 1) / longest, 1) : 0;
        int iu = c, is = c > 1 ? c : 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int u = __shfl_up_sync(0xffffffffu, iu, o), s = __shfl_up_sync(0xffffffffu, is, o);
            if (lane >= o) {
                iu += u;
                is += s;
            }
        }
        for (int i = 0; i < c; ++i) a.units[iu - c + i] = unit_of(order0, t, c, i, is - (c > 1 ? c : 0));
        const int heavy = __reduce_add_sync(0xffffffffu, (float)t > heavy_from * c ? c : 0);
        if (lane == 31) {
            a.plan->n_units = iu;
            a.plan->slots = is;
            a.plan->n_heavy = heavy;
            a.plan->n_apart = iu - heavy;
        }
        return;
    }
    if (tid < NC) s_units[tid] = s_cut[tid] = s_longest[tid] = 0;
    if (tid == 0) s_run[0] = s_run[1] = s_heavy = 0;
    __syncthreads();
    {
        int units[NC], cut[NC], longest[NC];
#pragma unroll
        for (int k = 0; k < NC; ++k) units[k] = cut[k] = longest[k] = 0;
        for (int x = tid; x < n_all; x += 256) {
            const int t = a.G * (x < 256 ? all_len0 : all_len[x]);
#pragma unroll
            for (int k = 0; k < NC; ++k) {
                const int c = t > cand[k] ? (t + cand[k] - 1) / cand[k] : 1;
                units[k] += c;
                if (c > 1) cut[k] += c;
                longest[k] = max(longest[k], c > 1 ? (t + c - 1) / c : t);
            }
        }
#pragma unroll
        for (int k = 0; k < NC; ++k) {
            units[k] = __reduce_add_sync(0xffffffffu, units[k]);
            cut[k] = __reduce_add_sync(0xffffffffu, cut[k]);
            longest[k] = __reduce_max_sync(0xffffffffu, longest[k]);
            if (lane == 0 && units[k] > 0) {
                atomicAdd(&s_units[k], units[k]);
                atomicAdd(&s_cut[k], cut[k]);
                atomicMax(&s_longest[k], longest[k]);
            }
        }
    }
    __syncthreads();
    if (warp == 0) {                        // lane k: candidate k
        const int k = lane & (NC - 1);
        int length;
        float heavy;
        choose(s_units[k], s_cut[k], s_longest[k], length, heavy);
        if (lane == 0) {
            s_len = length;
            s_heavy_from = heavy;
        }
    }
    __syncthreads();
    int longest = s_len;
    const float heavy_from = s_heavy_from;
    if (part != all) {                      // a part of the batch has no more cut units than the whole, but its slots are counted too
        if (tid == 0) s_cut[0] = 0;
        __syncthreads();
        int cut = 0;
        for (int x = tid; x < n; x += 256) {
            const int c = (a.G * len[x] + longest - 1) / longest;
            if (c > 1) cut += c;
        }
        if (cut) atomicAdd(&s_cut[0], cut);
        __syncthreads();
        if ((long long)s_cut[0] * a.Hkv > a.slots) longest = most;
    }
    // Where the traces do not fit in L2 together, all but `late` eighths of them come in the order of the batch, a head's units
    // and then the next head's: key blocks of a trace run together and share its Q and dO tiles and the lines of its dQ.  The
    // others come last, longest items first and of all heads together: as much work as it takes for all SMs to end together, where
    // the traces' lengths have nothing to do with their places in the batch (eighths of the traces, not of the tiles).
    const float part_share = (float)(a.pairs ? part->pair_tiles : part->blk_tiles) * a.G * a.Hkv / sms;
    const int late = a.by_trace ? (int)ceilf(8.f * (float)min(longest, most) / fmaxf(part_share, 1.f)) : 8;
    const bool by_trace = late <= BWD_MOST_LATE;
    auto is_late = [&](int block) { return ((a.mv.blk_trace[block] * late) & 7) < late; };        // evenly spread over the batch
    // List the units, the items' order kept (by trace: a pass for either part): prefix sums of the items' units and of their slots
    int n_apart = 0;
    for (int pass = by_trace ? 0 : 1; pass < 2; ++pass) {
        for (int x0 = 0; x0 < n; x0 += 256) {
            const int x = x0 + tid;
            int t = 0, block = 0;
            bool listed = x < n;
            if (listed && pass == 0) {
                block = x;
                t = max(a.mv.col_last[x] - a.mv.col_first[x] + 1, 0);
                listed = !is_late(x);
            } else if (listed) {
                t = x0 ? len[x] : len0;
                block = x0 ? order[x] : order0;
                listed = !by_trace || is_late(block);
            }
            t *= a.G;
            const int c = listed ? max((t + longest - 1) / longest, 1) : 0;
            int iu = c, is = c > 1 ? c : 0;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int u = __shfl_up_sync(0xffffffffu, iu, o), s = __shfl_up_sync(0xffffffffu, is, o);
                if (lane >= o) {
                    iu += u;
                    is += s;
                }
            }
            if (lane == 31) {
                s_scan[0][warp] = iu;
                s_scan[1][warp] = is;
            }
            __syncthreads();
            int bu = s_run[0], bs = s_run[1];
            for (int w = 0; w < warp; ++w) {
                bu += s_scan[0][w];
                bs += s_scan[1][w];
            }
            const int u0 = bu + iu - c, slot0 = bs + is - (c > 1 ? c : 0);
            if (c > 0 && (float)t > heavy_from * c) atomicAdd(&s_heavy, c);
            for (int i = 0; i < c; ++i)
                a.units[u0 + i] = unit_of(block, t, c, i, slot0);
            __syncthreads();
            if (tid == 255) {
                s_run[0] = bu + iu;
                s_run[1] = bs + is;
            }
            __syncthreads();
        }
        if (pass == 0) n_apart = s_run[0];
    }
    if (tid == 0) {
        a.plan->n_units = s_run[0];
        a.plan->slots = s_run[1];
        a.plan->n_heavy = by_trace ? 0 : s_heavy;
        a.plan->n_apart = by_trace ? n_apart : s_run[0] - s_heavy;
    }
}

// ---- pre-pass ---------------------------------------------------------------------------------
// D[h][tok] = sum_c dout[tok][h][c] * out[tok][h][c], and the fp32 dQ accumulator cleared in the same pass (it is
// the destination of the main kernel's reduce-adds).  16 bytes per lane and tensor, D/8 lanes per row, DOT_ROWS rows in
// flight per lane: the pass streams 2 x 2 B in and 4 B out per element and is bound by HBM.
constexpr int DOT_ROWS = 4;
template <int D>
__global__ void __launch_bounds__(256)
bwd_dot_kernel(const __nv_bfloat16* __restrict__ dout, const __nv_bfloat16* __restrict__ out,
               float* __restrict__ dvec, float* __restrict__ dq_acc, long long dq_ts, int total_tokens, int Hq, WsHeader* hdr,
               const __grid_constant__ BwdPlanArgs plan) {
    pdl_wait();
    if (blockIdx.x == 0) {                      // the first CTA has no rows
        if (threadIdx.x == 0) {
            hdr->magic = WS_MAGIC;
            hdr->status = KVS_OK;
        }
        if (plan.plan) bwd_plan(plan);
        return;
    }
    constexpr int LPR = D / 8;                  // lanes per row: 16 or 8
    constexpr int RPW = 32 / LPR;               // rows per warp and step
    const long long rows = (long long)total_tokens * Hq;
    const long long gw = ((long long)(blockIdx.x - 1) * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    const int sub = lane / LPR, c = lane % LPR;
    const long long row0 = gw * (RPW * DOT_ROWS) + sub;
    uint4 x[DOT_ROWS], y[DOT_ROWS];
#pragma unroll
    for (int r = 0; r < DOT_ROWS; ++r) {
        const long long row = row0 + (long long)r * RPW;
        if (row < rows) {
            x[r] = *reinterpret_cast<const uint4*>(dout + (size_t)row * D + c * 8);
            y[r] = *reinterpret_cast<const uint4*>(out + (size_t)row * D + c * 8);
        } else {
            x[r] = y[r] = make_uint4(0, 0, 0, 0);
        }
    }
    const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int r = 0; r < DOT_ROWS; ++r) {
        const long long row = row0 + (long long)r * RPW;
        const uint32_t xa[4] = {x[r].x, x[r].y, x[r].z, x[r].w}, ya[4] = {y[r].x, y[r].y, y[r].z, y[r].w};
        float acc = 0.f;
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            acc = fmaf(__uint_as_float(xa[e] << 16), __uint_as_float(ya[e] << 16), acc);
            acc = fmaf(__uint_as_float(xa[e] & 0xffff0000u), __uint_as_float(ya[e] & 0xffff0000u), acc);
        }
#pragma unroll
        for (int o = LPR / 2; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
        if (row < rows) {
            if (dq_acc) {
                float4* z = reinterpret_cast<float4*>(dq_acc + (size_t)(row / Hq) * dq_ts + (size_t)(row % Hq) * D + c * 8);
                z[0] = zero;
                z[1] = zero;
            }
            if (c == 0) dvec[(size_t)(row % Hq) * total_tokens + (row / Hq)] = acc;
        }
    }
}

// ---- post-pass --------------------------------------------------------------------------------
// acc: contiguous [tokens, row_elems]; dq: rows of row_elems elements, dq_ts elements apart
__global__ void bwd_cast_kernel(const float* __restrict__ acc, __nv_bfloat16* __restrict__ dq, size_t n4, int row_elems, long long dq_ts) {
    pdl_wait();
    const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n4) return;
    const float4 x = reinterpret_cast<const float4*>(acc)[i];
    uint2 w;
    w.x = pack_bf16(x.x, x.y);
    w.y = pack_bf16(x.z, x.w);
    const size_t e = i * 4;
    *reinterpret_cast<uint2*>(dq + (e / row_elems) * (size_t)dq_ts + e % row_elems) = w;
}

// ---- main -------------------------------------------------------------------------------------
// Warp-specialised, 16 warps in four warp groups:
//   warps 0-7   compute: one key row per thread, 64 of the 128 query columns each (P^T, dS^T)
//   warps 8-11  drain:   dQ tile, tensor memory -> registers -> swizzled shared memory -> TMA
//               reduce-add into the fp32 accumulator (global `red` instructions are processed at
//               about one thread per clock per SM, which alone would exceed the MMA time of a tile)
//   warp 12     producer (TMA for K, V, Q, dO; plain loads for lse and D)
//   warp 13     MMA issuer;   warp 14  list of units;   warp 15 idle (it only completes the warp group)
// Registers are re-balanced per warp group with setmaxnreg (compute 144, drain 144, the rest 80).
//
// Tensor memory (512 columns):  [0,128) S^T fp32, then P^T bf16 in [0,32) and [64,96)
//                               [128,256) dP^T fp32, then dQ fp32
//                               [256,256+D) dV     [384,384+D) dK
// Per iteration j (one (head, query block) tile) the tensor pipe runs, in this order,
//     dP^T(j) = V dO^T,  dV(j) += P^T dO,  S^T(j+1) = K Q^T,  dQ(j) = dS K,  dK(j) += dS^T Q
// while the compute warps run  dS(j), P(j+1)  and the drain warps empty dQ(j).  The softmax scale
// is folded into dS (dS = P (scale dP - scale D)), so dK and dQ leave the tensor core scaled.
// A CTA goes on with units of CTAs that have not started (cluster launch control).  Barriers run on across units, so that the
// next unit's K, V, Q and dO arrive and its first products run while the compute warps write out the last one's dK and dV and
// the last dQ is added; only what the last products read is waited for.  With a CTA per unit the launch, the chain of metadata
// loads, the set-up, the first loads, the write-out and the wait for the last adds stood beside the tiles: 12 of 138 us a unit on
// 12 traces of 1500 to 12000 tokens, 13 of 56 on 96 of 60 to 900.  Main kernel, a CTA per unit -> chained, us: 123 traces of 199
// to 350, 16 heads on 4, head_dim 64 211 -> 189; 40 of 100 to 1000, 4 on 4, head_dim 64 60.7 -> 51.3; 20 of 500 to 2000, 32 on 8
// 645 -> 610; 3 of 14000 with nothing evicted 12350 -> 11880.
// Rows of a dQ tile past the end of a trace are exactly zero (their P is zero), so the reduce-add
// of a whole 128-row box is harmless where it overlaps the next trace.
template <int D>
struct BwdSmem {
    static constexpr int TB = TILE * D * 2;
    static constexpr int STG_BYTES = TILE * 128;     // 128 rows x 32 fp32
    static constexpr int OFF_K = 0;
    static constexpr int OFF_V = TB;
    static constexpr int OFF_Q = 2 * TB;             // 2 stages
    static constexpr int OFF_DO = 4 * TB;            // 1 stage
    static constexpr int OFF_DS = 5 * TB;            // 128 keys x 128 queries bf16
    static constexpr int OFF_STG = OFF_DS + TILE * TILE * 2;   // 2 staging buffers for dQ chunks
    static constexpr int OFF_LSE = OFF_STG + 2 * STG_BYTES;    // 2 stages x 128 fp32: -lse * log2 e
    static constexpr int OFF_DVEC = OFF_LSE + 2 * TILE * 4;    // 2 stages x 128 fp32: -D * scale
    static constexpr int OFF_BAR = OFF_DVEC + 2 * TILE * 4;
    static constexpr int OFF_MISC = OFF_BAR + 22 * 8;          // tmem base, abort flag
    static constexpr int OFF_ASK = OFF_MISC + 16;              // the answer of the launch control
    static constexpr int OFF_WORK = OFF_ASK + 16;              // 2 slots
    static constexpr int TOTAL = OFF_WORK + 2 * (int)sizeof(BwdWork);
    static constexpr int MAX_DYN = 232448;                     // 227 KB
    static constexpr int DYN_BYTES = (TOTAL + 1024 > MAX_DYN) ? MAX_DYN : TOTAL + 1024;
};

template <int D>
__global__ void __launch_bounds__(BWD_THREADS, 1)
bwd_kernel(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_k,
           const __grid_constant__ CUtensorMap tm_v, const __grid_constant__ CUtensorMap tm_do,
           const __grid_constant__ CUtensorMap tm_dq, const __grid_constant__ MetaView mv,
           const __grid_constant__ BwdParams p) {
    using L = BwdSmem<D>;
    constexpr int NBOX = D / 64;
    constexpr int BOX_BYTES = TILE * 128;
    constexpr uint32_t TMEM_COLS = 512;
    constexpr uint32_t IDESC_ST = make_idesc(TILE, 0, 0);    // K-major x K-major, N = 128 queries
    constexpr uint32_t IDESC_KV = make_idesc(D, 0, 1);       // A from tensor memory, B MN-major, N = D
    constexpr uint32_t IDESC_DQ = make_idesc(D, 1, 1);       // A, B MN-major, N = D
    constexpr int HALF_D = D / 2;

    extern __shared__ uint8_t smem_raw[];

    const int tid = threadIdx.x;
    const int warp = tid >> 5;
    const int lane = tid & 31;
    pdl_wait();
    // meta_buf must be the one kvs_mask_meta wrote for these sizes: every index below comes out of it
    if (!meta_matches(mv.hdr, p.batch, p.total_tokens, p.max_seqlen)) {
        if (tid == 0 && blockIdx.x == 0) set_status(p.status, KVS_ERR_BAD_META);
        return;
    }
    const int n_items = mv.hdr->nblk_total;
    if (!bwd_has_unit(p, n_items, blockIdx.x)) return;
    int32_t* status = p.status;

    const uint32_t sraw = smem_u32(smem_raw);
    const uint32_t sbase = (sraw + 1023u) & ~1023u;
    if ((sbase - sraw) + L::TOTAL > (uint32_t)L::DYN_BYTES) {      // shared window not aligned as expected
        if (tid == 0) set_status(status, KVS_ERR_CUDA);
        return;
    }
    uint8_t* sgen = smem_raw + (sbase - sraw);
    const uint32_t sK = sbase + L::OFF_K, sV = sbase + L::OFF_V, sQ = sbase + L::OFF_Q, sDO = sbase + L::OFF_DO,
                   sDS = sbase + L::OFF_DS, sSTG = sbase + L::OFF_STG;
    uint32_t* s_tmem_base = reinterpret_cast<uint32_t*>(sgen + L::OFF_MISC);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(sgen + L::OFF_MISC + 4);
    const uint32_t bars = sbase + L::OFF_BAR;
    const uint32_t bar_kv = bars;
    auto bar_qfull = [&](int s) { return bars + 8 * (1 + s); };
    auto bar_ldfull = [&](int s) { return bars + 8 * (3 + s); };
    auto bar_qfree = [&](int s) { return bars + 8 * (5 + s); };
    const uint32_t bar_dofull = bars + 8 * 7, bar_dofree = bars + 8 * 8, bar_s = bars + 8 * 9, bar_dp = bars + 8 * 10,
                   bar_p = bars + 8 * 11, bar_dq = bars + 8 * 13, bar_drained = bars + 8 * 14,
                   bar_dss = bars + 8 * 15;
    auto bar_work = [&](int s) { return bars + 8 * (16 + s); };      // unit written
    auto bar_workfree = [&](int s) { return bars + 8 * (18 + s); };  // unit done by the producer, MMA, 4 drain and 8 compute warps
    const uint32_t bar_ask = bars + 8 * 12;                           // the launch control has answered
    const uint32_t bar_late = bars + 8 * 20;                          // the MMA warp is near the end of a unit
    const uint32_t bar_meet = bars + 8 * 21;                          // the 8 compute warps, twice in the epilogue of a cut unit
    volatile BwdWork* s_work = reinterpret_cast<volatile BwdWork*>(sgen + L::OFF_WORK);

    if (tid == 0) {
        *abort_flag = 0;
        mbar_init(bar_kv, 1);
        for (int s = 0; s < 2; ++s) {
            mbar_init(bar_qfull(s), 1);
            mbar_init(bar_ldfull(s), 32);
            mbar_init(bar_qfree(s), 1);
            mbar_init(bar_work(s), 1);
            mbar_init(bar_workfree(s), 14);
        }
        mbar_init(bar_dofull, 1);
        mbar_init(bar_dofree, 1);
        mbar_init(bar_s, 1);
        mbar_init(bar_dp, 1);
        mbar_init(bar_p, 8);
        mbar_init(bar_dss, 8);
        mbar_init(bar_dq, 1);
        mbar_init(bar_drained, 4);
        mbar_init(bar_ask, 1);
        mbar_init(bar_late, 1);
        mbar_init(bar_meet, 8);
        fence_mbar_init();
    }
    if (warp == 13) {
        tmem_alloc(smem_u32(s_tmem_base), TMEM_COLS);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *s_tmem_base;
    // The r-th unit of the CTA; false: there is none, or a wait gave up.  A role reads what it needs of it and arrives at the end
    // of it.
    auto take = [&](int r) {
        mbar_wait(bar_work(r & 1), (r >> 1) & 1, abort_flag, status);
        return (bool)__all_sync(0xffffffffu, s_work[r & 1].n_iter >= 0 && !*abort_flag);
    };
    auto done = [&](int r) {
        __syncwarp();
        if (lane == 0) mbar_arrive(bar_workfree(r & 1));
    };
    const uint32_t tmem_S = tmem;
    const uint32_t tmem_P = tmem + 128;
    const uint32_t tmem_dV = tmem + 256;
    const uint32_t tmem_dK = tmem + 384;

    if (warp >= 12) {
        reg_dec<80>();
        if (warp == 12) {
            // ================= producer =================
            float* sLse = reinterpret_cast<float*>(sgen + L::OFF_LSE);
            float* sDv = reinterpret_cast<float*>(sgen + L::OFF_DVEC);
            uint32_t J = 0;                                     // tiles of the CTA so far
            for (int r = 0; take(r); ++r) {
                const volatile BwdWork* work = s_work + (r & 1);
                const int tok0 = work->tok0, T = work->T, m_first = work->m_first, m_last = work->m_last, g = work->g;
                const uint32_t end = J + work->n_iter;
                int h = work->h_start, m = work->m_start;
                auto load_q = [&](uint32_t J, int h, int qtok) {
                    // Q(J): stage s, free once every MMA of tile J-2 has completed
                    const int s = J & 1;
                    if (J >= 2) mbar_wait(bar_qfree(s), ((J >> 1) + 1) & 1, abort_flag, status);
                    if (lane == 0) {
                        mbar_expect_tx(bar_qfull(s), L::TB);
                        for (int c = 0; c < NBOX; ++c) tma_load_3d(sQ + s * L::TB + c * BOX_BYTES, &tm_q, c * 64, h, qtok, bar_qfull(s));
                    }
                };
                if (J < end) {
                    load_q(J, h, tok0 + m * TILE);
                    // K is last read by the last unit's last dQ product, V before that
                    if (J > 0) mbar_wait(bar_dq, (J - 1) & 1, abort_flag, status);
                    if (lane == 0) {
                        const int ktok = tok0 + work->n * TILE;
                        mbar_expect_tx(bar_kv, 2 * L::TB);
                        for (int c = 0; c < NBOX; ++c) tma_load_3d(sK + c * BOX_BYTES, &tm_k, c * 64, g, ktok, bar_kv);
                        for (int c = 0; c < NBOX; ++c) tma_load_3d(sV + c * BOX_BYTES, &tm_v, c * 64, g, ktok, bar_kv);
                    }
                }
                for (const uint32_t first = J; J < end; ++J) {
                    const int s = J & 1;
                    const int qtok = tok0 + m * TILE;
                    if (J != first) load_q(J, h, qtok);
                    // lse(J), D(J): beside Q
                    const size_t rowbase = (size_t)h * p.total_tokens + qtok;
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const int i = lane * 4 + u;
                        const bool qv = (m * TILE + i) < T;
                        // stored negated (they are subtracted with one fused multiply-add); -inf makes P vanish
                        // for the rows past the end of the trace
                        sLse[s * TILE + i] = qv ? p.lse[rowbase + i] * -1.4426950408889634f : -INFINITY;
                        sDv[s * TILE + i] = qv ? p.dvec[rowbase + i] * -p.scale : 0.f;
                    }
                    mbar_arrive(bar_ldfull(s));
                    // dO(J): single buffer, free once dP(J-1) and dV(J-1) have completed
                    if (lane == 0) {
                        if (J >= 1) mbar_wait(bar_dofree, (J - 1) & 1, abort_flag, status);
                        mbar_expect_tx(bar_dofull, L::TB);
                        for (int c = 0; c < NBOX; ++c) tma_load_3d(sDO + c * BOX_BYTES, &tm_do, c * 64, h, qtok, bar_dofull);
                    }
                    __syncwarp();
                    if (++m > m_last) {
                        m = m_first;
                        ++h;
                    }
                }
                done(r);
            }
            if (*abort_flag) {                            // a wait gave up: let the copies in flight land, then leave
                const long long t0 = clock64();
                while (clock64() - t0 < 2000000) {}
            }
        } else if (warp == 14) {
            // ================= list of units =================
            // The first one is the CTA's own; after it units of CTAs of the grid that have not started, asked for a few tiles
            // before the end of the one before: what is asked for and found (about 3 us) lies beside those tiles, and the last
            // units still go to whoever is free first.
            int x = blockIdx.x, tiles = 0;                // of the unit before
            bool ok = true;
            for (int r = 0; ; ++r) {
                if (r > 0) {
                    mbar_wait_limit(bar_late, (r - 1) & 1, abort_flag, status, wait_limit_of(WAIT_LIMIT_CLOCKS, tiles));
                    if (*abort_flag) break;               // nothing is asked for that would not be waited for
                    if (lane == 0) {
                        mbar_expect_tx(bar_ask, 16);
                        ask_for_cta(sbase + L::OFF_ASK, bar_ask);
                    }
                    mbar_wait(bar_ask, (r - 1) & 1, abort_flag, status);
                    int y;
                    ok = cta_answer(sbase + L::OFF_ASK, x, y) && !*abort_flag;
                    fence_proxy_async();                  // the answer is read before the next one comes over it
                    __syncwarp();
                }
                BwdWork w;
                w.n = w.tok0 = w.T = w.m_first = w.m_last = w.h_start = w.m_start = w.g = w.cut = w.general = w.pad = 0;
                w.n_iter = -1;
                BwdUnit unit;
                if (ok && bwd_unit_of(p, mv.bwd_order, n_items, x, unit, w.g)) {
                    const int4 me = block_info(mv, unit.block);
                    const int G = p.Hq / p.Hkv;
                    w.n = me.z;
                    w.tok0 = me.x;
                    w.T = me.y;
                    w.m_first = mv.col_first[unit.block];           // == n unless the key slots were re-ordered
                    w.m_last = mv.col_last[unit.block];
                    w.general = mv.hdr->general != 0;
                    const int nm = w.m_last - w.m_first + 1;        // query blocks m_first .. m_last can see this key block
                    if (nm <= 0) {
                        w.n_iter = 0;                               // no query sees any key of the block (general metadata only)
                    } else {
                        w.n_iter = (unit.tile1 < 0 ? G * nm : unit.tile1) - unit.tile0;     // of the G * nm (head, query block) tiles
                        w.h_start = w.g * G + unit.tile0 / nm;
                        w.m_start = w.m_first + unit.tile0 % nm;
                    }
                    w.cut = unit.cut;
                }
                const int slot = r & 1;
                if (r >= 2) mbar_wait(bar_workfree(slot), ((r >> 1) + 1) & 1, abort_flag, status);
                if (*abort_flag) break;                   // the slot may still be read: no role may see another length of its unit
                tiles = w.n_iter;
                if (lane == 0) {
                    volatile int* dst = reinterpret_cast<volatile int*>(s_work + slot);
                    const int* src = reinterpret_cast<const int*>(&w);
#pragma unroll
                    for (int i = 0; i < (int)(sizeof(BwdWork) / 4); ++i) dst[i] = src[i];
                    mbar_arrive(bar_work(slot));
                }
                __syncwarp();
                if (w.n_iter < 0) break;
            }
        } else if (warp == 13) {
            // ================= MMA issuer (all lanes walk the loop, one elected lane issues) =================
            const bool leader = elect_one();
            // descriptors of stage 0; a stage or a k-step adds a constant to the 14-bit address field
            const uint64_t dK_k = smem_desc(sK, 16, 1024), dV_k = smem_desc(sV, 16, 1024);
            const uint64_t dQ_k = smem_desc(sQ, 16, 1024), dDO_k = smem_desc(sDO, 16, 1024);
            const uint64_t dK_mn = smem_desc(sK, BOX_BYTES, 1024), dDS_mn = smem_desc(sDS, BOX_BYTES, 1024);
            const uint64_t dDS_k = smem_desc(sDS, 16, 1024);
            const uint64_t dQ_mn = smem_desc(sQ, BOX_BYTES, 1024), dDO_mn = smem_desc(sDO, BOX_BYTES, 1024);
            constexpr uint64_t STAGE = (uint64_t)(L::TB >> 4);
            uint32_t J = 0;                                     // tiles of the CTA so far
            int loads = 0;                                      // units with tiles so far
            for (int r = 0; take(r); ++r) {
                const uint32_t first = J, end = J + s_work[r & 1].n_iter;
                if (first == end) {
                    if (lane == 0) mbar_arrive(bar_late);
                    done(r);
                    continue;
                }
                mbar_wait(bar_kv, loads & 1, abort_flag, status);
                ++loads;
                mbar_wait(bar_qfull(J & 1), (J >> 1) & 1, abort_flag, status);
                tc_fence_after();
                {
                    const uint64_t so = J & 1 ? STAGE : 0;
#pragma unroll
                    for (int kk = 0; kk < D / 16; ++kk) {
                        const uint64_t off = (uint64_t)(((kk >> 2) * BOX_BYTES + (kk & 3) * 32) >> 4);
                        if (leader) mma_ss(tmem_S, dK_k + off, dQ_k + so + off, IDESC_ST, kk > 0);
                    }
                }
                if (leader) mma_commit(bar_s);
                for (; J < end; ++J) {
                    const int s = J & 1;
                    const uint32_t ph = J & 1;
                    const uint64_t so = s ? STAGE : 0;
                    if (lane == 0 && (J + BWD_LATE == end || (J == first && end - first < BWD_LATE))) mbar_arrive(bar_late);
                    // dP^T(J) = V dO^T  (its columns hold dQ(J-1) until the drain warps have read it)
                    mbar_wait(bar_dofull, ph, abort_flag, status);
                    if (J > 0) mbar_wait(bar_drained, (J - 1) & 1, abort_flag, status);
                    tc_fence_after();
#pragma unroll
                    for (int kk = 0; kk < D / 16; ++kk) {
                        const uint64_t off = (uint64_t)(((kk >> 2) * BOX_BYTES + (kk & 3) * 32) >> 4);
                        if (leader) mma_ss(tmem_P, dV_k + off, dDO_k + off, IDESC_ST, kk > 0);
                    }
                    if (leader) mma_commit(bar_dp);
                    // dV(J) += P^T dO.  A unit's first one overwrites the last unit's dV (and dK later on): the compute warps
                    // have read both out before they write this tile's P.
                    mbar_wait(bar_p, ph, abort_flag, status);
                    tc_fence_after();
#pragma unroll
                    for (int kk = 0; kk < TILE / 16; ++kk)
                        if (leader) mma_ts(tmem_dV, tmem_S + (kk >> 2) * 64 + (kk & 3) * 8, dDO_mn + (uint64_t)(kk * 128), IDESC_KV,
                               (J != first) || (kk > 0));
                    if (leader) mma_commit(bar_dofree);
                    // S^T(J+1) = K Q^T
                    if (J + 1 < end) {
                        const uint64_t so1 = s ? 0 : STAGE;
                        mbar_wait(bar_qfull(s ^ 1), ((J + 1) >> 1) & 1, abort_flag, status);
                        tc_fence_after();
#pragma unroll
                        for (int kk = 0; kk < D / 16; ++kk) {
                            const uint64_t off = (uint64_t)(((kk >> 2) * BOX_BYTES + (kk & 3) * 32) >> 4);
                            if (leader) mma_ss(tmem_S, dK_k + off, dQ_k + so1 + off, IDESC_ST, kk > 0);
                        }
                        if (leader) mma_commit(bar_s);
                    }
                    // dQ(J) = dS K, then dK(J) += dS^T Q.  Both read dS from shared memory: the same swizzled buffer
                    // is the MN-major A operand of dQ (queries contiguous) and, read as [keys x queries] rows, the
                    // K-major A operand of dK; dQ goes first so that the drain can start while dK still runs.
                    mbar_wait(bar_dss, ph, abort_flag, status);
                    tc_fence_after();
#pragma unroll
                    for (int kk = 0; kk < TILE / 16; ++kk)
                        if (leader) mma_ss(tmem_P, dDS_mn + (uint64_t)(kk * 128), dK_mn + (uint64_t)(kk * 128), IDESC_DQ, kk > 0);
                    if (leader) mma_commit(bar_dq);
#pragma unroll
                    for (int kk = 0; kk < TILE / 16; ++kk) {
                        const uint64_t off = (uint64_t)(((kk >> 2) * BOX_BYTES + (kk & 3) * 32) >> 4);
                        if (leader) mma_ss(tmem_dK, dDS_k + off, dQ_mn + so + (uint64_t)(kk * 128), IDESC_KV, (J != first) || (kk > 0));
                    }
                    if (leader) mma_commit(bar_qfree(s));
                }
                done(r);
            }
        }
    } else if (warp >= 8) {
        // ================= drain warps: dQ(j), query rows on lanes =================
        reg_inc<144>();
        const int quad = warp & 3;
        const int row = quad * 32 + lane;
        const uint32_t lane_sel = (uint32_t)(quad * 32) << 16;
        uint8_t* stg_row = sgen + L::OFF_STG + row * 128;
        uint32_t J = 0;                                         // tiles of the CTA so far
        // the four warps meet at a named barrier in every tile: they take a unit together or not at all
        for (int r = 0; group_all(1, 128, take(r)); ++r) {
            const volatile BwdWork* work = s_work + (r & 1);
            const int tok0 = work->tok0, m_first = work->m_first, m_last = work->m_last;
            const uint32_t end = J + work->n_iter;
            int h = work->h_start, m = work->m_start;
            for (; J < end; ++J) {
                mbar_wait(bar_dq, J & 1, abort_flag, status);
                tc_fence_after();
                uint32_t o[D];
    #pragma unroll
                for (int ch = 0; ch < D / 32; ++ch) {
                    uint32_t t[32];
                    tmem_ld32(tmem_P + lane_sel + ch * 32, t);
    #pragma unroll
                    for (int e = 0; e < 32; ++e) o[ch * 32 + e] = t[e];
                }
                tmem_wait_ld();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(bar_drained);      // the columns may be overwritten from here on
                // chunks of 32 head-dim columns through two staging buffers
    #pragma unroll
                for (int ch = 0; ch < D / 32; ++ch) {
                    const int buf = ch & 1;
                    if (tid == 256) bulk_wait_read<1>();      // the reduce that last read this buffer has finished reading
                    named_bar_sync(1, 128);
    #pragma unroll
                    for (int c = 0; c < 8; ++c)
                        *reinterpret_cast<uint4*>(stg_row + buf * L::STG_BYTES + ((c ^ (row & 7)) << 4)) =
                            make_uint4(o[ch * 32 + c * 4], o[ch * 32 + c * 4 + 1], o[ch * 32 + c * 4 + 2], o[ch * 32 + c * 4 + 3]);
                    fence_proxy_async();
                    named_bar_sync(1, 128);
                    if (tid == 256) {
                        tma_reduce_add_3d(&tm_dq, ch * 32, h, tok0 + m * TILE, sSTG + buf * L::STG_BYTES);
                        bulk_commit();
                    }
                }
                if (++m > m_last) {
                    m = m_first;
                    ++h;
                }
            }
            done(r);
        }
        if (tid == 256) bulk_wait<0>();
    } else {
        // ================= compute warps =================
        reg_inc<144>();
        const int quad = warp & 3;
        const int half = warp >> 2;
        const int row = quad * 32 + lane;                  // TMEM lane: key row of S^T, dP^T
        const uint32_t lane_sel = (uint32_t)(quad * 32) << 16;
        const int col0 = half * 64;                        // this thread's 64 query columns
        const float* sLse = reinterpret_cast<const float*>(sgen + L::OFF_LSE);
        const float* sDv = reinterpret_cast<const float*>(sgen + L::OFF_DVEC);
        uint8_t* sDS_row = sgen + L::OFF_DS + half * BOX_BYTES + row * 128;
        float pv[64];
        uint32_t J = 0;                                         // tiles of the CTA so far
        // The compute warps meet by a bounded wait instead: deciding together at each unit cost units of 4 to 12 tiles 1 % (200
        // traces of 300 tokens, 32 heads on 8: 945 -> 954 us).
        uint32_t meets = 0;
        auto meet = [&] {
            __syncwarp();
            if (lane == 0) mbar_arrive(bar_meet);
            mbar_wait(bar_meet, meets++ & 1, abort_flag, status);
        };
        for (int r = 0; take(r); ++r) {
            const volatile BwdWork* work = s_work + (r & 1);
            const uint32_t end = J + work->n_iter;
            if (J == end) {                                         // a key block that no query sees: its gradients are zero
                bwd_zero_rows<D>(p, work->tok0 + work->n * TILE, min(TILE, work->T - work->n * TILE), work->g, 256);
                done(r);
                continue;
            }
            // queries [my_first, my_end) of the trace see this key; nobody sees a slot past the trace
            int my_end = 0, my_first = work->n * TILE + row;
            if (my_first < work->T) {
                const int at = work->tok0 + my_first;
                my_end = min(mv.evict[at], work->T);
                if (work->general) my_first = mv.kfirst[at];
            }
            int m = work->m_start;                             // query block of the tile of the next phase_p

            auto phase_p = [&](uint32_t j) {        // P^T(j) = exp2(S^T * c - lse), masked
                const int s = j & 1;
                const int lo = my_first - (m * TILE + col0), hi = my_end - (m * TILE + col0);     // columns [lo, hi) see the key
                m = (m == work->m_last) ? work->m_first : m + 1;       // read again, not kept: registers are short here
                mbar_wait(bar_ldfull(s), (j >> 1) & 1, abort_flag, status);
                mbar_wait(bar_s, j & 1, abort_flag, status);
                tc_fence_after();
                const float4* l4 = reinterpret_cast<const float4*>(sLse + s * TILE + col0);
                uint32_t r0[32], r1[32];
                tmem_ld32(tmem_S + lane_sel + col0, r0);
                tmem_ld32(tmem_S + lane_sel + col0 + 32, r1);
                tmem_wait_ld();
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
                tmem_st32(tmem_S + lane_sel + col0, pk);       // 64 queries -> 32 packed columns at [col0, col0+32)
                tmem_wait_st();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(bar_p);
            };

            auto phase_ds = [&](uint32_t j) {       // dS^T(j) = P^T (scale dP^T - scale D)
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
                // dS^T row -> shared memory, MN-major (queries contiguous), 128-byte swizzle: the 64 queries of
                // this half are the 128-byte row `row` of block `half`; 16-byte chunk c sits at (c ^ (row % 8))
#pragma unroll
                for (int c = 0; c < 8; ++c)
                    *reinterpret_cast<uint4*>(sDS_row + ((c ^ (row & 7)) << 4)) =
                        make_uint4(dk_[c * 4], dk_[c * 4 + 1], dk_[c * 4 + 2], dk_[c * 4 + 3]);
                fence_proxy_async();                     // dS visible to the tensor core's reads of shared memory
                tc_fence_before();                       // orders this thread's reads of dP^T before the dQ MMA that overwrites it
                __syncwarp();
                if (lane == 0) mbar_arrive(bar_dss);
            };

            phase_p(J);
            for (; J < end; ++J) {
                phase_ds(J);
                if (J + 1 < end) phase_p(J + 1);
            }

            // ---- epilogue: dK, dV of this key block, once every MMA has completed ----
            mbar_wait(bar_qfree((end - 1) & 1), ((end - 1) >> 1) & 1, abort_flag, status);
            tc_fence_after();
            // through the memory of dS, which nothing reads any more; the next unit's tiles are on their way into the others
            bwd_epilogue<D>(p, work->cut, work->g, 1, 0, tmem_dK + lane_sel + half * HALF_D, tmem_dV + lane_sel + half * HALF_D, row, half,
                            work->tok0 + work->n * TILE + quad * 32, work->T - work->n * TILE - quad * 32, sgen + L::OFF_DS + warp * 4096,
                            reinterpret_cast<volatile int*>(sgen + L::OFF_MISC + 8), meet);
            done(r);
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 13) {
        __syncwarp();
        tmem_dealloc(tmem, TMEM_COLS);
    }
}

template <int D>
static int launch_dot(const __nv_bfloat16* dout, const __nv_bfloat16* out, float* dvec, float* dq_acc, long long dq_ts, int total_tokens, int Hq,
                      WsHeader* hdr, const BwdPlanArgs& plan, cudaStream_t st) {
    const long long rows = (long long)total_tokens * Hq;
    const int rows_per_warp = (32 / (D / 8)) * DOT_ROWS;
    const long long warps = (rows + rows_per_warp - 1) / rows_per_warp;
    const int threads = 256;
    const long long blocks = (warps * 32 + threads - 1) / threads + 1;
    if (blocks > 0x7fffffffLL) return KVS_ERR_UNSUPPORTED;
    return launch_after(bwd_dot_kernel<D>, (unsigned)blocks, threads, 0, st, dout, out, dvec, dq_acc, dq_ts, total_tokens, Hq, hdr, plan);
}

template <int D>
static int launch_main(const CUtensorMap& tq, const CUtensorMap& tk, const CUtensorMap& tv, const CUtensorMap& tdo, const CUtensorMap& tdq,
                       const MetaView& mv, const BwdParams& p, unsigned units, cudaStream_t st) {
    auto kern = bwd_kernel<D>;
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, BwdSmem<D>::DYN_BYTES) != cudaSuccess) return cuda_refused();
    return launch_after(kern, units, BWD_THREADS, BwdSmem<D>::DYN_BYTES, st, tq, tk, tv, tdo, tdq, mv, p);
}

}  // namespace kvs

using namespace kvs;

extern "C" size_t kvs_attn_bwd_workspace_bytes(int total_tokens, int Hq, int Hkv, int head_dim, int grad_dtype) {
    if (total_tokens < 0 || Hq <= 0 || Hkv <= 0 || head_dim <= 0) return 0;
    if (grad_dtype != KVS_GRAD_BF16 && grad_dtype != KVS_GRAD_FP32) return 0;
    return bwd_ws_layout(total_tokens, Hq, head_dim, grad_dtype).total;
}

size_t kvs::bwd_base_bytes(int total_tokens, int Hq, int head_dim, int grad_dtype) {
    return bwd_ws_layout(total_tokens, Hq, head_dim, grad_dtype).base;
}
size_t kvs::bwd_cut_bytes(int total_tokens, int Hq, int head_dim, bool less) {
    const BwdWsLayout L = bwd_ws_layout(total_tokens, Hq, head_dim, KVS_GRAD_FP32, less ? BWD_MIN_UNIT_LESS : BWD_MIN_UNIT);
    return L.total - L.base;
}

namespace {
// CTA pairs take head_dim 128 where the traces are long: they read and stage less, and on long walks the chip runs at its power
// limit.  On short ones a pair's union of two query ranges and its costlier start weigh more, the more so the fewer heads share
// a key block.  Main kernel, single CTAs -> pairs, us (by tokens a trace, 48000 a batch, with nothing evicted 24000 to 32000; last-
// 4-turns, summary, nothing evicted, token-level):
//   32 heads on 8,  6000: 2844 -> 3064, 1980 -> 2307,  3694 ->  3441,  5932 ->  5832
//                  12000: 5293 -> 5120, 3437 -> 3440,  6040 ->  5495, 11404 -> 10971
//                  16000: 6687 -> 6436, 4443 -> 4403, 10129 ->  8952, 15039 -> 14283
//                  24000: 9750 -> 9072, 6520 -> 6232, 11745 -> 10639, 22404 -> 21227
//   16 on 16,      16000: 3506 -> 3463, 2410 -> 2515,  5152 ->  4734,  7524 ->  7429
//                  24000: 5060 -> 4838, 3456 -> 3427,  6000 ->  5501, 11329 -> 10872
// (28 on 4 and 16 on 2 are like 32 on 8.)  The mean length is what is known here that a caller cannot overstate, and no batch of
// short traces reaches it; a long trace with short ones beside it stays with single CTAs (40000 + 1 token: 11.7 instead of 10.8 ms).
bool use_pairs(int batch, int total_tokens, int G, int head_dim) {
    return head_dim == 128 && total_tokens / batch >= (G > 1 ? 16000 : 24000);
}

// in_ts: elements between consecutive tokens of q and of k, v; g_ts: of dq and of dk, dv (0: tensors of their own)
int bwd_impl(const void* dout, const void* q, const void* k, const void* v, long long in_ts, const void* out, const float* lse,
             const void* meta_buf, int batch, int total_tokens, int max_seqlen, int Hq, int Hkv, int head_dim,
             float softmax_scale, int grad_dtype, void* dq, void* dk, void* dv, long long g_ts, void* workspace,
             size_t workspace_bytes, kvs_stream_t stream, void* event_main_begin, void* event_main_end, const BwdWhole* part_of = nullptr) {
    cudaEvent_t ev0 = (cudaEvent_t)event_main_begin, ev1 = (cudaEvent_t)event_main_end;
    if (batch < 0 || total_tokens < 0 || max_seqlen < 0 || Hq <= 0 || Hkv <= 0) return KVS_ERR_INVALID_ARG;
    if (head_dim != 64 && head_dim != 128) return KVS_ERR_UNSUPPORTED;
    if (Hq % Hkv != 0 || Hq > 65535) return KVS_ERR_UNSUPPORTED;
    if (grad_dtype != KVS_GRAD_BF16 && grad_dtype != KVS_GRAD_FP32) return KVS_ERR_INVALID_ARG;
    if (total_tokens == 0 || batch == 0) return KVS_OK;
    if (!dout || !q || !k || !v || !out || !lse || !meta_buf || !dq || !dk || !dv || !workspace) return KVS_ERR_INVALID_ARG;
    if ((((uintptr_t)dout | (uintptr_t)q | (uintptr_t)k | (uintptr_t)v | (uintptr_t)out | (uintptr_t)dq | (uintptr_t)dk | (uintptr_t)dv) & 15) != 0)
        return KVS_ERR_ALIGNMENT;
    if (((uintptr_t)lse & 3) != 0 || ((uintptr_t)workspace & 255) != 0 || ((uintptr_t)meta_buf & 255) != 0) return KVS_ERR_ALIGNMENT;
    if (softmax_scale < 0.f || softmax_scale != softmax_scale) return KVS_ERR_INVALID_ARG;
    const BwdWhole whole = part_of ? *part_of : BwdWhole{meta_buf, batch, total_tokens, max_seqlen, Hkv, nullptr, false};
    const bool less = whole.cut_buf ? whole.cut_less : workspace_bytes < bwd_ws_layout(total_tokens, Hq, head_dim, grad_dtype).total;
    const int min_unit = less ? BWD_MIN_UNIT_LESS : BWD_MIN_UNIT;
    const BwdWsLayout W = bwd_ws_layout(total_tokens, Hq, head_dim, grad_dtype, min_unit);
    if (workspace_bytes < W.base) return KVS_ERR_WORKSPACE;
    int rc = check_device_sm100();
    if (rc != KVS_OK) return rc;
    const MetaLayout L = meta_layout(batch, total_tokens, max_seqlen);
    const MetaView mv = meta_view(meta_buf, L);
    const bool pair = use_pairs(whole.batch, whole.total_tokens, Hq / Hkv, head_dim);
    const int q_rows = pair ? TILE / 2 : TILE;       // rows of the boxes of q, dout and dq
    CUtensorMap tq, tk, tv, tdo, tdq;
    if ((rc = make_tmap_thd(&tq, q, total_tokens, Hq, head_dim, q_rows, in_ts)) != KVS_OK) return rc;
    if ((rc = make_tmap_thd(&tk, k, total_tokens, Hkv, head_dim, TILE, in_ts)) != KVS_OK) return rc;
    if ((rc = make_tmap_thd(&tv, v, total_tokens, Hkv, head_dim, TILE, in_ts)) != KVS_OK) return rc;
    if ((rc = make_tmap_thd(&tdo, dout, total_tokens, Hq, head_dim, q_rows)) != KVS_OK) return rc;
    cudaStream_t st = (cudaStream_t)stream;
    char* ws = (char*)workspace;
    const size_t nq = (size_t)total_tokens * Hq * head_dim;
    BwdParams p;
    p.batch = batch;
    p.total_tokens = total_tokens;
    p.max_seqlen = max_seqlen < total_tokens ? max_seqlen : total_tokens;
    p.Hq = Hq;
    p.Hkv = Hkv;
    p.scale = softmax_scale == 0.f ? 1.0f / sqrtf((float)head_dim) : softmax_scale;
    p.scale_log2 = p.scale * 1.4426950408889634f;
    p.lse = lse;
    p.dvec = (const float*)(ws + W.dvec);
    // bf16 gradients: dq is accumulated in the workspace (contiguous) and cast into place afterwards;
    // fp32 gradients: straight into dq, whatever its token stride
    const long long dq_ts_out = g_ts > 0 ? g_ts : (long long)Hq * head_dim;
    float* dq_acc = grad_dtype == KVS_GRAD_FP32 ? (float*)dq : (float*)(ws + W.dq_acc);
    const long long dq_ts = grad_dtype == KVS_GRAD_FP32 ? dq_ts_out : (long long)Hq * head_dim;
    if ((rc = make_tmap_f32_thd(&tdq, dq_acc, total_tokens, Hq, head_dim, q_rows, dq_ts)) != KVS_OK) return rc;
    p.dk = dk;
    p.dv = dv;
    p.dkv_ts = g_ts > 0 ? g_ts : (long long)Hkv * head_dim;
    p.grad_fp32 = grad_dtype == KVS_GRAD_FP32;
    p.status = &((WsHeader*)ws)->status;
    // Items and their units.  Without room for the plan (a workspace of the base size, or very many very short traces) the
    // items stay whole.
    const int ctas = pair ? 2 : 1;
    const long long both = ((long long)L.nb_cap + batch) / 2;         // sum of ceil(nb_b / 2) over the traces
    const int items = pair && both < L.nb_cap ? (int)both : L.nb_cap;
    const int slots = W.slots / ctas;
    char* cut = whole.cut_buf ? (char*)whole.cut_buf : ws + W.base;
    const bool planned = (whole.cut_buf || workspace_bytes >= W.total) && items + slots / Hkv <= W.unit_cap;
    BwdPlanArgs pa;
    memset(&pa, 0, sizeof(pa));
    if (planned) {
        const MetaLayout AL = meta_layout(whole.batch, whole.total_tokens, whole.max_seqlen);
        pa.all = meta_view(whole.meta_buf, AL);
        pa.mv = mv;
        pa.all_cap = AL.nb_cap;
        pa.cap = L.nb_cap;
        pa.all_batch = whole.batch;
        pa.all_tokens = whole.total_tokens;
        pa.all_maxlen = whole.max_seqlen < whole.total_tokens ? whole.max_seqlen : whole.total_tokens;
        pa.batch = batch;
        pa.tokens = total_tokens;
        pa.maxlen = p.max_seqlen;
        pa.pairs = pair;
        pa.by_trace = !pair && whole.batch >= BWD_MANY_TRACES && (long long)total_tokens * Hq * head_dim * 8 > BWD_L2_BYTES;
        pa.G = Hq / Hkv;
        pa.all_Hkv = whole.Hkv;
        pa.Hkv = Hkv;
        pa.all_slots = bwd_ws_layout(whole.total_tokens, whole.Hkv * pa.G, head_dim, grad_dtype, min_unit).slots / ctas;
        pa.slots = slots;
        pa.min_unit = min_unit;
        pa.plan = (BwdPlan*)(cut + W.plan);
        pa.units = (BwdUnit*)(cut + W.units);
        pa.arrived = (int32_t*)(cut + W.arrived);
        pa.arrived_n = 2 * W.slots;
    }
    p.plan = pa.plan;
    p.units = pa.units;
    p.arrived = pa.arrived;
    p.part = (float4*)(cut + W.part);
    // every cut of an item adds at most as many units as it takes slots
    const long long ctas_all = (long long)items * Hkv + (planned ? slots : 0);
    if (ctas_all > 0x3fffffffLL) return KVS_ERR_UNSUPPORTED;
    const __nv_bfloat16 *dout16 = (const __nv_bfloat16*)dout, *out16 = (const __nv_bfloat16*)out;
    rc = head_dim == 64 ? launch_dot<64>(dout16, out16, (float*)(ws + W.dvec), dq_acc, dq_ts, total_tokens, Hq, (WsHeader*)ws, pa, st)
                        : launch_dot<128>(dout16, out16, (float*)(ws + W.dvec), dq_acc, dq_ts, total_tokens, Hq, (WsHeader*)ws, pa, st);
    if (rc != KVS_OK) return rc;
    if (ev0 && cudaEventRecord(ev0, st) != cudaSuccess) return KVS_ERR_CUDA;
    rc = pair             ? launch_bwd_pair(tq, tk, tv, tdo, tdq, mv, p, (unsigned)ctas_all, st)
         : head_dim == 64 ? launch_main<64>(tq, tk, tv, tdo, tdq, mv, p, (unsigned)ctas_all, st)
                          : launch_main<128>(tq, tk, tv, tdo, tdq, mv, p, (unsigned)ctas_all, st);
    if (rc == KVS_OK && ev1 && cudaEventRecord(ev1, st) != cudaSuccess) return KVS_ERR_CUDA;
    if (rc != KVS_OK) return rc;
    if (grad_dtype == KVS_GRAD_BF16) {
        const size_t n4 = nq / 4;
        const size_t blocks = (n4 + 255) / 256;
        if (blocks > 0x7fffffffull) return KVS_ERR_UNSUPPORTED;
        if ((rc = launch_after(bwd_cast_kernel, (unsigned)blocks, 256, 0, st, (const float*)dq_acc, (__nv_bfloat16*)dq, n4, Hq * head_dim,
                               dq_ts_out)) != KVS_OK)
            return rc;
    }
    return KVS_OK;
}
}  // namespace

int kvs::bwd_of_chunk(const BwdWhole& whole, const void* dout, const void* q, const void* k, const void* v, const void* out, const float* lse,
                      const void* meta_buf, int batch, int total_tokens, int max_seqlen, int Hq, int Hkv, int head_dim, float softmax_scale,
                      int grad_dtype, void* dq, void* dk, void* dv, void* workspace, size_t workspace_bytes, kvs_stream_t stream) {
    return bwd_impl(dout, q, k, v, 0, out, lse, meta_buf, batch, total_tokens, max_seqlen, Hq, Hkv, head_dim, softmax_scale, grad_dtype, dq, dk,
                    dv, 0, workspace, workspace_bytes, stream, nullptr, nullptr, &whole);
}

extern "C" int kvs_attn_bwd_ex(const void* dout, const void* q, const void* k, const void* v, const void* out, const float* lse,
                               const void* meta_buf, int batch, int total_tokens, int max_seqlen, int Hq, int Hkv, int head_dim,
                               float softmax_scale, int grad_dtype, void* dq, void* dk, void* dv, void* workspace,
                               size_t workspace_bytes, kvs_stream_t stream, void* event_main_begin, void* event_main_end) {
    return bwd_impl(dout, q, k, v, 0, out, lse, meta_buf, batch, total_tokens, max_seqlen, Hq, Hkv, head_dim, softmax_scale, grad_dtype,
                    dq, dk, dv, 0, workspace, workspace_bytes, stream, event_main_begin, event_main_end);
}

extern "C" int kvs_attn_bwd_packed(const void* dout, const void* qkv, const void* out, const float* lse, const void* meta_buf,
                                   int batch, int total_tokens, int max_seqlen, int Hq, int Hkv, int head_dim, float softmax_scale,
                                   int grad_dtype, void* dqkv, void* workspace, size_t workspace_bytes, kvs_stream_t stream) {
    if (Hq <= 0 || Hkv <= 0 || head_dim <= 0) return KVS_ERR_INVALID_ARG;
    if (grad_dtype != KVS_GRAD_BF16 && grad_dtype != KVS_GRAD_FP32) return KVS_ERR_INVALID_ARG;
    if (total_tokens > 0 && batch > 0 && (!qkv || !dqkv)) return KVS_ERR_INVALID_ARG;
    const long long ts = (long long)(Hq + 2 * Hkv) * head_dim;
    const size_t gsz = grad_dtype == KVS_GRAD_FP32 ? 4 : 2;
    const char* in = (const char*)qkv;
    char* g = (char*)dqkv;
    return bwd_impl(dout, in, in + (size_t)Hq * head_dim * 2, in + (size_t)(Hq + Hkv) * head_dim * 2, ts, out, lse, meta_buf, batch,
                    total_tokens, max_seqlen, Hq, Hkv, head_dim, softmax_scale, grad_dtype, g, g + (size_t)Hq * head_dim * gsz,
                    g + (size_t)(Hq + Hkv) * head_dim * gsz, ts, workspace, workspace_bytes, stream, nullptr, nullptr);
}

extern "C" int kvs_attn_bwd(const void* dout, const void* q, const void* k, const void* v, const void* out, const float* lse,
                            const void* meta_buf, int batch, int total_tokens, int max_seqlen, int Hq, int Hkv, int head_dim,
                            float softmax_scale, int grad_dtype, void* dq, void* dk, void* dv, void* workspace,
                            size_t workspace_bytes, kvs_stream_t stream) {
    return kvs_attn_bwd_ex(dout, q, k, v, out, lse, meta_buf, batch, total_tokens, max_seqlen, Hq, Hkv, head_dim, softmax_scale,
                           grad_dtype, dq, dk, dv, workspace, workspace_bytes, stream, nullptr, nullptr);
}

