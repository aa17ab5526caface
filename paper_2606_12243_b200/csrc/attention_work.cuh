// What the attention kernels share: the cut of the keys, the CTA's work list, and small arithmetic.
//
// The split of the work is chosen on the device, from the lengths: either every (sequence, kv head, item) pair is cut into k
// ranges of tiles and the ranges are dealt to the CTAs in equal shares, or the tiles of all pairs laid end to end are cut
// into one range per CTA and row stream.  The cuts depend on the lengths, the heads and the grid only, so a one-stream and a
// two-stream launch cut alike and produce the same bits.  A pair that lies in several ranges is finished by all of their
// CTAs: each publishes its partial rows, goes on with its other items, and at its very end waits (bounded) for the other
// ranges of each such pair and merges its own slice of the rows, in range order.  All CTAs of a launch are resident together
// and publish before they wait, so no wait depends on another.
#pragma once
#include "common.cuh"
#include "tc_ptx.cuh"

namespace {

constexpr int HD = 128;                        // head dimension
constexpr int TKEYS = 128;                     // keys per tile
constexpr int HALF_BYTES = TKEYS * 128;        // 128 keys x 64 dims of bf16, as one TMA box lands
constexpr int SLOT_BYTES = 2 * HALF_BYTES;     // one tile of K or of V: dims 0..63, dims 64..127
constexpr int PART_ROW = HD + 2;               // floats per partial row: numerators, max (log2 units), sum
// costs in tiles: what an item costs besides its tiles (queries, first and last MMA, result), and a merge
constexpr int COST_ITEM = 4, COST_MERGE = 3;
constexpr int MAX_SPLITS = 16, MAX_SLOTS = 32; // ranges of a pair: cut evenly, in any case (a lane each when merged)

struct AttnWork {
    const float *q;             // [rows, H * HD] rotated queries
    float *part;                // [pair][slot]: partial rows
    __nv_bfloat16 *out;         // attention output planes (hi, lo)
    size_t out_plane;
    const int *len_eff;
    const TreeInfo *tree;
    int *status;
    const int *run_flag;        // null, or a device flag: the kernel leaves at once when it is zero
    int M, H, Hkv, max_batch, max_ctx, layer_ord;
    int batch, layer_ord2;      // second row stream: rows batch*M.., its own cache and layer ordinal
    int streams, ring_slots;
    int subs, rows_sub, rows8;  // items per kv head, query rows of each (but the last), the same rounded up to 8
    int slots;                  // ranges a pair may be cut into (the partial buffer's slots)
    int splits;                 // 0, or ranges per pair as asked for by the caller
    int w_one, w_two;           // the model's layers that run one row stream in a verify step, and those that run both
    unsigned long long m_recip; // 2^32 / M, rounded up: r / M for the few hundred query rows there are
    int *counters;              // per pair: arrivals, then finishers; zero between launches
    float scale;                // log2(e) / sqrt(hd)
};

struct Item { int pair, be, b, kvh, row0, rows, stream, split, n_split, n_ctx, k_begin, k_end, n_tiles, row_base; };

// The CTA's work list.  k > 0: its share of the k ranges of every pair; k == 0: its range of `per` tiles of one row stream, or
// of both in turn.
struct Cut { int k, per; };
struct ItemSrc { int s, s_end, range, b, g, off; };             // k > 0: the next item is `off`, the share ends at `range`
__device__ __forceinline__ void src_init(const AttnWork &a, const Cut &cut, int ranges, ItemSrc &c) {
    const int x = blockIdx.x;
    c.b = c.g = c.s = c.s_end = 0;
    if (cut.k > 0) {
        c.off = x * cut.per;
        c.range = min(a.streams * a.batch * a.Hkv * a.subs * cut.k, c.off + cut.per);
        return;
    }
    c.off = 0;
    if (a.streams * ranges <= (int)gridDim.x) {                // a CTA per range and stream
        c.s = x / ranges;
        c.s_end = c.s < a.streams ? c.s + 1 : c.s;
        c.range = x - c.s * ranges;
    } else {
        c.s_end = x < ranges ? a.streams : 0;
        c.range = x;
    }
}
// range `split` of n_split: tiles t0 .. t1 - 1 of pair (stream s, sequence b, item g of its kv heads)
__device__ __forceinline__ void set_item(const AttnWork &a, int s, int b, int g, int n_ctx, int t0, int t1, int split, int n_split, Item &it) {
    it.b = b; it.stream = s; it.be = s * a.batch + b;
    it.pair = it.be * a.Hkv * a.subs + g; it.kvh = g / a.subs;
    it.row0 = (g - it.kvh * a.subs) * a.rows_sub;
    it.rows = min(a.rows_sub, a.H / a.Hkv * a.M - it.row0);
    it.split = split; it.n_split = n_split;
    it.n_ctx = n_ctx; it.k_begin = t0 * TKEYS; it.k_end = min(n_ctx + a.M, t1 * TKEYS); it.n_tiles = t1 - t0;
    it.row_base = (((s ? a.layer_ord2 : a.layer_ord) * a.max_batch + b) * a.Hkv + it.kvh) * a.max_ctx;
}
__device__ __forceinline__ bool next_item(const AttnWork &a, const Cut &cut, ItemSrc &c, Item &it) {
    const int Hs = a.Hkv * a.subs;
    if (cut.k > 0) {
        while (c.off < c.range) {
            const int id = c.off++, bg = id / cut.k, split = id - bg * cut.k, be = bg / Hs, s = be / a.batch, b = be - s * a.batch;
            const int n_ctx = a.len_eff[b], tb = (n_ctx + a.M + TKEYS - 1) / TKEYS, n_split = min(cut.k, tb);
            if (split >= n_split) continue;                                                   // a short sequence has fewer ranges
            set_item(a, s, b, bg - be * Hs, n_ctx, split * tb / n_split, (split + 1) * tb / n_split, split, n_split, it);
            return true;
        }
        return false;
    }
    const int per = cut.per, lo = c.range * per, hi = lo + per;
    while (c.s < c.s_end) {
        if (c.b >= a.batch || c.off >= hi) { ++c.s; c.b = c.g = c.off = 0; continue; }      // done with this stream
        const int n_ctx = a.len_eff[c.b], tb = (n_ctx + a.M + TKEYS - 1) / TKEYS;
        if (c.off + Hs * tb <= lo) { c.off += Hs * tb; ++c.b; c.g = 0; continue; }            // this sequence ends before the range
        if (c.g == 0 && c.off < lo) c.g = (lo - c.off) / tb;                                  // its first pair that reaches into the range
        const int p_lo = c.off + c.g * tb, p_hi = p_lo + tb;
        if (c.g >= Hs) { c.off += Hs * tb; ++c.b; c.g = 0; continue; }
        if (p_lo >= hi) { ++c.s; c.b = c.g = c.off = 0; continue; }
        const int first = p_lo / per, last = (p_hi - 1) / per;
        set_item(a, c.s, c.b, c.g, n_ctx, max(lo, p_lo) - p_lo, min(hi, p_hi) - p_lo, c.range - first, last - first + 1, it);
        ++c.g;
        return true;
    }
    return false;
}
// The cut, by one warp: a lane per candidate k, and the even cut on the last lane.  Costs are summed over one-stream and
// two-stream layers, as the model has them, so that both kinds of launch choose alike.  (Per pair: 8 kv heads of one sequence,
// 17 tiles each: 9 ranges; 32 pairs: 4; 128 pairs on 148 CTAs: whole pairs, where an even cut would have two items and a
// merge per CTA.  Even: 160 pairs of 65 tiles.)
__device__ __forceinline__ void choose_cut(const AttnWork &a, int lane, Cut &cut, int &n_ranges) {
    int T = 0, tmax = 1;
    for (int b = lane; b < a.batch; b += 32) {
        const int tb = (a.len_eff[b] + a.M + TKEYS - 1) / TKEYS;
        T += tb;
        tmax = max(tmax, tb);
    }
    T = __reduce_add_sync(0xffffffffu, T) * a.Hkv * a.subs;
    tmax = __reduce_max_sync(0xffffffffu, tmax);
    const int G = gridDim.x, P = a.batch * a.Hkv * a.subs, kmax = max(1, min(MAX_SPLITS, a.slots)), k = lane + 1;
    // even cut: no pair in more ranges than it has slots
    const int per = a.slots < 2 ? T : max((T + G - 1) / G, (tmax + a.slots - 2) / (a.slots - 1)), ranges = (T + per - 1) / per;
    int cost = 1 << 26;
    if (k <= kmax && (a.splits == 0 || k == min(a.splits, kmax))) {
        const int item = (tmax + k - 1) / k + COST_ITEM, merge = k > 1 ? COST_MERGE : 0;
        cost = a.w_one * ((P * k + G - 1) / G * item + merge) + a.w_two * ((2 * P * k + G - 1) / G * item + merge);
    } else if (lane == 31 && a.splits == 0 && a.slots >= 2) {
        const int share = per + 2 * COST_ITEM;
        cost = a.w_one * (share + COST_MERGE) + a.w_two * ((2 * ranges <= G ? share : 2 * share) + COST_MERGE);
    }
    const unsigned best = __reduce_min_sync(0xffffffffu, ((unsigned)min(cost, 1 << 26) << 5) + lane) & 31u;
    cut.k = best == 31 ? 0 : (int)best + 1;
    cut.per = best == 31 ? per : (a.streams * P * ((int)best + 1) + G - 1) / G;
    n_ranges = ranges;
}
// A CTA that gave up (one thread): what it still owes the counters of its split pairs, `arrived` and `acked` of which it has
// counted in and out, so that they are zero for the next launch and the other CTAs do not wait for this one.
__device__ __forceinline__ void settle_counters(const AttnWork &a, const Cut &cut, int ranges, int arrived, int acked) {
    ItemSrc src;
    Item it;
    src_init(a, cut, ranges, src);
    for (int i = 0; next_item(a, cut, src, it); ) {
        if (it.n_split == 1) continue;
        if (i >= arrived) counter_arrive(a.counters + it.pair, it.n_split, it.n_split);
        if (i >= acked) counter_ack(a.counters + it.pair, it.n_split, it.n_split);
        ++i;
    }
}
// a query row's place in q and in the output
__device__ __forceinline__ size_t row_off(const AttnWork &a, const Item &i, int r) {
    const int g2 = i.row0 + r, hq = (int)((g2 * a.m_recip) >> 32);
    return ((size_t)(i.be * a.M + g2 - hq * a.M) * a.H + i.kvh * (a.H / a.Hkv) + hq) * HD;
}
// x0, x1 -> packed bf16 pairs hi = bf16(x), lo = bf16(x - hi); the low half word is the even element
__device__ __forceinline__ void split_pair(float x0, float x1, uint32_t &hi, uint32_t &lo) {
    const __nv_bfloat162 h = __floats2bfloat162_rn(x0, x1);
    hi = *reinterpret_cast<const uint32_t *>(&h);
    const __nv_bfloat162 l = __floats2bfloat162_rn(x0 - __uint_as_float(hi << 16), x1 - __uint_as_float(hi & 0xffff0000u));
    lo = *reinterpret_cast<const uint32_t *>(&l);
}

// everything but the rows of an item; floats of a partial slot: rows8 rows
inline void fill_work(const viasd_model *m, AttnWork &a, int layer_ord, int layer_ord2, int streams, int batch, int M) {
    const viasd_config &c = m->cfg;
    a.rows8 = (a.rows_sub + 7) / 8 * 8;
    a.q = m->ws.q; a.part = m->ws.part; a.out = (__nv_bfloat16 *)m->ws.attn;
    a.out_plane = m->ws.rows_alloc * (size_t)c.n_heads * HD;
    a.len_eff = m->ws.len_eff; a.tree = m->ws.tree; a.status = &m->ws.stats->device_status; a.run_flag = m->run_flag;
    a.M = M; a.H = c.n_heads; a.Hkv = c.n_kv_heads; a.max_batch = c.max_batch; a.max_ctx = c.max_ctx;
    a.layer_ord = layer_ord; a.scale = 1.4426950408889634f / sqrtf((float)HD);   // log2(e) / sqrt(hd)
    a.batch = batch; a.layer_ord2 = layer_ord2; a.streams = streams;
    a.counters = m->ws.attn_counters;
    // (always counted for two streams: the cuts must not depend on how many a launch has)
    const size_t slot_bytes = (size_t)2 * batch * c.n_kv_heads * a.subs * a.rows8 * PART_ROW * sizeof(float);
    const size_t fit = m->ws.part_bytes / slot_bytes;
    a.slots = fit > MAX_SLOTS ? MAX_SLOTS : (int)fit;
    a.splits = m->opt.attn_splits;
    a.w_one = c.n_layers - m->n_routed; a.w_two = m->n_routed;
    a.m_recip = ((1ull << 32) + M - 1) / M;
}
inline int work_grid(const viasd_model *m) {           // (the option: tests, long ranges per CTA on small cases)
    return m->opt.tk_grid >= 1 && m->opt.tk_grid < m->sm_count ? m->opt.tk_grid : m->sm_count;
}

}  // namespace
