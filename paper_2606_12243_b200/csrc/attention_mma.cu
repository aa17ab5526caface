// Block attention for up to 16 query rows per kv head and few tiles per CTA: mma.sync, K/V tiles staged by TMA.
//
// The query rows of a (sequence, kv head) are the G = H / Hkv query heads of that kv head times the M block rows, one 16-row
// MMA tile, so every K/V byte is read once for all of them.  Keys are the committed cache rows 0..n-1 plus the M block rows at
// slots n..n+M-1, the latter masked per query row by its ancestor bit set (causal for a chain, tree mask otherwise).
//
// What bounds it is a chain of latencies: queries from L2 (1000 cycles), S, softmax, P V per step, the merge of the warps and
// of the key ranges, a trip to L2 each way.  So the chain is kept short: a tile of 128 keys goes to four warps, 32 keys each,
// odd and even tiles to different warps, every warp on its own mbarriers with no step in common; the query fragments come
// straight from global memory; the warps are merged in one pass through shared memory; the ranges by a slice of the rows
// per CTA.  (With a CTA barrier on both sides of every tile, 16 keys per warp, the queries staged through shared memory,
// the warps merged pairwise and one CTA merging all ranges, 9 rows against 1033 keys took 27700 cycles from the dependency on.)
//
// Q is used as a bf16 hi + lo pair, and so is P, so that only the cache itself is bf16; fp32 accumulation.
// Split of the work: attention_work.cuh.  Partial rows: [rows8][128], then [rows8] (max, sum).
// Warp roles (288 threads): warps 0-7 compute, warp 8 requests K and V tiles (2-D TMA boxes of 64 dims x 128 keys, 128-byte
// swizzle) into a ring that runs across the CTA's items; tiles that lie wholly inside the committed context are requested
// before the kernel waits for its predecessor.  Every wait is bounded.
#include "common.cuh"
#include "attention_work.cuh"
#include "tc_ptx.cuh"
#include <stdlib.h>

namespace {

constexpr int WARPS = 8;
// Slots of one K or V tile; beside them the merge buffer's 64 KB.  Even and odd tiles go to different groups of warps with
// no step in common, and a parity wait is only good for a warp that has waited for the slot's use before: so every use of
// a slot belongs to one group.  (With five slots tile 3's K had the slot of tile 0's V: had that V landed after tile 1, the odd
// group would have taken it for its K.)
constexpr int RING = 4;
static_assert(RING % 4 == 0, "a slot's uses alternate between the groups of warps");

__device__ __forceinline__ void ldsm_x4(uint32_t addr, uint32_t (&r)[4]) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr));
}
__device__ __forceinline__ void ldsm_x4_t(uint32_t addr, uint32_t (&r)[4]) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr));
}
__device__ __forceinline__ void mma16816(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
// byte offset of (row, 16-byte chunk) in a 128-byte-swizzled tile whose rows are 128 bytes
__device__ __forceinline__ uint32_t sw128(int row, int chunk) { return (uint32_t)row * 128u + (uint32_t)((chunk ^ (row & 7)) << 4); }

// 32 keys of a tile against the query rows: one warp's step.  m, l, o: its running state (rows g and g + 8)
template <bool PLO, bool QLO>
struct Step {
    uint32_t qh[8][4];                          // the query rows as MMA A fragments, hi part; the lo part is in shared memory
    float m[2], l[2], o[16][4];

    __device__ __forceinline__ void scores(uint32_t kst, const uint4 *ql_sh, int r0, int lane, float (&s)[4][4]) {
        float t[4][4];                          // products with the lo part: a chain of their own
#pragma unroll
        for (int n = 0; n < 4; ++n)
#pragma unroll
            for (int e = 0; e < 4; ++e) s[n][e] = t[n][e] = 0.f;
        const int krow = r0 + (lane & 7) + ((lane >> 4) & 1) * 8;
#pragma unroll
        for (int ks = 0; ks < 8; ++ks) {        // dims 0..63 in the first half tile, 64..127 in the second
            uint32_t b[2][4], ql[4];
            if (QLO) { const uint4 x = ql_sh[ks * 32]; ql[0] = x.x; ql[1] = x.y; ql[2] = x.z; ql[3] = x.w; }
#pragma unroll
            for (int np = 0; np < 2; ++np) ldsm_x4(kst + (ks >> 2) * HALF_BYTES + sw128(krow + np * 16, (ks & 3) * 2 + ((lane >> 3) & 1)), b[np]);
#pragma unroll
            for (int np = 0; np < 2; ++np) {
                mma16816(s[np * 2], qh[ks], b[np][0], b[np][1]);
                mma16816(s[np * 2 + 1], qh[ks], b[np][2], b[np][3]);
                if (QLO) { mma16816(t[np * 2], ql, b[np][0], b[np][1]); mma16816(t[np * 2 + 1], ql, b[np][2], b[np][3]); }
            }
        }
#pragma unroll
        for (int n = 0; n < 4; ++n)
#pragma unroll
            for (int e = 0; e < 4; ++e) s[n][e] += t[n][e];
    }
    // online softmax (columns 8n + 2t, 8n + 2t + 1; log2 units)
    __device__ __forceinline__ void softmax(float (&s)[4][4]) {
        float mx[2] = {-INFINITY, -INFINITY}, corr[2], rs[2] = {0.f, 0.f}, ref[2];
#pragma unroll
        for (int n = 0; n < 4; ++n)
#pragma unroll
            for (int e = 0; e < 4; ++e) mx[e >> 1] = fmaxf(mx[e >> 1], s[n][e]);
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            mx[r] = fmaxf(mx[r], __shfl_xor_sync(0xffffffffu, mx[r], 1));
            mx[r] = fmaxf(mx[r], __shfl_xor_sync(0xffffffffu, mx[r], 2));
            const float mnew = fmaxf(m[r], mx[r]);
            corr[r] = (mnew == -INFINITY) ? 1.f : ex2(m[r] - mnew);
            m[r] = mnew;
            ref[r] = mnew == -INFINITY ? 0.f : mnew;                       // no visible key yet: every weight is 2^-inf
        }
#pragma unroll
        for (int n = 0; n < 4; ++n)
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                float p = ex2(s[n][e] - ref[e >> 1]);
                // without the lo part the MMA sees bf16(p): normalise by the sum of those same rounded values, or the
                // rounding of near-equal weights would not cancel
                if (!PLO) p = __bfloat162float(__float2bfloat16_rn(p));
                s[n][e] = p;
                rs[e >> 1] += p;
            }
#pragma unroll
        for (int r = 0; r < 2; ++r) l[r] = l[r] * corr[r] + rs[r];         // (summed over the four lanes of a row at the end)
        if (__any_sync(0xffffffffu, corr[0] != 1.f || corr[1] != 1.f)) {    // the running maximum moved: rescale
#pragma unroll
            for (int n = 0; n < 16; ++n) { o[n][0] *= corr[0]; o[n][1] *= corr[0]; o[n][2] *= corr[1]; o[n][3] *= corr[1]; }
        }
    }
    // O += P V: k-steps of 16 keys, 16 n-tiles of 8 dims; hi and lo part of P against each V fragment
    __device__ __forceinline__ void accumulate(uint32_t vst, int r0, int lane, const float (&s)[4][4]) {
#pragma unroll
        for (int ks = 0; ks < 2; ++ks) {
            uint32_t ph[4], pl[4];
            split_pair(s[2 * ks][0], s[2 * ks][1], ph[0], pl[0]);
            split_pair(s[2 * ks][2], s[2 * ks][3], ph[1], pl[1]);
            split_pair(s[2 * ks + 1][0], s[2 * ks + 1][1], ph[2], pl[2]);
            split_pair(s[2 * ks + 1][2], s[2 * ks + 1][3], ph[3], pl[3]);
            const int vrow = r0 + ks * 16 + (lane & 7) + ((lane >> 3) & 1) * 8;
#pragma unroll
            for (int np = 0; np < 8; ++np) {    // two n-tiles (16 dims) per ldmatrix.x4.trans
                uint32_t b[4];
                const int dchunk = np * 2 + (lane >> 4);             // 16-byte chunk of the 128 dims
                ldsm_x4_t(vst + (dchunk >> 3) * HALF_BYTES + sw128(vrow, dchunk & 7), b);
                mma16816(o[np * 2], ph, b[0], b[1]);
                mma16816(o[np * 2 + 1], ph, b[2], b[3]);
                if (PLO) { mma16816(o[np * 2], pl, b[0], b[1]); mma16816(o[np * 2 + 1], pl, b[2], b[3]); }
            }
        }
    }
};

// four normalised values of an output row as hi and lo planes
__device__ __forceinline__ void store_row(const AttnWork &a, size_t at, float4 v, float inv) {
    uint2 hi, lo;
    split_pair(v.x * inv, v.y * inv, hi.x, lo.x);
    split_pair(v.z * inv, v.w * inv, hi.y, lo.y);
    *reinterpret_cast<uint2 *>(a.out + at) = hi;
    *reinterpret_cast<uint2 *>(a.out + a.out_plane + at) = lo;
}

// PLO / QLO: use the lo parts of the probabilities / of the query too
template <bool PLO, bool QLO>
__global__ void __launch_bounds__(WARPS * 32 + 32, 1)
attention_mma_kernel(const __grid_constant__ CUtensorMap map_k, const __grid_constant__ CUtensorMap map_v,
                     const __grid_constant__ CUtensorMap map_k2, const __grid_constant__ CUtensorMap map_v2, const AttnWork a) {
    extern __shared__ uint8_t smem_raw[];
    __shared__ __align__(8) unsigned long long bars[2 * RING + 1];
    __shared__ int abort_sh, ranges_sh;
    __shared__ Cut cut_sh;
    __shared__ float2 ml_sh[WARPS][16];                 // per warp: a row's maximum and sum
    RUN_FLAG_EXIT(a.run_flag);
    PDL_TRIGGER();
    const int warp = uniform(threadIdx.x >> 5), lane = threadIdx.x & 31;
    const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    float *osm = reinterpret_cast<float *>(smem_raw + (base - smem_u32(smem_raw)) + RING * SLOT_BYTES);   // [warp][row][128 dims]
    auto full_bar = [&](int s) { return smem_u32(&bars[s]); };
    auto empty_bar = [&](int s) { return smem_u32(&bars[RING + s]); };
    const uint32_t wg_bar = smem_u32(&bars[2 * RING]);
    if (threadIdx.x == 0) {
        for (int s = 0; s < RING; ++s) { mbar_init(full_bar(s), 1); mbar_init(empty_bar(s), 4); }
        mbar_init(wg_bar, WARPS);
        abort_sh = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == 1) {
        Cut c;
        int n;
        choose_cut(a, lane, c, n);
        if (lane == 0) { cut_sh = c; ranges_sh = n; }
    }
    __syncthreads();
    const Cut cut{uniform(cut_sh.k), uniform(cut_sh.per)};
    const int ranges = uniform(ranges_sh);
    ItemSrc src;
    src_init(a, cut, ranges, src);
    Item it;

    if (warp == WARPS) {
        // ---------------- TMA producer: K and V of the CTA's tiles in turn ----------------
        if (elect_one()) {
            const uint64_t kvpol = l2_evict_first_policy();    // the cache passes through once per layer
            int j = 0, count = 0;
            bool ok = true, more = next_item(a, cut, src, it);
            auto issue_next = [&](bool context_only) -> bool {  // false: nothing (more) to request under this condition
                if (more && j >= 2 * it.n_tiles) { j = 0; more = next_item(a, cut, src, it); }
                if (!more) return false;
                const int k0 = it.k_begin + (j >> 1) * TKEYS;
                if (context_only && k0 + TKEYS > it.n_ctx) return false;   // this tile holds rows the previous kernel writes
                const int st = count % RING;
                if (count >= RING && !(ok = mbar_wait(empty_bar(st), ((count / RING) & 1) ^ 1, &abort_sh, a.status))) return false;
                const uint32_t dst = base + st * SLOT_BYTES;
                const CUtensorMap *mp = j & 1 ? (it.stream ? &map_v2 : &map_v) : (it.stream ? &map_k2 : &map_k);
                mbar_expect_tx(full_bar(st), SLOT_BYTES);
                tma_load_2d_hint(dst, mp, full_bar(st), 0, it.row_base + k0, kvpol);
                tma_load_2d_hint(dst + HALF_BYTES, mp, full_bar(st), 64, it.row_base + k0, kvpol);
                ++j; ++count;
                return true;
            };
            // committed context does not change during the pass: ask for it before waiting for the previous kernel
            while (count < RING && issue_next(true)) { }
            PDL_WAIT();
            while (ok && issue_next(false)) { }
        }
    } else {
        const int g = lane >> 2, t2 = (lane & 3) * 2, r0 = (warp & 3) * 32;   // rows g, g + 8; first column; this warp's keys of its tiles
        const size_t part_floats = (size_t)a.rows8 * PART_ROW;
        int c_tile = 0, wg_phase = 0, n_item = 0, arrived = 0, acked = 0;   // c_tile: tiles of earlier items
        bool ok = true;
        auto wg_sync = [&]() -> bool {
            __syncwarp();
            if (lane == 0) mbar_arrive(wg_bar);
            return warp_wait(wg_bar, wg_phase++ & 1, &abort_sh, a.status);
        };
        Step<PLO, QLO> st;
        uint4 *ql_sh = reinterpret_cast<uint4 *>(osm + warp * 16 * HD) + lane;   // the lo fragments, where the warp's state will go
        while (ok && next_item(a, cut, src, it)) {
            const float *qrow[2];
            unsigned long long anc[2];
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                const int row = min(g + 8 * i, it.rows - 1);     // rows past the end repeat the last one, unstored
                qrow[i] = a.q + row_off(a, it, row) + t2;
                anc[i] = a.tree[it.b].anc[row - (int)((row * a.m_recip) >> 32) * a.M];
            }
            if (n_item == 0) PDL_WAIT();
            else if (!(ok = wg_sync())) break;                   // the previous item's states have been read
            ++n_item;
#pragma unroll
            for (int h = 0; h < 2; ++h) {                        // half of the dims at a time: 16 loads in flight
                float2 v[4][4];
#pragma unroll
                for (int ks = 0; ks < 4; ++ks)
#pragma unroll
                    for (int e = 0; e < 4; ++e) v[ks][e] = __ldcg(reinterpret_cast<const float2 *>(qrow[e & 1] + (4 * h + ks) * 16 + (e >> 1) * 8));
#pragma unroll
                for (int ks = 0; ks < 4; ++ks) {
                    uint32_t lo[4];
#pragma unroll
                    for (int e = 0; e < 4; ++e) split_pair(v[ks][e].x * a.scale, v[ks][e].y * a.scale, st.qh[4 * h + ks][e], lo[e]);
                    ql_sh[(4 * h + ks) * 32] = make_uint4(lo[0], lo[1], lo[2], lo[3]);
                }
            }
            st.m[0] = st.m[1] = -INFINITY;
            st.l[0] = st.l[1] = 0.f;
#pragma unroll
            for (int n = 0; n < 16; ++n)
#pragma unroll
                for (int e = 0; e < 4; ++e) st.o[n][e] = 0.f;

            // odd and even tiles of the CTA go to different warps
            for (int t = ((c_tile & 1) ^ (warp >> 2)); t < it.n_tiles; t += 2) {
                const int ck = 2 * (c_tile + t), ks = ck % RING, vs = (ck + 1) % RING;
                const int j0 = it.k_begin + t * TKEYS + r0;
                const bool any = j0 < it.k_end;
                if (!(ok = warp_wait(full_bar(ks), (ck / RING) & 1, &abort_sh, a.status))) break;
                float s[4][4];
                if (any) {
                    st.scores(base + ks * SLOT_BYTES, ql_sh, r0, lane, s);
                    if (j0 + 32 > it.n_ctx || j0 + 32 > it.k_end) {
#pragma unroll
                        for (int n = 0; n < 4; ++n)
#pragma unroll
                            for (int e = 0; e < 4; ++e) {
                                const int j = j0 + n * 8 + t2 + (e & 1);
                                if (!(j < it.k_end && (j < it.n_ctx || ((anc[e >> 1] >> (j - it.n_ctx)) & 1ull)))) s[n][e] = -INFINITY;
                            }
                    }
                    st.softmax(s);
                }
                __syncwarp();
                if (lane == 0) mbar_arrive(empty_bar(ks));
                if (!(ok = warp_wait(full_bar(vs), ((ck + 1) / RING) & 1, &abort_sh, a.status))) break;
                if (any) {
                    if (j0 + 32 > it.k_end) zero_tile_rows(base + vs * SLOT_BYTES, HALF_BYTES, r0 + it.k_end - j0, r0 + 32, lane);   // (this warp's keys)
                    st.accumulate(base + vs * SLOT_BYTES, r0, lane, s);
                }
                __syncwarp();
                if (lane == 0) mbar_arrive(empty_bar(vs));
            }
            if (!ok) break;
            c_tile += it.n_tiles;

            // ---- the item's result: the warps' states through shared memory, columns swizzled against bank conflicts ----
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                float l = st.l[i];
                l += __shfl_xor_sync(0xffffffffu, l, 1);
                l += __shfl_xor_sync(0xffffffffu, l, 2);
                const int row = g + 8 * i;
                if (row >= it.rows) continue;
                if ((lane & 3) == 0) ml_sh[warp][row] = make_float2(st.m[i], l);
                float *dst = osm + (warp * 16 + row) * HD;
#pragma unroll
                for (int n = 0; n < 16; ++n)
                    *reinterpret_cast<float2 *>(dst + ((n * 8 + t2) ^ ((row & 3) << 3))) = make_float2(st.o[n][2 * i], st.o[n][2 * i + 1]);
            }
            if (!(ok = wg_sync())) break;
            const bool single = it.n_split == 1;
            float *pdst = a.part + ((size_t)it.pair * a.slots + it.split) * part_floats;
#pragma unroll 1
            for (int row = warp; row < it.rows; row += WARPS) {  // a row per warp, four dims per lane
                float m = -INFINITY, l = 0.f;
#pragma unroll
                for (int w = 0; w < WARPS; ++w) m = fmaxf(m, ml_sh[w][row].x);
                const float ref = m == -INFINITY ? 0.f : m;
                float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                for (int w = 0; w < WARPS; ++w) {
                    const float2 ml = ml_sh[w][row];
                    const float f = ex2(ml.x - ref);
                    const float4 x = *reinterpret_cast<const float4 *>(osm + (w * 16 + row) * HD + ((4 * lane) ^ ((row & 3) << 3)));
                    l = fmaf(ml.y, f, l);
                    v.x = fmaf(x.x, f, v.x); v.y = fmaf(x.y, f, v.y); v.z = fmaf(x.z, f, v.z); v.w = fmaf(x.w, f, v.w);
                }
                if (single) {
                    store_row(a, row_off(a, it, row) + 4 * lane, v, 1.f / l);
                } else {
                    *reinterpret_cast<float4 *>(pdst + row * HD + 4 * lane) = v;
                    if (lane == 0) *reinterpret_cast<float2 *>(pdst + (size_t)a.rows8 * HD + 2 * row) = make_float2(m, l);
                }
            }
            if (!single) {
                if (!(ok = wg_sync())) break;
                // (the barrier orders the group's stores before this thread's release, which is cumulative)
                if (threadIdx.x == 0) counter_arrive(a.counters + it.pair, it.n_split, it.n_split);
                ++arrived;
            }
        }
        // ---- the split pairs of this CTA's list: its slice of each one's rows ----
        src_init(a, cut, ranges, src);
        while (ok && next_item(a, cut, src, it)) {
            if (it.n_split == 1) continue;
            if (threadIdx.x == 0) counter_wait(a.counters + it.pair, it.n_split, it.n_split, &abort_sh, a.status);
            ++acked;
            if (!(ok = wg_sync())) break;
            const int rper = (it.rows + it.n_split - 1) / it.n_split, r_end = min(it.rows, (it.split + 1) * rper);
            const float *psrc = a.part + (size_t)it.pair * a.slots * part_floats;
#pragma unroll 1
            for (int row = it.split * rper + warp; row < r_end; row += WARPS) {
                // lane s holds range s's maximum and sum; the weights go round by shuffle
                float2 ml = make_float2(-INFINITY, 0.f);
                if (lane < it.n_split) ml = __ldcg(reinterpret_cast<const float2 *>(psrc + (size_t)lane * part_floats + (size_t)a.rows8 * HD + 2 * row));
                float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
                float w = 0.f, inv = 0.f;
#pragma unroll 1
                for (int s0 = 0; s0 < it.n_split; s0 += 4) {
                    float4 x[4];
#pragma unroll
                    for (int s = 0; s < 4; ++s)
                        x[s] = s0 + s < it.n_split ? __ldcg(reinterpret_cast<const float4 *>(psrc + (size_t)(s0 + s) * part_floats + row * HD + 4 * lane))
                                                   : make_float4(0.f, 0.f, 0.f, 0.f);
                    if (s0 == 0) {
                        w = ex2(ml.x - warp_max(ml.x));                          // (every row sees at least itself: finite)
                        inv = 1.f / warp_sum(ml.y * w);
                    }
#pragma unroll
                    for (int s = 0; s < 4; ++s) {
                        const float f = __shfl_sync(0xffffffffu, w, (s0 + s) & 31);
                        v.x = fmaf(x[s].x, f, v.x); v.y = fmaf(x[s].y, f, v.y); v.z = fmaf(x[s].z, f, v.z); v.w = fmaf(x[s].w, f, v.w);
                    }
                }
                store_row(a, row_off(a, it, row) + 4 * lane, v, inv);
            }
        }
        if (!ok && threadIdx.x == 0) settle_counters(a, cut, ranges, arrived, acked);
    }
    __syncwarp();
    if (abort_sh && threadIdx.x == 0) {
        // give copies that are still in flight time to land before shared memory goes away
        const long long t0 = clock64();
        while (clock64() - t0 < 400000) { }
    }
    __syncthreads();
}

}  // namespace

int attention_tensor_supported(const viasd_model *m) { return m->cfg.dtype == 1 && m->cfg.head_dim == HD && m->use_tc; }
int attention_mma_supported(const viasd_model *m, int M) {
    const viasd_config &c = m->cfg;
    return c.dtype == 1 && c.head_dim == HD && (c.n_heads / c.n_kv_heads) * M <= 16 && m->use_tc;
}

int attention_cache_maps(const viasd_model *m, CacheMaps &cm, const void *kc, const void *vc, int n_layers) {
    if (cm.k_ptr == kc && cm.v_ptr == vc) return VIASD_OK;
    const viasd_config &c = m->cfg;
    const uint64_t rows = (uint64_t)n_layers * c.max_batch * c.n_kv_heads * c.max_ctx;
    int rc;
    if ((rc = tc_make_map(&cm.k, kc, rows, HD, TKEYS))) return rc;
    if ((rc = tc_make_map(&cm.v, vc, rows, HD, TKEYS))) return rc;
    cm.k_ptr = kc; cm.v_ptr = vc;
    return VIASD_OK;
}

// streams = 1: one cache (full or slim).  streams = 2: rows [0, batch*M) against the full cache at layer_ord and
// rows [batch*M, 2*batch*M) against the slim cache at layer_ord2, in one launch.
int launch_attention_mma(viasd_model *m, const void *kc, const void *vc, bool slim, int layer_ord, const void *kc2,
                         const void *vc2, int layer_ord2, int streams, int batch, int M, cudaStream_t st) {
    const viasd_config &c = m->cfg;
    if (!attention_mma_supported(m, M)) return VIASD_EINVAL;
    CacheMaps &cm = slim ? m->cmaps_slim : m->cmaps_full;
    int rc;
    if ((rc = attention_cache_maps(m, cm, kc, vc, slim ? m->n_routed : c.n_layers))) return rc;
    CacheMaps *cm2 = &cm;
    if (streams == 2) {
        cm2 = &m->cmaps_slim;
        if ((rc = attention_cache_maps(m, *cm2, kc2, vc2, m->n_routed))) return rc;
    }
    AttnWork a;
    a.subs = 1;
    a.rows_sub = (c.n_heads / c.n_kv_heads) * M;
    a.ring_slots = RING;
    fill_work(m, a, layer_ord, layer_ord2, streams, batch, M);
    const size_t smem = 1024 + (size_t)RING * SLOT_BYTES + (size_t)WARPS * 16 * HD * sizeof(float);
    static std::atomic<bool> attr_done[64];
    if (int rc = once_on_device(attr_done, [&]() -> int {
        CUDA_TRY(cudaFuncSetAttribute(attention_mma_kernel<true, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
        CUDA_TRY(cudaFuncSetAttribute(attention_mma_kernel<false, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
        CUDA_TRY(cudaFuncSetAttribute(attention_mma_kernel<false, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
        return VIASD_OK;
    })) return rc;
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attr[1];
    pdl_config(cfg, attr, dim3(work_grid(m)), dim3(WARPS * 32 + 32), smem, st);
    const int lo_mode = m->opt.attn_lo;      // 2 = hi/lo for Q and P, 1 = hi/lo for Q only, 0 = plain bf16
    if (lo_mode >= 2) CUDA_TRY(cudaLaunchKernelEx(&cfg, attention_mma_kernel<true, true>, cm.k, cm.v, cm2->k, cm2->v, a));
    else if (lo_mode == 1) CUDA_TRY(cudaLaunchKernelEx(&cfg, attention_mma_kernel<false, true>, cm.k, cm.v, cm2->k, cm2->v, a));
    else CUDA_TRY(cudaLaunchKernelEx(&cfg, attention_mma_kernel<false, false>, cm.k, cm.v, cm2->k, cm2->v, a));
    LAUNCH_CHECK();
    return VIASD_OK;
}
