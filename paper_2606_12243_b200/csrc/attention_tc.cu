// Block attention on the 5th-generation tensor cores (tcgen05 + TMEM), bf16 caches, head_dim 128: query rows on the lanes.
//
// The M block rows of a sequence under all query heads of one kv head (dealt to items of at most 128 rows) against the
// committed context plus the block's own rows under the ancestor mask:
//
//   S[rows, 128 keys] = Q K^T      A = Q (shared memory, K-major, 2 or 3 bf16 planes: an MMA each into one S)
//                                  B = K tile exactly as its TMA box lands (K-major, 128-byte swizzle)
//   O[rows, 128 dims] += P V       A = P in TMEM (bf16 pairs, as many planes: an MMA each into one O)
//                                  B = V tile as it lands, read MN-major (keys are the contraction)
//
// Precision.  Up to 128 query rows per kv head queries and weights are bf16 pairs, as in the other two kernels; more rows
// belonged to an fp32 kernel, and three planes hold all of an fp32 value.  O is summed over the tiles in fp32 outside the MMAs
// (GROUP).  Error of the output against 64 bits, before / now: fp32 kernel / three planes 2.56 - 2.84e-6 / 2.53 - 2.56e-6
// (132 to 256 rows, 348 to 4033 keys), mma.sync / two planes 5.1 - 5.3e-6 / 5.0 - 5.1e-6 (36 to 108 rows); most of it is the
// output itself, which is stored as a bf16 pair.
//
// What bounds it: 32 (48) MMAs of 128 x 128 x 16 per tile, about 2300 (3200) cycles whatever the rows (so it is for 33 rows
// and more; fewer go to the kernels that put the keys on the lanes or use mma.sync), and with a few tiles per CTA the chain
// around them: queries, first S, softmax, last P V, result, merge.  Keeping the precision costs 0 - 3 % of a layer with a small
// feed-forward at two planes, 4 - 12 % at three (eight sequences, 33 rows each, 4000 keys: 206 us a layer, now 231; the fp32
// kernel took 2230).
//
// One TMEM lane is one query row; two warps share a lane quarter and take 64 of a tile's 128 keys each, exchanging row
// maxima once per tile.  The running maximum only moves when a tile exceeds it by 2^8 (the weights stay below 2^8
// otherwise, harmless in fp32), which makes rescaling O rare.  P overwrites S in place (per 16 keys 8
// columns of bf16 pairs hi, 8 of the next plane), two buffers; MMAs run in issue order, which is what lets Q K^T of tile t + 2
// reuse the buffer that P V of tile t reads.  The last tile of a range multiplies only the 16-key groups that it has.
//
// Split of the work: attention_work.cuh.  Partial rows: [32 groups of 4 dims][rows8] float4, then [rows8] (max, sum).
//
// Warp roles (320 threads): warp 0 requests K and V tiles by TMA into a ring that runs across the CTA's items, in the
// order the MMAs use them, warp 1 owns TMEM and issues the MMAs, warps 2-9 stage Q, run the softmax and write the result.
// Every wait is bounded: on expiry the CTA records VIASD_EDEVICE, lets its copies land and leaves.
#include "common.cuh"
#include "attention_work.cuh"
#include "tc_ptx.cuh"
#include <stdlib.h>

namespace {

constexpr int SW = 8;                          // softmax warps
constexpr int AT_THREADS = 64 + SW * 32;
constexpr int AT_MAX_SLOTS = 6;
constexpr int QROWS = 128 / SW;                // query rows a warp stages at most
// Tiles whose P V the tensor cores add up in one accumulator, before it is added to the item's sum in fp32 (rounded; what an
// MMA adds is cut off, so a sum over all tiles drifts towards zero: 36 rows against 1000 keys, error of the attention output
// 5.9e-6 over all tiles, 5.1e-6 with two, 5.0e-6 with one, where every added tile waits for the one before it to be read).
template <int PLANES> constexpr int GROUP = PLANES == 3 ? 1 : 2;
constexpr float RESCALE_GAP = 8.f;             // log2 units

constexpr uint32_t TM_S = 0, TM_O = 256, TM_X = 384;   // TMEM columns: S / P buffers (2 x 128), O of one tile (128), and the
                                                             // sum of the tiles' O (128), or third planes of P (2 x 64)

// The j-th of an item's 2 n requests, in the order the MMAs take them: K0 K1 V0 K2 V1 ... K(n-1) V(n-2) V(n-1)
__device__ __forceinline__ int request_tile(int j, int n, bool &is_v) {
    is_v = false;
    if (j == 0) return 0;
    if (j == 1) { is_v = n == 1; return n == 1 ? 0 : 1; }
    if ((j & 1) && (j + 1) / 2 < n) return (j + 1) / 2;
    is_v = true;
    return (j & 1) ? n - 1 : (j - 2) / 2;
}

// MN-major operand tile with the 128-byte swizzle: 64 contiguous elements along MN per row of 128 bytes,
// 8 rows (8 steps of the contraction) per 1024-byte group; groups `sbo` bytes apart along the contraction,
// 64-element blocks `lbo` bytes apart along MN.
__device__ __forceinline__ uint64_t smem_desc_mn(uint32_t addr, uint32_t lbo, uint32_t sbo) {
    return (uint64_t)((addr >> 4) & 0x3FFF) | ((uint64_t)((lbo >> 4) & 0x3FFF) << 16) | ((uint64_t)((sbo >> 4) & 0x3FFF) << 32) |
           (1ull << 46) | (2ull << 61);
}

// D[tmem] (+)= A[tmem] * B[smem]
__device__ __forceinline__ void tc_mma_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc, uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
        ::"r"(d_tmem), "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(accumulate) : "memory");
}

__device__ __forceinline__ void tc_ld32(uint32_t taddr, uint32_t (&r)[32]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];\n\t"
        "tcgen05.wait::ld.sync.aligned;"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]),
          "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]),
          "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]),
          "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr) : "memory");
}
// 32 columns from each of two places under one wait
__device__ __forceinline__ void tc_ld32x2(uint32_t ta, uint32_t tb, uint32_t (&r)[32], uint32_t (&s)[32]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
        : "=r"(r[0]),"=r"(r[1]),"=r"(r[2]),"=r"(r[3]),"=r"(r[4]),"=r"(r[5]),"=r"(r[6]),"=r"(r[7]),
          "=r"(r[8]),"=r"(r[9]),"=r"(r[10]),"=r"(r[11]),"=r"(r[12]),"=r"(r[13]),"=r"(r[14]),"=r"(r[15]),
          "=r"(r[16]),"=r"(r[17]),"=r"(r[18]),"=r"(r[19]),"=r"(r[20]),"=r"(r[21]),"=r"(r[22]),"=r"(r[23]),
          "=r"(r[24]),"=r"(r[25]),"=r"(r[26]),"=r"(r[27]),"=r"(r[28]),"=r"(r[29]),"=r"(r[30]),"=r"(r[31])
        : "r"(ta));
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
        : "=r"(s[0]),"=r"(s[1]),"=r"(s[2]),"=r"(s[3]),"=r"(s[4]),"=r"(s[5]),"=r"(s[6]),"=r"(s[7]),
          "=r"(s[8]),"=r"(s[9]),"=r"(s[10]),"=r"(s[11]),"=r"(s[12]),"=r"(s[13]),"=r"(s[14]),"=r"(s[15]),
          "=r"(s[16]),"=r"(s[17]),"=r"(s[18]),"=r"(s[19]),"=r"(s[20]),"=r"(s[21]),"=r"(s[22]),"=r"(s[23]),
          "=r"(s[24]),"=r"(s[25]),"=r"(s[26]),"=r"(s[27]),"=r"(s[28]),"=r"(s[29]),"=r"(s[30]),"=r"(s[31])
        : "r"(tb));
    // (an empty statement per half names the registers: no use of them is scheduled ahead of the wait)
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
    asm volatile("" : "+r"(r[0]),"+r"(r[1]),"+r"(r[2]),"+r"(r[3]),"+r"(r[4]),"+r"(r[5]),"+r"(r[6]),"+r"(r[7]),
          "+r"(r[8]),"+r"(r[9]),"+r"(r[10]),"+r"(r[11]),"+r"(r[12]),"+r"(r[13]),"+r"(r[14]),"+r"(r[15]),
          "+r"(r[16]),"+r"(r[17]),"+r"(r[18]),"+r"(r[19]),"+r"(r[20]),"+r"(r[21]),"+r"(r[22]),"+r"(r[23]),
          "+r"(r[24]),"+r"(r[25]),"+r"(r[26]),"+r"(r[27]),"+r"(r[28]),"+r"(r[29]),"+r"(r[30]),"+r"(r[31]));
    asm volatile("" : "+r"(s[0]),"+r"(s[1]),"+r"(s[2]),"+r"(s[3]),"+r"(s[4]),"+r"(s[5]),"+r"(s[6]),"+r"(s[7]),
          "+r"(s[8]),"+r"(s[9]),"+r"(s[10]),"+r"(s[11]),"+r"(s[12]),"+r"(s[13]),"+r"(s[14]),"+r"(s[15]),
          "+r"(s[16]),"+r"(s[17]),"+r"(s[18]),"+r"(s[19]),"+r"(s[20]),"+r"(s[21]),"+r"(s[22]),"+r"(s[23]),
          "+r"(s[24]),"+r"(s[25]),"+r"(s[26]),"+r"(s[27]),"+r"(s[28]),"+r"(s[29]),"+r"(s[30]),"+r"(s[31]));
}
__device__ __forceinline__ void tc_st32(uint32_t taddr, const uint32_t (&r)[32]) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], "
        "{%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31,%32};"
        ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]),
          "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]), "r"(r[16]), "r"(r[17]), "r"(r[18]), "r"(r[19]),
          "r"(r[20]), "r"(r[21]), "r"(r[22]), "r"(r[23]), "r"(r[24]), "r"(r[25]), "r"(r[26]), "r"(r[27]), "r"(r[28]), "r"(r[29]),
          "r"(r[30]), "r"(r[31])
        : "memory");
}
// x0, x1 -> three packed bf16 pairs whose sums are x0 and x1 to the last bit of fp32
__device__ __forceinline__ void split_triple(float x0, float x1, uint32_t &hi, uint32_t &mid, uint32_t &lo) {
    const __nv_bfloat162 h = __floats2bfloat162_rn(x0, x1);
    hi = *reinterpret_cast<const uint32_t *>(&h);
    split_pair(x0 - __uint_as_float(hi << 16), x1 - __uint_as_float(hi & 0xffff0000u), mid, lo);
}
__device__ __forceinline__ void tc_st16(uint32_t taddr, const uint32_t (&r)[16]) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};"
        ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]),
          "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]) : "memory");
}
__device__ __forceinline__ void tc_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// PLANES: bf16 planes of the queries and of the weights
template <int PLANES>
__global__ void __launch_bounds__(AT_THREADS, 1)
attention_tc_kernel(const __grid_constant__ CUtensorMap map_k, const __grid_constant__ CUtensorMap map_v,
                    const __grid_constant__ CUtensorMap map_k2, const __grid_constant__ CUtensorMap map_v2, const AttnWork a) {
    extern __shared__ uint8_t smem_raw[];
    __shared__ __align__(8) unsigned long long bars[2 * AT_MAX_SLOTS + 12];
    __shared__ uint32_t tmem_base_sh;
    __shared__ int abort_sh, ranges_sh;
    __shared__ Cut cut_sh;
    __shared__ float xch_sh[2][2][128];                 // exchange between the two warps of a lane quarter: [parity][half][row]

    RUN_FLAG_EXIT(a.run_flag);
    PDL_TRIGGER();
    const int warp = uniform(threadIdx.x >> 5), lane = threadIdx.x & 31;
    const int NS = a.ring_slots;
    // staged queries first (the MMA reads 128 rows from each 64-dim chunk: what lies behind the live rows is the ring)
    const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u, qchunk = (uint32_t)a.rows8 * 128u;
    const uint32_t qsm = base, ring = base + 2 * PLANES * qchunk;
    uint8_t *q_gen = smem_raw + (base - smem_u32(smem_raw));
    auto full_bar = [&](int s) { return smem_u32(&bars[s]); };
    auto empty_bar = [&](int s) { return smem_u32(&bars[AT_MAX_SLOTS + s]); };
    auto sfull_bar = [&](int b) { return smem_u32(&bars[2 * AT_MAX_SLOTS + b]); };
    auto pfull_bar = [&](int b) { return smem_u32(&bars[2 * AT_MAX_SLOTS + 2 + b]); };
    auto pvdone_bar = [&](int b) { return smem_u32(&bars[2 * AT_MAX_SLOTS + 4 + b]); };
    auto pair_bar = [&](int qt) { return smem_u32(&bars[2 * AT_MAX_SLOTS + 6 + qt]); };
    const uint32_t qfull_bar = smem_u32(&bars[2 * AT_MAX_SLOTS + 10]);
    const uint32_t wg_bar = smem_u32(&bars[2 * AT_MAX_SLOTS + 11]);      // the softmax warps among themselves (bounded, unlike bar.sync)

    if (threadIdx.x == 0) {
        for (int s = 0; s < NS; ++s) { mbar_init(full_bar(s), 1); mbar_init(empty_bar(s), 1); }
        for (int b = 0; b < 2; ++b) { mbar_init(sfull_bar(b), 1); mbar_init(pfull_bar(b), SW); mbar_init(pvdone_bar(b), 1); }
        for (int qt = 0; qt < 4; ++qt) mbar_init(pair_bar(qt), 2);
        mbar_init(qfull_bar, SW);
        mbar_init(wg_bar, SW);
        abort_sh = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == 2) {
        Cut c;
        int n;
        choose_cut(a, lane, c, n);
        if (lane == 0) { cut_sh = c; ranges_sh = n; }
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base_sh)), "r"(512) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = uniform(tmem_base_sh);
    const Cut cut{uniform(cut_sh.k), uniform(cut_sh.per)};
    const int ranges = uniform(ranges_sh);
    ItemSrc src;
    src_init(a, cut, ranges, src);
    Item it;

    if (warp == 0) {
        // ---------------- TMA producer: the CTA's requests, item after item ----------------
        if (lane == 0) {
            const uint64_t kvpol = l2_evict_first_policy();    // the cache passes through once per layer
            int j = 0, count = 0;
            bool ok = true, more = next_item(a, cut, src, it);
            auto issue_next = [&](bool context_only) -> bool {  // false: nothing (more) to request under this condition
                if (more && j >= 2 * it.n_tiles) { j = 0; more = next_item(a, cut, src, it); }
                if (!more) return false;
                bool is_v;
                const int k0 = it.k_begin + request_tile(j, it.n_tiles, is_v) * TKEYS;
                if (context_only && k0 + TKEYS > it.n_ctx) return false;   // this tile holds rows the previous kernel writes
                const int st = count % NS;
                if (count >= NS && !(ok = mbar_wait(empty_bar(st), ((count / NS) & 1) ^ 1, &abort_sh, a.status))) return false;
                const uint32_t dst = ring + st * SLOT_BYTES;
                const CUtensorMap *mp = is_v ? (it.stream ? &map_v2 : &map_v) : (it.stream ? &map_k2 : &map_k);
                mbar_expect_tx(full_bar(st), SLOT_BYTES);
                tma_load_2d_hint(dst, mp, full_bar(st), 0, it.row_base + k0, kvpol);
                tma_load_2d_hint(dst + HALF_BYTES, mp, full_bar(st), 64, it.row_base + k0, kvpol);
                ++j; ++count;
                return true;
            };
            // committed context does not change during the pass: ask for it before waiting for the previous kernel
            while (count < NS && issue_next(true)) { }
            PDL_WAIT();
            while (ok && issue_next(false)) { }
        }
    } else if (warp == 1) {
        // ---------------- MMA issuer ----------------
        const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((128u >> 4) << 24);          // without N
        const uint32_t idesc_pv = idesc | ((uint32_t)(HD >> 3) << 17) | (1u << 16);               // B (the V tile) is MN-major
        int st = 0, st_ph = 0, s_cnt = 0, n_q = 0;               // ring slot and its phase, tiles of the whole CTA, staged query sets
        bool ok = true;
        auto next_slot = [&]() { if (++st == NS) { st = 0; st_ph ^= 1; } };
        while (ok && next_item(a, cut, src, it)) {
            const int n = uniform(it.n_tiles), keys = uniform(it.k_end - it.k_begin);
            auto groups16 = [&](int t) { return (min(TKEYS, keys - t * TKEYS) + 15) >> 4; };   // 16-key groups of tile t
            auto issue_qk = [&](int t) -> bool {                 // tile t of the item, s_cnt + t of the CTA
                if (!warp_wait(full_bar(st), st_ph, &abort_sh, a.status)) return false;
                tc_fence_after();
                if (elect_one()) {
                    const uint64_t kd = smem_desc(ring + st * SLOT_BYTES), q0 = smem_desc(qsm), q_step = qchunk >> 4;
                    const uint32_t sb = (s_cnt + t) & 1, d = tmem + TM_S + sb * 128, id = idesc | ((uint32_t)(2 * groups16(t)) << 17);
                    // small planes first: what an MMA adds is cut off, not rounded, at the size of what it is added to (error of the
                    // output at 256 rows against 1000 keys 2.55e-6, the other way round 2.79e-6)
#pragma unroll
                    for (int i = 0; i < 8 * PLANES; ++i) {
                        const int ks = i & 7, plane = PLANES - 1 - (i >> 3);
                        const uint64_t kb = kd + (ks >> 2) * (HALF_BYTES >> 4) + (ks & 3) * 2, qa = q0 + (ks >> 2) * q_step + (ks & 3) * 2;
                        tc_mma(d, qa + 2 * plane * q_step, kb, id, i > 0 ? 1u : 0u);
                    }
                    tc_commit(empty_bar(st));
                    tc_commit(sfull_bar(sb));
                }
                __syncwarp();
                next_slot();
                return true;
            };
            // (staged queries also mean that the previous item's O has been read)
            if (!(ok = warp_wait(qfull_bar, n_q & 1, &abort_sh, a.status))) break;
            ++n_q;
            // issue order Q K^T(0), Q K^T(1), P V(0), Q K^T(2), P V(1), ...: Q K^T(t + 2) overwrites the buffer P V(t) reads
            if (!(ok = issue_qk(0))) break;
            if (n > 1 && !(ok = issue_qk(1))) break;
            for (int t = 0; t < n; ++t) {
                const int g = s_cnt + t, sb = g & 1;
                if (!(ok = warp_wait(full_bar(st), st_ph, &abort_sh, a.status))) break;
                if (!(ok = warp_wait(pfull_bar(sb), (g >> 1) & 1, &abort_sh, a.status))) break;
                const int live_keys = min(TKEYS, keys - t * TKEYS);
                if (live_keys & 15) zero_tile_rows(ring + st * SLOT_BYTES, HALF_BYTES, live_keys, (live_keys + 15) & ~15, lane);
                tc_fence_after();
                if (elect_one()) {
                    const uint64_t vd = smem_desc_mn(ring + st * SLOT_BYTES, HALF_BYTES, 1024);
                    const uint32_t pb = tmem + TM_S + sb * 128, p3 = tmem + TM_X + sb * 64;
                    const int nk = groups16(t);
#pragma unroll
                    for (int kk = 0; kk < 8; ++kk) {                  // 16 keys per step: two 8-key groups of 1024 bytes
                        if (kk >= nk) break;
#pragma unroll
                        for (int plane = PLANES - 1; plane >= 0; --plane)
                            tc_mma_ts(tmem + TM_O, plane == 2 ? p3 + kk * 8 : pb + kk * 16 + plane * 8, vd + kk * (2048 >> 4), idesc_pv,
                                      (plane < PLANES - 1 || kk > 0 || t % GROUP<PLANES> != 0) ? 1u : 0u);
                    }
                    tc_commit(empty_bar(st));                         // the slot is free once these MMAs have read it
                    tc_commit(pvdone_bar(sb));
                }
                __syncwarp();
                next_slot();
                if (t + 2 < n && !(ok = issue_qk(t + 2))) break;
            }
            s_cnt += n;
        }
    } else {
        // ---------------- softmax / result (warps 2..5 and 6..9 <-> TMEM lane quarters 2,3,0,1): one query row, half of the keys ----------------
        const int quarter = warp & 3, sw = warp - 2, half = sw >> 2, trow = quarter * 32 + lane, et = threadIdx.x - 64;
        const uint32_t tlane = tmem + ((uint32_t)(quarter * 32) << 16);
        const size_t part_floats = (size_t)a.rows8 * PART_ROW;
        int s_cnt = 0, x_cnt = 0, wg_phase = 0;                  // tiles (buffer phase), exchanges, group barriers
        int arrived = 0, acked = 0;                              // split pairs counted in and out
        bool ok = true, first = true;
        auto wg_sync = [&]() -> bool {
            __syncwarp();
            if (lane == 0) mbar_arrive(wg_bar);
            return warp_wait(wg_bar, wg_phase++ & 1, &abort_sh, a.status);
        };
        // the other half's value for this row (both warps of the lane quarter call it together)
        auto exchange = [&](float mine, float &other) -> bool {
            const int p = x_cnt & 1;
            xch_sh[p][half][trow] = mine;
            __syncwarp();
            if (lane == 0) mbar_arrive(pair_bar(quarter));
            const bool done = warp_wait(pair_bar(quarter), p, &abort_sh, a.status);
            other = xch_sh[p][half ^ 1][trow];
            ++x_cnt;
            return done;
        };
        while (ok && next_item(a, cut, src, it)) {
            const bool live = trow < it.rows, warp_live = quarter * 32 < it.rows;
            const size_t o0 = row_off(a, it, live ? trow : 0);
            const int g0 = it.row0 + (live ? trow : 0);
            const unsigned long long anc = a.tree[it.b].anc[g0 - (int)((g0 * a.m_recip) >> 32) * a.M];
            // stage the item's query rows as bf16 planes, pre-scaled, in the K-major 128-byte-swizzled layout the MMA
            // reads; a warp takes whole rows, all its loads in flight (addresses first: they do not wait for anything)
            uint32_t qrow[QROWS];
#pragma unroll
            for (int q = 0; q < QROWS; ++q) qrow[q] = (uint32_t)(row_off(a, it, min(sw + q * SW, it.rows - 1)) >> 2) + lane;
            if (first) PDL_WAIT();
            else if (!(ok = wg_sync())) break;                   // the rows staged in the query region have been written out
            first = false;
            float4 v[QROWS];
#pragma unroll
            for (int q = 0; q < QROWS; ++q) {
                v[q] = make_float4(0.f, 0.f, 0.f, 0.f);
                if (sw + q * SW < it.rows) v[q] = __ldcg(reinterpret_cast<const float4 *>(a.q) + qrow[q]);
            }
#pragma unroll
            for (int q = 0; q < QROWS; ++q) {
                const uint32_t r = sw + q * SW, d4 = 4 * lane, dc = d4 & 63;       // dc: dim inside its 64-dim chunk
                if (r >= (uint32_t)a.rows8) break;
                uint2 hi, lo, lo2;
                split_triple(v[q].x * a.scale, v[q].y * a.scale, hi.x, lo.x, lo2.x);
                split_triple(v[q].z * a.scale, v[q].w * a.scale, hi.y, lo.y, lo2.y);
                uint8_t *dst = q_gen + (d4 >> 6) * qchunk + r * 128u + (((dc >> 3) ^ (r & 7u)) << 4) + (dc & 7u) * 2u;
                *reinterpret_cast<uint2 *>(dst) = hi;
                *reinterpret_cast<uint2 *>(dst + 2 * qchunk) = lo;
                if (PLANES == 3) *reinterpret_cast<uint2 *>(dst + 4 * qchunk) = lo2;
            }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // generic writes -> the MMA's reads
            __syncwarp();
            if (lane == 0) mbar_arrive(qfull_bar);

            float m_run = -INFINITY, l_run = 0.f;                // m_run: the whole row's, l_run: of this half's keys
            // O of the tiles so far, this half's dims: in registers, or (two planes leave room) in TMEM, by rolled loops
            float o[PLANES == 3 ? 64 : 1];
#pragma unroll
            for (int e = 0; e < (PLANES == 3 ? 64 : 1); ++e) o[e] = 0.f;
            // Adds a group's O once its last P V (of tile g of the CTA) has written it, and moves the sum to the new maximum.  32
            // columns at a time; `first`: the sum is empty, `last`: it is not kept, but handed to `use`.
            auto add_group = [&](int g, float corr, bool first, bool last, auto use) -> bool {
                if (!warp_wait(pvdone_bar(g & 1), (g >> 1) & 1, &abort_sh, a.status)) return false;
                tc_fence_after();
                if (!warp_live) return true;
                if constexpr (PLANES == 3) {
#pragma unroll
                    for (int c = 0; c < 2; ++c) {
                        uint32_t r[32];
                        tc_ld32(tlane + TM_O + half * 64 + c * 32, r);
#pragma unroll
                        for (int e = 0; e < 32; ++e) r[e] = __float_as_uint(o[c * 32 + e] = (o[c * 32 + e] + __uint_as_float(r[e])) * corr);
                        if (last) use(c, r);
                    }
                } else {
#pragma unroll 1
                    for (int c = 0; c < 2; ++c) {
                        const uint32_t from = tlane + half * 64 + c * 32;
                        uint32_t r[32], s[32];
                        if (first) {
                            tc_ld32(from + TM_O, r);
                        } else {
                            tc_ld32x2(from + TM_O, from + TM_X, r, s);
#pragma unroll
                            for (int e = 0; e < 32; ++e) r[e] = __float_as_uint(__uint_as_float(r[e]) + __uint_as_float(s[e]));
                        }
                        if (last) { use(c, r); continue; }
#pragma unroll
                        for (int e = 0; e < 32; ++e) r[e] = __float_as_uint(__uint_as_float(r[e]) * corr);
                        tc_st32(from + TM_X, r);
                    }
                }
                return true;
            };
            for (int t = 0; t < it.n_tiles; ++t, ++s_cnt) {
                const int sb = s_cnt & 1;
                if (!(ok = warp_wait(sfull_bar(sb), (s_cnt >> 1) & 1, &abort_sh, a.status))) break;
                tc_fence_after();
                const int j0 = it.k_begin + t * TKEYS + half * 64;           // first key of this half
                const bool masked = j0 + 64 > it.n_ctx || j0 + 64 > it.k_end;
                const int cols = warp_live ? min(64, it.k_end - j0) : 0;     // columns of this half that hold scores (may be negative)
                const uint32_t tb = tlane + TM_S + sb * 128 + half * 64;
                // which of 32 keys from `key` on this row may see: inside the range, and committed context or an ancestor
                auto visible32 = [&](int key) -> uint32_t {
                    const int nr = it.k_end - key, nc = it.n_ctx - key;
                    const uint32_t in_range = nr >= 32 ? 0xffffffffu : nr <= 0 ? 0u : (1u << nr) - 1u;
                    const uint32_t in_ctx = nc >= 32 ? 0xffffffffu : nc <= 0 ? 0u : (1u << nc) - 1u;
                    const uint32_t tree_bits = nc >= 32 ? 0u : nc > 0 ? (uint32_t)(anc << nc) : (nc > -64 ? (uint32_t)(anc >> -nc) : 0u);
                    return in_range & (in_ctx | tree_bits);
                };
                auto load = [&](int c, uint32_t (&r)[32]) {                   // 32 scores, those out of sight -inf
                    tc_ld32(tb + c * 32, r);
                    if (masked) {
                        const uint32_t vis = visible32(j0 + c * 32);
#pragma unroll
                        for (int e = 0; e < 32; ++e) r[e] = (vis >> e) & 1u ? r[e] : 0xff800000u;
                    }
                };
                // pass 1: the row maximum (rolled: the loop bodies stay small enough to live in the instruction cache)
                float m_half = -INFINITY;
#pragma unroll 1
                for (int c = 0; c * 32 < cols; ++c) {
                    uint32_t r[32];
                    load(c, r);
#pragma unroll
                    for (int e = 0; e < 32; ++e) m_half = fmaxf(m_half, __uint_as_float(r[e]));
                }
                float m_tile;
                if (!(ok = exchange(m_half, m_tile))) break;
                m_tile = fmaxf(m_tile, m_half);
                float corr = 1.f;
                if (live && m_tile > m_run + RESCALE_GAP) {            // also the first tile with a visible key (m_run = -inf)
                    corr = (m_run == -INFINITY) ? 1.f : ex2(m_run - m_tile);
                    m_run = m_tile;
                }
                l_run *= corr;
                // pass 2: weights and their row sum; P replaces S in place
                const float m_use = m_run == -INFINITY ? 0.f : m_run;   // no visible key yet: every weight is 2^-inf
#pragma unroll 1
                for (int c = 0; c * 32 < cols; ++c) {
                    uint32_t r[32], w[32], w3[16];
                    load(c, r);
                    float l4[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
                    for (int e = 0; e < 32; e += 2) {
                        const float p0 = ex2(__uint_as_float(r[e]) - m_use), p1 = ex2(__uint_as_float(r[e + 1]) - m_use);
                        l4[(e >> 1) & 3] += p0 + p1;
                        const int at = (e >> 4) * 16 + ((e & 15) >> 1);
                        if (PLANES == 3) split_triple(p0, p1, w[at], w[at + 8], w3[e >> 1]);
                        else split_pair(p0, p1, w[at], w[at + 8]);
                    }
                    l_run += (l4[0] + l4[1]) + (l4[2] + l4[3]);
                    tc_st32(tb + c * 32, w);
                    if (PLANES == 3) tc_st16(tlane + TM_X + sb * 64 + half * 32 + c * 16, w3);
                }
                if (t > 0 && t % GROUP<PLANES> == 0) {
                    if (!(ok = add_group(s_cnt - 1, corr, t == GROUP<PLANES>, false, [](int, const uint32_t (&)[32]) {}))) break;
                } else if (t > 0 && __any_sync(0xffffffffu, corr != 1.f)) {
                    // rare: the maximum moved inside a group.  Its O, and the sum before it, move along.
                    if (!(ok = warp_wait(pvdone_bar(sb ^ 1), ((s_cnt - 1) >> 1) & 1, &abort_sh, a.status))) break;
                    tc_fence_after();
#pragma unroll 1
                    for (int c = 0; c < (t > GROUP<PLANES> ? 4 : 2); ++c) {
                        const uint32_t at = tlane + (c < 2 ? TM_O : TM_X) + half * 64 + (c & 1) * 32;
                        uint32_t r[32];
                        tc_ld32(at, r);
#pragma unroll
                        for (int e = 0; e < 32; ++e) r[e] = __float_as_uint(__uint_as_float(r[e]) * corr);
                        tc_st32(at, r);
                    }
                }
                tc_wait_st();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(pfull_bar(sb));             // P is in place, O may be overwritten
            }
            if (!ok) break;
            // ---- the item's result, once the last P V (and with it all earlier ones) has written O ----
            float l_other;
            if (!(ok = exchange(l_run, l_other))) break;
            const float l = half ? l_other + l_run : l_run + l_other;
            const bool single = it.n_split == 1;
            float *pdst = a.part + ((size_t)it.pair * a.slots + it.split) * part_floats;
            const float inv = 1.f / l;
            auto put = [&](int c, const uint32_t (&r)[32]) {
                if (single) {
                    // through the query region (every MMA that read it is done), so that whole rows go out together
#pragma unroll
                    for (int e = 0; e < 32; e += 8) {
                        uint4 hi, lo;
                        split_pair(__uint_as_float(r[e]) * inv, __uint_as_float(r[e + 1]) * inv, hi.x, lo.x);
                        split_pair(__uint_as_float(r[e + 2]) * inv, __uint_as_float(r[e + 3]) * inv, hi.y, lo.y);
                        split_pair(__uint_as_float(r[e + 4]) * inv, __uint_as_float(r[e + 5]) * inv, hi.z, lo.z);
                        split_pair(__uint_as_float(r[e + 6]) * inv, __uint_as_float(r[e + 7]) * inv, hi.w, lo.w);
                        if (live) {
                            uint8_t *dst = q_gen + trow * 256 + (((half * 8 + c * 4 + (e >> 3)) ^ (trow & 15)) << 4);
                            *reinterpret_cast<uint4 *>(dst) = hi;
                            *reinterpret_cast<uint4 *>(dst + 2 * qchunk) = lo;
                        }
                    }
                } else if (live) {
                    // lanes are rows: 512 contiguous bytes per store
#pragma unroll
                    for (int e = 0; e < 32; e += 4)
                        *reinterpret_cast<uint4 *>(pdst + ((size_t)(half * 16 + c * 8 + (e >> 2)) * a.rows8 + trow) * 4) = make_uint4(r[e], r[e + 1], r[e + 2], r[e + 3]);
                }
            };
            if (!(ok = add_group(s_cnt - 1, 1.f, it.n_tiles <= GROUP<PLANES>, true, put))) break;
            tc_fence_before();
            if (single) {
                float unused;
                if (!(ok = exchange(0.f, unused))) break;              // both halves of the rows are in place
                if (warp_live) {
#pragma unroll 1
                    for (int i = 0; i < 8; ++i) {
                        const int r = half * 16 + i * 2 + (lane >> 4), rr = quarter * 32 + r, ch = lane & 15;   // half a warp per row
                        const size_t ro = __shfl_sync(0xffffffffu, (unsigned long long)o0, r) + ch * 8;
                        if (rr >= it.rows) continue;
                        const uint8_t *from = q_gen + rr * 256 + ((ch ^ (rr & 15)) << 4);
                        *reinterpret_cast<uint4 *>(a.out + ro) = *reinterpret_cast<const uint4 *>(from);
                        *reinterpret_cast<uint4 *>(a.out + a.out_plane + ro) = *reinterpret_cast<const uint4 *>(from + 2 * qchunk);
                    }
                }
            } else {
                if (live && half == 0) *reinterpret_cast<float2 *>(pdst + (size_t)HD * a.rows8 + 2 * trow) = make_float2(m_run, l);
                if (!(ok = wg_sync())) break;
                // (the barrier orders the group's stores before this thread's release, which is cumulative)
                if (et == 0) counter_arrive(a.counters + it.pair, it.n_split, it.n_split);
                ++arrived;
            }
        }
        // ---- the split pairs of this CTA's list: its slice of each one's rows ----
        src_init(a, cut, ranges, src);
        while (ok && next_item(a, cut, src, it)) {
            if (it.n_split == 1) continue;
            if (et == 0) counter_wait(a.counters + it.pair, it.n_split, it.n_split, &abort_sh, a.status);
            ++acked;
            if (!(ok = wg_sync())) break;
            const int rper = (it.rows + it.n_split - 1) / it.n_split, r0 = min(it.rows, it.split * rper), nr = min(it.rows, r0 + rper) - r0;
            const float *psrc = a.part + (size_t)it.pair * a.slots * part_floats;
            // A lane takes a row, a warp every eighth group of dims.  All its pieces (16 bytes of a range's row) come into the idle
            // ring by asynchronous copies: one trip to L2 however many ranges there are, and no thread reads what another
            // copied, so there is no barrier.  (Loads into registers, 8 ranges at a time, were a trip of 1000 cycles per 8 ranges;
            // copies with a barrier and a warp per row for the weights 6800 cycles in all for 12 rows of 9 ranges.)
#pragma unroll 1
            for (int row = lane; row < nr; row += 32) {
                const float *from = psrc + ((size_t)sw * a.rows8 + r0 + row) * 4, *from_ml = psrc + (size_t)HD * a.rows8 + 2 * (r0 + row);
                const uint32_t at = qsm + (uint32_t)(sw * nr + row) * 16u, step = (uint32_t)(SW * nr) * 16u;
                const uint32_t at_ml = qsm + (uint32_t)(it.n_split * 4) * step + (uint32_t)(sw * nr + row) * 8u;
#pragma unroll 1
                for (int s = 0; s < it.n_split; ++s) {
#pragma unroll
                    for (int i = 0; i < 4; ++i)
                        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(at + (uint32_t)(4 * s + i) * step), "l"(from + (size_t)(i * SW * 4) * a.rows8) : "memory");
                    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(at_ml + (uint32_t)s * (step >> 1)), "l"(from_ml) : "memory");
                    from += part_floats; from_ml += part_floats;
                }
                __nv_bfloat16 *dst = a.out + row_off(a, it, r0 + row) + 4 * sw;
                asm volatile("cp.async.wait_all;" ::: "memory");
                const uint8_t *pieces = q_gen + (at - qsm);
                float2 *ml = reinterpret_cast<float2 *>(q_gen + (at_ml - qsm));
                const int ml_step = (int)(step >> 4);
                float m = -INFINITY, den = 0.f;
#pragma unroll 4
                for (int s = 0; s < it.n_split; ++s) m = fmaxf(m, ml[s * ml_step].x);   // (every row sees at least itself: finite)
#pragma unroll 4
                for (int s = 0; s < it.n_split; ++s) {
                    const float2 x = ml[s * ml_step];
                    const float w = ex2(x.x - m);
                    den = fmaf(x.y, w, den);
                    ml[s * ml_step].x = w;
                }
                const float inv = 1.f / den;
                float4 num[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) num[i] = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 2
                for (int s = 0; s < it.n_split; ++s) {
                    const float w = ml[s * ml_step].x;
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const float4 v = *reinterpret_cast<const float4 *>(pieces + (uint32_t)(4 * s + i) * step);
                        num[i].x = fmaf(v.x, w, num[i].x); num[i].y = fmaf(v.y, w, num[i].y);
                        num[i].z = fmaf(v.z, w, num[i].z); num[i].w = fmaf(v.w, w, num[i].w);
                    }
                }
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    uint2 hi, lo;
                    split_pair(num[i].x * inv, num[i].y * inv, hi.x, lo.x);
                    split_pair(num[i].z * inv, num[i].w * inv, hi.y, lo.y);
                    *reinterpret_cast<uint2 *>(dst + i * SW * 4) = hi;
                    *reinterpret_cast<uint2 *>(dst + a.out_plane + i * SW * 4) = lo;
                }
            }
        }
        if (!ok && et == 0) settle_counters(a, cut, ranges, arrived, acked);
    }

    // ---------------- teardown ----------------
    __syncwarp();
    if (abort_sh && threadIdx.x == 0) {
        // give copies and MMAs that are still in flight time to land before shared memory and TMEM go away
        const long long t0 = clock64();
        while (clock64() - t0 < 400000) { }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
    }
}

}  // namespace

// streams = 1: one cache (full or slim).  streams = 2: rows [0, batch*M) against the full cache at layer_ord and
// rows [batch*M, 2*batch*M) against the slim cache at layer_ord2, in one launch.
int launch_attention_tc(viasd_model *m, const void *kc, const void *vc, bool slim, int layer_ord, const void *kc2,
                        const void *vc2, int layer_ord2, int streams, int batch, int M, cudaStream_t st) {
    const viasd_config &c = m->cfg;
    CacheMaps &cm = slim ? m->cmaps_slim : m->cmaps_full;
    int rc;
    if ((rc = attention_cache_maps(m, cm, kc, vc, slim ? m->n_routed : c.n_layers))) return rc;
    CacheMaps *cm2 = &cm;
    if (streams == 2) {
        cm2 = &m->cmaps_slim;
        if ((rc = attention_cache_maps(m, *cm2, kc2, vc2, m->n_routed))) return rc;
    }
    const int QR = c.n_heads / c.n_kv_heads * M;
    AttnWork a;
    a.subs = (QR + 127) / 128;
    a.rows_sub = a.subs == 1 ? QR : ((QR + a.subs - 1) / a.subs + 7) / 8 * 8;
    a.subs = (QR + a.rows_sub - 1) / a.rows_sub;
    fill_work(m, a, layer_ord, layer_ord2, streams, batch, M);
    const int grid = work_grid(m);
    const int planes = QR > 128 ? 3 : 2;
    const size_t q_bytes = (size_t)a.rows8 * 256 * planes, smem_max = 229000;
    a.ring_slots = (int)((smem_max - 1024 - q_bytes) / SLOT_BYTES);
    if (a.ring_slots > AT_MAX_SLOTS) a.ring_slots = AT_MAX_SLOTS;
    const size_t smem = 1024 + q_bytes + (size_t)a.ring_slots * SLOT_BYTES;
    static std::atomic<bool> attr_done[64];
    if (int rc = once_on_device(attr_done, [&]() -> int {
        CUDA_TRY(cudaFuncSetAttribute(attention_tc_kernel<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_max));
        CUDA_TRY(cudaFuncSetAttribute(attention_tc_kernel<3>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_max));
        return VIASD_OK;
    })) return rc;
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attr[1];
    pdl_config(cfg, attr, dim3(grid), dim3(AT_THREADS), smem, st);
    CUDA_TRY(cudaLaunchKernelEx(&cfg, planes == 3 ? attention_tc_kernel<3> : attention_tc_kernel<2>, cm.k, cm.v, cm2->k, cm2->v, a));
    LAUNCH_CHECK();
    return VIASD_OK;
}
