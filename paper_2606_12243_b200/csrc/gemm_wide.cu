// Projection GEMM for many token rows: pairs of CTAs on one tcgen05.mma (cta_group::2).
//
//   y[rows, n] = x[rows, k] * W[n, k]^T        rows <= 256 per launch, x as bf16 hi + lo planes
//
// What bounds it.  Up to about 128 rows HBM, through the weights a CTA can keep in flight: in the one-CTA kernel
// (gemm_tc.cu) both planes of the activation tile sit beside every weight box, at 112 rows 28 KB of each 44 KB of ring.
// Here each CTA of a pair holds its own 128 weight rows and ONE of the two planes: the MMA's N dimension is [hi rows from
// CTA 0; lo rows from CTA 1], so a box of 64 columns costs 16 KB of weights plus rows * 128 B of activations per SM, and
// a launch takes up to 256 rows in two sub-tiles (512 TMEM columns), where the one-CTA kernel streams the weights once
// per 128 rows.  From about 200 rows on the tensor cores bound it (two planes: twice the product's operations).
//
// A tile is 2 x 128 output features (the MMA's M = 256); for the gate/up launch a CTA's 128 features are 64 of the gate
// and the matching 64 of the up matrix.  Stream-K over (tile pair, k-box) as in gemm_tc.cu: one contiguous range per
// pair; the cuts depend on n and k only, so a row's bits do not depend on how many rows share the launch.  A split
// tile is finished by the contributors that end in it: each keeps its own slice of the token rows in TMEM, publishes the
// rest, waits (bounded) for the other contributors and adds their rows in pair order.  The finishing is done a row per
// warp (lane l has features 4l..4l+3): 16-byte loads and stores, where a thread per feature needed a load, three stores
// and a chain of latencies per element.
//
// Warps (576 threads): 0 issues TMA loads (each CTA its own), 1 allocates TMEM and, in CTA 0, issues the MMAs, 2-17
// are four groups of four epilogue warps that take chunks of 8 rows in turn.  CTA 1's loads complete on CTA 0's full
// barriers; commits arrive on both CTAs' barriers.  Every mbarrier and counter wait is bounded: on expiry the CTA
// records VIASD_EDEVICE, lets its copies land and leaves (its partner's waits then expire the same way).
#include "common.cuh"
#include "gemm_tc.cuh"
#include "gemm_tc_device.cuh"

namespace {

constexpr int WGROUPS = 4;                     // groups of four epilogue warps
constexpr int WEPI = WGROUPS * 128;
constexpr int WTHREADS = 64 + WEPI;
constexpr int WROWS = TC_WIDE_ROWS;            // token rows per launch
constexpr int WSTAGES = 12;
constexpr uint32_t WBOX = TILE_F * TILE_K * 2; // a CTA's weight box: 128 features x 64 columns

// (all predicated to the lane with `on` != 0; the loops around them are run by the whole warp)
__device__ __forceinline__ uint32_t leader_addr(uint32_t own) {          // the same location in the pair's CTA 0
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(own), "r"(0));
    return r;
}
__device__ __forceinline__ void pair_load(uint32_t on, uint32_t dst, const CUtensorMap *map, uint32_t leader_bar, int x, int y) {
    asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.b32 q, %5, 0;\n\t"
                 "@q cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];\n\t}"
                 ::"r"(dst), "l"(map), "r"(leader_bar), "r"(x), "r"(y), "r"(on) : "memory");
}
__device__ __forceinline__ void pair_load_hint(uint32_t on, uint32_t dst, const CUtensorMap *map, uint32_t leader_bar, int x, int y, uint64_t pol) {
    asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.b32 q, %6, 0;\n\t"
                 "@q cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1, {%3, %4}], [%2], %5;\n\t}"
                 ::"r"(dst), "l"(map), "r"(leader_bar), "r"(x), "r"(y), "l"(pol), "r"(on) : "memory");
}
__device__ __forceinline__ void pair_mma(uint32_t on, uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc, uint32_t accumulate) {
    asm volatile("{\n\t.reg .pred p, q;\n\tsetp.ne.b32 p, %4, 0;\n\tsetp.ne.b32 q, %5, 0;\n\t"
                 "@q tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}"
                 ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate), "r"(on) : "memory");
}
__device__ __forceinline__ void pair_commit(uint32_t on, uint32_t bar) {              // arrives on both CTAs' barrier
    asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.b32 q, %2, 0;\n\t"
                 "@q tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;\n\t}"
                 ::"r"(bar), "h"((uint16_t)3), "r"(on) : "memory");
}
__device__ __forceinline__ void pair_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
template <int EPI>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(WTHREADS, 1)
gemm_wide_kernel(const __grid_constant__ CUtensorMap map_w0, const __grid_constant__ CUtensorMap map_w1,
                 const __grid_constant__ CUtensorMap map_w2, const __grid_constant__ CUtensorMap map_x, const TcParams p) {
    extern __shared__ uint8_t smem_raw[];
    __shared__ __align__(8) unsigned long long bars[2 * WSTAGES + 4];
    __shared__ uint32_t tmem_base_sh;
    __shared__ int abort_sh;
    __shared__ __align__(16) float xch[WGROUPS][CH * TILE_F];     // a chunk on its way from TMEM lanes to rows, per group
    __shared__ float inv_sh[WROWS];
    __shared__ int4 rowmeta[EPI == EPI_QKV_ROPE ? WROWS : 1];

    RUN_FLAG_EXIT(p.run_flag);
    const int warp = uniform(threadIdx.x >> 5), lane = threadIdx.x & 31;
    const uint32_t rank = blockIdx.x & 1;                         // this CTA's place in its pair
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    const int TH = p.nt, TT = p.tt;                               // rows per plane and sub-tile; sub-tiles
    // Weights and activations have rings of their own.  Weights come from HBM and are what the depth is for; activation
    // boxes come from L2 and need only a few slots.  A box's two loads still share one full barrier and one commit: box i's
    // weights and box i - (SW - SX)'s activations are requested when box i - SW has been read.
    const int SW = p.stages, SX = p.x_stages;
    const uint32_t x_bytes = (uint32_t)TH * 128u, xbox = TT * x_bytes;
    const uint32_t xring = smem_base + SW * WBOX;
    auto full_bar = [&](int s) { return smem_u32(&bars[s]); };
    auto empty_bar = [&](int s) { return smem_u32(&bars[WSTAGES + s]); };
    auto tfull_bar = [&](int b) { return smem_u32(&bars[2 * WSTAGES + b]); };
    auto tempty_bar = [&](int b) { return smem_u32(&bars[2 * WSTAGES + 2 + b]); };
    const uint32_t acc_cols = (uint32_t)TT * 2u * TH;

    if (threadIdx.x == 0) {
        for (int s = 0; s < SW; ++s) { mbar_init(full_bar(s), 1); mbar_init(empty_bar(s), 1); }
        for (int b = 0; b < 2; ++b) { mbar_init(tfull_bar(b), 1); mbar_init(tempty_bar(b), 2 * WGROUPS * 4); }
        abort_sh = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base_sh)), "r"(p.tmem_cols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    pair_sync();                                                  // both CTAs' barriers exist before either is signalled
    tc_fence_after();
    const uint32_t tmem_base = __shfl_sync(0xffffffffu, tmem_base_sh, 0);

    const int pair = blockIdx.x >> 1, ptiles = (p.n_tiles + 1) >> 1;
    const int total_units = ptiles * p.k_tiles;
    const int u_begin = min(total_units, pair * p.units_per_cta), u_end = min(total_units, u_begin + p.units_per_cta);

    if (warp == 0) {
        // ---------------- TMA producer: this CTA's weight rows and its plane of the activations ----------------
        const uint32_t on = elect_one(), lead = on && rank == 0;
        const int n_it = u_end - u_begin;
        const CUtensorMap *mw = &map_w0;
        int wrow = 0, kt = 0, ptile = 0;
        uint32_t w_tx = 0;                                        // bytes of both CTAs' weight boxes
        auto seg_of = [&](int tile, int &t0) { int s = 0; t0 = 0; while (s < 2 && tile >= p.seg_tile_end[s]) { t0 = p.seg_tile_end[s]; ++s; } return s; };
        auto enter_tile = [&]() {
            const int tile = 2 * ptile + (int)rank;
            if (EPI == EPI_SWIGLU) { wrow = tile * 64; w_tx = 4 * p.a_tx[0]; return; }
            int t0, t1;
            // (the tile past the end of an odd count reads rows beyond its matrix: zeros)
            const int s = seg_of(min(tile, p.n_tiles - 1), t0), so = seg_of(min(tile ^ 1, p.n_tiles - 1), t1);
            mw = s == 0 ? &map_w0 : (s == 1 ? &map_w1 : &map_w2);
            wrow = (tile - t0) * TILE_F;
            w_tx = p.a_tx[s] + p.a_tx[so];
        };
        auto advance = [&]() { if (++kt >= p.k_tiles) { kt = 0; ++ptile; enter_tile(); } };
        const uint64_t wpol = l2_evict_first_policy();
        const uint32_t x_tx = 2 * TT * p.b_tx;
        const int x_row = p.row0 + (rank ? p.lo_row_offset : 0);
        // CTA 0's barriers as both CTAs address them: one offset from this CTA's own
        const uint32_t to_lead = __shfl_sync(0xffffffffu, leader_addr(full_bar(0)) - full_bar(0), 0);
        auto load_w = [&](uint32_t base, uint32_t bar) {
            if (EPI == EPI_SWIGLU) {
                pair_load_hint(on, base, &map_w0, bar, kt * TILE_K, wrow, wpol);
                pair_load_hint(on, base + WBOX / 2, &map_w1, bar, kt * TILE_K, wrow, wpol);
            } else {
                pair_load_hint(on, base, mw, bar, kt * TILE_K, wrow, wpol);
            }
        };
        int xkt = 0;                                              // k-box of the next activation load
        auto load_x = [&](uint32_t base, uint32_t bar) {
            pair_load(on, base, &map_x, bar, xkt * TILE_K, x_row);
            if (TT == 2) pair_load(on, base + x_bytes, &map_x, bar, xkt * TILE_K, x_row + TH);
            if (++xkt >= p.k_tiles) xkt = 0;
        };
        ptile = u_begin / p.k_tiles; kt = u_begin - ptile * p.k_tiles; xkt = kt;
        enter_tile();
        // weights do not depend on the kernel before this one; activations do (programmatic dependent launch)
        const int pre_w = n_it < SW ? n_it : SW, pre_x = n_it < SX ? n_it : SX;
        for (int it = 0; it < pre_w; ++it, advance()) {
            // one arrival per phase, by CTA 0, for the bytes of both CTAs (the peer's may land before it)
            mbar_expect_tx_if(lead, full_bar(it), w_tx + x_tx);
            load_w(smem_base + it * WBOX, full_bar(it) + to_lead);
        }
        asm volatile("griddepcontrol.wait;" ::: "memory");
        for (int it = 0; it < pre_x; ++it) load_x(xring + it * xbox, full_bar(it) + to_lead);
        int st = 0, sx = 0, sf = pre_x == SW ? 0 : pre_x;         // weight slot, activation slot, and the barrier of its box
        uint32_t ph = 0;
        for (int done = 0; done + pre_x < n_it; ++done) {         // box `done` has been read: its two slots are free
            if (!warp_wait(empty_bar(st), ph, &abort_sh, p.status)) break;
            if (done + SW < n_it) {
                mbar_expect_tx_if(lead, full_bar(st), w_tx + x_tx);
                load_w(smem_base + st * WBOX, full_bar(st) + to_lead);
                advance();
            }
            load_x(xring + sx * xbox, full_bar(sf) + to_lead);
            if (++st == SW) { st = 0; ph ^= 1; }
            if (++sx == SX) sx = 0;
            if (++sf == SW) sf = 0;
        }
    } else if (warp == 1) {
        // ---------------- MMA issuer (CTA 0, for both) ----------------
        if (rank == 0) {
            const uint32_t on = elect_one();
            const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(2 * TH >> 3) << 17) | ((256u >> 4) << 24);
            int st = 0, sx = 0, acc_it = 0, u = u_begin;
            uint32_t ph = 0;
            Seg sg;
            bool ok = true;
            while (ok && next_seg(u, u_end, p.k_tiles, sg)) {
                const int buf = p.acc_bufs == 2 ? acc_it & 1 : 0;
                if (!(ok = warp_wait(tempty_bar(buf), (p.acc_bufs == 2 ? (acc_it >> 1) & 1 : acc_it & 1) ^ 1, &abort_sh, p.status))) break;
                tc_fence_after();
                const uint32_t d0 = tmem_base + buf * acc_cols;
                uint32_t acc = 0;
                for (int kt = sg.ka; kt < sg.kb; ++kt) {
                    if (!(ok = warp_wait(full_bar(st), ph, &abort_sh, p.status))) break;
                    tc_fence_after();
                    const uint64_t da = smem_desc(smem_base + st * WBOX), db = smem_desc(xring + sx * xbox), db2 = db + (x_bytes >> 4);
#pragma unroll
                    for (int k = 0; k < TILE_K / 16; ++k) {
                        pair_mma(on, d0, da + 2 * k, db + 2 * k, idesc, acc);
                        if (TT == 2) pair_mma(on, d0 + 2 * TH, da + 2 * k, db2 + 2 * k, idesc, acc);
                        acc = 1;
                    }
                    pair_commit(on, empty_bar(st));
                    if (++st == SW) { st = 0; ph ^= 1; }
                    if (++sx == SX) sx = 0;
                }
                if (ok) pair_commit(on, tfull_bar(buf));
                ++acc_it;
            }
        }
    } else {
        // ---------------- epilogue: TMEM lane quarter = warp & 3 ----------------
        const int quarter = warp & 3, f = quarter * 32 + lane, et = threadIdx.x - 64, group = et >> 7, gw = (et >> 5) & 3;
        const size_t slot_floats = (size_t)p.slot_rows * TILE_F;
        float *xg = xch[group];
        auto group_sync = [&]() { asm volatile("bar.sync %0, 128;" ::"r"(2 + group) : "memory"); };
        auto epi_sync = [&]() { asm volatile("bar.sync 1, %0;" ::"n"(WEPI) : "memory"); };
        asm volatile("griddepcontrol.wait;" ::: "memory");
        if (p.ssq_in && et < p.rows) {
            // 1/rms of an input row from its partial sums of squares: a thread per row, 32 loads in flight, in the order
            // of gemm_tc.cu (32 strided sub-sums, then a tree)
            const float *from = p.ssq_in + p.row0 + et;
            float acc[32];
#pragma unroll
            for (int i = 0; i < 32; ++i) acc[i] = 0.f;
#pragma unroll 1
            for (int j0 = 0; j0 < p.ssq_in_n; j0 += 32) {
                float v[32];
#pragma unroll
                for (int i = 0; i < 32; ++i) v[i] = j0 + i < p.ssq_in_n ? __ldcg(from + (size_t)(j0 + i) * p.ssq_stride) : 0.f;
#pragma unroll
                for (int i = 0; i < 32; ++i) acc[i] += v[i];
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
#pragma unroll
                for (int i = 0; i < o; ++i) acc[i] += acc[i + o];
            }
            inv_sh[et] = rsqrtf(acc[0] * p.inv_d + p.eps);
        }
        if (EPI == EPI_QKV_ROPE && et < p.rows) {
            // rows are laid out [stream][sequence][block row]; where a row's K/V go, worked out once
            const int row = p.row0 + et, stream = row >= p.split_row ? 1 : 0, rs = row - stream * p.split_row;
            const int b = rs / p.rope_M, i = rs - b * p.rope_M, n_ctx = p.len_eff[b];
            const int slot = (p.kv_keep && n_ctx + i < p.kv_keep[b]) ? -1 : n_ctx + i;
            const unsigned long long off = slot < 0 ? 0ull
                : (((unsigned long long)(stream ? p.layer_ord2 : p.layer_ord) * p.max_batch + b) * p.rope_Hkv * p.max_ctx + slot) * TILE_F;
            rowmeta[et] = make_int4(n_ctx + p.depth[(size_t)b * p.tree_stride + i], slot, (int)(unsigned)(off & 0xffffffffull),
                                    (int)((unsigned)(off >> 32) | ((unsigned)stream << 30)));
        }
        epi_sync();

        int acc_it = 0, u = u_begin, seg_i = 0;
        Seg sg;
        // (a wait that expires does not end this loop: all threads go on through the same barriers, none of which waits any
        // more for another CTA, see counter_wait)
        while (next_seg(u, u_end, p.k_tiles, sg)) {
            const int buf = acc_it % p.acc_bufs, tile = 2 * sg.tile + (int)rank;
            // one warp polls the barrier, the others sleep in a named barrier
            if (warp == 2) mbar_wait(tfull_bar(buf), (acc_it / p.acc_bufs) & 1, &abort_sh, p.status);
            epi_sync();
            tc_fence_after();
            const uint32_t t0 = tmem_base + ((uint32_t)(quarter * 32) << 16) + buf * acc_cols;
            // the sums of 8 token rows from r0 on, feature f: hi and lo products added
            auto load_chunk = [&](int r0, float (&g)[CH]) {
                const uint32_t c = r0 < TH ? r0 : r0 + TH;
                float lo[CH];
                tc_ld8x2(t0 + c, t0 + c + TH, g, lo);
#pragma unroll
                for (int j = 0; j < CH; ++j) g[j] += lo[j];
            };
            const bool live = tile < p.n_tiles;
            // what finishing a row reads besides the sums, asked for a chunk ahead (and, for the first chunk, before the waits)
            float4 aux[2][2];
            auto load_aux = [&](int r0, int r_end) {
                const int ra = r0 + 2 * gw;
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    const int r = ra + i;
                    if (r >= r_end || r >= p.rows) continue;
                    if (EPI == EPI_ADD_NORM) {
                        aux[i][0] = __ldcg(reinterpret_cast<const float4 *>(p.out_f32 + (size_t)(p.row0 + r) * p.ld_out + tile * TILE_F + 4 * lane));
                    } else if (EPI == EPI_QKV_ROPE) {
                        const size_t o = (size_t)rowmeta[r].x * 64 + (lane & 15) * 4;
                        aux[i][0] = *reinterpret_cast<const float4 *>(p.cosv + o);
                        aux[i][1] = *reinterpret_cast<const float4 *>(p.sinv + o);
                    }
                }
            };
#pragma unroll
            for (int i = 0; i < 4; ++i) aux[i >> 1][i & 1] = make_float4(0.f, 0.f, 0.f, 0.f);
            const bool whole = sg.ka == 0 && sg.kb == p.k_tiles;
            int row_begin = 0, row_end = live ? p.rows : 0, first = pair, n_c = 1, mine = 0;
            if (whole && live) load_aux(group * CH, row_end);
            if (!whole) {
                first = (sg.tile * p.k_tiles) / p.units_per_cta;
                const int last = ((sg.tile + 1) * p.k_tiles - 1) / p.units_per_cta;
                n_c = last - first + 1;
                mine = pair - first;
                const bool finisher = u >= u_end;                 // this range ends here; one that goes on only contributes
                const int last_end = min(total_units, (last + 1) * p.units_per_cta);
                const int n_fin = n_c - (last_end > (sg.tile + 1) * p.k_tiles ? 1 : 0);
                const int n_chunks = (p.rows + CH - 1) / CH, per = (n_chunks + n_fin - 1) / n_fin;
                row_begin = finisher && live ? min(p.rows, mine * per * CH) : p.rows;
                row_end = finisher && live ? min(p.rows, (mine + 1) * per * CH) : p.rows;
                load_aux(row_begin + group * CH, row_end);
                if (live) {
                    float *slot = p.scratch + ((size_t)blockIdx.x * 2 + (seg_i == 0 ? 0 : 1)) * slot_floats;
                    for (int c = group * CH; c < p.rows; c += WGROUPS * CH) {
                        if (c >= row_begin && c < row_end) continue;       // its own slice stays in TMEM
                        float g[CH];
                        load_chunk(c, g);
#pragma unroll
                        for (int j = 0; j < CH; ++j) slot[(size_t)(c + j) * TILE_F + f] = g[j];
                    }
                    epi_sync();
                    // (the barrier orders the CTA's stores before this release, which is cumulative)
                    if (et == 0) counter_arrive(p.counters + tile, n_c, n_fin);
                    if (finisher) {
                        if (et == 0) counter_wait(p.counters + tile, n_c, n_fin, &abort_sh, p.status);
                        epi_sync();
                    }
                }
            }
            float4 gain_a = make_float4(0.f, 0.f, 0.f, 0.f), gain_b = gain_a;
            if (EPI == EPI_ADD_NORM && row_begin < row_end) {
                gain_a = load_floats4(p.next_gain + tile * TILE_F + 4 * lane);
                gain_b = p.next_gain2 ? load_floats4(p.next_gain2 + tile * TILE_F + 4 * lane) : gain_a;
            }
            // The other contributors' rows are read where they are, a row per warp: 16-byte loads, four contributors of two rows
            // in flight, a chunk ahead (staged in the idle ring by bulk copies first: 13B batch 8 step 6.70 ms, then 6.37; 8B
            // tree batch 4 7.15, then 6.98; a chunk's loads only when its turn came and contributors past the fourth row by
            // row, a trip to L2 each: 8B batch 4 6.72, now 6.57; prompt chunk 25.1, now 24.5).
            const int others = n_c - 1;
            // contributor c's partial of this tile: its first piece of work, but for a first contributor that came from the tile before
            auto slot_of = [&](int c) {
                const int second = c == 0 && first * p.units_per_cta < sg.tile * p.k_tiles;
                return p.scratch + ((size_t)(2 * (first + c) + (int)rank) * 2 + second) * slot_floats + 4 * lane;
            };
            float4 part[4][2];
            auto load_part = [&](int c0, int ra) {
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    if (c0 + c < n_c && c0 + c != mine && ra < row_end) {
                        const float *from = slot_of(c0 + c);
#pragma unroll
                        for (int i = 0; i < 2; ++i)
                            part[c][i] = __ldcg(reinterpret_cast<const float4 *>(from + (size_t)min(ra + i, p.rows - 1) * TILE_F));
                    }
                }
            };
            load_part(0, row_begin + group * CH + 2 * gw);
#pragma unroll 1
            for (int r0 = row_begin + group * CH; r0 < row_end; r0 += WGROUPS * CH) {
                const int ra = r0 + 2 * gw;                        // this warp's two rows of the chunk
                float g[CH];
                load_chunk(r0, g);
                group_sync();                                      // the group has read its previous chunk
#pragma unroll
                for (int j = 0; j < CH; ++j) xg[j * TILE_F + f] = g[j];
                group_sync();
                float4 v[2];
#pragma unroll
                for (int i = 0; i < 2; ++i) v[i] = *reinterpret_cast<const float4 *>(xg + (2 * gw + i) * TILE_F + 4 * lane);
                if (others > 0) {                                  // in pair order, whoever adds them
                    const float4 own[2] = {v[0], v[1]};
                    v[0] = v[1] = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 1
                    for (int c0 = 0; c0 < n_c; c0 += 4) {
                        if (c0 > 0) load_part(c0, ra);
#pragma unroll
                        for (int c = 0; c < 4; ++c)
#pragma unroll
                            for (int i = 0; i < 2; ++i)
                                if (c0 + c < n_c) v[i] = add4(v[i], c0 + c == mine ? own[i] : part[c][i]);
                    }
                    load_part(0, ra + WGROUPS * CH);
                }
#pragma unroll
                for (int i = 0; i < 2; ++i)
                    if (ra + i < p.rows)
                        finish_row<EPI, true>(p, tile, ra + i, true, v[i], make_float4(0.f, 0.f, 0.f, 0.f), aux[i][0], aux[i][1], gain_a, gain_b, inv_sh, rowmeta, lane);
                load_aux(r0 + WGROUPS * CH, row_end);
            }
            // this tile's accumulator may be overwritten
            tc_fence_before();
            __syncwarp();
            if (lane == 0) asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(leader_addr(tempty_bar(buf))) : "memory");
            ++acc_it;
            ++seg_i;
        }
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
    pair_sync();                                                  // the peer's MMAs, loads and arrivals no longer touch this CTA
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(p.tmem_cols) : "memory");
    }
}

}  // namespace

// Rows per plane and sub-tile: the MMA's N is 2 x this, in steps of 32 columns.
int tc_wide_th(int rows) {
    const int per = rows > 128 ? (rows + 1) / 2 : rows;
    return per < 16 ? 16 : (per + 15) / 16 * 16;
}

int launch_gemm_wide(const TcLaunch &L, cudaStream_t st) {
    if (L.rows < 1 || L.rows > WROWS || !L.has_lo) return VIASD_EINVAL;
    TcParams p;
    tc_fill_params(L, p);
    const bool dual = L.epi == EPI_SWIGLU;
    p.tt = L.rows > 128 ? 2 : 1;
    p.slot_rows = (L.rows + CH - 1) / CH * CH;
    p.k_tiles = (L.k + TILE_K - 1) / TILE_K;
    if (dual) p.n_tiles = (L.seg_n[0] + 63) / 64;                  // 64 gate and 64 up features per CTA tile
    if (p.n_tiles <= 0 || p.k_tiles <= 0) return VIASD_OK;
    const int units = ((p.n_tiles + 1) / 2) * p.k_tiles;
    static int resident[64];                                       // pairs the device holds at once, asked once per device
    int dev = 0;
    CUDA_TRY(cudaGetDevice(&dev));
    if (dev < 0 || dev >= 64) return VIASD_EUNSUPPORTED;
    if (!resident[dev]) {
        const int most = 204 * 1024;
        CUDA_TRY(cudaFuncSetAttribute(gemm_wide_kernel<EPI_SWIGLU>, cudaFuncAttributeMaxDynamicSharedMemorySize, most));
        CUDA_TRY(cudaFuncSetAttribute(gemm_wide_kernel<EPI_ADD_NORM>, cudaFuncAttributeMaxDynamicSharedMemorySize, most));
        CUDA_TRY(cudaFuncSetAttribute(gemm_wide_kernel<EPI_QKV_ROPE>, cudaFuncAttributeMaxDynamicSharedMemorySize, most));
        CUDA_TRY(cudaFuncSetAttribute(gemm_wide_kernel<EPI_STORE>, cudaFuncAttributeMaxDynamicSharedMemorySize, most));
        cudaLaunchConfig_t q{};
        cudaLaunchAttribute cluster[1];
        cluster[0].id = cudaLaunchAttributeClusterDimension;
        cluster[0].val.clusterDim.x = 2; cluster[0].val.clusterDim.y = 1; cluster[0].val.clusterDim.z = 1;
        q.gridDim = dim3(2); q.blockDim = dim3(WTHREADS); q.dynamicSmemBytes = most; q.attrs = cluster; q.numAttrs = 1;
        int n = 0;
        CUDA_TRY(cudaOccupancyMaxActiveClusters(&n, gemm_wide_kernel<EPI_QKV_ROPE>, &q));
        if (n < 1) return VIASD_EUNSUPPORTED;
        resident[dev] = n;
    }
    // the finishers of a split tile wait for its other contributors: all pairs have to be resident at once
    int pairs = L.sm_count / 2 < resident[dev] ? L.sm_count / 2 : resident[dev];
    if (pairs > units) pairs = units;
    p.units_per_cta = (units + pairs - 1) / pairs;
    pairs = (units + p.units_per_cta - 1) / p.units_per_cta;
    const size_t xbox = (size_t)p.tt * p.nt * 128, ring = (size_t)(L.ring_kb > 0 ? L.ring_kb : 200) * 1024;
    // Activation slots: 3 with two sub-tiles (a box's MMAs take 900 cycles, L2 answers in 1500); with one, as many as weight
    // slots, since a short range has all its weights in the ring when its dependency is met and then waits for
    // activations only (14 boxes of the 4096 x 4096 projection with 4 slots: 1 us longer).  What is left is weights.
    p.x_stages = p.tt == 2 ? 3 : (int)(ring / (xbox + WBOX));
    if (p.x_stages > 8) p.x_stages = 8;
    while (p.x_stages > 2 && ring < p.x_stages * xbox + 2 * WBOX) --p.x_stages;
    if (p.x_stages < 2) p.x_stages = 2;
    const int stages = ring > p.x_stages * xbox ? (int)((ring - p.x_stages * xbox) / WBOX) : 0;
    p.stages = stages < p.x_stages ? p.x_stages : stages > WSTAGES ? WSTAGES : stages;
    const int acc_cols = p.tt * 2 * p.nt;
    p.acc_bufs = 2 * acc_cols <= 512 ? 2 : 1;
    const int cols = p.acc_bufs * acc_cols;
    p.tmem_cols = cols <= 32 ? 32 : cols <= 64 ? 64 : cols <= 128 ? 128 : cols <= 256 ? 256 : 512;
    const size_t smem = p.stages * (size_t)WBOX + p.x_stages * xbox + 1024;
    const CUtensorMap &w0 = *L.map_w[0], &w1 = *L.map_w[L.n_seg > 1 ? 1 : 0], &w2 = *L.map_w[L.n_seg > 2 ? 2 : 0];
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attr[1];
    pdl_config(cfg, attr, dim3(2 * pairs), dim3(WTHREADS), smem, st, !L.ordered);
    switch (L.epi) {
    case EPI_SWIGLU: CUDA_TRY(cudaLaunchKernelEx(&cfg, gemm_wide_kernel<EPI_SWIGLU>, w0, w1, w2, *L.map_x, p)); break;
    case EPI_ADD_NORM: CUDA_TRY(cudaLaunchKernelEx(&cfg, gemm_wide_kernel<EPI_ADD_NORM>, w0, w1, w2, *L.map_x, p)); break;
    case EPI_QKV_ROPE: CUDA_TRY(cudaLaunchKernelEx(&cfg, gemm_wide_kernel<EPI_QKV_ROPE>, w0, w1, w2, *L.map_x, p)); break;
    case EPI_STORE: CUDA_TRY(cudaLaunchKernelEx(&cfg, gemm_wide_kernel<EPI_STORE>, w0, w1, w2, *L.map_x, p)); break;
    default: return VIASD_EINVAL;
    }
    LAUNCH_CHECK();
    return VIASD_OK;
}
