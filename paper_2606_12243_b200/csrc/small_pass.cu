// A whole forward pass of a small model in one launch: embedding, every layer, output head, for both verifiers at once.
//
// What bounds a small model is neither HBM nor the tensor cores but the chain of launches: a pass of two to six layers whose
// weights fit L2 is 25 to 36 kernels of 4 - 10 us, each a launch (or a dependency), a trip to L2 for the activations and a
// few hundred cycles of arithmetic.  Here the CTAs of one cooperative launch go through the stages together, a grid barrier
// (an arrival counter in L2) between two stages, five per layer:
//
//   1 RMSNorm, Q/K/V projection, rotary embedding, KV append      4 RMSNorm, gate / up projection, SwiGLU
//   2 attention, a (stream, sequence, kv head, key range) per CTA 5 down projection, residual
//   3 output projection, residual                                 and at the end: final RMSNorm, output head
//
// A projection's unit is 8 or 16 output features by one CTA; its eight warps share k in groups of 32, and their sums meet in
// shared memory.  A unit's weights do not depend on the pass, so a warp asks for those of the next projection (cp.async)
// between its arrival at a barrier and the wait there.  Activations come from L2 after the barrier, each warp its own groups of
// k of all rows.
//
// bf16 models: mma.sync m16n8k16, weights exact, activations as bf16 pairs hi + lo as in the kernels for large models (a unit
// is too small for a tcgen05 tile: 8 features against 128 lanes).  fp32 models: CUDA cores, fp32 throughout.  A row's results do
// not depend on whether one or both verifiers' rows are in the launch, nor on the values of other rows; on how many there are only by
// the key ranges of its attention (Grouping::ranges).
//
// One step, launches before / one launch: two fp32 layers of d 256, 5 rows 145 / 69 us; four bf16 layers of d 512, 9 rows 164 / 120.
// What bounds it now (cycles per stage): stores to arrival 1000, arrival to exit 1000, activations from L2 700 - 2400 (every CTA
// reads all rows), arithmetic 500 - 2500, finishing 600; attention 8000 with the merge of its key ranges.
#include "common.cuh"
#include "tc_ptx.cuh"
#include <string.h>
#include <type_traits>

namespace {

constexpr int SP_WARPS = 8, SP_THREADS = 32 * SP_WARPS;
constexpr int KG = 32;                          // columns of k per group
constexpr int XGROUP = KG * 4 + 16;             // bytes of a staged row's group (16 more than it has keep 16-byte reads off each other's banks)
constexpr int SP_ROWS = SMALL_PASS_MAX_ROWS;    // token rows of both streams together
constexpr int SP_QG = 16;                       // query rows of an attention item
constexpr int SP_SPLITS = 8;                    // key ranges of an attention pair, at most
constexpr int NU = 2, TN = 2 * NU;              // units a CTA works on together, and their tiles of 8 features

struct SpLayer {
    const void *wq, *wk, *wv, *wo, *wg, *wu, *wd;
    const float *n1, *n2, *next[2];             // gains; per stream, that of the norm behind this layer
    int ord[2];                                 // the layer's place in each stream's cache, -1: the stream does not take part
};
struct SpArgs {
    int B, M, R, streams;                       // rows per sequence, rows per stream (B * M)
    int d, ff, qd, V, H, Hkv, n_layers, max_batch, max_ctx, nsplit, att_items;   // att_items: of one stream
    int first[2];                               // each stream's first layer: its input is the embedding
    int skip;                                   // rows of every sequence in front of the block's own (replay pass): no logits
    float eps, inv_d, att_scale;
    const void *embed, *head;
    const float *final_norm, *cosv, *sinv;
    void *kc[2], *vc[2];
    float *logits[2];
    float *h, *part;                            // residual stream; partial rows of the attention
    uint4 *xn, *q, *attn, *act;                 // inputs of the projections and of the attention, in chunks (see put_elem)
    float *ssq;                                 // [row][d / 8] sums of squares of the residual stream
    float2 *part_ml;
    const int *len, *pending, *draft_tok, *parent, *row_tok, *kv_keep;
    int N, per_seq, full_pass, kv_vec;          // kv_vec: the caches are aligned to 16 bytes
    TreeInfo *tree;
    int *len_eff;
    DeviceStats *stats;
    const int *run_flag;
    int *counters;                              // which set; the two sets: barriers, used in turn, and arrivals of each attention pair's ranges
    int set_words;
    int red_bytes, w_bytes, x_bytes;            // shared memory: sums; a stage's weights; a warp's staged activations,
    int x_groups, x_rows;                       // that many groups of k (bf16) of that many rows (fp32: all groups) at a time
    SpLayer layer[SMALL_PASS_MAX_LAYERS];
};

__device__ __forceinline__ void cp16(uint32_t dst, const void *src, bool on) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(on ? 16 : 0) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cp_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }
__device__ __forceinline__ float4 lds4(const float *p) { return *reinterpret_cast<const float4 *>(p); }
__device__ __forceinline__ uint4 ldsu4(const void *p) { return *reinterpret_cast<const uint4 *>(p); }
__device__ __forceinline__ void mma_bf16(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void ldsm_x4(uint32_t addr, uint32_t (&r)[4]) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void ldsm_x4_t(uint32_t addr, uint32_t (&r)[4]) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void split_bf16(float x0, float x1, uint32_t &hi, uint32_t &lo) {
    const __nv_bfloat162 h = __floats2bfloat162_rn(x0, x1);
    hi = *reinterpret_cast<const uint32_t *>(&h);
    const __nv_bfloat162 l = __floats2bfloat162_rn(x0 - __uint_as_float(hi << 16), x1 - __uint_as_float(hi & 0xffff0000u));
    lo = *reinterpret_cast<const uint32_t *>(&l);
}
// four consecutive elements of a caller's array as floats
__device__ __forceinline__ float4 load4(const float *p) { return load_floats4(p); }
__device__ __forceinline__ float4 load4(const __nv_bfloat16 *p) {
    if (reinterpret_cast<uintptr_t>(p) & 7) return make_float4(to_f32(p[0]), to_f32(p[1]), to_f32(p[2]), to_f32(p[3]));
    const uint2 u = __ldg(reinterpret_cast<const uint2 *>(p));
    return make_float4(__uint_as_float(u.x << 16), __uint_as_float(u.x & 0xffff0000u), __uint_as_float(u.y << 16), __uint_as_float(u.y & 0xffff0000u));
}

// What a projection (or the attention, the queries) multiplies is kept in chunks of eight columns, 32 bytes: eight floats, or for
// bf16 models the eight hi parts and then the eight lo parts, so that a consumer's fragment is two 16-byte reads and no
// arithmetic.
__device__ __forceinline__ void put_elem(float *, uint4 *buf, size_t chunk, int f, float v) { reinterpret_cast<float *>(buf + 2 * chunk)[f] = v; }
__device__ __forceinline__ void put_elem(__nv_bfloat16 *, uint4 *buf, size_t chunk, int f, float v) {
    __nv_bfloat16 *to = reinterpret_cast<__nv_bfloat16 *>(buf + 2 * chunk) + f;
    const __nv_bfloat16 hi = __float2bfloat16_rn(v);
    to[0] = hi;
    to[8] = __float2bfloat16_rn(v - __bfloat162float(hi));
}
// four columns from 4 * half on
__device__ __forceinline__ void put_four(float *, uint8_t *chunk, int half, float4 v) { *reinterpret_cast<float4 *>(chunk + 16 * half) = v; }
__device__ __forceinline__ void put_four(__nv_bfloat16 *, uint8_t *chunk, int half, float4 v) {
    uint2 hi, lo;
    split_bf16(v.x, v.y, hi.x, lo.x);
    split_bf16(v.z, v.w, hi.y, lo.y);
    *reinterpret_cast<uint2 *>(chunk + 8 * half) = hi;
    *reinterpret_cast<uint2 *>(chunk + 16 + 8 * half) = lo;
}

enum { ST_QKV, ST_O, ST_GU, ST_DOWN, ST_HEAD };
__host__ __device__ constexpr int stage_tiles(int st) { return st == ST_O || st == ST_DOWN ? 1 : 2; }   // tiles of 8 features per unit
__host__ __device__ constexpr bool stage_norm(int st) { return st == ST_QKV || st == ST_GU || st == ST_HEAD; }

template <typename T, int HD, int MT>
struct Pass {
    static constexpr bool BF = std::is_same<T, __nv_bfloat16>::value;
    static constexpr int WGROUP = BF ? 512 : 1024, WSTEP = SP_WARPS * WGROUP;    // bytes of 8 features x 32 columns; of all warps'
    // attention: keys per tile, bytes of a staged row (16 more than the row, for the banks)
    static constexpr int TKS = HD * (int)sizeof(T) <= 256 ? 64 : 32, KVROW = HD * (int)sizeof(T) + 16, KV_BYTES = 2 * TKS * KVROW;

    struct Shared {
        SpLayer layer[SMALL_PASS_MAX_LAYERS];                   // (read by number from the launch's arguments, each pointer was a miss)
        float inv[SP_ROWS];                                     // the norm's factor of every row
        float q[SP_QG][HD + 4];                                 // query rows, in chunks
        float s[SP_QG][TKS + 4];                                // scores, or fp32 probabilities, of a tile
        __nv_bfloat16 ph[SP_QG][TKS + 8], pl[SP_QG][TKS + 8];   // probabilities as bf16 pairs
        float corr[SP_QG];
        // query rows of the CTA's first attention item, and of a later one: ancestors; token row * H + head
        unsigned long long q_anc[2][SP_QG];
        int q_at[2][SP_QG];
        unsigned long long anc[SP_ROWS];                        // per row of a stream
        int tok[SP_ROWS], pos[SP_ROWS], slot[SP_ROWS], n_ctx[SP_ROWS], seq[SP_ROWS];
        TreeInfo tree[SP_WARPS];
        int par[SP_WARPS][VIASD_MAX_ROWS_PER_SEQ];
        int *counters;                                          // this launch's set
        int n_bar, abort_flag, last;
    };
    struct Range { int pair, s, b, kvh, row0, rows, split, n, k0, k1; };

    const SpArgs &a;
    Shared &sh;
    float *red;                                                 // [warp][row][feature] the warps' sums of the units in hand
    uint8_t *wbuf;                                              // weights of the stage to come
    uint8_t *xbuf;                                              // this warp's staged activations, in one place with
    uint8_t *kvbuf;                                             // two K/V tiles: no stage uses both
    const int tid, warp, lane, g, c;

    __device__ Pass(const SpArgs &a_, uint8_t *smem) : a(a_), sh(*reinterpret_cast<Shared *>(smem)), tid(threadIdx.x), warp(threadIdx.x >> 5),
        lane(threadIdx.x & 31), g((threadIdx.x & 31) >> 2), c(threadIdx.x & 3) {
        red = reinterpret_cast<float *>(smem + (sizeof(Shared) + 127) / 128 * 128);
        wbuf = reinterpret_cast<uint8_t *>(red) + a.red_bytes;
        kvbuf = wbuf + a.w_bytes;
        xbuf = kvbuf + (size_t)warp * a.x_bytes;
    }

    template <int ST> __device__ __forceinline__ int stage_k() const { return ST == ST_O ? a.qd : ST == ST_DOWN ? a.ff : a.d; }
    template <int ST> __device__ __forceinline__ int stage_per() const { return (stage_k<ST>() + KG * SP_WARPS - 1) / (KG * SP_WARPS); }   // groups of k per warp
    template <int ST> __device__ __forceinline__ int stage_units() const {
        return ST == ST_QKV ? (a.H + 2 * a.Hkv) * (HD / 16) : ST == ST_GU ? a.ff / 8 : ST == ST_HEAD ? (a.V + 15) / 16 : a.d / 8;
    }
    // weight row of feature `f` (0..7) of a unit's tile; null past the last one
    template <int ST> __device__ __forceinline__ const T *weight(const SpLayer &l, int unit, int tile, int f) const {
        const void *w;
        int row;
        if (ST == ST_QKV) {
            const int hh = unit / (HD / 16), p = (unit % (HD / 16)) * 8 + f + tile * (HD / 2);         // a pair of rotary partners
            w = hh < a.H ? l.wq : hh < a.H + a.Hkv ? l.wk : l.wv;
            row = (hh < a.H ? hh : hh < a.H + a.Hkv ? hh - a.H : hh - a.H - a.Hkv) * HD + p;
        } else if (ST == ST_HEAD) {
            row = unit * 16 + tile * 8 + f;
            w = row < a.V ? a.head : nullptr;
        } else {
            w = ST == ST_GU ? (tile ? l.wu : l.wg) : ST == ST_O ? l.wo : l.wd;
            row = unit * 8 + f;
        }
        return w ? reinterpret_cast<const T *>(w) + (size_t)row * stage_k<ST>() : nullptr;
    }
    // This warp's share of the weights of all of the CTA's units (every lane brings what it will itself read): [tile][group][warp]
    template <int ST> __device__ __forceinline__ void prefetch(const SpLayer &l) {
        constexpr int NT = stage_tiles(ST);
        const int K = stage_k<ST>(), per = stage_per<ST>(), units = stage_units<ST>();
        uint32_t dst = smem_u32(wbuf) + warp * WGROUP + lane * 16;
#pragma unroll 1
        for (int u = blockIdx.x; u < units; u += gridDim.x) {
#pragma unroll
            for (int t = 0; t < NT; ++t) {
                const T *row = weight<ST>(l, u, t, g);
                int k = warp * KG + c * 8;
                const T *src = row + k;
#pragma unroll 2
                for (int i = 0; i < per; ++i, dst += WSTEP, k += KG * SP_WARPS, src += KG * SP_WARPS) {
                    const bool on = (ST != ST_HEAD || row) && k < K;
                    cp16(dst, on ? src : reinterpret_cast<const T *>(a.head), on);
                    if (!BF) cp16(dst + 512, on ? src + 4 : reinterpret_cast<const T *>(a.head), on);
                }
            }
        }
        cp_commit();
    }

    // All CTAs have arrived, and what they stored before is seen behind this; `meanwhile` runs between arrival and wait.  (A ninth
    // warp for the barriers, so that no warp's prefetch waits behind the release: 168 registers for all, mini 121 -> 127 us.)
    template <typename F> __device__ __forceinline__ void barrier(F meanwhile) {
        int *ctr = sh.counters + (sh.n_bar & 1);                // (ahead of the barrier: its latency is not the arrival's)
        __syncthreads();
        // (a counter is used again two barriers later: by then every CTA has acknowledged its last use)
        if (tid == 0) counter_arrive(ctr, gridDim.x, gridDim.x);
        meanwhile();
        if (tid == 0) counter_wait(sh.counters + (sh.n_bar++ & 1), gridDim.x, gridDim.x, &sh.abort_flag, &a.stats->device_status);
        __syncthreads();
    }

    // Behind a barrier, so that all CTAs know their set: the other one, which the launch before this one used, becomes the
    // next launch's, from zero.  Counters come back to zero by themselves, also when a wait expires; one that is off all the same
    // (a launch that was cut short, a stray write) costs one launch its results, not the handle.  (Cleared at a launch's head they
    // would meet arrivals of CTAs that are further on, and by a kernel in front of it every pass would pay a launch.)
    __device__ __forceinline__ void hand_over() {
        if (blockIdx.x) return;
        const int next = sh.counters == a.counters + SMALL_PASS_LINE ? 1 : 0;
        for (int i = tid; i < a.set_words; i += SP_THREADS) a.counters[SMALL_PASS_LINE + next * a.set_words + i] = 0;
        if (tid == 0) a.counters[0] = next;
    }

    // ---- the input of k-groups i0 .. i0 + n - 1 of this warp, rows r_lo .. r_lo + r_n - 1, to shared memory ----
    __device__ __forceinline__ uint8_t *staged(int j, int row, int r_n) const { return xbuf + (j * r_n + row) * XGROUP; }
    template <int ST> __device__ __forceinline__ bool from_embedding(int layer, int s) const { return ST == ST_QKV && a.first[s] == layer; }
    __device__ __forceinline__ const T *embedding(int r) const { return reinterpret_cast<const T *>(a.embed) + (size_t)sh.tok[r >= a.R ? r - a.R : r] * a.d; }
    template <int ST> __device__ __forceinline__ void stage_x(int layer, int i0, int n, int r_lo, int r_n) {
        const int K = stage_k<ST>(), sub = lane >> 3, piece = lane & 7;      // 16 bytes of a group's 128
        if (from_embedding<ST>(layer, 0) || from_embedding<ST>(layer, 1)) {
            for (int j = 0; j < n; ++j)
                for (int x = sub; x < r_n; x += 4) {
                    const int r = r_lo + x, k = (warp + SP_WARPS * (i0 + j)) * KG + piece * 4;
                    if (!from_embedding<ST>(layer, r >= a.R)) continue;
                    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
                    if (k < K) {
                        const float4 e = load4(embedding(r) + k), gn = load_floats4(sh.layer[layer].n1 + k);
                        v = make_float4(e.x * gn.x, e.y * gn.y, e.z * gn.z, e.w * gn.w);
                    }
                    put_four((T *)nullptr, staged(j, x, r_n) + (piece >> 1) * 32, piece & 1, v);
                }
        }
        const uint4 *from = (ST == ST_DOWN ? a.act : ST == ST_O ? a.attn : a.xn) + (size_t)(r_lo + sub) * (K / 4) + piece;
        uint32_t dst = smem_u32(staged(0, sub, r_n)) + piece * 16;
        int group = warp + SP_WARPS * i0;
#pragma unroll 1
        for (int j = 0; j < n; ++j, group += SP_WARPS, dst += r_n * XGROUP) {
            const bool in = group * KG + (piece >> 1) * 8 < K;
            const uint4 *src = from + (in ? group * (KG / 4) : 0);
            uint32_t to = dst;
#pragma unroll 4
            for (int x = sub; x < r_n; x += 4, src += K, to += 4 * XGROUP) {         // (four rows of K / 4 pieces)
                if (ST == ST_QKV && from_embedding<ST>(layer, r_lo + x >= a.R)) continue;
                cp16(to, src, in);
            }
        }
    }
    // The norm's factors: eight lanes per row, from the sums of squares that the projection before this one left, or from the
    // embedding.  Asked for ahead of the activations (behind their 30 KB the answer took twice as long), added up behind them.
    struct NormPart { float v[8]; };
    template <int ST> __device__ __forceinline__ void norm_ask(int layer, int rows, NormPart &p) {
        const int n = a.d / 8, f = lane & 7, r = min(warp * 4 + (lane >> 3), rows - 1);
        if (warp * 4 >= rows || from_embedding<ST>(layer, r >= a.R)) return;
        const float *src = a.ssq + (size_t)r * n + f;
#pragma unroll
        for (int x = 0; x < 8; ++x) p.v[x] = f + 8 * x < n ? __ldcg(src + 8 * x) : 0.f;
    }
    template <int ST> __device__ __forceinline__ void norm_factors(int layer, int rows, const NormPart &p) {
        const int n = a.d / 8, f = lane & 7;
        for (int r0 = warp * 4; r0 < rows; r0 += SP_WARPS * 4) {
            const int r = min(r0 + (lane >> 3), rows - 1);
            float q = 0.f;
            if (from_embedding<ST>(layer, r >= a.R)) {
                const T *e = embedding(r);
#pragma unroll 4
                for (int k = f; k < n; k += 8) {
                    const float4 v = load4(e + 8 * k), w = load4(e + 8 * k + 4);
                    q += ((v.x * v.x + v.y * v.y) + (v.z * v.z + v.w * v.w)) + ((w.x * w.x + w.y * w.y) + (w.z * w.z + w.w * w.w));
                }
            } else {
                const float *src = a.ssq + (size_t)r * n;
#pragma unroll
                for (int x = 0; x < 8; ++x) q += r0 == warp * 4 ? p.v[x] : f + 8 * x < n ? __ldcg(src + f + 8 * x) : 0.f;
#pragma unroll 4
                for (int k = f + 64; k < n; k += 8) q += __ldcg(src + k);
            }
#pragma unroll
            for (int o = 4; o > 0; o >>= 1) q += __shfl_xor_sync(0xffffffffu, q, o);
            if (f == 0) sh.inv[r] = rsqrtf(q * a.inv_d + a.eps);
        }
    }
    // bf16: sums over this warp's staged groups, NTL tiles (weights from w on), rows 16 m + g and + 8; hi and lo products apart
    template <int NTL> __device__ __forceinline__ void multiply(float (&acc)[MT][TN][4], float (&al)[MT][2][4], const uint8_t *w, int per, int i0, int n, int rows) {
        constexpr bool APART = NTL <= 2;                         // (two chains of products; with four tiles there are enough of them)
        const uint8_t *at[MT][2];                                // rows g, g + 8 (past the end: the last one again, unstored)
#pragma unroll
        for (int m = 0; m < MT; ++m)
#pragma unroll
            for (int e = 0; e < 2; ++e) at[m][e] = staged(0, min(m * 16 + g + 8 * e, rows - 1), rows) + c * 32;
        w += i0 * WSTEP;
#pragma unroll 1
        for (int j = 0; j < n; ++j, w += WSTEP) {
            uint4 b[NTL];
#pragma unroll
            for (int t = 0; t < NTL; ++t) b[t] = ldsu4(w + t * per * WSTEP);
#pragma unroll
            for (int m = 0; m < MT; ++m) {
                const uint4 ha = ldsu4(at[m][0]), la = ldsu4(at[m][0] + 16), hb = ldsu4(at[m][1]), lb = ldsu4(at[m][1] + 16);
                at[m][0] += rows * XGROUP; at[m][1] += rows * XGROUP;
                const uint32_t h0[4] = {ha.x, hb.x, ha.y, hb.y}, h1[4] = {ha.z, hb.z, ha.w, hb.w};
                const uint32_t l0[4] = {la.x, lb.x, la.y, lb.y}, l1[4] = {la.z, lb.z, la.w, lb.w};
#pragma unroll
                for (int t = 0; t < NTL; ++t) { mma_bf16(APART ? al[m][t & 1] : acc[m][t], l0, b[t].x, b[t].y); if (APART) mma_bf16(acc[m][t], h0, b[t].x, b[t].y); }
                if (!APART) {
#pragma unroll
                    for (int t = 0; t < NTL; ++t) mma_bf16(acc[m][t], h0, b[t].x, b[t].y);
                }
#pragma unroll
                for (int t = 0; t < NTL; ++t) { mma_bf16(APART ? al[m][t & 1] : acc[m][t], l1, b[t].z, b[t].w); if (APART) mma_bf16(acc[m][t], h1, b[t].z, b[t].w); }
                if (!APART) {
#pragma unroll
                    for (int t = 0; t < NTL; ++t) mma_bf16(acc[m][t], h1, b[t].z, b[t].w);
                }
            }
        }
    }
    // fp32: up to eight staged rows from r0 on; lane (g, c): feature g of each tile, columns 8c .. 8c+7 of every group
    template <int NTL> __device__ __forceinline__ void multiply(const uint8_t *w, int per, int r0, int r_n, float *to) {
        float s[8][NTL];
#pragma unroll
        for (int r = 0; r < 8; ++r)
#pragma unroll
            for (int t = 0; t < NTL; ++t) s[r][t] = 0.f;
#pragma unroll 2
        for (int j = 0; j < per; ++j, w += WSTEP) {
            float4 b[NTL][2];
#pragma unroll
            for (int t = 0; t < NTL; ++t) {
                b[t][0] = *reinterpret_cast<const float4 *>(w + t * per * WSTEP);
                b[t][1] = *reinterpret_cast<const float4 *>(w + t * per * WSTEP + 512);
            }
#pragma unroll
            for (int r = 0; r < 8; ++r) {
                const float *src = reinterpret_cast<const float *>(staged(j, min(r0 + r, r_n - 1), r_n)) + c * 8;
                const float4 v0 = lds4(src), v1 = lds4(src + 4);
#pragma unroll
                for (int t = 0; t < NTL; ++t) {
                    s[r][t] = fmaf(v0.x, b[t][0].x, s[r][t]); s[r][t] = fmaf(v0.y, b[t][0].y, s[r][t]);
                    s[r][t] = fmaf(v0.z, b[t][0].z, s[r][t]); s[r][t] = fmaf(v0.w, b[t][0].w, s[r][t]);
                    s[r][t] = fmaf(v1.x, b[t][1].x, s[r][t]); s[r][t] = fmaf(v1.y, b[t][1].y, s[r][t]);
                    s[r][t] = fmaf(v1.z, b[t][1].z, s[r][t]); s[r][t] = fmaf(v1.w, b[t][1].w, s[r][t]);
                }
            }
        }
#pragma unroll
        for (int r = 0; r < 8; ++r) {
#pragma unroll
            for (int t = 0; t < NTL; ++t) {
                s[r][t] += __shfl_xor_sync(0xffffffffu, s[r][t], 1);
                s[r][t] += __shfl_xor_sync(0xffffffffu, s[r][t], 2);
            }
            float v = s[r][0];                                   // lane (g, c) stores tile c's sum
            if (NTL >= 2) v = c & 1 ? s[r][NTL >= 2 ? 1 : 0] : v;
            if (NTL == 4) v = c & 2 ? (c & 1 ? s[r][NTL - 1] : s[r][NTL >= 3 ? 2 : 0]) : v;
            if (c < NTL && r0 + r < r_n) to[r * (TN * 8)] = v;
        }
    }
    // What finishing a sum reads besides it, asked for ahead of the arithmetic: the residual and the gain, or cosine and sine.
    template <int ST> __device__ __forceinline__ float2 aux(int layer, int unit, int r, int f) const {
        if (ST == ST_O || ST == ST_DOWN) {
            const int col = unit * 8 + f, s = r >= a.R;
            const SpLayer &l = sh.layer[layer];
            const bool emb = ST == ST_O && a.first[s] == layer;
            return make_float2(emb ? to_f32<T>(embedding(r)[col]) : __ldcg(a.h + (size_t)r * a.d + col), __ldg((ST == ST_O ? l.n2 : l.next[s]) + col));
        }
        if (ST == ST_QKV) {
            const size_t o = (size_t)sh.pos[r >= a.R ? r - a.R : r] * (HD / 2) + (unit % (HD / 16)) * 8 + f;
            return make_float2(__ldg(a.cosv + o), __ldg(a.sinv + o));
        }
        return make_float2(0.f, 0.f);
    }
    // ---- a projection: the sums of every row for the CTA's units, two units at a time (with one after the other, the CTAs that
    // have two took half as long again: gate / up of d_ff 1408 is 176 units on 148 CTAs) ----
    template <int ST> __device__ __forceinline__ void project(int layer, int rows) {
        constexpr int NT = stage_tiles(ST);
        const int per = stage_per<ST>(), units = stage_units<ST>(), batch = min(per, a.x_groups);
        const uint8_t *w = wbuf + warp * WGROUP + lane * 16;
        bool fresh = true;
#pragma unroll 1
        for (int u = blockIdx.x; u < units; u += NU * gridDim.x) {
            const bool two = u + (int)gridDim.x < units;
            const int n_t = two ? 2 * NT : NT, total = rows * 8 * (two ? 2 : 1);     // tiles in hand; sums to finish
            // element e of them: feature e & 7 of a row of the first unit, then of the second
            auto row_of = [&](int e) { return (e >= rows * 8 ? e - rows * 8 : e) >> 3; };
            auto unit_of = [&](int e) { return e >= rows * 8 ? u + (int)gridDim.x : u; };
            const float2 ax0 = tid < total ? aux<ST>(layer, unit_of(tid), row_of(tid), tid & 7) : make_float2(0.f, 0.f);
            const bool norm = stage_norm(ST) && fresh;
            NormPart np;
            if (norm) norm_ask<ST>(layer, rows, np);
            if (BF) {
                float acc[MT][TN][4], al[MT][2][4] = {};         // al: the lo parts' products; added at the end, however many batches k came in
#pragma unroll
                for (int m = 0; m < MT; ++m)
#pragma unroll
                    for (int t = 0; t < TN; ++t)
#pragma unroll
                        for (int e = 0; e < 4; ++e) acc[m][t][e] = 0.f;
#pragma unroll 1
                for (int i0 = 0; i0 < per; i0 += batch) {
                    const int n = min(batch, per - i0);
                    if (fresh || batch < per) {
                        __syncwarp();                            // what was staged before has been read
                        stage_x<ST>(layer, i0, n, 0, rows);
                        if (norm && i0 == 0) norm_factors<ST>(layer, rows, np);
                        cp_wait_all();
                        __syncwarp();
                    }
                    if constexpr (BF) { if (two) multiply<2 * NT>(acc, al, w, per, i0, n, rows); else multiply<NT>(acc, al, w, per, i0, n, rows); }
                }
#pragma unroll
                for (int m = 0; m < MT; ++m)
#pragma unroll
                    for (int e = 0; e < 2; ++e)
                        if (m * 16 + g + 8 * e < rows) {
                            float *to = red + (warp * rows + m * 16 + g + 8 * e) * (TN * 8) + 2 * c;
#pragma unroll
                            for (int t = 0; t < TN; ++t) if (t < n_t) *reinterpret_cast<float2 *>(to + t * 8) = t < 2 ? make_float2(acc[m][t][2 * e] + al[m][t][2 * e], acc[m][t][2 * e + 1] + al[m][t][2 * e + 1])
                                                                                                 : make_float2(acc[m][t][2 * e], acc[m][t][2 * e + 1]);
                        }
            } else {
                // a few rows at a time, all of this warp's k
#pragma unroll 1
                for (int r_lo = 0; r_lo < rows; r_lo += a.x_rows) {
                    const int r_n = min(a.x_rows, rows - r_lo);
                    const bool stage = fresh || rows > a.x_rows;
                    if (stage) {
                        __syncwarp();
                        stage_x<ST>(layer, 0, per, r_lo, r_n);
                    }
                    if (norm && r_lo == 0) norm_factors<ST>(layer, rows, np);
                    if (stage) { cp_wait_all(); __syncwarp(); }
#pragma unroll 1
                    for (int r0 = 0; r0 < r_n; r0 += 8) {
                        float *to = red + (warp * rows + r_lo + r0) * (TN * 8) + c * 8 + g;
                        if constexpr (!BF) { if (two) multiply<2 * NT>(w, per, r0, r_n, to); else multiply<NT>(w, per, r0, r_n, to); }
                    }
                }
            }
            w += n_t * per * WSTEP;
            __syncthreads();
#pragma unroll 1
            for (int e0 = 0; e0 < total; e0 += SP_THREADS) {
                const int e = min(e0 + tid, total - 1), f = e & 7, r = row_of(e);
                const float *from = red + r * (TN * 8) + (e >= rows * 8 ? NT * 8 : 0) + f;
                float x[2] = {0.f, 0.f};
#pragma unroll
                for (int t = 0; t < NT; ++t)
#pragma unroll
                    for (int i = 0; i < SP_WARPS; ++i) x[t] += from[i * rows * (TN * 8) + t * 8];
                if (stage_norm(ST)) { x[0] *= sh.inv[r]; x[1] *= sh.inv[r]; }
                finish<ST>(layer, unit_of(e), r, f, x[0], x[1], e0 > 0 ? aux<ST>(layer, unit_of(e), r, f) : ax0, e0 + tid < total);
            }
            fresh = false;
            if (u + NU * (int)gridDim.x < units) __syncthreads();
        }
    }
    // row r, feature f of a unit: the sums of its first tile and of its second one (whole warps; on: to be stored)
    template <int ST> __device__ __forceinline__ void finish(int layer, int unit, int r, int f, float x, float y, float2 ax, bool on) {
        const int s = r >= a.R, rs = r - s * a.R;
        T *const type = nullptr;
        if (ST == ST_O || ST == ST_DOWN) {
            // the residual stream, and what the norm behind it needs: x * gain, sums of x^2 per eight columns
            x += ax.x;
            float q = x * x;
#pragma unroll
            for (int o = 4; o > 0; o >>= 1) q += __shfl_xor_sync(0xffffffffu, q, o);
            if (!on) return;
            a.h[(size_t)r * a.d + unit * 8 + f] = x;
            put_elem(type, a.xn, (size_t)r * (a.d / 8) + unit, f, x * ax.y);
            if (f == 0) a.ssq[(size_t)r * (a.d / 8) + unit] = q;
            return;
        }
        if (!on) return;
        if (ST == ST_QKV) {
            const int hh = unit / (HD / 16), p8 = unit % (HD / 16), p = p8 * 8 + f;
            if (hh < a.H + a.Hkv) {
                const float y1 = x * ax.x - y * ax.y, y2 = y * ax.x + x * ax.y;
                x = y1; y = y2;
            }
            if (hh < a.H) {
                const size_t chunk = ((size_t)r * a.H + hh) * (HD / 8) + p8;
                put_elem(type, a.q, chunk, f, x * a.att_scale);
                put_elem(type, a.q, chunk + HD / 16, f, y * a.att_scale);
            } else if (sh.slot[rs] >= 0) {
                const int kv = hh < a.H + a.Hkv ? hh - a.H : hh - a.H - a.Hkv;
                T *dst = reinterpret_cast<T *>(hh < a.H + a.Hkv ? a.kc[s] : a.vc[s]) +
                         ((((size_t)sh.layer[layer].ord[s] * a.max_batch + sh.seq[rs]) * a.Hkv + kv) * a.max_ctx + sh.slot[rs]) * HD + p;
                dst[0] = from_f32<T>(x); dst[HD / 2] = from_f32<T>(y);
            }
        } else if (ST == ST_GU) {
            const float e = BF ? __expf(-x) : expf(-x);
            put_elem(type, a.act, (size_t)r * (a.ff / 8) + unit, f, x / (1.f + e) * y);
        } else {
            const int b = sh.seq[rs], i = rs - b * a.M - a.skip, n = unit * 16 + f;
            if (i < 0) return;                                  // a replayed row
            float *dst = a.logits[s] + ((size_t)b * (a.M - a.skip) + i) * a.V + n;
            if (n < a.V) dst[0] = x;
            if (n + 8 < a.V) dst[8] = y;
        }
    }

    // ---- attention: item = (stream, sequence, kv head, group of query rows, key range); its rows' tables to place `tab` ----
    __device__ __forceinline__ void att_item(int id, int tab, Range &it) const {
        const int grp = a.H / a.Hkv, QR = grp * a.M, qgroups = (QR + SP_QG - 1) / SP_QG;
        it.pair = id / a.nsplit;
        it.split = id - it.pair * a.nsplit;
        const int x = it.pair / qgroups, qg = it.pair - x * qgroups, be = x / a.Hkv;
        it.kvh = x - be * a.Hkv;
        it.s = be >= a.B; it.b = be - it.s * a.B;
        it.row0 = qg * SP_QG;
        it.rows = min(SP_QG, QR - it.row0);
        it.n = sh.n_ctx[it.b * a.M];
        const int Tk = it.n + a.M, chunk = ((Tk + a.nsplit - 1) / a.nsplit + 31) / 32 * 32;
        it.k0 = min(Tk, it.split * chunk);
        it.k1 = min(Tk, it.k0 + chunk);
        if (tid < SP_QG) {                                      // (rows past the end repeat the last one, unstored)
            const int qi = it.row0 + min(tid, it.rows - 1), h = qi / a.M, i = qi - h * a.M;
            sh.q_anc[tab][tid] = sh.anc[it.b * a.M + i];
            sh.q_at[tab][tid] = (it.s * a.R + it.b * a.M + i) * a.H + it.kvh * grp + h;
        }
    }
    __device__ __forceinline__ void load_kv(const Range &it, int ord, int k0, uint8_t *buf) {
        const size_t base = (((size_t)ord * a.max_batch + it.b) * a.Hkv + it.kvh) * (size_t)a.max_ctx * HD;
        const T *kc = reinterpret_cast<const T *>(a.kc[it.s]) + base, *vc = reinterpret_cast<const T *>(a.vc[it.s]) + base;
        constexpr int PIECES = HD * (int)sizeof(T) / 16;
        const uint32_t dst = smem_u32(buf);
#pragma unroll 4
        for (int e = tid; e < TKS * PIECES; e += SP_THREADS) {
            const int j = e / PIECES, p = e - j * PIECES;
            const bool on = k0 + j < it.k1;                     // (what the cache holds past the block is not read into the result: zeros)
            const size_t o = (size_t)(on ? k0 + j : it.k0) * HD + p * (16 / sizeof(T));
            if (BF || a.kv_vec) {
                cp16(dst + j * KVROW + p * 16, kc + o, on);
                cp16(dst + TKS * KVROW + j * KVROW + p * 16, vc + o, on);
            } else {                                            // an fp32 cache need only be aligned to its element
                T *to = reinterpret_cast<T *>(buf + j * KVROW + p * 16);
#pragma unroll
                for (int x = 0; x < 16 / (int)sizeof(T); ++x) {
                    to[x] = on ? __ldcg(kc + o + x) : T(0.f);
                    to[x + TKS * KVROW / (int)sizeof(T)] = on ? __ldcg(vc + o + x) : T(0.f);
                }
            }
        }
        cp_commit();
    }
    // softmax of a tile's scores: rows warp and warp + 8 (NR 2) side by side.  (bf16: rows without a probability are not stored either.)
    template <int NR> __device__ __forceinline__ void softmax(float (&m)[2], float (&lsum)[2], float (&o)[2][4]) {
        constexpr int NK = TKS / 32, DPL = HD / 32;
        float x[NR][NK], mx[NR], ref[NR], corr[NR], sum[NR];
#pragma unroll
        for (int r = 0; r < NR; ++r) {
            mx[r] = -INFINITY; sum[r] = 0.f;
#pragma unroll
            for (int y = 0; y < NK; ++y) { x[r][y] = sh.s[warp + SP_WARPS * r][lane + 32 * y]; mx[r] = fmaxf(mx[r], x[r][y]); }
        }
#pragma unroll
        for (int z = 16; z > 0; z >>= 1)
#pragma unroll
            for (int r = 0; r < NR; ++r) mx[r] = fmaxf(mx[r], __shfl_xor_sync(0xffffffffu, mx[r], z));
#pragma unroll
        for (int r = 0; r < NR; ++r) {
            const int row = warp + SP_WARPS * r;
            const float mnew = fmaxf(m[r], mx[r]);
            ref[r] = mnew == -INFINITY ? 0.f : mnew;             // (no visible key yet: weights are e^-inf)
            corr[r] = mnew == -INFINITY ? 1.f : BF ? ex2(m[r] - ref[r]) : expf(m[r] - ref[r]);
            m[r] = mnew;
#pragma unroll
            for (int y = 0; y < NK; ++y) {
                const float p = BF ? ex2(x[r][y] - ref[r]) : expf(x[r][y] - ref[r]);
                sum[r] += p;
                if constexpr (BF) {
                    const __nv_bfloat16 hi = __float2bfloat16_rn(p);
                    sh.ph[row][lane + 32 * y] = hi;
                    sh.pl[row][lane + 32 * y] = __float2bfloat16_rn(p - __bfloat162float(hi));
                } else {
                    sh.s[row][lane + 32 * y] = p;
                }
            }
            if constexpr (BF) { if (lane == 0) sh.corr[row] = corr[r]; }
            else {
#pragma unroll
                for (int y = 0; y < DPL; ++y) o[r][y] *= corr[r];
            }
        }
#pragma unroll
        for (int z = 16; z > 0; z >>= 1)
#pragma unroll
            for (int r = 0; r < NR; ++r) sum[r] += __shfl_xor_sync(0xffffffffu, sum[r], z);
#pragma unroll
        for (int r = 0; r < NR; ++r) lsum[r] = lsum[r] * corr[r] + sum[r];
    }
    // first: the CTA's first item, whose first tile may have been asked for
    __device__ __forceinline__ void attention(const SpLayer &l, int items, const Range &first, bool asked) {
        constexpr int NK = TKS / 32, DPL = HD / 32;             // keys of a row, and fp32 dims of an output row, per lane
        Range it = first;
        int tab = 0;
#pragma unroll 1
        for (int id = blockIdx.x; id < items; ) {
            const int tiles = (it.k1 - it.k0 + TKS - 1) / TKS, ord = l.ord[it.s];
            const int *q_at = sh.q_at[tab];
#pragma unroll
            for (int x = 0; x < SP_QG * HD / 4 / SP_THREADS; ++x) {
                const int e = tid + x * SP_THREADS, r = e / (HD / 4), piece = e - r * (HD / 4);
                cp16(smem_u32(&sh.q[r][piece * 4]), a.q + (size_t)q_at[r] * (HD / 4) + piece, true);
            }
            if (tiles > 0 && !asked) load_kv(it, ord, it.k0, kvbuf);
            asked = false;
            float m[2] = {-INFINITY, -INFINITY}, lsum[2] = {0.f, 0.f};       // of rows warp and warp + 8, in every lane
            float o[2][4];                                       // bf16: dims 16 warp + 8 n + 2c, + 1 of rows g and g + 8; fp32: dims DPL lane ... of rows warp, warp + 8
#pragma unroll
            for (int r = 0; r < 2; ++r)
#pragma unroll
                for (int x = 0; x < 4; ++x) o[r][x] = 0.f;
#pragma unroll 1
            for (int t = 0; t < tiles; ++t) {
                cp_wait_all();
                __syncthreads();                                // the tile has landed; the other buffer has been read
                if (t + 1 < tiles) load_kv(it, ord, it.k0 + (t + 1) * TKS, kvbuf + ((t + 1) & 1) * KV_BYTES);
                const uint8_t *kb = kvbuf + (t & 1) * KV_BYTES, *vb = kb + TKS * KVROW;
                const int j0 = it.k0 + t * TKS;
                auto seen = [&](int row, int j) { return j < it.k1 && (j < it.n || ((sh.q_anc[tab][row] >> (j - it.n)) & 1ull)); };
                // scores: bf16 eight keys per warp; fp32 a key per lane, blocks of 32 keys and groups of rows to the warps
                if constexpr (BF) {
                    float sc[2][4] = {};                         // products with the hi and with the lo parts
#pragma unroll
                    for (int x = 0; x < HD / 32; ++x) {
                        const uint4 b = ldsu4(kb + (warp * 8 + g) * KVROW + (x * 32 + c * 8) * 2);
                        const uint4 ha = ldsu4(&sh.q[g][x * 32 + c * 8]), la = ldsu4(&sh.q[g][x * 32 + c * 8 + 4]);
                        const uint4 hb = ldsu4(&sh.q[g + 8][x * 32 + c * 8]), lb = ldsu4(&sh.q[g + 8][x * 32 + c * 8 + 4]);
                        const uint32_t h0[4] = {ha.x, hb.x, ha.y, hb.y}, h1[4] = {ha.z, hb.z, ha.w, hb.w};
                        const uint32_t l0[4] = {la.x, lb.x, la.y, lb.y}, l1[4] = {la.z, lb.z, la.w, lb.w};
                        mma_bf16(sc[0], h0, b.x, b.y); mma_bf16(sc[1], l0, b.x, b.y);
                        mma_bf16(sc[0], h1, b.z, b.w); mma_bf16(sc[1], l1, b.z, b.w);
                    }
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        const int row = g + 8 * (e >> 1), key = warp * 8 + 2 * c + (e & 1);
                        sh.s[row][key] = seen(row, j0 + key) ? sc[0][e] + sc[1][e] : -INFINITY;
                    }
                } else {
                    const int key = (warp % NK) * 32 + lane;
                    const uint8_t *kr = kb + key * KVROW;
#pragma unroll 1
                    for (int row = warp / NK; row < it.rows; row += SP_WARPS / NK) {
                        float p4[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 8
                        for (int dd = 0; dd < HD; dd += 4) {
                            const float4 kv = *reinterpret_cast<const float4 *>(kr + dd * 4), qv = lds4(&sh.q[row][dd]);
                            p4[0] = fmaf(qv.x, kv.x, p4[0]); p4[1] = fmaf(qv.y, kv.y, p4[1]);
                            p4[2] = fmaf(qv.z, kv.z, p4[2]); p4[3] = fmaf(qv.w, kv.w, p4[3]);
                        }
                        sh.s[row][key] = seen(row, j0 + key) ? (p4[0] + p4[1]) + (p4[2] + p4[3]) : -INFINITY;
                    }
                }
                __syncthreads();
                if (warp + SP_WARPS < it.rows) softmax<2>(m, lsum, o);
                else if (warp < it.rows) softmax<1>(m, lsum, o);
                if constexpr (BF) {
                    __syncthreads();
                    // 16 dims per warp
                    const float c0 = g < it.rows ? sh.corr[g] : 1.f, c1 = g + 8 < it.rows ? sh.corr[g + 8] : 1.f;
#pragma unroll
                    for (int n = 0; n < 2; ++n) { o[n][0] *= c0; o[n][1] *= c0; o[n][2] *= c1; o[n][3] *= c1; }
#pragma unroll
                    for (int ks = 0; ks < TKS / 16; ++ks) {
                        uint32_t ph[4], pl[4], b[4];
                        const int pr = lane & 15, pc = ks * 16 + (lane >> 4) * 8;
                        ldsm_x4(smem_u32(&sh.ph[pr][pc]), ph);
                        ldsm_x4(smem_u32(&sh.pl[pr][pc]), pl);
                        ldsm_x4_t(smem_u32(vb + (ks * 16 + (lane & 15)) * KVROW + (warp * 16 + (lane >> 4) * 8) * 2), b);
                        mma_bf16(o[0], pl, b[0], b[1]); mma_bf16(o[1], pl, b[2], b[3]);
                        mma_bf16(o[0], ph, b[0], b[1]); mma_bf16(o[1], ph, b[2], b[3]);
                    }
                } else {
                    __syncwarp();
#pragma unroll
                    for (int r = 0; r < 2; ++r) {
                        const int row = warp + SP_WARPS * r;
                        if (row >= it.rows) continue;
#pragma unroll 4
                        for (int j = 0; j < TKS; j += 4) {
                            const float4 p = lds4(&sh.s[row][j]);
                            const float pj[4] = {p.x, p.y, p.z, p.w};
#pragma unroll
                            for (int e = 0; e < 4; ++e) {
                                const float *vr = reinterpret_cast<const float *>(vb + (j + e) * KVROW) + lane * DPL;
                                if constexpr (DPL == 4) {
                                    const float4 v = lds4(vr);
                                    o[r][0] = fmaf(pj[e], v.x, o[r][0]); o[r][1] = fmaf(pj[e], v.y, o[r][1]);
                                    o[r][2] = fmaf(pj[e], v.z, o[r][2]); o[r][3] = fmaf(pj[e], v.w, o[r][3]);
                                } else {
                                    const float2 v = *reinterpret_cast<const float2 *>(vr);
                                    o[r][0] = fmaf(pj[e], v.x, o[r][0]); o[r][1] = fmaf(pj[e], v.y, o[r][1]);
                                }
                            }
                        }
                    }
                }
            }
            if (tiles == 0) { cp_wait_all(); __syncthreads(); }
            // ---- partial rows: [token row, head][range] ----
            if constexpr (BF) {
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    if (g + 8 * e >= it.rows) continue;
                    float *dst = a.part + ((size_t)q_at[g + 8 * e] * a.nsplit + it.split) * HD + warp * 16 + 2 * c;
                    *reinterpret_cast<float2 *>(dst) = make_float2(o[0][2 * e], o[0][2 * e + 1]);
                    *reinterpret_cast<float2 *>(dst + 8) = make_float2(o[1][2 * e], o[1][2 * e + 1]);
                }
            }
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                const int row = warp + SP_WARPS * r;
                if (row >= it.rows) continue;
                const size_t pr = (size_t)q_at[row] * a.nsplit + it.split;
                if constexpr (!BF) {
                    float *dst = a.part + pr * HD + lane * DPL;
                    if constexpr (DPL == 4) *reinterpret_cast<float4 *>(dst) = make_float4(o[r][0], o[r][1], o[r][2], o[r][3]);
                    else *reinterpret_cast<float2 *>(dst) = make_float2(o[r][0], o[r][1]);
                }
                if (lane == 0) a.part_ml[pr] = make_float2(m[r], lsum[r]);
            }
            // ---- the last of the pair's CTAs to get here merges the ranges, in their order ----
            __syncthreads();
            if (tid == 0) {
                unsigned old;
                asm volatile("atom.acq_rel.gpu.global.inc.u32 %0, [%1], %2;" : "=r"(old) : "l"(sh.counters + 2 + it.pair), "r"(a.nsplit - 1) : "memory");
                sh.last = old == (unsigned)a.nsplit - 1;
            }
            __syncthreads();
            if (sh.last) {
                // a row per warp, four dims per lane (HD 64: one half of the lanes repeats the other), all ranges in flight
                const int col = lane % (HD / 4);
#pragma unroll 1
                for (int row = warp; row < it.rows; row += SP_WARPS) {
                    const size_t z = (size_t)q_at[row] * a.nsplit;
                    const float2 w = __ldcg(a.part_ml + z + min(lane, a.nsplit - 1));
                    float4 p[SP_SPLITS];
#pragma unroll
                    for (int y = 0; y < SP_SPLITS; ++y) if (y < a.nsplit) p[y] = __ldcg(reinterpret_cast<const float4 *>(a.part + (z + y) * HD + col * 4));
                    const float mx = warp_max(w.x);              // (every row sees itself: finite)
                    const float f = BF ? ex2(w.x - mx) : expf(w.x - mx);
                    float sum = 0.f;
                    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                    for (int y = 0; y < SP_SPLITS; ++y) if (y < a.nsplit) {
                        const float fy = __shfl_sync(0xffffffffu, f, y), ly = __shfl_sync(0xffffffffu, w.y, y);
                        sum = fmaf(ly, fy, sum);
                        v.x = fmaf(p[y].x, fy, v.x); v.y = fmaf(p[y].y, fy, v.y); v.z = fmaf(p[y].z, fy, v.z); v.w = fmaf(p[y].w, fy, v.w);
                    }
                    if (lane < HD / 4)
                        put_four((T *)nullptr, reinterpret_cast<uint8_t *>(a.attn + (size_t)q_at[row] * (HD / 4) + (col >> 1) * 2), col & 1,
                                 make_float4(v.x / sum, v.y / sum, v.z / sum, v.w / sum));
                }
            }
            id += gridDim.x;
            if (id < items) {
                __syncthreads();                                // this item's tables and tiles have been read
                tab = 1;
                att_item(id, tab, it);
                __syncthreads();
            }
        }
    }

    // ---- what the pass needs of the draft: every CTA for itself, CTA 0 also for the kernels behind this one ----
    __device__ __forceinline__ void prepare() {
        if (tid == SP_THREADS - 1) { sh.n_bar = sh.abort_flag = 0; sh.counters = a.counters + SMALL_PASS_LINE + (__ldcg(a.counters) & 1) * a.set_words; }
        if (a.row_tok) {                                        // a replay pass: its preparation has run
            for (int r = tid; r < a.R; r += SP_THREADS) {
                const int b = r / a.M, i = r - b * a.M, n = a.len_eff[b], at = n + i;
                sh.anc[r] = a.tree[b].anc[i]; sh.pos[r] = n + a.tree[b].depth[i]; sh.tok[r] = a.row_tok[r];
                sh.slot[r] = a.kv_keep && at < a.kv_keep[b] ? -1 : at; sh.n_ctx[r] = n; sh.seq[r] = b;
            }
            __syncthreads();
            return;
        }
        for (int b = warp; b < a.B; b += SP_WARPS) {
            TreeInfo &t = sh.tree[warp];
            const int l = a.len[b], n = min(max(l, 0), a.max_ctx - a.M);
            build_tree(&t, a.parent + (a.per_seq ? (size_t)b * a.N : 0), a.N, a.stats, sh.par[warp]);
            if (n != l) a.stats->device_status = VIASD_ECAPACITY;
            for (int i = lane; i < a.M; i += 32) {
                const int r = b * a.M + i;
                int tok = i == 0 ? a.pending[b] : a.draft_tok[b * a.N + i - 1];
                if (tok < 0 || tok >= a.V) { a.stats->device_status = VIASD_EDEVICE; tok = 0; }
                sh.anc[r] = t.anc[i]; sh.pos[r] = n + t.depth[i]; sh.tok[r] = tok;
                sh.slot[r] = n + i; sh.n_ctx[r] = n; sh.seq[r] = b;
            }
            if (blockIdx.x == 0) {
                int *dst = reinterpret_cast<int *>(a.tree + b);
                const int *src = reinterpret_cast<const int *>(&t);
                // (rows past the block's hold nothing that is read)
                for (int i = lane; i < (int)(sizeof(TreeInfo) / sizeof(int)); i += 32) dst[i] = src[i];
                if (lane == 0) a.len_eff[b] = n;
            }
            __syncwarp();
        }
        if (blockIdx.x == 0 && tid == 0 && a.full_pass) a.stats->full_ran = 1;       // the full verifier's cache receives this block's rows
        __syncthreads();
    }

    __device__ __forceinline__ void run() {
        for (int i = tid; i < a.n_layers * (int)(sizeof(SpLayer) / 4); i += SP_THREADS)
            reinterpret_cast<int *>(sh.layer)[i] = reinterpret_cast<const int *>(a.layer)[i];
        __syncthreads();
        prefetch<ST_QKV>(sh.layer[0]);
        prepare();
        Range first;
        const bool any = (int)blockIdx.x < a.streams * a.att_items;          // (one stream's items come first: the same in every layer)
        if (any) att_item(blockIdx.x, 0, first);
#pragma unroll 1
        for (int li = 0; li < a.n_layers; ++li) {
            const SpLayer &l = sh.layer[li];
            const int streams = a.streams == 2 && l.ord[1] >= 0 ? 2 : 1, rows = streams * a.R, items = streams * a.att_items;
            project<ST_QKV>(li, rows);
            bool asked = false;
            barrier([&] {
                asked = any && (int)blockIdx.x < items && first.k0 < first.k1 && first.k0 + TKS <= first.n;   // a first tile wholly inside the committed context
                if (asked) load_kv(first, l.ord[first.s], first.k0, kvbuf);
                prefetch<ST_O>(l);
            });
            attention(l, items, first, asked);
            barrier([] {});
            project<ST_O>(li, rows);
            barrier([&] { prefetch<ST_GU>(l); });
            project<ST_GU>(li, rows);
            barrier([&] { prefetch<ST_DOWN>(l); });
            project<ST_DOWN>(li, rows);
            barrier([&] { if (li + 1 < a.n_layers) prefetch<ST_QKV>(sh.layer[li + 1]); else prefetch<ST_HEAD>(l); });
        }
        hand_over();
        project<ST_HEAD>(a.n_layers, a.streams * a.R);
    }
};

template <typename T, int HD, int MT>
__global__ void __launch_bounds__(SP_THREADS, 1) small_pass_kernel(const __grid_constant__ SpArgs a) {
    extern __shared__ __align__(128) uint8_t sp_smem[];
    RUN_FLAG_EXIT(a.run_flag);
    PDL_TRIGGER();
    using P = Pass<T, HD, MT>;
    P pass(a, sp_smem);
    pass.run();
}

constexpr size_t SP_SMEM = 227 * 1024;

// Shared memory of a pass; false where it does not fit.  Nothing here depends on how many of the verifiers are in the launch.
template <typename T, int HD, int MT>
bool plan(const viasd_config &c, int rows, int grid, SpArgs &a, size_t &smem) {
    using P = Pass<T, HD, MT>;
    const int k[5] = {c.d_model, c.n_heads * HD, c.d_model, c.d_ff, c.d_model};
    const int units[5] = {(c.n_heads + 2 * c.n_kv_heads) * (HD / 16), c.d_model / 8, c.d_ff / 8, c.d_model / 8, (c.vocab + 15) / 16};
    size_t w = 0;
    int per = 0;
    for (int s = ST_QKV; s <= ST_HEAD; ++s) {
        const int p = (k[s] + KG * SP_WARPS - 1) / (KG * SP_WARPS), mine = (units[s] + grid - 1) / grid;
        const size_t bytes = (size_t)mine * p * stage_tiles(s) * P::WSTEP;
        w = bytes > w ? bytes : w;
        per = p > per ? p : per;
    }
    a.red_bytes = rows * TN * 8 * SP_WARPS * (int)sizeof(float);
    const size_t fixed = (sizeof(typename P::Shared) + 127) / 128 * 128 + a.red_bytes + w, row = (size_t)XGROUP * SP_WARPS;    // row: one group of k, all warps
    if (fixed + 2 * P::KV_BYTES > SP_SMEM) return false;
    const size_t room = SP_SMEM - fixed;
    a.x_groups = per; a.x_rows = rows;
    if (P::BF) {
        while (a.x_groups > 1 && (size_t)a.x_groups * rows * row > room) --a.x_groups;
    } else {
        a.x_rows = rows < 16 ? rows : 16;
        if ((size_t)per * a.x_rows * row > room && a.x_rows > 8) a.x_rows = 8;
    }
    const size_t x = (size_t)a.x_groups * a.x_rows * row;
    if (x > room) return false;
    a.w_bytes = (int)w;
    a.x_bytes = a.x_groups * a.x_rows * XGROUP;
    smem = fixed + (x > 2 * (size_t)P::KV_BYTES ? x : 2 * (size_t)P::KV_BYTES);
    return true;
}

template <typename T, int HD, int MT>
int launch(SpArgs &a, const viasd_config &c, int rows, int grid, cudaStream_t st) {
    size_t smem = 0;
    if (!plan<T, HD, MT>(c, rows, grid, a, smem)) return VIASD_EINVAL;
    static std::atomic<bool> attr_done[64];
    if (int rc = once_on_device(attr_done, [&]() -> int {
        CUDA_TRY(cudaFuncSetAttribute(small_pass_kernel<T, HD, MT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SP_SMEM));
        return VIASD_OK;
    })) return rc;
    cudaLaunchConfig_t cfg{};
    cudaLaunchAttribute attr[1];
    cfg.gridDim = dim3(grid); cfg.blockDim = dim3(SP_THREADS); cfg.dynamicSmemBytes = smem; cfg.stream = st;
    attr[0].id = cudaLaunchAttributeCooperative;                // the CTAs wait for one another: all of them are resident, or none is
    attr[0].val.cooperative = 1;
    cfg.attrs = attr; cfg.numAttrs = 1;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, small_pass_kernel<T, HD, MT>, a);
    if (e == cudaErrorCooperativeLaunchTooLarge) {               // (a context with a share of the SMs only)
        (void)cudaGetLastError();
        return SMALL_PASS_NO_ROOM;
    }
    CUDA_TRY(e);
    LAUNCH_CHECK();
    return VIASD_OK;
}

// F(type, head dim, row tiles) for a pass of `rows` rows
#define SP_DISPATCH(m, rows, F)                                                                             \
    ((m)->cfg.dtype == 0 ? ((m)->cfg.head_dim == 64 ? F(float, 64, 1) : F(float, 128, 1))                   \
                         : ((rows) <= 16 ? F(__nv_bfloat16, 128, 1) : (rows) <= 32 ? F(__nv_bfloat16, 128, 2) : F(__nv_bfloat16, 128, 4)))

}  // namespace

// Token rows of a launch at most: 64, or fewer where the shared memory of 64 does not fit; 0: not even M rows do.
static int launch_rows(const viasd_model *m, int M) {
    for (int rows = SP_ROWS; rows >= M && rows >= 8; rows -= 8) {
        SpArgs a;
        size_t smem;
#define SP_PLAN(T, HD, MT) plan<T, HD, MT>(m->cfg, rows, m->sm_count, a, smem)
        if (SP_DISPATCH(m, rows, SP_PLAN)) return rows;
#undef SP_PLAN
    }
    return 0;
}

// How a call's sequences share launches (M: rows of one).  They form groups of n, the last one maybe smaller; a launch has a group of
// both verifiers' rows, or as many groups of one verifier's as fit.  The cuts of a sequence's key ranges depend on its group's
// size alone, so that they are the same whatever is launched; a last group that is cut otherwise has launches of its own.
struct Grouping {
    int batch, n, per_one;          // groups that a launch of one verifier's rows takes
    bool fits_both;
    int pairs;                      // attention pairs of a sequence
    int part_seqs;                  // sequences of one verifier whose partial rows any launch has, at most
    int sms, tiles; size_t part_room;
    // as many ranges as keep the CTAs busy with both verifiers, one per 64 keys of the cache's capacity at most, within the partial buffer;
    // of a short context (they are cut on the device, at whole 32s) some are half a tile, or empty and merged as nothing
    int ranges(int b0) const {
        int ns = sms / (2 * (batch - b0 < n ? batch - b0 : n) * pairs);
        if (ns > tiles) ns = tiles;
        if (ns > SP_SPLITS) ns = SP_SPLITS;
        if ((size_t)ns > part_room) ns = (int)part_room;
        return ns < 1 ? 1 : ns;
    }
    int take(int b0, bool both) const {                             // sequences of the launch that begins with b0
        const int most = both ? n : per_one * n, left = batch - b0;
        if (left > most) return most;
        const int full = left / n * n;
        return full && full < left && ranges(b0 + full) != ranges(b0) ? full : left;
    }
    int launches(bool both) const {
        int count = 0;
        for (int b0 = 0; b0 < batch; b0 += take(b0, both)) ++count;
        return count;
    }
};
static Grouping grouping(const viasd_model *m, int batch, int M, int most) {
    const viasd_config &c = m->cfg;
    Grouping g;
    g.batch = batch;
    g.fits_both = 2 * M <= most;
    const int rows = g.fits_both ? 2 * M : M, n = most / rows < batch ? most / rows : batch, groups = (batch + n - 1) / n;
    // Groups of equal size, or all but the last as large as fits: whichever has fewer eights of rows (6 sequences of 7 rows as 4 + 2, not 3 + 3:
    // 175 us, else 181), equal ones where that is the same (6 of 6 rows as 3 + 3, not 5 + 1: 224 us, else 264)
    auto eights = [&](int size) {
        const int full = batch / size, last = batch - full * size;
        return full * ((size * rows + 7) / 8) + (last * rows + 7) / 8;
    };
    const int even = (batch + groups - 1) / groups;
    g.n = eights(even) <= eights(n) ? even : n;
    g.per_one = most / (g.n * M);
    g.pairs = c.n_kv_heads * ((c.n_heads / c.n_kv_heads * M + SP_QG - 1) / SP_QG);
    g.part_seqs = g.per_one * g.n < batch ? g.per_one * g.n : batch;
    if (2 * g.n > g.part_seqs) g.part_seqs = 2 * g.n;
    g.sms = m->sm_count; g.tiles = (c.max_ctx + 63) / 64;
    g.part_room = m->ws.part_bytes / ((size_t)g.part_seqs * M * c.n_heads * (c.head_dim + 2) * sizeof(float));
    return g;
}

// Which passes go this way.  us, this way / launch by launch (three layers, one of them routed; one step):
//   fp32, d 256: 5 rows 90 / 177 (context 100), 132 / 335 (4000); 18 rows 136 / 267, 198 / 500; 32 rows 156 / 351, 334 / 635;
//         d 768, 9 rows 257 / 503
//   bf16, d 512, 4 kv heads: 5 rows 84 / 114 (100), 118 / 131 (4000); 9 rows 96 / 124, 132 / 141; 18 rows 119 / 135, 165 / 152;
//         28 rows 137 / 143 (100), 148 / 152 (1000), 227 / 177 (4000); 1 kv head: 27 rows 134 / 146, 142 / 157, 171 / 174;
//         four layers, context 300: d 768, 18 rows 195 / 200, 27 rows 231 / 213; d 1024, 9 rows 189 / 207
// so fp32 always where one launch holds a verifier's rows (527 drawn shapes: none slower); bf16 while the rows a CTA reads (rows x the
// layer's columns of input, 2944 at d 512) and the tiles of keys per CTA are few: then tcgen05 GEMMs and attention overtake it.
// fp32 in several launches: each one more costs a layer's barriers, 17 us, which rows x columns have to win back, and attention by
// the tile of keys.  Of 1109 drawn calls (d 64 - 1024, 1 - 64 rows per sequence, batch 2 - 64, context 70 - 4000, steps and
// prompt chunks) 81 are slower in launches, 0.58 times as fast at worst; of the 985 on this side of the line 17 are (0.77), of
// those on the other 22 would have gained more than a fifth.  Drawn again with groups of equal size: 5 of 516 (0.83), none.
// d 192, d_ff 2816, 24 x 6 rows, a sequence per launch: 2310 / 1498; d 256, 16 x 27 rows 2738 / 4343 (context 300), 3365 / 4828 (2000);
// d 768, 16 x 9 rows 1978 / 2305.  Key tiles are counted by the cache's capacity, as the lengths are on the device.
// A launch has all weights of a stage in shared memory, the output head's too (plan): at 148 SMs fp32 of d 256 up to a vocabulary of
// 16576, bf16 of d 512 up to 14208, of d 768 up to 9472; beyond that a model goes launch by launch.
// bf16 steps of 33 - 64 rows of both verifiers (the kernel's instance for 64, whose padding and smaller stages of input tell) go this way
// where a step's estimate is the smaller one: per layer 15.2 us and what a CTA multiplies and its tiles of keys take, against
// 26.4 us and weights, rows and keys, fitted to 2688 drawn steps of 2 - 32 rows per verifier (median error 3 %, 7 % in a tenth).  Without it 242
// of them are slower in one launch (0.74 at worst; d 640, two layers, 21 rows 124 / 116 us), with it 77 (0.87; drawn again: 90 of 2728, 0.86); 35 of those it
// sends launch by launch would have gained 5 % or more.  A single pass follows the step, as both compute the same bits.
static bool one_launch_gains(const viasd_model *m, const Grouping &g, int rows) {
    const viasd_config &c = m->cfg;
    auto up = [](long long a, long long b) { return (double)((a + b - 1) / b); };
    auto units = [&](long long n) { return up(n, m->sm_count); };
    auto chunks = [&](int k) { return up(k, KG * SP_WARPS); };
    const int d = c.d_model, ff = c.d_ff, qd = c.n_heads * c.head_dim, kvd = c.n_kv_heads * c.head_dim, routed = m->n_routed, other = c.n_layers - routed;
    const double products = (units((qd + 2 * kvd) / 16) + units(ff / 8)) * chunks(d) + units(d / 8) * (chunks(qd) + chunks(ff));
    const long long pairs = (long long)g.batch * g.pairs, ns = g.ranges(0);
    auto layer = [&](int streams) { return units(streams * pairs * ns) * (15.2 + 1.6 * up(c.max_ctx, 64 * ns)) + 0.029 * streams * rows * products; };
    const double one = 32 + routed * layer(2) + other * layer(1) + 0.029 * 2 * rows * chunks(d) * units((c.vocab + 15) / 16) +
                       (d > 512 ? routed * 3.1 * (d - 512) / 128 : 0);
    const double params = (double)d * (2 * qd + 2 * kvd) + 3. * d * ff;
    const double many = 26.4 * (c.n_layers + 1) + 0.21 * rows * (c.n_layers + routed) + 1.29e-6 * (c.n_layers * params + (double)c.vocab * d) +
                        1e-3 * c.max_ctx * (1.52 * c.n_layers + 0.051 * pairs * (c.n_layers + routed));
    return one <= many;
}

bool small_pass_takes(const viasd_model *m, const viasd_cache *cache, int batch, int M, bool replay) {
    const viasd_config &c = m->cfg;
    const ModelOptions &o = m->opt;
    if (!o.one_launch || (c.dtype == 1 && !m->fused)) return false;
    // the options of kernels that such a pass does not have
    if (o.attn_kernel || o.attn_splits || o.attn_lo != 2 || o.tk_grid || o.tk_flat >= 0 || o.ring_kb || o.epi_groups) return false;
    if (c.n_layers > SMALL_PASS_MAX_LAYERS) return false;
    const int most = launch_rows(m, M);
    if (most == 0) return false;
    const Grouping g = grouping(m, batch, M, most);
    const long long rows = (long long)batch * M, columns = 2LL * c.d_model + c.n_heads * c.head_dim + c.d_ff;
    if (c.dtype == 0) {
        const long long launches = (batch + most / M - 1) / (most / M), seqs = g.take(0, false), ns = g.ranges(0), range = ns * (c.head_dim == 64 ? 64 : 32);
        const long long tiles = (seqs * g.pairs * ns + m->sm_count - 1) / m->sm_count * ((c.max_ctx + range - 1) / range);   // of a CTA
        if (launches > 1 && rows * columns < 59000 * (launches - 1) + 800 * launches * tiles * (c.head_dim / 64)) return false;
    } else {
        if (2 * rows > most) return false;
        const long long tiles = 2LL * batch * g.pairs * ((c.max_ctx + 63) / 64);
        if (rows * columns * m->sm_count + 3 * 2944 * tiles > 36LL * 2944 * m->sm_count) return false;
        if (!replay && rows > 16 && !one_launch_gains(m, g, (int)rows)) return false;
        // (caches that are not aligned are refused by the path with tensor maps over them)
        if (((uintptr_t)cache->k_full | (uintptr_t)cache->v_full | (uintptr_t)cache->k_slim | (uintptr_t)cache->v_slim) & 15) return false;
    }
    return true;
}

// Sequences b0 .. b0 + n - 1 of a pass.  mode 0: full verifier, 1: slim verifier, 2: both; replay: rows in front of every
// sequence's own (prepared before this call)
static int launch_group(viasd_model *m, const viasd_cache *cache, const viasd_draft *d, const Grouping &g, int b0, int n, int mode, int replay,
                        float *logits_full, float *logits_slim, cudaStream_t st) {
    const viasd_config &c = m->cfg;
    SpArgs a;
    memset(&a, 0, sizeof(a));
    a.B = n; a.N = d->n_nodes; a.M = d->n_nodes + 1 + replay; a.R = a.B * a.M; a.streams = mode == 2 ? 2 : 1;
    a.d = c.d_model; a.ff = c.d_ff; a.qd = c.n_heads * c.head_dim; a.V = c.vocab; a.H = c.n_heads; a.Hkv = c.n_kv_heads;
    a.max_batch = c.max_batch; a.max_ctx = c.max_ctx; a.skip = replay;
    a.eps = c.rms_eps; a.inv_d = 1.0f / (float)c.d_model;
    a.att_scale = (c.dtype == 1 ? 1.4426950408889634f : 1.0f) / sqrtf((float)c.head_dim);
    a.embed = m->embed; a.head = m->lm_head; a.final_norm = m->final_norm; a.cosv = m->ws.rope_cos; a.sinv = m->ws.rope_sin;
    const size_t kv0 = (size_t)b0 * c.n_kv_heads * c.max_ctx * c.head_dim * (c.dtype == 0 ? 4 : 2);
    auto from = [&](void *cache_of_first) { return (void *)((char *)cache_of_first + kv0); };
    const bool slim_first = mode == 1;
    a.kc[0] = from(slim_first ? cache->k_slim : cache->k_full); a.vc[0] = from(slim_first ? cache->v_slim : cache->v_full);
    a.kc[1] = from(cache->k_slim); a.vc[1] = from(cache->v_slim);
    const size_t out0 = (size_t)b0 * (a.M - replay) * c.vocab;
    a.logits[0] = (slim_first ? logits_slim : logits_full) + out0; a.logits[1] = mode == 2 ? logits_slim + out0 : nullptr;
    a.kv_vec = (((uintptr_t)cache->k_full | (uintptr_t)cache->v_full | (uintptr_t)cache->k_slim | (uintptr_t)cache->v_slim) & 15) == 0;
    a.h = m->ws.h; a.xn = (uint4 *)m->ws.a; a.q = (uint4 *)m->ws.q; a.attn = (uint4 *)m->ws.attn; a.act = (uint4 *)m->ws.act;
    a.ssq = (float *)m->ws.a_head;                              // (what a pass of many launches packs the head's input into)
    a.len = cache->len + b0; a.pending = cache->pending + b0; a.draft_tok = d->draft_tok + (size_t)b0 * a.N;
    a.per_seq = d->per_sequence; a.parent = d->parent + (d->per_sequence ? (size_t)b0 * a.N : 0);
    a.row_tok = replay ? m->ws.row_tok + (size_t)b0 * a.M : nullptr; a.kv_keep = replay ? cache->len_full + b0 : nullptr;
    a.full_pass = mode != 1;
    a.tree = m->ws.tree + b0; a.len_eff = m->ws.len_eff + b0; a.stats = m->ws.stats; a.run_flag = m->run_flag;
    a.counters = m->ws.pass_counters; a.set_words = small_pass_set(c);
    a.first[0] = 0; a.first[1] = -1;
    for (int l = 0; l < c.n_layers; ++l) {
        int so = -1;
        for (int o = 0; o < m->n_routed; ++o) if (m->routed[o] == l) so = o;
        if (mode == 1 && so < 0) continue;
        SpLayer &s = a.layer[a.n_layers];
        s.wq = m->wq[l]; s.wk = m->wk[l]; s.wv = m->wv[l]; s.wo = m->wo[l]; s.wg = m->wg[l]; s.wu = m->wu[l]; s.wd = m->wd[l];
        s.n1 = m->norm1[l]; s.n2 = m->norm2[l];
        s.ord[0] = mode == 1 ? so : l;
        s.ord[1] = mode == 2 ? so : -1;
        if (s.ord[1] >= 0 && a.first[1] < 0) a.first[1] = a.n_layers;
        ++a.n_layers;
    }
    for (int i = 0; i < a.n_layers; ++i) {
        SpLayer &s = a.layer[i];
        s.next[0] = i + 1 < a.n_layers ? a.layer[i + 1].n1 : m->final_norm;
        s.next[1] = m->final_norm;
        for (int j = i + 1; j < a.n_layers; ++j) if (a.layer[j].ord[1] >= 0) { s.next[1] = a.layer[j].n1; break; }
    }
    a.nsplit = g.ranges(b0);
    a.att_items = a.B * g.pairs * a.nsplit;
    a.part = m->ws.part;
    a.part_ml = reinterpret_cast<float2 *>(m->ws.part + (size_t)g.part_seqs * a.M * c.n_heads * a.nsplit * c.head_dim);
    const int rows = a.streams * a.R;
#define SP_LAUNCH(T, HD, MT) launch<T, HD, MT>(a, c, rows, m->sm_count, st)
    return SP_DISPATCH(m, rows, SP_LAUNCH);
#undef SP_LAUNCH
}

// A pass that small_pass_takes; SMALL_PASS_NO_ROOM if the device does not hold its CTAs at once (nothing has been launched then, and
// it goes launch by launch).  More sequences than a launch holds (fp32) go in groups, as many of them in each as fit: with both
// verifiers' rows, or with one's where that makes fewer launches times layers.  (Groups of as many as would fit with both, whichever
// were in the launch, left half of a single verifier's rows empty: 16 prompts' chunks of 17 rows were 32 launches, not 12.)
int launch_small_pass(viasd_model *m, const viasd_cache *cache, const viasd_draft *d, int mode, int replay, float *logits_full,
                      float *logits_slim, cudaStream_t st) {
    const int M = d->n_nodes + 1 + replay, most = launch_rows(m, M);
    if (most < M) return VIASD_EINVAL;
    const Grouping g = grouping(m, d->batch, M, most);
    const bool together = mode == 2 && g.fits_both && g.launches(true) * m->cfg.n_layers <= g.launches(false) * (m->cfg.n_layers + m->n_routed);
    for (int b0 = 0, nb; b0 < d->batch; b0 += nb) {
        nb = g.take(b0, together);
        auto group = [&](int which) { return launch_group(m, cache, d, g, b0, nb, which, replay, logits_full, logits_slim, st); };
        int rc;
        if (together) {
            if ((rc = group(2))) return rc;
            continue;
        }
        if (mode != 0 && (rc = group(1))) return rc;
        if (mode != 1 && (rc = group(0))) return rc;
    }
    return VIASD_OK;
}
