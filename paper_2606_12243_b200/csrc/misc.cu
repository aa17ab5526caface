// Small memory-bound kernels of the decoder block and the cache bookkeeping:
// rotary table, embedding gather with the per-pass preparation (tree layout, row tokens, clamped lengths),
// RMSNorm, rotary embedding + KV append, KV commit.
#include "common.cuh"

// ---------------------------------------------------------------------------------------------
// rotary table: cos/sin(pos * theta^(-2p/hd)), computed in double once per handle
// ---------------------------------------------------------------------------------------------
__global__ void rope_table_kernel(float *cosv, float *sinv, int max_ctx, int half, double theta) {
    int idx = blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= max_ctx * half) return;
    int pos = idx / half, p = idx % half;
    double inv = pow(theta, -2.0 * (double)p / (double)(2 * half));
    double ang = (double)pos * inv;
    cosv[idx] = (float)cos(ang);
    sinv[idx] = (float)sin(ang);
}

int launch_rope_table(const viasd_model *m, cudaStream_t st) {
    int half = m->cfg.head_dim / 2;
    int n = m->cfg.max_ctx * half;
    rope_table_kernel<<<(n + 255) / 256, 256, 0, st>>>(m->ws.rope_cos, m->ws.rope_sin, m->cfg.max_ctx, half,
                                                       (double)m->cfg.rope_theta);
    LAUNCH_CHECK();
    return VIASD_OK;
}

// ---------------------------------------------------------------------------------------------
// per-pass preparation: part of the embedding kernels
// ---------------------------------------------------------------------------------------------
// The first CTAs of an embedding launch, one per sequence, lay out the sequence's tree and clamp its length; a row's CTA
// finds its own token.  (As a kernel of its own in front of the embedding, and again in front of the commit, this was 7 us
// each time, most of it the launch.)  What attention reads of it before its dependency wait - tree and length - is complete
// because the pass's first QKV launch is an ordinary one: nothing after it starts before the embedding has ended.
// Arrival counters of the GEMMs and of attention, zero between launches.  After a wait that expired they may not be: a pass
// that finds the status word saying so starts from clean ones (nothing before it in the stream is still running).
struct Counters { int *gemm, *attn; int n_gemm, n_attn; };
__device__ __forceinline__ int pass_status(const DeviceStats *stats) { return *reinterpret_cast<const volatile int *>(&stats->device_status); }
__device__ __forceinline__ void clear_counters_if_failed(const Counters &c, int status, int thread, int threads) {
    if (status != VIASD_EDEVICE) return;
    for (int i = thread; i < c.n_gemm; i += threads) c.gemm[i] = 0;
    for (int i = thread; i < c.n_attn; i += threads) c.attn[i] = 0;
}
static Counters counters_of(const viasd_model *m) {
    return Counters{m->ws.gemm_counters, m->ws.attn_counters, (int)m->ws.n_counters,
                    (int)attn_counter_count(m->cfg.max_batch, m->cfg.n_heads, m->cfg.n_kv_heads)};
}

struct PrepArgs {
    TreeInfo *tree; int *len_eff; DeviceStats *stats;
    const int *len, *pending, *draft_tok, *parent;       // parent: [N] shared by the batch, or [B, N] when per_seq
    const int *row_tok;                                  // not null: a replay pass, whose preparation has run (no sequence CTAs)
    int per_seq, B, N, max_ctx, vocab, full_pass;
    Counters counters;
};
__device__ __forceinline__ int prep_ctas(const PrepArgs &p) { return p.row_tok ? 0 : p.B; }
__device__ __forceinline__ int clamped_len(const int *len, int b, int max_ctx, int M, DeviceStats *stats) {
    const int l = len[b], c = min(max(l, 0), max_ctx - M);
    if (c != l) stats->device_status = VIASD_ECAPACITY;
    return c;
}
__device__ __forceinline__ void prep_sequence(const PrepArgs &p, int b, int *par_sh) {       // by the CTA's first warp
    const int status = b == 0 ? pass_status(p.stats) : 0;        // (asked for ahead of the tree, used behind it)
    build_tree(p.tree + b, p.parent + (p.per_seq ? (size_t)b * p.N : 0), p.N, p.stats, par_sh);
    if (threadIdx.x == 0) {
        if (b == 0 && p.full_pass) p.stats->full_ran = 1;      // the full verifier's cache receives this block's rows
        p.len_eff[b] = clamped_len(p.len, b, p.max_ctx, p.N + 1, p.stats);
    }
    clear_counters_if_failed(p.counters, status, threadIdx.x, 32);
}
__device__ __forceinline__ int prep_token(const PrepArgs &p, int r) {
    if (p.row_tok) return p.row_tok[r];
    const int M = p.N + 1, b = r / M, i = r - b * M;
    int t = i == 0 ? p.pending[b] : p.draft_tok[b * p.N + i - 1];
    if (t < 0 || t >= p.vocab) { p.stats->device_status = VIASD_EDEVICE; t = 0; }
    return t;
}
static PrepArgs prep_args(const viasd_model *m, const viasd_cache *c, const viasd_draft *d, bool full_pass, bool replay) {
    return PrepArgs{m->ws.tree, m->ws.len_eff, m->ws.stats, c->len, c->pending, d->draft_tok, d->parent,
                    replay ? m->ws.row_tok : nullptr, d->per_sequence, d->batch, d->n_nodes, m->cfg.max_ctx, m->cfg.vocab, full_pass ? 1 : 0,
                    counters_of(m)};
}

// Preparation of a replay pass (routed execution policy): the block of every sequence is extended, in front, by its
// last G committed tokens, so that the rows are
//     row 0 .. G-1 : tokens[len - G .. len - 1]  (a chain; row 0 plays the pending token's part)
//     row G        : the pending token
//     row G+1+n    : draft node n (its parent moved along)
// against a context of len - G rows.  The full verifier recomputes K/V of the G committed tokens (the same values
// where its cache had them, the missing ones where a skipped pass left a gap) on its way to the block's own rows.
__global__ void prep_replay_kernel(TreeInfo *tree, int *len_eff, int *row_tok, DeviceStats *stats, const int *len,
                                   const int *pending, const int *draft_tok, const int *parent, int per_seq,
                                   const int *tokens, int B, int N, int G, int max_ctx, int vocab, const Counters counters, const int *run_flag) {
    RUN_FLAG_EXIT(run_flag);
    clear_counters_if_failed(counters, pass_status(stats), threadIdx.x, blockDim.x);
    const int Mx = G + N + 1;
    if (threadIdx.x == 0) stats->full_ran = 1;
    for (int b = threadIdx.x; b < B; b += blockDim.x) {
        TreeInfo *t = tree + b;
        const int *par = parent + (per_seq ? (size_t)b * N : 0);
        t->anc[0] = 1ull;
        t->depth[0] = 0;
        for (int i = 0; i < Mx; ++i) { t->first_child[i] = -1; t->next_sibling[i] = -1; }
        for (int e = 0; e < G + N; ++e) {                       // extended node e is row e + 1
            int p = e < G ? e - 1 : par[e - G];
            const int i = e + 1;
            if (e >= G) {
                if (p == -2) { t->anc[i] = 1ull << i; t->depth[i] = 0; continue; }
                if (p < -1 || p >= e - G) { stats->device_status = VIASD_EDEVICE; p = -1; }
                p = p < 0 ? G - 1 : G + p;
            }
            const int pr = p + 1;
            t->anc[i] = t->anc[pr] | (1ull << i);
            t->depth[i] = t->depth[pr] + 1;
        }
        const int l = len[b] - G;
        const int c = min(max(l, 0), max_ctx - Mx);
        if (c != l) stats->device_status = VIASD_ECAPACITY;     // fewer than G committed tokens, or no room for the rows
        len_eff[b] = c;
    }
    for (int r = threadIdx.x; r < B * Mx; r += blockDim.x) {
        const int b = r / Mx, i = r % Mx;
        const int base = max(len[b] - G, 0);
        int t = i < G ? tokens[(size_t)b * max_ctx + min(base + i, max_ctx - 1)] : i == G ? pending[b] : draft_tok[b * N + i - G - 1];
        if (t < 0 || t >= vocab) { stats->device_status = VIASD_EDEVICE; t = 0; }
        row_tok[r] = t;
    }
}

int launch_prep_replay(const viasd_model *m, const viasd_cache *c, const viasd_draft *d, int G, cudaStream_t st) {
    prep_replay_kernel<<<1, 128, 0, st>>>(m->ws.tree, m->ws.len_eff, m->ws.row_tok, m->ws.stats, c->len, c->pending,
                                          d->draft_tok, d->parent, d->per_sequence, c->tokens, d->batch, d->n_nodes, G,
                                          m->cfg.max_ctx, m->cfg.vocab, counters_of(m), m->run_flag);
    LAUNCH_CHECK();
    return VIASD_OK;
}

// The block's own rows (the last M of every sequence's G + M) of the head's input and of its row statistics, packed
// for the output head: row b * (G + M) + G + i -> row b * M + i.  One CTA per row.
__global__ void compact_head_rows_kernel(__nv_bfloat16 *dst, const __nv_bfloat16 *src, size_t plane, float *ssq_dst,
                                         const float *ssq_src, int ssq_stride, int ssq_n, int d, int M, int G,
                                         const int *run_flag) {
    RUN_FLAG_EXIT(run_flag);
    PDL_TRIGGER();
    const int r = blockIdx.x, b = r / M, i = r % M, from = b * (G + M) + G + i;
    const uint4 *s0 = reinterpret_cast<const uint4 *>(src + (size_t)from * d), *s1 = reinterpret_cast<const uint4 *>(src + plane + (size_t)from * d);
    uint4 *d0 = reinterpret_cast<uint4 *>(dst + (size_t)r * d), *d1 = reinterpret_cast<uint4 *>(dst + plane + (size_t)r * d);
    for (int c = threadIdx.x; c < d / 8; c += blockDim.x) { d0[c] = s0[c]; d1[c] = s1[c]; }
    for (int e = threadIdx.x; e < ssq_n; e += blockDim.x) ssq_dst[(size_t)e * ssq_stride + r] = ssq_src[(size_t)e * ssq_stride + from];
}

int launch_compact_head_rows(const viasd_model *m, int batch, int M, int G, cudaStream_t st) {
    const viasd_config &c = m->cfg;
    compact_head_rows_kernel<<<batch * M, 128, 0, st>>>((__nv_bfloat16 *)m->ws.a_head, (const __nv_bfloat16 *)m->ws.a,
        m->ws.rows_alloc * (size_t)c.d_model, m->ws.ssq_head, m->ws.ssq, (int)m->ws.rows_alloc, (c.d_model / 128) * 4,
        c.d_model, M, G, m->run_flag);
    LAUNCH_CHECK();
    return VIASD_OK;
}

// ---------------------------------------------------------------------------------------------
// embedding gather: h[r] = E[token of row r]
// ---------------------------------------------------------------------------------------------
template <typename T>
__global__ void embed_kernel(float *h, const T *E, const PrepArgs p, int d) {
    __shared__ int par_sh[VIASD_MAX_ROWS_PER_SEQ];
    PDL_TRIGGER();
    const int r = (int)blockIdx.x - prep_ctas(p);
    if (r < 0) { if (threadIdx.x < 32) prep_sequence(p, blockIdx.x, par_sh); return; }
    const T *src = E + (size_t)prep_token(p, r) * d;
    for (int i = threadIdx.x; i < d; i += blockDim.x) h[(size_t)r * d + i] = to_f32<T>(src[i]);
}

// One embedding row by one CTA of 8 warps: h = E[tok], a = hi/lo(h * gain), sums of h^2 per 32 features.
// The row and the gains are loaded in batches of eight independent loads per thread: the embedding rows are cold in
// HBM, and one load per loop trip made this kernel a chain of memory round trips.
__device__ __forceinline__ void embed_row(float *h, __nv_bfloat16 *a, size_t plane, float *ssq, int ssq_stride,
                                          const __nv_bfloat16 *src, const float *gain, int r, int d, int warp, int lane) {
    for (int base0 = 0; base0 < d; base0 += 8 * 256) {
        float v[8], g[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const int base = base0 + j * 256, i = base + warp * 32 + lane;   // d is a multiple of 128: whole warps stay in range
            const bool on = base + warp * 32 < d;
            v[j] = on ? __bfloat162float(src[i]) : 0.f;
            g[j] = on ? gain[i] : 0.f;
        }
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const int base = base0 + j * 256, i = base + warp * 32 + lane;
            if (base + warp * 32 < d) {
                h[(size_t)r * d + i] = v[j];
                store_act<__nv_bfloat16>(a, plane, (size_t)r * d + i, v[j] * g[j]);
                const float sq = warp_sum(v[j] * v[j]);
                if (lane == 0) ssq[(size_t)(i >> 5) * ssq_stride + r] = sq;   // (tile * 4 + quarter) == feature / 32
            }
        }
    }
}

// Embedding gather fused with the preparation of the first RMSNorm of the pass (tensor-core path):
// h = E[tok]; a = hi/lo(h * gain); partial sums of h^2 per 32 features in the layout the GEMM epilogue reads.
// Rows from `rows` on are the second stream's (both verifiers in one sweep): the same tokens, prepared for the slim
// verifier's first routed layer.
__global__ void __launch_bounds__(256)
embed_norm_kernel(float *h, __nv_bfloat16 *a, size_t plane, float *ssq, int ssq_stride, const __nv_bfloat16 *E,
                  const float *gain_full, const float *gain_slim, const PrepArgs p, int d, int rows, const int *run_flag) {
    RUN_FLAG_EXIT(run_flag);
    __shared__ int par_sh[VIASD_MAX_ROWS_PER_SEQ];
    const int r = (int)blockIdx.x - prep_ctas(p), warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    PDL_TRIGGER();
    PDL_WAIT();
    if (r < 0) { if (warp == 0) prep_sequence(p, blockIdx.x, par_sh); return; }
    const __nv_bfloat16 *src = E + (size_t)prep_token(p, r < rows ? r : r - rows) * d;
    embed_row(h, a, plane, ssq, ssq_stride, src, r < rows ? gain_full : gain_slim, r, d, warp, lane);
}

int launch_embed_norm(const viasd_model *m, const viasd_cache *c, const viasd_draft *d, bool full_pass, bool replay, const float *gain,
                      const float *gain_slim, int rows, cudaStream_t st) {
    const PrepArgs p = prep_args(m, c, d, full_pass, replay);
    CUDA_TRY(launch_chained(embed_norm_kernel, (replay ? 0 : d->batch) + (gain_slim ? 2 : 1) * rows, 256, st,
        m->ws.h, (__nv_bfloat16 *)m->ws.a, m->ws.rows_alloc * m->cfg.d_model, m->ws.ssq, (int)m->ws.rows_alloc,
        (const __nv_bfloat16 *)m->embed, gain, gain_slim, p, m->cfg.d_model, rows, m->run_flag));
    LAUNCH_CHECK();
    return VIASD_OK;
}

int launch_embed(const viasd_model *m, const viasd_cache *c, const viasd_draft *d, bool full_pass, int rows, cudaStream_t st) {
    const PrepArgs p = prep_args(m, c, d, full_pass, false);
    if (m->cfg.dtype == 0)
        embed_kernel<float><<<d->batch + rows, 256, 0, st>>>(m->ws.h, (const float *)m->embed, p, m->cfg.d_model);
    else
        embed_kernel<__nv_bfloat16><<<d->batch + rows, 256, 0, st>>>(m->ws.h, (const __nv_bfloat16 *)m->embed, p, m->cfg.d_model);
    LAUNCH_CHECK();
    return VIASD_OK;
}

// ---------------------------------------------------------------------------------------------
// RMSNorm: a[r] = h[r] / sqrt(mean(h[r]^2) + eps) * gain, written in the model dtype
// ---------------------------------------------------------------------------------------------
template <typename T>
__global__ void __launch_bounds__(256)
rmsnorm_kernel(T *a, size_t plane, const float *h, const float *gain, int d, float eps) {
    __shared__ float red[8];
    PDL_TRIGGER();
    PDL_WAIT();
    const int r = blockIdx.x;
    const float4 *x4 = reinterpret_cast<const float4 *>(h + (size_t)r * d);
    constexpr int MAXV = 8;                           // up to 8 float4 per thread: d <= 8192 stays in registers
    const int nv = d >> 2;
    float4 v[MAXV];
    float s = 0.f;
#pragma unroll
    for (int j = 0; j < MAXV; ++j) {
        const int i = threadIdx.x + j * 256;
        if (i < nv) { v[j] = x4[i]; s += v[j].x * v[j].x + v[j].y * v[j].y + v[j].z * v[j].z + v[j].w * v[j].w; }
    }
    for (int i = threadIdx.x + MAXV * 256; i < nv; i += 256) { float4 t = x4[i]; s += t.x * t.x + t.y * t.y + t.z * t.z + t.w * t.w; }
    s = warp_sum(s);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
    __syncthreads();
    float tot = 0.f;
#pragma unroll
    for (int w = 0; w < 8; ++w) tot += red[w];
    const float inv = rsqrtf(tot / (float)d + eps);
    auto emit = [&](int i, float4 t) {
        const float4 g = load_floats4(gain + 4 * i);
        const size_t o = (size_t)r * d + (size_t)i * 4;
        store_act<T>(a, plane, o, t.x * inv * g.x);
        store_act<T>(a, plane, o + 1, t.y * inv * g.y);
        store_act<T>(a, plane, o + 2, t.z * inv * g.z);
        store_act<T>(a, plane, o + 3, t.w * inv * g.w);
    };
#pragma unroll
    for (int j = 0; j < MAXV; ++j) {
        const int i = threadIdx.x + j * 256;
        if (i < nv) emit(i, v[j]);
    }
    for (int i = threadIdx.x + MAXV * 256; i < nv; i += 256) emit(i, x4[i]);
}

int launch_rmsnorm(const viasd_model *m, const float *gain, int rows, cudaStream_t st) {
    if (m->cfg.dtype == 0)
        CUDA_TRY(launch_chained(rmsnorm_kernel<float>, rows, 256, st, (float *)m->ws.a, 0, m->ws.h, gain, m->cfg.d_model, m->cfg.rms_eps));
    else
        CUDA_TRY(launch_chained(rmsnorm_kernel<__nv_bfloat16>, rows, 256, st, (__nv_bfloat16 *)m->ws.a, m->ws.rows_alloc * m->cfg.d_model,
                                m->ws.h, gain, m->cfg.d_model, m->cfg.rms_eps));
    LAUNCH_CHECK();
    return VIASD_OK;
}

// ---------------------------------------------------------------------------------------------
// rotary embedding of q and k, KV append at slot len + row
// ---------------------------------------------------------------------------------------------
template <typename T>
__global__ void rope_append_kernel(float *q_out, T *kc, T *vc, const float *qkv, const float *cosv, const float *sinv,
                                   const int *len_eff, const TreeInfo *tree, int M, int H, int Hkv, int hd,
                                   int max_batch, int max_ctx, int layer_ord) {
    int r = blockIdx.x, head = blockIdx.y;
    PDL_TRIGGER();
    PDL_WAIT();
    int b = r / M, i = r % M;
    int half = hd >> 1;
    int n = len_eff[b];
    int pos = n + tree[b].depth[i], slot = n + i;
    const float *src = qkv + (size_t)r * (H + 2 * Hkv) * hd + (size_t)head * hd;
    for (int p = threadIdx.x; p < half; p += blockDim.x) {
        float x1 = src[p], x2 = src[p + half];
        if (head < H + Hkv) {
            float c = cosv[(size_t)pos * half + p], s = sinv[(size_t)pos * half + p];
            float y1 = x1 * c - x2 * s, y2 = x2 * c + x1 * s;
            if (head < H) {
                float *dst = q_out + (size_t)r * H * hd + (size_t)head * hd;
                dst[p] = y1;
                dst[p + half] = y2;
            } else {
                int g = head - H;
                T *dst = kc + ((((size_t)layer_ord * max_batch + b) * Hkv + g) * max_ctx + slot) * hd;
                dst[p] = from_f32<T>(y1);
                dst[p + half] = from_f32<T>(y2);
            }
        } else {
            int g = head - H - Hkv;
            T *dst = vc + ((((size_t)layer_ord * max_batch + b) * Hkv + g) * max_ctx + slot) * hd;
            dst[p] = from_f32<T>(x1);
            dst[p + half] = from_f32<T>(x2);
        }
    }
}

int launch_rope_append(const viasd_model *m, void *kc, void *vc, int layer_ord, int batch, int M, cudaStream_t st) {
    const viasd_config &c = m->cfg;
    dim3 grid(batch * M, c.n_heads + 2 * c.n_kv_heads);
    int threads = c.head_dim / 2 < 32 ? 32 : c.head_dim / 2;
    if (c.dtype == 0)
        CUDA_TRY(launch_chained(rope_append_kernel<float>, grid, threads, st, m->ws.q, (float *)kc, (float *)vc, m->ws.qkv,
            m->ws.rope_cos, m->ws.rope_sin, m->ws.len_eff, m->ws.tree, M, c.n_heads, c.n_kv_heads, c.head_dim,
            c.max_batch, c.max_ctx, layer_ord));
    else
        // (an ordinary launch: the attention kernel behind it reads lengths and tree ahead of its wait)
        rope_append_kernel<__nv_bfloat16><<<grid, threads, 0, st>>>(m->ws.q, (__nv_bfloat16 *)kc,
            (__nv_bfloat16 *)vc, m->ws.qkv, m->ws.rope_cos, m->ws.rope_sin, m->ws.len_eff, m->ws.tree, M, c.n_heads,
            c.n_kv_heads, c.head_dim, c.max_batch, c.max_ctx, layer_ord);
    LAUNCH_CHECK();
    return VIASD_OK;
}

// ---------------------------------------------------------------------------------------------
// KV commit: compact the accepted path, advance len / pending / tokens
// ---------------------------------------------------------------------------------------------
// A warp moves the path's rows of one (layer, sequence, kv head), K by its first half and V by its second, eight rows in
// flight, in pieces of 16 bytes where the caches are aligned to that (an fp32 cache, or one of head_dim 64, need not be), else
// of one element; the last CTA to finish advances the lengths (nobody reads them before).  (Three launches -
// lengths, rows one 2-byte column per thread and row after row, advance - were 15 to 27 us.)
struct CommitArgs {
    void *kf, *vf, *ks, *vs;
    int *len, *len_full, *pending, *tokens;
    const int *n_acc, *path, *n_emit, *out_tok;
    DeviceStats *stats;
    int B, N, L, Ls, layer0, Hkv, row_vecs, max_batch, max_ctx, slim_only;   // row_vecs: pieces of a K (or V) row
};
constexpr int COMMIT_WARPS = 8;

template <typename Piece>
__global__ void __launch_bounds__(32 * COMMIT_WARPS) commit_kernel(const CommitArgs a) {
    __shared__ int last_sh;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, M = a.N + 1;
    const int item = blockIdx.x * COMMIT_WARPS + warp, n_items = (a.L + a.Ls - a.layer0) * a.B * a.Hkv;
    PDL_WAIT();
    const bool full_ran = a.stats->full_ran != 0;
    if (item < n_items) {
        const int g = item % a.Hkv, b = (item / a.Hkv) % a.B, layer = a.layer0 + item / (a.Hkv * a.B);
        const bool is_full = layer < a.L;
        if (full_ran || !is_full) {                            // else the full verifier's cache did not receive this block
            const int half = lane >> 4, l16 = lane & 15;
            Piece *base = reinterpret_cast<Piece *>(is_full ? (half ? a.vf : a.kf) : (half ? a.vs : a.ks)) +
                          (((size_t)(is_full ? layer : layer - a.L) * a.max_batch + b) * a.Hkv + g) * (size_t)a.max_ctx * a.row_vecs;
            const int n = clamped_len(a.len, b, a.max_ctx, M, a.stats), na = min(a.n_acc[b], a.N);
            // a path's nodes never come before their position (node >= j), so rows only move down and no row that is still to
            // be moved is overwritten; an invalid entry ends the path
            bool more = true;
            for (int j0 = 0; more && j0 < na; j0 += 8) {
                int src[8];
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const int node = j0 + j < na ? a.path[b * a.N + j0 + j] : -1;
                    more = more && node >= j0 + j && node < a.N;
                    src[j] = more && node != j0 + j ? n + 1 + node : -1;
                }
                for (int c = l16; c < a.row_vecs; c += 16) {
                    Piece v[8];
#pragma unroll
                    for (int j = 0; j < 8; ++j) if (src[j] >= 0) v[j] = base[(size_t)src[j] * a.row_vecs + c];
#pragma unroll
                    for (int j = 0; j < 8; ++j) if (src[j] >= 0) base[(size_t)(n + 1 + j0 + j) * a.row_vecs + c] = v[j];
                }
            }
        }
    }
    if (a.slim_only) return;
    __syncthreads();
    if (threadIdx.x == 0) {
        int old;
        asm volatile("atom.acq_rel.gpu.global.add.s32 %0, [%1], 1;" : "=r"(old) : "l"(&a.stats->commit_ctas) : "memory");
        last_sh = old == (int)gridDim.x - 1;
        if (last_sh) a.stats->commit_ctas = 0;
    }
    __syncthreads();
    if (!last_sh) return;
    for (int b = threadIdx.x; b < a.B; b += blockDim.x) {
        const int n = clamped_len(a.len, b, a.max_ctx, M, a.stats), ne = min(max(a.n_emit[b], 0), a.N + 1);
        // the full verifier's cache is complete up to the new length exactly when its pass ran in this step
        if (a.len_full && full_ran) a.len_full[b] = n + ne;
        if (b == 0 && !full_ran) ++a.stats->full_skipped;
        if (ne == 0) continue;
        if (a.tokens) {
            a.tokens[(size_t)b * a.max_ctx + n] = a.pending[b];
            for (int j = 0; j + 1 < ne; ++j) a.tokens[(size_t)b * a.max_ctx + n + 1 + j] = a.out_tok[b * (a.N + 1) + j];
        }
        a.len[b] = n + ne;
        a.pending[b] = a.out_tok[b * (a.N + 1) + ne - 1];
    }
}

// slim_only: move the accepted rows in this handle's slim cache and nothing else (lengths, pending token and token
// list belong to the handle that commits last)
int launch_commit(const viasd_model *m, viasd_cache *c, const viasd_draft *d, const viasd_result *r, bool slim_only,
                  cudaStream_t st) {
    const viasd_config &cf = m->cfg;
    CommitArgs a;
    a.kf = c->k_full; a.vf = c->v_full; a.ks = c->k_slim; a.vs = c->v_slim;
    a.len = c->len; a.len_full = c->len_full; a.pending = c->pending; a.tokens = c->tokens;
    a.n_acc = r->n_acc; a.path = r->path; a.n_emit = r->n_emit; a.out_tok = r->out_tok;
    a.stats = m->ws.stats;
    a.B = d->batch; a.N = d->n_nodes; a.L = cf.n_layers; a.Ls = m->n_routed; a.layer0 = slim_only ? cf.n_layers : 0;
    a.Hkv = cf.n_kv_heads; 
    a.max_batch = cf.max_batch; a.max_ctx = cf.max_ctx; a.slim_only = slim_only ? 1 : 0;
    const int items = (cf.n_layers + m->n_routed - a.layer0) * d->batch * cf.n_kv_heads;
    const bool vec = (((uintptr_t)a.kf | (uintptr_t)a.vf | (uintptr_t)a.ks | (uintptr_t)a.vs) & 15) == 0;
    auto kernel = vec ? commit_kernel<uint4> : cf.dtype == 0 ? commit_kernel<uint32_t> : commit_kernel<uint16_t>;
    a.row_vecs = vec ? cf.head_dim * (cf.dtype == 0 ? 4 : 2) / 16 : cf.head_dim;
    CUDA_TRY(launch_chained(kernel, (items + COMMIT_WARPS - 1) / COMMIT_WARPS, 32 * COMMIT_WARPS, st, a));
    LAUNCH_CHECK();
    return VIASD_OK;
}
