// Choice of the attention kernel, and the CUDA-core kernel for fp32 models and head_dim 64.
// KV-append attention over a drafted block: each of the M query rows of a sequence attends to the
// committed cache rows 0..n-1 and to the block rows on its own root path (causal mask for a chain,
// ancestor mask for a tree).  Split-KV: a CTA handles one (sequence, kv head, key range, group of
// query rows), keeps an online softmax per query row and writes unnormalised partials; a second
// kernel merges the key ranges.
#include "common.cuh"
#include <string.h>
#include <stdlib.h>
#include <type_traits>

namespace {

constexpr int TK = 32;          // keys per shared-memory tile
constexpr int QG = 16;          // query rows per CTA (2 per warp, 8 warps)
constexpr int ATT_WARPS = 8;

// VEC: K and V are aligned to 16 bytes (the caller's caches need not be)
template <typename T, int HD, bool VEC>
__global__ void __launch_bounds__(ATT_WARPS * 32)
attention_split_kernel(float *__restrict__ part, const float *__restrict__ q, const T *__restrict__ kc,
                       const T *__restrict__ vc, const int *__restrict__ len_eff, const TreeInfo *__restrict__ tree,
                       int M, int H, int Hkv, int max_batch, int max_ctx, int layer_ord, int nsplit, float scale,
                       const int *run_flag) {
    RUN_FLAG_EXIT(run_flag);
    __shared__ float Qs[QG][HD];
    __shared__ float Ks[TK][HD + 1];
    __shared__ float Vs[TK][HD];
    constexpr int DPL = HD / 32;                     // output dims per lane
    PDL_TRIGGER();
    PDL_WAIT();
    const int b = blockIdx.x / Hkv, g = blockIdx.x % Hkv, split = blockIdx.y, qg = blockIdx.z;
    const int grp = H / Hkv, QR = grp * M;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int n = len_eff[b], Tk = n + M;
    int chunk = (Tk + nsplit - 1) / nsplit;
    chunk = (chunk + TK - 1) / TK * TK;
    const int k_begin = split * chunk, k_end = min(Tk, k_begin + chunk);

    // stage this CTA's query rows, pre-scaled
    for (int idx = threadIdx.x; idx < QG * HD; idx += blockDim.x) {
        int qq = idx / HD, dd = idx % HD;
        int qidx = qg * QG + qq;
        float v = 0.f;
        if (qidx < QR) {
            int h = g * grp + qidx / M, i = qidx % M;
            v = q[((size_t)(b * M + i) * H + h) * HD + dd] * scale;
        }
        Qs[qq][dd] = v;
    }
    float mrun[2] = {-INFINITY, -INFINITY}, lrun[2] = {0.f, 0.f}, o[2][DPL];
#pragma unroll
    for (int r = 0; r < 2; ++r)
#pragma unroll
        for (int c = 0; c < DPL; ++c) o[r][c] = 0.f;
    unsigned long long anc[2];
    int qrow[2];
#pragma unroll
    for (int r = 0; r < 2; ++r) {
        int qidx = qg * QG + warp * 2 + r;
        qrow[r] = qidx < QR ? qidx : -1;
        anc[r] = qidx < QR ? tree[b].anc[qidx % M] : 0ull;
    }
    const size_t cbase = (((size_t)layer_ord * max_batch + b) * Hkv + g) * (size_t)max_ctx * HD;

    for (int k0 = k_begin; k0 < k_end; k0 += TK) {
        __syncthreads();
        // 16-byte loads, all of a thread's in flight together; an element at a time where the caches are not aligned to that
        constexpr int VE = VEC ? 16 / (int)sizeof(T) : 1, NV = VEC ? TK * HD / VE / (ATT_WARPS * 32) : 4;
        constexpr int STEP = NV * VE * ATT_WARPS * 32;
        using Piece = typename std::conditional<VEC, uint4, T>::type;
        static_assert(TK * HD % STEP == 0, "whole pieces per thread");
#pragma unroll 1
        for (int at = 0; at < TK * HD; at += STEP) {
            Piece kraw[NV], vraw[NV];
#pragma unroll
            for (int q = 0; q < NV; ++q) {
                const int idx = at + (threadIdx.x + q * ATT_WARPS * 32) * VE, j = idx / HD;
                const size_t o = cbase + (size_t)min(k0 + j, k_end - 1) * HD + idx % HD;
                kraw[q] = *reinterpret_cast<const Piece *>(kc + o);
                vraw[q] = *reinterpret_cast<const Piece *>(vc + o);
            }
#pragma unroll
            for (int q = 0; q < NV; ++q) {
                const int idx = at + (threadIdx.x + q * ATT_WARPS * 32) * VE, j = idx / HD, dd = idx % HD;
                const bool in = k0 + j < k_end;
                alignas(16) T kv[VE], vv[VE];
                *reinterpret_cast<Piece *>(kv) = kraw[q];
                *reinterpret_cast<Piece *>(vv) = vraw[q];
#pragma unroll
                for (int e = 0; e < VE; ++e) { Ks[j][dd + e] = in ? to_f32<T>(kv[e]) : 0.f; Vs[j][dd + e] = in ? to_f32<T>(vv[e]) : 0.f; }
            }
        }
        __syncthreads();
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            if (qrow[r] < 0) continue;
            const int j = k0 + lane;
            const bool valid = j < k_end && (j < n || ((anc[r] >> (j - n)) & 1ull));
            float s = 0.f;
            const float *qs = Qs[warp * 2 + r];
#pragma unroll 8
            for (int dd = 0; dd < HD; ++dd) s = fmaf(qs[dd], Ks[lane][dd], s);
            s = valid ? s : -INFINITY;
            float mnew = fmaxf(mrun[r], warp_max(s));
            if (mnew == -INFINITY) continue;                     // nothing visible yet
            float p = valid ? expf(s - mnew) : 0.f;
            float corr = expf(mrun[r] - mnew);                   // exp(-inf) = 0 on the first tile
            lrun[r] = lrun[r] * corr + warp_sum(p);
#pragma unroll
            for (int c = 0; c < DPL; ++c) o[r][c] *= corr;
#pragma unroll 8
            for (int jj = 0; jj < TK; ++jj) {
                float pj = __shfl_sync(0xffffffffu, p, jj);
#pragma unroll
                for (int c = 0; c < DPL; ++c) o[r][c] = fmaf(pj, Vs[jj][lane + 32 * c], o[r][c]);
            }
            mrun[r] = mnew;
        }
    }
#pragma unroll
    for (int r = 0; r < 2; ++r) {
        if (qrow[r] < 0) continue;
        int h = g * grp + qrow[r] / M, i = qrow[r] % M;
        float *dst = part + ((((size_t)b * H + h) * M + i) * nsplit + split) * (HD + 2);
#pragma unroll
        for (int c = 0; c < DPL; ++c) dst[lane + 32 * c] = o[r][c];
        if (lane == 0) { dst[HD] = mrun[r]; dst[HD + 1] = lrun[r]; }
    }
}

template <typename T, int HD>
__global__ void attention_combine_kernel(T *__restrict__ out, size_t plane, const float *__restrict__ part, int M, int H,
                                         int nsplit, const int *run_flag) {
    RUN_FLAG_EXIT(run_flag);
    const int r = blockIdx.x, h = blockIdx.y;        // r = b * M + i
    PDL_TRIGGER();
    PDL_WAIT();
    const int b = r / M, i = r % M;
    const float *src = part + (((size_t)b * H + h) * M + i) * (size_t)nsplit * (HD + 2);
    float mmax = -INFINITY;
    for (int s = 0; s < nsplit; ++s) mmax = fmaxf(mmax, src[(size_t)s * (HD + 2) + HD]);
    for (int dd = threadIdx.x; dd < HD; dd += blockDim.x) {
        float num = 0.f, den = 0.f;
        for (int s = 0; s < nsplit; ++s) {
            const float *p = src + (size_t)s * (HD + 2);
            float ms = p[HD];
            if (ms == -INFINITY) continue;
            float w = expf(ms - mmax);
            num = fmaf(p[dd], w, num);
            den = fmaf(p[HD + 1], w, den);
        }
        store_act<T>(out, plane, ((size_t)r * H + h) * HD + dd, num / den);
    }
}

template <typename T, int HD>
int run(const viasd_model *m, const void *kc, const void *vc, int layer_ord, int batch, int M, int nsplit,
        cudaStream_t st) {
    const viasd_config &c = m->cfg;
    const int grp = c.n_heads / c.n_kv_heads;
    const int qgroups = (grp * M + QG - 1) / QG;
    dim3 grid(batch * c.n_kv_heads, nsplit, qgroups);
    const bool vec = (((uintptr_t)kc | (uintptr_t)vc) & 15) == 0;
    CUDA_TRY(launch_chained(vec ? attention_split_kernel<T, HD, true> : attention_split_kernel<T, HD, false>, grid, ATT_WARPS * 32, st, m->ws.part, m->ws.q, (const T *)kc,
        (const T *)vc, m->ws.len_eff, m->ws.tree, M, c.n_heads, c.n_kv_heads, c.max_batch, c.max_ctx, layer_ord, nsplit,
        1.0f / sqrtf((float)HD), m->run_flag));
    LAUNCH_CHECK();
    CUDA_TRY(launch_chained(attention_combine_kernel<T, HD>, dim3(batch * M, c.n_heads), HD < 128 ? HD : 128, st, (T *)m->ws.attn,
        sizeof(T) == 2 ? m->ws.rows_alloc * (size_t)c.n_heads * HD : 0, m->ws.part, M, c.n_heads, nsplit, m->run_flag));
    LAUNCH_CHECK();
    return VIASD_OK;
}

}  // namespace

int attention_nsplit(const viasd_model *m, int batch, int M) {
    const viasd_config &c = m->cfg;
    const int grp = c.n_heads / c.n_kv_heads;
    const int qgroups = (grp * M + QG - 1) / QG;
    int ctas = batch * c.n_kv_heads * qgroups;
    int nsplit = (2 * m->sm_count + ctas - 1) / ctas;
    int by_len = (c.max_ctx + TK - 1) / TK;          // at least one tile per split: with few CTAs a tile is a chain of latencies
    if (nsplit > by_len) nsplit = by_len;
    if (nsplit > 16) nsplit = 16;
    if (nsplit < 1) nsplit = 1;
    // never beyond what the partial buffer holds
    size_t per_split = (size_t)batch * c.n_heads * M * (c.head_dim + 2) * sizeof(float);
    while (nsplit > 1 && per_split * nsplit > m->ws.part_bytes) --nsplit;
    return nsplit;
}

// Key ranges per (sequence, kv head) for the keys-on-lanes kernel, from a small cost model: items are dealt to
// CTAs in equal contiguous shares, each item costs a fixed part (query staging, merge, partial) plus its tiles,
// and every extra range adds merge work.  Depends on batch, heads and M only, so the one-stream and the two-stream
// launch cut the keys at the same places and produce the same bits.
static int tk_nsplit(const viasd_model *m, int batch, int M, int streams, int subs, int rows) {
    const viasd_config &c = m->cfg;
    const int base = batch * c.n_kv_heads * subs, sms = m->sm_count;      // subs: items per kv head
    const int tiles = (c.max_ctx + 127) / 128;
    const int max_s = tiles < 16 ? tiles : 16;                  // the partial buffer holds 16 ranges per (row, head)
    // microseconds, roughly: a tile costs its softmax chain, 1.1 - 1.8 us with 8 - 32 rows per item, an item 5 - 10 us of
    // query staging, result rows and merge
    const double t_tile = rows > 16 ? 1.8 : rows > 8 ? 1.3 : 1.1, t_item = rows > 16 ? 8.0 : 5.0;
    // One choice for the whole model, whichever call runs (the cuts must not depend on it): the routed layers are
    // charged as two-stream launches, as the verify step runs them, the others as one-stream launches.
    const int n_dual = m->n_routed, n_single = c.n_layers - m->n_routed;
    int best = 1;
    double best_cost = 1e30;
    for (int s = 1; s <= max_s; ++s) {
        const int tpi = ((tiles + s - 1) / s);
        double cost = 0.15 * s * (n_dual + n_single);
        for (int st2 = 1; st2 <= 2; ++st2) {
            const int n = base * s * st2, ipc = (n + sms - 1) / sms;
            cost += (st2 == 2 ? n_dual : n_single) * ipc * (tpi * t_tile + t_item);
        }
        if (cost < best_cost - 1e-9) { best_cost = cost; best = s; }
    }
    if (m->opt.attn_splits >= 1 && m->opt.attn_splits <= max_s) best = m->opt.attn_splits;
    size_t per_split = (size_t)streams * batch * c.n_heads * M * (c.head_dim + 2) * sizeof(float);
    while (best > 1 && per_split * best > m->ws.part_bytes) --best;
    return best;
}

// Attention on the tensor cores: the choice of the kernel.
static int mma_attention(viasd_model *m, const void *kc, const void *vc, bool slim, int layer_ord, const void *kc2,
                         const void *vc2, int layer_ord2, int streams, int batch, int M, cudaStream_t st) {
    const viasd_config &c = m->cfg;
    // VIASD_OPT_ATTENTION_KERNEL: mma.sync (up to 16 query rows per kv head), tcgen05 with the query rows on the TMEM lanes
    // (any), or tcgen05 with the keys on the lanes (up to 32 rows per item); by default, as below.
    const int kind = m->opt.attn_kernel == 1 ? 0 : m->opt.attn_kernel == 2 ? 1 : m->opt.attn_kernel == 3 ? 2 : 3;   // 0 mma, 1 tc, 2 tk, 3 default
    const int QR = (c.n_heads / c.n_kv_heads) * M;
    // More than 32 query rows per kv head: the rows-on-lanes kernel, whose tile costs the same whatever the rows (per layer,
    // 32 / 8 heads, against the better of the two others: 36 rows, 1 sequence of 2048 -1.7 us, 16 sequences of 1000 -16 us;
    // 108 rows, 1 sequence of 100 -2.7 us, of 2048 -5, 4 sequences of 2048 -12, 16 of 1000 -66; at 32 rows and 2048 keys or
    // more it is 0.6 - 1.5 us behind).  17 - 32 rows: keys-on-lanes, whose MMAs are that much narrower, from one tile per SM
    // on (24 rows, 1 sequence of 8000 -3.2 us), rows-on-lanes for less (1 sequence of 100: -4.8 us, of 600 -2.2).  Up to 16
    // rows: mma.sync, whose chain is the shortest for a few tiles, until keys-on-lanes streams 36 tiles per SM (32 kv heads,
    // 9 rows: 2 sequences of 2048 +11 us, 4 of 2048 (31 tiles) +5, 8 of 1500 (45) -9; 8 kv heads, 16 rows, 8 of 4000 +4.6).
    // Tiles of both row streams, whichever the launch has: the choice must not depend on it.
    const long long tiles_two = 2LL * batch * c.n_kv_heads * ((c.max_ctx + 127) / 128);
    const int grp = c.n_heads / c.n_kv_heads, hpi = attention_tk_heads_per_item(grp, M);
    const int subs = hpi ? grp / hpi : 1, QRi = hpi * M;       // keys-on-lanes: items per kv head, query rows per item
    int use = kind != 3 ? kind : QR > 32 ? 1 : QR > 16 ? (tiles_two >= m->sm_count ? 2 : 1) : tiles_two >= 36LL * m->sm_count ? 2 : 0;
    if (use == 2 && !hpi) use = 0;
    if (use == 0 && !attention_mma_supported(m, M)) use = 1;   // (asked for by option, with more rows than its one query tile)
    if (use == 1) return launch_attention_tc(m, kc, vc, slim, layer_ord, kc2, vc2, layer_ord2, streams, batch, M, st);
    if (use == 0) return launch_attention_mma(m, kc, vc, slim, layer_ord, kc2, vc2, layer_ord2, streams, batch, M, st);
    // The keys-on-lanes kernel deals tiles, not key ranges, evenly to the CTAs (nsplit 0) when the partial buffer has its 16
    // slots per (row, head): whole (sequence, head) items leave SMs idle (320 items on 148 SMs: a quarter of them).  Its
    // merges are then always fused.  Not with more than 16 query rows per kv head: there an item's fixed cost (staging 32
    // rows of queries, 32 rows of results) is worth a dozen tiles, and the extra item per CTA cost more than the balance
    // won (32B batch-16 step 36.5 -> 39.0 ms).  VIASD_OPT_TK_FLAT overrides.
    const size_t need = (size_t)streams * batch * c.n_heads * M * 16 * (c.head_dim + 2) * sizeof(float);
    if ((m->opt.tk_flat >= 0 ? m->opt.tk_flat != 0 : QR <= 16) && subs == 1 && need <= m->ws.part_bytes)
        return launch_attention_tk(m, kc, vc, slim, layer_ord, kc2, vc2, layer_ord2, streams, batch, M, 0, 1, st);
    const int nsplit = tk_nsplit(m, batch, M, streams, subs, QRi);
    const bool fuse = nsplit > 1 && QRi * nsplit <= 160;
    int rc = launch_attention_tk(m, kc, vc, slim, layer_ord, kc2, vc2, layer_ord2, streams, batch, M, nsplit, fuse ? 1 : 0, st);
    if (rc || nsplit == 1 || fuse) return rc;
    CUDA_TRY(launch_chained(attention_combine_kernel<__nv_bfloat16, 128>, dim3(streams * batch * M, c.n_heads), 128, st,
        (__nv_bfloat16 *)m->ws.attn, m->ws.rows_alloc * (size_t)c.n_heads * 128, m->ws.part, M, c.n_heads, nsplit, m->run_flag));
    LAUNCH_CHECK();
    return VIASD_OK;
}

int launch_attention(viasd_model *m, const void *kc, const void *vc, bool slim, int layer_ord, int batch, int M,
                     cudaStream_t st) {
    const viasd_config &c = m->cfg;
    if (attention_tensor_supported(m)) {
        return mma_attention(m, kc, vc, slim, layer_ord, nullptr, nullptr, 0, 1, batch, M, st);
    }
    int nsplit = attention_nsplit(m, batch, M);
    if (c.dtype == 0) {
        if (c.head_dim == 64) return run<float, 64>(m, kc, vc, layer_ord, batch, M, nsplit, st);
        if (c.head_dim == 128) return run<float, 128>(m, kc, vc, layer_ord, batch, M, nsplit, st);
    } else {
        if (c.head_dim == 64) return run<__nv_bfloat16, 64>(m, kc, vc, layer_ord, batch, M, nsplit, st);
        if (c.head_dim == 128) return run<__nv_bfloat16, 128>(m, kc, vc, layer_ord, batch, M, nsplit, st);
    }
    return VIASD_EINVAL;
}

// Both verifiers in one launch: the full stream's rows against the full cache, the slim stream's rows against the
// slim cache (tensor-core kernel only).
int launch_attention_dual(viasd_model *m, const void *kf, const void *vf, int layer_full, const void *ks, const void *vs,
                          int ord_slim, int batch, int M, cudaStream_t st) {
    return mma_attention(m, kf, vf, false, layer_full, ks, vs, ord_slim, 2, batch, M, st);
}
