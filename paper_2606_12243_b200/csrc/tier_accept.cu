// Confidence tiers and accept / resolve.
//
// Tiers (App. B, Eq. B.1-B.3): per drafted token v, d = l[v] - max_u l[u] on the gating logits;
// tier 0 if d >= log_tau_hi, 1 if d >= log_tau_lo, else 2.  Asked for alone (phase 1) a kernel with one CTA per gating
// row scans the vocabulary; asked for together with the walk, the tiers come from the row statistics the walk needs anyway.
//
// Accept kernel (Algorithm 2, per-position loop; Algorithm 1, what is appended; App. A, Eq. A.2-A.3):
// one CTA per sequence (a cluster of 8 or 16 when it samples over a large vocabulary) walks the draft from the pending
// token: children of the current row are tried in index order; tier-0 children are taken at once, tier-1 children are
// judged by q', tier-2 children by q.  The first row where no child passes ends the walk and the strongest judge that
// rejected there emits the replacement token.  The walk is sequential over depth, so everything that can be known before
// it is: a row-statistics kernel (a CTA per logits row, or per part of one, one sweep) leaves each row's maximum, argmax
// and softmax denominator, in parts, and the walk starts by fetching the tree and every node's two logits at once, so that a test is
// arithmetic on shared memory.  Only a rejection in sampling mode (residual, Eq. A.3) and the final draw sweep the
// vocabulary: one sweep and one exchange among the cluster's CTAs each.  An element of a residual is worked out from the logits
// by replaying the rejections so far (a handful of scalars), in the arithmetic of Eq. A.3 round by round; every FOLD of them at
// one position are written out and the replay starts from there, so that a star of many children stays linear.  CTAs exchange their sums by storing them into each other's shared memory before one cluster barrier; every
// CTA adds them in the same order, so all of them walk the same way.
#include "common.cuh"
#include <string.h>
#include <stdlib.h>

namespace {

constexpr int ACC_THREADS = 512, ACC_WARPS = ACC_THREADS / 32;
constexpr int MAX_TEAM = 16;
constexpr int MAXJ = VIASD_MAX_JUDGES;    // verifiers that may judge a drafted token (the last one is q); 2 for three tiers
constexpr int KINDS = MAXJ + 1;           // distributions kept per position: the proposal and the judges
constexpr int ACC_TEAM = 8;               // CTAs per sequence in sampling mode (a portable cluster size)
// Rejections at one position that are replayed per element before they are written out.  Rejected children of one position,
// us, all written out as they come / all replayed / eight at a time: 63, vocabulary 128256 933 / 1264 / 457, 8000 495 / 1167 /
// 373, 1024 195 / - / 194; 12, vocabulary 128256 218 / 138 / 109.
constexpr int FOLD = 8;

// ---- counter-based uniforms -------------------------------------------------------------------
__device__ __forceinline__ unsigned long long mix64(unsigned long long z) {
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}
constexpr unsigned long long GAMMA = 0x9E3779B97F4A7C15ull;
__device__ __forceinline__ unsigned long long stream_key(unsigned long long seed, unsigned long long step, int b,
                                                         int stream) {
    unsigned long long k = mix64(seed + GAMMA);
    k = mix64(k + step * GAMMA + 1ull);
    return mix64(k + (unsigned long long)(b * 256 + stream) * GAMMA + 2ull);
}
// 23 random bits -> (k + 0.5) / 2^23: exact in fp32, strictly inside (0, 1)
__device__ __forceinline__ float unit_f32(unsigned long long key, unsigned long long idx) {
    unsigned long long w = mix64(key + idx * GAMMA + 3ull);
    return ((float)(w >> 41) + 0.5f) * 1.1920928955078125e-7f;
}

// ---- block reductions: in every thread; sh: a buffer nobody reads any more ----------------------
struct MaxIdx { float v; int i; };
__device__ __forceinline__ MaxIdx better(MaxIdx a, MaxIdx b) {   // larger value, lowest index on ties
    if (b.v > a.v || (b.v == a.v && b.i < a.i)) return b;
    return a;
}
__device__ __forceinline__ MaxIdx warp_argmax(MaxIdx x) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        MaxIdx y;
        y.v = __shfl_xor_sync(0xffffffffu, x.v, o);
        y.i = __shfl_xor_sync(0xffffffffu, x.i, o);
        x = better(x, y);
    }
    return x;
}
__device__ __forceinline__ MaxIdx no_idx() { MaxIdx r; r.v = -INFINITY; r.i = 0x7fffffff; return r; }
__device__ MaxIdx block_argmax(MaxIdx x, MaxIdx *sh) {
    x = warp_argmax(x);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = x;
    __syncthreads();
    const int lane = threadIdx.x & 31;
    return warp_argmax(lane < (int)(blockDim.x >> 5) ? sh[lane] : no_idx());
}
__device__ float block_sum(float x, float *sh) {
    x = warp_sum(x);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = x;
    __syncthreads();
    const int lane = threadIdx.x & 31;
    return warp_sum(lane < (int)(blockDim.x >> 5) ? sh[lane] : 0.f);
}
__device__ float block_max(float x, float *sh) {
    x = warp_max(x);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = x;
    __syncthreads();
    const int lane = threadIdx.x & 31;
    return warp_max(lane < (int)(blockDim.x >> 5) ? sh[lane] : -INFINITY);
}

// ---- tier kernel ------------------------------------------------------------------------------
// n thresholds in descending order cut the log-confidence axis into n + 1 tiers: tier 0 (accepted outright) from
// log_tau[0] up, tier k between log_tau[k] and log_tau[k - 1], tier n (the full verifier) below log_tau[n - 1].
struct TierCuts { int n; float log_tau[MAXJ]; };
// grid (gate rows per sequence, B).  conf_source 0: gate row of node n = prow[n], rows = drafter logits
// [B, R, V]; conf_source 1: gate row = parent[n] + 1, rows = slim logits [B, M, V].
__global__ void __launch_bounds__(1024)
tier_kernel(unsigned char *__restrict__ tier, float *__restrict__ conf, DeviceStats *stats,
            const float *__restrict__ gate_logits, const int *__restrict__ draft_tok, const int *__restrict__ prow,
            const int *__restrict__ parent, int per_seq, int conf_source, int rows_per_seq, int N, int V, TierCuts cuts) {
    __shared__ float sh[32];
    const int gr = blockIdx.x, b = blockIdx.y;
    if (per_seq) { prow += (size_t)b * N; parent += (size_t)b * N; }     // every sequence has its own tree
    const float *row = gate_logits + ((size_t)b * rows_per_seq + gr) * V;
    float mx = -INFINITY;
    if ((V & 3) == 0 && ((uintptr_t)row & 15) == 0) {
        const float4 *r4 = reinterpret_cast<const float4 *>(row);
        for (int i = threadIdx.x; i < V / 4; i += blockDim.x) {
            float4 v = r4[i];
            mx = fmaxf(mx, fmaxf(fmaxf(v.x, v.y), fmaxf(v.z, v.w)));
        }
    } else {
        for (int i = threadIdx.x; i < V; i += blockDim.x) mx = fmaxf(mx, row[i]);
    }
    mx = block_max(mx, sh);
    for (int n = threadIdx.x; n < N; n += blockDim.x) {
        if (parent[n] == -2) {                                   // unused node of this sequence's tree
            if (gr == 0) { tier[b * N + n] = 0; conf[b * N + n] = 0.f; }
            continue;
        }
        int g = conf_source == 0 ? prow[n] : parent[n] + 1;
        const bool ok = g >= 0 && g < rows_per_seq;              // no such gate row: an error, and the strictest tier
        if (g != gr && (ok || gr > 0)) continue;
        if (!ok) stats->device_status = VIASD_EDEVICE;
        int t = draft_tok[b * N + n];
        t = min(max(t, 0), V - 1);
        float d = ok ? row[t] - mx : -INFINITY;
        int tr = 0;                                              // thresholds descend: the first one d reaches names the tier
        while (tr < cuts.n && d < cuts.log_tau[tr]) ++tr;
        tier[b * N + n] = (unsigned char)tr;
        conf[b * N + n] = d;
        atomicAdd(&stats->tier_count[tr == 0 ? 0 : (tr == cuts.n ? 2 : 1)], 1ull);   // accepted / some slim verifier / q
        if (tr > 0 && tr < cuts.n) stats->need_slim = 1;
        if (tr == cuts.n) stats->need_full = 1;
    }
    if (gr == 0 && b == 0 && threadIdx.x == 0) atomicAdd(&stats->steps, 1ull);
}

// ---- row statistics ---------------------------------------------------------------------------
// One-dimensional grid over rows, kind by kind, and parts (RowUnits): kind 0 = drafter rows [B, R, V], kind k = judge k's rows
// [B, M, V] (the last judge is q).
// Per row: max, argmax (lowest index on ties) and, when wanted, sum exp((l - max) / T).
// HBM-bound: every row once.  Maximum and denominator come from one sweep (a running reference per thread, moved when it is
// exceeded by e^20); two sweeps read a batch's rows twice from HBM, 16 sequences' 1040 rows of 0.5 MB being far more than L2
// holds.  Eight 16-byte loads per thread in flight: few rows are bound by what a CTA has under way.
// A row's statistics are kept in parts, which the walk puts together.  Whole turns of two CTAs per SM take whole rows, part after
// part; what is left over goes a part per CTA, so that one sequence's 66 rows fill the chip and the last of 1040 rows' turns is a
// quarter as long (a part's numbers are the same either way).
constexpr int RS_STRIDE = VIASD_MAX_ROWS_PER_SEQ, RS_THREADS = 512, RS_BATCH = 8;
constexpr float RS_GAP = 20.f;
struct RowStats { float *mx; int *arg; float *z; };       // each [B, KINDS, RS_STRIDE, parts]
// (by the vocabulary: a row's sums do not depend on the call's other rows)
int row_parts(int vocab) { return vocab >= 65536 ? ROW_STAT_PARTS : vocab >= 16384 ? 2 : 1; }
struct RowPtrs { const float *p[KINDS]; };                // drafter logits, then each judge's

template <bool WANT_Z>
struct RowAcc {
    float ref, lim, s;
    MaxIdx best;
    __device__ __forceinline__ void init() { ref = lim = -INFINITY; s = 0.f; best = no_idx(); }
    // N values from index i on, in pieces of four `step` apart
    template <int N>
    __device__ __forceinline__ void add(const float (&x)[N], int i, int step, ExpScale scale, float gap) {
        float bm = x[0];
#pragma unroll
        for (int e = 1; e < N; ++e) bm = fmaxf(bm, x[e]);
        if (bm > best.v) {                                 // rare after the first batches
            best.v = bm;
#pragma unroll
            for (int e = N - 1; e >= 0; --e) if (x[e] == bm) best.i = i + (e >> 2) * step + (e & 3);
        }
        if (!WANT_Z) return;
        if (bm > lim) {
            s *= exp_scaled(ref - bm, scale);
            ref = bm;
            lim = bm + gap;
        }
        const float r = ref == -INFINITY ? 0.f : ref;
#pragma unroll
        for (int e = 0; e < N; ++e) s += exp_scaled(x[e] - r, scale);
    }
};

struct RowUnits { int B, R, M, whole, parts; };           // rows: [drafter rows of all sequences, unless R is 0][judge 1's] ..., the first `whole` by a CTA each
template <bool WANT_Z>
__global__ void __launch_bounds__(RS_THREADS, 2)
row_stats_kernel(RowStats rs, RowPtrs src, RowUnits un, int V, ExpScale scale, float gap, DeviceStats *stats, int clear_needs,
                 TreeInfo *tree, const int *parent, int per_seq) {
    // tree != null: no forward pass of the same call has laid the trees out, so the first CTAs do, one per sequence
    constexpr int WARPS = RS_THREADS / 32;
    __shared__ float sh_z[ROW_STAT_PARTS][WARPS];
    __shared__ MaxIdx sh_m[ROW_STAT_PARTS][WARPS];
    __shared__ int par_sh[VIASD_MAX_ROWS_PER_SEQ];
    PDL_TRIGGER();
    PDL_WAIT();
    const int x = blockIdx.x, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (clear_needs && x == 0 && tid == 0) stats->need_slim = stats->need_full = 0;
    if (tree && x < un.B && tid < 32) build_tree(tree + x, parent + (per_seq ? (size_t)x * (un.M - 1) : 0), un.M - 1, stats, par_sh);
    const int id = x < un.whole ? x : un.whole + (x - un.whole) / un.parts;
    const int first = x < un.whole ? 0 : (x - un.whole) % un.parts, last = x < un.whole ? un.parts : first + 1;
    const bool drafter = id < un.B * un.R;
    const int rows = drafter ? un.R : un.M, at = drafter ? id : id - un.B * un.R, kind = drafter ? 0 : 1 + at / (un.B * un.M);
    const int br = drafter ? at : at % (un.B * un.M), b = br / rows, r = br - b * rows;
    const float *row = src.p[kind] + (size_t)br * V;
    // up to three values in front of the first 16-byte boundary (an odd vocabulary), then 16-byte pieces, then the rest
    const int head = min(V, (int)((4 - ((reinterpret_cast<uintptr_t>(row) >> 2) & 3)) & 3)), n4 = (V - head) >> 2, tail = V - head - 4 * n4;
    const float4 *r4 = reinterpret_cast<const float4 *>(row + head);
    const int per = (n4 + un.parts - 1) / un.parts;
#pragma unroll 1
    for (int part = first; part < last; ++part) {
        const int end = min(n4, (part + 1) * per);               // this part's pieces
        RowAcc<WANT_Z> acc;
        acc.init();
        if (part == 0 && tid < head) { const float v[1] = {row[tid]}; acc.add(v, tid, 0, scale, gap); }
        int i0 = part * per + tid;
#pragma unroll 1
        for (; i0 < end; i0 += RS_BATCH * RS_THREADS) {
            float v[4 * RS_BATCH];
            if (i0 + (RS_BATCH - 1) * RS_THREADS < end) {
#pragma unroll
                for (int j = 0; j < RS_BATCH; ++j) {
                    const float4 u = r4[i0 + j * RS_THREADS];
                    v[4 * j] = u.x; v[4 * j + 1] = u.y; v[4 * j + 2] = u.z; v[4 * j + 3] = u.w;
                }
            } else {                                             // the last pieces, all in flight too (two at a time: a part of 8016 pieces took 1.5 times as long)
#pragma unroll
                for (int j = 0; j < RS_BATCH; ++j) {
                    const float4 u = i0 + j * RS_THREADS < end ? r4[i0 + j * RS_THREADS] : make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY);
                    v[4 * j] = u.x; v[4 * j + 1] = u.y; v[4 * j + 2] = u.z; v[4 * j + 3] = u.w;
                }
            }
            acc.add(v, head + 4 * i0, 4 * RS_THREADS, scale, gap);
        }
        if (part == un.parts - 1 && tid < tail) { const float v[1] = {row[V - tail + tid]}; acc.add(v, V - tail + tid, 0, scale, gap); }
        const MaxIdx best = warp_argmax(acc.best);
        float z = 0.f;
        if (WANT_Z) z = warp_sum(acc.ref == -INFINITY ? 0.f : acc.s * exp_scaled(acc.ref - best.v, scale));
        if (lane == 0) { sh_m[part][warp] = best; sh_z[part][warp] = z; }
    }
    __syncthreads();
    if (warp >= last - first) return;
    const int part = first + warp;                               // a warp per part
    const MaxIdx mine = lane < WARPS ? sh_m[part][lane] : no_idx(), best = warp_argmax(mine);
    const float z = WANT_Z ? warp_sum(mine.v == -INFINITY ? 0.f : sh_z[part][lane & (WARPS - 1)] * exp_scaled(mine.v - best.v, scale)) : 0.f;
    if (lane == 0) {
        const size_t o = (((size_t)b * KINDS + kind) * RS_STRIDE + r) * un.parts + part;
        rs.mx[o] = best.v;
        rs.arg[o] = best.i;
        rs.z[o] = z;
    }
}

// ---- accept kernel ----------------------------------------------------------------------------
struct AcceptArgs {
    RowStats rs;
    int parts;                               // of a row's statistics
    const float *judges[KINDS];              // [1..n_judges]: each judge's logits [B, M, V], weakest first, q last
    const float *drafter;                    // [B, R, V]
    float *fold;                             // [B, KINDS, V]: numerators with the rejections folded in, each thread's own
    int vec;                                 // all rows are 16-byte aligned: sweeps take 16 bytes at a time
    int n_judges;
    const int *draft_tok, *prow, *parent;    // [B, N], [N], [N]
    unsigned char *tier;                     // [B, N]
    float *conf;                             // [B, N]: written with the tiers
    const TreeInfo *tree;
    int *n_acc, *path, *out_tok, *n_emit, *corr_src;
    unsigned char *judge;
    DeviceStats *stats;
    int N, R, V;
    int mode, strict_break, emit_bonus;
    ExpScale scale;
    float inv_temp, log1m_alpha, inv_beta;
    float log_acc_rel[KINDS];                // greedy gate per judging tier
    unsigned long long seed, step;
    int do_tier, conf_source;                // do_tier: this launch also assigns the tiers, from the row statistics
    TierCuts cuts;
    // Probe (routed execution policy): the same walk on the slim verifier's logits alone.  It stops where the full
    // verifier's judgment (a tier-2 node, or the bonus token at a leaf) would be needed and raises *need_full; it also
    // raises it when a sequence's backlog (len - len_full) plus this step's tokens would outgrow the replay window.
    // Writes no result.
    int per_seq;                             // prow is [B, N] and every sequence has its own tree
    int probe, replay_rows;
    int *need_full;
    const int *len, *len_full;
};

struct Rejection { int t, v; float sj, sp; };  // judging tier, token, 1 / (beta Z_judge) (negative: the residual vanished), 1 / Z_proposal

struct Walk {                                  // per CTA: everything the walk reads
    int first_child[RS_STRIDE], next_sibling[RS_STRIDE], tok[RS_STRIDE], prow[RS_STRIDE], tier[RS_STRIDE];
    int judged[RS_STRIDE], path[RS_STRIDE];
    float xj[RS_STRIDE], x0[RS_STRIDE];        // logit of the node's token in its judge's row and in its drafter row
    float jv[2][RS_STRIDE], pv[2][RS_STRIDE];  // numerators of the token of each child of this position, after the rejections so far
                                               // (alternate positions: the test that ended the last one may still be reading)
    float mx[KINDS][RS_STRIDE], z[KINDS][RS_STRIDE];
    int arg[KINDS][RS_STRIDE];
    Rejection rej[RS_STRIDE];
    int tier_count[3];
};

// The CTAs of a sequence (a thread-block cluster in sampling mode, else one CTA).  Each sweeps its share of the vocabulary.
struct Team {
    unsigned rank, size;
    float2 (*slots)[MAX_TEAM];     // [2]: what every CTA of the team has sent, by exchange parity
    int phase;
};
__device__ __forceinline__ void team_barrier() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// Every CTA's two values in lanes 0 .. size - 1 of every warp (others: `none`).  A CTA stores its own into all others'
// shared memory and one barrier follows: reading sixteen CTAs' slots one after the other took longer than the sweep.
// (Slots alternate: a CTA sends again into a parity only after the barrier that its readers of it have passed.)
__device__ __forceinline__ float2 team_exchange(float2 v, float2 none, Team &tm) {
    float2 (&slot)[MAX_TEAM] = tm.slots[tm.phase & 1];
    ++tm.phase;
    if (threadIdx.x < tm.size) {
        uint32_t a;
        asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"((uint32_t)__cvta_generic_to_shared(&slot[tm.rank])), "r"(threadIdx.x));
        asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};" ::"r"(a), "f"(v.x), "f"(v.y) : "memory");
    }
    team_barrier();
    const int lane = threadIdx.x & 31;
    return lane < (int)tm.size ? slot[lane] : none;
}

// f(x, y, i) for this CTA's share of a row's indices, N at a time from i on; x, y: the values of two rows there (y: 0 when b
// is null).  Four consecutive values to a thread, whatever the alignment, which only decides how they are loaded: what a thread
// writes at an index it reads again.
template <typename F>
__device__ __forceinline__ void sweep_rows(const float *a, const float *b, int V, bool vec, const Team &tm, F f) {
    const int n4 = V >> 2, per = (n4 + (int)tm.size - 1) / (int)tm.size, lo = (int)tm.rank * per, hi = min(n4, lo + per);
    // eight loads in flight, then a rolled loop over pieces of four values (indexed, so they pass through local memory): a
    // CTA has 16 values per thread and sweep; unrolled, their code came from a cold instruction cache (8 us a sweep), one
    // at a time they are a chain of latencies
#pragma unroll 1
    for (int i0 = lo + threadIdx.x; i0 < hi; i0 += 4 * ACC_THREADS) {
        float4 x[4], y[4];
        if (vec) {
            const float4 *a4 = reinterpret_cast<const float4 *>(a), *b4 = reinterpret_cast<const float4 *>(b);
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int i = min(i0 + j * ACC_THREADS, hi - 1);
                x[j] = a4[i];
                y[j] = b ? b4[i] : make_float4(0.f, 0.f, 0.f, 0.f);
            }
        } else {
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int i = 4 * min(i0 + j * ACC_THREADS, hi - 1);
                x[j] = make_float4(a[i], a[i + 1], a[i + 2], a[i + 3]);
                y[j] = b ? make_float4(b[i], b[i + 1], b[i + 2], b[i + 3]) : make_float4(0.f, 0.f, 0.f, 0.f);
            }
        }
        const int n = min(4, (hi - i0 + ACC_THREADS - 1) / ACC_THREADS);
#pragma unroll 1
        for (int j = 0; j < n; ++j) {
            const float u[4] = {x[j].x, x[j].y, x[j].z, x[j].w}, v[4] = {y[j].x, y[j].y, y[j].z, y[j].w};
            f(u, v, 4 * (i0 + j * ACC_THREADS));
        }
    }
    const int i = 4 * n4 + (int)threadIdx.x;                      // the last few of a vocabulary that is no multiple of four
    if (tm.rank == 0 && i < V) {
        const float u[1] = {a[i]}, v[1] = {b ? b[i] : 0.f};
        f(u, v, i);
    }
}

// Numerators at tokens i, i + 1, ... after the rejections so far: the judge of tier t (starting from jt) and the proposal (pr).
// Eq. A.3 round by round: the rejecting judge becomes its residual against the proposal (kept as it is if the residual
// vanishes); the rejected token leaves the proposal.
template <int N>
__device__ __forceinline__ void replay(const Rejection *rej, int n, int i, int t, float (&jt)[N], float (&pr)[N]) {
    for (int k = 0; k < n; ++k) {
        const Rejection r = rej[k];
        if (r.t == t && r.sj >= 0.f) {
#pragma unroll
            for (int e = 0; e < N; ++e) jt[e] = fmaxf(0.f, jt[e] * r.sj - pr[e] * r.sp);
        }
#pragma unroll
        for (int e = 0; e < N; ++e) pr[e] = i + e == r.v ? 0.f : pr[e];
    }
}

__global__ void __launch_bounds__(ACC_THREADS, 2)
accept_kernel(AcceptArgs a) {
    __shared__ Walk w;
    __shared__ MaxIdx shm[ACC_WARPS];
    __shared__ float sh[4][ACC_WARPS];
    __shared__ float2 slots[2][MAX_TEAM];
    Team tm;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(tm.rank));
    asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(tm.size));
    tm.slots = slots; tm.phase = 0;
    PDL_TRIGGER();
    PDL_WAIT();
    const int tid = threadIdx.x;
    const int b = blockIdx.x / tm.size, N = a.N, M = N + 1, V = a.V;
    const bool sampling = a.mode == 1, writes = tm.rank == 0 && !a.probe;     // writes: this CTA stores the results
    const int J = a.n_judges;                                 // tier J is the full verifier's
    const unsigned long long k_acc = stream_key(a.seed, a.step, b, 0), k_gum = stream_key(a.seed, a.step, b, 1);

    // ---- everything the walk reads, at once
    if (tid < 3) w.tier_count[tid] = 0;
    const size_t st0 = (size_t)b * KINDS * RS_STRIDE;
    for (int e = tid; e < (J + 1) * RS_STRIDE; e += ACC_THREADS) {
        const int k = e / RS_STRIDE, r = e - k * RS_STRIDE;
        if (r >= (k == 0 ? a.R : M)) continue;
        MaxIdx best = no_idx(), m[ROW_STAT_PARTS];
        float z[ROW_STAT_PARTS], sum = 0.f;
#pragma unroll
        for (int i = 0; i < ROW_STAT_PARTS; ++i) {
            const size_t o = (st0 + e) * a.parts + min(i, a.parts - 1);
            m[i].v = a.rs.mx[o]; m[i].i = a.rs.arg[o]; z[i] = a.rs.z[o];
        }
#pragma unroll
        for (int i = 0; i < ROW_STAT_PARTS; ++i) if (i < a.parts) best = better(best, m[i]);
#pragma unroll
        for (int i = 0; i < ROW_STAT_PARTS; ++i) if (i < a.parts && m[i].v != -INFINITY) sum += z[i] * exp_scaled(m[i].v - best.v, a.scale);
        w.mx[k][r] = best.v; w.z[k][r] = sum; w.arg[k][r] = best.i == 0x7fffffff ? 0 : best.i;
    }
    for (int r = tid; r < M; r += ACC_THREADS) w.first_child[r] = a.tree[b].first_child[r];
    __syncthreads();
    for (int n = tid; n < N; n += ACC_THREADS) {
        const int par = a.parent[(a.per_seq ? (size_t)b * N : 0) + n], pr = a.prow[(a.per_seq ? (size_t)b * N : 0) + n];
        const int v = min(max(a.draft_tok[b * N + n], 0), V - 1);
        w.next_sibling[n] = a.tree[b].next_sibling[n];
        w.tok[n] = v;
        w.judged[n] = 0;
        const bool pr_ok = pr >= 0 && pr < a.R, used = par != -2;      // -2: unused node of this sequence's tree
        w.prow[n] = pr_ok ? pr : 0;
        if (used && sampling && !pr_ok) a.stats->device_status = VIASD_EDEVICE;
        const float x0 = a.drafter && used ? a.drafter[((size_t)b * a.R + w.prow[n]) * V + v] : 0.f;
        w.x0[n] = x0;
        int t;
        if (a.do_tier) {
            t = 0;
            float d = 0.f;
            const int g = a.conf_source == 0 ? pr : par + 1;
            if (used) {
                // no such gate row: an error, and the strictest tier, as in the tier kernel
                d = -INFINITY;
                if (a.conf_source ? g < 0 || g >= M : !pr_ok) a.stats->device_status = VIASD_EDEVICE;
                else d = a.conf_source == 0 ? x0 - w.mx[0][g] : a.judges[1][((size_t)b * M + g) * V + v] - w.mx[1][g];
                while (t < a.cuts.n && d < a.cuts.log_tau[t]) ++t;      // thresholds descend: the first one d reaches names the tier
                atomicAdd(&w.tier_count[t == 0 ? 0 : (t == a.cuts.n ? 2 : 1)], 1);       // accepted / some slim verifier / q
            }
            if (writes) { a.tier[b * N + n] = (unsigned char)t; a.conf[b * N + n] = d; }
        } else {
            t = a.tier[b * N + n];
        }
        t = min(t, J);
        w.tier[n] = t;
        w.xj[n] = t > 0 && par >= -1 && par < N && a.judges[t] ? a.judges[t][((size_t)b * M + par + 1) * V + v] : 0.f;
    }
    if (tm.size > 1) team_barrier(); else __syncthreads();    // (every CTA of the cluster runs: its slots may be written)
    if (a.do_tier && writes && tid < 3) {
        if (w.tier_count[tid]) {
            atomicAdd(&a.stats->tier_count[tid], (unsigned long long)w.tier_count[tid]);
            if (tid == 1) a.stats->need_slim = 1;
            if (tid == 2) a.stats->need_full = 1;
        }
        if (b == 0 && tid == 0) atomicAdd(&a.stats->steps, 1ull);
    }

    // What rejections at this position have been folded into the arrays of a.fold: the first `n_fold`, those of the judges in
    // `folded` (bit t; bit 0: the proposal's array is in use).
    int n_fold = 0;
    unsigned folded = 0;
    auto fold_row = [&](int k) { return a.fold + ((size_t)b * KINDS + k) * V; };
    auto judge_row = [&](int t, int cur) -> const float * { return folded >> t & 1 ? fold_row(t) : a.judges[t] + ((size_t)b * M + cur) * V; };
    auto proposal_row = [&](const float *r0) -> const float * { return folded & 1 ? fold_row(0) : r0; };
    // the judge's and the proposal's numerators from i on after n_rej rejections, from what judge_row and proposal_row hold there
    auto numerators = [&](int t, int i, const auto &xt, float mxt, const auto &x0, float mx0, int n_rej, auto &jt, auto &pr) {
        constexpr int N = sizeof(jt) / sizeof(float);
        const bool ft = folded >> t & 1, f0 = folded & 1;
#pragma unroll
        for (int e = 0; e < N; ++e) {
            jt[e] = ft ? xt[e] : exp_scaled(xt[e] - mxt, a.scale);
            pr[e] = f0 ? x0[e] : exp_scaled(x0[e] - mx0, a.scale);
        }
        replay(w.rej + n_fold, n_rej - n_fold, i, t, jt, pr);
    };

    // argmax_v (log weight(v) - log(-log u_v)): a draw from the judge of tier t at block row `cur` after n_rej rejections
    auto draw = [&](int t, int cur, const float *r0, float mx0, int n_rej) -> int {
        const float *rt = a.judges[t] + ((size_t)b * M + cur) * V;
        const float mxt = w.mx[t][cur];
        MaxIdx best = no_idx();
        sweep_rows(n_rej ? judge_row(t, cur) : rt, n_rej ? proposal_row(r0) : nullptr, V, a.vec, tm, [&](const auto &xt, const auto &x0, int i) {
            constexpr int N = sizeof(xt) / sizeof(float);
            float jt[N], pr[N];
            if (n_rej) numerators(t, i, xt, mxt, x0, mx0, n_rej, jt, pr);
#pragma unroll
            for (int e = 0; e < N; ++e) {
                // log weight; through the residuals once there are any
                const float lw = n_rej ? logf(jt[e]) : (xt[e] - mxt) * a.inv_temp;
                const float u = unit_f32(k_gum, ((unsigned long long)cur << 32) + (unsigned long long)(i + e));
                MaxIdx c; c.v = !n_rej || jt[e] > 0.f ? lw - logf(-logf(u)) : -INFINITY; c.i = i + e;
                best = better(best, c);
            }
        });
        best = block_argmax(best, shm);
        if (tm.size > 1) {
            const float2 got = team_exchange(make_float2(best.v, __int_as_float(best.i)), make_float2(-INFINITY, __int_as_float(0x7fffffff)), tm);
            MaxIdx c; c.v = got.x; c.i = __float_as_int(got.y);
            best = warp_argmax(c);
        }
        return best.i == 0x7fffffff ? 0 : best.i;
    };

    int cur = 0, n_acc = 0, corr = -1, corr_src = 0, parity = 0, draw_t = 0, n_rej = 0, pos = 0;
    const float *r0 = nullptr;                                   // the drafter row of this position and its maximum
    float mx0 = 0.f;
    bool needs_q = false;
    while (true) {
        int c = w.first_child[cur];
        n_rej = n_fold = 0;
        folded = 0;
        r0 = nullptr;
        if (c < 0) {                                             // leaf: whole path accepted
            if (a.emit_bonus && a.probe) { needs_q = true; break; }
            if (a.emit_bonus) {
                corr_src = draw_t = J;
            }
            break;
        }
        // the distributions of this position: the proposal (drafter row) and the judges; Z: denominators after n_rej rejections
        float Z[KINDS];
#pragma unroll
        for (int k = 0; k < KINDS; ++k) Z[k] = k >= 1 && k <= J && a.judges[k] ? w.z[k][cur] : 0.f;
        int failed = 0, taken = -1, taken_tier = 0, row0 = -1;
        for (; c >= 0; c = w.next_sibling[c]) {
            const int t = w.tier[c], v = w.tok[c];
            if (t == 0) {
                taken = c; taken_tier = 0;
                if (tid == 0) w.judged[c] = 1;
                break;
            }
            if (t == J && a.probe) { needs_q = true; break; }     // from here on the walk depends on q
            const float mxt = w.mx[t][cur];
            bool pass;
            float Zt = 0.f;
            if (!sampling) {
                pass = (w.xj[c] - mxt) >= a.log_acc_rel[t];
            } else {
                if (!r0) {
                    row0 = w.prow[c];
                    r0 = a.drafter + ((size_t)b * a.R + row0) * V;
                    mx0 = w.mx[0][row0];
                    Z[0] = w.z[0][row0];
                    pos ^= 1;
                    for (int n = tid; n < N; n += ACC_THREADS) {      // (of the children of this row; the others' are not used)
                        // a child that names another drafter row than its elder sibling is still tested against that sibling's
                        const float x0 = w.prow[n] == row0 ? w.x0[n] : r0[w.tok[n]];
                        w.jv[pos][n] = exp_scaled(w.xj[n] - w.mx[w.tier[n]][cur], a.scale);
                        w.pv[pos][n] = exp_scaled(x0 - mx0, a.scale);
                    }
                    __syncthreads();
                }
#pragma unroll
                for (int k = 1; k < KINDS; ++k) if (k == t) Zt = Z[k];
                const float u = unit_f32(k_acc, (unsigned long long)c);
                const float lp = logf(w.pv[pos][c] / Z[0]);
                const float lj = logf(w.jv[pos][c] / Zt);
                pass = (logf(u) + a.log1m_alpha + lp) < lj;       // u < j(v) / ((1 - alpha) p(v)), Eq. A.2
            }
            if (pass) {
                taken = c; taken_tier = t;
                if (tid == 0) w.judged[c] = 1 | (t << 4);
                break;
            }
            if (tid == 0) w.judged[c] = 2 | (t << 4);
            failed = max(failed, t);
            if (sampling) {
                // the masses of the judge's residual and of the proposal without the rejected token
                const float sj = a.inv_beta / Zt, sp = 1.f / Z[0];
                if (n_rej - n_fold == FOLD) {
                    // the judges that have rejected, the proposal with the last of them (all start from its old values)
                    unsigned write = 0;
                    for (int k = 0; k < n_rej; ++k) write |= 1u << w.rej[k].t;
                    for (int k = 1; k <= J; ++k) {
                        if (!(write >> k & 1)) continue;
                        const bool last = write >> (k + 1) == 0;
                        float *to = fold_row(k), *to0 = fold_row(0);
                        const float mxk = w.mx[k][cur];
                        sweep_rows(judge_row(k, cur), proposal_row(r0), V, a.vec, tm, [&](const auto &xt, const auto &x0, int i) {
                            constexpr int N = sizeof(xt) / sizeof(float);
                            float jt[N], pr[N];
                            numerators(k, i, xt, mxk, x0, mx0, n_rej, jt, pr);
#pragma unroll
                            for (int e = 0; e < N; ++e) { to[i + e] = jt[e]; if (last) to0[i + e] = pr[e]; }
                        });
                    }
                    folded |= write | 1u;
                    n_fold = n_rej;
                }
                float s = 0.f, z = 0.f;
                sweep_rows(judge_row(t, cur), proposal_row(r0), V, a.vec, tm, [&](const auto &xt, const auto &x0, int i) {
                    constexpr int N = sizeof(xt) / sizeof(float);
                    float jt[N], pr[N];
                    numerators(t, i, xt, mxt, x0, mx0, n_rej, jt, pr);
#pragma unroll
                    for (int e = 0; e < N; ++e) {
                        s += fmaxf(0.f, jt[e] * sj - pr[e] * sp);
                        z += i + e == v ? 0.f : pr[e];
                    }
                });
                s = block_sum(s, sh[2 * parity]);
                z = block_sum(z, sh[2 * parity + 1]);
                parity ^= 1;
                if (tm.size > 1) {
                    const float2 got = team_exchange(make_float2(s, z), make_float2(0.f, 0.f), tm);
                    s = warp_sum(got.x);
                    z = warp_sum(got.y);
                }
                const Rejection r{t, v, s > 0.f ? sj : -1.f, sp};
                if (tid == 0) w.rej[n_rej] = r;
                ++n_rej;
                for (int n = tid; n < N; n += ACC_THREADS) {
                    float jt[1] = {w.jv[pos][n]}, pr[1] = {w.pv[pos][n]};
                    replay(&r, 1, w.tok[n], w.tier[n], jt, pr);
                    w.jv[pos][n] = jt[0];
                    w.pv[pos][n] = pr[0];
                }
#pragma unroll
                for (int k = 1; k < KINDS; ++k) if (k == t && s > 0.f) Z[k] = s;
                if (z > 0.f) Z[0] = z;
                __syncthreads();
            }
        }
        if (needs_q) break;
        if (taken >= 0) {
            if (a.strict_break && taken_tier >= 1 && taken_tier < J) {
                corr = w.tok[taken];
                corr_src = taken_tier;
                break;
            }
            if (tid == 0) w.path[n_acc] = taken;
            ++n_acc;
            cur = taken + 1;
            continue;                                             // (rej is written again only behind a barrier of the next sweep)
        }
        corr_src = draw_t = failed;
        break;
    }
    if (draw_t > 0) corr = sampling ? draw(draw_t, cur, r0, mx0, n_rej) : w.arg[draw_t][cur];
    __syncthreads();
    if (tm.rank != 0) return;                                     // (nothing is sent to this CTA any more)
    if (a.probe) {
        if (tid == 0) {
            // tokens this step emits if q is not asked: the accepted nodes and the replacement (or nothing at a leaf)
            const int ne = n_acc + (corr >= 0 ? 1 : 0);
            const bool room = a.len[b] - a.len_full[b] + ne <= a.replay_rows && a.len[b] >= a.replay_rows;
            if (needs_q || !room) atomicExch(a.need_full, 1);
        }
        return;
    }
    const int ne = n_acc + (corr >= 0 ? 1 : 0);
    for (int n = tid; n < N; n += ACC_THREADS) a.judge[b * N + n] = (unsigned char)w.judged[n];
    for (int j = tid; j < n_acc; j += ACC_THREADS) {
        a.path[b * N + j] = w.path[j];
        a.out_tok[b * (N + 1) + j] = w.tok[w.path[j]];
    }
    if (tid == 0) {
        if (corr >= 0) a.out_tok[b * (N + 1) + n_acc] = corr;
        a.n_acc[b] = n_acc;
        a.n_emit[b] = ne;
        a.corr_src[b] = corr_src;
        atomicAdd(&a.stats->emitted, (unsigned long long)ne);
        atomicAdd(&a.stats->accepted, (unsigned long long)n_acc);
    }
}

TierCuts tier_cuts(const JudgeSet &js) {
    TierCuts c;
    c.n = js.n;
    for (int k = 0; k < MAXJ; ++k) c.log_tau[k] = k < js.n ? js.log_tau[k] : 0.f;
    return c;
}

}  // namespace

int launch_tier(const viasd_model *m, const viasd_draft *d, const viasd_params *p, const JudgeSet &js, viasd_result *r,
                cudaStream_t st) {
    const int M = d->n_nodes + 1;
    if (js.n < 1 || js.n > MAXJ) return VIASD_EINVAL;
    CUDA_TRY(cudaMemsetAsync(&m->ws.stats->need_slim, 0, 2 * sizeof(int), st));
    const float *gate = p->conf_source == 0 ? d->drafter_logits : js.logits[0];   // Alg. 2 gates with the slim(mest) verifier
    const int rows = p->conf_source == 0 ? d->n_prows : M;
    if (!gate) return VIASD_EINVAL;
    const TierCuts cuts = tier_cuts(js);
    // (a CTA per gate row: with few rows the launch is bound by the loads each CTA has in flight, hence 1024 threads)
    tier_kernel<<<dim3(rows, d->batch), 1024, 0, st>>>(r->tier, r->conf, m->ws.stats, gate, d->draft_tok, d->prow,
        d->parent, d->per_sequence, p->conf_source, rows, d->n_nodes, m->cfg.vocab, cuts);
    LAUNCH_CHECK();
    return VIASD_OK;
}

// A cluster of 16 CTAs (beyond the portable 8) where the device takes it: asked once per device.
static bool accept_team16_ok() {
    static int state[64];                    // 0 unknown, 1 yes, -1 no
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return false;
    if (state[dev] == 0) {
        state[dev] = -1;
        if (cudaFuncSetAttribute(accept_kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess) {
            cudaLaunchConfig_t cfg;
            memset(&cfg, 0, sizeof(cfg));
            cfg.gridDim = dim3(16); cfg.blockDim = dim3(ACC_THREADS);
            cudaLaunchAttribute attr[1];
            attr[0].id = cudaLaunchAttributeClusterDimension;
            attr[0].val.clusterDim.x = 16; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
            cfg.attrs = attr; cfg.numAttrs = 1;
            int n = 0;
            if (cudaOccupancyMaxActiveClusters(&n, accept_kernel, &cfg) == cudaSuccess && n >= 1) state[dev] = 1;
        }
        (void)cudaGetLastError();
    }
    return state[dev] == 1;
}

int launch_accept(const viasd_model *m, const viasd_draft *d, const viasd_params *p, const JudgeSet &js, viasd_result *r,
                  bool tree_ready, bool do_tier, cudaStream_t st, const AcceptProbe *probe) {
    if (js.n < 1 || js.n > MAXJ) return VIASD_EINVAL;
    if (d->n_prows > RS_STRIDE) return VIASD_EINVAL;
    AcceptArgs a;
    {
        float *base = m->ws.accept_scratch;
        const size_t n = (size_t)m->cfg.max_batch * KINDS * RS_STRIDE * ROW_STAT_PARTS;
        a.parts = row_parts(m->cfg.vocab);
        a.rs.mx = base; a.rs.arg = reinterpret_cast<int *>(base + n); a.rs.z = base + 2 * n;
        RowPtrs src;
        src.p[0] = p->mode == 1 || (do_tier && p->conf_source == 0) ? d->drafter_logits : nullptr;
        int judges = 0;
        for (int k = 1; k < KINDS; ++k) src.p[k] = nullptr;
        for (int k = 1; k <= js.n; ++k) if (js.logits[k - 1]) { src.p[k] = js.logits[k - 1]; judges = k; }   // (those of a probe come without q)
        RowUnits un{d->batch, src.p[0] ? d->n_prows : 0, d->n_nodes + 1, 0, a.parts};
        const int rows = un.B * (un.R + un.M * judges), turn = 2 * m->sm_count;
        un.whole = a.parts > 1 ? rows / turn * turn : rows;
        auto kernel = p->mode == 1 ? row_stats_kernel<true> : row_stats_kernel<false>;
        const float temperature = p->mode == 1 ? p->temperature : 1.f;
        CUDA_TRY(launch_chained(kernel, un.whole + (rows - un.whole) * a.parts, RS_THREADS, st, a.rs, src, un, m->cfg.vocab,
            exp_scale(temperature), RS_GAP * temperature, m->ws.stats, do_tier ? 1 : 0, tree_ready ? nullptr : m->ws.tree, d->parent, d->per_sequence));
        LAUNCH_CHECK();
    }
    a.judges[0] = nullptr;
    for (int k = 1; k < KINDS; ++k) a.judges[k] = k <= js.n ? js.logits[k - 1] : nullptr;
    a.n_judges = js.n;
    a.drafter = d->drafter_logits;
    a.fold = m->ws.accept_fold;
    uintptr_t rows16 = (uintptr_t)a.drafter;
    for (int k = 1; k <= js.n; ++k) rows16 |= (uintptr_t)a.judges[k];
    a.vec = m->cfg.vocab % 4 == 0 && (rows16 & 15) == 0;
    a.draft_tok = d->draft_tok; a.prow = d->prow; a.parent = d->parent; a.tier = r->tier; a.conf = r->conf; a.tree = m->ws.tree;
    a.do_tier = do_tier ? 1 : 0; a.conf_source = p->conf_source;
    a.cuts = tier_cuts(js);
    a.n_acc = r->n_acc; a.path = r->path; a.out_tok = r->out_tok; a.n_emit = r->n_emit; a.corr_src = r->corr_src;
    a.judge = r->judge; a.stats = m->ws.stats;
    a.N = d->n_nodes; a.R = d->n_prows; a.V = m->cfg.vocab;
    a.mode = p->mode; a.strict_break = p->strict_break; a.emit_bonus = p->emit_bonus;
    a.inv_temp = 1.0f / p->temperature;
    a.scale = exp_scale(p->mode == 1 ? p->temperature : 1.f);
    a.log1m_alpha = log1pf(-p->alpha);
    a.inv_beta = 1.0f / p->beta;
    // greedy gates: log_acc_rel[1] for every slim verifier, log_acc_rel[2] for q
    for (int k = 0; k < KINDS; ++k) a.log_acc_rel[k] = k == 0 ? p->log_acc_rel[0] : k < js.n ? p->log_acc_rel[1] : p->log_acc_rel[2];
    a.seed = p->seed; a.step = p->step;
    a.per_seq = d->per_sequence;
    a.probe = probe ? 1 : 0;
    a.replay_rows = probe ? probe->replay_rows : 0;
    a.need_full = probe ? probe->need_full : nullptr;
    a.len = probe ? probe->len : nullptr;
    a.len_full = probe ? probe->len_full : nullptr;
    // sampling over a large vocabulary: a cluster of CTAs per sequence shares every sweep of the vocabulary
    int team = (p->mode == 1 && m->cfg.vocab >= 16384) ? ACC_TEAM : 1;
    if (team == ACC_TEAM && m->cfg.vocab >= 65536 && accept_team16_ok()) team = 16;     // every sweep of the vocabulary is shared
    { const int t = m->opt.accept_team; if (t == 1 || t == 2 || t == 4 || t == 8) team = t; }
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attr[2];
    pdl_config(cfg, attr, dim3(d->batch * team), dim3(ACC_THREADS), 0, st);
    if (team > 1) {
        attr[cfg.numAttrs].id = cudaLaunchAttributeClusterDimension;
        attr[cfg.numAttrs].val.clusterDim.x = team; attr[cfg.numAttrs].val.clusterDim.y = 1; attr[cfg.numAttrs].val.clusterDim.z = 1;
        ++cfg.numAttrs;
    }
    CUDA_TRY(cudaLaunchKernelEx(&cfg, accept_kernel, a));
    LAUNCH_CHECK();
    return VIASD_OK;
}
