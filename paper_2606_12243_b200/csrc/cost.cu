// KL-style verification cost of a judge against a proposal, per logits row (Eq. 11; smooth margin of App. F).
//
//   lp = log softmax(proposal / T), lq = log softmax(judge / T)
//   z1 = log(1 - alpha) + lp - lq,  z2 = log(beta) + lp - lq
//   R  = sum_v exp(lp) phi(z1) + sum_v exp(lq) phi(z2),   phi = max(0, .) or tau log(1 + exp(. / tau))
//
// HBM-bound: 2 rows of V floats in, one float out.  Two sweeps: the first finds each row's maximum and denominator
// together (a running reference per thread, moved only when it is exceeded by e^20), the second the sums.  A row pair is
// 1.2 MB at a vocabulary of 152064: with a CTA per row six hundred of them are in flight, nothing is left in L2 for the
// second sweep, and every sweep comes from HBM.  So a cluster of CTAs shares a row pair, exchanging its results through
// distributed shared memory in rank order - reproducible, and the same for a row whatever rows come with it - and works
// through the rows one after the other (a launch of one cluster per row spends longer starting clusters than reading).
// The block cost of Eq. 10 is the sum of the rows, added up by one thread in row order.
#include "common.cuh"
#include <string.h>

namespace {

constexpr int COST_THREADS = 512, COST_WARPS = COST_THREADS / 32, MAX_TEAM = 4;
constexpr int BATCH = 4;                        // 16-byte loads of each row in flight per thread
constexpr float REF_GAP = 20.f;                 // a thread's reference may be exceeded by this much (in exponent units)

__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ void push_f32(float *own, unsigned rank, float v) {       // into the same place of CTA `rank`
    uint32_t a;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"((uint32_t)__cvta_generic_to_shared(own)), "r"(rank));
    asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(a), "f"(v) : "memory");
}
struct Share { unsigned rank, size; };          // this CTA's place among the CTAs of its row
__device__ __forceinline__ void row_barrier(const Share &s) {
    if (s.size > 1) { cluster_arrive(); cluster_wait(); } else __syncthreads();
}
__device__ __forceinline__ Share row_share() {
    Share s;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(s.rank));
    asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(s.size));
    return s;
}

struct MaxOp {
    static __device__ __forceinline__ float none() { return -INFINITY; }
    __device__ __forceinline__ float operator()(float a, float b) const { return fmaxf(a, b); }
};
struct SumOp {
    static __device__ __forceinline__ float none() { return 0.f; }
    __device__ __forceinline__ float operator()(float a, float b) const { return a + b; }
};
template <typename Op>
__device__ __forceinline__ float warp_all(float v, Op op) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = op(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}
// K values per thread -> the CTA's combined values, in every thread.  sh: a buffer of this call's own
template <int K, typename Op>
__device__ __forceinline__ void block_combine(float (&v)[K], float (*sh)[COST_WARPS], Op op) {
#pragma unroll
    for (int k = 0; k < K; ++k) {
        v[k] = warp_all(v[k], op);
        if ((threadIdx.x & 31) == 0) sh[k][threadIdx.x >> 5] = v[k];
    }
    __syncthreads();
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int k = 0; k < K; ++k) v[k] = warp_all(lane < COST_WARPS ? sh[k][lane] : Op::none(), op);
}

// This CTA's share of a pair of rows: f(Count<n>, x, y) for batches of n values of either row.  16-byte loads behind a head
// of up to three values where the two rows are aligned alike (an odd vocabulary shifts both).
template <int N> struct Count { static constexpr int n = N; };
template <typename F>
__device__ __forceinline__ void sweep_pair(const float *a, const float *b, int V, const Share &sh, F f) {
    float x[4 * BATCH], y[4 * BATCH];
    if (((reinterpret_cast<uintptr_t>(a) ^ reinterpret_cast<uintptr_t>(b)) & 15) == 0) {
        const int head = min(V, (int)((4 - ((reinterpret_cast<uintptr_t>(a) >> 2) & 3)) & 3)), n4 = (V - head) >> 2;
        const int tail = V - head - 4 * n4, per = (n4 + (int)sh.size - 1) / (int)sh.size;
        const int lo = min(n4, (int)sh.rank * per), hi = min(n4, lo + per);
        const float4 *a4 = reinterpret_cast<const float4 *>(a + head), *b4 = reinterpret_cast<const float4 *>(b + head);
        int i0 = lo + threadIdx.x;
#pragma unroll 1
        for (; i0 + (BATCH - 1) * COST_THREADS < hi; i0 += BATCH * COST_THREADS) {
#pragma unroll
            for (int j = 0; j < BATCH; ++j) {
                const float4 u = a4[i0 + j * COST_THREADS], w = b4[i0 + j * COST_THREADS];
                x[4 * j] = u.x; x[4 * j + 1] = u.y; x[4 * j + 2] = u.z; x[4 * j + 3] = u.w;
                y[4 * j] = w.x; y[4 * j + 1] = w.y; y[4 * j + 2] = w.z; y[4 * j + 3] = w.w;
            }
            f(Count<4 * BATCH>(), x, y);
        }
#pragma unroll 1
        for (; i0 < hi; i0 += COST_THREADS) {
            const float4 u = a4[i0], w = b4[i0];
            x[0] = u.x; x[1] = u.y; x[2] = u.z; x[3] = u.w;
            y[0] = w.x; y[1] = w.y; y[2] = w.z; y[3] = w.w;
            f(Count<4>(), x, y);
        }
        // the few values outside the 16-byte pieces
        const int e = (int)threadIdx.x;
        if (sh.rank == 0 && e < head + tail) {
            x[0] = e < head ? a[e] : a[V - tail + e - head];
            y[0] = e < head ? b[e] : b[V - tail + e - head];
            f(Count<1>(), x, y);
        }
    } else {
        for (int i = sh.rank * COST_THREADS + threadIdx.x; i < V; i += sh.size * COST_THREADS) { x[0] = a[i]; y[0] = b[i]; f(Count<1>(), x, y); }
    }
}

// Running maximum and denominator of one row, per thread: sum of exp((x - ref) / T).
struct Denom {
    float ref, lim, mx, s;
    __device__ __forceinline__ void init() { ref = lim = mx = -INFINITY; s = 0.f; }
    template <int N>
    __device__ __forceinline__ void add(Count<N>, const float (&x)[4 * BATCH], ExpScale scale, float gap) {
        float bm = x[0];
#pragma unroll
        for (int e = 1; e < N; ++e) bm = fmaxf(bm, x[e]);
        if (bm > lim) {                             // the first values, or far above the reference: rare
            s *= exp_scaled(ref - bm, scale);
            ref = bm;
            lim = bm + gap;
        }
        mx = fmaxf(mx, bm);
        const float r = ref == -INFINITY ? 0.f : ref;
#pragma unroll
        for (int e = 0; e < N; ++e) s += exp_scaled(x[e] - r, scale);
    }
    __device__ __forceinline__ float at(float m, ExpScale scale) const { return ref == -INFINITY ? 0.f : s * exp_scaled(ref - m, scale); }
};

__device__ __forceinline__ float phi(float z, int smooth, float tau, float inv_tau) {
    if (!smooth) return fmaxf(z, 0.f);
    const float t = z * inv_tau;                              // tau log(1 + e^t), without overflow for large t
    return tau * (fmaxf(t, 0.f) + log1pf(expf(-fabsf(t))));
}

// A cluster works through the rows blockIdx.x / team, + the number of clusters, ...  One barrier per row: the CTAs' maxima
// and denominators go to every CTA of the row before it (double-buffered by row), a row's cost to CTA 0, which adds it up
// after the next row's barrier.
template <int SMOOTH>
__global__ void __launch_bounds__(COST_THREADS, 2)
kl_cost_kernel(float *__restrict__ cost_rows, const float *__restrict__ judge, const float *__restrict__ proposal, int rows, int V,
               ExpScale scale, float inv_temp, float log1m_alpha, float log_beta, float tau) {
    __shared__ float sh_mx[2][COST_WARPS], sh_s[2][COST_WARPS], sh_c[1][COST_WARPS], part[2][4][MAX_TEAM], fin[2][MAX_TEAM];
    const Share me = row_share();
    const int lane = threadIdx.x & 31, clusters = gridDim.x / me.size;
    const bool on = lane < (int)me.size;
    const float gap = REF_GAP / inv_temp, inv_tau = SMOOTH ? 1.f / tau : 0.f;
    row_barrier(me);                                          // every CTA of the cluster runs: its shared memory may be written
    int buf = 0, before = -1;
    auto finish_before = [&]() {                              // the row before this one, by one warp of CTA 0
        if (before >= 0 && me.rank == 0 && threadIdx.x < 32) {
            const float r = warp_all(on ? fin[buf ^ 1][lane] : 0.f, SumOp());
            if (lane == 0) cost_rows[before] = r;
        }
    };
    for (int row = blockIdx.x / me.size; row < rows; before = row, row += clusters, buf ^= 1) {
        const float *jq = judge + (size_t)row * V, *pp = proposal + (size_t)row * V;
        Denom dq, dp;
        dq.init(); dp.init();
        sweep_pair(jq, pp, V, me, [&](auto n, const float (&q)[4 * BATCH], const float (&p)[4 * BATCH]) { dq.add(n, q, scale, gap); dp.add(n, p, scale, gap); });
        float m[2] = {dq.mx, dp.mx};
        block_combine<2>(m, sh_mx, MaxOp());                  // this CTA's maxima (-inf if it has no share) ...
        float z[2] = {dq.at(m[0], scale), dp.at(m[1], scale)};
        block_combine<2>(z, sh_s, SumOp());                   // ... and denominators relative to them
        if (threadIdx.x < me.size) {
            push_f32(&part[buf][0][me.rank], threadIdx.x, m[0]); push_f32(&part[buf][1][me.rank], threadIdx.x, m[1]);
            push_f32(&part[buf][2][me.rank], threadIdx.x, z[0]); push_f32(&part[buf][3][me.rank], threadIdx.x, z[1]);
        }
        row_barrier(me);
        finish_before();
        const float a = on ? part[buf][0][lane] : -INFINITY, b = on ? part[buf][1][lane] : -INFINITY;
        const float mq = warp_all(a, MaxOp()), mp = warp_all(b, MaxOp());
        const float zq = warp_all(a == -INFINITY ? 0.f : part[buf][2][lane] * exp_scaled(a - mq, scale), SumOp());
        const float zp = warp_all(b == -INFINITY ? 0.f : part[buf][3][lane] * exp_scaled(b - mp, scale), SumOp());
        // lp - lq as (p - q) / T plus a constant of the row that is worked out from small numbers, the weights' denominators
        // outside the sums: log q and log p themselves are of the order of ten, and their last bit was the cost's error
        // (vocabulary 152064: 7.4e-7 rms, now 2.8e-7)
        const float shift = fmaf(mq - mp, inv_temp, logf(zq / zp)), sh1 = log1m_alpha + shift, sh2 = log_beta + shift;
        float acc_p = 0.f, acc_q = 0.f;
        sweep_pair(jq, pp, V, me, [&](auto n, const float (&q)[4 * BATCH], const float (&p)[4 * BATCH]) {
#pragma unroll
            for (int e = 0; e < decltype(n)::n; ++e) {
                const float d = p[e] - q[e];
                acc_p += exp_scaled(p[e] - mp, scale) * phi(fmaf(d, inv_temp, sh1), SMOOTH, tau, inv_tau);
                acc_q += exp_scaled(q[e] - mq, scale) * phi(fmaf(d, inv_temp, sh2), SMOOTH, tau, inv_tau);
            }
        });
        float acc[1] = {acc_p / zp + acc_q / zq};
        block_combine<1>(acc, sh_c, SumOp());
        if (threadIdx.x == 0) push_f32(&fin[buf][me.rank], 0, acc[0]);
    }
    row_barrier(me);
    if (me.rank != 0) return;
    finish_before();
}

// Region masses (Eq. B.8-B.10): per row, the mass of p = softmax(proposal / T) on the tokens the gating row places in
// region A (d >= log tau_hi), B (log tau_lo <= d < log tau_hi) and C (below), d = l[u] - max l in fp32 exactly as the
// tier kernel decides a drafted token.  Built like the cost kernel: maxima, then the sums.  (scale2 = log2(e) / T: the masses
// are shares of one sum, in which a scale that is slightly off cancels.)
__global__ void __launch_bounds__(COST_THREADS, 2)
region_mass_kernel(float *__restrict__ mass, const float *__restrict__ gate, const float *__restrict__ proposal, int rows, int V,
                   float scale2, float log_tau_hi, float log_tau_lo) {
    __shared__ float sh_mx[2][COST_WARPS], sh_s[3][COST_WARPS], part[2][2][MAX_TEAM], fin[2][3][MAX_TEAM];
    const Share me = row_share();
    const int lane = threadIdx.x & 31, clusters = gridDim.x / me.size;
    const bool on = lane < (int)me.size;
    row_barrier(me);
    int buf = 0, before = -1;
    auto finish_before = [&]() {
        if (before >= 0 && me.rank == 0 && threadIdx.x < 32) {
            float r[3];
#pragma unroll
            for (int c = 0; c < 3; ++c) r[c] = warp_all(on ? fin[buf ^ 1][c][lane] : 0.f, SumOp());
            const float inv = 1.f / (r[0] + r[1] + r[2]);
            if (lane < 3) mass[(size_t)before * 3 + lane] = (lane == 0 ? r[0] : lane == 1 ? r[1] : r[2]) * inv;
        }
    };
    for (int row = blockIdx.x / me.size; row < rows; before = row, row += clusters, buf ^= 1) {
        const float *gg = gate + (size_t)row * V, *pp = proposal + (size_t)row * V;
        float v[2] = {-INFINITY, -INFINITY};
        sweep_pair(gg, pp, V, me, [&](auto n, const float (&g)[4 * BATCH], const float (&p)[4 * BATCH]) {
#pragma unroll
            for (int e = 0; e < decltype(n)::n; ++e) { v[0] = fmaxf(v[0], g[e]); v[1] = fmaxf(v[1], p[e]); }
        });
        block_combine<2>(v, sh_mx, MaxOp());
        if (threadIdx.x < me.size) { push_f32(&part[buf][0][me.rank], threadIdx.x, v[0]); push_f32(&part[buf][1][me.rank], threadIdx.x, v[1]); }
        row_barrier(me);
        finish_before();
        const float mg = warp_all(on ? part[buf][0][lane] : -INFINITY, MaxOp()), mp = warp_all(on ? part[buf][1][lane] : -INFINITY, MaxOp());
        float m[3] = {0.f, 0.f, 0.f};
        sweep_pair(gg, pp, V, me, [&](auto n, const float (&g)[4 * BATCH], const float (&p)[4 * BATCH]) {
#pragma unroll
            for (int e = 0; e < decltype(n)::n; ++e) {
                const float d = g[e] - mg, x = ex2((p[e] - mp) * scale2);
                m[0] += d >= log_tau_hi ? x : 0.f;
                m[1] += d < log_tau_hi && d >= log_tau_lo ? x : 0.f;
                m[2] += d >= log_tau_lo ? 0.f : x;            // (log_tau_lo <= log_tau_hi; a NaN counts here)
            }
        });
        block_combine<3>(m, sh_s, SumOp());
        if (threadIdx.x < 3) push_f32(&fin[buf][threadIdx.x][me.rank], 0, threadIdx.x == 0 ? m[0] : threadIdx.x == 1 ? m[1] : m[2]);
    }
    row_barrier(me);
    if (me.rank != 0) return;
    finish_before();
}

// total[c] = the sum over rows of v[r * C + c] divided by `over`, added up in row order by one thread per column; the values
// come in through shared memory (one load after the other from L2 they were 20 us at a thousand rows)
__global__ void __launch_bounds__(1024) row_sum_kernel(float *total, const float *v, int rows, int C, float over) {
    __shared__ float buf[6144];
    const int per = 6144 / C;
    float s = 0.f;
    for (int r0 = 0; r0 < rows; r0 += per) {
        const int n = min(per, rows - r0);
        __syncthreads();
        for (int i = threadIdx.x; i < n * C; i += blockDim.x) buf[i] = v[(size_t)r0 * C + i];
        __syncthreads();
        if ((int)threadIdx.x < C) {
#pragma unroll 8
            for (int r = 0; r < n; ++r) s += buf[r * C + threadIdx.x];
        }
    }
    if ((int)threadIdx.x < C) total[threadIdx.x] = s / over;
}

// CTAs per row: by the vocabulary (a row's bits do not depend on the call's other rows).  1021 rows, us with 1 / 2 / 4 / 8
// CTAs per row: vocabulary 152064 cost 364 / 361 / 342 / 413, masses 361 / 360 / 296 / 331 (four: 74 row pairs of 1.2 MB in
// flight, most of which L2 holds; eight: each exchange idles more threads than the better hit rate wins); 50257 cost 133 /
// 124 / 165 / 262.  The smooth margin is bound by its logarithms: two.
int row_team(int vocab, bool smooth) { return vocab >= 65536 && !smooth ? 4 : vocab >= 16384 ? 2 : 1; }

template <typename... P, typename... A>
int launch_rows(void (*kernel)(P...), int rows, int team, int (&resident)[64][MAX_TEAM + 1], cudaStream_t st, A... args) {
    cudaLaunchConfig_t cfg;
    memset(&cfg, 0, sizeof(cfg));
    cfg.blockDim = dim3(COST_THREADS);
    cfg.gridDim = dim3(team);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = team; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int dev = 0;
    CUDA_TRY(cudaGetDevice(&dev));
    if (dev < 0 || dev >= 64) return VIASD_EUNSUPPORTED;
    if (!resident[dev][team]) {                               // clusters the device holds at once, asked once
        int n = 0;
        CUDA_TRY(cudaOccupancyMaxActiveClusters(&n, kernel, &cfg));
        resident[dev][team] = n < 1 ? 1 : n;
    }
    cfg.gridDim = dim3((rows < resident[dev][team] ? rows : resident[dev][team]) * team);
    cfg.numAttrs = team > 1 ? 1 : 0;                          // (a CTA by itself: no cluster to set up)
    CUDA_TRY(cudaLaunchKernelEx(&cfg, kernel, args...));
    LAUNCH_CHECK();
    return VIASD_OK;
}

}  // namespace

extern "C" int viasd_region_mass(const float *gate_logits, const float *proposal_logits, int rows, int vocab, float temperature,
                                 float log_tau_hi, float log_tau_lo, float *mass, float *mean, void *stream) {
    if (!gate_logits || !proposal_logits || !mass || rows < 1 || vocab < 1) return VIASD_EINVAL;
    if (!(temperature > 0.f) || !(log_tau_lo <= log_tau_hi)) return VIASD_EINVAL;
    cudaStream_t st = (cudaStream_t)stream;
    static int resident[64][MAX_TEAM + 1];
    int rc = launch_rows(region_mass_kernel, rows, row_team(vocab, false), resident, st, mass, gate_logits, proposal_logits, rows, vocab,
                         (1.0f / temperature) * 1.44269504f, log_tau_hi, log_tau_lo);
    if (rc) return rc;
    if (mean) {
        row_sum_kernel<<<1, 1024, 0, st>>>(mean, mass, rows, 3, (float)rows);
        LAUNCH_CHECK();
    }
    return VIASD_OK;
}

extern "C" int viasd_kl_cost(const float *judge_logits, const float *proposal_logits, int rows, int vocab, float temperature,
                             float alpha, float beta, int margin, float tau, float *cost_rows, float *cost_total,
                             void *stream) {
    if (!judge_logits || !proposal_logits || !cost_rows || rows < 1 || vocab < 1) return VIASD_EINVAL;
    if (!(temperature > 0.f) || !(alpha >= 0.f) || !(alpha < 1.f) || !(beta > 0.f)) return VIASD_EINVAL;
    if (margin != 0 && margin != 1) return VIASD_EINVAL;
    if (margin == 1 && !(tau > 0.f)) return VIASD_EINVAL;
    cudaStream_t st = (cudaStream_t)stream;
    static int resident[2][64][MAX_TEAM + 1];
    int rc = launch_rows(margin ? kl_cost_kernel<1> : kl_cost_kernel<0>, rows, row_team(vocab, margin == 1), resident[margin], st, cost_rows, judge_logits,
                         proposal_logits, rows, vocab, exp_scale(temperature), 1.0f / temperature, log1pf(-alpha), logf(beta), tau);
    if (rc) return rc;
    if (cost_total) {
        row_sum_kernel<<<1, 1024, 0, st>>>(cost_total, cost_rows, rows, 1, 1.f);
        LAUNCH_CHECK();
    }
    return VIASD_OK;
}
