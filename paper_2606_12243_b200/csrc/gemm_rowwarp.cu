// Generic CUDA-core GEMM y[rows, n] = x[rows, k] * W[n, k]^T for a handful of rows.
// One warp owns FEAT output features and streams their weight rows once with 16-byte loads; the
// activation vector it multiplies with is reused across the FEAT features from registers.  Four features where that still
// gives every SM a CTA (a 256 x 256 projection is 8 CTAs of four-feature warps, each a chain of dependent loads); below that
// one, or two from a size on that is the lower the more rows share a weight's load.  us with 1 / 2 / 4 features, 9 rows: 1024 x
// 1024 9.0 / 11.3 / 19.7, 2048 x 2048 29.9 / 20.9 / 39.2, 4096 x 2048 49.8 / 39.7 / 40.6, 6144 x 1024 40.0 / 28.5 / 21.9; 5 rows: 2048 x
// 2048 14.4 / 15.7 / 24.8, 3072 x 768 11.2 / 6.6 / 12.3; 1 row: 4096 x 2048 10.7 / 12.6 / 15.1.  With a feature per warp, the loads of several k-steps in flight, no branches between
// them, the rows' read-modify-writes side by side and launches that overlap, the 14 GEMMs of the two-layer fp32 step
// (d = 256) take 114 us instead of 211.
// Serves the fp32 model configuration and any shape the tensor-core kernels do not take.
#include "common.cuh"

namespace {

template <typename T> struct Vec;                 // 16 bytes of T
template <> struct Vec<float> { static constexpr int N = 4; };
template <> struct Vec<__nv_bfloat16> { static constexpr int N = 8; };

template <typename T>
__device__ __forceinline__ void load16(const T *p, float (&out)[Vec<T>::N]);
template <>
__device__ __forceinline__ void load16<float>(const float *p, float (&out)[4]) {
    float4 v = *reinterpret_cast<const float4 *>(p);
    out[0] = v.x; out[1] = v.y; out[2] = v.z; out[3] = v.w;
}
template <>
__device__ __forceinline__ void load16<__nv_bfloat16>(const __nv_bfloat16 *p, float (&out)[8]) {
    uint4 v = *reinterpret_cast<const uint4 *>(p);
    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        out[2 * i] = __uint_as_float(w[i] << 16);
        out[2 * i + 1] = __uint_as_float(w[i] & 0xffff0000u);
    }
}

constexpr int WARPS = 8;

struct SegTable { const void *w[3]; int end[3]; int count; };

template <typename T>
__device__ __forceinline__ const T *weight_row(const SegTable &s, int n, int k) {
    int base = 0;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        if (i < s.count && n < s.end[i]) return reinterpret_cast<const T *>(s.w[i]) + (size_t)(n - base) * k;
        base = s.end[i];
    }
    return nullptr;
}

// RC rows are kept in registers at a time; more rows loop (weights then come from L2).
template <typename T, int RC, int EPI, int FEAT>
__global__ void __launch_bounds__(WARPS * 32)
gemm_rowwarp_kernel(const T *__restrict__ x, size_t x_plane, SegTable segs, int rows, int k, int n_total,
                    float *__restrict__ out_f32, T *__restrict__ out_act, size_t act_plane, int ld_out) {
    constexpr int VN = Vec<T>::N;
    PDL_TRIGGER();
    PDL_WAIT();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int group = blockIdx.x * WARPS + warp;
    constexpr int UNROLL = FEAT > 2 ? 1 : RC <= 4 ? 4 : 2;          // k-steps with their loads in flight together
    constexpr int HF = EPI == EPI_SWIGLU ? FEAT / 2 : FEAT;
    const T *wrow[FEAT];
    int feat[FEAT];
    if (EPI == EPI_SWIGLU) {
        // HF features from f0 on of the gate matrix and the same of the up matrix
        const int ff = segs.end[0];
        const int f0 = group * HF;
        if (f0 >= ff) return;
#pragma unroll
        for (int j = 0; j < HF; ++j) {
            int f = f0 + j;
            feat[j] = f; feat[HF + j] = f;
            bool ok = f < ff;
            wrow[j] = ok ? reinterpret_cast<const T *>(segs.w[0]) + (size_t)f * k : nullptr;
            wrow[HF + j] = ok ? reinterpret_cast<const T *>(segs.w[1]) + (size_t)f * k : nullptr;
        }
    } else {
        const int n0 = group * FEAT;
        if (n0 >= n_total) return;
#pragma unroll
        for (int j = 0; j < FEAT; ++j) {
            feat[j] = n0 + j;
            wrow[j] = (n0 + j < n_total) ? weight_row<T>(segs, n0 + j, k) : nullptr;
        }
    }
    for (int r0 = 0; r0 < rows; r0 += RC) {
        float acc[RC][FEAT];
#pragma unroll
        for (int r = 0; r < RC; ++r)
#pragma unroll
            for (int j = 0; j < FEAT; ++j) acc[r][j] = 0.f;
#pragma unroll UNROLL
        for (int k0 = lane * VN; k0 < k; k0 += 32 * VN) {
            float wv[FEAT][VN];
#pragma unroll
            for (int j = 0; j < FEAT; ++j) {
                if (wrow[j]) load16<T>(wrow[j] + k0, wv[j]);
                else {
#pragma unroll
                    for (int e = 0; e < VN; ++e) wv[j][e] = 0.f;
                }
            }
            // (rows past the end repeat the last one, unstored: a branch around a load would keep it behind the loads before it)
#pragma unroll
            for (int r = 0; r < RC; ++r) {
                const T *xr = x + (size_t)min(r0 + r, rows - 1) * k + k0;
                float xv[VN];
                load16<T>(xr, xv);
                if (x_plane) {                          // bf16 activations come as hi + lo planes
                    float lo[VN];
                    load16<T>(xr + x_plane, lo);
#pragma unroll
                    for (int e = 0; e < VN; ++e) xv[e] += lo[e];
                }
#pragma unroll
                for (int j = 0; j < FEAT; ++j)
#pragma unroll
                    for (int e = 0; e < VN; ++e) acc[r][j] = fmaf(xv[e], wv[j][e], acc[r][j]);
            }
        }
#pragma unroll
        for (int r = 0; r < RC; ++r)
#pragma unroll
            for (int j = 0; j < FEAT; ++j) acc[r][j] = warp_sum(acc[r][j]);
        // lane r finishes row r0 + r: the rows' read-modify-writes run side by side
        if (lane < RC && r0 + lane < rows) {
            float mine[FEAT];
#pragma unroll
            for (int j = 0; j < FEAT; ++j) {
                mine[j] = acc[0][j];
#pragma unroll
                for (int r = 1; r < RC; ++r) mine[j] = lane == r ? acc[r][j] : mine[j];
            }
            const size_t row = r0 + lane;
            if (EPI == EPI_SWIGLU) {
#pragma unroll
                for (int j = 0; j < HF; ++j) {
                    if (!wrow[j]) continue;
                    const float g = mine[j], u = mine[HF + j], s = g / (1.f + expf(-g));
                    store_act<T>(out_act, act_plane, row * ld_out + feat[j], s * u);
                }
            } else {
#pragma unroll
                for (int j = 0; j < FEAT; ++j) {
                    if (!wrow[j]) continue;
                    float *dst = out_f32 + row * ld_out + feat[j];
                    if (EPI == EPI_ADD) *dst += mine[j]; else *dst = mine[j];
                }
            }
        }
    }
}

template <typename T, int RC>
int dispatch_epi(const T *x, size_t x_plane, const SegTable &s, int rows, int k, int n_total, int epi, float *out_f32,
                 T *out_act, size_t act_plane, int ld_out, int sms, cudaStream_t st) {
    const int outs = epi == EPI_SWIGLU ? 2 * s.end[0] : n_total;            // weight rows in all
    const bool two = RC > 8 ? outs >= 12 * sms : RC > 4 && outs >= 16 * sms;
    const int feat = outs >= 4 * WARPS * sms ? 4 : two || epi == EPI_SWIGLU ? 2 : 1;
#define ROWWARP(KIND, F)                                                                                                    \
    CUDA_TRY(launch_chained(gemm_rowwarp_kernel<T, RC, KIND, F>, ((outs + F - 1) / F + WARPS - 1) / WARPS, WARPS * 32, st,   \
                            x, x_plane, s, rows, k, n_total, out_f32, out_act, act_plane, ld_out))
    switch (epi) {
    case EPI_STORE: if (feat == 4) ROWWARP(EPI_STORE, 4); else if (feat == 2) ROWWARP(EPI_STORE, 2); else ROWWARP(EPI_STORE, 1); break;
    case EPI_ADD: if (feat == 4) ROWWARP(EPI_ADD, 4); else if (feat == 2) ROWWARP(EPI_ADD, 2); else ROWWARP(EPI_ADD, 1); break;
    case EPI_SWIGLU: if (feat == 4) ROWWARP(EPI_SWIGLU, 4); else ROWWARP(EPI_SWIGLU, 2); break;
    default: return VIASD_EINVAL;
    }
#undef ROWWARP
    LAUNCH_CHECK();
    return VIASD_OK;
}

template <typename T>
int dispatch_rows(const T *x, size_t x_plane, const SegTable &s, int rows, int k, int n_total, int epi, float *out_f32,
                  T *out_act, size_t act_plane, int ld_out, int sms, cudaStream_t st) {
    if (rows <= 4) return dispatch_epi<T, 4>(x, x_plane, s, rows, k, n_total, epi, out_f32, out_act, act_plane, ld_out, sms, st);
    if (rows <= 8) return dispatch_epi<T, 8>(x, x_plane, s, rows, k, n_total, epi, out_f32, out_act, act_plane, ld_out, sms, st);
    return dispatch_epi<T, 12>(x, x_plane, s, rows, k, n_total, epi, out_f32, out_act, act_plane, ld_out, sms, st);
}

}  // namespace

int launch_gemm_rowwarp(const void *x, size_t x_plane, const GemmSegs &segs, int rows, int k, int dtype,
                        int epilogue, float *out_f32, void *out_act, size_t act_plane, int ld_out, int sms, cudaStream_t st) {
    if (rows <= 0) return VIASD_OK;
    if (k % 8 != 0) return VIASD_EINVAL;
    SegTable s;
    int total = 0;
    s.count = segs.count;
    for (int i = 0; i < 3; ++i) {
        s.w[i] = i < segs.count ? segs.w[i] : nullptr;
        if (i < segs.count) total += segs.n[i];
        s.end[i] = total;
    }
    if (epilogue == EPI_SWIGLU && (segs.count != 2 || segs.n[0] != segs.n[1])) return VIASD_EINVAL;
    if (dtype == 0)
        return dispatch_rows<float>((const float *)x, 0, s, rows, k, total, epilogue, out_f32, (float *)out_act, 0, ld_out, sms, st);
    return dispatch_rows<__nv_bfloat16>((const __nv_bfloat16 *)x, x_plane, s, rows, k, total, epilogue, out_f32,
                                        (__nv_bfloat16 *)out_act, act_plane, ld_out, sms, st);
}
