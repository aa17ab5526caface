// Device-side pieces of the tcgen05 GEMM kernel: tile constants, the unit-range walk of the stream-K
// schedule and the fused epilogues.
#pragma once
#include "common.cuh"
#include "gemm_tc.cuh"
#include "tc_ptx.cuh"

namespace {

constexpr int TILE_F = 128;          // output features per tile (MMA M)
constexpr int TILE_K = 64;           // bf16 per k-block: 128 bytes, one swizzle row
constexpr int MAX_STAGES = 12;

constexpr int CH = 8;                // token rows per epilogue chunk
__device__ __forceinline__ void tc_ld8(uint32_t taddr, float (&v)[CH]) {
    uint32_t r[8];
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 8; ++i) v[i] = __uint_as_float(r[i]);
}

// two groups of columns with one wait (hi and lo columns of a chunk): the second load does not wait for the first
__device__ __forceinline__ void tc_ld8x2(uint32_t ta, uint32_t tb, float (&a)[CH], float (&b)[CH]) {
    uint32_t r[8], q[8];
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(ta));
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(q[0]), "=r"(q[1]), "=r"(q[2]), "=r"(q[3]), "=r"(q[4]), "=r"(q[5]), "=r"(q[6]), "=r"(q[7])
                 : "r"(tb));
    // the wait names the registers: no use of them may be scheduled ahead of it
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),
                   "+r"(q[0]), "+r"(q[1]), "+r"(q[2]), "+r"(q[3]), "+r"(q[4]), "+r"(q[5]), "+r"(q[6]), "+r"(q[7])
                 :: "memory");
#pragma unroll
    for (int i = 0; i < 8; ++i) { a[i] = __uint_as_float(r[i]); b[i] = __uint_as_float(q[i]); }
}

struct Seg { int tile, ka, kb; };      // one contiguous piece of this CTA's unit range inside a tile

__device__ __forceinline__ bool next_seg(int &u, int u1, int k_tiles, Seg &s) {
    if (u >= u1) return false;
    s.tile = u / k_tiles;
    s.ka = u - s.tile * k_tiles;
    s.kb = min(k_tiles, s.ka + (u1 - u));
    u += s.kb - s.ka;
    return true;
}

// ---- finishing, a token row per warp: lane l holds features 4l .. 4l+3 of the tile -------------------------------
__device__ __forceinline__ float4 add4(float4 a, float4 b) { return make_float4(a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w); }
__device__ __forceinline__ float4 scale4(float4 a, float s) { return make_float4(a.x * s, a.y * s, a.z * s, a.w * s); }
__device__ __forceinline__ uint2 pack4(float4 v) {
    const __nv_bfloat162 a = __floats2bfloat162_rn(v.x, v.y), b = __floats2bfloat162_rn(v.z, v.w);
    return make_uint2(*reinterpret_cast<const uint32_t *>(&a), *reinterpret_cast<const uint32_t *>(&b));
}
// live: store; else (a dry pass that warms the instruction cache) ask for the line, so that the first store does not start
// with an address-translation miss
template <typename V>
__device__ __forceinline__ void put(bool live, void *dst, V v) {
    if (live) *reinterpret_cast<V *>(dst) = v;
    else asm volatile("prefetch.global.L2 [%0];" ::"l"(dst));
}
// four values as hi and lo planes (x = hi + lo to about 16 mantissa bits)
__device__ __forceinline__ void store_pair4(bool live, __nv_bfloat16 *dst, size_t plane, float4 v) {
    const __nv_bfloat16 h0 = __float2bfloat16_rn(v.x), h1 = __float2bfloat16_rn(v.y), h2 = __float2bfloat16_rn(v.z), h3 = __float2bfloat16_rn(v.w);
    const uint2 hi = make_uint2((uint32_t)__bfloat16_as_ushort(h0) | ((uint32_t)__bfloat16_as_ushort(h1) << 16),
                                (uint32_t)__bfloat16_as_ushort(h2) | ((uint32_t)__bfloat16_as_ushort(h3) << 16));
    put(live, dst, hi);
    put(live, dst + plane, pack4(make_float4(v.x - __bfloat162float(h0), v.y - __bfloat162float(h1),
                                             v.z - __bfloat162float(h2), v.w - __bfloat162float(h3))));
}

// One token row of a tile: v = the row's full sums (u: those of the up matrix, EPI_SWIGLU of the one-CTA kernel).
// HALVES (pair kernel): lanes 0..15 hold 64 gate features, lanes 16..31 the matching up features.
// aux0 / aux1: the residual row (EPI_ADD_NORM), or the row's cosines and sines (EPI_QKV_ROPE).
template <int EPI, bool HALVES>
__device__ __forceinline__ void finish_row(const TcParams &p, int tile, int row, bool live, float4 v, float4 u, float4 aux0, float4 aux1,
                                           float4 gain_a, float4 gain_b, const float *inv_sh, const int4 *rowmeta, int lane) {
    const int grow = p.row0 + row;
    if (EPI != EPI_ADD_NORM && p.ssq_in) {                                 // the input was h * gain without its RMS factor
        v = scale4(v, inv_sh[row]);
        if (EPI == EPI_SWIGLU && !HALVES) u = scale4(u, inv_sh[row]);
    }
    if (EPI == EPI_SWIGLU) {
        if (HALVES) {
            // lanes 0..15 have four gate features each, lanes 16..31 the matching up features: they trade two, so that every lane has
            // two of both (with lanes 0..15 doing all four: prompt chunk 24.71 ms, now 24.30; steps of many rows within their runs' spread)
            const bool low = lane < 16;
            const float r0 = __shfl_xor_sync(0xffffffffu, low ? v.z : v.x, 16), r1 = __shfl_xor_sync(0xffffffffu, low ? v.w : v.y, 16);
            const float g0 = low ? v.x : r0, g1 = low ? v.y : r1, u0 = low ? r0 : v.z, u1 = low ? r1 : v.w;
            const int n = tile * 64 + 4 * (lane & 15) + (low ? 0 : 2);
            if (n < p.seg_n[0]) {                                          // (d_ff is a multiple of 8)
                const float y0 = g0 / (1.f + __expf(-g0)) * u0, y1 = g1 / (1.f + __expf(-g1)) * u1;
                const __nv_bfloat16 h0 = __float2bfloat16_rn(y0), h1 = __float2bfloat16_rn(y1);
                const __nv_bfloat162 l = __floats2bfloat162_rn(y0 - __bfloat162float(h0), y1 - __bfloat162float(h1));
                __nv_bfloat16 *dst = p.out_act + (size_t)grow * p.ld_out + n;
                put(live, dst, (uint32_t)__bfloat16_as_ushort(h0) | ((uint32_t)__bfloat16_as_ushort(h1) << 16));
                put(live, dst + p.act_plane, *reinterpret_cast<const uint32_t *>(&l));
            }
            return;
        }
        const int n = tile * TILE_F + 4 * lane;
        if (n < p.seg_n[0]) {
            const float4 y = make_float4(v.x / (1.f + __expf(-v.x)) * u.x, v.y / (1.f + __expf(-v.y)) * u.y,
                                         v.z / (1.f + __expf(-v.z)) * u.z, v.w / (1.f + __expf(-v.w)) * u.w);
            store_pair4(live, p.out_act + (size_t)grow * p.ld_out + n, p.act_plane, y);
        }
        return;
    }
    int s = 0, t0 = 0, nbase = 0;
    while (s < 2 && tile >= p.seg_tile_end[s]) { t0 = p.seg_tile_end[s]; nbase += p.seg_n[s]; ++s; }
    const int nin = (tile - t0) * TILE_F + 4 * lane, n = nbase + nin;
    if (EPI == EPI_STORE) {                                                // (also EPI_ADD: the unfused residual update)
        if (nin >= p.seg_n[s]) return;
        float *dst = grow < p.split_row ? p.out_f32 + (size_t)grow * p.ld_out + n                 // the second stream's rows go
                                        : p.out_f32_2 + (size_t)(grow - p.split_row) * p.ld_out + n;   // to the second output
        if (p.out_vec4 && nin + 3 < p.seg_n[s]) {
            if (p.epi == EPI_ADD && live) v = add4(*reinterpret_cast<const float4 *>(dst), v);
            put(live, dst, v);
            return;
        }
        const float e[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) if (nin + i < p.seg_n[s]) put(live, dst + i, p.epi == EPI_ADD && live ? dst[i] + e[i] : e[i]);
    } else if (EPI == EPI_ADD_NORM) {
        // residual update, and what the next RMSNorm needs: h * gain as planes, sums of h^2 per 32 features
        v = add4(v, aux0);
        const size_t o = (size_t)grow * p.ld_out + n;                      // (d_model is a multiple of 128)
        put(live, p.out_f32 + o, v);
        const float4 g = grow < p.split_row ? gain_a : gain_b;
        store_pair4(live, p.next_act + o, p.next_plane, make_float4(v.x * g.x, v.y * g.y, v.z * g.z, v.w * g.w));
        float q = (v.x * v.x + v.y * v.y) + (v.z * v.z + v.w * v.w);
#pragma unroll
        for (int d = 4; d > 0; d >>= 1) q += __shfl_xor_sync(0xffffffffu, q, d);
        if ((lane & 7) == 0) put(live, p.ssq_out + ((size_t)tile * 4 + (lane >> 3)) * p.ssq_stride + grow, q);
    } else {                                                               // EPI_QKV_ROPE: the tile is one head of 128 dims
        const int4 rm = rowmeta[row];
        if (s < 2) {
            float4 w;                                                      // the rotary partner (dim ^ 64)
            w.x = __shfl_xor_sync(0xffffffffu, v.x, 16); w.y = __shfl_xor_sync(0xffffffffu, v.y, 16);
            w.z = __shfl_xor_sync(0xffffffffu, v.z, 16); w.w = __shfl_xor_sync(0xffffffffu, v.w, 16);
            const float sg = lane < 16 ? -1.f : 1.f;
            v = make_float4(v.x * aux0.x + sg * w.x * aux1.x, v.y * aux0.y + sg * w.y * aux1.y,
                            v.z * aux0.z + sg * w.z * aux1.z, v.w * aux0.w + sg * w.w * aux1.w);
        }
        const int head = tile - t0;
        if (s == 0) {
            put(live, p.q_out + ((size_t)grow * p.rope_H + head) * TILE_F + 4 * lane, v);
        } else if (rm.y >= 0) {
            const size_t off = ((size_t)((unsigned)rm.w & 0x3fffffffu) << 32) | (unsigned)rm.z;
            __nv_bfloat16 *c0 = s == 1 ? p.kc : p.vc, *c1 = s == 1 ? p.kc2 : p.vc2;
            __nv_bfloat16 *dst = (((unsigned)rm.w >> 30) & 1u ? c1 : c0) + off + (size_t)head * p.max_ctx * TILE_F + 4 * lane;
            put(live, dst, pack4(v));
        }
    }
}

}  // namespace
