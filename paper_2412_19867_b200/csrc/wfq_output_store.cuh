// What the floating-point and the integer output transform have in common: the epilogue, the stores of y and
// the launch shape.
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <type_traits>

#include "wfq_internal.h"

namespace wfq {
namespace {

// One rounding to the 16-bit output type: kind 1 = fp16, 2 = bf16 (round to nearest even).
__device__ __forceinline__ uint16_t to_bits16(float v, int kind)
{
    return kind == 2 ? __bfloat16_as_ushort(__float2bfloat16_rn(v)) : __half_as_ushort(__float2half_rn(v));
}
__device__ __forceinline__ uint32_t to_bits16x2(float lo, float hi, int kind)
{
    return (uint32_t)to_bits16(lo, kind) | ((uint32_t)to_bits16(hi, kind) << 16);
}

// t / (1 + exp(-t)).  The reciprocal is the hardware's approximation with one Newton step: __frcp_rn rounds correctly but
// takes several times the instructions, which bounded the SiLU layers (forward, two layers of 640 channels 32x32 49.8 ->
// 46.6 us, 64x64 F(6,3) 34.6 -> 32.9 us; 16 images 10x10, 128 channels 13.8 -> 11.9 us).  Over all 2^32 floats the
// results are the same but for 34 033 below t = -87, where the reciprocal is denormal; the error against 64 bits is that of
// __expf (at most 3.0, 15.5 and 64.3 units in the last place up to |t| = 1, 16 and 87; rms 0.32, 1.8 and 11).  A quarter of
// 1 + exp(-t) keeps the reciprocal a normal number for every finite exp(-t); where that overflows the step's NaN becomes
// -1 and the reciprocal stays 0.
__device__ __forceinline__ float silu(float t)
{
    const float d = fmaf(__expf(-t), 0.25f, 0.25f);
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(d));
    r = fmaf(r, fmaxf(fmaf(-d, r, 1.f), -1.f), r);
    return t * (0.25f * r);
}
// Optional epilogue on the spatial-domain outputs of one row segment: per-output-channel
// bias, then ReLU or SiLU (act: 0 none, 1 ReLU, 2 SiLU).
template <int M>
__device__ __forceinline__ void epilogue(float (&o)[M], float bias, int act)
{
#pragma unroll
    for (int v = 0; v < M; ++v) {
        float t = o[v] + bias;
        if (act == 1) t = fmaxf(t, 0.f);
        else if (act == 2) t = silu(t);
        o[v] = t;
    }
}

// STORE: 2 = 16-byte stores straight from the
// registers (F(4,3), W a multiple of 4: neighbouring lanes then write neighbouring 16 bytes
// and a warp fills whole sectors), 1 = every other even W, 0 = odd W: the m-float row
// segments of a tile are 24 (or 16) bytes apart, so that direct stores would write every
// 32-byte sector of y in several pieces, and the L2 takes a piece as long as a whole sector
// (measured for F(6,3) with 8-byte stores: 2.3 sector writes per sector of y, and the
// kernel bound by them).  The CTA therefore collects its tiles' outputs in shared memory,
// one array per output row u with the tiles side by side exactly as they lie in the image
// row, and copies them out with consecutive lanes on consecutive 8 bytes (even W) or
// consecutive floats (odd W).  A thread keeps its place in the rows and goes down them: tile, limits and offset are
// formed once per place instead of once per element (most of the instructions of the copy; forward, 128 tiles x 512
// channels of 7x7 images, two layers, 55.7 -> 53.1 us; ten 22x15 images, 64 channels, integer transforms 24.8 -> 23.6).
// What one thread per tile of a CTA's TT (64 or 128) tiles has computed goes to y: `row_of(u, o)` gives row u of the
// thread's tile (called once per u), base is the offset of y[img][k][h0][w0].
template <int M, int STORE, int TT>
struct StoreShared {
    float out[STORE != 2 ? M * TT * M : 1];       // [u][tile][v]
    int tile_base[STORE != 2 ? TT : 1];           // offset of the tile's y[.][.][h0][w0]
    int tile_lim[STORE != 2 ? TT : 1];            // valid rows * 16 + valid columns
};

template <int M, int STORE, bool EPI, int TT, typename RowOf>
__device__ __forceinline__ void store_tiles(const RowOf &row_of, StoreShared<M, STORE, TT> &sm, bool live, size_t base,
                                            int h0, int w0, int k, float *__restrict__ y, const Geometry &g,
                                            const float *__restrict__ bias, int act, int out_half)
{
    // 16-bit output (epilogue variants only; out_half 1 = fp16, 2 = bf16): y points at 2-byte storage
    // of the same shape
    [[maybe_unused]] uint16_t *yh = reinterpret_cast<uint16_t *>(y);
    float *out_s = sm.out;
    int *tile_base = sm.tile_base, *tile_lim = sm.tile_lim;
    if constexpr (STORE != 2) {
        const int j = threadIdx.x;
        if (live) {
            const float bk = (EPI && bias) ? __ldg(bias + k) : 0.f;
#pragma unroll
            for (int u = 0; u < M; ++u) {
                float o[M];
                row_of(u, o);
                if constexpr (EPI) epilogue<M>(o, bk, act);
                float2 *dst = reinterpret_cast<float2 *>(out_s + (u * TT + j) * M);
#pragma unroll
                for (int v2 = 0; v2 < M; v2 += 2) dst[v2 / 2] = make_float2(o[v2], o[v2 + 1]);
            }
        }
        tile_base[j] = (int)base;
        tile_lim[j] = live ? (min(M, g.H - h0) * 16 + min(M, g.W - w0)) : 0;
        __syncthreads();
        if constexpr (STORE == 0) {
            // float f of a row: tile f / M, column f % M
#pragma unroll
            for (int i = 0; i < M; ++i) {
                const int f = threadIdx.x + i * TT;
                const int tj = f / M, v1 = f - tj * M;
                const int lim = tile_lim[tj], rows = v1 < (lim & 15) ? lim >> 4 : 0;
                size_t off = (size_t)tile_base[tj] + v1;
                const float *src = out_s + f;
#pragma unroll
                for (int u = 0; u < M; ++u) {
                    if (u < rows) {
                        if (EPI && out_half) yh[off] = to_bits16(src[u * TT * M], out_half);
                        else y[off] = src[u * TT * M];
                    }
                    off += g.W;
                }
            }
            return;
        }
        // pair q of a row: tile q / (M/2), columns 2 * (q % (M/2)) and the next
        constexpr int PPT = M / 2;                // pairs per tile row
#pragma unroll
        for (int i = 0; i < PPT; ++i) {
            const int q = threadIdx.x + i * TT;
            const int tj = q / PPT, v2 = 2 * (q - tj * PPT);
            const int lim = tile_lim[tj], rows = v2 < (lim & 15) ? lim >> 4 : 0;    // W even: both columns or none
            size_t off = (size_t)tile_base[tj] + v2;
            const float2 *src = reinterpret_cast<const float2 *>(out_s) + q;
#pragma unroll
            for (int u = 0; u < M; ++u) {
                if (u < rows) {
                    const float2 r = src[u * TT * PPT];
                    if (EPI && out_half) *reinterpret_cast<uint32_t *>(yh + off) = to_bits16x2(r.x, r.y, out_half);
                    else *reinterpret_cast<float2 *>(y + off) = r;
                }
                off += g.W;
            }
        }
    } else {
        float *row = y + base;
        uint16_t *rowh = yh + base;
        const bool full_w = (w0 + M <= g.W);
        const float bk = (EPI && bias) ? __ldg(bias + k) : 0.f;
#pragma unroll
        for (int u = 0; u < M; ++u) {
            float o[M];
            row_of(u, o);
            if constexpr (EPI) epilogue<M>(o, bk, act);
            if (h0 + u < g.H) {
                if (EPI && out_half) {
                    if (full_w) {
                        *reinterpret_cast<uint2 *>(rowh) = make_uint2(to_bits16x2(o[0], o[1], out_half),
                                                                      to_bits16x2(o[2], o[3], out_half));
                    } else {
#pragma unroll
                        for (int v2 = 0; v2 < M; ++v2)
                            if (w0 + v2 < g.W) rowh[v2] = to_bits16(o[v2], out_half);
                    }
                } else if (full_w) {
                    *reinterpret_cast<float4 *>(row) = make_float4(o[0], o[1], o[2], o[3]);
                } else {
#pragma unroll
                    for (int v2 = 0; v2 < M; ++v2)
                        if (w0 + v2 < g.W) row[v2] = o[v2];
                }
            }
            row += g.W;
            rowh += g.W;
        }
    }
}

// F(6,3): CTAs of 64 tiles where they leave at least a twentieth fewer threads without a tile than CTAs
// of 128: 36 tiles of 1280 channels (forward 47.6 -> 45.7 us; of 640 with an epilogue 45.0 -> 38.7 us), 800
// tiles of 128 channels with an epilogue (36.4 -> 33.7 us), 162 of 256 (26.6 -> 25.9 us).  With about
// the same number of threads they are no better (121 tiles of 640 channels 41.2 -> 41.8 us, 3200 and 1600
// tiles within 0.3 us), and F(4,3) and F(2,3) gain nothing from them (32 tiles of 1280 channels 26.5 ->
// 26.8 us, 3136 tiles of 128 channels 23.9 -> 24.4 us).  The integer kernels gain more: forward with one scale
// per tile, 36 tiles of 640 channels 28.6 -> 26.3 us, with one per row 48.5 -> 34.1 us; 800 tiles of 64
// channels 30.9 -> 29.9 and 50.1 -> 37.3 us.
bool half_ctas(const Geometry &g)
{
    const long long by64 = ((long long)g.T + 63) / 64 * 64, by128 = ((long long)g.T + 127) / 128 * 128;
    return g.m == 6 && 20 * by64 <= 19 * by128;
}

// Calls f with <M, STORE, TT> as integral constants.  y is 16-byte aligned; rows of an even W keep 8-byte
// alignment for every tile.
template <typename F>
cudaError_t with_store(int m, int W, bool half, F f)
{
    using std::integral_constant;
    constexpr integral_constant<int, 0> odd{};
    constexpr integral_constant<int, 1> even{};
    constexpr integral_constant<int, 2> fours{};
    constexpr integral_constant<int, 64> t64{};
    constexpr integral_constant<int, 128> t128{};
    if (m == 2) {
        constexpr integral_constant<int, 2> m2{};
        return W % 2 == 0 ? f(m2, even, t128) : f(m2, odd, t128);
    }
    if (m == 4) {
        constexpr integral_constant<int, 4> m4{};
        return W % 4 == 0 ? f(m4, fours, t128) : W % 2 == 0 ? f(m4, even, t128) : f(m4, odd, t128);
    }
    constexpr integral_constant<int, 6> m6{};
    if (half) return W % 2 == 0 ? f(m6, even, t64) : f(m6, odd, t64);
    return W % 2 == 0 ? f(m6, even, t128) : f(m6, odd, t128);
}

template <typename F>
cudaError_t with_store(const Geometry &g, F f) { return with_store(g.m, g.W, half_ctas(g), f); }

cudaLaunchConfig_t output_config(const wfq_plan &plan, cudaStream_t stream, bool pdl, cudaLaunchAttribute *attr)
{
    const int tt = half_ctas(plan.geo) ? 64 : 128;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((plan.geo.T + tt - 1) / tt, plan.geo.K);
    cfg.blockDim = dim3(tt);
    cfg.stream = stream;
    attr->id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr->val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = pdl ? 1 : 0;
    return cfg;
}

}  // namespace
}  // namespace wfq
