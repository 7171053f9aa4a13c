// What the NCHW input transforms with strips in shared memory have in common: staging of a work item's input
// strip (cp.async), patch loads from it, and the group quantizer of a work item's transformed values.
#pragma once

#include <cuda_fp16.h>

#include "wfq_internal.h"

namespace wfq {
namespace {

constexpr int K1_THREADS = 128;
constexpr int K1_WP = 16;        // staged columns per row (image columns w_base .. w_base+15)
constexpr int K1_WPV = 24;       // the same where rows are copied in aligned 16-byte pieces (w_base a multiple of 8)

// ---- patch load from the staged strip ---------------------------------------------
// `ch` points at the channel's plane in smem; `col0` is the (even) smem column whose
// successor is the tile's first input column.
template <int NN>
__device__ __forceinline__ void load_patch(const __half *ch, int col0, float (&d)[NN][NN])
{
#pragma unroll
    for (int a = 0; a < NN; ++a) {
        const __half2 *row = reinterpret_cast<const __half2 *>(ch + a * K1_WP + col0);
        float v[NN + 2];
#pragma unroll
        for (int w = 0; w < (NN + 2) / 2; ++w) {
            const float2 f = __half22float2(row[w]);
            v[2 * w] = f.x;
            v[2 * w + 1] = f.y;
        }
#pragma unroll
        for (int b = 0; b < NN; ++b) d[a][b] = v[b + 1];
    }
}

// The same from a strip staged in 16-byte pieces (rows of K1_WPV columns, channel stride a
// multiple of 16 bytes and an odd number of 16-byte units): 16-byte loads, for which the eight
// lanes of a quarter warp then hit eight different groups of four banks.  `k0` is the first of
// the two 16-byte pieces that hold columns col0 .. col0 + NN + 1, WO the 32-bit word of col0
// inside them (col0 is even); both are the same for all lanes of the warp.
template <int NN, int WO>
__device__ __forceinline__ void load_patch_vec(const __half *ch, int k0, float (&d)[NN][NN])
{
#pragma unroll
    for (int a = 0; a < NN; ++a) {
        const uint4 *row = reinterpret_cast<const uint4 *>(ch + a * K1_WPV) + k0;
        const uint4 q0 = row[0], q1 = row[1];
        const uint32_t w[8] = {q0.x, q0.y, q0.z, q0.w, q1.x, q1.y, q1.z, q1.w};
        float v[NN + 2];
#pragma unroll
        for (int i = 0; i < (NN + 2) / 2; ++i) {
            const float2 f = __half22float2(*reinterpret_cast<const __half2 *>(&w[WO + i]));
            v[2 * i] = f.x;
            v[2 * i + 1] = f.y;
        }
#pragma unroll
        for (int b = 0; b < NN; ++b) d[a][b] = v[b + 1];
    }
}
template <int NN>
__device__ __forceinline__ void load_patch_vec(const __half *ch, int col0, float (&d)[NN][NN])
{
    const int k0 = col0 >> 3;
    switch ((col0 & 7) >> 1) {            // warp-uniform
        case 0: load_patch_vec<NN, 0>(ch, k0, d); break;
        case 1: load_patch_vec<NN, 1>(ch, k0, d); break;
        case 2: load_patch_vec<NN, 2>(ch, k0, d); break;
        default: load_patch_vec<NN, 3>(ch, k0, d); break;
    }
}
template <int NN>
__device__ __forceinline__ void load_patch_vec(const float *, int, float (&)[NN][NN]) {}   // fp16 only

template <int NN>
__device__ __forceinline__ void load_patch(const float *ch, int col0, float (&d)[NN][NN])
{
#pragma unroll
    for (int a = 0; a < NN; ++a)
#pragma unroll
        for (int b = 0; b < NN; ++b) d[a][b] = ch[a * K1_WP + col0 + 1 + b];
}

// Codes: round v*inv to the nearest integer (ties to even) and keep the low byte.
// fl32(v*inv) + 1.5*2^23 is exact up to the rounding to an integer, and the sum's bit
// pattern is 0x4B400000 + q for |q| <= 2^22.
// Packed f32x2 multiply (one instruction for two products, each correctly rounded).
__device__ __forceinline__ float2 mul2_rn(float2 a, float2 b)
{
    float2 d;
    asm("{\n\t.reg .b64 ra, rb, rd;\n\t"
        "mov.b64 ra, {%2, %3};\n\tmov.b64 rb, {%4, %5};\n\t"
        "mul.rn.f32x2 rd, ra, rb;\n\t"
        "mov.b64 {%0, %1}, rd;\n\t}"
        : "=f"(d.x), "=f"(d.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return d;
}

// One code: fl32(v*inv), then + 1.5*2^23; two separately rounded scalar operations, as
// the quantizer is defined.  (A packed multiply followed by a packed add, written as
// intrinsics or as PTX, came out as one fused multiply-add: it rounds once and decides
// near-ties differently, and a single differing code of an outlier-dominated group can
// move the final output by more than the end-to-end tolerance.)
__device__ __forceinline__ uint32_t code_bits(float v, float inv)
{
    return __float_as_uint(__fadd_rn(__fmul_rn(v, inv), 12582912.f));
}
__device__ __forceinline__ uint32_t codes4(float4 v, float inv)
{
    return __byte_perm(__byte_perm(code_bits(v.x, inv), code_bits(v.y, inv), 0x0040),
                       __byte_perm(code_bits(v.z, inv), code_bits(v.w, inv), 0x0040), 0x5410);
}

// X = Z * (s + sl), rounded once: fma(z, s, z * sl) (the factor is held as two floats).
__device__ __forceinline__ float4 scale4(float4 v, float2 s2, float2 sl2)
{
    const float2 a = make_float2(v.x, v.y), b = make_float2(v.z, v.w);
    const float2 lo = __ffma2_rn(a, s2, mul2_rn(a, sl2));
    const float2 hi = __ffma2_rn(b, s2, mul2_rn(b, sl2));
    return make_float4(lo.x, lo.y, hi.x, hi.y);
}

__device__ __forceinline__ float absmax4(float m, float4 v)
{
    return fmaxf(fmaxf(fmaxf(m, fabsf(v.x)), fabsf(v.y)), fmaxf(fabsf(v.z), fabsf(v.w)));
}

// 32-byte store (one full sector); `p` must be 32-byte aligned.
__device__ __forceinline__ void st_global_v8_b32(void *p, uint32_t a, uint32_t b, uint32_t c, uint32_t d,
                                                 uint32_t e, uint32_t f, uint32_t g, uint32_t h)
{
    asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};"
                 ::"l"(p), "r"(a), "r"(b), "r"(c), "r"(d), "r"(e), "r"(f), "r"(g), "r"(h)
                 : "memory");
}

__device__ __forceinline__ void cp_async_4(uint32_t dst, const void *src, bool valid)
{
    const int n = valid ? 4 : 0;   // 0 source bytes: the destination is zero filled
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst), "l"(src), "r"(n) : "memory");
}
__device__ __forceinline__ void cp_async_16(uint32_t dst, const void *src, bool valid)
{
    const int n = valid ? 16 : 0;
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(n) : "memory");
}
__device__ __forceinline__ void cp_async_commit()
{
    asm volatile("cp.async.commit_group;" ::: "memory");
}
template <int N>
__device__ __forceinline__ void cp_async_wait_group()   // all but the N newest groups are done
{
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// ---- strip staging -----------------------------------------------------------------
// smem column j of the strip holds image column w_base + j (w_base even); rows are
// image rows h_base .. h_base + NN - 1; anything outside the image is zero.
template <typename Tin, int NN>
__device__ __forceinline__ void stage_strip(Tin *sm, const Tin *__restrict__ x, const Geometry &g,
                                            const K1Params &prm, int img, int c_base, int h_base,
                                            int w_base)
{
    const size_t HW = (size_t)g.H * g.W;
    const Tin *ximg = x + ((size_t)img * g.C + c_base) * HW;
    // Each thread owns one (row, column) slot of the strip and walks over the channels,
    // so its bounds test and addresses are computed once.
    if (sizeof(Tin) == 2 && prm.vec16) {
        // 16-byte pieces: W and w_base are multiples of 8 and x is 16-byte aligned, so a piece
        // lies inside the image or outside it as a whole
        constexpr int CPR = K1_WPV / 8;                        // copies per row
        constexpr int ROWS = K1_THREADS / CPR;
        constexpr int CSLOTS = ROWS / NN;
        const int jc = threadIdx.x % CPR;
        const int rs = threadIdx.x / CPR;
        const int a = rs % NN, cslot = rs / NN;
        if (cslot < CSLOTS) {
            const int h = h_base + a, w = w_base + 8 * jc;
            const bool ok = h >= 0 && h < g.H && w >= 0 && w < g.W;
            const Tin *src = ok ? ximg + (size_t)cslot * HW + (size_t)h * g.W + w : x;
            const size_t src_step = ok ? (size_t)CSLOTS * HW : 0;
            uint32_t dst = static_cast<uint32_t>(__cvta_generic_to_shared(sm)) +
                           (uint32_t)((cslot * prm.CS + a * K1_WPV + 8 * jc) * sizeof(Tin));
            const uint32_t dst_step = (uint32_t)(CSLOTS * prm.CS * sizeof(Tin));
            for (int c = cslot; c < prm.CB; c += CSLOTS) {
                cp_async_16(dst, src, ok);
                src += src_step;
                dst += dst_step;
            }
        }
    } else if (sizeof(Tin) == 4 || prm.pair) {
        constexpr int EPC = sizeof(Tin) == 4 ? 1 : 2;          // elements per 4-byte copy
        constexpr int CPR = K1_WP / EPC;                       // copies per row
        constexpr int ROWS = K1_THREADS / CPR;                 // rows covered by one pass
        constexpr int CSLOTS = ROWS / NN;                      // channels covered by one pass
        const int jc = threadIdx.x % CPR;
        const int rs = threadIdx.x / CPR;
        const int a = rs % NN, cslot = rs / NN;
        if (cslot < CSLOTS) {
            const int h = h_base + a, w = w_base + EPC * jc;
            const bool ok = h >= 0 && h < g.H && w >= 0 && w < g.W;   // W even for pairs: both or none
            const Tin *src = ok ? ximg + (size_t)cslot * HW + (size_t)h * g.W + w : x;
            const size_t src_step = ok ? (size_t)CSLOTS * HW : 0;
            uint32_t dst = static_cast<uint32_t>(__cvta_generic_to_shared(sm)) +
                           (uint32_t)((cslot * prm.CS + a * K1_WP + EPC * jc) * sizeof(Tin));
            const uint32_t dst_step = (uint32_t)(CSLOTS * prm.CS * sizeof(Tin));
            for (int c = cslot; c < prm.CB; c += CSLOTS) {
                cp_async_4(dst, src, ok);
                src += src_step;
                dst += dst_step;
            }
        }
    } else {
        // fp16 with an odd W or a 2-byte aligned base: plain 2-byte loads, eight channels
        // in flight per thread (these copies are complete when the function returns)
        constexpr int ROWS = K1_THREADS / K1_WP;               // 8 row slots per pass
        constexpr int CSLOTS = ROWS / NN;                      // 1
        const int j = threadIdx.x % K1_WP;
        const int rs = threadIdx.x / K1_WP;
        const int a = rs % NN, cslot = rs / NN;
        if (cslot < CSLOTS) {
            const int h = h_base + a, w = w_base + j;
            const bool ok = h >= 0 && h < g.H && w >= 0 && w < g.W;
            const Tin *src = ximg + (size_t)cslot * HW + (size_t)h * g.W + w;
            Tin *dst = sm + cslot * prm.CS + a * K1_WP + j;
            for (int c = cslot; c < prm.CB; c += 8 * CSLOTS) {     // CB is a multiple of 32
                Tin v[8];
#pragma unroll
                for (int u = 0; u < 8; ++u) v[u] = ok ? __ldg(src + (size_t)u * CSLOTS * HW) : Tin(0);
#pragma unroll
                for (int u = 0; u < 8; ++u) dst[u * CSLOTS * prm.CS] = v[u];
                src += (size_t)8 * CSLOTS * HW;
                dst += 8 * CSLOTS * prm.CS;
            }
        }
    }
}

// ---- group abs-max and scale (the quantizer of Section 2, one scale per group) ------
// amax >= 0.  Returns the stored scale and the reciprocal used for the codes.
__device__ __forceinline__ void group_scale(float amax, float &scale, float &inv)
{
    const bool nz = amax >= 1e-30f;
    scale = nz ? __fdiv_rn(amax, 127.f) : 0.f;
    inv = nz ? __fdiv_rn(127.f, amax) : 0.f;
}

// ---- phase 2 of a work item: quantize, one (tile, group, position) per thread -------------
// Zs holds the transformed values of `ntile` tiles as [tile][position][CB + 4] fp32; the item is
// tiles tw0 .. of tile row `srow` (= image * TH + tile row) and channels c_base .. c_base + CB.
template <int P, int GSR, int SPLIT, bool SCALED = true>
__device__ __forceinline__ void quantize_item(const float *__restrict__ Zs, int CBP, int ntile, int ng, int gs,
                                              int srow, int tw0, int c_base, const Geometry &g,
                                              const InputScales &tab, int8_t *__restrict__ Xq,
                                              float *__restrict__ sX)
{
    // X = Z * (caller's per-position factor) is formed here, one rounding, as the
    // quantizer's input; then abs-max, scale, reciprocal and codes.
    const int g_base = c_base / gs;
    if constexpr (GSR > 0) {
        // whole warps walk the loop so that the lanes sharing a group can shuffle
        const int tasks = ntile * ng * P * SPLIT;
        for (int base = 0; base < tasks; base += K1_THREADS) {
            const int task = base + (int)threadIdx.x;
            const bool act = task < tasks;          // the lanes of a group are all in or all out
            const int tk = act ? task : 0;
            const int part = tk % SPLIT, rest = tk / SPLIT;
            const int q = rest / P, p = rest - q * P;
            const int tl = q >> (ng - 1), grp = q - tl * ng;        // one or two groups per item
            const int t = srow * g.TW + tw0 + tl;
            const float4 *src = reinterpret_cast<const float4 *>(Zs + (size_t)(tl * P + p) * CBP + grp * gs +
                                                                 part * GSR);
            int8_t *dst = Xq + ((size_t)p * g.T + t) * g.C + c_base + grp * gs + part * GSR;
            const float sp = tab.in_scale[p], sl = tab.in_scale_lo[p];
            const float2 sp2 = make_float2(sp, sp), sl2 = make_float2(sl, sl);
            float4 v[GSR / 4];
            float amax = 0.f;
#pragma unroll
            for (int k = 0; k < GSR / 4; ++k) {
                v[k] = SCALED ? scale4(src[k], sp2, sl2) : src[k];
                amax = absmax4(amax, v[k]);
            }
            if constexpr (SPLIT >= 2) amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, 1));
            if constexpr (SPLIT >= 4) amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, 2));
            float scale, inv;
            group_scale(amax, scale, inv);
            if (act) {
#pragma unroll
                for (int k = 0; k < GSR / 32; ++k)        // 32 codes = one full sector per store
                    st_global_v8_b32(dst + 32 * k, codes4(v[8 * k], inv), codes4(v[8 * k + 1], inv),
                                     codes4(v[8 * k + 2], inv), codes4(v[8 * k + 3], inv),
                                     codes4(v[8 * k + 4], inv), codes4(v[8 * k + 5], inv),
                                     codes4(v[8 * k + 6], inv), codes4(v[8 * k + 7], inv));
                if (part == 0) sX[((size_t)p * g.G + g_base + grp) * g.Ts + t] = scale;
            }
        }
    } else {
        const int tasks = ntile * ng * P;
        for (int task = threadIdx.x; task < tasks; task += K1_THREADS) {
            const int q = task / P, p = task - q * P;
            const int tl = q >> (ng - 1), grp = q - tl * ng;        // one or two groups per item
            const int t = srow * g.TW + tw0 + tl;
            const float4 *src = reinterpret_cast<const float4 *>(Zs + (size_t)(tl * P + p) * CBP + grp * gs);
            int8_t *dst = Xq + ((size_t)p * g.T + t) * g.C + c_base + grp * gs;
            const float sp = tab.in_scale[p], sl = tab.in_scale_lo[p];
            const float2 sp2 = make_float2(sp, sp), sl2 = make_float2(sl, sl);
            auto val = [&](int k) { return SCALED ? scale4(src[k], sp2, sl2) : src[k]; };
            float scale, inv;
            float amax = 0.f;
            for (int k = 0; k < gs / 4; ++k) amax = absmax4(amax, val(k));
            group_scale(amax, scale, inv);
            for (int k = 0; k < gs / 32; ++k)
                st_global_v8_b32(dst + 32 * k, codes4(val(8 * k), inv), codes4(val(8 * k + 1), inv),
                                 codes4(val(8 * k + 2), inv), codes4(val(8 * k + 3), inv),
                                 codes4(val(8 * k + 4), inv), codes4(val(8 * k + 5), inv),
                                 codes4(val(8 * k + 6), inv), codes4(val(8 * k + 7), inv));
            sX[((size_t)p * g.G + g_base + grp) * g.Ts + t] = scale;
        }
    }
}

}  // namespace
}  // namespace wfq
