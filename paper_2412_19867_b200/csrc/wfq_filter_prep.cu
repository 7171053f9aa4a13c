// Offline filter path: W = S_G V_G w V_G^T S_G (Section 4.1) in fp64, one rounding to
// fp32, then group-wise int8 quantization along the input channels, stored
// position-major Wq[P][K][C] with scales sW[P][G][K], in one kernel.
#include <cmath>
#include <type_traits>

#include "wfq_internal.h"

namespace wfq {
namespace {

// Rows of V_{n x 3}: (f^0 g^2, f^1 g^1, f^2 g^0) for the points 0, 1, -1, 2, -2, [1/2, -1/2,] infinity;
// products of the filter scales.
struct FilterTables {
    double va[kMaxN], vb[kMaxN], vc[kMaxN];
    double ss[kMaxP];         // sG_i * sG_j at i * n + j
    float w_limit;            // |w| up to here: every transformed value is finite
};

// A warp handles one output channel and a run of CW input channels (whole groups: 128 channels for
// groups of 32 and 64, otherwise one group); a lane owns four neighbouring channels (eight, in two
// runs, for groups above 128), so that eight lanes are 32 channels.  Per row of n positions a lane
// transforms its channels in fp64, rounds once, and the eight lanes exchange their abs-max so that
// each ends up with that of one position: one scale and one reciprocal per lane instead of n, sent
// back by shuffles.  Codes leave as one word per lane (128 contiguous bytes per warp and position),
// the scales of the CTA's eight output channels through shared memory as whole sectors.
// Bound: latency of about ten dependent instructions per transformed value (3-4 of them fp64) at the 12 warps
// per SM that the filters of four channels in fp64 leave room for: 2.2 of 4 issue slots per cycle and SM are
// used.  Nothing but w, Wq and sW touches memory.  640 -> 1280 channels, F(6,3), groups of 64 (82 MB in and
// out, 13 us at 6.55 TB/s): 45 us alone, 47 us back to back.  Groups above 128 hold twice the filters per lane (two
// CTAs per SM, 28 bytes spilled): 1280 -> 640 channels, groups of 256, 64 us; groups of 160, whose second run of lanes
// is three quarters empty, 640 -> 1280 channels 92 us.  The former pair of kernels (one thread per filter, then one thread per group
// reading serially, through an fp32 array four times the size of Wq taken from the stream-ordered
// allocator) took 690 us, and 20 ms when the device was idle in between and the pool had been given back.
constexpr int FP_WARPS = 4;       // warps per CTA
constexpr int FP_KPW = 2;         // output channels per warp, one after the other
constexpr int FP_KB = FP_WARPS * FP_KPW;

template <int M, int Q>
__global__ void __launch_bounds__(32 * FP_WARPS, Q == 1 ? 3 : 2)
filter_prep_kernel(const float *__restrict__ w, int8_t *__restrict__ Wq, float *__restrict__ sW, int K, int C,
                   int gs, int k_pitch, int qmax, int vec_in, int word_out,
                   const __grid_constant__ FilterTables tab)
{
    constexpr int NN = M + 2, P = NN * NN;
    constexpr int CWMAX = 128 * Q;                              // channels a warp can hold
    __shared__ __align__(16) float w_s[FP_WARPS][CWMAX * 9];
    __shared__ float sc_s[P * 4][FP_KB];                        // [position, group of the run][output channel]
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int og = gs >> 5;                                     // runs of 32 channels per group
    const int gw = og == 1 ? 4 : og == 2 ? 2 : 1;               // groups per warp
    const int ncb = (C + gw * gs - 1) / (gw * gs);              // runs of CW channels
    const int kb = (int)blockIdx.x / ncb;
    const int c0 = ((int)blockIdx.x - kb * ncb) * (gw * gs);
    const int nch = min(gw * gs, C - c0);                       // whole groups
    const int k0 = kb * FP_KB;
    const float fq = (float)qmax;
    const size_t plane = (size_t)K * C;                         // codes per position

    for (int kk = 0; kk < FP_KPW; ++kk) {
        const int kl = warp * FP_KPW + kk, k = k0 + kl;
        if (k >= K) break;                                      // the whole warp
        const float *src = w + ((size_t)k * C + c0) * 9;
        __syncwarp();
        if (vec_in) {                                           // 16-byte aligned w: 32 channels are 72 pieces
            const float4 *s4 = reinterpret_cast<const float4 *>(src);
            float4 *d4 = reinterpret_cast<float4 *>(w_s[warp]);
            for (int i = lane; i < nch * 9 / 4; i += 32) d4[i] = __ldg(s4 + i);
        } else {
            for (int i = lane; i < nch * 9; i += 32) w_s[warp][i] = __ldg(src + i);
        }
        __syncwarp();

        double f[4 * Q][9];
        bool on[Q], finite = true;
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            const int cl = 128 * q + 4 * lane;                  // first of the lane's four channels
            on[q] = cl < nch;
            const float4 *s4 = reinterpret_cast<const float4 *>(w_s[warp] + (on[q] ? cl : 0) * 9);
            float v[36];
#pragma unroll
            for (int i = 0; i < 9; ++i) {
                const float4 t = on[q] ? s4[i] : make_float4(0.f, 0.f, 0.f, 0.f);
                v[4 * i] = t.x; v[4 * i + 1] = t.y; v[4 * i + 2] = t.z; v[4 * i + 3] = t.w;
            }
            float top = 0.f;
#pragma unroll
            for (int i = 0; i < 36; ++i) top = fmaxf(top, fabsf(v[i]));
#pragma unroll
            for (int i = 0; i < 36; ++i) finite = finite && v[i] == v[i];
            finite = finite && top <= tab.w_limit;
#pragma unroll
            for (int e = 0; e < 4; ++e)
#pragma unroll
                for (int i = 0; i < 9; ++i) f[4 * q + e][i] = (double)v[9 * e + i];
        }

        auto rows = [&](auto all_finite) {
            constexpr bool FINITE = decltype(all_finite)::value;
            int8_t *dst = Wq + (size_t)k * C + c0 + 4 * lane;
#pragma unroll 1
            for (int i = 0; i < NN; ++i) {
                const double a = tab.va[i], b = tab.vb[i], c = tab.vc[i];
                float v[4 * Q][NN];
                float m[8];
#pragma unroll
                for (int j = 0; j < 8; ++j) m[j] = 0.f;
#pragma unroll
                for (int e = 0; e < 4 * Q; ++e) {
                    // The factors are powers of two or zero: every product is exact, fused or not.
                    double t[3];                                // row i of V_G w
#pragma unroll
                    for (int col = 0; col < 3; ++col) t[col] = a * f[e][col] + b * f[e][3 + col] + c * f[e][6 + col];
#pragma unroll
                    for (int j = 0; j < NN; ++j) {              // times row j of V_G
                        const double p = j == 0 ? 0.0 : j == 1 ? 1.0 : j == 2 ? -1.0 : j == 3 ? 2.0 : j == 4 ? -2.0
                                       : j == 5 ? 0.5 : -0.5;
                        double u;
                        // products with zero carry an infinity or NaN along and are otherwise left out
                        if (j == NN - 1) u = FINITE ? t[2] : 0.0 * t[0] + 0.0 * t[1] + t[2];
                        else if (j == 0) u = FINITE ? t[0] : t[0] + 0.0 * t[1] + 0.0 * t[2];
                        else u = t[0] + p * t[1] + p * p * t[2];
                        v[e][j] = (float)(tab.ss[i * NN + j] * u);
                        m[j] = fmaxf(m[j], fabsf(v[e][j]));     // ignores NaN
                    }
                }
                // abs-max over the eight lanes of a run: each exchange halves the positions a lane keeps
                float m4[4], m2[2], amax;
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    m4[j] = fmaxf(lane & 4 ? m[j + 4] : m[j],
                                  __shfl_xor_sync(0xffffffffu, lane & 4 ? m[j] : m[j + 4], 4));
#pragma unroll
                for (int j = 0; j < 2; ++j)
                    m2[j] = fmaxf(lane & 2 ? m4[j + 2] : m4[j],
                                  __shfl_xor_sync(0xffffffffu, lane & 2 ? m4[j] : m4[j + 2], 2));
                amax = fmaxf(lane & 1 ? m2[1] : m2[0], __shfl_xor_sync(0xffffffffu, lane & 1 ? m2[0] : m2[1], 1));
                if (og >= 2) amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, 8));
                if (og >= 3) amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, 16));
                float scale = 0.f, inv = 0.f;                   // of position j = lane & 7
                if (amax >= 1e-30f) {
                    scale = __fdiv_rn(amax, fq);
                    inv = __fdiv_rn(fq, amax);
                }
                const int run = lane >> 3;
                const bool first = og == 1 ? true : og == 2 ? (run & 1) == 0 : run == 0;
                if (first && (lane & 7) < NN)
                    sc_s[(i * NN + (lane & 7)) * 4 + (og == 1 ? run : og == 2 ? run >> 1 : 0)][kl] = scale;
#pragma unroll
                for (int j = 0; j < NN; ++j) {
                    const float invj = __shfl_sync(0xffffffffu, inv, (lane & 24) | j);
#pragma unroll
                    for (int q = 0; q < Q; ++q) {
                        uint32_t b[4];
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            // round half to even by the addition of 1.5 * 2^23, |product| <= 127 up to
                            // rounding; inf * 0 and NaN give code 0
                            const float t = __fmul_rn(v[4 * q + e][j], invj);
                            b[e] = FINITE || t == t ? __float_as_uint(__fadd_rn(t, 12582912.f)) : 0u;
                        }
                        const uint32_t word = __byte_perm(__byte_perm(b[0], b[1], 0x0040),
                                                          __byte_perm(b[2], b[3], 0x0040), 0x5410);
                        if (on[q]) {
                            if (word_out) {
                                *reinterpret_cast<uint32_t *>(dst + 128 * q) = word;
                            } else {
#pragma unroll
                                for (int e = 0; e < 4; ++e) dst[128 * q + e] = (int8_t)(word >> (8 * e));
                            }
                        }
                    }
                    dst += plane;
                }
            }
        };
        // w_limit keeps every transformed value finite; anything else takes the careful variant
        if (__all_sync(0xffffffffu, finite)) rows(std::true_type{});
        else rows(std::false_type{});
    }
    __syncthreads();
    // scales: eight output channels of a (position, group) are one sector of sW (rows k_pitch floats apart)
    const int ng = nch / gs, G = C / gs, g0 = c0 / gs;
    for (int idx = threadIdx.x; idx < P * ng * FP_KB; idx += 32 * FP_WARPS) {
        const int kl = idx % FP_KB, r = idx / FP_KB;
        const int p = r / ng, gl = r - p * ng;
        if (k0 + kl < K) sW[((size_t)p * G + g0 + gl) * k_pitch + k0 + kl] = sc_s[p * 4 + gl][kl];
    }
}

// Wq[P][K][C], sW[P][G][k_pitch] from w[K][C][3][3]; no memory besides these.
cudaError_t run_filter_prep(const float *w, int8_t *Wq, float *sW, int K, int C, int m, int gs, int k_pitch, int qmax,
                            const double *sG, cudaStream_t stream)
{
    const int n = m + 2, og = gs / 32;
    static const double pts[7] = {0.0, 1.0, -1.0, 2.0, -2.0, 0.5, -0.5};
    FilterTables tab;
    for (int i = 0; i < n; ++i) {
        tab.va[i] = i < n - 1 ? 1.0 : 0.0;
        tab.vb[i] = i < n - 1 ? pts[i] : 0.0;
        tab.vc[i] = i < n - 1 ? pts[i] * pts[i] : 1.0;
    }
    double top = 0.0;
    for (int i = 0; i < n; ++i)
        for (int j = 0; j < n; ++j) {
            tab.ss[i * n + j] = sG[i] * sG[j];
            top = std::fmax(top, std::fabs(tab.ss[i * n + j]));
        }
    // a transformed value is at most (1 + 2 + 4)^2 |w| |sG_i sG_j| in magnitude, up to rounding
    tab.w_limit = (float)std::fmin(std::ldexp(1.0, 126) / (64.0 * top), 1e37);
    const int cw = og <= 2 ? 128 : gs;                          // input channels per warp
    const int vec_in = (reinterpret_cast<uintptr_t>(w) & 15u) == 0, word_out = (reinterpret_cast<uintptr_t>(Wq) & 3u) == 0;
    auto kern = og > 4 ? (m == 2 ? filter_prep_kernel<2, 2> : m == 4 ? filter_prep_kernel<4, 2> : filter_prep_kernel<6, 2>)
                       : (m == 2 ? filter_prep_kernel<2, 1> : m == 4 ? filter_prep_kernel<4, 1> : filter_prep_kernel<6, 1>);
    const unsigned grid = (unsigned)((C + cw - 1) / cw) * (unsigned)((K + FP_KB - 1) / FP_KB);
    kern<<<grid, 32 * FP_WARPS, 0, stream>>>(w, Wq, sW, K, C, gs, k_pitch, qmax, vec_in, word_out, tab);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_filter_prep(const wfq_plan &plan, const float *w_dev, cudaStream_t stream)
{
    const Geometry &g = plan.geo;
    return run_filter_prep(w_dev, plan.Wq, plan.sW, g.K, g.C, g.m, g.gs, g.Kp, plan.w_bits == 4 ? 7 : 127, plan.sG, stream);
}

// 4-bit filter codes of the exported blob: byte j = code 2j in the low nibble, code 2j+1 in the
// high nibble, two's complement.  One thread per 8 codes (two words in, one word out).
namespace {
__global__ void pack_nibbles_kernel(const uint2 *__restrict__ codes, uint32_t *__restrict__ packed, size_t words)
{
    const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= words) return;
    const uint2 c = codes[i];
    uint32_t out = 0;
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        out |= ((c.x >> (8 * e)) & 0xfu) << (4 * e);
        out |= ((c.y >> (8 * e)) & 0xfu) << (16 + 4 * e);
    }
    packed[i] = out;
}

__global__ void unpack_nibbles_kernel(const uint32_t *__restrict__ packed, uint2 *__restrict__ codes, size_t words)
{
    const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= words) return;
    const uint32_t w = packed[i];
    uint2 c = make_uint2(0u, 0u);
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        // sign extension of a nibble: shift it to the top of an int, arithmetic shift back
        const int lo = ((int)(w << (28 - 4 * e))) >> 28;
        const int hi = ((int)(w << (12 - 4 * e))) >> 28;
        c.x |= ((uint32_t)lo & 0xffu) << (8 * e);
        c.y |= ((uint32_t)hi & 0xffu) << (8 * e);
    }
    codes[i] = c;
}
}  // namespace

cudaError_t launch_pack_nibbles(const int8_t *codes, void *packed, size_t n_codes, cudaStream_t stream)
{
    const size_t words = n_codes / 8;
    if (words == 0) return cudaSuccess;
    pack_nibbles_kernel<<<(unsigned)((words + 255) / 256), 256, 0, stream>>>(
        reinterpret_cast<const uint2 *>(codes), static_cast<uint32_t *>(packed), words);
    return cudaGetLastError();
}

cudaError_t launch_unpack_nibbles(const void *packed, int8_t *codes, size_t n_codes, cudaStream_t stream)
{
    const size_t words = n_codes / 8;
    if (words == 0) return cudaSuccess;
    unpack_nibbles_kernel<<<(unsigned)((words + 255) / 256), 256, 0, stream>>>(
        static_cast<const uint32_t *>(packed), reinterpret_cast<uint2 *>(codes), words);
    return cudaGetLastError();
}

}  // namespace wfq

// ---- filter quantization into the caller's buffers, without any allocation ------------
extern "C" wfq_status_t wfq_quantize_filters_static(const float *w_dev, int K, int C, int m,
                                                    int group_size, const float *sG_host,
                                                    int8_t *wq_dev, float *sw_dev, void *stream)
{
    using namespace wfq;
    if (!w_dev || !wq_dev || !sw_dev) return WFQ_ERR_INVALID_ARG;
    if (K < 1 || C < 1 || m < 1 || group_size < 1) return WFQ_ERR_INVALID_ARG;
    if ((m != 2 && m != 4 && m != 6) || group_size % 32 != 0 || group_size > 256 || C % group_size != 0)
        return WFQ_ERR_UNSUPPORTED;
    const int n = m + 2, P = n * n;
    const unsigned long long need = (unsigned long long)P * (unsigned long long)K * (unsigned long long)C;
    if (need > WFQ_STATIC_SCRATCH_FLOATS) return WFQ_ERR_SCRATCH_TOO_SMALL;

    static const double std2[4] = {1.0, 0.5, 0.5, 1.0};
    static const double std4[6] = {1.0 / 4, -1.0 / 6, -1.0 / 6, 1.0 / 24, 1.0 / 24, 1.0};
    static const double std6[8] = {1.0, -2.0 / 9, -2.0 / 9, 1.0 / 90, 1.0 / 90, 32.0 / 45, 32.0 / 45, 1.0};
    double sG[kMaxN];
    for (int i = 0; i < n; ++i) {
        sG[i] = sG_host ? (double)sG_host[i] : (m == 2 ? std2[i] : m == 4 ? std4[i] : std6[i]);
        if (!std::isfinite(sG[i]) || sG[i] == 0.0) return WFQ_ERR_INVALID_ARG;
    }

    int device = -1;
    if (cudaGetDevice(&device) != cudaSuccess) return WFQ_ERR_CUDA;
    int major = 0;
    if (cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, device) != cudaSuccess)
        return WFQ_ERR_CUDA;
    if (major != 10) return WFQ_ERR_UNSUPPORTED;
    return run_filter_prep(w_dev, wq_dev, sw_dev, K, C, m, group_size, K, 127, sG,
                           reinterpret_cast<cudaStream_t>(stream)) == cudaSuccess ? WFQ_OK : WFQ_ERR_CUDA;
}
