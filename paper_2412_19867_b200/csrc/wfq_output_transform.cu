// Output transform y = V_A S_A Y S_A V_A^T (Section 4.1): one thread per
// (output channel, tile).  Lanes run along the tile index, so the P plane reads of
// Y[P][K][Tp] are 128-byte coalesced; the m-float row segments of neighbouring tiles are
// contiguous in y[N][K][H][W] and are written in whole sectors.  P*4 bytes read
// and m*m*4 bytes written per thread against ~150 flops.
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <type_traits>

#include "wfq_int_quant.cuh"
#include "wfq_internal.h"
#include "wfq_ptx.cuh"

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

// F(2,3), points 0, 1, -1, inf: V_A = [1,1,1,0; 0,1,-1,1] (the sign of the textbook's last column is
// in the standard S_A).
__device__ __forceinline__ void at_f23(const float (&v)[4], float (&o)[2])
{
    o[0] = v[0] + v[1] + v[2];
    o[1] = v[1] - v[2] + v[3];
}

// 1-D output transform with V_A = V_{n x m}^T for the points 0, 1, -1, 2, -2, inf:
//   o_u = sum_i f_i^u y_i (i < 5) + [u == 3] y_5
__device__ __forceinline__ void at_f43(const float (&v)[6], float (&o)[4])
{
    const float s1 = v[1] + v[2], d1 = v[1] - v[2];
    const float s2 = v[3] + v[4], d2 = v[3] - v[4];
    o[0] = v[0] + s1 + s2;
    o[1] = fmaf(2.f, d2, d1);
    o[2] = fmaf(4.f, s2, s1);
    o[3] = fmaf(8.f, d2, d1) + v[5];
}

// Points 0, 1, -1, 2, -2, 1/2, -1/2, inf.
__device__ __forceinline__ void at_f63(const float (&v)[8], float (&o)[6])
{
    const float s1 = v[1] + v[2], d1 = v[1] - v[2];
    const float s2 = v[3] + v[4], d2 = v[3] - v[4];
    const float s3 = v[5] + v[6], d3 = v[5] - v[6];
    o[0] = v[0] + s1 + s2 + s3;
    o[1] = fmaf(2.f, d2, d1) + 0.5f * d3;
    o[2] = fmaf(4.f, s2, s1) + 0.25f * s3;
    o[3] = fmaf(8.f, d2, d1) + 0.125f * d3;
    o[4] = fmaf(16.f, s2, s1) + 0.0625f * s3;
    o[5] = fmaf(32.f, d2, d1) + 0.03125f * d3 + v[7];
}

template <int M>
__device__ __forceinline__ void at_1d(const float (&v)[M + 2], float (&o)[M])
{
    if constexpr (M == 2) at_f23(v, o);
    else if constexpr (M == 4) at_f43(v, o);
    else at_f63(v, o);
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
        else if (act == 2) t = t * __frcp_rn(1.f + __expf(-t));   // exp overflow: t * 0
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
// consecutive floats (odd W).
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
            // float f of row u: tile f / M, column f % M
#pragma unroll
            for (int u = 0; u < M; ++u) {
                const float *row = out_s + u * TT * M;
#pragma unroll
                for (int i = 0; i < M; ++i) {
                    const int f = threadIdx.x + i * TT;
                    const int tj = f / M, v1 = f - tj * M;
                    const int lim = tile_lim[tj];
                    if (u < (lim >> 4) && v1 < (lim & 15)) {
                        const size_t off = (size_t)tile_base[tj] + (size_t)u * g.W + v1;
                        if (EPI && out_half) yh[off] = to_bits16(row[f], out_half);
                        else y[off] = row[f];
                    }
                }
            }
            return;
        }
        // pair q of row u: tile q / (M/2), columns 2 * (q % (M/2)) and the next
        constexpr int PPT = M / 2;                // pairs per tile row
#pragma unroll
        for (int u = 0; u < M; ++u) {
            const float2 *row = reinterpret_cast<const float2 *>(out_s + u * TT * M);
#pragma unroll
            for (int i = 0; i < PPT; ++i) {
                const int q = threadIdx.x + i * TT;
                const int tj = q / PPT, v2 = 2 * (q - tj * PPT);
                const int lim = tile_lim[tj];
                if (u < (lim >> 4) && v2 < (lim & 15)) {    // W even: both columns or none
                    const size_t off = (size_t)tile_base[tj] + (size_t)u * g.W + v2;
                    if (EPI && out_half) *reinterpret_cast<uint32_t *>(yh + off) = to_bits16x2(row[q].x, row[q].y, out_half);
                    else *reinterpret_cast<float2 *>(y + off) = row[q];
                }
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

// LOAD: how Y is loaded, 0 plain, 1 marked for early eviction from L2 (evict_early below), 2 as the flag says.
// flags: output type (0 fp32, 1 fp16, 2 bf16), plus kEarlyFlag.  One argument for both: a further one makes a launch
// longer (layers of 12.2 us that wait for launches 12.7 us).
constexpr int kEarlyFlag = 4;
template <int M, int STORE, bool EPI, int TT, int LOAD>
__global__ void __launch_bounds__(TT, (M == 6 ? (EPI ? 6 : 7) : 8) * 128 / TT)
output_transform_kernel(const float *__restrict__ Y, float *__restrict__ y, Geometry g,
                        ScaleTables tab, const float *__restrict__ bias, int act, int flags)
{
    constexpr int NN = M + 2;
    const int out_half = flags & (kEarlyFlag - 1);
    __shared__ __align__(16) StoreShared<M, STORE, TT> sm;
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    const int k = blockIdx.y;
    ptx::grid_dependency_wait();   // Y comes from the kernel launched before this one
    const bool live = t < g.T;
    if (STORE == 2 && !live) return;

    float tmp[M][NN];
    int h0 = 0, w0 = 0;
    size_t base = 0;
    if (live) {
        const size_t plane = (size_t)g.K * g.Tp;
        const float *src = Y + (size_t)k * g.Tp + t;
        float v[NN][NN];
        auto load = [&](auto one) {
#pragma unroll
            for (int i = 0; i < NN; ++i)
#pragma unroll
                for (int j = 0; j < NN; ++j) {
                    v[i][j] = one(src);
                    src += plane;
                }
        };
        if (LOAD == 1 || (LOAD == 2 && (flags & kEarlyFlag))) load([](const float *q) { return __ldcs(q); });
        else if (M == 6) load([](const float *q) { return __ldcg(q); });
        else load([](const float *q) { return __ldg(q); });
#pragma unroll
        for (int i = 0; i < NN; ++i)
#pragma unroll
            for (int j = 0; j < NN; ++j) v[i][j] *= tab.out_scale[i * NN + j];

        // columns: tmp[u][j] = sum_i VA[u][i] v[i][j]
#pragma unroll
        for (int j = 0; j < NN; ++j) {
            float col[NN], o[M];
#pragma unroll
            for (int i = 0; i < NN; ++i) col[i] = v[i][j];
            at_1d<M>(col, o);
#pragma unroll
            for (int u = 0; u < M; ++u) tmp[u][j] = o[u];
        }
        const int tw = t % g.TW;
        const int tq = t / g.TW;
        const int th = tq % g.TH;
        const int img = tq / g.TH;
        h0 = th * M;
        w0 = tw * M;
        base = (((size_t)img * g.K + k) * g.H + h0) * g.W + w0;
    }

    auto row_of = [&](int u, float (&o)[M]) { at_1d<M>(tmp[u], o); };
    store_tiles<M, STORE, EPI, TT>(row_of, sm, live, base, h0, w0, k, y, g, bias, act, out_half);
}

// ---- the fully quantized output transform (Eq. quant-y) ------------------------------------
//   y~ = s_qA^2 s_qY  Q(V_A S_A / s_qA)  Q(Y~ / s_qY) Q(S_A V_A^T / s_qA)
// one thread per (tile, output channel) as above, on integer codes; the results leave through the
// same stores.
// MODE 1: one scale per tile; MODE 2: one scale per row, then one per column.
template <int M, int STORE, int MODE, int TT>
__global__ void __launch_bounds__(TT)
output_transform_int_kernel(const float *__restrict__ Y, float *__restrict__ y, Geometry g,
                            const __grid_constant__ FullQuantTables tab, const float *__restrict__ bias, int act, int out_half)
{
    constexpr int NN = M + 2;
    __shared__ __align__(16) StoreShared<M, STORE, TT> sm;
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    const int k = blockIdx.y;
    ptx::grid_dependency_wait();   // Y comes from the kernel launched before this one
    const bool live = t < g.T;
    if (STORE == 2 && !live) return;
    const size_t plane = (size_t)g.K * g.Tp;
    const float *src = Y + (size_t)k * g.Tp + (live ? t : 0);
    float v[NN][NN];
#pragma unroll
    for (int i = 0; i < NN; ++i)
#pragma unroll
        for (int j = 0; j < NN; ++j) v[i][j] = src[(size_t)(i * NN + j) * plane];

    float out[M][M];
    if constexpr (MODE == 1) {
        float amax = 0.f;
#pragma unroll
        for (int i = 0; i < NN; ++i)
#pragma unroll
            for (int j = 0; j < NN; ++j) amax = fmaxf(amax, fabsf(v[i][j]));
        const double sqY = __ddiv_rn((double)amax, kIntQmax);
        const float rinv = __fdiv_rn(127.f, amax);
        int tmp[NN][M];         // Q(Y) Q(S_A V_A^T): [i][v]
#pragma unroll
        for (int i = 0; i < NN; ++i) {
            int q[NN];
#pragma unroll
            for (int j = 0; j < NN; ++j) q[j] = code_of_float(v[i][j], amax, rinv);
#pragma unroll
            for (int c = 0; c < M; ++c) {
                int s = 0;
#pragma unroll
                for (int j = 0; j < NN; ++j) s += q[j] * tab.ATq[c * NN + j];
                tmp[i][c] = s;
            }
        }
        const double sA2 = __dmul_rn(tab.sqA, tab.sqA);
#pragma unroll
        for (int u = 0; u < M; ++u)
#pragma unroll
            for (int c = 0; c < M; ++c) {
                int s = 0;
#pragma unroll
                for (int i = 0; i < NN; ++i) s += tab.ATq[u * NN + i] * tmp[i][c];
                out[u][c] = (float)__dmul_rn(__dmul_rn((double)s, sA2), sqY);
            }
    } else {
        double Z[NN][M];        // rows keep their scale: Q(Y_i) Q(S_A V_A^T) s_qA s_row(i)
#pragma unroll
        for (int i = 0; i < NN; ++i) {
            float amax = 0.f;
#pragma unroll
            for (int j = 0; j < NN; ++j) amax = fmaxf(amax, fabsf(v[i][j]));
            const double sr = __ddiv_rn((double)amax, kIntQmax);
            const float rinv = __fdiv_rn(127.f, amax);
            int q[NN];
#pragma unroll
            for (int j = 0; j < NN; ++j) q[j] = code_of_float(v[i][j], amax, rinv);
#pragma unroll
            for (int c = 0; c < M; ++c) {
                int s = 0;
#pragma unroll
                for (int j = 0; j < NN; ++j) s += q[j] * tab.ATq[c * NN + j];
                Z[i][c] = __dmul_rn(__dmul_rn((double)s, tab.sqA), sr);
            }
        }
#pragma unroll
        for (int c = 0; c < M; ++c) {
            double amax = 0.0;
#pragma unroll
            for (int i = 0; i < NN; ++i) amax = fmax(amax, fabs(Z[i][c]));
            const double sc = __ddiv_rn(amax, kIntQmax);
            const double rc = amax > 0.0 ? __ddiv_rn(1.0, sc) : 0.0;
            int q[NN];
#pragma unroll
            for (int i = 0; i < NN; ++i) q[i] = amax > 0.0 ? code_of(Z[i][c], sc, rc) : 0;
#pragma unroll
            for (int u = 0; u < M; ++u) {
                int s = 0;
#pragma unroll
                for (int i = 0; i < NN; ++i) s += tab.ATq[u * NN + i] * q[i];
                out[u][c] = (float)__dmul_rn(__dmul_rn((double)s, tab.sqA), sc);
            }
        }
    }

    const int tw = t % g.TW, th = (t / g.TW) % g.TH, img = t / (g.TW * g.TH);
    const int h0 = th * M, w0 = tw * M;
    const size_t base = (((size_t)img * g.K + k) * g.H + h0) * g.W + w0;
    auto row_of = [&](int u, float (&o)[M]) {
#pragma unroll
        for (int c = 0; c < M; ++c) o[c] = out[u][c];
    };
    store_tiles<M, STORE, true, TT>(row_of, sm, live, base, h0, w0, k, y, g, bias, act, out_half);
}

}  // namespace

namespace {

// F(6,3): CTAs of 64 tiles where they leave at least a twentieth fewer threads without a tile than CTAs
// of 128: 36 tiles of 1280 channels (forward 47.6 -> 45.7 us; of 640 with an epilogue 45.0 -> 38.7 us), 800
// tiles of 128 channels with an epilogue (36.4 -> 33.7 us), 162 of 256 (26.6 -> 25.9 us).  With about
// the same number of threads they are no better (121 tiles of 640 channels 41.2 -> 41.8 us, 3200 and 1600
// tiles within 0.3 us), and F(4,3) and F(2,3) gain nothing from them (32 tiles of 1280 channels 26.5 ->
// 26.8 us, 3136 tiles of 128 channels 23.9 -> 24.4 us).
bool half_ctas(const Geometry &g)
{
    const long long by64 = ((long long)g.T + 63) / 64 * 64, by128 = ((long long)g.T + 127) / 128 * 128;
    return g.m == 6 && 20 * by64 <= 19 * by128;
}

// How Y, which is read once, is loaded.  Marked for early eviction it leaves L2 before what the next kernels
// read.  That helps where Y takes a good part of the 126 MB of L2 (forward, F(6,3), plain -> marked: 33 MB 28.4 ->
// 28.1 us, 66 MB 47.5 -> 45.9 us, 98 MB 73.5 -> 69.1 us, 133 MB 92.4 -> 89.1 us; F(4,3) 47 MB 45.3 -> 44.5 us, 94 MB
// 77.2 -> 73.4 us; F(2,3) 51 MB 39.4 -> 38.5 us) and is no better or worse where it is small (20 MB 22.8 -> 23.0 us,
// 24 MB 25.3 -> 25.6 us).  With Y and y together beyond twice L2 most of Y has left by itself, and F(6,3) is better
// off without the mark (Y 199 MB with fp32 y 125.8 -> 127.5 us, 393 MB 227.6 -> 238.8 us; 199 MB with fp16 y, just below
// the limit, 127.2 -> 124.7 us); F(4,3) and F(2,3) are not (377 MB 131.4 -> 129.0 us, 336 MB 165.2 -> 158.3 us).
bool evict_early(const wfq_plan &plan)
{
    const Geometry &g = plan.geo;
    const size_t Y = (size_t)g.P * g.K * g.Tp * sizeof(float);
    const size_t y = (size_t)g.N * g.K * g.H * g.W * (plan.out_half ? 2 : 4);
    return Y >= (size_t)32 << 20 && (g.m != 6 || Y + y <= (size_t)256 << 20);
}
// With two forms of the loads in the kernel the compiler issues all of them before the arithmetic, which is faster
// than one form scheduled into it (forward, 600 tiles of 320 channels 35.5 -> 34.5 us, 243 of 128 14.2 -> 13.8 us, F(4,3)
// 2048 of 128 24.3 -> 24.0 us).  The F(6,3) variants with an epilogue have no registers for it (80 with 4 to 16 bytes
// spilled; 256 tiles of 1280 channels 80.9 us, with one form 75.8 us).
constexpr bool both_loads(int m, bool epi, int tt) { return tt == 128 && !(m == 6 && epi); }

template <int M, int STORE, bool EPI, int TT>
auto variant(bool early)
{
    if constexpr (both_loads(M, EPI, TT)) return output_transform_kernel<M, STORE, EPI, TT, 2>;
    else return early ? output_transform_kernel<M, STORE, EPI, TT, 1> : output_transform_kernel<M, STORE, EPI, TT, 0>;
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

// One-time attribute setting (per device): the staged variants want twelve or more half CTAs of
// 5-10 KB of shared memory per SM.
cudaError_t setup_output_transform()
{
    auto carveout = [](auto m, auto store, auto tt) {
        constexpr int M = decltype(m)::value, STORE = decltype(store)::value, TT = decltype(tt)::value;
        if (STORE == 2) return cudaSuccess;
        cudaError_t e = cudaSuccess;
        for (auto kern : {variant<M, STORE, false, TT>(false), variant<M, STORE, false, TT>(true),
                          variant<M, STORE, true, TT>(false), variant<M, STORE, true, TT>(true)})
            if (e == cudaSuccess)
                e = cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout,
                                         (int)cudaSharedmemCarveoutMaxShared);
        return e;
    };
    for (int m = 2; m <= 6; m += 2)
        for (int W : {1, 2})
            for (bool half : {false, true}) {
                const cudaError_t e = with_store(m, W, half, carveout);
                if (e != cudaSuccess) return e;
            }
    return cudaSuccess;
}

cudaError_t launch_output_transform(const wfq_plan &plan, float *y_dev, cudaStream_t stream, bool pdl)
{
    cudaLaunchAttribute attr[1];
    const cudaLaunchConfig_t cfg = output_config(plan, stream, pdl, attr);
    return with_store(plan.geo, [&](auto m, auto store, auto tt) {
        constexpr int M = decltype(m)::value, STORE = decltype(store)::value, TT = decltype(tt)::value;
        const bool epi = plan.bias || plan.act || plan.out_half, early = evict_early(plan);
        return cudaLaunchKernelEx(&cfg, epi ? variant<M, STORE, true, TT>(early) : variant<M, STORE, false, TT>(early),
                                  (const float *)plan.ws.Y, y_dev, plan.geo, plan.tables, plan.bias, plan.act,
                                  plan.out_half | (early ? kEarlyFlag : 0));
    });
}

cudaError_t launch_output_transform_int(const wfq_plan &plan, float *y_dev, cudaStream_t stream, bool pdl)
{
    cudaLaunchAttribute attr[1];
    const cudaLaunchConfig_t cfg = output_config(plan, stream, pdl, attr);
    return with_store(plan.geo, [&](auto m, auto store, auto tt) {
        constexpr int M = decltype(m)::value, STORE = decltype(store)::value, TT = decltype(tt)::value;
        return cudaLaunchKernelEx(&cfg, plan.fq_output == 1 ? output_transform_int_kernel<M, STORE, 1, TT>
                                                            : output_transform_int_kernel<M, STORE, 2, TT>,
                                  (const float *)plan.ws.Y, y_dev, plan.geo, plan.fq, plan.bias, plan.act, plan.out_half);
    });
}

}  // namespace wfq
