// Output transform y = V_A S_A Y S_A V_A^T (Section 4.1): one thread per
// (output channel, tile).  Lanes run along the tile index, so the P plane reads of
// Y[P][K][Tp] are 128-byte coalesced; the m-float row segments of neighbouring tiles are
// contiguous in y[N][K][H][W] and are written in whole sectors.  P*4 bytes read
// and m*m*4 bytes written per thread against ~150 flops.
#include "wfq_internal.h"
#include "wfq_output_store.cuh"
#include "wfq_ptx.cuh"

namespace wfq {
namespace {

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

// LOAD: how Y is loaded, 0 plain, 1 marked for early eviction from L2 (evict_early below), 2 as the flag says.
// flags: output type (0 fp32, 1 fp16, 2 bf16), plus kEarlyFlag.  One argument for both: a further one makes a launch
// longer (layers of 12.2 us that wait for launches 12.7 us).
constexpr int kEarlyFlag = 4;
// F(6,3): registers for five CTAs of 128 tiles per SM (89 to 96) instead of seven (72; six with an epilogue, 80).  The
// 64 loads of a thread then stand further ahead of the arithmetic, and most layers are one wave of fewer CTAs anyway
// (forward, 36 tiles x 1280 channels 41.5 -> 40.6 us, 925 x 48 16.8 -> 16.0 us, 126 x 256 16.5 -> 16.2 us; several waves,
// 3200 x 64, 40.1 -> 40.2 us).  Four CTAs (125 registers) are no better, nor are six for F(4,3).
template <int M, int STORE, bool EPI, int TT, int LOAD>
__global__ void __launch_bounds__(TT, (M == 6 ? 5 : 8) * 128 / TT)
output_transform_kernel(const float *__restrict__ Y, float *__restrict__ y, Geometry g,
                        OutputScales tab, const float *__restrict__ bias, int act, int flags)
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
        const int tq = t / g.by_TW, img = tq / g.by_TH;
        h0 = (tq - img * g.TH) * M;
        w0 = (t - tq * g.TW) * M;
        base = (((size_t)img * g.K + k) * g.H + h0) * g.W + w0;
    }

    auto row_of = [&](int u, float (&o)[M]) { at_1d<M>(tmp[u], o); };
    store_tiles<M, STORE, EPI, TT>(row_of, sm, live, base, h0, w0, k, y, g, bias, act, out_half);
}

}  // namespace

namespace {

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
// 2048 of 128 24.3 -> 24.0 us).  The F(6,3) variants with an epilogue are better off with one form (1600 tiles of 128
// channels 34.4 us, with two 35.4 us).
constexpr bool both_loads(int m, bool epi, int tt) { return tt == 128 && !(m == 6 && epi); }

template <int M, int STORE, bool EPI, int TT>
auto variant(bool early)
{
    if constexpr (both_loads(M, EPI, TT)) return output_transform_kernel<M, STORE, EPI, TT, 2>;
    else return early ? output_transform_kernel<M, STORE, EPI, TT, 1> : output_transform_kernel<M, STORE, EPI, TT, 0>;
}

}  // namespace

// One-time attribute setting (per device): the staged variants want twelve or more half CTAs of
// 5-10 KB of shared memory per SM.  (The integer kernels, fewer per SM because of their registers, are up to 7 %
// slower with the same attribute.)
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

}  // namespace wfq
