// Fused input transform + group-wise int8 quantization.
//
//   X = S_B V_B x V_B^T S_B   (Section 4.1), fp32, never stored to global memory
//   per (position, tile, channel group): amax -> scale, codes (Section 2 quantizer,
//   one scale per group, dynamic abs-max)
//
// A work item is TB neighbouring tiles of one tile row and CB input channels (one or two
// whole groups); persistent CTAs walk over the items.  Per item, separated by block
// barriers (where shared memory allows it without costing a resident CTA, the next
// item's strip is staged into a second buffer while this one is processed):
//   stage    the zero-padded input strip (n rows x 16 columns x CB channels) goes to
//            shared memory with 4-byte cp.async copies, all in flight at once
//   phase 1  thread <-> (tile, channel): the n x n patch is transformed with the
//            standard-scaled B^T (small integers / dyadic rationals as add/fma chains)
//            and written as fp32 to a shared [tile][position][channel] array (lanes
//            along the channel: conflict free)
//   phase 2  thread <-> (tile, group, position): it reads the group's values of that
//            position with 16-byte loads (rows 4 floats longer than the channel block:
//            conflict free), multiplies them by the caller's per-position factor, takes
//            the abs-max serially, derives scale and reciprocal once, rounds with the
//            1.5*2^23 trick (same result as mul + round-half-even convert; scalar multiply
//            and add, each rounded) and stores 32 codes per 32-byte store.
// The abs-max over a group of up to 64 channels therefore needs no shuffles; groups of 128
// or 256 channels are shared by two or four neighbouring lanes (64 channels each, one or two
// shuffles for the abs-max); other group sizes read shared memory twice instead of holding
// the group in registers.
#include <cuda_fp16.h>

#include "wfq_internal.h"
#include "wfq_ptx.cuh"
#include "wfq_strip.cuh"

namespace wfq {
namespace {

// ---- 1-D input transforms with the standard B^T ------------------------------------

// F(2,3) (the textbook matrices): rows [1,0,-1,0] [0,1,1,0] [0,-1,1,0] [0,1,0,-1]
__device__ __forceinline__ void bt_1d(const float (&d)[4], float (&r)[4])
{
    r[0] = d[0] - d[2];
    r[1] = d[1] + d[2];
    r[2] = d[2] - d[1];
    r[3] = d[1] - d[3];
}

// F(4,3): rows [4,0,-5,0,1,0] [0,-4,-4,1,1,0] [0,4,-4,-1,1,0] [0,-2,-1,2,1,0]
//              [0,2,-1,-2,1,0] [0,4,0,-5,0,1]
__device__ __forceinline__ void bt_1d(const float (&d)[6], float (&r)[6])
{
    r[0] = fmaf(4.f, d[0], fmaf(-5.f, d[2], d[4]));
    const float a = fmaf(-4.f, d[2], d[4]);
    const float b = fmaf(-4.f, d[1], d[3]);
    r[1] = a + b;
    r[2] = a - b;
    const float c = d[4] - d[2];
    const float t = d[3] - d[1];
    r[3] = fmaf(2.f, t, c);
    r[4] = fmaf(-2.f, t, c);
    r[5] = fmaf(4.f, d[1], fmaf(-5.f, d[3], d[5]));
}

// F(6,3): rows [1,0,-21/4,0,21/4,0,-1,0] [0,1,1,-17/4,-17/4,1,1,0]
//   [0,-1,1,17/4,-17/4,-1,1,0] [0,1/2,1/4,-5/2,-5/4,2,1,0] [0,-1/2,1/4,5/2,-5/4,-2,1,0]
//   [0,2,4,-5/2,-5,1/2,1,0] [0,-2,4,5/2,-5,-1/2,1,0] [0,-1,0,21/4,0,-21/4,0,1]
__device__ __forceinline__ void bt_1d(const float (&d)[8], float (&r)[8])
{
    r[0] = fmaf(5.25f, d[4] - d[2], d[0] - d[6]);
    r[7] = fmaf(5.25f, d[3] - d[5], d[7] - d[1]);
    const float a = fmaf(-4.25f, d[4], d[2] + d[6]);
    const float b = fmaf(-4.25f, d[3], d[1] + d[5]);
    r[1] = a + b;
    r[2] = a - b;
    const float c = fmaf(-1.25f, d[4], fmaf(0.25f, d[2], d[6]));
    const float e = fmaf(2.f, d[5], fmaf(-2.5f, d[3], 0.5f * d[1]));
    r[3] = c + e;
    r[4] = c - e;
    const float f = fmaf(-5.f, d[4], fmaf(4.f, d[2], d[6]));
    const float g = fmaf(0.5f, d[5], fmaf(-2.5f, d[3], 2.f * d[1]));
    r[5] = f + g;
    r[6] = f - g;
}

// The same two transforms on two columns at once (packed f32x2 arithmetic: one
// instruction per pair, each component rounded as in the scalar form).
__device__ __forceinline__ float2 f2(float v) { return make_float2(v, v); }

__device__ __forceinline__ void bt_1d(const float2 (&d)[4], float2 (&r)[4])
{
    r[0] = __ffma2_rn(f2(-1.f), d[2], d[0]);
    r[1] = __fadd2_rn(d[1], d[2]);
    r[2] = __ffma2_rn(f2(-1.f), d[1], d[2]);
    r[3] = __ffma2_rn(f2(-1.f), d[3], d[1]);
}

__device__ __forceinline__ void bt_1d(const float2 (&d)[6], float2 (&r)[6])
{
    r[0] = __ffma2_rn(f2(4.f), d[0], __ffma2_rn(f2(-5.f), d[2], d[4]));
    const float2 a = __ffma2_rn(f2(-4.f), d[2], d[4]);
    const float2 b = __ffma2_rn(f2(-4.f), d[1], d[3]);
    r[1] = __fadd2_rn(a, b);
    r[2] = __ffma2_rn(f2(-1.f), b, a);
    const float2 c = __ffma2_rn(f2(-1.f), d[2], d[4]);
    const float2 t = __ffma2_rn(f2(-1.f), d[1], d[3]);
    r[3] = __ffma2_rn(f2(2.f), t, c);
    r[4] = __ffma2_rn(f2(-2.f), t, c);
    r[5] = __ffma2_rn(f2(4.f), d[1], __ffma2_rn(f2(-5.f), d[3], d[5]));
}

__device__ __forceinline__ void bt_1d(const float2 (&d)[8], float2 (&r)[8])
{
    r[0] = __ffma2_rn(f2(5.25f), __ffma2_rn(f2(-1.f), d[2], d[4]), __ffma2_rn(f2(-1.f), d[6], d[0]));
    r[7] = __ffma2_rn(f2(5.25f), __ffma2_rn(f2(-1.f), d[5], d[3]), __ffma2_rn(f2(-1.f), d[1], d[7]));
    const float2 a = __ffma2_rn(f2(-4.25f), d[4], __fadd2_rn(d[2], d[6]));
    const float2 b = __ffma2_rn(f2(-4.25f), d[3], __fadd2_rn(d[1], d[5]));
    r[1] = __fadd2_rn(a, b);
    r[2] = __ffma2_rn(f2(-1.f), b, a);
    const float2 c = __ffma2_rn(f2(-1.25f), d[4], __ffma2_rn(f2(0.25f), d[2], d[6]));
    const float2 e = __ffma2_rn(f2(2.f), d[5], __ffma2_rn(f2(-2.5f), d[3], __fmul2_rn(f2(0.5f), d[1])));
    r[3] = __fadd2_rn(c, e);
    r[4] = __ffma2_rn(f2(-1.f), e, c);
    const float2 f = __ffma2_rn(f2(-5.f), d[4], __ffma2_rn(f2(4.f), d[2], d[6]));
    const float2 g = __ffma2_rn(f2(0.5f), d[5], __ffma2_rn(f2(-2.5f), d[3], __fmul2_rn(f2(2.f), d[1])));
    r[5] = __fadd2_rn(f, g);
    r[6] = __ffma2_rn(f2(-1.f), g, f);
}

__device__ __forceinline__ float to_float32(float v) { return v; }
__device__ __forceinline__ float to_float32(__half v) { return __half2float(v); }

// Z = B^T d B with the standard B^T, written to out[p * pitch] for p = i*NN + j.
template <int NN>
__device__ __forceinline__ void transform_patch(float (&d)[NN][NN], float *__restrict__ out, int pitch)
{
#pragma unroll
    for (int b = 0; b < NN; b += 2) {   // columns, two at a time: d <- B^T d
        float2 col[NN], r[NN];
#pragma unroll
        for (int a = 0; a < NN; ++a) col[a] = make_float2(d[a][b], d[a][b + 1]);
        bt_1d(col, r);
#pragma unroll
        for (int a = 0; a < NN; ++a) {
            d[a][b] = r[a].x;
            d[a][b + 1] = r[a].y;
        }
    }
#pragma unroll
    for (int i = 0; i < NN; ++i) {   // rows: Z[i][:] = (B^T d)[i][:] B
        float r[NN];
        bt_1d(d[i], r);
#pragma unroll
        for (int j = 0; j < NN; ++j) out[(i * NN + j) * pitch] = r[j];
    }
}

// ---- the kernel ----------------------------------------------------------------------
// GSR > 0: channels a thread holds in registers during phase 2 (32 or 64); a group is GSR *
// SPLIT channels, SPLIT neighbouring lanes share it and exchange their abs-max by shuffle.
// GSR == 0: any group size, one thread per group, phase 2 reads shared memory twice.
template <int M, typename Tin, int GSR, int SPLIT>
__global__ void __launch_bounds__(K1_THREADS, 4)
input_transform_kernel(const Tin *__restrict__ x, int8_t *__restrict__ Xq,
                       float *__restrict__ sX, Geometry g, InputScales tab, K1Params prm)
{
    constexpr int NN = M + 2;
    constexpr int P = NN * NN;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    // This kernel is launched with programmatic stream serialization: it may become
    // resident while the kernel before it in the stream (normally the previous layer's output
    // transform) drains, and waits here, before its first global access, until that kernel has
    // completed and its writes are visible.
    ptx::grid_dependency_wait();
    // The contraction kernel launched behind this one may start its prologue and its filter
    // stream now (it waits for this grid's completion before it touches Xq or sX).  Not before the
    // wait: the kernel in front of this one may be the filter preparation, whose codes that stream
    // reads.  The order costs nothing on the whole (forward, 60 layers: 0.4 % less time than the other way
    // round, between 4 % less and 1 % more: 28x28 NHWC 36.4 -> 35.2 us, 784 tiles x 320 channels 33.3 -> 33.5 us).
    ptx::grid_launch_dependents();
    // two strip buffers (the next item is staged while this one is transformed), then Z
    float *Zs = reinterpret_cast<float *>(smem_raw + (1 + prm.dbuf) * prm.strip_bytes);   // [tile][position][CBP]
    const int CBP = prm.CB + 4;   // 16-byte aligned rows an odd number of 16-byte units apart

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    constexpr int NWARP = K1_THREADS / 32;
    const int cb32 = prm.CB >> 5;
    const int gs = GSR > 0 ? GSR * SPLIT : g.gs;
    const int ng = prm.CB / gs;

    // item -> (tile row, chunk of tiles, channel block); channel blocks vary fastest so
    // that CTAs running side by side read the same image rows
    auto stage_item = [&](int item, int buf) {
        const int rest = item / prm.by_NCB, cblk = item - rest * prm.NCB;
        const int srow = rest / prm.by_NCH, chunk = rest - srow * prm.NCH;
        const int img = srow / g.by_TH, th = srow - img * g.TH;
        // first staged column: two left of the first tile's first output column, or (16-byte
        // pieces) the multiple of 8 at or below the first input column
        const int first = chunk * prm.TB * M - 1;
        const int w_base = prm.vec16 ? ((first + 8) & ~7) - 8 : first - 1;
        stage_strip<Tin, NN>(reinterpret_cast<Tin *>(smem_raw + buf * prm.strip_bytes), x, g, prm, img,
                             cblk * prm.CB, th * M - 1, w_base);
        cp_async_commit();
    };

    int item = blockIdx.x;
    if (item < prm.items) stage_item(item, 0);
    for (int it = 0; item < prm.items; ++it, item += gridDim.x) {
        const int buf = prm.dbuf ? (it & 1) : 0;
        const int next = item + gridDim.x;
        if (!prm.dbuf) {
            // one buffer: this item's copies were issued after the previous item's patches had been
            // read (below), and landed while that item was quantized
            cp_async_wait_group<0>();
        } else if (next < prm.items) {
            stage_item(next, buf ^ 1);
            cp_async_wait_group<1>();          // this item's copies have landed
        } else {
            cp_async_wait_group<0>();
        }
        __syncthreads();

        const Tin *strip = reinterpret_cast<const Tin *>(smem_raw + buf * prm.strip_bytes);
        const int rest = item / prm.by_NCB, cblk = item - rest * prm.NCB;
        const int srow = rest / prm.by_NCH, chunk = rest - srow * prm.NCH;   // srow = img*TH + th
        const int tw0 = chunk * prm.TB;
        const int ntile = min(prm.TB, g.TW - tw0);
        const int c_base = cblk * prm.CB;

        // ---- phase 1: transform, one (tile, channel) per thread ----------------------
        const int voff = tw0 * M - 2 - (((tw0 * M - 1 + 8) & ~7) - 8);   // 16-byte pieces: column of tile 0 minus one
        for (int wt = warp; wt < ntile * cb32; wt += NWARP) {
            const int tl = wt / prm.by_cb32;
            const int c = (wt - tl * cb32) * 32 + lane;
            float d[NN][NN];
            if (sizeof(Tin) == 2 && prm.vec16) load_patch_vec<NN>(strip + c * prm.CS, tl * M + voff, d);
            else load_patch<NN>(strip + c * prm.CS, tl * M, d);
            transform_patch<NN>(d, Zs + (size_t)tl * P * CBP + c, CBP);
        }
        __syncthreads();
        if (!prm.dbuf && next < prm.items) stage_item(next, 0);   // the strip buffer is free: refill it now

        quantize_item<P, GSR, SPLIT>(Zs, CBP, ntile, ng, gs, srow, tw0, c_base, g, tab, Xq, sX);
        __syncthreads();   // Z and this strip buffer are free again
    }
}

// ---- the same for an NHWC input ---------------------------------------------------------
// x[N][H][W][C]: the channels are innermost, so the strip of a work item is one 4-D TMA box
// {CB channels, TB * m + 2 columns, n rows, 1 image} (zero fill outside the image, no alignment
// condition on the row or column it starts at) and lands as [row][column][channel]; a thread
// reads its patch with the lanes along the channels (no bank conflicts, no realignment).  One
// thread issues the copy of an item as soon as the buffer it goes to has been read; everything
// else is the kernel above: transform, [tile][position][channel] array, quantize_item.
struct K1NhwcShared {
    uint64_t full[2];        // the strip of a buffer has landed
    volatile int abort;
};

template <int M, typename Tin, int GSR, int SPLIT>
__global__ void __launch_bounds__(K1_THREADS, 4)
input_transform_nhwc_kernel(const __grid_constant__ CUtensorMap tmx, int8_t *__restrict__ Xq,
                            float *__restrict__ sX, Geometry g, InputScales tab, K1Params prm, int *status,
                            long long wait_cycles)
{
    constexpr int NN = M + 2;
    constexpr int P = NN * NN;
    extern __shared__ __align__(16) unsigned char smem_dyn[];
    __shared__ K1NhwcShared sh;
    // a TMA destination must be 128-byte aligned; the dynamic part starts wherever the static part
    // ends, so the strips start at the next multiple of 128 (the launch adds 128 bytes for this)
    unsigned char *smem_raw = ptx::align_smem<128>(smem_dyn);
    ptx::grid_dependency_wait();
    ptx::grid_launch_dependents();
    float *Zs = reinterpret_cast<float *>(smem_raw + (1 + prm.dbuf) * prm.strip_bytes);   // [tile][position][CBP]
    const int CBP = prm.CB + 4;
    const int WB = prm.TB * M + 2;                     // columns of the box
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    constexpr int NWARP = K1_THREADS / 32;
    const int cb32 = prm.CB >> 5;
    const int gs = GSR > 0 ? GSR * SPLIT : g.gs;
    const int ng = prm.CB / gs;
    const WaitCtx ctx{&sh.abort, status, wait_cycles};
    const uint32_t box_bytes = (uint32_t)(NN * WB * prm.CB * (int)sizeof(Tin));

    if (threadIdx.x == 0) {
        ptx::mbar_init(ptx::smem_u32(&sh.full[0]), 1);
        ptx::mbar_init(ptx::smem_u32(&sh.full[1]), 1);
        sh.abort = 0;
        ptx::fence_mbar_init();
        ptx::prefetch_tmap(&tmx);
    }
    __syncthreads();

    // thread 0 only
    auto issue = [&](int item, int buf) {
        const int rest = item / prm.by_NCB, cblk = item - rest * prm.NCB;
        const int srow = rest / prm.by_NCH, chunk = rest - srow * prm.NCH;
        const int img = srow / g.by_TH, th = srow - img * g.TH;
        const uint32_t bar = ptx::smem_u32(&sh.full[buf]);
        ptx::mbar_arrive_expect_tx(bar, box_bytes);
        ptx::tma_load_4d(ptx::smem_u32(smem_raw + buf * prm.strip_bytes), &tmx, bar, cblk * prm.CB,
                         chunk * prm.TB * M - 1, th * M - 1, img);
    };

    const int stride = (int)gridDim.x;
    int item = blockIdx.x;
    int issued = 0;                                     // items whose copy has been issued (thread 0)
    if (threadIdx.x == 0) {
        if (item < prm.items) { issue(item, 0); ++issued; }
        if (prm.dbuf && item + stride < prm.items) { issue(item + stride, 1); ++issued; }
    }
    bool ok = true;
    int it = 0;
    for (; item < prm.items; ++it, item += stride) {
        const int buf = prm.dbuf ? (it & 1) : 0;
        const uint32_t parity = (uint32_t)(prm.dbuf ? (it >> 1) : it) & 1u;
        ok = wait_warp(ptx::smem_u32(&sh.full[buf]), parity, ctx, kWaitStripFull);
        if (!ok) break;

        const Tin *strip = reinterpret_cast<const Tin *>(smem_raw + buf * prm.strip_bytes);
        const int rest = item / prm.by_NCB, cblk = item - rest * prm.NCB;
        const int srow = rest / prm.by_NCH, chunk = rest - srow * prm.NCH;
        const int tw0 = chunk * prm.TB;
        const int ntile = min(prm.TB, g.TW - tw0);
        const int c_base = cblk * prm.CB;

        // ---- phase 1: transform, one (tile, channel) per thread ----------------------
        for (int wt = warp; wt < ntile * cb32; wt += NWARP) {
            const int tl = wt / prm.by_cb32;
            const int c = (wt - tl * cb32) * 32 + lane;
            float d[NN][NN];
            const Tin *src = strip + (size_t)(tl * M) * prm.CB + c;
#pragma unroll
            for (int a = 0; a < NN; ++a)
#pragma unroll
                for (int b = 0; b < NN; ++b) d[a][b] = to_float32(src[(a * WB + b) * prm.CB]);
            transform_patch<NN>(d, Zs + (size_t)tl * P * CBP + c, CBP);
        }
        __syncthreads();
        // the strip buffer has been read: the item that uses it next may be copied now
        if (threadIdx.x == 0) {
            const int nxt = item + (prm.dbuf ? 2 : 1) * stride;
            if (nxt < prm.items) { issue(nxt, buf); ++issued; }
        }
        quantize_item<P, GSR, SPLIT>(Zs, CBP, ntile, ng, gs, srow, tw0, c_base, g, tab, Xq, sX);
        __syncthreads();   // Z is free again
    }
    if (!ok && threadIdx.x == 0) {
        // a copy never arrived: give the ones still in flight a bounded time to land before the
        // shared memory goes away (copies issued: `issued`, consumed: `it`)
        for (int k = it; k < issued; ++k) {
            const int b = prm.dbuf ? (k & 1) : 0;
            drain(ptx::smem_u32(&sh.full[b]), (uint32_t)(prm.dbuf ? (k >> 1) : k) & 1u);
        }
    }
}

// Resident CTAs per SM and the attribute calls need the kernel symbol: one entry per
// instantiation.
template <int M, typename Tin, int GSR, int SPLIT>
int k1_resident(size_t smem)
{
    return resident_ctas_per_sm(input_transform_kernel<M, Tin, GSR, SPLIT>, K1_THREADS, smem, 32);
}

template <int M, typename Tin, int GSR, int SPLIT>
cudaError_t k1_setup()
{
    auto kern = input_transform_kernel<M, Tin, GSR, SPLIT>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
    if (e != cudaSuccess) return e;
    return cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout,
                                (int)cudaSharedmemCarveoutMaxShared);
}

template <int M, typename Tin, int GSR, int SPLIT>
cudaError_t launch_k1(const wfq_plan &plan, const void *x_dev, cudaStream_t stream)
{
    // 16-byte pieces need a 16-byte aligned x; the plan holds a second parameter set without them
    const bool vec = plan.k1v.vec16 && plan.k1_choice != 3 && (reinterpret_cast<uintptr_t>(x_dev) & 15u) == 0;
    const K1Params &prm = vec ? plan.k1v : plan.k1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)prm.grid);
    cfg.blockDim = dim3(K1_THREADS);
    cfg.dynamicSmemBytes = prm.smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, input_transform_kernel<M, Tin, GSR, SPLIT>, static_cast<const Tin *>(x_dev),
                              plan.ws.Xq, plan.ws.sX, plan.geo, plan.tables, prm);
}

template <int M, typename Tin, int GSR, int SPLIT>
int k1n_resident(size_t smem)
{
    return resident_ctas_per_sm(input_transform_nhwc_kernel<M, Tin, GSR, SPLIT>, K1_THREADS, smem, 32);
}

template <int M, typename Tin, int GSR, int SPLIT>
cudaError_t k1n_setup()
{
    auto kern = input_transform_nhwc_kernel<M, Tin, GSR, SPLIT>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, 226 * 1024);
    if (e != cudaSuccess) return e;
    return cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout,
                                (int)cudaSharedmemCarveoutMaxShared);
}

template <int M, typename Tin, int GSR, int SPLIT>
cudaError_t launch_k1n(const wfq_plan &plan, cudaStream_t stream)
{
    const K1Params &prm = plan.k1n;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)prm.grid);
    cfg.blockDim = dim3(K1_THREADS);
    cfg.dynamicSmemBytes = prm.smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, input_transform_nhwc_kernel<M, Tin, GSR, SPLIT>, plan.tmap_xn, plan.ws.Xq,
                              plan.ws.sX, plan.geo, plan.tables, prm, plan.status, plan.wait_cycles);
}

// What to do with the instantiation that serves (m, dtype, group size).
enum K1Op { kK1Launch, kK1Resident, kK1Setup, kK1nLaunch, kK1nResident, kK1nSetup };

template <int M, typename Tin>
long long k1_by_gs(K1Op op, int gs, const wfq_plan *plan, const void *x, cudaStream_t s, size_t smem)
{
#define WFQ_K1_CASE(GSR, SPLIT)                                                        \
    switch (op) {                                                                      \
        case kK1Launch: return (long long)launch_k1<M, Tin, GSR, SPLIT>(*plan, x, s);  \
        case kK1Resident: return k1_resident<M, Tin, GSR, SPLIT>(smem);                \
        case kK1Setup: return (long long)k1_setup<M, Tin, GSR, SPLIT>();               \
        case kK1nLaunch: return (long long)launch_k1n<M, Tin, GSR, SPLIT>(*plan, s);   \
        case kK1nResident: return k1n_resident<M, Tin, GSR, SPLIT>(smem);              \
        default: return (long long)k1n_setup<M, Tin, GSR, SPLIT>();                    \
    }
    if (gs == 32) { WFQ_K1_CASE(32, 1) }
    if (gs == 64) { WFQ_K1_CASE(64, 1) }
    if (gs == 128) { WFQ_K1_CASE(64, 2) }
    if (gs == 256) { WFQ_K1_CASE(64, 4) }
    WFQ_K1_CASE(0, 1)
#undef WFQ_K1_CASE
}

long long k1_op(K1Op op, int m, bool f16, int gs, const wfq_plan *plan, const void *x, cudaStream_t s,
                size_t smem)
{
    if (m == 2)
        return f16 ? k1_by_gs<2, __half>(op, gs, plan, x, s, smem) : k1_by_gs<2, float>(op, gs, plan, x, s, smem);
    if (m == 4)
        return f16 ? k1_by_gs<4, __half>(op, gs, plan, x, s, smem) : k1_by_gs<4, float>(op, gs, plan, x, s, smem);
    return f16 ? k1_by_gs<6, __half>(op, gs, plan, x, s, smem) : k1_by_gs<6, float>(op, gs, plan, x, s, smem);
}

}  // namespace

void plan_k1(wfq_plan &plan, K1Params &prm, bool vec16, ResidentFn resident_of)
{
    const Geometry &g = plan.geo;
    const bool f16 = plan.in_dtype == WFQ_F16;
    const int NN = g.n, P = g.P, M = g.m;
    const int esz = f16 ? 2 : 4;
    prm.vec16 = vec16 ? 1 : 0;
    prm.TB = (K1_WP - 3) / M;                      // 2 tiles for F(6,3), 3 for F(4,3)
    prm.CB = g.gs;
    if (g.gs == 32 && g.C % 64 == 0) prm.CB = 64;  // two groups per CTA
    // channel stride: an odd number of 32-bit words, so lanes that walk over channels
    // hit different banks; with 16-byte pieces an odd number of 16-byte units (16-byte loads)
    int cs = NN * K1_WP;
    if (vec16) { cs = NN * K1_WPV; if ((cs / 8) % 2 == 0) cs += 8; }
    else if (esz == 2) { cs += 2; if ((cs / 2) % 2 == 0) cs += 2; }
    else if (cs % 2 == 0) cs += 1;
    prm.CS = cs;
    prm.strip_bytes = (prm.CB * cs * esz + 15) / 16 * 16;
    prm.pair = (g.W % 2 == 0);                     // x is 4-byte aligned (checked by the entry points)
    auto smem_bytes = [&]() {
        return (1 + prm.dbuf) * (size_t)prm.strip_bytes + (size_t)prm.TB * P * (prm.CB + 4) * sizeof(float);
    };
    // Large groups get fewer tiles per item (aim: two or more CTAs per SM).  The second
    // strip buffer is used only where it does not cost a resident CTA (registers allow four).
    prm.dbuf = 0;
    while (prm.TB > 1 && smem_bytes() > 113 * 1024) --prm.TB;
    // the same number of chunks per tile row with evenly sized chunks (four tiles: 2 + 2, not 3 + 1)
    prm.NCH = (g.TW + prm.TB - 1) / prm.TB;
    prm.TB = (g.TW + prm.NCH - 1) / prm.NCH;
    {
        const size_t per_sm = 227 * 1024, one = smem_bytes() + 1024;
        const size_t two = one + prm.strip_bytes;
        const size_t n1 = per_sm / one < 4 ? per_sm / one : 4, n2 = per_sm / two < 4 ? per_sm / two : 4;
        if (n2 >= 1 && n2 == n1) prm.dbuf = 1;
    }
    prm.smem = (int)smem_bytes();
    prm.NCB = g.C / prm.CB;
    prm.items = g.N * g.TH * prm.NCH * prm.NCB;
    prm.by_NCH = FastDiv(prm.NCH);
    prm.by_NCB = FastDiv(prm.NCB);
    prm.by_cb32 = FastDiv(prm.CB / 32);
    // persistent CTAs: as many as fit on the device at once
    const int per_sm = resident_of(plan, (size_t)prm.smem);
    const int resident = per_sm * (plan.sm_count > 0 ? plan.sm_count : 1);
    prm.grid = prm.items < resident ? prm.items : resident;
}

// The same for the NHWC kernel: the strip is the dense TMA box [n][TB * m + 2][CB].
static void plan_k1_nhwc(wfq_plan &plan)
{
    const Geometry &g = plan.geo;
    const bool f16 = plan.in_dtype == WFQ_F16;
    const int NN = g.n, P = g.P, M = g.m;
    const int esz = f16 ? 2 : 4;
    K1Params &prm = plan.k1n;
    prm = plan.k1;
    prm.vec16 = 0;
    prm.TB = (K1_WP - 3) / M;
    prm.CB = g.gs;
    if (g.gs == 32 && g.C % 64 == 0) prm.CB = 64;
    auto strip = [&]() { return ((NN * (prm.TB * M + 2) * prm.CB * esz + 127) / 128) * 128; };
    auto smem_bytes = [&]() {     // 128 bytes of slack for the alignment of the strips
        return 128 + (1 + prm.dbuf) * (size_t)strip() + (size_t)prm.TB * P * (prm.CB + 4) * sizeof(float);
    };
    prm.dbuf = 0;
    while (prm.TB > 1 && smem_bytes() > 113 * 1024) --prm.TB;
    prm.NCH = (g.TW + prm.TB - 1) / prm.TB;
    prm.TB = (g.TW + prm.NCH - 1) / prm.NCH;
    {
        const size_t per_sm = 226 * 1024, one = smem_bytes() + 1024;
        const size_t two = one + strip();
        const size_t n1 = per_sm / one < 4 ? per_sm / one : 4, n2 = per_sm / two < 4 ? per_sm / two : 4;
        if (n2 >= 1 && n2 == n1) prm.dbuf = 1;
    }
    prm.strip_bytes = strip();
    prm.CS = 0;
    prm.smem = (int)smem_bytes();
    prm.NCB = g.C / prm.CB;
    prm.items = g.N * g.TH * prm.NCH * prm.NCB;
    prm.by_NCH = FastDiv(prm.NCH);
    prm.by_NCB = FastDiv(prm.NCB);
    prm.by_cb32 = FastDiv(prm.CB / 32);
    const int per_sm = (int)k1_op(kK1nResident, M, f16, g.gs, nullptr, nullptr, nullptr, (size_t)prm.smem);
    const int resident = per_sm * (plan.sm_count > 0 ? plan.sm_count : 1);
    prm.grid = prm.items < resident ? prm.items : resident;
}

// Work-item shape, shared-memory layout and grid of the cp.async kernel for this plan: one set
// with 4-byte (or 2-byte) copies for any x, and where fp16 rows are whole 16-byte pieces (W a
// multiple of 8) a second one with 16-byte copies, used when x is 16-byte aligned.
void plan_input_transform(wfq_plan &plan)
{
    const bool vec16 = plan.in_dtype == WFQ_F16 && plan.geo.W % 8 == 0;
    auto resident_of = [](const wfq_plan &p, size_t smem) {
        return (int)k1_op(kK1Resident, p.geo.m, p.in_dtype == WFQ_F16, p.geo.gs, nullptr, nullptr, nullptr, smem);
    };
    plan_k1(plan, plan.k1, false, resident_of);
    plan.k1v = plan.k1;
    if (vec16) plan_k1(plan, plan.k1v, true, resident_of);
    plan_k1_nhwc(plan);
    plan.tmap_xn_base = nullptr;
    plan.tmap_xn_tc_base = nullptr;
}

cudaError_t setup_input_transform()
{
    const int sizes[5] = {32, 64, 128, 256, 96};
    for (int m = 2; m <= 6; m += 2)
        for (int f16 = 0; f16 < 2; ++f16)
            for (int gs : sizes) {
                cudaError_t e = (cudaError_t)k1_op(kK1Setup, m, f16 != 0, gs, nullptr, nullptr, nullptr, 0);
                if (e != cudaSuccess) return e;
                e = (cudaError_t)k1_op(kK1nSetup, m, f16 != 0, gs, nullptr, nullptr, nullptr, 0);
                if (e != cudaSuccess) return e;
            }
    return cudaSuccess;
}

cudaError_t launch_input_transform(wfq_plan &plan, const void *x_dev, cudaStream_t stream)
{
    const Geometry &g = plan.geo;
    if (plan.in_nhwc) {
        // x[N][H][W][C] as a 4-D tensor (C, W, H, N) with boxes of one work item's strip
        if ((reinterpret_cast<uintptr_t>(x_dev) & 15u) != 0) return cudaErrorInvalidValue;
        const unsigned long long esz0 = plan.in_dtype == WFQ_F16 ? 2 : 4;
        // tensor cores where they apply (fp16, groups of 32 or 64, C a multiple of 64, F(4,3) / F(6,3)),
        // unless the debug option asks for the plain kernel
        if (input_transform_tcn_applies(plan) && plan.k1_choice != 1) {
            if (plan.tmap_xn_tc_base != x_dev) {
                const unsigned long long dims[4] = {(unsigned long long)g.C, (unsigned long long)g.W,
                                                    (unsigned long long)g.H, (unsigned long long)g.N};
                const unsigned long long strides[3] = {(unsigned long long)g.C * esz0,
                                                       (unsigned long long)g.W * g.C * esz0,
                                                       (unsigned long long)g.H * g.W * g.C * esz0};
                unsigned box[4];
                input_transform_tcn_box(plan, box);
                if (!encode_tmap(&plan.tmap_xn_tc, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 4, x_dev, dims, strides, box,
                                 CU_TENSOR_MAP_SWIZZLE_128B))
                    return cudaErrorInvalidValue;
                plan.tmap_xn_tc_base = x_dev;
            }
            return launch_input_transform_tcn(plan, stream);
        }
        if (plan.tmap_xn_base != x_dev) {
            const unsigned long long esz = plan.in_dtype == WFQ_F16 ? 2 : 4;
            const unsigned long long dims[4] = {(unsigned long long)g.C, (unsigned long long)g.W,
                                                (unsigned long long)g.H, (unsigned long long)g.N};
            const unsigned long long strides[3] = {(unsigned long long)g.C * esz, (unsigned long long)g.W * g.C * esz,
                                                   (unsigned long long)g.H * g.W * g.C * esz};
            const unsigned box[4] = {(unsigned)plan.k1n.CB, (unsigned)(plan.k1n.TB * g.m + 2), (unsigned)g.n, 1u};
            if (!encode_tmap(&plan.tmap_xn, plan.in_dtype == WFQ_F16 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT16
                                                                      : CU_TENSOR_MAP_DATA_TYPE_FLOAT32,
                             4, x_dev, dims, strides, box, CU_TENSOR_MAP_SWIZZLE_NONE))
                return cudaErrorInvalidValue;
            plan.tmap_xn_base = x_dev;
        }
        return (cudaError_t)k1_op(kK1nLaunch, g.m, plan.in_dtype == WFQ_F16, g.gs, &plan, x_dev, stream, 0);
    }
    // tensor-core kernel: fp16 input that a TMA tensor map (16-byte aligned base) can describe
    // (automatic = the cp.async kernel: the tensor-core one measured no faster on any configured layer)
    if (plan.k1tc.use && plan.k1_choice == 2 && (reinterpret_cast<uintptr_t>(x_dev) & 15u) == 0) {
        if (plan.k1tc.mode != 2 && plan.tmap_x_base != x_dev) {
            const unsigned long long hw = (unsigned long long)g.H * g.W;
            bool ok;
            if (plan.k1tc.mode == 0) {
                const unsigned long long dims[3] = {(unsigned long long)g.W, (unsigned long long)g.H,
                                                    (unsigned long long)g.N * g.C};
                const unsigned long long strides[2] = {(unsigned long long)g.W * 2, hw * 2};
                ok = encode_tmap(&plan.tmap_x, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 3, x_dev, dims, strides,
                                 plan.k1tc.box, CU_TENSOR_MAP_SWIZZLE_NONE);
            } else {
                const unsigned long long dims[2] = {hw, (unsigned long long)g.N * g.C};
                const unsigned long long strides[1] = {hw * 2};
                ok = encode_tmap(&plan.tmap_x, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, x_dev, dims, strides,
                                 plan.k1tc.box, CU_TENSOR_MAP_SWIZZLE_NONE);
            }
            if (!ok) return cudaErrorInvalidValue;
            plan.tmap_x_base = x_dev;
        }
        return launch_input_transform_tc(plan, x_dev, stream);
    }
    return (cudaError_t)k1_op(kK1Launch, g.m, plan.in_dtype == WFQ_F16, g.gs, &plan, x_dev, stream, 0);
}

}  // namespace wfq
