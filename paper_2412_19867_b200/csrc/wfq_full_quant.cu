// The paper's fully quantized transforms (Section 4.1), as an optional mode of the plan:
//   input   X~ = s_qB^2 s_qx  Q(S_B V_B / s_qB)  Q(x / s_qx)  Q(V_B^T S_B / s_qB)      (Eq. quant-B)
//   output  y~ = s_qA^2 s_qY  Q(V_A S_A / s_qA)  Q(Y~ / s_qY) Q(S_A V_A^T / s_qA)      (Eq. quant-y)
// with Q the symmetric 8-bit abs-max quantizer of Section 2 (codes in [-127, 127], round half to
// even, scale = abs-max / 127).  The matrix products run on integer codes in int32 (exact); the
// quantizers decide in fp64 (scale = amax / 127, code = rint(v / scale)), which makes every code a
// function of the input values alone, not of an instruction order.  The contraction between the
// two transforms (Eq. quant-Y) is the same kernel as in the floating-point-transform mode: the
// input kernel hands it int8 codes and group scales of fp32(X~), the output kernel reads its fp32 Y.
//
// Readings where the paper is silent: s_qB and s_qA are one scale per matrix (they appear squared);
// s_qx is one scale per (tile, group of `group size` input channels), shared by the n x n patches of
// those channels; s_qY is one scale per (tile, output channel) ("tile") or one per row of the n x n
// matrix for the product with the right-hand matrix, whose result is quantized again per column for
// the left-hand product ("row": Section 3.2 asks for per-tile or per-row/column scales of Y).
//
// The kernels share the staging, group quantization and stores of their floating-point counterparts
// (wfq_strip.cuh, wfq_output_store.cuh; the quantizer in wfq_int_quant.cuh) but are compiled here: the code
// of a source file is loaded onto a device as a whole, and only plans in this mode need theirs (in the
// files of their counterparts they made a process's first plan 14 ms longer).
#include <cmath>

#include "wfq_int_quant.cuh"
#include "wfq_internal.h"
#include "wfq_output_store.cuh"
#include "wfq_ptx.cuh"
#include "wfq_strip.cuh"

namespace wfq {

namespace {

// Points of F(4,3) and F(6,3) (Section 3.1), the last one at infinity.
const double kPoints2[3] = {0.0, 1.0, -1.0};
const double kPoints4[5] = {0.0, 1.0, -1.0, 2.0, -2.0};
const double kPoints6[7] = {0.0, 1.0, -1.0, 2.0, -2.0, 0.5, -0.5};
// Standard-scaled B^T of the paper's supplementary and its row scales: V_B = diag(1 / s) B^T.
const double kStdBT2[16] = {1, 0, -1, 0,   0, 1, 1, 0,   0, -1, 1, 0,   0, 1, 0, -1};
const double kStdRow2[4] = {1.0, 2.0, 2.0, -1.0};
const double kStdBT4[36] = {4, 0, -5, 0, 1, 0,   0, -4, -4, 1, 1, 0,   0, 4, -4, -1, 1, 0,
                            0, -2, -1, 2, 1, 0,  0, 2, -1, -2, 1, 0,   0, 4, 0, -5, 0, 1};
const double kStdRow4[6] = {4.0, -6.0, -6.0, 24.0, 24.0, 1.0};
const double kStdBT6[64] = {
    1, 0, -5.25, 0, 5.25, 0, -1, 0,        0, 1, 1, -4.25, -4.25, 1, 1, 0,
    0, -1, 1, 4.25, -4.25, -1, 1, 0,       0, 0.5, 0.25, -2.5, -1.25, 2, 1, 0,
    0, -0.5, 0.25, 2.5, -1.25, -2, 1, 0,   0, 2, 4, -2.5, -5, 0.5, 1, 0,
    0, -2, 4, 2.5, -5, -0.5, 1, 0,         0, -1, 0, 5.25, 0, -5.25, 0, 1};
const double kStdRow6[8] = {1.0, -4.5, -4.5, 90.0, 90.0, 45.0 / 32, 45.0 / 32, 1.0};

// Q of a whole matrix: one scale, codes rint(v / scale).
double quantize_matrix(const double *mat, int count, int *codes)
{
    double amax = 0.0;
    for (int i = 0; i < count; ++i) amax = std::fmax(amax, std::fabs(mat[i]));
    const double s = amax / kIntQmax;
    for (int i = 0; i < count; ++i) {
        double q = s > 0.0 ? std::nearbyint(mat[i] / s) : 0.0;     // round half to even (default mode)
        q = std::fmin(std::fmax(q, -kIntQmax), kIntQmax);
        codes[i] = (int)q;
    }
    return s;
}

}  // namespace

// Codes and scales of the two transform matrices for the plan's current scale vectors.
void build_full_quant_tables(wfq_plan &plan)
{
    const Geometry &g = plan.geo;
    const int n = g.n, m = g.m;
    FullQuantTables &tab = plan.fq;
    const double *bt = m == 2 ? kStdBT2 : m == 4 ? kStdBT4 : kStdBT6;
    const double *row = m == 2 ? kStdRow2 : m == 4 ? kStdRow4 : kStdRow6;
    const double *pts = m == 2 ? kPoints2 : m == 4 ? kPoints4 : kPoints6;
    double BT[kMaxN * kMaxN], AT[kMaxN * kMaxN];
    // S_B V_B: V_B = V^{-T}, each entry the correctly rounded quotient of two exact numbers
    for (int i = 0; i < n; ++i)
        for (int a = 0; a < n; ++a) BT[i * n + a] = plan.sB[i] * (bt[i * n + a] / row[i]);
    // V_A S_A: V_A[u][i] = point_i^u, the point at infinity contributes to the last row only
    for (int u = 0; u < m; ++u)
        for (int i = 0; i < n; ++i) {
            double va = i < n - 1 ? 1.0 : (u == m - 1 ? 1.0 : 0.0);
            if (i < n - 1)
                for (int e = 0; e < u; ++e) va *= pts[i];          // exact: small powers of 0, 1, 2, 1/2
            AT[u * n + i] = va * plan.sA[i];
        }
    for (int i = 0; i < kMaxN * kMaxN; ++i) tab.BTq[i] = tab.ATq[i] = 0;
    const double sqB = quantize_matrix(BT, n * n, tab.BTq);
    tab.sqB2 = sqB * sqB;
    tab.sqA = quantize_matrix(AT, m * n, tab.ATq);
}

namespace {

// ---- the fully quantized input transform (Eq. quant-B) ------------------------------------
//   X~ = s_qB^2 s_qx  Q(S_B V_B / s_qB)  Q(x / s_qx)  Q(V_B^T S_B / s_qB)
// with one s_qx per (tile, channel group) over the group's n x n patches; fp32(X~) is what the group
// quantizer of the contraction's operand sees.  Work items, staging and quantization are those of
// the kernel above; in between every (tile, channel) first contributes its patch to the abs-max of its
// 32 channels (one warp reduction), then quantizes the patch (code_of_float) and forms the two
// integer products.  32x32 C=640 F(4,3), two images: 15.5 us (latency of
// the phases at 16 warps per SM, 45 % of the issue slots); with one CTA per (tile, group), each thread
// reading its patch element by element from global memory (32 rows of memory per load instruction)
// and all codes decided in fp64, 24.8 us.
template <int M, typename Tin, int GSR, int SPLIT>
__global__ void __launch_bounds__(K1_THREADS, 4)
input_transform_int_kernel(const Tin *__restrict__ x, int8_t *__restrict__ Xq, float *__restrict__ sX, Geometry g,
                           const __grid_constant__ FullQuantTables tab, K1Params prm)
{
    constexpr int NN = M + 2;
    constexpr int P = NN * NN;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ float amax_s[(K1_WP - 3) / M][8];               // [tile][run of 32 channels]
    ptx::grid_dependency_wait();
    ptx::grid_launch_dependents();
    float *Zs = reinterpret_cast<float *>(smem_raw + (1 + prm.dbuf) * prm.strip_bytes);   // [tile][position][CBP]
    const int CBP = prm.CB + 4;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    constexpr int NWARP = K1_THREADS / 32;
    const int cb32 = prm.CB >> 5;
    const int gs = GSR > 0 ? GSR * SPLIT : g.gs;
    const int ng = prm.CB / gs, gs32 = gs >> 5;

    auto stage_item = [&](int item, int buf) {
        const int rest = item / prm.by_NCB, cblk = item - rest * prm.NCB;
        const int srow = rest / prm.by_NCH, chunk = rest - srow * prm.NCH;
        const int img = srow / g.by_TH, th = srow - img * g.TH;
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
            cp_async_wait_group<0>();
        } else if (next < prm.items) {
            stage_item(next, buf ^ 1);
            cp_async_wait_group<1>();
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
        const int voff = tw0 * M - 2 - (((tw0 * M - 1 + 8) & ~7) - 8);
        auto patch = [&](int tl, int c, float (&d)[NN][NN]) {
            if (sizeof(Tin) == 2 && prm.vec16) load_patch_vec<NN>(strip + c * prm.CS, tl * M + voff, d);
            else load_patch<NN>(strip + c * prm.CS, tl * M, d);
        };

        for (int wt = warp; wt < ntile * cb32; wt += NWARP) {
            const int tl = wt / prm.by_cb32, c32 = wt - tl * cb32;
            float d[NN][NN], m = 0.f;
            patch(tl, c32 * 32 + lane, d);
#pragma unroll
            for (int a = 0; a < NN; ++a)
#pragma unroll
                for (int b = 0; b < NN; ++b) m = fmaxf(m, fabsf(d[a][b]));     // ignores NaN
            const unsigned top = __reduce_max_sync(0xffffffffu, __float_as_uint(m));
            if (lane == 0) amax_s[tl][c32] = __uint_as_float(top);
        }
        __syncthreads();
        for (int wt = warp; wt < ntile * cb32; wt += NWARP) {
            const int tl = wt / prm.by_cb32, c32 = wt - tl * cb32;
            const int c = c32 * 32 + lane;
            float amax = 0.f;                                    // of the group of these 32 channels
            for (int k = c32 / gs32 * gs32, e = k + gs32; k < e; ++k) amax = fmaxf(amax, amax_s[tl][k]);
            float d[NN][NN];
            patch(tl, c, d);
            const float rinv = __fdiv_rn(127.f, amax);
            int q[NN][NN], tmp[NN][NN];
#pragma unroll
            for (int a = 0; a < NN; ++a)
#pragma unroll
                for (int b = 0; b < NN; ++b) q[a][b] = code_of_float(d[a][b], amax, rinv);
#pragma unroll
            for (int b = 0; b < NN; ++b)
#pragma unroll
                for (int i = 0; i < NN; ++i) {
                    int s = 0;
#pragma unroll
                    for (int a = 0; a < NN; ++a) s += tab.BTq[i * NN + a] * q[a][b];
                    tmp[i][b] = s;
                }
            const double scale = __dmul_rn(tab.sqB2, __ddiv_rn((double)amax, kIntQmax));
            float *out = Zs + (size_t)tl * P * CBP + c;
#pragma unroll
            for (int i = 0; i < NN; ++i)
#pragma unroll
                for (int j = 0; j < NN; ++j) {
                    int s = 0;
#pragma unroll
                    for (int b = 0; b < NN; ++b) s += tmp[i][b] * tab.BTq[j * NN + b];
                    out[(i * NN + j) * CBP] = (float)__dmul_rn((double)s, scale);
                }
        }
        __syncthreads();
        if (!prm.dbuf && next < prm.items) stage_item(next, 0);   // the strip buffer is free: refill it now

        quantize_item<P, GSR, SPLIT, false>(Zs, CBP, ntile, ng, gs, srow, tw0, c_base, g, InputScales{}, Xq, sX);
        __syncthreads();   // Z and this strip buffer are free again
    }
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

    const int tq = t / g.by_TW, img = tq / g.by_TH;
    const int tw = t - tq * g.TW, th = tq - img * g.TH;
    const int h0 = th * M, w0 = tw * M;
    const size_t base = (((size_t)img * g.K + k) * g.H + h0) * g.W + w0;
    auto row_of = [&](int u, float (&o)[M]) {
#pragma unroll
        for (int c = 0; c < M; ++c) o[c] = out[u][c];
    };
    store_tiles<M, STORE, true, TT>(row_of, sm, live, base, h0, w0, k, y, g, bias, act, out_half);
}

template <int M, typename Tin, int GSR, int SPLIT>
int k1i_resident(size_t smem)
{
    return resident_ctas_per_sm(input_transform_int_kernel<M, Tin, GSR, SPLIT>, K1_THREADS, smem, 32);
}

template <int M, typename Tin, int GSR, int SPLIT>
cudaError_t k1i_setup()
{
    auto kern = input_transform_int_kernel<M, Tin, GSR, SPLIT>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, 226 * 1024);
    if (e != cudaSuccess) return e;
    return cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout,
                                (int)cudaSharedmemCarveoutMaxShared);
}

template <int M, typename Tin, int GSR, int SPLIT>
cudaError_t launch_k1i(const wfq_plan &plan, const void *x_dev, cudaStream_t stream)
{
    const bool vec = plan.k1iv.vec16 && plan.k1_choice != 3 && (reinterpret_cast<uintptr_t>(x_dev) & 15u) == 0;
    const K1Params &prm = vec ? plan.k1iv : plan.k1i;
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
    return cudaLaunchKernelEx(&cfg, input_transform_int_kernel<M, Tin, GSR, SPLIT>, static_cast<const Tin *>(x_dev),
                              plan.ws.Xq, plan.ws.sX, plan.geo, plan.fq, prm);
}

// What to do with the instantiation of the input transform that serves (m, dtype, group size).
enum IntOp { kLaunch, kResident, kSetup };

template <int M, typename Tin>
long long int_by_gs(IntOp op, const wfq_plan &plan, const void *x, cudaStream_t s, size_t smem)
{
    auto go = [&](auto gsr, auto split) -> long long {
        constexpr int GSR = decltype(gsr)::value, SPLIT = decltype(split)::value;
        if (op == kLaunch) return (long long)launch_k1i<M, Tin, GSR, SPLIT>(plan, x, s);
        if (op == kResident) return k1i_resident<M, Tin, GSR, SPLIT>(smem);
        return (long long)k1i_setup<M, Tin, GSR, SPLIT>();
    };
    using std::integral_constant;
    switch (plan.geo.gs) {
        case 32: return go(integral_constant<int, 32>{}, integral_constant<int, 1>{});
        case 64: return go(integral_constant<int, 64>{}, integral_constant<int, 1>{});
        case 128: return go(integral_constant<int, 64>{}, integral_constant<int, 2>{});
        case 256: return go(integral_constant<int, 64>{}, integral_constant<int, 4>{});
        default: return go(integral_constant<int, 0>{}, integral_constant<int, 1>{});
    }
}

long long int_op(IntOp op, const wfq_plan &plan, const void *x, cudaStream_t s, size_t smem)
{
    const bool f16 = plan.in_dtype == WFQ_F16;
    switch (plan.geo.m) {
        case 2: return f16 ? int_by_gs<2, __half>(op, plan, x, s, smem) : int_by_gs<2, float>(op, plan, x, s, smem);
        case 4: return f16 ? int_by_gs<4, __half>(op, plan, x, s, smem) : int_by_gs<4, float>(op, plan, x, s, smem);
        default: return f16 ? int_by_gs<6, __half>(op, plan, x, s, smem) : int_by_gs<6, float>(op, plan, x, s, smem);
    }
}

}  // namespace

// Work-item shapes of the integer input transform and the attributes of the one kernel that the plan uses.  With
// the plan's device current; geometry, dtype and device are known.
cudaError_t plan_input_transform_int(wfq_plan &plan)
{
    const cudaError_t e = (cudaError_t)int_op(kSetup, plan, nullptr, nullptr, 0);
    if (e != cudaSuccess) return e;
    auto resident_of = [](const wfq_plan &p, size_t smem) { return (int)int_op(kResident, p, nullptr, nullptr, smem); };
    plan_k1(plan, plan.k1i, false, resident_of);
    plan.k1iv = plan.k1i;
    if (plan.in_dtype == WFQ_F16 && plan.geo.W % 8 == 0) plan_k1(plan, plan.k1iv, true, resident_of);
    return cudaSuccess;
}

// NCHW input, any group size of the plan.
cudaError_t launch_input_transform_int(const wfq_plan &plan, const void *x_dev, cudaStream_t stream)
{
    return (cudaError_t)int_op(kLaunch, plan, x_dev, stream, 0);
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
