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
// The kernels stand beside their floating-point counterparts, whose staging, group quantization and
// stores they share (wfq_input_transform.cu, wfq_output_transform.cu; the quantizer in
// wfq_int_quant.cuh); here are the codes of the two matrices, which they take as parameters.
#include <cmath>

#include "wfq_int_quant.cuh"
#include "wfq_internal.h"

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

}  // namespace wfq
