// Winograd-domain contraction with per-group dequantization (Eq. quant-Y):
//   for every position p:  Y_p[t][k] = sum_g sX[p,g,t] * sW[p,g,k] * acc_g[t][k],
//   acc_g[t][k] = sum_{c in g} Xq_p[t][c] * Wq_p[k][c]     (int8 x int8 -> int32)
//
// Persistent, warp-specialised sm_100a kernel, two CTAs per SM.  A unit of work is
// (position p, block of 128 rows, block of BN columns).  "Rows" are the 128 TMEM lanes
// of the accumulator: tiles in the normal orientation, output channels in the swapped
// one (used when there are few tiles, so that all 128 lanes carry real work); columns
// are the other of the two.  Both operands are K-major int8 (channels contiguous).
//
// Every mbarrier hand-over costs the thread that makes it a few hundred cycles, so the
// roles synchronise per *chunk* of up to CG channel groups (128 channels when the group
// size divides 128), not per group.  A chunk owns one TMEM slot of 128 columns (its
// groups side by side, BN columns each) and one slot of the scale ring.
//   warp 0   TMA producer: 128 x 128 B of the row operand and BN x 128 B of the column
//            operand per stage (128-byte swizzle), ring of NSTAGES
//   warp 1   allocates TMEM; one lane issues tcgen05.mma kind::i8 (M=128, N=BN, K=32 per
//            instruction): waits for a stage and, at the start of a chunk, for its TMEM
//            slot; commits the stage back to the producer and the chunk to the epilogue
//   warp 2   scale loader: per chunk, 128 row scales and BN column scales per group into
//            the chunk's scale slot (bulk copies); their arrival counts on the same barrier as the MMAs'
//   warps 4-7   epilogue: warp % 4 selects the 32 TMEM lanes the warp may read; each warp
//            handles all BN columns of its lanes.  Per chunk: wait for accumulators and
//            scales, then per group tcgen05.ld the int32 sums, convert and scale into fp32
//            registers (packed f32x2 multiply / fma), release the slot; after the last
//            chunk of a unit write Y[p][k][t].
// The second CTA of the SM runs the same pipeline on other units, which hides part of the
// hand-over latencies; the stores of Y leave through the TMA unit (rows = tiles).
// What bounds it: the epilogue warps.  14x14 with groups of 32 (1024 tiles x 256 channels, F(4,3): 3.9
// units of four chunks per CTA, 75 M group sums), this kernel launched back to back on warm operands,
// 20.7 us from launch to launch; with clock reads in the epilogue, which cost 10 %: a chunk of 2 x 64
// columns takes 1110 cycles (840 with one CTA per SM) and 140 pass until the next one is complete, a
// unit's first chunk comes after 460 and handing its Y to the TMA unit takes 780; 26 k cycles, 13.5 us,
// in all, and 0.5 us in front of them.
// Four epilogue warps per CTA: eight, with half of the columns each, are 1 % slower (forward, ten
// layers), and the registers for 64 sums and two blocks of 16 leave no room for more.
// Every wait is bounded; on expiry the CTA records where, stops, drains and frees TMEM.
#include "wfq_internal.h"
#include "wfq_ptx.cuh"

namespace wfq {

namespace {

constexpr int BM = 128;        // rows per unit (MMA M, TMEM lanes)
constexpr int BK = 128;        // bytes (= int8 channels) per pipeline stage
constexpr int UK = 32;         // channels per MMA instruction
constexpr int NSTAGES = 3;     // shared-memory operand stages
constexpr int NSLOT = 2;       // TMEM / scale slots (chunks in flight)
constexpr int SLOT_COLS = 128; // TMEM columns per slot
constexpr int TMEM_COLS = NSLOT * SLOT_COLS;
constexpr int A_BYTES = BM * BK;
constexpr int NUM_EPI_WARPS = 4;   // one per 32 TMEM lanes
constexpr int FIRST_EPI_WARP = 4;
constexpr int NUM_THREADS = 32 * (FIRST_EPI_WARP + NUM_EPI_WARPS);

// Pieces of 16 columns in a part of a cut unit: halves of 64 and of 32 columns, thirds of 48.
__host__ __device__ constexpr int part_pieces(int bn) { return bn == 64 ? 2 : 1; }

struct Shared {
    uint64_t full[NSTAGES];     // operands of a stage have landed
    uint64_t empty[NSTAGES];    // the MMAs reading a stage have completed
    uint64_t acc_full[NSLOT];      // the MMAs of a chunk have completed and its scales have landed
    uint64_t slot_free[NSLOT];     // all epilogue warps are done with a chunk
    uint64_t mma_done;             // after a wait that ran out: every MMA issued has completed
    uint32_t tmem_base;
    volatile int abort;
};

// Normal orientation: the epilogue hands Y to the TMA unit through shared memory.  Three stages leave the room for it
// and are no slower than four (forward, ten layers within 0.2 %; swapped, 36 tiles x 1280 channels F(6,3) 44.0 -> 43.6 us).
template <int BN, bool SWAP>
struct Cfg {
    static constexpr int STORE_BYTES = SWAP ? 0 : BM * BN * 4;
    static constexpr int B_BYTES = BN * BK;
    static constexpr int STAGE_BYTES = A_BYTES + B_BYTES;
    static constexpr int CG_MAX = SLOT_COLS / BN;             // groups per chunk at most
    static constexpr int GROUP_SCALE_FLOATS = BM + BN;        // row scales, then column scales
    static constexpr int SLOT_SCALE_FLOATS = CG_MAX * GROUP_SCALE_FLOATS;
    static constexpr size_t SMEM_BYTES = 1024 /*alignment slack*/ + (size_t)NSTAGES * STAGE_BYTES + STORE_BYTES +
                                         (size_t)NSLOT * SLOT_SCALE_FLOATS * sizeof(float) + sizeof(Shared);
};

struct GemmArgs {
    const float *row_scale;   // [P][G][row_pitch]: sX (normal) or sW (swapped)
    const float *col_scale;   // [P][G][col_pitch]: sW (normal) or sX (swapped)
    int row_pitch, col_pitch;
    int rows, cols;           // valid rows / columns: (T, K) normal, (K, T) swapped
    int cg;                   // groups per chunk
    int items;                // work items: whole units, then the parts of the units that are cut (plan_gemm_units)
    int whole;                // whole units
    FastDiv by_NT, by_MT;     // blocks of columns and of rows
    float *Y;                 // [P][K][Tp]
    int32_t *acc_dump;        // [P][T][K][G] or null
    int *status;
    long long wait_cycles;    // limit of every mbarrier wait (about a second by default)
    int debug_skip_stage;     // >= 0: CTA 0's producer skips the loads of this stage (test hook)
    long long l2_prefetch_bytes;   // per CTA: filter bytes it may ask into L2 ahead of the previous kernel's end
};

// A work item: a unit, or a part of it: `np` pieces of 16 columns from piece p0 on.
struct Item { int p, mt, nt, p0, np; };
template <int BN, bool CUT>
__device__ __forceinline__ Item item_of(const GemmArgs &a, int i, int MT, int NT)
{
    Item it;
    it.p0 = 0;
    it.np = BN / 16;
    if (CUT && i >= a.whole) {
        constexpr int PARTS = BN / (16 * part_pieces(BN));
        const int part = i - a.whole;
        i = a.whole + part / PARTS;
        it.p0 = part % PARTS * part_pieces(BN);
        it.np = part_pieces(BN);
    }
    const int r = i / a.by_NT;
    it.nt = i - r * NT;
    it.p = r / a.by_MT;
    it.mt = r - it.p * MT;
    return it;
}

// MMA issue loop for the common shapes in which the chunks tile a stage exactly
// (GSTEPS MMAs per group, CGT groups per chunk, GSTEPS * CGT in {2, 4} MMAs per chunk):
// per chunk one slot wait, the chunk's MMAs as straight-line code with constant
// descriptor offsets and accumulate flags, one commit.  The generic loop in the kernel
// spends several hundred cycles per MMA on its bookkeeping, which made the issuing
// warp the bottleneck of every layer with more than one chunk per unit.
template <int BN, bool SWAP, bool CUT, int GSTEPS, int CGT>
__device__ __forceinline__ void mma_issue_aligned(Shared *sh, uint32_t tiles_lo, uint32_t tmem_base,
                                                  const GemmArgs &args, int MT, int NT, int KB,
                                                  int last_slices, const WaitCtx &ctx)
{
    using C = Cfg<BN, SWAP>;
    constexpr int CHUNK_STEPS = GSTEPS * CGT;            // MMAs per chunk
    constexpr int NCH = (BK / UK) / CHUNK_STEPS;         // chunks per stage
    static_assert(NCH >= 1 && NCH * CHUNK_STEPS == BK / UK, "chunks must tile a stage");
    constexpr uint32_t dhi = ptx::smem_desc_sw128_hi();
    const uint32_t full0 = ptx::smem_u32(&sh->full[0]), empty0 = ptx::smem_u32(&sh->empty[0]);
    const uint32_t acc0 = ptx::smem_u32(&sh->acc_full[0]), free0 = ptx::smem_u32(&sh->slot_free[0]);
    int stage = 0, slot = 0;
    uint32_t phase = 0, sphase = 0;
    for (int i = blockIdx.x; i < args.items; i += gridDim.x) {
        const Item it = item_of<BN, CUT>(args, i, MT, NT);
        const uint32_t idesc = ptx::idesc_i8(BM, 16 * it.np);
        for (int kb = 0; kb < KB; ++kb) {
            const int nslice = kb == KB - 1 ? last_slices : BK / UK;
            if (!wait_warp(full0 + 8u * stage, phase, ctx, kWaitSmemFull))
                return;
            const uint32_t a_lo = tiles_lo + (uint32_t)(stage * (C::STAGE_BYTES >> 4));
            const uint32_t b_lo = a_lo + (uint32_t)(A_BYTES >> 4) + (uint32_t)(it.p0 * (16 * BK >> 4));
#pragma unroll
            for (int c = 0; c < NCH; ++c) {
                if (c * CHUNK_STEPS < nslice) {           // the chunk has at least one group
                    if (!wait_warp(free0 + 8u * slot, sphase ^ 1u, ctx, kWaitTmemEmpty))
                        return;
                    ptx::tc_fence_after();
                    if (ptx::elect_one()) {
                        const uint32_t d = tmem_base + (uint32_t)(slot * SLOT_COLS);
                        if ((c + 1) * CHUNK_STEPS <= nslice) {
#pragma unroll
                            for (int s = 0; s < CHUNK_STEPS; ++s) {
                                const uint32_t off = 2u * (uint32_t)(c * CHUNK_STEPS + s);
                                if (s % GSTEPS) ptx::umma_i8_lo<true>(d + (s / GSTEPS) * BN, a_lo + off, b_lo + off, dhi, idesc);
                                else ptx::umma_i8_lo<false>(d + (s / GSTEPS) * BN, a_lo + off, b_lo + off, dhi, idesc);
                            }
                        } else {
                            // last stage of a unit whose channel count is not a multiple of 128
#pragma unroll
                            for (int s = 0; s < CHUNK_STEPS; ++s) {
                                const uint32_t off = 2u * (uint32_t)(c * CHUNK_STEPS + s);
                                if (c * CHUNK_STEPS + s < nslice) {
                                    if (s % GSTEPS) ptx::umma_i8_lo<true>(d + (s / GSTEPS) * BN, a_lo + off, b_lo + off, dhi, idesc);
                                    else ptx::umma_i8_lo<false>(d + (s / GSTEPS) * BN, a_lo + off, b_lo + off, dhi, idesc);
                                }
                            }
                        }
                        ptx::umma_commit(acc0 + 8u * slot);
                    }
                    __syncwarp();
                    if (++slot == NSLOT) { slot = 0; sphase ^= 1u; }
                }
            }
            if (ptx::elect_one()) ptx::umma_commit(empty0 + 8u * stage);
            __syncwarp();
            if (++stage == NSTAGES) { stage = 0; phase ^= 1u; }
        }
    }
}

// What the epilogue keeps through the kernel: the warp's tensor memory, the scale slots, its part of the staging for Y.
struct EpiCtx {
    uint32_t tmem;
    const float *scales;
    unsigned char *out;
    int quarter, lane, nchunk;
};

// One work item in the epilogue: NP * 16 columns from column block0 + c0 on, c0 inside the unit's block of BN columns.
template <int BN, bool SWAP, bool DUMP, bool CUT, int NP>
__device__ __forceinline__ bool epilogue_unit(Shared *sh, const CUtensorMap &tmY, const GemmArgs &a, const Geometry &g,
                                              const WaitCtx &ctx, const EpiCtx &ec, int p, int mt, int block0, int c0,
                                              int &slot, uint32_t &sphase)
{
    using C = Cfg<BN, SWAP>;
    constexpr int CW = 16 * NP;                                // columns of the item
    constexpr int SW = CUT ? 16 * part_pieces(BN) : BN;        // columns of a store (a box of tmap_y)
    const int quarter = ec.quarter, lane = ec.lane;
    const int row = mt * BM + quarter * 32 + lane;    // tile (normal) or channel (swapped)
    const int col0 = block0 + c0;                     // first column
    // warp-uniform: does this warp own any valid row and column of the unit?
    const bool active = (mt * BM + quarter * 32 < a.rows) && (col0 < a.cols);
    const bool row_ok = row < a.rows;
    float2 acc[CW / 2];
#pragma unroll
    for (int j = 0; j < CW / 2; ++j) acc[j] = make_float2(0.f, 0.f);

    for (int ch = 0; ch < ec.nchunk; ++ch) {
        const int g0 = ch * a.cg, ng = min(a.cg, g.G - g0);
        if (!wait_warp(ptx::smem_u32(&sh->acc_full[slot]), sphase, ctx, kWaitTmemFull)) return false;
        if (active) {
            ptx::tc_fence_after();
            const float *sc = ec.scales + (size_t)slot * C::SLOT_SCALE_FLOATS;
            for (int j = 0; j < ng; ++j) {
                const uint32_t taddr = ec.tmem + (uint32_t)(slot * SLOT_COLS + j * BN);
                const float rs = sc[j * C::GROUP_SCALE_FLOATS + quarter * 32 + lane];
                const float2 rs2 = make_float2(rs, rs);
                const float4 *cs4 = reinterpret_cast<const float4 *>(sc + j * C::GROUP_SCALE_FLOATS + BM + c0);
                uint32_t rr[2][16];
                ptx::tmem_ld_x16(taddr, rr[0]);
#pragma unroll
                for (int h = 0; h < CW / 16; ++h) {          // 16 columns at a time, the next 16 on their way
                    uint32_t (&r)[16] = rr[h & 1];
                    ptx::tmem_ld_wait(r);
                    if (h + 1 < CW / 16) ptx::tmem_ld_x16(taddr + (uint32_t)(16 * (h + 1)), rr[(h + 1) & 1]);
                    if constexpr (DUMP) {
                        if (row_ok) {
#pragma unroll
                            for (int i = 0; i < 16; ++i) {
                                const int col = col0 + 16 * h + i;
                                if (col < a.cols) {
                                    const size_t t = SWAP ? col : row, k = SWAP ? row : col;
                                    a.acc_dump[(((size_t)p * g.T + t) * g.K + k) * g.G + g0 + j] =
                                        (int32_t)r[i];
                                }
                            }
                        }
                    } else {
#pragma unroll
                        for (int q = 0; q < 4; ++q) {
                            const float4 cs = cs4[4 * h + q];
                            float2 f0 = make_float2(__int2float_rn((int32_t)r[4 * q + 0]),
                                                    __int2float_rn((int32_t)r[4 * q + 1]));
                            float2 f1 = make_float2(__int2float_rn((int32_t)r[4 * q + 2]),
                                                    __int2float_rn((int32_t)r[4 * q + 3]));
                            f0 = __fmul2_rn(f0, rs2);
                            f1 = __fmul2_rn(f1, rs2);
                            acc[8 * h + 2 * q] = __ffma2_rn(f0, make_float2(cs.x, cs.y), acc[8 * h + 2 * q]);
                            acc[8 * h + 2 * q + 1] =
                                __ffma2_rn(f1, make_float2(cs.z, cs.w), acc[8 * h + 2 * q + 1]);
                        }
                    }
                }
            }
            ptx::tc_fence_before();
        }
        __syncwarp();
        if (ptx::elect_one()) ptx::mbar_arrive(ptx::smem_u32(&sh->slot_free[slot]));
        if (++slot == NSLOT) { slot = 0; sphase ^= 1u; }
    }

    if constexpr (!DUMP && SWAP) {
        if (active && row_ok) {
            // row = output channel, columns = tiles: contiguous in Y[p][k][:];
            // 32-byte stores so that every instruction fills whole sectors
            float *dst = a.Y + ((size_t)p * g.K + row) * g.Tp + col0;
#pragma unroll
            for (int j8 = 0; j8 < CW / 8; ++j8)
                if (col0 + 8 * j8 + 7 < g.Tp)
                    ptx::st_global_v8(dst + 8 * j8, acc[4 * j8].x, acc[4 * j8].y, acc[4 * j8 + 1].x,
                                      acc[4 * j8 + 1].y, acc[4 * j8 + 2].x, acc[4 * j8 + 2].y,
                                      acc[4 * j8 + 3].x, acc[4 * j8 + 3].y);
        }
    } else if constexpr (!DUMP) {
        if (active) {
            // row = tile: the warp's columns go to shared memory as rows of 32 tiles and from there to Y[p][k][t] by
            // tiled stores, which leave out what lies beyond K or T (rounded up to 16 bytes, inside the padding of the
            // row), while the warp goes on with the next item.  Stored by the warp itself (64 stores of 128 bytes) they
            // held it up for as long as L2 took them (about 1400 cycles a unit): forward, 1024 tiles x 256 channels in
            // groups of 32 43.1 -> 42.6 us, F(6,3) 128 tiles x 512 channels, two layers, 57.0 -> 55.5 us
            float *out_lane = reinterpret_cast<float *>(ec.out) + lane;
            if (lane == 0) ptx::bulk_wait_read();
            __syncwarp();
#pragma unroll
            for (int j = 0; j < CW / 2; ++j) {
                out_lane[(2 * j) * 32] = acc[j].x;
                out_lane[(2 * j + 1) * 32] = acc[j].y;
            }
            ptx::fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0) {
#pragma unroll
                for (int h = 0; h < CW; h += SW)
                    if (col0 + h < a.cols)
                        ptx::tma_store_3d(&tmY, ptx::smem_u32(ec.out) + (uint32_t)(h * 128), mt * BM + quarter * 32,
                                          col0 + h, p);
                ptx::bulk_commit();
            }
            __syncwarp();
        }
    }
    return true;
}

template <int BN, bool SWAP, bool DUMP, bool CUT>
__global__ void __launch_bounds__(NUM_THREADS, 2)
gemm_dequant_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                    const __grid_constant__ CUtensorMap tmY, GemmArgs a, Geometry g)
{
    using C = Cfg<BN, SWAP>;
    extern __shared__ unsigned char smem_raw[];
    // 1024-byte alignment: the 128-byte swizzle atoms repeat every 1024 bytes
    unsigned char *tiles = ptx::align_smem<1024>(smem_raw);
    unsigned char *store = tiles + (size_t)NSTAGES * C::STAGE_BYTES;
    float *scales = reinterpret_cast<float *>(store + C::STORE_BYTES);
    Shared *sh = reinterpret_cast<Shared *>(scales + (size_t)NSLOT * C::SLOT_SCALE_FLOATS);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int MT = (a.rows + BM - 1) / BM, NT = (a.cols + BN - 1) / BN;
    const int KB = (g.C + BK - 1) / BK;          // stages per unit
    const int gs_steps = g.gs / UK;              // MMAs per group
    const int cg = a.cg;                         // groups per chunk
    const int nchunk = (g.G + cg - 1) / cg;      // chunks per unit
    const WaitCtx ctx{&sh->abort, a.status, a.wait_cycles};

    if (threadIdx.x == 0) {
        for (int s = 0; s < NSTAGES; ++s) {
            ptx::mbar_init(ptx::smem_u32(&sh->full[s]), 1);
            ptx::mbar_init(ptx::smem_u32(&sh->empty[s]), 1);
        }
        for (int b = 0; b < NSLOT; ++b) {
            ptx::mbar_init(ptx::smem_u32(&sh->acc_full[b]), DUMP ? 1 : 2);   // MMAs, scales
            ptx::mbar_init(ptx::smem_u32(&sh->slot_free[b]), NUM_EPI_WARPS);
        }
        ptx::mbar_init(ptx::smem_u32(&sh->mma_done), 1);
        sh->abort = 0;
        ptx::fence_mbar_init();
    }
    if (warp == 1) {
        ptx::tmem_alloc(ptx::smem_u32(&sh->tmem_base), TMEM_COLS);
        ptx::tmem_relinquish();
    }
    ptx::tc_fence_before();
    __syncthreads();
    ptx::tc_fence_after();
    const uint32_t tmem_base = sh->tmem_base;

    // Everything above may overlap the kernel that produces Xq and sX.  So may the filter
    // stream, which does not depend on it: before waiting for that kernel the producer loads
    // the filter half of its first stages and asks for the filter tiles of its first units
    // to be brought into L2 (bounded by a per-CTA share of `l2_prefetch_bytes`).  Filters written by a
    // kernel before that one are complete: the input transforms let this grid start only after their own
    // wait for it.
    constexpr int W_ROWS = SWAP ? BM : BN;                 // filter rows of a stage
    // stages of the first unit whose filter half is loaded early
    const int pre = (a.l2_prefetch_bytes > 0 && (int)blockIdx.x < a.items) ? (KB < NSTAGES ? KB : NSTAGES) : 0;
    if (warp == 0 && ptx::elect_one()) {
        ptx::prefetch_tmap(&tmA);
        ptx::prefetch_tmap(&tmB);
        if (!SWAP) ptx::prefetch_tmap(&tmY);
        const CUtensorMap *tmW = SWAP ? &tmA : &tmB;
        long long budget = a.l2_prefetch_bytes;
        for (int i = blockIdx.x, first = 1; i < a.items && budget > 0; i += gridDim.x, first = 0) {
            const Item it = item_of<BN, CUT>(a, i, MT, NT);
            const int p = it.p, wrow = SWAP ? it.mt * BM : it.nt * BN;
            for (int kb = 0; kb < KB && budget > 0; ++kb) {
                if (first && kb < pre) {
                    if (!(blockIdx.x == 0 && kb == a.debug_skip_stage)) {
                        const uint32_t bar = ptx::smem_u32(&sh->full[kb]);
                        const uint32_t dst = ptx::smem_u32(tiles + (size_t)kb * C::STAGE_BYTES) + (SWAP ? 0 : A_BYTES);
                        ptx::mbar_arrive_expect_tx(bar, C::STAGE_BYTES);
                        ptx::tma_load_3d(dst, tmW, bar, kb * BK, wrow, p);
                    }
                } else {
                    ptx::tma_prefetch_l2_3d(tmW, kb * BK, wrow, p);
                    budget -= W_ROWS * BK;
                }
            }
        }
    }
    if (warp == 0) __syncwarp();
    ptx::grid_dependency_wait();

    if (warp == 0) {
        // ---------------- TMA producer ----------------
        // All 32 lanes walk the loop and wait together; an elected one issues the copies.
        // (A warp whose other lanes sit at the final block barrier while one lane works
        // gets scheduled far too rarely.)
        int stage = 0;
        uint32_t phase = 0;
        long long issued = 0;
        bool ok = true;
        for (int i = blockIdx.x; i < a.items && ok; i += gridDim.x) {
            const Item it = item_of<BN, CUT>(a, i, MT, NT);
            const int nt = it.nt, mt = it.mt, p = it.p;
            for (int kb = 0; kb < KB; ++kb) {
                ok = wait_warp(ptx::smem_u32(&sh->empty[stage]), phase ^ 1u, ctx, kWaitSmemEmpty);
                if (!ok) break;
                if (ptx::elect_one() && !(blockIdx.x == 0 && issued == a.debug_skip_stage)) {
                    const uint32_t bar = ptx::smem_u32(&sh->full[stage]);
                    const uint32_t a_dst = ptx::smem_u32(tiles + (size_t)stage * C::STAGE_BYTES);
                    if (issued >= pre) {
                        ptx::mbar_arrive_expect_tx(bar, C::STAGE_BYTES);
                        ptx::tma_load_3d(a_dst, &tmA, bar, kb * BK, mt * BM, p);
                        ptx::tma_load_3d(a_dst + A_BYTES, &tmB, bar, kb * BK, nt * BN, p);
                    } else if (SWAP) {      // the filter half of this stage is already on its way
                        ptx::tma_load_3d(a_dst + A_BYTES, &tmB, bar, kb * BK, nt * BN, p);
                    } else {
                        ptx::tma_load_3d(a_dst, &tmA, bar, kb * BK, mt * BM, p);
                    }
                }
                __syncwarp();
                ++issued;
                if (++stage == NSTAGES) { stage = 0; phase ^= 1u; }
            }
        }
        if (!ok || sh->abort) {
            // give copies still in flight a bounded time to land before the CTA exits
            int s = stage;
            uint32_t ph = phase;
            const long long n = issued < NSTAGES ? issued : NSTAGES;
            for (long long i = 0; i < n; ++i) {
                if (--s < 0) { s = NSTAGES - 1; ph ^= 1u; }
                drain(ptx::smem_u32(&sh->full[s]), ph);
            }
        }
    } else if (warp == 1) {
        // ---------------- MMA issuer ----------------
        // The warp stays converged; an elected lane issues every MMA and commit.  Its instructions
        // form one dependent chain, so the descriptors are advanced with 32-bit adds and
        // the accumulate flag is a constant of the instruction.
        constexpr uint32_t dhi = ptx::smem_desc_sw128_hi();
        const uint32_t tiles_lo = ptx::smem_desc_sw128_lo(ptx::smem_u32(tiles));
        const int chunk_steps = cg * gs_steps;       // MMAs per full chunk
        const int last_slices = (g.C - (KB - 1) * BK) / UK;
        int stage = 0, slot = 0;
        uint32_t phase = 0, sphase = 0;
        bool ok = true;
        // shapes whose chunks tile a stage exactly take the straight-line issue loop
        if (gs_steps == 2 && cg == 2) {
            mma_issue_aligned<BN, SWAP, CUT, 2, 2>(sh, tiles_lo, tmem_base, a, MT, NT, KB, last_slices, ctx);
            ok = false;
        } else if (gs_steps == 4 && cg == 1) {
            mma_issue_aligned<BN, SWAP, CUT, 4, 1>(sh, tiles_lo, tmem_base, a, MT, NT, KB, last_slices, ctx);
            ok = false;
        } else if (gs_steps == 1 && cg == C::CG_MAX && C::CG_MAX <= 4) {
            mma_issue_aligned<BN, SWAP, CUT, 1, (C::CG_MAX <= 4 ? C::CG_MAX : 4)>(sh, tiles_lo, tmem_base, a, MT, NT,
                                                                                  KB, last_slices, ctx);
            ok = false;
        }
        for (int i = blockIdx.x; i < a.items && ok; i += gridDim.x) {
            const Item it = item_of<BN, CUT>(a, i, MT, NT);
            const uint32_t idesc = ptx::idesc_i8(BM, 16 * it.np);
            int step = 0;          // MMA step within the chunk
            int in_group = 0;      // MMA step within the group
            uint32_t dcol = 0;     // TMEM column of the current group
            for (int kb = 0; kb < KB && ok; ++kb) {
                ok = wait_warp(ptx::smem_u32(&sh->full[stage]), phase, ctx, kWaitSmemFull);
                if (!ok) break;
                ptx::tc_fence_after();
                // a 32-byte step along K inside the swizzled rows is +2 in the address field
                const uint32_t a_lo = tiles_lo + (uint32_t)(stage * (C::STAGE_BYTES >> 4));
                const uint32_t b_lo = a_lo + (uint32_t)(A_BYTES >> 4) + (uint32_t)(it.p0 * (16 * BK >> 4));
                const int nslice = min(BK, g.C - kb * BK) / UK;
                for (int s = 0; s < nslice; ++s) {
                    if (step == 0) {
                        // start of a chunk: its TMEM slot must have been drained
                        ok = wait_warp(ptx::smem_u32(&sh->slot_free[slot]), sphase ^ 1u, ctx, kWaitTmemEmpty);
                        if (!ok) break;
                        ptx::tc_fence_after();
                        dcol = tmem_base + (uint32_t)(slot * SLOT_COLS);
                    }
                    if (ptx::elect_one()) {
                        if (in_group) ptx::umma_i8_lo<true>(dcol, a_lo + 2 * s, b_lo + 2 * s, dhi, idesc);
                        else ptx::umma_i8_lo<false>(dcol, a_lo + 2 * s, b_lo + 2 * s, dhi, idesc);
                    }
                    ++step;
                    if (++in_group == gs_steps) { in_group = 0; dcol += BN; }
                    if (step == chunk_steps) {
                        if (ptx::elect_one()) ptx::umma_commit(ptx::smem_u32(&sh->acc_full[slot]));
                        step = 0;
                        if (++slot == NSLOT) { slot = 0; sphase ^= 1u; }
                    }
                }
                if (!ok) break;
                if (ptx::elect_one()) ptx::umma_commit(ptx::smem_u32(&sh->empty[stage]));
                __syncwarp();
                if (++stage == NSTAGES) { stage = 0; phase ^= 1u; }
            }
            if (ok && step != 0) {
                // the last chunk of the unit has fewer groups than a full one
                if (ptx::elect_one()) ptx::umma_commit(ptx::smem_u32(&sh->acc_full[slot]));
                __syncwarp();
                if (++slot == NSLOT) { slot = 0; sphase ^= 1u; }
            }
        }
    } else if (warp == 2) {
        // ---------------- scale loader ----------------
        if (!DUMP) {
            int slot = 0;
            uint32_t sphase = 0;
            long long issued = 0;
            bool ok = true;
            for (int i = blockIdx.x; i < a.items && ok; i += gridDim.x) {
                const Item it = item_of<BN, CUT>(a, i, MT, NT);
                const int nt = it.nt, mt = it.mt, p = it.p;
                for (int ch = 0; ch < nchunk; ++ch) {
                    const int g0 = ch * cg, ng = min(cg, g.G - g0);
                    ok = wait_warp(ptx::smem_u32(&sh->slot_free[slot]), sphase ^ 1u, ctx, kWaitScaleEmpty);
                    if (!ok) break;
                    const uint32_t bar = ptx::smem_u32(&sh->acc_full[slot]);
                    const uint32_t dst = ptx::smem_u32(scales + (size_t)slot * C::SLOT_SCALE_FLOATS);
                    if (ptx::elect_one()) ptx::mbar_arrive_expect_tx(bar, (uint32_t)(ng * C::GROUP_SCALE_FLOATS * 4));
                    __syncwarp();
                    // lane j copies the row scales of group j, lane 4 + j its column scales
                    if (lane < 8 && (lane & 3) < ng) {
                        const int j = lane & 3;
                        const size_t pg = (size_t)p * g.G + g0 + j;
                        const uint32_t d = dst + (uint32_t)(j * C::GROUP_SCALE_FLOATS * 4);
                        if (lane < 4)
                            ptx::bulk_load(d, a.row_scale + pg * a.row_pitch + mt * BM, BM * 4, bar);
                        else
                            ptx::bulk_load(d + BM * 4, a.col_scale + pg * a.col_pitch + nt * BN, BN * 4, bar);
                    }
                    __syncwarp();
                    ++issued;
                    if (++slot == NSLOT) { slot = 0; sphase ^= 1u; }
                }
            }
            if (!ok || sh->abort) {      // where the chunk's MMAs were not issued this runs out its limit, the copies land
                int s = slot;
                uint32_t ph = sphase;
                const long long n = issued < NSLOT ? issued : NSLOT;
                for (long long i = 0; i < n; ++i) {
                    if (--s < 0) { s = NSLOT - 1; ph ^= 1u; }
                    drain(ptx::smem_u32(&sh->acc_full[s]), ph);
                }
            }
        }
    } else if (warp >= FIRST_EPI_WARP) {
        // ---------------- epilogue ----------------
        const int quarter = warp & 3;                         // TMEM lanes this warp may read
        int slot = 0;
        uint32_t sphase = 0;
        bool ok = true;
        const EpiCtx ec{tmem_base + ((uint32_t)(quarter * 32) << 16), scales,
                        store + quarter * (C::STORE_BYTES / NUM_EPI_WARPS), quarter, lane, nchunk};
        // The parts of cut units (at most one per CTA) run code of their own: a bound on the pieces inside the unrolled
        // loops keeps the compiler from interleaving them (34 layers 5 % slower, up to 13 %)
        for (int i = blockIdx.x; i < a.whole && ok; i += gridDim.x) {
            const Item it = item_of<BN, false>(a, i, MT, NT);
            ok = epilogue_unit<BN, SWAP, DUMP, CUT, BN / 16>(sh, tmY, a, g, ctx, ec, it.p, it.mt, it.nt * BN, 0, slot,
                                                             sphase);
        }
        const int tail = a.whole + (int)blockIdx.x;
        if (CUT && tail < a.items && ok) {
            const Item it = item_of<BN, CUT>(a, tail, MT, NT);
            ok = epilogue_unit<BN, SWAP, DUMP, CUT, part_pieces(BN)>(sh, tmY, a, g, ctx, ec, it.p, it.mt, it.nt * BN,
                                                                     16 * it.p0, slot, sphase);
        }
        if constexpr (!DUMP && !SWAP) {
            if (lane == 0) ptx::bulk_wait();
            __syncwarp();
        }
    }

    ptx::tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        if (sh->abort) {      // a wait ran out: MMAs may still be reading the stages and writing the accumulators
            if (ptx::elect_one()) ptx::umma_commit(ptx::smem_u32(&sh->mma_done));
            __syncwarp();
            drain(ptx::smem_u32(&sh->mma_done), 0);
        }
        ptx::tc_fence_after();
        ptx::tmem_dealloc(tmem_base, TMEM_COLS);
    }
}

// Groups per chunk: as many whole groups as fit into 128 channels (one stage) and into one TMEM slot; group sizes that
// do not divide 128 get one group per chunk.
int groups_per_chunk(int gs, int bn)
{
    if (BK % gs != 0) return 1;
    return BK / gs < SLOT_COLS / bn ? BK / gs : SLOT_COLS / bn;
}

template <int BN, bool SWAP, bool DUMP>
cudaError_t launch_variant(const wfq_plan &plan, int32_t *acc_dump, cudaStream_t stream, bool pdl)
{
    using C = Cfg<BN, SWAP>;
    const Geometry &g = plan.geo;
    GemmArgs a;
    a.row_scale = SWAP ? plan.sW : plan.ws.sX;
    a.col_scale = SWAP ? plan.ws.sX : plan.sW;
    a.row_pitch = SWAP ? g.Kp : g.Ts;
    a.col_pitch = SWAP ? g.Ts : g.Kp;
    a.rows = SWAP ? g.K : g.T;
    a.cols = SWAP ? g.T : g.K;
    a.cg = groups_per_chunk(g.gs, BN);
    a.Y = plan.ws.Y;
    a.acc_dump = acc_dump;
    a.status = plan.status;
    a.wait_cycles = plan.wait_cycles;
    a.debug_skip_stage = plan.debug_skip_gemm_stage;
    const int MT = (a.rows + BM - 1) / BM, NT = (a.cols + BN - 1) / BN;
    const int units = g.P * MT * NT;
    a.whole = DUMP ? units : plan.gemm_whole;     // the debug output is not cut
    a.items = a.whole + (units - a.whole) * plan.gemm_parts;
    a.by_NT = plan.gemm_by_nt;
    a.by_MT = plan.gemm_by_mt;
    const int grid = a.items < plan.gemm_ctas ? a.items : plan.gemm_ctas;   // the layout above is for this grid alone
    // the filters share L2 (126 MB) with Xq, sX and Y: at most 48 MB of them are asked for early
    a.l2_prefetch_bytes = pdl ? (48LL << 20) / grid : 0;
    auto kern = gemm_dequant_kernel<BN, SWAP, DUMP, false>;
    if constexpr (BN != 16 && !DUMP)
        if (plan.gemm_parts > 1) kern = gemm_dequant_kernel<BN, SWAP, DUMP, true>;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3(NUM_THREADS);
    cfg.dynamicSmemBytes = C::SMEM_BYTES;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = pdl ? 1 : 0;
    const CUtensorMap &tmA = SWAP ? plan.tmap_wq : plan.tmap_xq;
    const CUtensorMap &tmB = SWAP ? plan.tmap_xq : plan.tmap_wq;
    return cudaLaunchKernelEx(&cfg, kern, tmA, tmB, plan.tmap_y, a, g);
}

// ---- tensor-pipe rate of tcgen05.mma kind::i8 -----------------------------------------
// One CTA per SM issues `mmas` accumulating 128 x BN x 32 MMAs on operands that stay in
// shared memory (no global traffic), then waits (bounded) for the last one.  Timed by the
// caller with events: grid * mmas * 2 * 128 * BN * 32 operations.
struct PeakShared { uint64_t done; uint32_t tmem_base; volatile int abort; };

template <int BN>
__global__ void __launch_bounds__(128, 1) mma_peak_kernel(int mmas, int *status, long long wait_cycles)
{
    extern __shared__ unsigned char smem_raw[];
    unsigned char *tiles = ptx::align_smem<1024>(smem_raw);
    constexpr int BYTES = (BM + BN) * BK;
    PeakShared *sh = reinterpret_cast<PeakShared *>(tiles + BYTES);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int i = threadIdx.x; i < BYTES / 4; i += blockDim.x) reinterpret_cast<uint32_t *>(tiles)[i] = 0x01010101u;
    if (threadIdx.x == 0) {
        ptx::mbar_init(ptx::smem_u32(&sh->done), 1);
        sh->abort = 0;
        ptx::fence_mbar_init();
    }
    if (warp == 0) {
        ptx::tmem_alloc(ptx::smem_u32(&sh->tmem_base), BN < 32 ? 32 : BN);
        ptx::tmem_relinquish();
    }
    ptx::fence_proxy_async_smem();
    ptx::tc_fence_before();
    __syncthreads();
    ptx::tc_fence_after();
    const uint32_t tmem = sh->tmem_base;
    if (warp == 0) {
        const WaitCtx ctx{&sh->abort, status, wait_cycles};
        if (lane == 0) {
            constexpr uint32_t idesc = ptx::idesc_i8(BM, BN);
            constexpr uint32_t dhi = ptx::smem_desc_sw128_hi();
            const uint32_t a_lo = ptx::smem_desc_sw128_lo(ptx::smem_u32(tiles));
            const uint32_t b_lo = a_lo + (uint32_t)(A_BYTES >> 4);
            for (int i = 0; i < mmas; i += 4) {
                ptx::umma_i8_lo<true>(tmem, a_lo, b_lo, dhi, idesc);
                ptx::umma_i8_lo<true>(tmem, a_lo + 2, b_lo + 2, dhi, idesc);
                ptx::umma_i8_lo<true>(tmem, a_lo + 4, b_lo + 4, dhi, idesc);
                ptx::umma_i8_lo<true>(tmem, a_lo + 6, b_lo + 6, dhi, idesc);
            }
            ptx::umma_commit(ptx::smem_u32(&sh->done));
        }
        __syncwarp();
        wait_warp(ptx::smem_u32(&sh->done), 0, ctx, kWaitTmemFull);
    }
    ptx::tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        ptx::tc_fence_after();
        ptx::tmem_dealloc(tmem, BN < 32 ? 32 : BN);
    }
}

template <int BN>
cudaError_t launch_peak(int grid, int mmas, int *status, long long wait_cycles, cudaStream_t stream)
{
    const int smem = 1024 + (BM + BN) * BK + (int)sizeof(PeakShared);
    cudaError_t e = cudaFuncSetAttribute(mma_peak_kernel<BN>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    mma_peak_kernel<BN><<<grid, 128, smem, stream>>>(mmas, status, wait_cycles);
    return cudaGetLastError();
}

template <int BN, bool SWAP, bool DUMP>
cudaError_t setup_variant()
{
    if constexpr (BN != 16 && !DUMP) {
        const cudaError_t e = cudaFuncSetAttribute(gemm_dequant_kernel<BN, SWAP, DUMP, true>,
                                                   cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                   (int)Cfg<BN, SWAP>::SMEM_BYTES);
        if (e != cudaSuccess) return e;
    }
    return cudaFuncSetAttribute(gemm_dequant_kernel<BN, SWAP, DUMP, false>,
                                cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Cfg<BN, SWAP>::SMEM_BYTES);
}

}  // namespace

// One-time attribute setting for the kernels of this file (per device).
cudaError_t setup_gemm()
{
    cudaError_t e = setup_variant<16, true, true>();
    if (e == cudaSuccess) e = setup_variant<16, true, false>();
    if (e == cudaSuccess) e = setup_variant<16, false, true>();
    if (e == cudaSuccess) e = setup_variant<16, false, false>();
    if (e == cudaSuccess) e = setup_variant<32, true, true>();
    if (e == cudaSuccess) e = setup_variant<32, true, false>();
    if (e == cudaSuccess) e = setup_variant<48, true, true>();
    if (e == cudaSuccess) e = setup_variant<48, true, false>();
    if (e == cudaSuccess) e = setup_variant<64, true, true>();
    if (e == cudaSuccess) e = setup_variant<64, true, false>();
    if (e == cudaSuccess) e = setup_variant<64, false, true>();
    if (e == cudaSuccess) e = setup_variant<64, false, false>();
    return e;
}

cudaError_t launch_mma_peak(const wfq_plan &plan, int n_cols, int mmas, cudaStream_t stream)
{
    const int grid = plan.sm_count;
    switch (n_cols) {
        case 64: return launch_peak<64>(grid, mmas, plan.status, plan.wait_cycles, stream);
        case 128: return launch_peak<128>(grid, mmas, plan.status, plan.wait_cycles, stream);
        case 256: return launch_peak<256>(grid, mmas, plan.status, plan.wait_cycles, stream);
        default: return cudaErrorInvalidValue;
    }
}

// Which units are cut into parts along their columns, and the box of the stores of Y.  A last round that leaves CTAs
// without a unit takes as long as a full one; where it holds no more units than parts of them have room, each CTA of
// it takes a part (forward: 360 units of 5 chunks on 296 CTAs 33.4 -> 32.4 us, 640 units 35.8 -> 34.9 us, swapped in
// thirds of 48 columns 43.6 -> 42.5 us, 54 units of 3 chunks 13.8 -> 12.8 us).  Units of one chunk are no shorter in
// parts (84 of 972 units with 40 columns 23.9 -> 24.5 us), nor is a unit whose columns all lie in its first part.
// Quarters of 64 columns, where they fit, are as good as halves (F(2,3) 1216 channels 78.9 -> 77.0 us, 640 units
// 34.9 -> 35.4 us).
bool plan_gemm_units(wfq_plan &plan)
{
    const Geometry &g = plan.geo;
    const int bn = plan.gemm_bn, rows = plan.gemm_swap ? g.K : g.T, cols = plan.gemm_swap ? g.T : g.K;
    const int units = g.P * ((rows + BM - 1) / BM) * ((cols + bn - 1) / bn);
    int ctas = plan.debug_gemm_ctas > 0 ? plan.debug_gemm_ctas : 2 * plan.sm_count;     // two per SM
    if (ctas < 1) ctas = 1;
    const int rest = units % ctas;
    const int part = 16 * part_pieces(bn), parts = bn / part;
    const int cg = groups_per_chunk(g.gs, bn);
    const bool cut = parts > 1 && rest > 0 && parts * rest <= ctas && (g.G + cg - 1) / cg > 1 && cols > part;
    plan.gemm_ctas = ctas;
    plan.gemm_whole = cut ? units - rest : units;
    plan.gemm_parts = cut ? parts : 1;
    plan.gemm_by_nt = FastDiv((cols + bn - 1) / bn);
    plan.gemm_by_mt = FastDiv((rows + BM - 1) / BM);
    const unsigned long long dims[3] = {(unsigned long long)g.T, (unsigned long long)g.K, (unsigned long long)g.P};
    const unsigned long long strides[2] = {(unsigned long long)g.Tp * 4, (unsigned long long)g.K * g.Tp * 4};
    const unsigned box[3] = {32u, (unsigned)(cut ? part : bn), 1u};
    return encode_tmap(&plan.tmap_y, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, plan.ws.Y, dims, strides, box,
                       CU_TENSOR_MAP_SWIZZLE_NONE);
}

int gemm_block_m() { return BM; }

// Orientation and column block of the contraction for a layer: rows (TMEM lanes) are
// tiles unless the swapped orientation leaves less padded work.
void gemm_choose(const Geometry &g, bool *swap, int *bn)
{
    auto up = [](long long v, int b) { return (v + b - 1) / b * b; };
    const long long normal = up(g.T, BM) * up(g.K, 64);
    // swapped: the tile columns are padded to a multiple of the column block (32, 48 or 64:
    // every padded column is promoted like a real one); the largest block among the least padded
    int bn_sw = 64;
    for (int c : {48, 32})
        if (up(g.T, c) < up(g.T, bn_sw)) bn_sw = c;
    const long long swapped = up(g.K, BM) * up(g.T, bn_sw);
    *swap = 5 * swapped < 4 * normal;   // swapped stores are less efficient: want >= 20 % less work
    *bn = *swap ? bn_sw : 64;
}

cudaError_t launch_gemm(const wfq_plan &plan, int32_t *acc_dump, cudaStream_t stream, bool pdl)
{
    const bool dump = acc_dump != nullptr;
    // 16 columns: never chosen by gemm_choose, only by the debug option (the shape a contraction
    // fused with the output transform would be confined to by its accumulator space)
    if (plan.gemm_bn == 16) {
        if (plan.gemm_swap)
            return dump ? launch_variant<16, true, true>(plan, acc_dump, stream, pdl)
                        : launch_variant<16, true, false>(plan, acc_dump, stream, pdl);
        return dump ? launch_variant<16, false, true>(plan, acc_dump, stream, pdl)
                    : launch_variant<16, false, false>(plan, acc_dump, stream, pdl);
    }
    if (plan.gemm_swap) {
        if (plan.gemm_bn == 32)
            return dump ? launch_variant<32, true, true>(plan, acc_dump, stream, pdl)
                        : launch_variant<32, true, false>(plan, acc_dump, stream, pdl);
        if (plan.gemm_bn == 48)
            return dump ? launch_variant<48, true, true>(plan, acc_dump, stream, pdl)
                        : launch_variant<48, true, false>(plan, acc_dump, stream, pdl);
        return dump ? launch_variant<64, true, true>(plan, acc_dump, stream, pdl)
                    : launch_variant<64, true, false>(plan, acc_dump, stream, pdl);
    }
    return dump ? launch_variant<64, false, true>(plan, acc_dump, stream, pdl)
                : launch_variant<64, false, false>(plan, acc_dump, stream, pdl);
}

}  // namespace wfq
