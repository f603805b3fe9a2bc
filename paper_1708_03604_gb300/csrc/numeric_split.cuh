// The split paths on the tensor cores (TF32x3, BF16x3, BF16x6): device code and
// launchers, one translation unit per precision (k_split_*.cu), and the parts of
// it that the packing and the Ozaki kernels in k_numeric.cu share.
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "bsm_internal.cuh"
#include "numeric_debug.cuh"

namespace bsm {

namespace {

constexpr int kWarpsPerCta = 4;             // default warps per CTA
constexpr int kThreadsNum = kWarpsPerCta * 32;

// =====================================================================
// Tensor-core split path
// =====================================================================
// Packed fragment planes.  For a logical R x T operand in role X (mma "A"
// operand) the tiles are (kt, mt) with MT = ceil(R/16), kt over K steps;
// for a logical T x S operand in role Y ("B" operand) tiles are (kt, nt)
// with NT = ceil(S/8).  Words per lane per tile:
//   prec      K step   X words   Y words
//   TF32x3       8        8         4      (hi[4] lo[4] | hi[2] lo[2])
//   BF16x3      16        8         4      (hi[4] lo[4] | hi[2] lo[2])
//   BF16x6      16       12         8      (p0[4] p1[4] p2[4] | p0[2] p1[2] p2[2] pad[2])
// Inside a tile the words are chunk-major: 16-byte chunk c of lane L at word
// c * 128 + 4 * L (X chunk = one piece, Y chunk = two pieces), so a 16-byte
// copy of the warp reads 512 contiguous bytes.  In X blocks of up to 8 and of
// 17 to 24 rows the registers of rows 8..15 (v1, v3) of the last tile row are all
// zeros: its tiles hold v0 and v2 of every piece only, HW words per lane, two
// pieces to a chunk.
template <int PREC> struct PrecTraits;
// whether the last tile row of a block of R rows is half a tile.  Higher blocks
// keep whole tiles: their half would take a second copy of every pass in the 2 x
// PN instance, and 300 rows of blocks of 1 to 40 lost 12% to the larger code.
__host__ __device__ constexpr bool half_tile(int R) { return R <= 8 || (R > 16 && R <= 24); }
template <> struct PrecTraits<BSM_P_TF32x3> { static constexpr int K = 8, XW = 8, HW = 4, YW = 4, NP = 2; };
template <> struct PrecTraits<BSM_P_BF16x3> { static constexpr int K = 16, XW = 8, HW = 4, YW = 4, NP = 2; };
template <> struct PrecTraits<BSM_P_BF16x6> { static constexpr int K = 16, XW = 12, HW = 8, YW = 8, NP = 3; };

__device__ __forceinline__ void mma_tf32(float (&d)[4], const uint32_t (&a)[4], const uint32_t (&b)[2]) {
    asm(
        "mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
        "{%0,%1,%2,%3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}
__device__ __forceinline__ void mma_bf16(float (&d)[4], const uint32_t (&a)[4], const uint32_t (&b)[2]) {
    asm(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
        "{%0,%1,%2,%3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

template <int PREC>
__device__ __forceinline__ void mma_piece(float (&d)[4], const uint32_t (&a)[4], const uint32_t (&b)[2]) {
    if constexpr (PREC == BSM_P_TF32x3) mma_tf32(d, a, b);
    else mma_bf16(d, a, b);
}

// Per-lane staging ring: every lane copies its own fragment words of the
// next (product, k-step) steps from global memory into its private slots of
// shared memory with cp.async and reads back only those words, so the ring
// needs no warp barrier -- only each lane's own cp.async.wait_group.  A stage
// is chunk-major like the packs (chunk c of lane L at word c * 128 + 4 * L):
// every 16-byte copy and read of the warp covers 512 contiguous bytes.
// Stages, and words per lane of a stage for passes of at most PM x PN tiles.
// A kernel instance compiled for smaller passes holds fewer accumulators and
// a smaller ring, so more warps fit on an SM.
// HALF: the last of the PM tile rows is a half tile.
template <int PREC, int PM, int PN, bool HALF> struct RingTraits {
    static constexpr int STAGES = PREC == BSM_P_BF16x6 ? 3 : 4;
    static constexpr int SW = (PM - 1) * PrecTraits<PREC>::XW + (HALF ? PrecTraits<PREC>::HW : PrecTraits<PREC>::XW) +
                              PN * PrecTraits<PREC>::YW;
};

template <int PREC, int PM, int PN, bool HALF>
__host__ __device__ constexpr int ring_words_per_warp() {
    return RingTraits<PREC, PM, PN, HALF>::STAGES * 32 * RingTraits<PREC, PM, PN, HALF>::SW;
}

__device__ __forceinline__ uint32_t smem_addr(const void *p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
// 16-byte asynchronous copy global -> shared, cached in L2 only (the staged
// fragment words are read once per warp)
__device__ __forceinline__ void cp_async16_cg(uint32_t dst, const void *src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src));
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N)); }

// Compensated (Kahan) addition of b into the pair (hi, lo), value hi + lo:
// the low part lost by each addition is fed into the next one (4 FP32 adds;
// error below about 2u of the sum of |b|, u = 2^-24).
__device__ __forceinline__ void kahan_acc(float &hi, float &lo, float b) {
    const float y = __fadd_rn(b, lo);
    const float t = __fadd_rn(hi, y);
    lo = __fsub_rn(y, __fsub_rn(t, hi));
    hi = t;
}

// FP32 -> FP64 (exact).  Widening by integer bit operations instead of the
// conversion instruction was measured no faster on GB300: the FP64 additions,
// not the conversions, are what the FP64 running sum pays for.
__device__ __forceinline__ double widen(float f) { return (double)f; }

// The value of a compensated pair (hi, lo) plus a last partial sum b, in
// FP64: b is first added into the pair in FP32 (one more compensated step),
// then the pair is widened and added once.
__device__ __forceinline__ double pair_total(float hi, float lo, float b) {
    kahan_acc(hi, lo, b);
    return widen(hi) + widen(lo);
}

// One pass over a super tile of MTC x NTC (at most 2 x 3) fragment tiles
// starting at (mt0, nt0) of output block q: at most 32 x 24 output elements.
// FF: cross-product sum as a compensated float pair (Kahan after every |F| block
// products); otherwise an FP64 sum refreshed every F products.  HALF: the last
// of the MTC tile rows is a half tile; rows 8..15 of its MMAs are zeros, and half
// of its sums and X words fall away.  RT: the ring of the kernel instance.
//
// Bound by the issue of instructions: a product of 23 x 23 x 23 takes 54 MMAs,
// and the copies, fragment reads and sums around them are as many again.  So the
// cursors are running pointers, no tile of a pass is tested (every one exists),
// and the empty half of a half tile is neither copied nor summed.
// Numeric pass in TF32x3, before and after, blocks of 5: 15.4 -> 11.7 ms (8e7
// products), of 13: 3.36 -> 2.87 (6.8e6), of 23: 2.17 -> 1.76 (1.2e6), of 32: 2.08
// -> 1.80 (4.5e5); 3,000 block rows of 5/13/23: 65 -> 49.
template <int PREC, int MTC, int NTC, bool FF, typename RT, bool DUAL, bool HALF>
__device__ __forceinline__ void tc_pass(const NumericArgs &a, int64_t q, int lane, int mt0, int nt0,
                                        uint32_t *ring) {
    using PT = PrecTraits<PREC>;
    constexpr int ST = RT::STAGES, SW = RT::SW;
    const int32_t orc = a.out_blk_rc[q];
    const int R = rc_rows(orc), S = rc_cols(orc);
    const int MT = (R + 15) >> 4, NT = (S + 7) >> 3;
    const int64_t p0 = a.seg_ptr[q], p1 = a.seg_ptr[q + 1];
    const uint32_t *XP = static_cast<const uint32_t *>(a.x_pack);
    const uint32_t *YP = static_cast<const uint32_t *>(a.y_pack);
    // FP64 mode: flush_every > 0 products per FP64 add; compensated mode:
    // |flush_every| products per compensated addition (0 means 1)
    const int F = a.flush_every > 0 ? a.flush_every : (a.flush_every < 0 ? -a.flush_every : 1);
    uint32_t *myring = ring + 4 * lane;  // chunk c of stage st at myring + st * 32 * SW + 128 * c
    const uint32_t ring_s = smem_addr(myring);
    constexpr int XC = PT::XW / 4, HC = PT::HW / 4, YC = PT::YW / 4;  // chunks per tile
    constexpr int XT = (MTC - 1) * XC + (HALF ? HC : XC);             // X chunks of a stage
    // words of one k-step of an X and a Y block
    const int xk = 32 * (PT::XW * (MT - 1) + (half_tile(R) ? PT::HW : PT::XW)), yk = 32 * PT::YW * NT;
    XP += mt0 * (32 * PT::XW) + 4 * lane;
    YP += nt0 * (32 * PT::YW) + 4 * lane;
    // accumulator elements of a lane that count in tile row i
    auto elems = [](int i) { return HALF && i == MTC - 1 ? 2 : 4; };

    // DUAL (1-row instances summing more than one block product in the tensor
    // core, F > 1): the piece products of a k-step alternate between two
    // accumulators (term t into acc if t is even, acc2 if odd), so that the
    // tensor core's chain of dependent MMAs on one tile is about half as long;
    // the two are added (FP32, to nearest) where the single one was read
    float acc[MTC][NTC][4], acc2[DUAL ? MTC : 1][DUAL ? NTC : 1][4];
    float shi[FF ? MTC : 1][FF ? NTC : 1][4], slo[FF ? MTC : 1][FF ? NTC : 1][4];
    double s64[FF ? 1 : MTC][FF ? 1 : NTC][4];
#pragma unroll
    for (int i = 0; i < MTC; ++i)
#pragma unroll
        for (int j = 0; j < NTC; ++j)
#pragma unroll
            for (int v = 0; v < 4; ++v) {
                acc[i][j][v] = 0.f;
                if constexpr (DUAL) acc2[i][j][v] = 0.f;
                if constexpr (FF) {
                    shi[i][j][v] = 0.f;
                    slo[i][j][v] = 0.f;
                } else {
                    s64[i][j][v] = 0.0;
                }
            }
    int since = 0;
    for (int64_t pb = p0; pb < p1; pb += 32) {
        const int nb = (int)min((int64_t)32, p1 - pb);
        // metadata of up to 32 products, one per lane
        int64_t mxo = 0, myo = 0;
        int mkt = 0;
        if (lane < nb) {
            const int32_t ix = a.px[pb + lane], iy = a.py[pb + lane];
            const int32_t xrc = a.x_blk_rc[ix];
            const int Tn = a.x_trans ? rc_rows(xrc) : rc_cols(xrc);
            mxo = a.x_pack_off[ix];
            myo = a.y_pack_off[iy];
            mkt = (Tn + PT::K - 1) / PT::K;
        }
        int nsteps = mkt;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) nsteps += __shfl_xor_sync(0xffffffffu, nsteps, o);
        // producer cursor over the (product, k-step) sequence
        int pu = 0, pk = __shfl_sync(0xffffffffu, mkt, 0);  // product; its k-steps left
        const uint32_t *xs = XP + __shfl_sync(0xffffffffu, mxo, 0), *ys = YP + __shfl_sync(0xffffffffu, myo, 0);
        auto produce = [&](uint32_t dst) {
#pragma unroll
            for (int i = 0; i < MTC; ++i)
#pragma unroll
                for (int c = 0; c < (HALF && i == MTC - 1 ? HC : XC); ++c)
                    cp_async16_cg(dst + 512u * (i * XC + c), xs + i * (32 * PT::XW) + 128 * c);
#pragma unroll
            for (int j = 0; j < NTC; ++j)
#pragma unroll
                for (int c = 0; c < YC; ++c)
                    cp_async16_cg(dst + 512u * (XT + j * YC + c), ys + j * (32 * PT::YW) + 128 * c);
            xs += xk;
            ys += yk;
            if (--pk == 0) {
                ++pu;
                const int src_lane = pu < nb ? pu : 0;
                xs = XP + __shfl_sync(0xffffffffu, mxo, src_lane);
                ys = YP + __shfl_sync(0xffffffffu, myo, src_lane);
                pk = __shfl_sync(0xffffffffu, mkt, src_lane);
            }
        };
#pragma unroll
        for (int st = 0; st < ST - 1; ++st) {
            if (st < nsteps) produce(ring_s + (uint32_t)(st * 128 * SW));
            cp_async_commit();
        }
        int cu = 0, ck = __shfl_sync(0xffffffffu, mkt, 0);
        uint32_t rd = 0, wr = (ST - 1) * 128 * SW;  // bytes into the ring of the stages read and filled
        for (int s = 0; s < nsteps; ++s) {
            if (s + ST - 1 < nsteps) produce(ring_s + wr);
            cp_async_commit();
            cp_async_wait<ST - 1>();
            const uint32_t *w = myring + rd / 4;
            rd = rd == (ST - 1) * 128 * SW ? 0 : rd + 128 * SW;
            wr = wr == (ST - 1) * 128 * SW ? 0 : wr + 128 * SW;
            uint32_t fa[MTC][PT::NP][4];
#pragma unroll
            for (int i = 0; i < MTC; ++i) {
                if (HALF && i == MTC - 1) {
#pragma unroll
                    for (int pc = 0; pc < PT::NP; pc += 2) {
                        const uint4 v = *reinterpret_cast<const uint4 *>(w + 128 * (i * XC + (pc >> 1)));
                        fa[i][pc][0] = v.x; fa[i][pc][1] = 0u; fa[i][pc][2] = v.y; fa[i][pc][3] = 0u;
                        if (pc + 1 < PT::NP) {
                            fa[i][pc + 1][0] = v.z; fa[i][pc + 1][1] = 0u; fa[i][pc + 1][2] = v.w; fa[i][pc + 1][3] = 0u;
                        }
                    }
                } else {
#pragma unroll
                    for (int pc = 0; pc < PT::NP; ++pc) {
                        const uint4 v = *reinterpret_cast<const uint4 *>(w + 128 * (i * XC + pc));
                        fa[i][pc][0] = v.x; fa[i][pc][1] = v.y; fa[i][pc][2] = v.z; fa[i][pc][3] = v.w;
                    }
                }
            }
            uint32_t fb[NTC][PT::NP][2];
#pragma unroll
            for (int j = 0; j < NTC; ++j) {
                const uint32_t *wy = w + 128 * (XT + j * YC);
                const uint4 v = *reinterpret_cast<const uint4 *>(wy);
                fb[j][0][0] = v.x; fb[j][0][1] = v.y; fb[j][1][0] = v.z; fb[j][1][1] = v.w;
                if constexpr (PT::NP == 3) {
                    const uint2 u = *reinterpret_cast<const uint2 *>(wy + 128);
                    fb[j][2][0] = u.x; fb[j][2][1] = u.y;
                }
            }
            // piece products, smallest first; consecutive mma instructions go
            // to different tiles so their accumulator chains overlap
            constexpr int NTERM = PT::NP == 2 ? 3 : 6;
            constexpr int TA[6] = {1, 0, 0, 0, 0, 0}, TB[6] = {0, 1, 0, 0, 0, 0};
            constexpr int SA[6] = {2, 1, 0, 1, 0, 0}, SB[6] = {0, 1, 2, 0, 1, 0};
#pragma unroll
            for (int t = 0; t < NTERM; ++t) {
                const int ia = PT::NP == 2 ? TA[t] : SA[t];
                const int ib = PT::NP == 2 ? TB[t] : SB[t];
#pragma unroll
                for (int j = 0; j < NTC; ++j)
#pragma unroll
                    for (int i = 0; i < MTC; ++i) {
                        if (DUAL && (t & 1)) mma_piece<PREC>(acc2[DUAL ? i : 0][DUAL ? j : 0], fa[i][ia], fb[j][ib]);
                        else mma_piece<PREC>(acc[i][j], fa[i][ia], fb[j][ib]);
                    }
            }
            if (--ck == 0) {  // a block product is complete
                ++cu;
                ck = __shfl_sync(0xffffffffu, mkt, cu < nb ? cu : 0);
                if (++since == F) {
                    since = 0;
#pragma unroll
                    for (int i = 0; i < MTC; ++i)
#pragma unroll
                        for (int j = 0; j < NTC; ++j)
#pragma unroll
                            for (int v = 0; v < elems(i); ++v) {
                                float part = acc[i][j][v];
                                if constexpr (DUAL) {
                                    part = __fadd_rn(part, acc2[DUAL ? i : 0][DUAL ? j : 0][v]);
                                    acc2[DUAL ? i : 0][DUAL ? j : 0][v] = 0.f;
                                }
                                if constexpr (FF) kahan_acc(shi[i][j][v], slo[i][j][v], part);
                                else s64[i][j][v] += widen(part);
                                acc[i][j][v] = 0.f;
                            }
                }
            }
        }
        cp_async_wait<0>();
    }
    // epilogue: fragment element v of tile (i, j) sits at
    // row (mt0+i)*16 + g + 8*(v>=2), column (nt0+j)*8 + 2*t4 + (v&1)
    const int g = lane >> 2, t4 = lane & 3;
    const int64_t out_off = a.out_blk_off[q];
    const int64_t old = (a.beta != 0.0 && a.old_off) ? a.old_off[q] : -1;
#pragma unroll
    for (int i = 0; i < MTC; ++i)
#pragma unroll
        for (int j = 0; j < NTC; ++j)
#pragma unroll
            for (int v = 0; v < elems(i); ++v) {
                const int r = (mt0 + i) * 16 + g + ((v >> 1) << 3);
                const int c = (nt0 + j) * 8 + 2 * t4 + (v & 1);
                if (r < R && c < S) {
                    double sum;
                    float part = acc[i][j][v];
                    if constexpr (DUAL) part = __fadd_rn(part, acc2[DUAL ? i : 0][DUAL ? j : 0][v]);
                    if constexpr (FF) sum = pair_total(shi[i][j][v], slo[i][j][v], part);
                    else sum = s64[i][j][v] + widen(part);
                    double val = a.alpha == 1.0 ? sum : a.alpha * sum;
                    const int64_t e = (int64_t)r * S + c;
                    if (a.dtype == BSM_FP64) {
                        if (old >= 0) val = fma(a.beta, static_cast<const double *>(a.old_data)[old + e], val);
                        static_cast<double *>(a.out_data)[out_off + e] = val;
                    } else {
                        if (old >= 0) val = fma(a.beta, (double)static_cast<const float *>(a.old_data)[old + e], val);
                        static_cast<float *>(a.out_data)[out_off + e] = (float)val;
                    }
                }
            }
}

// the passes over tile rows mt0 .. mt0 + MTC - 1
template <int PREC, int MTC, bool FF, int PN, typename RT, bool DUAL, bool HALF>
__device__ __forceinline__ void tc_row(const NumericArgs &a, int64_t q, int lane, int mt0, int NT, int pn, uint32_t *ring) {
    for (int nt0 = 0; nt0 < NT; nt0 += pn) {
        const int ntc = min(pn, NT - nt0);
        if (PN == 1 || ntc == 1) tc_pass<PREC, MTC, 1, FF, RT, DUAL, HALF>(a, q, lane, mt0, nt0, ring);
        else if constexpr (PN >= 2) {
            if (PN == 2 || ntc == 2) tc_pass<PREC, MTC, 2, FF, RT, DUAL, HALF>(a, q, lane, mt0, nt0, ring);
            else if constexpr (PN >= 3) tc_pass<PREC, MTC, 3, FF, RT, DUAL, HALF>(a, q, lane, mt0, nt0, ring);
        }
    }
}

// The blocks that an instance takes: kAny of any height; of one class: kWhole
// without a half tile, kHalf of exactly PM tile rows, the last a half one.
enum TcHeights { kAny, kWhole, kHalf };

template <int PREC, bool FF, int PM, int PN, bool DUAL, TcHeights H>
__device__ __forceinline__ void tc_item(const NumericArgs &a, int64_t q, int lane, uint32_t *ring) {
    using RT = RingTraits<PREC, PM, PN, H == kHalf>;
    const int32_t orc = a.out_blk_rc[q];
    const int MT = (rc_rows(orc) + 15) >> 4, NT = (rc_cols(orc) + 7) >> 3;
    const int pm = min(PM, a.pass_mt > 0 ? a.pass_mt : PM), pn = min(PN, a.pass_nt > 0 ? a.pass_nt : PN);
    if constexpr (H == kHalf) {
        tc_row<PREC, PM, FF, PN, RT, DUAL, true>(a, q, lane, 0, NT, pn, ring);
    } else {
        const bool half = H == kAny && half_tile(rc_rows(orc));
        for (int mt0 = 0; mt0 < MT; mt0 += pm) {
            const int mtc = min(pm, MT - mt0);
            const bool h = half && mt0 + mtc == MT;
            if (PM == 1 || mtc == 1) {
                if (!h) tc_row<PREC, 1, FF, PN, RT, DUAL, false>(a, q, lane, mt0, NT, pn, ring);
                else if constexpr (H == kAny) tc_row<PREC, 1, FF, PN, RT, DUAL, true>(a, q, lane, mt0, NT, pn, ring);
            } else if constexpr (PM == 2) {
                if (!h) tc_row<PREC, 2, FF, PN, RT, DUAL, false>(a, q, lane, mt0, NT, pn, ring);
                else if constexpr (H == kAny) tc_row<PREC, 2, FF, PN, RT, DUAL, true>(a, q, lane, mt0, NT, pn, ring);
            }
        }
    }
}

// Tiny output blocks (at most 16 elements, 5 x 5 on request) on the split
// paths: the same narrow pieces multiplied with FP32 FMA on CUDA cores (a
// product of two TF32 or BF16 pieces is exact in FP32), FP32 sum inside a block
// product, the same compensated (or FP64) sum across products.  A 16 x 8 MMA
// tile would be almost all padding for such blocks.  One lane owns one element:
// a lane per block leaves a few blocks with long product lists to a few warps
// (2,700 blocks of ragged sizes 1..40: 7.0 ms).
template <int PREC, bool FF>
__device__ __forceinline__ void cs_element(const NumericArgs &a, int64_t q, int e) {
    constexpr int NP = PrecTraits<PREC>::NP;
    const int32_t orc = a.out_blk_rc[q];
    const int R = rc_rows(orc), S = rc_cols(orc), r = e / S, c = e - r * S;
    const int64_t p1 = a.seg_ptr[q + 1];
    const int64_t old = (a.beta != 0.0 && a.old_off) ? a.old_off[q] : -1;
    const int F = a.flush_every > 0 ? a.flush_every : (a.flush_every < 0 ? -a.flush_every : 1);
    float acc = 0.f, shi = 0.f, slo = 0.f;
    double s64 = 0.0;
    int since = 0;
    for (int64_t p = a.seg_ptr[q]; p < p1; ++p) {
        const int32_t ix = a.px[p], iy = a.py[p];
        const int32_t xrc = a.x_blk_rc[ix];
        const int Tn = a.x_trans ? rc_rows(xrc) : rc_cols(xrc);
        const int xs_t = a.x_trans ? R : 1, ys_t = a.y_trans ? 1 : S;
        const float *xe = a.x_plain + (a.x_blk_off[ix] + r * (a.x_trans ? 1 : Tn)) * NP;
        const float *ye = a.y_plain + (a.y_blk_off[iy] + c * (a.y_trans ? Tn : 1)) * NP;
#pragma unroll 4
        for (int t = 0; t < Tn; ++t) {
            if constexpr (NP == 2) {
                const float2 xv = __ldg(reinterpret_cast<const float2 *>(xe + (int64_t)t * xs_t * NP));
                const float2 yv = __ldg(reinterpret_cast<const float2 *>(ye + (int64_t)t * ys_t * NP));
                acc = fmaf(xv.y, yv.x, acc);
                acc = fmaf(xv.x, yv.y, acc);
                acc = fmaf(xv.x, yv.x, acc);
            } else {
                const float *xt = xe + (int64_t)t * xs_t * NP, *yt = ye + (int64_t)t * ys_t * NP;
                const float x0 = __ldg(xt), x1 = __ldg(xt + 1), x2 = __ldg(xt + 2);
                const float y0 = __ldg(yt), y1 = __ldg(yt + 1), y2 = __ldg(yt + 2);
                acc = fmaf(x2, y0, acc);
                acc = fmaf(x1, y1, acc);
                acc = fmaf(x0, y2, acc);
                acc = fmaf(x1, y0, acc);
                acc = fmaf(x0, y1, acc);
                acc = fmaf(x0, y0, acc);
            }
        }
        if (++since == F) {
            since = 0;
            if constexpr (FF) kahan_acc(shi, slo, acc);
            else s64 += widen(acc);
            acc = 0.f;
        }
    }
    const double sum = FF ? pair_total(shi, slo, acc) : s64 + widen(acc);
    double val = a.alpha == 1.0 ? sum : a.alpha * sum;
    const int64_t out = a.out_blk_off[q] + e;
    if (a.dtype == BSM_FP64) {
        if (old >= 0) val = fma(a.beta, static_cast<const double *>(a.old_data)[old + e], val);
        static_cast<double *>(a.out_data)[out] = val;
    } else {
        if (old >= 0) val = fma(a.beta, (double)static_cast<const float *>(a.old_data)[old + e], val);
        static_cast<float *>(a.out_data)[out] = (float)val;
    }
}

// PM x PN: the largest pass this instance runs.  Items [i0, i1) of the
// order, a warp each on the tensor cores: every item before the lane items
// (a.group < 0), or the blocks of one height class (a.group, split_group).
template <int PREC, bool FF, int PM, int PN, bool DUAL, TcHeights H>
__global__ void __launch_bounds__(kThreadsNum) k_numeric_tc(NumericArgs a) {
    extern __shared__ __align__(16) uint32_t tc_smem[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t *ring = tc_smem + warp * ring_words_per_warp<PREC, PM, PN, H == kHalf>();
    if (a.status && *a.status != 0) return;
    int64_t i0 = 0, i1 = a.n_items - (a.n_lane_items ? *a.n_lane_items : 0);
    if (a.group > 0) i0 = a.item_groups[a.group - 1];
    if (a.group >= 0 && a.group < kSplitGroups - 1) i1 = a.item_groups[a.group];
    unsigned long long *ctr = a.work_counter + max(a.group, 0);
    while (true) {
        int64_t t = 0;
        if (lane == 0) t = (int64_t)atomicAdd(ctr, 1ull);
        t = __shfl_sync(0xffffffffu, t, 0) + i0;
        if (t >= i1) break;
        int64_t q = t;
        if (a.item_order) q = (int64_t)((uint32_t)a.item_order[q] & 0x7fffffffu);
        BSM_DBG_WARP_SKIP(a, q, lane)
        tc_item<PREC, FF, PM, PN, DUAL, H>(a, q, lane, ring);
    }
}

// The last *n_lane_items items of the order: tiny blocks marked for the
// CUDA-core variant, kTinyItems per ticket (a kernel of their own, so that the
// tensor-core instances do not carry its registers).
constexpr int kTinyItems = 8;
template <int PREC, bool FF>
__global__ void __launch_bounds__(kThreadsNum) k_numeric_tc_lane(NumericArgs a) {
    const int lane = threadIdx.x & 31;
    if (a.status && *a.status != 0) return;
    const int64_t n_lane = *a.n_lane_items;
    const int64_t lane0 = a.n_items - n_lane;
    unsigned long long *ctr = a.work_counter + kSplitGroups;
    while (true) {
        int64_t t = 0;
        if (lane == 0) t = (int64_t)atomicAdd(ctr, 1ull);
        t = __shfl_sync(0xffffffffu, t, 0) * kTinyItems;
        if (t >= n_lane) break;
        int32_t q = -1;
        int size = 0;
        if (lane < kTinyItems && t + lane < n_lane) {
            q = (int32_t)((uint32_t)a.item_order[lane0 + t + lane] & 0x7fffffffu);
            const int32_t rc = a.out_blk_rc[q];
            size = rc_rows(rc) * rc_cols(rc);
        }
        // lanes per block, by the ticket's largest
        const int most = __reduce_max_sync(0xffffffffu, size), g = most <= 4 ? 4 : most <= 16 ? 16 : 32;
        for (int i = lane / g; i - lane / g < kTinyItems; i += 32 / g) {
            const int32_t qi = __shfl_sync(0xffffffffu, q, i);
            const int e = lane % g;
            if (e < __shfl_sync(0xffffffffu, size, i) && BSM_DBG_LANE_OK(a, qi)) cs_element<PREC, FF>(a, qi, e);
        }
    }
}

template <typename K>
int persistent_grid(K kernel, int64_t n_items, size_t smem = 0, int threads = kThreadsNum, int ctas_per_sm = 0) {
    int per_sm = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, threads, smem);
    if (per_sm < 1) per_sm = 1;
    if (ctas_per_sm > 0 && ctas_per_sm < per_sm) per_sm = ctas_per_sm;
    int64_t g = (int64_t)num_sms() * per_sm;
    const int warps = threads / 32;
    const int64_t need = (n_items + warps - 1) / warps;
    if (g > need) g = need;
    if (g < 1) g = 1;
    return (int)g;
}

template <int PREC, bool FF, int PM, int PN, bool DUAL, TcHeights H>
cudaError_t launch_tc_inst(const NumericArgs &a, cudaStream_t s, int threads, int *grid) {
    const size_t smem = sizeof(uint32_t) * (size_t)ring_words_per_warp<PREC, PM, PN, H == kHalf>() * (threads / 32);
    cudaError_t e = cudaFuncSetAttribute(k_numeric_tc<PREC, FF, PM, PN, DUAL, H>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    *grid = persistent_grid(k_numeric_tc<PREC, FF, PM, PN, DUAL, H>, a.n_items, smem, threads, a.ctas_per_sm);
    k_numeric_tc<PREC, FF, PM, PN, DUAL, H><<<*grid, threads, smem, s>>>(a);
    count_launch(1);
    return cudaGetLastError();
}

// 1-row instances with two accumulators where F > 1 block products share the
// tensor core's sum
template <int PREC, bool FF, int PM, int PN, TcHeights H>
cudaError_t launch_tc_pass(const NumericArgs &a, cudaStream_t s, int threads, int *grid) {
    const int F = a.flush_every > 0 ? a.flush_every : (a.flush_every < 0 ? -a.flush_every : 1);
    if constexpr (PM == 1) {
        if (F > 1) return launch_tc_inst<PREC, FF, PM, PN, true, H>(a, s, threads, grid);
    }
    return launch_tc_inst<PREC, FF, PM, PN, false, H>(a, s, threads, grid);
}

template <int PREC, bool FF, int PM, TcHeights H>
cudaError_t launch_tc_pm(const NumericArgs &a, cudaStream_t s, int threads, int *grid, int pn) {
    if (pn >= 3) return launch_tc_pass<PREC, FF, PM, 3, H>(a, s, threads, grid);
    if (pn == 2) return launch_tc_pass<PREC, FF, PM, 2, H>(a, s, threads, grid);
    return launch_tc_pass<PREC, FF, PM, 1, H>(a, s, threads, grid);
}

// With item groups, the default, an instance for every height class that the
// output has: fewer registers, a smaller ring and less code each, so more warps
// per SM.  Otherwise one instance by the largest pass asked for (pass_mt 1 or 2,
// pass_nt 1..3, default 2 x 3).  Then the lane items.
template <int PREC, bool FF>
cudaError_t launch_tc_ff(const NumericArgs &a, cudaStream_t s, int threads, int *grid) {
    const int pn = a.pass_nt > 0 ? a.pass_nt : 3;
    cudaError_t e = cudaSuccess;
    NumericArgs b = a;
    if (a.item_groups) {
        *grid = 0;  // reported: the first launch's
        for (b.group = 0; b.group < kSplitGroups && e == cudaSuccess; ++b.group) {
            if (!(a.group_mask >> b.group & 1)) continue;
            int g = 0;
            e = b.group == 0   ? launch_tc_pm<PREC, FF, 2, kWhole>(b, s, threads, &g, pn)
                : b.group == 1 ? launch_tc_pass<PREC, FF, 2, 3, kHalf>(b, s, threads, &g)
                : b.group == 2 ? launch_tc_pm<PREC, FF, 1, kWhole>(b, s, threads, &g, pn)
                               : launch_tc_pass<PREC, FF, 1, 3, kHalf>(b, s, threads, &g);
            if (*grid == 0) *grid = g;
        }
    } else {
        b.group = -1;
        e = a.pass_mt == 1 ? launch_tc_pm<PREC, FF, 1, kAny>(b, s, threads, grid, pn)
                           : launch_tc_pm<PREC, FF, 2, kAny>(b, s, threads, grid, pn);
    }
    if (e == cudaSuccess && a.n_lane_items) {
        const int g = persistent_grid(k_numeric_tc_lane<PREC, FF>, a.n_items / kTinyItems + 1, 0, kThreadsNum, a.ctas_per_sm);
        k_numeric_tc_lane<PREC, FF><<<g, kThreadsNum, 0, s>>>(a);
        count_launch(1);
        e = cudaGetLastError();
    }
    return e;
}

template <int PREC>
cudaError_t launch_tc(const NumericArgs &a, cudaStream_t s, int threads, int *grid) {
    return a.flush_every > 0 ? launch_tc_ff<PREC, false>(a, s, threads, grid)
                             : launch_tc_ff<PREC, true>(a, s, threads, grid);
}

}  // namespace

}  // namespace bsm
