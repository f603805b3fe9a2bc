// Numeric phase: every output block accumulates its list of small dense
// block products (the "batches" of DBCSR, Bethune et al. 2017 §2) in a fixed
// order, owned by exactly one warp -- the GPU analogue of the paper's static
// assignment of an A row-block to one thread, so no atomics touch C.
//
// One generic contraction serves the forward product and both adjoints:
//   out_q = alpha * sum_{p in seg(q)} X_p . Y_p  (+ beta * old_q)
// with X_p a logical R x T block and Y_p a logical T x S block, either stored
// as is or transposed:
//   forward  C_ij  = sum_k A_ik . B_kj          X = A,      Y = B
//   adjoint  dA_ik = sum_j dC_ij . B_kj^T       X = dC,     Y = B^T
//   adjoint  dB_kj = sum_i A_ik^T . dC_ij       X = A^T,    Y = dC
//
// Two arithmetic paths:
//   * CUDA cores: FP64 FMA; one lane owns a fixed set of output elements (the
//     plain FP64 path is in k_group.cu, FP32 data in k_tile.cu, few blocks
//     of either in k_warp.cu).
//   * Tensor cores (mma.sync m16n8k8 TF32 / m16n8k16 BF16): operands were
//     split beforehand into 2 or 3 narrow pieces (hi, lo[, lo2]) and packed
//     in mma fragment order; the cross products of the pieces accumulate in
//     FP32 inside the tensor core and are added into an FP64 accumulator
//     every `flush_every` block products.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <atomic>

#include "bsm_internal.cuh"
#include "numeric_debug.cuh"
#include "numeric_split.cuh"
#include "numeric_warp.cuh"

namespace bsm {

namespace {

// =====================================================================
// FP64 FMA on the CUDA cores, a warp or a lane per output block: the small
// blocks of the FP64 tensor-core and Ozaki paths (BSM_P_FP64 has k_group.cu and,
// for few blocks, k_warp.cu, FP32 data k_tile.cu)
// =====================================================================
__device__ __forceinline__ void cc_dispatch(const NumericArgs &a, int64_t q, int lane) {
    warp_block<double, false>(a, q, lane);
}

// Tiny output blocks (at most 16 elements): one lane owns a whole block, so a
// warp advances 32 blocks at once instead of leaving most lanes idle.
__device__ __forceinline__ void cc_lane_item(const NumericArgs &a, int64_t q) {
    constexpr int L = 16;
    const double *__restrict__ X = static_cast<const double *>(a.x_data);
    const double *__restrict__ Y = static_cast<const double *>(a.y_data);
    double *__restrict__ O = static_cast<double *>(a.out_data);
    const int32_t orc = a.out_blk_rc[q];
    const int R = rc_rows(orc), S = rc_cols(orc);
    const int RS = R * S;
    const int64_t out_off = a.out_blk_off[q];
    const int64_t p0 = a.seg_ptr[q], p1 = a.seg_ptr[q + 1];
    const int64_t old = (a.beta != 0.0 && a.old_off) ? a.old_off[q] : -1;
    double acc[L];
#pragma unroll
    for (int e = 0; e < L; ++e) {
        acc[e] = 0.0;
    }
    for (int64_t p = p0; p < p1; ++p) {
        const int32_t ix = a.px[p], iy = a.py[p];
        const double *xb = X + a.x_blk_off[ix];
        const double *yb = Y + a.y_blk_off[iy];
        const int32_t xrc = a.x_blk_rc[ix];
        const int Tn = a.x_trans ? rc_rows(xrc) : rc_cols(xrc);
        const int xs_r = a.x_trans ? 1 : Tn, xs_t = a.x_trans ? R : 1;
        const int ys_t = a.y_trans ? 1 : S, ys_s = a.y_trans ? Tn : 1;
        for (int t = 0; t < Tn; ++t) {
#pragma unroll
            for (int e = 0; e < L; ++e) {
                if (e < RS) {
                    const int r = e / S, c = e - r * S;
                    acc[e] = fma(__ldg(xb + r * xs_r + t * xs_t), __ldg(yb + t * ys_t + c * ys_s), acc[e]);
                }
            }
        }
    }
    const double *OLD = static_cast<const double *>(a.old_data);
#pragma unroll
    for (int e = 0; e < L; ++e) {
        if (e < RS) {
            double v = acc[e];
            v = a.alpha * v;
            if (old >= 0) v = fma(a.beta, OLD[old + e], v);
            O[out_off + e] = v;
        }
    }
}

// Fixed shapes of the lane-per-block mode: column t of the X block and row t
// of the Y block are loaded once per k and applied as a rank-1 update.
template <int R, int S>
__device__ __forceinline__ void cc_lane_fixed(const NumericArgs &a, int64_t q) {
    const double *__restrict__ X = static_cast<const double *>(a.x_data);
    const double *__restrict__ Y = static_cast<const double *>(a.y_data);
    double *__restrict__ O = static_cast<double *>(a.out_data);
    const int64_t out_off = a.out_blk_off[q];
    const int64_t p0 = a.seg_ptr[q], p1 = a.seg_ptr[q + 1];
    const int64_t old = (a.beta != 0.0 && a.old_off) ? a.old_off[q] : -1;
    double acc[R][S];
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
        for (int c = 0; c < S; ++c) {
            acc[r][c] = 0.0;
        }
    for (int64_t p = p0; p < p1; ++p) {
        const int32_t ix = a.px[p], iy = a.py[p];
        const double *xb = X + a.x_blk_off[ix];
        const double *yb = Y + a.y_blk_off[iy];
        const int32_t xrc = a.x_blk_rc[ix];
        const int Tn = a.x_trans ? rc_rows(xrc) : rc_cols(xrc);
        const int xs_r = a.x_trans ? 1 : Tn, xs_t = a.x_trans ? R : 1;
        const int ys_t = a.y_trans ? 1 : S, ys_s = a.y_trans ? Tn : 1;
        for (int t = 0; t < Tn; ++t) {
            double xv[R], yv[S];
#pragma unroll
            for (int r = 0; r < R; ++r) xv[r] = __ldg(xb + r * xs_r + t * xs_t);
#pragma unroll
            for (int c = 0; c < S; ++c) yv[c] = __ldg(yb + t * ys_t + c * ys_s);
#pragma unroll
            for (int r = 0; r < R; ++r)
#pragma unroll
                for (int c = 0; c < S; ++c) acc[r][c] = fma(xv[r], yv[c], acc[r][c]);
        }
    }
    const double *OLD = static_cast<const double *>(a.old_data);
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
        for (int c = 0; c < S; ++c) {
            const int e = r * S + c;
            double v = acc[r][c];
            v = a.alpha * v;
            if (old >= 0) v = fma(a.beta, OLD[old + e], v);
            O[out_off + e] = v;
        }
}

__device__ __forceinline__ void cc_lane_dispatch(const NumericArgs &a, int64_t q) {
    const int32_t orc = a.out_blk_rc[q];
    switch ((rc_rows(orc) << 8) | rc_cols(orc)) {
        case 0x101: cc_lane_fixed<1, 1>(a, q); break;
        case 0x102: cc_lane_fixed<1, 2>(a, q); break;
        case 0x201: cc_lane_fixed<2, 1>(a, q); break;
        case 0x202: cc_lane_fixed<2, 2>(a, q); break;
        case 0x104: cc_lane_fixed<1, 4>(a, q); break;
        case 0x401: cc_lane_fixed<4, 1>(a, q); break;
        case 0x204: cc_lane_fixed<2, 4>(a, q); break;
        case 0x402: cc_lane_fixed<4, 2>(a, q); break;
        case 0x404: cc_lane_fixed<4, 4>(a, q); break;
        case 0x505: cc_lane_fixed<5, 5>(a, q); break;
        case 0x606: cc_lane_fixed<6, 6>(a, q); break;
        default: cc_lane_item(a, q); break;
    }
}

// =====================================================================
// FP64 tensor-core path (BSM_P_FP64_DMMA): mma.sync m8n8k4 with FP64
// operands and accumulators.  Fragment layout of m8n8k4 (lane = 4 g + t4):
// A (8 x 4, row) holds X(g, t4); B (4 x 8, col) holds Y(t4, g); the
// accumulator holds D(g, 2 t4) and D(g, 2 t4 + 1).  One warp per output
// block; blocks of at least 8 x 8 elements run here, in passes of up to
// 3 x 3 tiles of 8 x 8 (24 x 24 elements), every block product in ascending
// k steps of 4 with zero padding past the block edges.  Smaller output
// blocks run the FP64 FMA code.
// =====================================================================
__device__ __forceinline__ void dmma(double (&d)[2], double a, double b) {
    asm volatile("mma.sync.aligned.m8n8k4.row.col.f64.f64.f64.f64 {%0,%1}, {%2}, {%3}, {%0,%1};"
                 : "+d"(d[0]), "+d"(d[1])
                 : "d"(a), "d"(b));
}

template <int MTC, int NTC>
__device__ __forceinline__ void dmma_pass(const NumericArgs &a, int64_t q, int lane, int mt0, int nt0) {
    const double *__restrict__ X = static_cast<const double *>(a.x_data);
    const double *__restrict__ Y = static_cast<const double *>(a.y_data);
    const int32_t orc = a.out_blk_rc[q];
    const int R = rc_rows(orc), S = rc_cols(orc);
    const int64_t p0 = a.seg_ptr[q], p1 = a.seg_ptr[q + 1];
    const int g = lane >> 2, t4 = lane & 3;
    double acc[MTC][NTC][2];
#pragma unroll
    for (int i = 0; i < MTC; ++i)
#pragma unroll
        for (int j = 0; j < NTC; ++j) acc[i][j][0] = acc[i][j][1] = 0.0;
    // rows of X and columns of Y this lane loads (clamped reads are masked)
    int xr[MTC], ys[NTC];
    bool xv[MTC], yv[NTC];
#pragma unroll
    for (int i = 0; i < MTC; ++i) {
        xr[i] = (mt0 + i) * 8 + g;
        xv[i] = xr[i] < R;
    }
#pragma unroll
    for (int j = 0; j < NTC; ++j) {
        ys[j] = (nt0 + j) * 8 + g;
        yv[j] = ys[j] < S;
    }
    for (int64_t p = p0; p < p1; ++p) {
        const int32_t ix = a.px[p], iy = a.py[p];
        const double *xb = X + a.x_blk_off[ix];
        const double *yb = Y + a.y_blk_off[iy];
        const int32_t xrc = a.x_blk_rc[ix];
        const int Tn = a.x_trans ? rc_rows(xrc) : rc_cols(xrc);
        const int xs_r = a.x_trans ? 1 : Tn, xs_t = a.x_trans ? R : 1;
        const int ys_t = a.y_trans ? 1 : S, ys_s = a.y_trans ? Tn : 1;
        for (int t0 = 0; t0 < Tn; t0 += 4) {
            const int t = t0 + t4;
            const bool tv = t < Tn;
            double fa[MTC], fb[NTC];
#pragma unroll
            for (int i = 0; i < MTC; ++i) fa[i] = (tv && xv[i]) ? __ldg(xb + xr[i] * xs_r + t * xs_t) : 0.0;
#pragma unroll
            for (int j = 0; j < NTC; ++j) fb[j] = (tv && yv[j]) ? __ldg(yb + t * ys_t + ys[j] * ys_s) : 0.0;
#pragma unroll
            for (int i = 0; i < MTC; ++i)
#pragma unroll
                for (int j = 0; j < NTC; ++j) dmma(acc[i][j], fa[i], fb[j]);
        }
    }
    double *O = static_cast<double *>(a.out_data);
    const double *OLD = static_cast<const double *>(a.old_data);
    const int64_t out_off = a.out_blk_off[q];
    const int64_t old = (a.beta != 0.0 && a.old_off) ? a.old_off[q] : -1;
#pragma unroll
    for (int i = 0; i < MTC; ++i)
#pragma unroll
        for (int j = 0; j < NTC; ++j)
#pragma unroll
            for (int v = 0; v < 2; ++v) {
                const int r = (mt0 + i) * 8 + g, c = (nt0 + j) * 8 + 2 * t4 + v;
                if (r < R && c < S) {
                    const int64_t e = (int64_t)r * S + c;
                    double val = a.alpha * acc[i][j][v];
                    if (old >= 0) val = fma(a.beta, OLD[old + e], val);
                    O[out_off + e] = val;
                }
            }
}

__device__ __forceinline__ void dmma_item(const NumericArgs &a, int64_t q, int lane) {
    const int32_t orc = a.out_blk_rc[q];
    const int MT = (rc_rows(orc) + 7) >> 3, NT = (rc_cols(orc) + 7) >> 3;
    const int pm = a.pass_mt > 0 ? a.pass_mt : 3, pn = a.pass_nt > 0 ? a.pass_nt : 3;
    for (int mt0 = 0; mt0 < MT; mt0 += pm) {
        const int mtc = min(pm, MT - mt0);
        for (int nt0 = 0; nt0 < NT; nt0 += pn) {
            const int ntc = min(pn, NT - nt0);
            switch (mtc * 4 + ntc) {
                case 5: dmma_pass<1, 1>(a, q, lane, mt0, nt0); break;
                case 6: dmma_pass<1, 2>(a, q, lane, mt0, nt0); break;
                case 7: dmma_pass<1, 3>(a, q, lane, mt0, nt0); break;
                case 9: dmma_pass<2, 1>(a, q, lane, mt0, nt0); break;
                case 10: dmma_pass<2, 2>(a, q, lane, mt0, nt0); break;
                case 11: dmma_pass<2, 3>(a, q, lane, mt0, nt0); break;
                case 13: dmma_pass<3, 1>(a, q, lane, mt0, nt0); break;
                case 14: dmma_pass<3, 2>(a, q, lane, mt0, nt0); break;
                default: dmma_pass<3, 3>(a, q, lane, mt0, nt0); break;
            }
        }
    }
}

__global__ void __launch_bounds__(kThreadsNum) k_numeric_dmma(NumericArgs a) {
    const int lane = threadIdx.x & 31;
    if (a.status && *a.status != 0) return;
    unsigned long long *ctr = a.work_counter;
    const int64_t n_lane = a.n_lane_items ? *a.n_lane_items : 0;
    const int64_t n0 = a.n_items - n_lane;
    const int64_t tickets = n0 + (n_lane + 31) / 32;
    while (true) {
        int64_t t = 0;
        if (lane == 0) t = (int64_t)atomicAdd(ctr, 1ull);
        t = __shfl_sync(0xffffffffu, t, 0);
        if (t >= tickets) break;
        if (t < n0) {
            int64_t q = t;
            if (a.item_order) q = (int64_t)((uint32_t)a.item_order[q] & 0x7fffffffu);
            BSM_DBG_WARP_SKIP(a, q, lane)
            const int32_t orc = a.out_blk_rc[q];
            if (rc_rows(orc) >= 8 && rc_cols(orc) >= 8) dmma_item(a, q, lane);
            else cc_dispatch(a, q, lane);
        } else {
            const int64_t idx = n0 + (t - n0) * 32 + lane;
            if (idx < a.n_items) {
                const int64_t q = (int64_t)((uint32_t)a.item_order[idx] & 0x7fffffffu);
                if (BSM_DBG_LANE_OK(a, q)) cc_lane_dispatch(a, q);
            }
        }
    }
}

// =====================================================================
// Ozaki-style error-free slicing (BSM_P_OZAKI)
// =====================================================================
// Error-free transformation of a product into products of short-mantissa
// operands (Ozaki, Ogita, Oishi and Rump, 2012).  With 2^e the largest power
// of two not above max |x| over a line (a logical row of X, a logical column
// of Y), every x of the line is cut into integer digits
//   x * 2^(7-e) = d_0 + d_1 2^-9 + ... + d_5 2^-45 + rest,   |rest| <= 2^-46,
// d_0 = rint(x * 2^(7-e)) and each next digit the rounded remainder times 2^9,
// so |d_p| <= 256 and the slice d_p * 2^(-9p) is exact in BF16.  A slice
// product of level l = p + q lies on the grid 2^(-9l) (in units of the line
// pair's scale 2^(ex+ey-14)); products of one level summed in the tensor
// core's FP32 accumulator stay exact while the sum stays below 2^24 grid
// units: a level holding c slice pairs takes 2^24 / (c * 2^16) terms of k,
// 64 for level 3 (4 pairs).  Levels 0..3 have exact FP32 sums; before more
// than kOzWindow terms of k they are converted to integers and added into a
// 64-bit fixed-point sum with unit 2^-27 (exact; a window adds less than
// 2^49.01 units, so 8192 windows fit, after which the sum is moved into the
// output element).  Levels 4 and 5 (11 pairs, below 2^-33 of level 0) have
// a rounded FP32 sum each per window (the tensor core's FP32 additions round
// toward zero, so they are restarted every window; two sums rather than one
// keep every accumulator's chain of dependent MMAs at 6 per k-step or less),
// whose window values add up in an FP32 sum with round-to-nearest on the
// CUDA cores; levels >= 6 are dropped (below 2^-50 of level 0).  Per term of k the error is below 2^-44
// of 2^(ex+ey): the rounded sums plus the cut digits and levels.
constexpr int kOzSlices = 6;
constexpr int kOzLevels = 6;    // FP32 sums: levels 0, 1, 2, 3 exact, 4 and 5 rounded (one each,
                                // so that no accumulator takes more than 6 of a k-step's 21 MMAs)
constexpr int kOzWindow = 64;
constexpr int kOzSpillWindows = 8192;
constexpr int kOzStages = 3;
constexpr int kOzXW = 4 * kOzSlices;                 // X words per lane per tile
constexpr int kOzYW = 2 * kOzSlices;                 // Y words per lane per tile
constexpr int kOzHW = 2 * kOzSlices;                 // X words of a tile that is half a tile one way
constexpr int kOzQW = 8;                             // X words of a quarter tile, Y words of a half one
// words of one k-step of an X block of R rows and of a Y block of S columns; HK:
// the last step where at most 8 terms of k are left
template <bool HK> __host__ __device__ constexpr int oz_xstep(int R) {
    return 32 * ((HK ? kOzHW : kOzXW) * ((R - 1) / 16) +
                 (half_rows(R) ? (HK ? kOzQW : kOzHW) : (HK ? kOzHW : kOzXW)));
}
__host__ __device__ constexpr int oz_xstep_whole(int R) { return 32 * kOzXW * ((R + 15) / 16); }
template <bool HK> __host__ __device__ constexpr int oz_ystep(int S) { return 32 * (HK ? kOzQW : kOzYW) * ((S + 7) / 8); }
// ring words per lane per stage for passes of at most MAXN tiles (1 x MAXN)
template <int MAXN>
__host__ __device__ constexpr int oz_sw() { return kOzXW + MAXN * kOzYW; }
template <int MAXN>
__host__ __device__ constexpr int oz_ring_words_per_warp() { return kOzStages * 32 * oz_sw<MAXN>(); }
// Packed tiles are chunk-major: chunk c (16 bytes) of lane L at word
// c * 128 + 4 * L, so one 16-byte cp.async per lane reads 512 contiguous
// bytes.  X tile: chunk p = plane p (registers v0..v3); Y tile: chunk c =
// planes 2c and 2c+1 (registers v0, v1 each; lanes with bit 3 set hold the two
// 8-byte halves swapped, so 8-byte reads of 16 lanes hit 16 distinct bank
// pairs).  A ring stage is chunk-major the same way (chunk c of lane L at
// word c * 128 + 4 * L): each 16-byte copy and read of the warp covers 512
// contiguous bytes of shared memory.
// Half tiles: where at most 8 rows of an X block fall into its last tile row (HM:
// registers v1, v3 would be zeros) or at most 8 terms of k into its last step (HK:
// v2, v3, and v1 of Y), another slice takes the empty half, so that one MMA does
// the work of two (of four where both hold):
//   HM  chunk c = {p.v0, p'.v0, p.v2, p'.v2}, p = 2c, p' = p + 1: rows 0..7 of the
//       MMA's result hold level p + q, rows 8..15 level p + q + 1 of the same rows
//   HK  chunk c = {p.v0, p.v1, p'.v0, p'.v1} against Y {q, q-1}: the terms (p, q)
//       and (p', q - 1) of one level
//   both  chunk c = v0 of p = 4c, p + 1, p + 2, p + 3 against Y {q, q-2}: level
//       p + q from p and p + 2 below, level p + q + 1 from p + 1 and p + 3 above
// With HK the Y slices are words, 4c..4c+3 in chunk c.  21 MMAs a tile and k-step
// become 12, 12 and 8.  (The same packs with zeros in the empty half were slower
// than whole tiles: 2,000 banded rows of 23 62.5 ms, 57.3 with m16n8k8, against 55.0.)

// The MMAs of one k-step from its ring stage (w: this lane's words).  acc[l]: level
// l; with HM level l in rows 0..7, level l + 1 in rows 8..15 (of acc[5] not used).
template <int NTC, bool HM, bool HK>
__device__ __forceinline__ void oz_step(float (&acc)[kOzLevels][NTC][4], const uint32_t *w, int hswz) {
    constexpr int XC = HM && HK ? kOzQW / 4 : HM || HK ? kOzHW / 4 : kOzXW / 4, YC = (HK ? kOzQW : kOzYW) / 4;
    constexpr int PC = kOzSlices / XC + (HM && HK ? 1 : 0);  // slices per chunk: 1, 2 or 4
    constexpr int top = kOzLevels - 1;
    uint32_t fa[XC][4];
#pragma unroll
    for (int c = 0; c < XC; ++c) {
        const uint4 v = *reinterpret_cast<const uint4 *>(w + 128 * c);
        fa[c][0] = v.x; fa[c][1] = v.y; fa[c][2] = v.z; fa[c][3] = v.w;
    }
    if constexpr (HK) {
        uint32_t y[NTC][kOzSlices];
#pragma unroll
        for (int j = 0; j < NTC; ++j) {
            const uint4 v = *reinterpret_cast<const uint4 *>(w + 128 * (XC + j * YC));
            const uint2 u = *reinterpret_cast<const uint2 *>(w + 128 * (XC + j * YC + 1));
            y[j][0] = v.x; y[j][1] = v.y; y[j][2] = v.z; y[j][3] = v.w; y[j][4] = u.x; y[j][5] = u.y;
        }
        constexpr int D = HM ? 2 : 1;  // the slice of Y in the upper half of k is q - D
#pragma unroll
        for (int q = kOzSlices - 1; q >= 0; --q) {
            uint32_t fb[NTC][2];
#pragma unroll
            for (int j = 0; j < NTC; ++j) {
                fb[j][0] = y[j][q];
                fb[j][1] = q >= D ? y[j][q >= D ? q - D : 0] : 0u;
            }
#pragma unroll
            for (int c = XC - 1; c >= 0; --c)
                if (PC * c + q <= top)
#pragma unroll
                    for (int j = 0; j < NTC; ++j) mma_bf16(acc[PC * c + q <= top ? PC * c + q : 0][j], fa[c], fb[j]);
        }
    } else {
        // Y slice q (read when needed) with every X slice of level <= 5
#pragma unroll
        for (int q = kOzSlices - 1; q >= 0; --q) {
            uint32_t fb[NTC][2];
#pragma unroll
            for (int j = 0; j < NTC; ++j) {
                const uint2 v = *reinterpret_cast<const uint2 *>(
                    w + 128 * (XC + j * YC + (q >> 1)) + 2 * ((q & 1) ^ hswz));
                fb[j][0] = v.x; fb[j][1] = v.y;
            }
#pragma unroll
            for (int c = XC - 1; c >= 0; --c)
                if (PC * c + q <= top)
#pragma unroll
                    for (int j = 0; j < NTC; ++j) mma_bf16(acc[PC * c + q <= top ? PC * c + q : 0][j], fa[c], fb[j]);
        }
    }
}

// One pass over a 1 x NTC super tile (16 x 8*NTC output elements) at (mt0, nt0),
// staged through a ring laid out for passes of at most MAXN tiles.  HM: half a tile
// of rows; HKS: some product has an HK step (the multiply's inner sizes tell); WT:
// packs of whole tiles and k-steps.
//
// Bound by the latency of a warp's steps at eight warps an SM: 2,000 banded rows of
// 23, the kernels of the half and of the whole tile rows, tensor pipe 42% and 48%
// busy, issue 35% and 32%.  Two CTAs of four warps fit, in the whole-row kernel by
// its 200 registers, in the half-row one by its staging ring of 90 KB (with 166
// registers three would; half a tile row needs 12 of the ring's 24 X words a lane).
// Then the L2 reads, 15 chunks of 512 bytes to the 63 MMAs of a whole step.
// Blocks of 23 end in half a tile both ways: four whole steps a product,
// 252 MMAs and 60 chunks, became 159 and 40.5.  Numeric pass of 2,000 banded rows
// of 23 (1.96e7 products) 55.0 -> 47.5 ms, of blocks of 5 (8e7) 26.0 -> 19.8, of 13
// (6.9e6) 7.34 -> 7.16, of 32 (4.6e5) 4.44 -> 4.13, the last two from the running
// pointers and untested tiles alone.
template <int NTC, int MAXN, bool HM, bool HKS, bool WT>
__device__ __forceinline__ void oz_pass(const NumericArgs &a, int64_t q, int lane, int mt0, int nt0,
                                        uint32_t *ring) {
    constexpr int ST = kOzStages, SW = oz_sw<MAXN>();
    const int32_t orc = a.out_blk_rc[q];
    const int R = rc_rows(orc), S = rc_cols(orc);
    const int64_t p0 = a.seg_ptr[q], p1 = a.seg_ptr[q + 1];
    const uint32_t *XP = static_cast<const uint32_t *>(a.x_pack) + 4 * lane;
    const uint32_t *YP = static_cast<const uint32_t *>(a.y_pack) + 4 * lane;
    const int xk = WT ? oz_xstep_whole(R) : oz_xstep<false>(R), yk = oz_ystep<false>(S);
    constexpr int NV = HM ? 2 : 4;  // accumulator elements of a lane that count
    double *O = static_cast<double *>(a.out_data);
    const int64_t out_off = a.out_blk_off[q];
    uint32_t *myring = ring + 4 * lane;  // chunk c of stage st at myring + st * 32 * SW + 128 * c
    const uint32_t ring_s = smem_addr(myring);
    const int hswz = (lane >> 3) & 1;  // 8-byte half order inside a Y chunk
    const int g = lane >> 2, t4 = lane & 3;
    float acc[kOzLevels][NTC][4];
    long long fx[NTC][4];  // exact sum of levels 0..3, unit 2^-27
    float low[NTC][4];     // sum of the windows' level 4..5 sums
#pragma unroll
    for (int j = 0; j < NTC; ++j)
#pragma unroll
        for (int v = 0; v < 4; ++v) {
            fx[j][v] = 0;
            low[j][v] = 0.f;
#pragma unroll
            for (int l = 0; l < kOzLevels; ++l) acc[l][j][v] = 0.f;
        }
    int kacc = 0;      // terms of k in the open exact window
    int nwin = 0;      // windows added into fx since it was last moved out
    bool spilled = false;
    // levels 0..3 -> fx (integers below 2^24 on their grids, so the conversions are exact)
    auto close_window = [&]() {
#pragma unroll
        for (int j = 0; j < NTC; ++j)
#pragma unroll
            for (int v = 0; v < NV; ++v) {
                // element v of level l: with HM in two sums, below and (v + 2) above
                auto level = [&](int l, float scale) -> long long {
                    long long t = __float2int_rn(acc[l][j][v] * scale);
                    if (HM && l > 0) t += __float2int_rn(acc[HM && l > 0 ? l - 1 : 0][j][(v + 2) & 3] * scale);
                    return t;
                };
                fx[j][v] += (level(0, 1.f) << 27) + (level(1, 512.f) << 18) + (level(2, 262144.f) << 9) + level(3, 134217728.f);
                float l4 = acc[4][j][v], l5 = acc[5][j][v];
                if constexpr (HM) {
                    l4 = __fadd_rn(l4, acc[3][j][(v + 2) & 3]);
                    l5 = __fadd_rn(l5, acc[4][j][(v + 2) & 3]);
                }
                low[j][v] = __fadd_rn(low[j][v], __fadd_rn(l4, l5));
            }
#pragma unroll
        for (int j = 0; j < NTC; ++j)
#pragma unroll
            for (int v = 0; v < 4; ++v) {
#pragma unroll
                for (int l = 0; l < kOzLevels; ++l) acc[l][j][v] = 0.f;
            }
        if (++nwin == kOzSpillWindows) {  // keep fx far from 2^63: move it into the output
            nwin = 0;
#pragma unroll
            for (int j = 0; j < NTC; ++j)
#pragma unroll
                for (int v = 0; v < NV; ++v) {
                    const int r = mt0 * 16 + g + ((v >> 1) << 3);
                    const int c = (nt0 + j) * 8 + 2 * t4 + (v & 1);
                    if (r < R && c < S) {
                        const double part = (double)fx[j][v] * 0x1p-27;
                        const int64_t e = out_off + (int64_t)r * S + c;
                        O[e] = spilled ? O[e] + part : part;
                    }
                    fx[j][v] = 0;
                }
            spilled = true;
        }
    };
    for (int64_t pb = p0; pb < p1; pb += 32) {
        const int nb = (int)min((int64_t)32, p1 - pb);
        int64_t mxo = 0, myo = 0;
        int mtn = 0;
        if (lane < nb) {
            const int32_t ix = a.px[pb + lane], iy = a.py[pb + lane];
            const int32_t xrc = a.x_blk_rc[ix];
            mtn = a.x_trans ? rc_rows(xrc) : rc_cols(xrc);
            mxo = a.x_pack_off[ix];
            myo = a.y_pack_off[iy];
        }
        int nsteps = (mtn + 15) >> 4;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) nsteps += __shfl_xor_sync(0xffffffffu, nsteps, o);
        // producer cursor: product, terms of k left in it, its next k-step
        int pu = 0, pk = __shfl_sync(0xffffffffu, mtn, 0);
        const uint32_t *xs = XP + __shfl_sync(0xffffffffu, mxo, 0), *ys = YP + __shfl_sync(0xffffffffu, myo, 0);
        auto produce = [&](uint32_t dst) {
            if (HKS && pk <= 8) {
                constexpr int XC = (HM ? kOzQW : kOzHW) / 4, YC = kOzQW / 4;
                const uint32_t *x = xs + mt0 * (32 * kOzHW), *y = ys + nt0 * (32 * kOzQW);
#pragma unroll
                for (int c = 0; c < XC; ++c) cp_async16_cg(dst + 512u * c, x + 128 * c);
#pragma unroll
                for (int c = 0; c < NTC * YC; ++c) cp_async16_cg(dst + 512u * (XC + c), y + 128 * c);
            } else {
                constexpr int XC = (HM ? kOzHW : kOzXW) / 4, YC = kOzYW / 4;
                const uint32_t *x = xs + mt0 * (32 * kOzXW), *y = ys + nt0 * (32 * kOzYW);
#pragma unroll
                for (int c = 0; c < XC; ++c) cp_async16_cg(dst + 512u * c, x + 128 * c);
#pragma unroll
                for (int c = 0; c < NTC * YC; ++c) cp_async16_cg(dst + 512u * (XC + c), y + 128 * c);
                xs += xk;
                ys += yk;
            }
            pk -= 16;
            if (pk <= 0) {
                ++pu;
                const int src_lane = pu < nb ? pu : 0;
                xs = XP + __shfl_sync(0xffffffffu, mxo, src_lane);
                ys = YP + __shfl_sync(0xffffffffu, myo, src_lane);
                pk = __shfl_sync(0xffffffffu, mtn, src_lane);
            }
        };
#pragma unroll
        for (int st = 0; st < ST - 1; ++st) {
            if (st < nsteps) produce(ring_s + (uint32_t)(st * 128 * SW));
            cp_async_commit();
        }
        int cu = 0, ck = __shfl_sync(0xffffffffu, mtn, 0);  // product, terms of k left in it
        uint32_t rd = 0, wr = (ST - 1) * 128 * SW;  // bytes into the ring of the stages read and filled
        for (int s = 0; s < nsteps; ++s) {
            if (s + ST - 1 < nsteps) produce(ring_s + wr);
            cp_async_commit();
            cp_async_wait<ST - 1>();
            const uint32_t *w = myring + rd / 4;
            rd = rd == (ST - 1) * 128 * SW ? 0 : rd + 128 * SW;
            wr = wr == (ST - 1) * 128 * SW ? 0 : wr + 128 * SW;
            // close the exact window before it would pass kOzWindow terms of k
            const int kact = min(16, ck);
            if (kacc + kact > kOzWindow) {
                close_window();
                kacc = 0;
            }
            kacc += kact;
            if (HKS && ck <= 8) oz_step<NTC, HM, true>(acc, w, hswz);
            else oz_step<NTC, HM, false>(acc, w, hswz);
            ck -= 16;
            if (ck <= 0) {
                ++cu;
                ck = __shfl_sync(0xffffffffu, mtn, cu < nb ? cu : 0);
            }
        }
        cp_async_wait<0>();
    }
    close_window();
    // epilogue: scale by 2^(ex + ey - 14) of the element's row and column
    const int64_t old = (a.beta != 0.0 && a.old_off) ? a.old_off[q] : -1;
    const bool any = p1 > p0;
    const int32_t xl0 = any ? a.x_line0[a.px[p0]] : 0;
    const int32_t yl0 = any ? a.y_line0[a.py[p0]] : 0;
    int ex[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int r = mt0 * 16 + g + 8 * h;
        ex[h] = (any && r < R) ? a.x_exp[xl0 + r] - 1023 : 0;
    }
#pragma unroll
    for (int j = 0; j < NTC; ++j) {
        int ey[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int c = (nt0 + j) * 8 + 2 * t4 + h;
            ey[h] = (any && c < S) ? a.y_exp[yl0 + c] - 1023 : 0;
        }
#pragma unroll
        for (int v = 0; v < NV; ++v) {
            const int r = mt0 * 16 + g + ((v >> 1) << 3);
            const int c = (nt0 + j) * 8 + 2 * t4 + (v & 1);
            if (r < R && c < S) {
                const int64_t e = (int64_t)r * S + c;
                double sum = (double)fx[j][v] * 0x1p-27 + (double)low[j][v];
                if (spilled) sum += O[out_off + e];
                double val = a.alpha * ldexp(sum, ex[v >> 1] + ey[v & 1] - 14);
                if (old >= 0) val = fma(a.beta, static_cast<const double *>(a.old_data)[old + e], val);
                O[out_off + e] = val;
            }
        }
    }
}

template <int MAXN, bool HM, bool HKS, bool WT>
__device__ __forceinline__ void oz_row(const NumericArgs &a, int64_t q, int lane, int mt0, int NT, int pn, uint32_t *ring) {
    for (int nt0 = 0; nt0 < NT; nt0 += pn) {
        const int left = min(NT - nt0, pn);
        if (MAXN == 1 || left == 1) oz_pass<1, MAXN, HM, HKS, WT>(a, q, lane, mt0, nt0, ring);
        else if constexpr (MAXN >= 2) {
            if (MAXN == 2 || left == 2) oz_pass<2, MAXN, HM, HKS, WT>(a, q, lane, mt0, nt0, ring);
            else if constexpr (MAXN >= 3) oz_pass<3, MAXN, HM, HKS, WT>(a, q, lane, mt0, nt0, ring);
        }
    }
}

// the half tile row of a block (HM) or its whole ones; all as whole ones (WT)
template <int MAXN, bool HM, bool HKS, bool WT>
__device__ __forceinline__ void oz_item(const NumericArgs &a, int64_t q, int lane, uint32_t *ring) {
    const int32_t orc = a.out_blk_rc[q];
    const int R = rc_rows(orc), NT = (rc_cols(orc) + 7) >> 3;
    const int pn = MAXN == 3 ? 3 : MAXN == 1 ? 1 : (a.pass_nt == 1 ? 1 : 2);
    const int whole = WT ? (R + 15) >> 4 : (R + 7) >> 4;
    if constexpr (HM) {
        if (half_rows(R)) oz_row<MAXN, true, HKS, WT>(a, q, lane, whole, NT, pn, ring);
    } else {
        for (int mt0 = 0; mt0 < whole; ++mt0) oz_row<MAXN, false, HKS, WT>(a, q, lane, mt0, NT, pn, ring);
    }
}

// The half tile rows run in kernels of their own: with both kinds in one, the code
// of a warp's two passes fell out of the instruction cache where blocks have few
// products (497 block rows of 23, 5 products a block: 7.1 ms, 5.2 before).
// Items [0, n0): a warp each on the tensor cores; items [n0, n_items): tiny
// blocks one per lane with plain FP64 FMA (exact enough, no slicing needed).
template <int MAXN, bool HM, bool HKS, bool WT>
__global__ void __launch_bounds__(kThreadsNum) k_numeric_oz(NumericArgs a) {
    extern __shared__ __align__(16) uint32_t oz_smem[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t *ring = oz_smem + warp * oz_ring_words_per_warp<MAXN>();
    if (a.status && *a.status != 0) return;
    // items [i0, i1): every item before the lane items (a.group < 0), or one
    // group: blocks of two tile columns and more (0), of one tile column (1)
    const int64_t n_lane = a.n_lane_items ? *a.n_lane_items : 0;
    int64_t i0 = 0, i1 = a.n_items - n_lane;
    if (a.group == 0) i1 = a.item_groups[0];
    if (a.group == 1) i0 = a.item_groups[0];
    // work_counter[2] is the lane items'
    unsigned long long *ctr = a.work_counter + (HM ? 3 : 0) + (a.group > 0 ? a.group : 0);
    while (true) {
        int64_t t = 0;
        if (lane == 0) t = (int64_t)atomicAdd(ctr, 1ull);
        t = __shfl_sync(0xffffffffu, t, 0) + i0;
        if (t >= i1) break;
        int64_t q = t;
        if (a.item_order) q = (int64_t)((uint32_t)a.item_order[q] & 0x7fffffffu);
        BSM_DBG_WARP_SKIP(a, q, lane)
        oz_item<MAXN, HM, HKS, WT>(a, q, lane, ring);
    }
}

// The lane items of the Ozaki path: plain FP64 FMA, one lane per block.
__global__ void __launch_bounds__(kThreadsNum) k_numeric_oz_lane(NumericArgs a) {
    const int lane = threadIdx.x & 31;
    if (a.status && *a.status != 0) return;
    const int64_t n_lane = *a.n_lane_items;
    const int64_t lane0 = a.n_items - n_lane;
    unsigned long long *ctr = a.work_counter + 2;
    while (true) {
        int64_t t = 0;
        if (lane == 0) t = (int64_t)atomicAdd(ctr, 1ull);
        t = __shfl_sync(0xffffffffu, t, 0);
        if (t * 32 >= n_lane) break;
        const int64_t idx = lane0 + t * 32 + lane;
        if (idx < a.n_items) {
            const int64_t q = (int64_t)((uint32_t)a.item_order[idx] & 0x7fffffffu);
            if (BSM_DBG_LANE_OK(a, q)) cc_lane_dispatch(a, q);
        }
    }
}

// =====================================================================
// Operand splitting and fragment packing
// =====================================================================
__device__ __forceinline__ uint32_t f32_to_tf32(float x) {
    uint32_t r;
    asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(x));
    return r;
}

// Split x into `np` pieces of the precision's narrow type, most significant
// first; returns the bit patterns (TF32 in 32 bits, BF16 in the low 16).
template <int PREC>
__device__ __forceinline__ void split_value(double x, uint32_t (&out)[3]) {
    if constexpr (PREC == BSM_P_TF32x3) {
        const uint32_t hi = f32_to_tf32((float)x);
        const double r = x - (double)__uint_as_float(hi);
        out[0] = hi;
        out[1] = f32_to_tf32((float)r);
        out[2] = 0;
    } else {
        const __nv_bfloat16 h0 = __double2bfloat16(x);
        const double r1 = x - (double)__bfloat162float(h0);
        const __nv_bfloat16 h1 = __double2bfloat16(r1);
        const double r2 = r1 - (double)__bfloat162float(h1);
        const __nv_bfloat16 h2 = __double2bfloat16(r2);
        out[0] = __bfloat16_as_ushort(h0);
        out[1] = __bfloat16_as_ushort(h1);
        out[2] = __bfloat16_as_ushort(h2);
    }
}

template <typename T>
__device__ __forceinline__ double elem(const T *b, int R, int Tn, int trans, int r, int t) {
    // logical R x Tn block, stored R x Tn (trans=0) or Tn x R (trans=1)
    if (r >= R || t >= Tn) return 0.0;
    return (double)(trans ? b[(int64_t)t * R + r] : b[(int64_t)r * Tn + t]);
}

// words of one block's packing
__device__ __forceinline__ int64_t pack_words(int R, int C, int role_y, int prec, bool whole) {
    const int K = (prec == BSM_P_TF32x3) ? 8 : 16;
    if (prec == BSM_P_OZAKI) {
        const int T = role_y ? R : C;
        const int hk = !whole && ((T - 1) & 15) < 8, kf = (T + 15) / 16 - hk;  // half and whole k-steps
        return role_y ? (int64_t)kf * oz_ystep<false>(C) + hk * oz_ystep<true>(C)
                      : (int64_t)kf * (whole ? oz_xstep_whole(R) : oz_xstep<false>(R)) + hk * oz_xstep<true>(R);
    }
    if (!role_y) {
        const int XW = prec == BSM_P_BF16x6 ? 12 : 8;
        const int last = !half_tile(R) ? XW : prec == BSM_P_BF16x6 ? 8 : 4;
        return (int64_t)((R - 1) / 16 * XW + last) * ((C + K - 1) / K) * 32;
    }
    const int YW = prec == BSM_P_BF16x6 ? 8 : 4;
    return (int64_t)((R + K - 1) / K) * ((C + 7) / 8) * 32 * YW;
}

// logical dims of block b for the role: X is R x T, Y is T x S
__device__ __forceinline__ void logical_dims(int32_t rc, int trans, int &rows, int &cols) {
    rows = trans ? rc_cols(rc) : rc_rows(rc);
    cols = trans ? rc_rows(rc) : rc_cols(rc);
}

__global__ void k_pack_sizes(int64_t nnzb, const int32_t *blk_rc, int role_y, int trans, int prec, bool whole,
                             int64_t *words, unsigned long long *other) {
    unsigned long long sum = 0;
    for (int64_t b = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; b < nnzb;
         b += (int64_t)gridDim.x * blockDim.x) {
        int rows, cols;
        logical_dims(blk_rc[b], trans, rows, cols);
        words[b] = pack_words(rows, cols, role_y, prec, whole);
        if (other) sum += (unsigned long long)pack_words(rows, cols, role_y, prec, !whole);
    }
    if (!other) return;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    if ((threadIdx.x & 31) == 0 && sum) atomicAdd(other, sum);
}

// one warp per block; lane L writes its fragment words of every tile
template <typename T, int PREC>
__global__ void k_pack(int64_t nnzb, const int64_t *blk_off, const int32_t *blk_rc, const T *data,
                       int role_y, int trans, const int64_t *pack_off, uint32_t *pack, const int32_t *status) {
    using PT = PrecTraits<PREC>;
    if (status && *status != 0) return;
    const int lane = threadIdx.x & 31;
    const int g = lane >> 2, t4 = lane & 3;
    const int64_t wid = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarp = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t b = wid; b < nnzb; b += nwarp) {
        const T *src = data + blk_off[b];
        int rows, cols;
        logical_dims(blk_rc[b], trans, rows, cols);
        // element accessor of the logical rows x cols block
        auto at = [&](int r, int c) -> double {
            return elem<T>(src, rows, cols, trans, r, c);
        };
        uint32_t *dst = pack + pack_off[b];
        uint32_t sp[3];
        if (!role_y) {
            const int MT = (rows + 15) / 16, KT = (cols + PT::K - 1) / PT::K;
            const bool half = half_tile(rows);
            const int xk = 32 * (PT::XW * (MT - 1) + (half ? PT::HW : PT::XW));
            for (int kt = 0; kt < KT; ++kt)
                for (int mt = 0; mt < MT; ++mt) {
                    // chunk pc (piece pc, registers v0..v3) of this lane at word 128 * pc
                    uint32_t *w = dst + (kt * xk + mt * (32 * PT::XW)) + 4 * lane;
                    const int r0 = mt * 16 + g, k0 = kt * PT::K;
                    if (half && mt == MT - 1) {  // v0, v2 of piece pc at word 128 * (pc >> 1) + 2 * (pc & 1)
                        uint32_t z[2][4] = {};
#pragma unroll
                        for (int v = 0; v < 2; ++v) {
                            if constexpr (PREC == BSM_P_TF32x3) {
                                split_value<PREC>(at(r0, k0 + t4 + 4 * v), sp);
                                z[0][v] = sp[0];
                                z[0][2 + v] = sp[1];
                            } else {
                                uint32_t lo[3], hi[3];
                                split_value<PREC>(at(r0, k0 + 2 * t4 + 8 * v), lo);
                                split_value<PREC>(at(r0, k0 + 2 * t4 + 8 * v + 1), hi);
#pragma unroll
                                for (int pc = 0; pc < PT::NP; ++pc)
                                    z[pc >> 1][2 * (pc & 1) + v] = lo[pc] | (hi[pc] << 16);
                            }
                        }
#pragma unroll
                        for (int c = 0; c < PT::HW / 4; ++c)
                            *reinterpret_cast<uint4 *>(w + 128 * c) = make_uint4(z[c][0], z[c][1], z[c][2], z[c][3]);
                        continue;
                    }
                    if constexpr (PREC == BSM_P_TF32x3) {
                        const int rr[4] = {r0, r0 + 8, r0, r0 + 8};
                        const int kk[4] = {k0 + t4, k0 + t4, k0 + t4 + 4, k0 + t4 + 4};
                        for (int v = 0; v < 4; ++v) {
                            split_value<PREC>(at(rr[v], kk[v]), sp);
                            w[v] = sp[0];
                            w[128 + v] = sp[1];
                        }
                    } else {
                        // reg v holds (row, k) and (row, k+1)
                        const int rr[4] = {r0, r0 + 8, r0, r0 + 8};
                        const int kk[4] = {k0 + 2 * t4, k0 + 2 * t4, k0 + 2 * t4 + 8, k0 + 2 * t4 + 8};
                        for (int v = 0; v < 4; ++v) {
                            uint32_t lo[3], hi[3];
                            split_value<PREC>(at(rr[v], kk[v]), lo);
                            split_value<PREC>(at(rr[v], kk[v] + 1), hi);
                            for (int pc = 0; pc < PT::NP; ++pc) w[128 * pc + v] = lo[pc] | (hi[pc] << 16);
                        }
                    }
                }
        } else {
            const int KT = (rows + PT::K - 1) / PT::K, NT = (cols + 7) / 8;
            for (int kt = 0; kt < KT; ++kt)
                for (int nt = 0; nt < NT; ++nt) {
                    // piece pc, registers v0 v1 at word 128 * (pc >> 1) + 2 * (pc & 1)
                    uint32_t *w = dst + (int64_t)(kt * NT + nt) * (32 * PT::YW) + 4 * lane;
                    const int n0 = nt * 8 + g, k0 = kt * PT::K;
                    if constexpr (PREC == BSM_P_TF32x3) {
                        const int kk[2] = {k0 + t4, k0 + t4 + 4};
                        for (int v = 0; v < 2; ++v) {
                            split_value<PREC>(at(kk[v], n0), sp);
                            w[v] = sp[0];
                            w[2 + v] = sp[1];
                        }
                    } else {
                        const int kk[2] = {k0 + 2 * t4, k0 + 2 * t4 + 8};
                        for (int v = 0; v < 2; ++v) {
                            uint32_t lo[3], hi[3];
                            split_value<PREC>(at(kk[v], n0), lo);
                            split_value<PREC>(at(kk[v] + 1, n0), hi);
                            for (int pc = 0; pc < PT::NP; ++pc) w[128 * (pc >> 1) + 2 * (pc & 1) + v] = lo[pc] | (hi[pc] << 16);
                        }
                        if constexpr (PT::NP == 3) {  // padding words of the second chunk
                            w[128 + 2] = 0;
                            w[128 + 3] = 0;
                        }
                    }
                }
        }
    }
}

// Unpacked pieces: out[e*NP + p] = piece p of element e (as an FP32 value)
template <typename T, int PREC>
__global__ void k_split_plain(int64_t n, const T *data, float *out) {
    constexpr int NP = PrecTraits<PREC>::NP;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x) {
        uint32_t sp[3];
        split_value<PREC>((double)data[e], sp);
#pragma unroll
        for (int p = 0; p < NP; ++p) {
            float v;
            if constexpr (PREC == BSM_P_TF32x3) v = __uint_as_float(sp[p]);
            else v = __bfloat162float(__ushort_as_bfloat16((unsigned short)sp[p]));
            out[e * NP + p] = v;
        }
    }
}

// Digits of x on its line's grid (see the Ozaki section above): slice p is
// d_p * 2^(-9p) as BF16 bits, exact.  e = unbiased exponent of the line.
__device__ __forceinline__ void oz_slices(double x, int e, uint32_t (&out)[kOzSlices]) {
    // The recursion y_0 = x * 2^(7-e), d_p = rint(y_p), y_(p+1) = (y_p - d_p) * 512
    // is exact in FP64 (y_p - d_p is exact, |y_p - d_p| <= 1/2), so it is run on
    // the integers: r = |x| * 2^(62-e) truncated (below 2^63; `sticky` records
    // whether anything was cut), digit p = r / 2^(55-9p) rounded half to even
    // with the cut part counted, r minus the digit.  The same digits as the
    // FP64 recursion -- signs of zero digits included -- without the FP64 pipe.
    const unsigned long long b = (unsigned long long)__double_as_longlong(x);
    const unsigned long long mag = b & 0x7fffffffffffffffull;
    if (mag == 0) {  // padding and exact zeros
#pragma unroll
        for (int p = 0; p < kOzSlices; ++p) out[p] = 0u;
        return;
    }
    const bool neg = (b >> 63) != 0;
    int ex = (int)(mag >> 52);
    unsigned long long m = mag & 0xfffffffffffffull;
    if (ex) m |= 1ull << 52;
    else ex = 1;
    // |x| * 2^(62-e) = m * 2^(ex - 1013 - e), ex - 1013 - e <= 11 and m < 2^53 (2^52 for ex = 1)
    const int sh = ex - 1013 - e;
    long long r;
    bool sticky;
    if (sh >= 0) {
        r = (long long)(m << sh);
        sticky = false;
    } else if (sh > -64) {
        r = (long long)(m >> -sh);
        sticky = (m & ((1ull << -sh) - 1ull)) != 0ull;
    } else {
        r = 0;
        sticky = true;
    }
#pragma unroll
    for (int p = 0; p < kOzSlices; ++p) {
        const int k = 55 - 9 * p;
        const long long rp = r;
        long long q = r >> k;  // floor
        const long long rem = r - (long long)((unsigned long long)q << k);
        const long long half = 1ll << (k - 1);
        if (rem > half || (rem == half && (sticky || (q & 1)))) ++q;
        r = (long long)((unsigned long long)r - ((unsigned long long)q << k));
        // d_p * 2^(-9p) with |d_p| <= 256: exact in FP32 and in BF16; a zero digit
        // takes the sign of the remainder it rounded (rint keeps it)
        float v = (float)q * __int_as_float((127 - 9 * p) << 23);
        if (neg) v = -v;
        if (q == 0) v = (neg ? (rp > 0 || (rp == 0 && sticky)) : (rp < 0)) ? -0.0f : 0.0f;
        out[p] = __bfloat16_as_ushort(__float2bfloat16_rn(v));
    }
}

// Ozaki fragment planes of FP64 data: the tiles of k_pack's BF16 layout with
// kOzSlices planes, chunk-major inside a tile; X element (r, k) uses the
// exponent of line line0[b] + r, Y element (k, n) that of line line0[b] + n.
template <bool WHOLE>
__global__ void k_pack_oz(int64_t nnzb, const int64_t *blk_off, const int32_t *blk_rc, const double *data,
                          int role_y, int trans, const int64_t *pack_off, uint32_t *pack, const int32_t *line0,
                          const int32_t *exps, const int32_t *status) {
    if (status && *status != 0) return;
    const int lane = threadIdx.x & 31;
    const int g = lane >> 2, t4 = lane & 3;
    const int64_t wid = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarp = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t b = wid; b < nnzb; b += nwarp) {
        const double *src = data + blk_off[b];
        int rows, cols;
        logical_dims(blk_rc[b], trans, rows, cols);
        const int32_t l0 = line0[b];
        uint32_t *dst = pack + pack_off[b];
        uint32_t lo[kOzSlices], hi[kOzSlices];
        if (!role_y) {
            const int MT = (rows + 15) / 16, KT = (cols + 15) / 16;
            for (int kt = 0; kt < KT; ++kt)
                for (int mt = 0; mt < MT; ++mt) {
                    const bool hk = !WHOLE && cols - 16 * kt <= 8, hm = !WHOLE && rows - 16 * mt <= 8;
                    uint32_t *w = dst + kt * (WHOLE ? oz_xstep_whole(rows) : oz_xstep<false>(rows)) + mt * (32 * (hk ? kOzHW : kOzXW)) + 4 * lane;
                    const int r0 = mt * 16 + g, k0 = kt * 16;
                    const int rr[4] = {r0, r0 + 8, r0, r0 + 8};
                    const int kk[4] = {k0 + 2 * t4, k0 + 2 * t4, k0 + 2 * t4 + 8, k0 + 2 * t4 + 8};
                    int u = 0;  // registers kept so far
#pragma unroll
                    for (int v = 0; v < 4; ++v) {
                        if ((hm && (v & 1)) || (hk && v >= 2)) continue;
                        const int e = rr[v] < rows ? exps[l0 + rr[v]] - 1023 : 0;
                        oz_slices(elem<double>(src, rows, cols, trans, rr[v], kk[v]), e, lo);
                        oz_slices(elem<double>(src, rows, cols, trans, rr[v], kk[v] + 1), e, hi);
#pragma unroll
                        for (int p = 0; p < kOzSlices; ++p)
                            w[hm && hk ? 128 * (p >> 2) + (p & 3) : hm ? 128 * (p >> 1) + 2 * u + (p & 1)
                              : hk ? 128 * (p >> 1) + 2 * (p & 1) + u : 128 * p + v] =
                                lo[p] | (hi[p] << 16);
                        ++u;
                    }
                    if (hm && hk) w[128 + 2] = w[128 + 3] = 0;  // padding words
                }
        } else {
            const int KT = (rows + 15) / 16, NT = (cols + 7) / 8;
            for (int kt = 0; kt < KT; ++kt)
                for (int nt = 0; nt < NT; ++nt) {
                    const bool hk = !WHOLE && rows - 16 * kt <= 8;
                    uint32_t *w = dst + kt * oz_ystep<false>(cols) + nt * (32 * (hk ? kOzQW : kOzYW)) + 4 * lane;
                    const int n0 = nt * 8 + g, k0 = kt * 16;
                    const int e = n0 < cols ? exps[l0 + n0] - 1023 : 0;
                    const int kk[2] = {k0 + 2 * t4, k0 + 2 * t4 + 8};
                    for (int v = 0; v < (hk ? 1 : 2); ++v) {
                        oz_slices(elem<double>(src, rows, cols, trans, kk[v], n0), e, lo);
                        oz_slices(elem<double>(src, rows, cols, trans, kk[v] + 1, n0), e, hi);
#pragma unroll
                        for (int p = 0; p < kOzSlices; ++p)
                            w[hk ? 128 * (p >> 2) + (p & 3) : 128 * (p >> 1) + 2 * ((p & 1) ^ ((lane >> 3) & 1)) + v] =
                                lo[p] | (hi[p] << 16);
                    }
                    if (hk) w[128 + 2] = w[128 + 3] = 0;  // padding words
                }
        }
    }
}

// line0[b] for every block: first global line of the block (one warp per block row)
__global__ void k_oz_line0(int32_t nbr, const int64_t *row_ptr, const int32_t *col_idx, const int32_t *row_start,
                           const int32_t *col_start, int by_rows, int32_t *line0) {
    const int lane = threadIdx.x & 31;
    const int64_t wid = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarp = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t i = wid; i < nbr; i += nwarp)
        for (int64_t b = row_ptr[i] + lane; b < row_ptr[i + 1]; b += 32)
            line0[b] = by_rows ? row_start[i] : col_start[col_idx[b]];
}

// exps[line] = max over the line of the biased exponent field of |x| (one warp
// per block, a lane per line of the block)
__global__ void k_oz_line_exp(int64_t nnzb, const int64_t *blk_off, const int32_t *blk_rc, const double *data,
                              const int32_t *line0, int by_rows, int32_t *exps) {
    const int lane = threadIdx.x & 31;
    const int64_t wid = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarp = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t b = wid; b < nnzb; b += nwarp) {
        const double *src = data + blk_off[b];
        const int R = rc_rows(blk_rc[b]), C = rc_cols(blk_rc[b]);
        const int nl = by_rows ? R : C, len = by_rows ? C : R;
        for (int l = lane; l < nl; l += 32) {
            int m = 0;
            for (int t = 0; t < len; ++t) {
                const double x = by_rows ? src[(int64_t)l * C + t] : src[(int64_t)t * C + l];
                m = max(m, (int)((unsigned long long)__double_as_longlong(x) >> 52) & 0x7ff);
            }
            atomicMax(&exps[line0[b] + l], m);
        }
    }
}

// Set bit 31 of order[t] when the block order[t] is computed by the CUDA-core
// variant: variant_of_class[size_index[rows] * ns + size_index[cols]] != 0.
__global__ void k_mark_variant(int64_t n, int32_t *order, const int32_t *blk_rc, const int32_t *size_index,
                               int32_t ns, const int8_t *variant_of_class, unsigned long long *marked) {
    unsigned long long cnt = 0;
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < n; t += (int64_t)gridDim.x * blockDim.x) {
        const int32_t q = order[t] & 0x7fffffff;
        const int32_t rc = blk_rc[q];
        if (variant_of_class[size_index[rc_rows(rc)] * ns + size_index[rc_cols(rc)]]) {
            order[t] = (int32_t)((uint32_t)q | 0x80000000u);
            cnt++;
        }
    }
    if (marked && cnt) atomicAdd(marked, cnt);
}

template <int MAXN, bool HM, bool HKS, bool WT = false>
cudaError_t launch_oz_inst(const NumericArgs &a, cudaStream_t s, int threads, int *grid) {
    const size_t smem = sizeof(uint32_t) * (size_t)oz_ring_words_per_warp<MAXN>() * (threads / 32);
    cudaError_t e =
        cudaFuncSetAttribute(k_numeric_oz<MAXN, HM, HKS, WT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    *grid = persistent_grid(k_numeric_oz<MAXN, HM, HKS, WT>, a.n_items, smem, threads, a.ctas_per_sm);
    k_numeric_oz<MAXN, HM, HKS, WT><<<*grid, threads, smem, s>>>(a);
    count_launch(1);
    return cudaGetLastError();
}

// The kernels for the tile rows that the output's block sizes can have, without
// the code of half steps where no inner size has them: blocks of 32 took 4.6 ms
// with it and 4.2 without (4.4 before either; 457,000 products).
template <int MAXN, bool HM>
cudaError_t launch_oz_rows(const NumericArgs &a, cudaStream_t s, int threads, int *grid) {
    return a.half_mask & kHalfInner ? launch_oz_inst<MAXN, HM, true>(a, s, threads, grid)
                                    : launch_oz_inst<MAXN, HM, false>(a, s, threads, grid);
}

template <int MAXN>
cudaError_t launch_oz(const NumericArgs &a, cudaStream_t s, int threads, int *grid) {
    if (a.half_mask & kAllWhole) return launch_oz_inst<MAXN, false, false, true>(a, s, threads, grid);
    cudaError_t e = cudaSuccess;
    if (a.half_mask & kHalfRows) e = launch_oz_rows<MAXN, true>(a, s, threads, grid);
    if (e == cudaSuccess && (a.half_mask & kWholeRows)) e = launch_oz_rows<MAXN, false>(a, s, threads, grid);
    return e;
}

}  // namespace

int num_sms() {
    static std::atomic<int> count{0};
    int n = count.load(std::memory_order_relaxed);
    if (n == 0) {
        int dev = 0;
        if (cudaGetDevice(&dev) != cudaSuccess ||
            cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n <= 0)
            n = 1;
        count.store(n, std::memory_order_relaxed);
    }
    return n;
}

// Whether the output has too few blocks for lane groups and register tiles, which
// share warps among blocks of one shape: then a warp per block (k_warp.cu).  Times of
// a warp per block over those of the sharing kernel, uniform patterns, 0.7 to 40
// products a block:
//   FP64  5 x 5        5,000 blocks 0.87-0.93   20,000 0.74-1.07    78,000 1.31-1.34
//         8 x 8        5,000 0.89-0.98          40,000 0.74-0.90   160,000 0.98-1.16
//         13 x 13      5,000 0.92-0.97          20,000 0.87-1.02    78,000 1.05-1.09
//         23 x 23      3,000 0.87-0.95          20,000 1.01-1.05
//         32 x 32      1,500 0.84-1.09          10,000 1.08-1.12
//         5/13/23      5,000 0.62-0.77          80,000 0.82-0.90   160,000 1.08-1.28
//         2/6          5,000 0.83-0.96          40,000 0.70-0.76   160,000 1.51-2.00
//   FP32  5 x 5        5,000 0.79-0.85          20,000 0.83-1.74
//         13 x 13      3,000 0.90-1.24          10,000 1.15-1.38
//         5/13         5,000 0.78-0.97          20,000 0.78-1.11
//         23 x 23, 32 x 32 and more: 1.2 to 3 from 1,000 on
static bool few_blocks(const NumericArgs &a) {
    const int area = a.max_out_rows * a.max_out_cols;
    int per_sm;
    if (area <= 16) per_sm = 0;
    else if (a.dtype == BSM_FP64) per_sm = a.out_shapes > 1 ? (area <= 64 ? 400 : 800) : area > 288 ? 32 : area % 32 == 0 ? 400 : 200;
    else per_sm = a.out_shapes > 1 ? (area <= 576 ? 100 : 0) : area <= 64 ? 64 : 0;
    return a.n_items <= (int64_t)per_sm * num_sms();
}

cudaError_t launch_numeric(const NumericArgs &args, cudaStream_t s, NumericLaunch *info) {
    NumericArgs a = args;
    a.unit_alpha = a.alpha == 1.0;
    a.has_old = a.beta != 0.0 && a.old_off;
    NumericLaunch li{BSM_K_NONE, -1, 0, 0, 0, 0};
    if (info) *info = li;
    if (a.n_items == 0) return cudaSuccess;
    cudaError_t e = cudaMemsetAsync(a.work_counter, 0, kWorkCounters * sizeof(unsigned long long), s);
    if (e != cudaSuccess) return e;
    const bool tc = a.prec == BSM_P_TF32x3 || a.prec == BSM_P_BF16x3 || a.prec == BSM_P_BF16x6;
    // the mma.sync kernels run 2 or 4 warps per CTA (compiled for at most 4,
    // which keeps their register count at three CTAs per SM)
    const int tc_threads = (a.cta_warps == 2 ? 2 : 4) * 32;
    int grid = 0;
    if (a.prec == BSM_P_OZAKI) {
        // passes of up to 3 tiles (the default) take the instance with the
        // wider ring; with item groups the blocks of one tile column run in
        // the 1-tile instance
        const bool wide = a.pass_nt != 1 && a.pass_nt != 2;
        NumericArgs b = a;
        b.group = a.item_groups ? 0 : -1;
        e = wide ? launch_oz<3>(b, s, tc_threads, &grid) : launch_oz<2>(b, s, tc_threads, &grid);
        if (e == cudaSuccess && a.item_groups) {
            int g1 = 0;
            b.group = 1;
            e = launch_oz<1>(b, s, tc_threads, &g1);
        }
        if (e == cudaSuccess && a.n_lane_items) {
            const int g = persistent_grid(k_numeric_oz_lane, a.n_items / 32 + 1, 0, kThreadsNum, a.ctas_per_sm);
            k_numeric_oz_lane<<<g, kThreadsNum, 0, s>>>(a);
            count_launch(1);
            e = cudaGetLastError();
        }
        li = NumericLaunch{BSM_K_OZAKI_MMA, -1, tc_threads, grid, 1, wide ? 3 : (a.pass_nt == 1 ? 1 : 2)};
    } else if (a.prec == BSM_P_FP64_DMMA && a.dtype == BSM_FP64) {
        grid = persistent_grid(k_numeric_dmma, a.n_items, 0, kThreadsNum, a.ctas_per_sm);
        k_numeric_dmma<<<grid, kThreadsNum, 0, s>>>(a);
        li = NumericLaunch{BSM_K_FP64_MMA, -1, kThreadsNum, grid, a.pass_mt > 0 ? a.pass_mt : 3,
                           a.pass_nt > 0 ? a.pass_nt : 3};
    } else if (!tc) {
        const int area = a.max_out_rows * a.max_out_cols;
        const bool few = few_blocks(a);
        // the build by the largest output block: narrow up to 288 elements and
        // beyond the wide ladder's single pass (768), wide between, where its
        // larger Q fill more lane slots; narrow and wide in ms (3e10 useful
        // FLOP, 10% occupancy): 16 x 16 23.9 and 24.3, 17 x 17 27.4 and 25.6,
        // 18 x 18 26.2 and 25.1, 20 x 20 25.0 and 25.1, 23 x 23 26.1 and 24.8,
        // 24 x 24 24.0 and 24.2, 32 x 32 24.5 and 24.7.  The tuner may ask for
        // either; the small build only ever runs when every output block has at
        // most 16 elements
        int build = area > 0 && area <= 16 ? kCcSmall : area <= 288 || area > 768 ? kCcNarrow : kCcWide;
        if (a.fp64_build == 1 && build != kCcSmall) build = kCcNarrow;
        if (a.fp64_build == 2 && build != kCcSmall) build = kCcWide;
        if (few) e = launch_numeric_warp(a, build == kCcWide, s, &grid);
        else if (a.dtype == BSM_FP64) e = launch_numeric_group(a, build, s, &grid);
        else e = launch_numeric_tile(a, s, &grid);
        if (a.dtype != BSM_FP64) build = -1;
        li = NumericLaunch{BSM_K_FP64_CORES, build, kThreadsNum, grid, 0, 0};
    } else {
        if (a.prec == BSM_P_TF32x3) e = launch_split_tf32x3(a, s, tc_threads, &grid);
        else if (a.prec == BSM_P_BF16x3) e = launch_split_bf16x3(a, s, tc_threads, &grid);
        else e = launch_split_bf16x6(a, s, tc_threads, &grid);
        li = NumericLaunch{BSM_K_SPLIT_MMA, -1, tc_threads, grid,
                           a.item_groups ? 0 : (a.pass_mt > 0 ? a.pass_mt : 2), a.pass_nt > 0 ? a.pass_nt : 3};
    }
    if (e != cudaSuccess) return e;
    if (info) *info = li;
    if (!tc && a.prec != BSM_P_OZAKI) count_launch(1);  // the split and Ozaki paths count their own
    return cudaGetLastError();
}

uint32_t numeric_debug_bits(cudaStream_t s) {
    return read_debug_bits(s) | group_debug_bits(s) | tile_debug_bits(s) | warp_debug_bits(s) | split_tf32x3_debug_bits(s) |
           split_bf16x3_debug_bits(s) | split_bf16x6_debug_bits(s);
}

cudaError_t launch_split_plain(const bsm_mat *M, int prec, float *out, cudaStream_t s) {
    if (M->data_len == 0) return cudaSuccess;
    int64_t g = (M->data_len + 255) / 256;
    if (g > 152 * 32) g = 152 * 32;
    const bool f64 = M->dtype == BSM_FP64;
    if (prec == BSM_P_TF32x3) {
        if (f64) k_split_plain<double, BSM_P_TF32x3><<<(unsigned)g, 256, 0, s>>>(M->data_len, static_cast<const double *>(M->data), out);
        else k_split_plain<float, BSM_P_TF32x3><<<(unsigned)g, 256, 0, s>>>(M->data_len, static_cast<const float *>(M->data), out);
    } else if (prec == BSM_P_BF16x3) {
        if (f64) k_split_plain<double, BSM_P_BF16x3><<<(unsigned)g, 256, 0, s>>>(M->data_len, static_cast<const double *>(M->data), out);
        else k_split_plain<float, BSM_P_BF16x3><<<(unsigned)g, 256, 0, s>>>(M->data_len, static_cast<const float *>(M->data), out);
    } else {
        if (f64) k_split_plain<double, BSM_P_BF16x6><<<(unsigned)g, 256, 0, s>>>(M->data_len, static_cast<const double *>(M->data), out);
        else k_split_plain<float, BSM_P_BF16x6><<<(unsigned)g, 256, 0, s>>>(M->data_len, static_cast<const float *>(M->data), out);
    }
    count_launch(1);
    return cudaGetLastError();
}

int split_pieces(int prec) { return prec == BSM_P_BF16x6 ? 3 : 2; }

cudaError_t launch_oz_lines(const bsm_mat *M, int by_rows, int32_t *line0, int32_t *exps, cudaStream_t s) {
    if (M->nnzb == 0) return cudaSuccess;
    if (M->dtype != BSM_FP64 || !M->row_start || !M->col_start) return cudaErrorInvalidValue;
    int64_t g = ((int64_t)M->nbr * 32 + 255) / 256;
    if (g > 152 * 32) g = 152 * 32;
    k_oz_line0<<<(unsigned)g, 256, 0, s>>>(M->nbr, M->row_ptr, M->col_idx, M->row_start, M->col_start, by_rows,
                                           line0);
    g = (M->nnzb * 32 + 255) / 256;
    if (g > 152 * 32) g = 152 * 32;
    k_oz_line_exp<<<(unsigned)g, 256, 0, s>>>(M->nnzb, M->blk_off, M->blk_rc, static_cast<const double *>(M->data),
                                              line0, by_rows, exps);
    count_launch(2);
    return cudaGetLastError();
}

cudaError_t launch_mark_variant(int64_t n, int32_t *order, const int32_t *blk_rc, const int32_t *size_index, int32_t ns,
                                const int8_t *variant_of_class, unsigned long long *marked, cudaStream_t s) {
    if (n == 0) return cudaSuccess;
    int64_t g = (n + 255) / 256;
    if (g > 152 * 32) g = 152 * 32;
    k_mark_variant<<<(unsigned)g, 256, 0, s>>>(n, order, blk_rc, size_index, ns, variant_of_class, marked);
    count_launch(1);
    return cudaGetLastError();
}

cudaError_t launch_pack_sizes(const bsm_mat *M, int role_y, int trans, int prec, bool whole, int64_t *pack_words,
                              unsigned long long *other, cudaStream_t s) {
    if (M->nnzb == 0) return cudaSuccess;
    int64_t g = (M->nnzb + 255) / 256;
    if (g > 152 * 32) g = 152 * 32;
    k_pack_sizes<<<(unsigned)g, 256, 0, s>>>(M->nnzb, M->blk_rc, role_y, trans, prec, whole, pack_words, other);
    count_launch(1);
    return cudaGetLastError();
}

cudaError_t launch_pack(const bsm_mat *M, int role_y, int trans, int prec, bool whole, const int64_t *pack_off,
                        void *pack, const int32_t *status, cudaStream_t s, const int32_t *line0,
                        const int32_t *exps) {
    if (M->nnzb == 0) return cudaSuccess;
    int64_t g = (M->nnzb * 32 + 255) / 256;
    if (g > 152 * 32) g = 152 * 32;
    uint32_t *p = static_cast<uint32_t *>(pack);
    const bool f64 = M->dtype == BSM_FP64;
    if (prec == BSM_P_OZAKI) {
        if (!f64 || !line0 || !exps) return cudaErrorInvalidValue;
        const double *d = static_cast<const double *>(M->data);
        if (whole)
            k_pack_oz<true><<<(unsigned)g, 256, 0, s>>>(M->nnzb, M->blk_off, M->blk_rc, d, role_y, trans, pack_off, p,
                                                        line0, exps, status);
        else
            k_pack_oz<false><<<(unsigned)g, 256, 0, s>>>(M->nnzb, M->blk_off, M->blk_rc, d, role_y, trans, pack_off, p,
                                                         line0, exps, status);
        count_launch(1);
        return cudaGetLastError();
    }
#define BSM_PACK_CASE(PREC)                                                                           \
    if (f64)                                                                                          \
        k_pack<double, PREC><<<(unsigned)g, 256, 0, s>>>(M->nnzb, M->blk_off, M->blk_rc,              \
                                                         static_cast<const double *>(M->data), role_y, \
                                                         trans, pack_off, p, status);                         \
    else                                                                                              \
        k_pack<float, PREC><<<(unsigned)g, 256, 0, s>>>(M->nnzb, M->blk_off, M->blk_rc,               \
                                                        static_cast<const float *>(M->data), role_y,   \
                                                        trans, pack_off, p, status);
    if (prec == BSM_P_TF32x3) {
        BSM_PACK_CASE(BSM_P_TF32x3)
    } else if (prec == BSM_P_BF16x3) {
        BSM_PACK_CASE(BSM_P_BF16x3)
    } else {
        BSM_PACK_CASE(BSM_P_BF16x6)
    }
#undef BSM_PACK_CASE
    count_launch(1);
    return cudaGetLastError();
}

}  // namespace bsm
