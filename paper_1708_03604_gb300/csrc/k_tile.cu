// FP32 data on the CUDA cores: register tiles in lane groups.
//
// Every output block is the sum of its small dense block products (Bethune et
// al. 2017 §2): each product is one chain of FP32 fused multiply-adds per
// element in ascending k, the products are added up in FP64 in ascending order
// -- per element the same operations whatever the tile below.
//
// What bounds it: with an element per lane and term of k, two loads per FMA.
// A group of LR x LC lanes owns a block and each lane a TR x TC tile of it, TR +
// TC loads for TR TC FMAs; 32 / (LR LC) groups of a warp walk their own product
// lists side by side.  Next come the FP64 additions, one per element and product
// at 16 cycles a warp and SM, so tiles that leave lanes idle cost there.
//
// Measured against an element per lane (ms of the kernel, 3e10 useful FLOP each,
// uniform patterns of 10% occupancy): 5 x 5 blocks 34.0 -> 9.1, 8 x 8 17.7 -> 6.5,
// 13 x 13 11.5 -> 7.0, 16 x 16 9.3 -> 4.4, 23 x 23 9.8 -> 3.2, 32 x 32 8.2 -> 3.7,
// mixed 5/13/23 20.5 -> 7.7.
#include <cuda_runtime.h>

#include <type_traits>

#include "numeric_items.cuh"

namespace bsm {

namespace {

// tiles of up to kTileCols columns and `ROWS` rows are compiled: 4 where every
// block has at most 288 elements (96 registers, five CTAs an SM: 16 x 16 blocks
// 4.8 -> 4.1 ms), 6 elsewhere (128 registers, four CTAs: 23 x 23 4.3 -> 3.2 ms).
// Held to those they spill (ptxas: 386 and 234 bytes of stores, 218 and 140 of loads)
constexpr int kTileCols = 4;

// cycles of a line, and of the way from product to product
constexpr float kLine = 0.6f, kWay = 70.f;

struct TilePlan {
    int lr, lc, tr, tc;
};

// The lanes and tile of an m x n block, the cheapest in cycles per block
// product: the FP64 additions (16 per tile element), the loads (a line of 128
// bytes a cycle: a load touches `lr` rows of X or `lc` columns of Y in every
// group, one line where they lie side by side), the FMAs' issue and the way
// from product to product; several passes where the lanes' tiles do not cover
// the block.  Every lane of the warp rates lane + 1 rows of lanes.
template <int ROWS>
__device__ TilePlan tile_plan(int m, int n, bool spread, const NumericArgs &a, int lane) {
    const int lr = lane + 1;
    const float k = 0.5f * (float)(m + n);
    float best = 3.0e38f;
    int best_lc = 1;
    for (int lc = 1; lr * lc <= 32 && lr <= m && lc <= n; ++lc) {
        const int tr = min(ROWS, (m + lr - 1) / lr), tc = min(kTileCols, (n + lc - 1) / lc);
        const int passes = ((m + lr * tr - 1) / (lr * tr)) * ((n + lc * tc - 1) / (lc * tc));
        const int groups = 32 / (lr * lc);
        const float x_lines = a.x_trans ? 1.f : fminf((float)lr, (float)lr * k * (1.f / 32.f) + 1.f);
        const float y_lines = a.y_trans ? fminf((float)lc, (float)lc * k * (1.f / 32.f) + 1.f) : 1.f;
        const float loads = (float)groups * ((float)tr * x_lines + (float)tc * y_lines);
        const float cycles = 16.f * (float)(tr * tc) + k * (fmaxf(1.3f * (float)(tr + tc), kLine * loads) + 0.25f * (float)(tr * tc)) + kWay;
        // products of different length run for the longest of the warp's groups
        const float wait = a.mixed_k ? 1.f + 0.1f * (float)(31 - __clz(groups)) : 1.f;
        const float cost = cycles * (float)passes * wait / (float)(spread ? 1 : groups);
        if (cost < best) {
            best = cost;
            best_lc = lc;
        }
    }
    const uint32_t key = __float_as_uint(best);  // ordered as the value
    const int win = __ffs(__ballot_sync(0xffffffffu, key == __reduce_min_sync(0xffffffffu, key))) - 1;
    const int r = win + 1, c = __shfl_sync(0xffffffffu, best_lc, win);
    return TilePlan{r, c, min(ROWS, (m + r - 1) / r), min(kTileCols, (n + c - 1) / c)};
}

// Blocks of shape m x n from `run`, until the next one has another shape or
// none is left.
template <int TR, int TC>
__device__ __forceinline__ void tile_run(const NumericArgs &a, ItemRun &run, int lane, int m, int n, int lr, int lc) {
    constexpr int TU = TR + TC <= 4 ? 4 : 2;
    const float *__restrict__ X = static_cast<const float *>(a.x_data);
    const float *__restrict__ Y = static_cast<const float *>(a.y_data);
    const int g = lr * lc, groups = 32 / g, gi = lane / g, l = lane - gi * g;
    const int lrow = l / lc, lcol = l - lrow * lc;
    const bool member = gi < groups;
    const unsigned before = (1u << (gi * g & 31)) - 1u;  // lanes of the groups before this one
    const int32_t shape = (m << 16) | n;
    const int xs_t = a.x_trans ? m : 1, ys_t = a.y_trans ? 1 : n;
    // products per FP64 addition
    const int every = a.flush_every > 0 && !a.each_product.has(m, n) ? a.flush_every : 1;

    double acc[TR][TC];
    float part[TR][TC];
    int xo[TR], yo[TC];
    auto clear = [&]() {
#pragma unroll
        for (int i = 0; i < TR; ++i)
#pragma unroll
            for (int j = 0; j < TC; ++j) {
                acc[i][j] = 0.0;
                part[i][j] = 0.f;
            }
    };
    clear();  // defined on every path (see k_group.cu)
#pragma unroll
    for (int i = 0; i < TR; ++i) xo[i] = 0;
#pragma unroll
    for (int j = 0; j < TC; ++j) yo[j] = 0;
    bool act = false, closed = false;
    int32_t item = 0, p = 0, pe = 0;    // the block and its products left, [p, pe)
    int r0 = 0, c0 = 0;                 // first row and column of the pass
    int tn = -1, since = 0;             // terms of k of the product at p; products since an addition
    const float *xp = X, *yp = Y;
    int64_t nxo = 0, nyo = 0;           // one product ahead
    int ntn = 0;
    int32_t ix2 = 0, iy2 = 0;           // two ahead

    auto load_offsets = [&](int32_t ix, int32_t iy) {
        const int32_t rc = a.x_blk_rc[ix];
        nxo = a.x_blk_off[ix];
        nyo = a.y_blk_off[iy];
        ntn = a.x_trans ? rc_rows(rc) : rc_cols(rc);
    };
    auto advance = [&]() {
        xp = X + nxo;
        yp = Y + nyo;
        if (ntn != tn) {
            tn = ntn;
            const int xs_r = a.x_trans ? 1 : tn, ys_s = a.y_trans ? tn : 1;
            // rows and columns past the block: element 0
#pragma unroll
            for (int i = 0; i < TR; ++i) xo[i] = r0 + lrow + lr * i < m ? (r0 + lrow + lr * i) * xs_r : 0;
#pragma unroll
            for (int j = 0; j < TC; ++j) yo[j] = c0 + lcol + lc * j < n ? (c0 + lcol + lc * j) * ys_s : 0;
        }
        if (pe - p > 1) load_offsets(ix2, iy2);
        if (pe - p > 2) {
            ix2 = a.px[p + 2];
            iy2 = a.py[p + 2];
        }
    };
    auto begin = [&]() {
        clear();
        since = 0;
        tn = -1;
        advance();
    };
    // the product's sums into FP64.  The conversion is exact and takes a warp 16
    // cycles of the FP64 pipe like the addition, so it is done on the bits; zero,
    // subnormal and non-finite sums (in any slot of the lane) go the usual way.
    auto add_up = [&]() {
        since = 0;
        bool usual = false;
#pragma unroll
        for (int i = 0; i < TR; ++i)
#pragma unroll
            for (int j = 0; j < TC; ++j)
                usual |= (__float_as_uint(part[i][j]) & 0x7fffffffu) - 0x800000u >= 0x7f000000u;
        if (usual) {
#pragma unroll
            for (int i = 0; i < TR; ++i)
#pragma unroll
                for (int j = 0; j < TC; ++j) {
                    double w;
                    asm volatile("cvt.f64.f32 %0, %1;" : "=d"(w) : "f"(part[i][j]));
                    acc[i][j] += w;
                    part[i][j] = 0.f;
                }
            return;
        }
#pragma unroll
        for (int i = 0; i < TR; ++i)
#pragma unroll
            for (int j = 0; j < TC; ++j) {
                const uint32_t u = __float_as_uint(part[i][j]);
                acc[i][j] += __hiloint2double((int)((u & 0x80000000u) | (((u & 0x7fffffffu) >> 3) + ((1023u - 127u) << 20))),
                                              (int)(u << 29));
                part[i][j] = 0.f;
            }
    };
    auto store = [&]() {
        float *__restrict__ O = static_cast<float *>(a.out_data) + a.out_blk_off[item];
        const int64_t old = a.has_old ? a.old_off[item] : -1;
        const float *OLD = static_cast<const float *>(a.old_data) + old;
        auto each = [&](auto value) {
#pragma unroll
            for (int i = 0; i < TR; ++i)
#pragma unroll
                for (int j = 0; j < TC; ++j) {
                    const int r = r0 + lrow + lr * i, c = c0 + lcol + lc * j;
                    if (r < m && c < n) O[r * n + c] = (float)value(acc[i][j], r * n + c);
                }
        };
        if (a.unit_alpha && old < 0) each([&](double v, int) { return v; });
        else if (old < 0) each([&](double v, int) { return a.alpha * v; });
        else each([&](double v, int e) { return fma(a.beta, (double)OLD[e], a.alpha * v); });
    };
    // the next pass over the block; false when it is done
    auto next_pass = [&]() {
        c0 += lc * TC;
        if (c0 >= n) {
            c0 = 0;
            r0 += lr * TR;
        }
        return r0 < m;
    };
    auto terms = [&](auto count) {
        constexpr int N = decltype(count)::value;
        float xv[N][TR], yv[N][TC];
#pragma unroll
        for (int q = 0; q < N; ++q) {
#pragma unroll
            for (int i = 0; i < TR; ++i) xv[q][i] = __ldg(xp + xo[i]);
#pragma unroll
            for (int j = 0; j < TC; ++j) yv[q][j] = __ldg(yp + yo[j]);
            xp += xs_t;
            yp += ys_t;
        }
#pragma unroll
        for (int q = 0; q < N; ++q)
#pragma unroll
            for (int i = 0; i < TR; ++i)
#pragma unroll
                for (int j = 0; j < TC; ++j) part[i][j] = fmaf(xv[q][i], yv[q][j], part[i][j]);
    };

    for (;;) {
        // groups without a block take the next ones of this shape
        while (!closed) {
            const unsigned need = __ballot_sync(0xffffffffu, member && !act && l == 0);
            if (!need) break;
            if (!items_left(a, run, lane)) {
                closed = true;
                break;
            }
            const int count = min(__popc(need), run.count - run.cur);
            const int rank = __popc(need & before), slot = run.cur + rank;
            const bool want = member && !act && rank < count;
            const Window &w = *run.w;
            const unsigned other = __ballot_sync(0xffffffffu, want && l == 0 && w.shape[slot] != shape);
            const int take = other ? __popc(need & (other & (0u - other)) - 1u) : count;
            if (want && rank < take) {
                item = w.item[slot];
                p = w.p[slot];
                pe = w.pe[slot];
                r0 = c0 = 0;
                if (p < pe) {
                    if (BSM_DBG_LANE_OK(a, item)) {
                        act = true;
                        nxo = w.xoff[slot];
                        nyo = w.yoff[slot];
                        ntn = w.tn[slot];
                        ix2 = w.ix[slot];
                        iy2 = w.iy[slot];
                        begin();
                    }
                } else {  // no product: alpha * 0 + beta * old
                    clear();
                    do store();
                    while (next_pass());
                }
            }
            run.cur += take;
            closed = other != 0u;
            __syncwarp();  // the window may be overwritten
        }
        if (!__ballot_sync(0xffffffffu, act)) break;
        if (act) {
            int s = 0;
#pragma unroll 1
            for (; s + TU <= tn; s += TU) terms(std::integral_constant<int, TU>{});
#pragma unroll 1
            for (; s < tn; ++s) terms(std::integral_constant<int, 1>{});
            if (++since == every || p + 1 == pe) add_up();
            if (++p < pe) {
                advance();
            } else {
                store();
                act = next_pass();
                if (act) {
                    p = (int32_t)a.seg_ptr[item];
                    load_offsets(a.px[p], a.py[p]);
                    if (pe - p > 1) {
                        ix2 = a.px[p + 1];
                        iy2 = a.py[p + 1];
                    }
                    begin();
                }
            }
        }
        __syncwarp();
    }
}

template <int ROWS>
__global__ void __launch_bounds__(kGroupThreads, ROWS == 4 ? 5 : 4) k_numeric_tile(NumericArgs a) {
    __shared__ Window windows[kGroupThreads / 32];
    if (a.status && *a.status != 0) return;
    const int lane = threadIdx.x & 31;
    // a few blocks for each warp of the grid: a warp per block, so that all work
    const bool spread = a.n_items <= 4 * (int64_t)gridDim.x * (kGroupThreads / 32);
    ItemRun run{&windows[threadIdx.x >> 5], 0, 0, a.n_items};
    while (items_left(a, run, lane)) {
        const int32_t rc = run.w->shape[run.cur];
        const int m = rc_rows(rc), n = rc_cols(rc);
        const TilePlan pl = tile_plan<ROWS>(m, n, spread, a, lane);
        // one element per lane in as many passes as it takes, the default, takes every
        // shape: whatever the plan, the run ends
        switch (pl.tr * 8 + pl.tc) {
            default:
#define BSM_TILE(TR, TC) \
    case TR * 8 + TC:                                                             \
        if constexpr (TR <= ROWS) tile_run<TR, TC>(a, run, lane, m, n, pl.lr, pl.lc); \
        break;
#define BSM_TILE_ROW(TR) BSM_TILE(TR, 1) BSM_TILE(TR, 2) BSM_TILE(TR, 3) BSM_TILE(TR, 4)
            BSM_TILE_ROW(1) BSM_TILE_ROW(2) BSM_TILE_ROW(3) BSM_TILE_ROW(4) BSM_TILE_ROW(5) BSM_TILE_ROW(6)
#undef BSM_TILE_ROW
#undef BSM_TILE
        }
    }
}

}  // namespace

cudaError_t launch_numeric_tile(const NumericArgs &a, cudaStream_t s, int *grid) {
    static std::atomic<int> low{0}, high{0};
    if (a.max_out_rows * a.max_out_cols <= 288) return launch_persistent(k_numeric_tile<4>, low, a, s, grid);
    return launch_persistent(k_numeric_tile<6>, high, a, s, grid);
}

uint32_t tile_debug_bits(cudaStream_t s) { return read_debug_bits(s); }

}  // namespace bsm
