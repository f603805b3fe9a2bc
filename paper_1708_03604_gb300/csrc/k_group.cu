// FP64 numeric kernel on the CUDA cores (FP64 FMA): lane groups.
//
// Every output block accumulates its list of small dense block products
// (Bethune et al. 2017 §2) in ascending product, then ascending k, one FP64
// fused multiply-add per element and term of k -- the same chain of FMAs per
// element whatever the layout below, so results do not depend on it.
//
// What bounds it: GB300's FP64 pipe, one warp-wide FMA every 16 cycles per SM
// whether 32 lanes are used or one.  So the layout is chosen to leave as few
// lanes idle as possible: a group of g lanes owns a block and each of its lanes
// Q = ceil(m n / g) elements, 32 / g groups of a warp work on blocks of one
// shape side by side, each walking its own product list and taking the next
// block when it is done.  A warp per block (g = 32, Q = ceil(m n / 32)) fills
// 36 of 64 slots of a 6 x 6 block and 65 of 96 of a 5 x 13 one; 8 groups of 4
// lanes fill 288 of 288, 6 groups of 5 lanes 390 of 416.
//
// Measured against a warp per block (useful TFLOP/s of the kernel, uniform
// patterns of 10% occupancy, 1.256 being the pipe's rate): 4 x 4 blocks 0.83 ->
// 1.13, 5 x 5 0.60 -> 1.08, 6 x 6 0.62 -> 1.21, 8 x 8 1.18 -> 1.24, 13 x 13 1.05
// -> 1.18, 16 x 16 1.08 -> 1.25, 23 x 23 1.14 -> 1.20, 32 x 32 1.07 -> 1.23,
// mixed 5/13/23 0.87 -> 1.12.
#include <cuda_runtime.h>

#include <atomic>
#include <type_traits>

#include "bsm_internal.cuh"
#include "numeric_items.cuh"

namespace bsm {

namespace {

// Elements per lane (Q) compiled into each build; the widest sets the register
// count and with it how many warps an SM holds: small 64 registers, narrow 80 (24
// warps), wide 128 (16).  Held to those by the launch bounds they spill (ptxas:
// 8, 796 and 492 bytes of stores, 36, 460 and 176 of loads); the FP64 pipe is 97%
// (1,200 rows of 5/13/23) to 99% busy (2,000 banded rows of 23 x 23) all the same.
constexpr uint32_t q_bit(int q) { return 1u << q; }
constexpr uint32_t kQSmall = q_bit(1) | q_bit(2) | q_bit(3) | q_bit(4);
constexpr uint32_t kQNarrow = kQSmall | q_bit(5) | q_bit(6) | q_bit(7) | q_bit(8) | q_bit(9) | q_bit(11) | q_bit(13);
constexpr uint32_t kQWide = kQNarrow | q_bit(15) | q_bit(17) | q_bit(19) | q_bit(21) | q_bit(24);
// Q of the layouts whose lanes keep one row or one column
constexpr uint32_t kQShared = kQNarrow;
// whether Q = q is compiled into a build; any q (a shift by 32 is undefined)
__host__ __device__ constexpr bool has_q(uint32_t mask, int q) { return q < 32 && ((mask >> q) & 1u); }
static_assert(has_q(kQWide, 24) && !has_q(kQWide, 31) && !has_q(kQWide, 32));
static_assert(has_q(kQSmall, 1) && has_q(kQNarrow, 1) && has_q(kQWide, 1));

template <int BUILD>
__host__ __device__ constexpr uint32_t q_mask() {
    return BUILD == kCcSmall ? kQSmall : BUILD == kCcNarrow ? kQNarrow : kQWide;
}
__host__ __device__ constexpr int q_max(uint32_t mask) {
    int q = 0;
    for (int b = 1; b < 32; ++b)
        if (mask & (1u << b)) q = b;
    return q;
}

// Layouts.  Element (r, c) of a lane's slot u, l its number in the group:
//   kFlat  the block in row-major order, element l + g u
//   kRow   in column-major order with g a multiple of m: every slot of a lane
//          has one row, so X is loaded once per term of k
//   kCol   in row-major order with g a multiple of n: one column per lane, Y
//          is loaded once per term of k
enum { kFlat = 0, kRow = 1, kCol = 2 };

struct GroupPlan {
    int mode, q, g;
};

// The layout of an m x n block, the cheapest in cycles per block and term of
// k: the larger of the FP64 pipe's (16 per slot) and of the load path's (two
// 128-byte lines a cycle: groups times the lines they touch), and a few for the
// loop, so that one pass goes before several; ties to the wider group (fewer
// blocks in flight, less divergence).  Every lane of the warp rates
// the group size lane + 1 in each layout, and a whole warp per block with
// lane + 1 slots in as many passes over the products as it takes.
template <uint32_t MASK>
__device__ GroupPlan group_plan(int m, int n, bool spread, int lane) {
    const int rs = m * n, blk_lines = (((m + n) / 2 * max(m, n) * 8) >> 7) + 1;
    uint32_t best = 0xffffffffu;
    int best_mode = kFlat, best_q = 0, best_g = 32;
    const int kavg = max(1, (m + n) / 2);
    auto rate = [&](int mode, int q, int g, int groups, int passes, int lines) {
        const int per_term = max(16 * q, groups * (lines * kavg + 5) / (2 * kavg)) + 3 + 24 / kavg;
        const uint32_t cost = (uint32_t)(per_term * passes * 64 / groups) * 32u + (uint32_t)(32 - g);
        if (cost < best) {
            best = cost;
            best_mode = mode;
            best_q = q;
            best_g = g;
        }
    };
    if (has_q(MASK, lane + 1)) {
        const int q = lane + 1, rows = min(min(m, (31 + n) / n + 1), blk_lines), cols = (min(32, n) * 8 >> 7) + 1;
        rate(kFlat, q, 32, 1, (rs + 32 * q - 1) / (32 * q), q * (rows + cols));
    }
    for (int mode = 0; mode < 3 && !spread; ++mode) {
        const int g = lane + 1, groups = 32 / g, dim = mode == kRow ? m : n;
        if (mode != kFlat && g % dim != 0) continue;
        const int need = mode == kFlat ? (rs + g - 1) / g : ((mode == kRow ? n : m) + g / dim - 1) / (g / dim);
        const uint32_t mask = mode == kFlat ? MASK : MASK & kQShared;
        if (need > q_max(mask)) continue;
        const int q = __ffs(mask >> need) - 1 + need;
        const int rows = min(min(m, (g + n - 1) / n + 1), blk_lines), cols = (min(g, n) * 8 >> 7) + 1;
        rate(mode, q, g, groups, 1,
             mode == kFlat ? q * (rows + cols) : mode == kRow ? min(m, blk_lines) + q : q * min((g - 1) / n + 1, blk_lines) + cols);
    }
    const uint32_t top = __reduce_min_sync(0xffffffffu, best);
    const int win = __ffs(__ballot_sync(0xffffffffu, best == top)) - 1;
    const GroupPlan pl{__shfl_sync(0xffffffffu, best_mode, win), __shfl_sync(0xffffffffu, best_q, win),
                       __shfl_sync(0xffffffffu, best_g, win)};
    // only layouts that are compiled are rated; a block without one would never be
    // taken from the window, so it would go to one that takes every shape
    return has_q(pl.mode == kFlat ? MASK : MASK & kQShared, pl.q) ? pl : GroupPlan{kFlat, 1, 32};
}

// Blocks of shape m x n from `run`, until the next one has another shape or
// none is left.
template <int Q, int MODE>
__device__ __forceinline__ void group_run(const NumericArgs &a, ItemRun &run, int lane, int m, int n, int g) {
    constexpr int NX = MODE == kRow ? 1 : Q, NY = MODE == kCol ? 1 : Q;
    constexpr int TU = Q <= 2 ? 4 : Q <= 9 ? 2 : 1;
    const double *__restrict__ X = static_cast<const double *>(a.x_data);
    const double *__restrict__ Y = static_cast<const double *>(a.y_data);
    const int groups = 32 / g, gi = lane / g, l = lane - gi * g;
    const bool member = gi < groups;
    const unsigned before = (1u << (gi * g & 31)) - 1u;  // lanes of the groups before this one
    const int rs = m * n;
    const int32_t shape = (m << 16) | n;
    // step from slot to slot, in rows and columns
    const int dr = MODE == kRow ? 0 : g / n, dc = MODE == kFlat ? g % n : MODE == kRow ? g / m : 0;
    const int xs_t = a.x_trans ? m : 1, ys_t = a.y_trans ? 1 : n;

    double acc[Q];
    int xo[NX], yo[NY];
    // defined on every path: what may be read before it is written would
    // count as live from the start of the kernel
#pragma unroll
    for (int u = 0; u < Q; ++u) acc[u] = 0.0;
#pragma unroll
    for (int u = 0; u < NX; ++u) xo[u] = 0;
#pragma unroll
    for (int u = 0; u < NY; ++u) yo[u] = 0;
    bool act = false, closed = false;
    int32_t item = 0, p = 0, pe = 0;    // the block and its products left, [p, pe)
    int e0 = 0;                         // first element of the pass (blocks of several passes)
    int tn = -1, t = 0;                 // terms of k of the product at p, and those done
    const double *xp = X, *yp = Y;      // its operands at term t
    // one product ahead: offsets and terms of p + 1; two ahead: indices of p + 2
    int64_t nxo = 0, nyo = 0;
    int ntn = 0;
    int32_t ix2 = 0, iy2 = 0;

    // row and column of the lane's first slot (of the pass)
    int r0 = 0, c0 = 0;
    auto set_first = [&]() {
        const int e = e0 + l;
        r0 = MODE == kRow ? e % m : e / n;
        c0 = MODE == kRow ? e / m : e % n;
    };
    // opaque copies: the slots' rows and columns follow from them in a few
    // instructions and are not worth registers across the product loop
    auto first = [&](int &r, int &c) {
        r = r0;
        c = c0;
        asm volatile("" : "+r"(r), "+r"(c));
    };
    auto next = [&](int &r, int &c) {
        r += dr;
        c += dc;
        if constexpr (MODE == kFlat) {
            if (c >= n) {
                c -= n;
                ++r;
            }
        }
    };
    // operand offsets of every slot for products of `k` terms (slots past the block: element 0)
    auto set_offsets = [&](int k) {
        const int xs_r = a.x_trans ? 1 : k, ys_s = a.y_trans ? k : 1;
        int r, c;
        first(r, c);
        if constexpr (MODE == kRow) xo[0] = r * xs_r;
        if constexpr (MODE == kCol) yo[0] = c * ys_s;
#pragma unroll
        for (int u = 0; u < Q; ++u) {
            const bool in = r < m && c < n;
            if constexpr (MODE != kRow) xo[u] = in ? r * xs_r : 0;
            if constexpr (MODE != kCol) yo[u] = in ? c * ys_s : 0;
            next(r, c);
        }
    };
    auto load_offsets = [&](int32_t ix, int32_t iy) {
        const int32_t rc = a.x_blk_rc[ix];
        nxo = a.x_blk_off[ix];
        nyo = a.y_blk_off[iy];
        ntn = a.x_trans ? rc_rows(rc) : rc_cols(rc);
    };
    // make product p current and fetch ahead
    auto advance = [&]() {
        xp = X + nxo;
        yp = Y + nyo;
        t = 0;
        if (ntn != tn) {
            tn = ntn;
            set_offsets(tn);
        }
        if (pe - p > 1) load_offsets(ix2, iy2);
        if (pe - p > 2) {
            ix2 = a.px[p + 2];
            iy2 = a.py[p + 2];
        }
    };
    // start a pass at product p, whose operands are in nxo, nyo, ntn and the
    // next product's indices in ix2, iy2
    auto begin = [&]() {
#pragma unroll
        for (int u = 0; u < Q; ++u) acc[u] = 0.0;
        tn = -1;
        advance();
    };
    // Without a scale or an old block nothing here runs on the FP64 pipe: groups
    // end one by one, and each instruction would cost a whole warp's (a scale
    // and a comparison made 6 x 6 blocks 28.5 ms instead of 24.9, 6.9e7 products).
    auto store = [&]() {
        double *__restrict__ O = static_cast<double *>(a.out_data) + a.out_blk_off[item];
        const int64_t old = a.has_old ? a.old_off[item] : -1;
        const double *OLD = static_cast<const double *>(a.old_data) + old;
        int r, c;
        first(r, c);
        auto each = [&](auto value) {
#pragma unroll
            for (int u = 0; u < Q; ++u) {
                if (r < m && c < n) O[r * n + c] = value(acc[u], r * n + c);
                next(r, c);
            }
        };
        if (a.unit_alpha && old < 0) each([&](double v, int) { return v; });
        else if (a.unit_alpha) each([&](double v, int e) { return fma(a.beta, OLD[e], v); });
        else if (old < 0) each([&](double v, int) { return a.alpha * v; });
        else each([&](double v, int e) { return fma(a.beta, OLD[e], a.alpha * v); });
    };

    // `N` terms of k at once: the loads of all of them before the first FMA, so
    // that few slots still cover the load latency
    auto terms = [&](auto count) {
        constexpr int N = decltype(count)::value;
        double xv[N][NX], yv[N][NY];
#pragma unroll
        for (int i = 0; i < N; ++i) {
#pragma unroll
            for (int u = 0; u < NX; ++u) xv[i][u] = __ldg(xp + xo[u]);
#pragma unroll
            for (int u = 0; u < NY; ++u) yv[i][u] = __ldg(yp + yo[u]);
            xp += xs_t;
            yp += ys_t;
        }
#pragma unroll
        for (int i = 0; i < N; ++i)
#pragma unroll
            for (int u = 0; u < Q; ++u) acc[u] = fma(xv[i][MODE == kRow ? 0 : u], yv[i][MODE == kCol ? 0 : u], acc[u]);
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
                e0 = 0;
                set_first();
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
#pragma unroll
                    for (int u = 0; u < Q; ++u) acc[u] = 0.0;
                    for (; e0 < rs; e0 += MODE == kFlat ? g * Q : rs) {
                        set_first();
                        store();
                    }
                }
            }
            run.cur += take;
            closed = other != 0u;
            __syncwarp();  // the window may be overwritten
        }
        const int steps = (int)__reduce_min_sync(0xffffffffu, act ? (unsigned)(tn - t) : 0xffffffffu);
        if (steps < 0) break;  // no group has a block
        if (act) {
            int s = 0;
            if constexpr (TU > 1) {
#pragma unroll 1
                for (; s + TU <= steps; s += TU) terms(std::integral_constant<int, TU>{});
            }
#pragma unroll 1
            for (; s < steps; ++s) terms(std::integral_constant<int, 1>{});
            t += steps;
            if (t == tn) {
                if (++p < pe) {
                    advance();
                } else {
                    store();
                    e0 += g * Q;
                    if (MODE == kFlat && e0 < rs) {  // the next elements of a large block
                        p = (int32_t)a.seg_ptr[item];
                        set_first();
                        load_offsets(a.px[p], a.py[p]);
                        if (pe - p > 1) {
                            ix2 = a.px[p + 1];
                            iy2 = a.py[p + 1];
                        }
                        begin();
                    } else {
                        act = false;
                    }
                }
            }
        }
        __syncwarp();
    }
}

template <int BUILD>
__global__ void __launch_bounds__(kGroupThreads, BUILD == kCcSmall ? 8 : BUILD == kCcNarrow ? 6 : 4)
k_numeric_group(NumericArgs a) {
    constexpr uint32_t MASK = q_mask<BUILD>();
    if (a.status && *a.status != 0) return;
    const int lane = threadIdx.x & 31;
    // a few blocks for each warp of the grid (tiny blocks; others are few_blocks then):
    // a warp per block, so that all work
    const bool spread = a.n_items <= 4 * (int64_t)gridDim.x * (kGroupThreads / 32);
    __shared__ Window windows[kGroupThreads / 32];
    ItemRun run{&windows[threadIdx.x >> 5], 0, 0, a.n_items};
    while (items_left(a, run, lane)) {
        const int32_t rc = run.w->shape[run.cur];
        const int m = rc_rows(rc), n = rc_cols(rc);
        const GroupPlan pl = group_plan<MASK>(m, n, spread, lane);
        switch (pl.mode * 32 + pl.q) {
#define BSM_Q_MODE(Q, MODE, MASK_)                                                   \
    case MODE * 32 + Q:                                                              \
        if constexpr (has_q(MASK_, Q)) group_run<Q, MODE>(a, run, lane, m, n, pl.g); \
        break;
#define BSM_Q(Q) BSM_Q_MODE(Q, kFlat, MASK) BSM_Q_MODE(Q, kRow, MASK &kQShared) BSM_Q_MODE(Q, kCol, MASK &kQShared)
            BSM_Q(1) BSM_Q(2) BSM_Q(3) BSM_Q(4) BSM_Q(5) BSM_Q(6) BSM_Q(7) BSM_Q(8)
            BSM_Q(9) BSM_Q(11) BSM_Q(13) BSM_Q(15) BSM_Q(17) BSM_Q(19) BSM_Q(21) BSM_Q(24)
#undef BSM_Q
#undef BSM_Q_MODE
        }
    }
}

template <int BUILD>
cudaError_t launch_build(const NumericArgs &a, cudaStream_t s, int *grid) {
    static std::atomic<int> resident{0};
    return launch_persistent(k_numeric_group<BUILD>, resident, a, s, grid);
}

}  // namespace

cudaError_t launch_numeric_group(const NumericArgs &a, int build, cudaStream_t s, int *grid) {
    if (build == kCcSmall) return launch_build<kCcSmall>(a, s, grid);
    if (build == kCcNarrow) return launch_build<kCcNarrow>(a, s, grid);
    return launch_build<kCcWide>(a, s, grid);
}

uint32_t group_debug_bits(cudaStream_t s) { return read_debug_bits(s); }

}  // namespace bsm
