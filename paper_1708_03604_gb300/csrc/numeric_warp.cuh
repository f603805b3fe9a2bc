// An output block by a warp on the CUDA cores: a lane owns every 32nd element.
#pragma once

#include "bsm_internal.cuh"

namespace bsm {
namespace {

// FP64 data: one chain of FP64 fused multiply-adds per element, ascending product,
// then ascending k.  FP32 data: such a chain in FP32 over flush_every products (one
// for the shapes of a.each_product), the chains' sums added in FP64.  Per element
// the operations of the lane groups (k_group.cu) and the register tiles (k_tile.cu).
template <typename T, int Q>
__device__ __forceinline__ void warp_item(const NumericArgs &a, int64_t q, int lane) {
    const T *__restrict__ X = static_cast<const T *>(a.x_data);
    const T *__restrict__ Y = static_cast<const T *>(a.y_data);
    T *__restrict__ O = static_cast<T *>(a.out_data);
    const int32_t orc = a.out_blk_rc[q];
    const int R = rc_rows(orc), S = rc_cols(orc);
    const int RS = R * S;
    const int64_t out_off = a.out_blk_off[q];
    const int64_t p0 = a.seg_ptr[q], p1 = a.seg_ptr[q + 1];
    const int64_t old = (a.beta != 0.0 && a.old_off) ? a.old_off[q] : -1;
    const T *OLD = static_cast<const T *>(a.old_data);
    const int F = sizeof(T) == 4 && a.flush_every > 0 && !a.each_product.has(R, S) ? a.flush_every : 1;

    for (int e0 = 0; e0 < RS; e0 += 32 * Q) {
        int rr[Q], ss[Q];
        double acc[Q];
        T part[Q];
#pragma unroll
        for (int u = 0; u < Q; ++u) {
            const int e = e0 + lane + 32 * u;
            const bool v = e < RS;
            rr[u] = v ? e / S : 0;
            ss[u] = v ? e % S : 0;
            acc[u] = 0.0;
            part[u] = T(0);
        }
        int since = 0;
        for (int64_t p = p0; p < p1; ++p) {
            const int32_t ix = a.px[p], iy = a.py[p];
            const T *xb = X + a.x_blk_off[ix];
            const T *yb = Y + a.y_blk_off[iy];
            const int32_t xrc = a.x_blk_rc[ix];
            const int Tn = a.x_trans ? rc_rows(xrc) : rc_cols(xrc);
            const int xs_r = a.x_trans ? 1 : Tn, xs_t = a.x_trans ? R : 1;
            const int ys_t = a.y_trans ? 1 : S, ys_s = a.y_trans ? Tn : 1;
            int xo[Q], yo[Q];
#pragma unroll
            for (int u = 0; u < Q; ++u) {
                xo[u] = rr[u] * xs_r;
                yo[u] = ss[u] * ys_s;
            }
            for (int t = 0; t < Tn; ++t) {
#pragma unroll
                for (int u = 0; u < Q; ++u) {
                    const T xv = __ldg(xb + xo[u] + t * xs_t);
                    const T yv = __ldg(yb + t * ys_t + yo[u]);
                    part[u] = fma(xv, yv, part[u]);
                }
            }
            if constexpr (sizeof(T) == 4) {
                if (++since == F) {
                    since = 0;
#pragma unroll
                    for (int u = 0; u < Q; ++u) {
                        acc[u] += (double)part[u];
                        part[u] = T(0);
                    }
                }
            }
        }
#pragma unroll
        for (int u = 0; u < Q; ++u) {
            const int e = e0 + lane + 32 * u;
            if (e < RS) {
                double v = sizeof(T) == 8 ? (double)part[u] : acc[u] + (double)part[u];
                v = a.alpha * v;
                if (old >= 0) v = fma(a.beta, (double)OLD[old + e], v);
                O[out_off + e] = (T)v;
            }
        }
    }
}

// up to 9 elements a lane and pass (24 if WIDE), more passes over the products for larger blocks
template <typename T, bool WIDE>
__device__ __forceinline__ void warp_block(const NumericArgs &a, int64_t q, int lane) {
    const int32_t orc = a.out_blk_rc[q];
    const int need = (rc_rows(orc) * rc_cols(orc) + 31) >> 5;
    if (need <= 1) return warp_item<T, 1>(a, q, lane);
    if (need <= 2) return warp_item<T, 2>(a, q, lane);
    if (need <= 3) return warp_item<T, 3>(a, q, lane);
    if (need <= 4) return warp_item<T, 4>(a, q, lane);
    if (need <= 6) return warp_item<T, 6>(a, q, lane);
    if constexpr (WIDE) {
        if (need <= 8) return warp_item<T, 8>(a, q, lane);
        if (need <= 10) return warp_item<T, 10>(a, q, lane);
        if (need <= 12) return warp_item<T, 12>(a, q, lane);
        if (need <= 14) return warp_item<T, 14>(a, q, lane);
        if (need <= 17) return warp_item<T, 17>(a, q, lane);
        if (need <= 20) return warp_item<T, 20>(a, q, lane);
        return warp_item<T, 24>(a, q, lane);
    } else {
        warp_item<T, 9>(a, q, lane);
    }
}

}  // namespace
}  // namespace bsm
