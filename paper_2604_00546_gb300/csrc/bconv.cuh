// Device side of the fast base conversions (see BconvTarget).
#pragma once
#include "ckks_kernels.h"

// (sum_i y_i [B/b_i]_t + add) mod t, canonical; add up to the add_max the target was made for
template <int NS, int W>
__device__ __forceinline__ void bconv(const BconvTarget& T, const u64 (&y)[NS][W], const u64 (&add)[W],
                                      u64 (&out)[W]) {
    if (T.mode == 0) {
        u64 a0[W], a1[W];
#pragma unroll
        for (int w = 0; w < W; ++w) {
            a0[w] = add[w];
            a1[w] = 0;
        }
#pragma unroll
        for (int i = 0; i < NS; ++i) {
            const uint4 h = T.hat[i];
#pragma unroll
            for (int w = 0; w < W; ++w) {
                const u32 xl = (u32)y[i][w], xh = (u32)(y[i][w] >> 32);
                a1[w] = mad_wide(xh, h.w, mad_wide(xl, h.y, a1[w]));
                a0[w] = mad_wide(xh, h.z, mad_wide(xl, h.x, a0[w]));
            }
        }
#pragma unroll
        for (int w = 0; w < W; ++w) {
            const u64 r = mad_wide((u32)a1[w], T.mul, mad_wide((u32)(a1[w] >> 32), T.c2, a0[w]));
            const u64 f = fold_top(r, T.bsh, T.c);
            out[w] = min(f, f - T.q);
        }
    } else if (T.mode == 1) {
        u64 sum[W];
#pragma unroll
        for (int w = 0; w < W; ++w) sum[w] = add[w];
#pragma unroll
        for (int i = 0; i < NS; i += 2) {
            const uint4 h = T.hat[i], g = i + 1 < NS ? T.hat[i + 1 < NS ? i + 1 : i] : make_uint4(0, 0, 0, 0);
#pragma unroll
            for (int w = 0; w < W; ++w) {
                const u32 xl = (u32)y[i][w], xh = (u32)(y[i][w] >> 32);
                u64 a1 = mad_wide(xh, h.w, mul_wide(xl, h.y));
                u64 a0 = mad_wide(xh, h.z, mul_wide(xl, h.x));
                if (i + 1 < NS) {
                    const u64 z = y[i + 1 < NS ? i + 1 : i][w];
                    a1 = mad_wide((u32)(z >> 32), g.w, mad_wide((u32)z, g.y, a1));
                    a0 = mad_wide((u32)(z >> 32), g.z, mad_wide((u32)z, g.x, a0));
                }
                sum[w] += fold_top(mad_wide((u32)a1, T.mul, mad_wide((u32)(a1 >> 32), T.c2, a0)), T.bsh, T.c);
            }
        }
#pragma unroll
        for (int w = 0; w < W; ++w) {
            const u64 f = fold_top(sum[w], T.bsh, T.c);
            out[w] = min(f, f - T.q);
        }
    } else {
        for (int w = 0; w < W; ++w) {
            AccK a{0, 0, 0};
            Acc128 acc{0, 0};
#pragma unroll
            for (int i = 0; i < NS; ++i) {
                const u64 x = split30(y[i][w]);
                mack(a, x, sum30(x), (u64)T.hat[i].y << 32 | T.hat[i].x);
                if (i % 4 == 3) flushk(acc, a);  // operands below 2^61
            }
            flushk(acc, a);
            const u64 r = redc(mul_shoup(acc.hi, 1, T.one_s, T.q), acc.lo, T.q, T.qinv);
            out[w] = add_mod(r, mul_shoup(add[w], 1, T.one_s, T.q), T.q);
        }
    }
}
