// Device-side 64-bit RNS arithmetic for sm_103a.
//
// Residues are kept canonical ([0, q)) between kernels. Products by constants
// use Shoup's precomputed quotient (w' = floor(w * 2^64 / q)); products of two
// variable residues and multiply-accumulate chains use Montgomery reduction
// with R = 2^64 (one operand stored pre-multiplied by R, or a second
// reduction by R^2 mod q). All primes are below 2^61, which the lazy
// accumulation bounds below rely on.
#pragma once
#include <cuda_runtime.h>
#include <cstdint>

typedef uint64_t u64;
typedef unsigned int u32;

struct DevPrime {
    u64 q;       // modulus
    u64 qinv;    // q^-1 mod 2^64 (Montgomery)
    u64 r2;      // 2^128 mod q
    u64 one_s;   // floor(2^64 / q): Shoup quotient of 1 (x mod q for any 64-bit x)
    // constants of the NTT's products by twiddles (see TwClass)
    u64 c2;      // classes 0, 1: 2^(S + 32) mod q, below 2^32
    u64 off;     // classes 0, 1: the smallest multiple of q not below the bound of a product
    u64 big;     // class 1: the largest multiple of q up to 2^63
    u32 bsh;     // classes 0, 1: bits(q) - 32
    u32 c;       // classes 0, 1: 2^bits(q) - q
    u32 cls;     // twiddle class
    u32 fold63;  // fold_top brings every value below 2^63 to below 2q
    uint4 tw_ninv;   // N^-1 as a twiddle of the class
    uint4 tw_wninv;  // N^-1 times the inverse transform's last twiddle, likewise
};

// Products x w by the twiddles of the NTT. A twiddle is 16 bytes, in the format of its prime's
// class:
//
// Classes 0 and 1 store w and v = w 2^32 mod q, each split at bit S: (w mod 2^S, w >> S, v mod
// 2^S, v >> S). With x = xh 2^32 + xl the sum xl w + xh v = a0 + a1 2^S is congruent to x w, and
// a1's high word counts the 2^(S+32) in it, which are worth c2 = 2^(S+32) mod q each:
//   r = a0 + (a1 mod 2^32) 2^S + (a1 >> 32) c2.
// That is six 32 x 32 + 64 -> 64 multiply-adds and nothing else, where the 64-bit Shoup product
// (quotient x ws >> 64, then x w - quotient q) takes five, four 32-bit products and the carries
// between them. On GB300 a wide product costs 4.2 issue cycles a warp, a 32-bit product or a shift
// 2, an add 1; butterflies with operands in registers measured 29 cycles a warp against 39 (44
// with a conditional subtraction of Harvey's ranges). r is not reduced below 2q: it lies in
// [0, bound),
//   bound = (a1max >> 32) c2 + 2^(S+32) + 2^(S+33),
// and twiddle_class() accepts a prime only when the sums of a transform stay below 2^64:
//   class 0 (S = 20, primes of at most 51 bits close below a power of two): 16 products and a
//     residue fit in 64 bits, so a forward transform needs no conditional subtraction at all;
//   class 1 (S = 29, up to 60 bits): a product and a value below 2^63 fit.
// Class 2 (any prime below 2^61): (w, floor(w 2^64 / q)), the Shoup product.
constexpr int kTwS0 = 20, kTwS1 = 29;

__device__ __forceinline__ u64 mul_wide(u32 a, u32 b) {
    u64 r;
    asm("mul.wide.u32 %0, %1, %2;" : "=l"(r) : "r"(a), "r"(b));
    return r;
}
__device__ __forceinline__ u64 mad_wide(u32 a, u32 b, u64 c) {
    u64 r;
    asm("mad.wide.u32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
    return r;
}

// x w, lazily reduced (any 64-bit x); qm: class 2 the modulus, else DevPrime::c2
template <int CLS>
__device__ __forceinline__ u64 mul_tw(u64 x, const uint4& w, u64 qm) {
    if constexpr (CLS == 2) {
        const u64 W = (u64)w.y << 32 | w.x, WS = (u64)w.w << 32 | w.z;
        return x * W - __umul64hi(x, WS) * qm;  // in [0, 2q)
    } else {
        constexpr int S = CLS == 0 ? kTwS0 : kTwS1;
        const u32 xl = (u32)x, xh = (u32)(x >> 32);
        const u64 a1 = mad_wide(xh, w.w, mul_wide(xl, w.y));
        const u64 a0 = mad_wide(xh, w.z, mul_wide(xl, w.x));
        return mad_wide((u32)a1, 1u << S, mad_wide((u32)(a1 >> 32), (u32)qm, a0));
    }
}

// any value of a transform to below 2q (classes 0, 1: to below 2^bits(q) plus a little, at most
// 2q): the bits from bits(q) up times c = 2^bits(q) - q
__device__ __forceinline__ u64 fold_top(u64 v, u32 bsh, u32 c) {
    const u32 vh = (u32)(v >> 32);
    const u32 h = vh >> bsh;
    return mad_wide(h, c, (u64)(vh - (h << bsh)) << 32 | (u32)v);
}

__device__ __forceinline__ u64 add_mod(u64 a, u64 b, u64 q) {
    u64 s = a + b;
    return s >= q ? s - q : s;
}
__device__ __forceinline__ u64 sub_mod(u64 a, u64 b, u64 q) { return a >= b ? a - b : a + q - b; }

// x * w mod q for a constant w with Shoup quotient ws; any 64-bit x. Lazily: in [0, 2q).
__device__ __forceinline__ u64 mul_shoup_lazy(u64 x, u64 w, u64 ws, u64 q) { return x * w - __umul64hi(x, ws) * q; }
__device__ __forceinline__ u64 mul_shoup(u64 x, u64 w, u64 ws, u64 q) {
    u64 hi = __umul64hi(x, ws);
    u64 r = x * w - hi * q;
    return r >= q ? r - q : r;
}

// Montgomery reduction of T = hi * 2^64 + lo with hi < q: returns T * 2^-64 mod q in [0, q).
__device__ __forceinline__ u64 redc(u64 hi, u64 lo, u64 q, u64 qinv) {
    u64 m = lo * qinv;
    u64 t = __umul64hi(m, q);
    return hi >= t ? hi - t : hi - t + q;
}

struct Acc128 {
    u64 lo, hi;
};
// acc += x y
__device__ __forceinline__ void mac_full(Acc128& a, u64 x, u64 y) {
    const u32 xl = (u32)x, xh = (u32)(x >> 32), yl = (u32)y, yh = (u32)(y >> 32);
    const u64 p0 = mul_wide(xl, yl), m0 = mad_wide(xh, yl, p0 >> 32), m1 = mad_wide(xl, yh, (u64)(u32)m0);
    const u64 hi = mad_wide(xh, yh, (m0 >> 32) + (m1 >> 32)), lo = m1 << 32 | (u32)p0;
    asm("add.cc.u64 %0, %0, %2;\n\taddc.u64 %1, %1, %3;" : "+l"(a.lo), "+l"(a.hi) : "l"(lo), "l"(hi));
}
// a sum of at most two products of residues to its canonical residue, for a prime of class 0 or 1:
// everything from bit bits(q) up is worth c = 2^bits(q) - q per unit, three times over (no
// quotient, no Montgomery factor: 40 issue cycles a warp against 45 for each of mul_mod's two
// reductions)
__device__ __forceinline__ u64 reduce_sum(const Acc128& a, const DevPrime& P) {
    const u32 w1 = (u32)(a.lo >> 32), w2 = (u32)a.hi, w3 = (u32)(a.hi >> 32), mask = (1u << P.bsh) - 1;
    const u64 p0 = mad_wide(__funnelshift_r(w1, w2, P.bsh), P.c, (u64)(w1 & mask) << 32 | (u32)a.lo);
    const u64 p1 = mad_wide(__funnelshift_r(w2, w3, P.bsh), P.c, p0 >> 32);
    const u64 r = mad_wide((u32)(p1 >> P.bsh), P.c, (u64)((u32)p1 & mask) << 32 | (u32)p0);
    const u64 f = fold_top(r, P.bsh, P.c);
    return min(f, f - P.q);
}

// Products of residues below 2^60 from 30-bit halves: x = xh 2^30 + xl, y = yh 2^30 + yl,
// x y = xl yl + (xl yh + xh yl) 2^30 + xh yh 2^60. Each partial product is below 2^60, so up
// to 8 products sum in three 64-bit words, a1 holding the middle terms (below 2^64), with no
// carries. split30 packs (xl, xh) into the low and high 32-bit words. Residues below 2^61 have
// xh, yh below 2^31, partial products below 2^62 and middle terms below 2^62: up to 4 products.
struct Acc3 {
    u64 a0, a1, a2;
};
__device__ __forceinline__ u64 split30(u64 x) { return (x & 0x3fffffffull) | ((x >> 30) << 32); }
// acc += hi 2^64 + lo, one add-with-carry chain
__device__ __forceinline__ void add128(Acc128& acc, u64 lo, u64 hi) {
    asm("add.cc.u64 %0, %0, %2;\n\taddc.u64 %1, %1, %3;" : "+l"(acc.lo), "+l"(acc.hi) : "l"(lo), "l"(hi));
}
// acc += a0 + a1 2^30 + a2 2^60, then a = 0
__device__ __forceinline__ void flush30(Acc128& acc, Acc3& a) {
    add128(acc, a.a0, 0);
    add128(acc, a.a1 << 30, a.a1 >> 34);
    add128(acc, a.a2 << 60, a.a2 >> 4);
    a.a0 = a.a1 = a.a2 = 0;
}

// Karatsuba form of the same sums, three multiply-adds per product:
//   x y = xl yl + ((xl + xh)(yl + yh) - xl yl - xh yh) 2^30 + xh yh 2^60.
// am = sum (xl + xh)(yl + yh) may wrap modulo 2^64, but the middle term sum (xl yh + xh yl) is
// below 8 * 2 * 2^60 = 2^64 for up to 8 products (residues below 2^61: 4 * 2 * 2^61, up to 4), so
// am - a0 - a2 modulo 2^64 is exact.
// xsum = xl + xh is passed in (it is shared by every product with the same x).
struct AccK {
    u64 a0, am, a2;
};
__device__ __forceinline__ u32 sum30(u64 xs) { return (u32)xs + (u32)(xs >> 32); }
__device__ __forceinline__ void mack(AccK& a, u64 xs, u32 xsum, u64 ys) {
    const u32 xl = (u32)xs, xh = (u32)(xs >> 32), yl = (u32)ys, yh = (u32)(ys >> 32);
    a.a0 += (u64)xl * yl;
    a.am += (u64)xsum * (yl + yh);
    a.a2 += (u64)xh * yh;
}
// acc += the products summed in a, then a = 0
__device__ __forceinline__ void flushk(Acc128& acc, AccK& a) {
    Acc3 t{a.a0, a.am - a.a0 - a.a2, a.a2};
    flush30(acc, t);
    a.a0 = a.am = a.a2 = 0;
}

// a * b mod q for two variable residues: REDC(REDC(a b) * R^2)
__device__ __forceinline__ u64 mul_mod(u64 a, u64 b, const DevPrime& P) {
    u64 t = redc(__umul64hi(a, b), a * b, P.q, P.qinv);
    return redc(__umul64hi(t, P.r2), t * P.r2, P.q, P.qinv);
}

// x * R mod q (Montgomery form)
__device__ __forceinline__ u64 to_mont(u64 x, const DevPrime& P) {
    return redc(__umul64hi(x, P.r2), x * P.r2, P.q, P.qinv);
}

// Automorphism sigma_g in evaluation form: position k holds the value at
// psi^(2 brev(k) + 1); sigma_g(a) at that point is a at psi^((2 brev(k)+1) g).
__device__ __forceinline__ u32 galois_src_index(u32 k, u32 g, int logN) {
    u32 e = 2u * (__brev(k) >> (32 - logN)) + 1u;
    u32 M = 2u << logN;
    u32 e2 = (u32)(((u64)e * g) & (M - 1));
    return __brev((e2 - 1u) >> 1) >> (32 - logN);
}
