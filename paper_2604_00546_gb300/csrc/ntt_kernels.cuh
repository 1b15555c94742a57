// Batched negacyclic NTT / inverse NTT over 64-bit primes.
//
// Forward: Cooley-Tukey with twiddles psi^brev(k) (natural-order input,
// evaluation-order output: position k = A(psi^(2 brev(k)+1))). Inverse:
// Gentleman-Sande with psi^-brev(k), then N^-1.
//
// The log N stages are split in two passes over an R x C view of the
// polynomial (N = R C): the first log R stages only couple elements of one
// column (stride C), the remaining log C stages only couple elements of one
// row (contiguous). Each pass loads its tile once and writes it once. Inside a
// pass every thread keeps 2^RB elements in registers (RB = 3 or 4) and runs up
// to RB radix-2 stages on them; the elements are re-distributed through shared
// memory between these phases, so a 256-point sub-transform costs 2 exchanges
// with 8 elements a thread and 1 with 16. Index arithmetic is shifts and masks only.
//
// The passes are bound by the issue of integer multiplications, so the butterfly's product
// is the cheapest one its prime allows (TwClass in dev_arith.cuh) and residues stay lazily
// reduced between stages:
//   class 0  forward: sums only grow, 16 stages stay below 2^64; inverse: the sums of a phase
//            (at most 4 stages) grow sixteenfold and are folded at its end;
//   class 1  one conditional subtraction of `big` (about 2^63) per butterfly;
//   class 2  Harvey's ranges: forward [0, 4q), inverse [0, 2q).
// The last pass returns canonical residues.
// Twiddle of the butterfly pairing x and x + 2^b, in either direction:
// tw[(M + J) >> (b + 1)] where J is the global index of x and M = R for the
// column pass, N for the row pass.
#pragma once
#include <cooperative_groups.h>
#include <type_traits>

#include "ckks_kernels.h"

namespace ntt_kernels {


// polynomial e of an extension map: digit and position
__device__ __forceinline__ void ext_at(const ExtMap& m, int e, int* digit, int* pos) {
    int d = 0;
    while (d + 1 < m.ndig && e >= m.npos - m.ns[d]) e -= m.npos - m.ns[d++];
    *digit = d;
    *pos = e < m.lo[d] ? e : e + m.ns[d];
}

__device__ __forceinline__ u64* poly_at(const PolyBatch& b, int p, int N, int* prime) {
    if (b.split && p >= b.split) {
        const int q = p - b.split;
        *prime = b.pm2.idx[q % b.pm2.period];
        return b.base2 + (long long)(q / b.inner2) * b.outer2 + (long long)(q % b.inner2) * N;
    }
    if (b.ext.n) {
        int d, pos;
        ext_at(b.ext, p % b.ext.n, &d, &pos);
        *prime = pos < b.ext.limbs ? pos : b.ext.pbase + pos - b.ext.limbs;
        return b.base + (long long)(p / b.ext.n) * b.outer + (long long)(d * b.ext.npos + pos) * N;
    }
    *prime = b.pm.idx[p % b.pm.period];
    return b.base + (long long)(p / b.inner) * b.outer + (long long)(p % b.inner) * N;
}

template <int W>
__device__ __forceinline__ void ld_vec(u64 (&r)[W], const u64* p) {
    if constexpr (W == 2) {
        const ulonglong2 t = *reinterpret_cast<const ulonglong2*>(p);
        r[0] = t.x;
        r[1] = t.y;
    } else {
        r[0] = *p;
    }
}
template <int W>
__device__ __forceinline__ void st_vec(u64* p, const u64 (&r)[W]) {
    if constexpr (W == 2) *reinterpret_cast<ulonglong2*>(p) = make_ulonglong2(r[0], r[1]);
    else *p = r[0];
}
// W consecutive values from index k of second-segment poly p (PolyBatch::rs)
template <int W>
__device__ __forceinline__ void rs_load(u64 (&v)[W], const PolyBatch& b, int p, int k, int N, u64 q) {
    const int jt = p - b.split, l = b.rs.l;
    const u64 w = __ldg(b.rs.pinv + l), ws = __ldg(b.rs.pinv_s + l);
    u64 dd[W] = {};
    ld_vec(v, b.rs.acc + ((long long)jt * b.rs.npos + l) * N + k);
    if (b.rs.d) ld_vec(dd, b.rs.d + (((long long)(jt >> 1) * 3 + (jt & 1)) * (l + 1) + l) * N + k);
#pragma unroll
    for (int i = 0; i < W; ++i) v[i] = add_mod(mul_shoup(v[i], w, ws, q), dd[i], q);
}
__device__ __forceinline__ bool rs_poly(const PolyBatch& b, int p) { return b.rs.acc && p >= b.split; }

// where the first pass reads poly p: its source when the batch has one, else its place
__device__ __forceinline__ const u64* poly_in(const PolyBatch& b, int p, int N, const u64* x) {
    return b.src ? b.src + (long long)(p / b.inner) * b.src_outer + (long long)(p % b.inner) * N : x;
}

// poly p's own final constants of an inverse transform, if its batch has them
__device__ __forceinline__ const uint4* poly_post(const PolyBatch& b, int p) {
    return b.post && !(b.split && p >= b.split) ? b.post + 2 * (p % b.pm.period) : nullptr;
}

// element index of register e of thread tau in a phase whose RB bits start at LO
template <int RB, int LO>
__device__ __forceinline__ int phase_x(int tau, int e) {
    return ((tau >> LO) << (LO + RB)) | (e << LO) | (tau & ((1 << LO) - 1));
}

// Phases of a 2^LOG-point pass with RB bits of the element index in registers: phase PH holds
// bits [LO, LO + RB) and runs the stages on bits [BFROM, BTO). Forward phases take bits in
// descending order, inverse ones ascending; with RB = 4 (two phases) the inverse ones mirror the
// forward ones, so both directions share the order of the row pass's twiddles.
template <int RB, int LOG, bool INV, int PH>
struct PhaseInfo {
    static constexpr int P = (LOG + RB - 1) / RB;
    static constexpr int DOWN = LOG - RB * (PH + 1) > 0 ? LOG - RB * (PH + 1) : 0;
    static constexpr int UP = RB == 4 ? (PH == 0 ? 0 : LOG - 4) : (RB * PH < LOG - RB ? RB * PH : LOG - RB);
    static constexpr int LO = INV ? UP : DOWN;
    static constexpr int BFROM = !INV ? LO : RB == 4 ? LO : RB * PH;
    static constexpr int BTO = !INV ? LOG - RB * PH
                               : RB == 4 ? (PH == 0 ? LOG - 4 : LOG)
                                         : (RB * PH + RB < LOG ? RB * PH + RB : LOG);
    static_assert(RB != 4 || P == 2, "radix-16 passes have two phases");
};
template <int RB, int LOG, bool INV>
struct LastLo {
    static constexpr int v = PhaseInfo<RB, LOG, INV, PhaseInfo<RB, LOG, INV, 0>::P - 1>::LO;
};

// Epilogues of the forward row pass (the last pass of a forward transform): instead of
// storing the transformed values of poly p in place, the fused epilogue finishes the operation
// the transform belonged to, on W = 1 or 2 consecutive indices from k (16-byte accesses for 2). It
// has two parts: load() fetches the operands, put() computes and stores. The outputs may alias the
// operands, so the compiler cannot move a load above the store before it; a thread loads the
// operands of four places and then stores four (one by one, their memory latencies added up: the
// row pass of EpiRelinRescale took 141 us for 192 polynomials, 74 more than without an epilogue).
// Values arrive below 2q; every epilogue ends them in a product by a constant, and Shoup's product
// is exact for any 64-bit operand, so differences are lifted by 2q instead of reduced.
template <int W>
struct EpiOps {
    u64 a[W], b[W], c[W];
};
// a polynomial's constants in its epilogue (factors m, n with Shoup quotients, a term t), read when
// the pass starts
struct EpiK {
    u64 m, ms, n, ns, t;
};
struct EpiStore {
    __device__ __forceinline__ EpiK consts(int) const { return EpiK{}; }
};

template <class E>
constexpr bool in_place = std::is_same<E, EpiStore>::value;


// r += a term below q, mod q
template <int W>
__device__ __forceinline__ void add_vec(u64 (&r)[W], const u64 (&a)[W], u64 q) {
#pragma unroll
    for (int w = 0; w < W; ++w) r[w] = add_mod(r[w], a[w], q);
}

// Template diagonals: Montgomery form as 30-bit halves into the database's tiles.
struct EpiDiag {
    u64* diags;
    int d0, ell, nl, N;
    __device__ __forceinline__ EpiK consts(int) const { return EpiK{}; }
    template <int W>
    __device__ __forceinline__ void load(EpiOps<W>&, int, int) const {}
    template <int W>
    __device__ __forceinline__ void put(const EpiK&, const EpiOps<W>&, int p, int k, const u64 (&v)[W],
                                        const DevPrime& P) const {
        u64 o[W];
#pragma unroll
        for (int w = 0; w < W; ++w) o[w] = split30(to_mont(v[w], P));
        st_vec(diags + diag_word(p % nl, k, d0 + p / nl, ell, N), o);
    }
};

// ModDown combine: poly p = (job, component t, limb i) of the P -> Q conversions; out =
// (acc_Q - v) P^-1 (+ sigma_g(c0) for rotations, + the ct addend for relinearisation; a
// rotation may add a ciphertext as well, as in x + Rot(x)).
struct EpiModDown {
    MDJobs jobs;
    int npos, level, logN;
    const u64* pinv;
    const u64* pinv_s;
    __device__ __forceinline__ EpiK consts(int p) const {
        const int i = p % (level + 1);
        return EpiK{pinv[i], pinv_s[i], 0, 0, 0};
    }
    template <int W>
    __device__ __forceinline__ void load(EpiOps<W>& o, int p, int k) const {
        const int L1 = level + 1, N = 1 << logN;
        const int r = p % (2 * L1), t = r / L1, i = r % L1;
        const MDJob& J = jobs.j[p / (2 * L1)];
        ld_vec(o.a, J.acc + ((long long)t * npos + i) * N + k);
        if ((J.mode & 1) && t == 0) {  // modes 1, 3
#pragma unroll
            for (int w = 0; w < W; ++w)
                o.b[w] = J.add[(long long)i * N + galois_src_index((u32)(k + w), J.galois, logN)];
        }
        if (J.mode & 2) ld_vec(o.c, (J.mode == 3 ? J.add2 : J.add) + ((long long)t * J.add_cap + i) * N + k);
    }
    template <int W>
    __device__ __forceinline__ void put(const EpiK& K, const EpiOps<W>& x, int p, int k, const u64 (&v)[W],
                                        const DevPrime& P) const {
        const u64 q = P.q;
        const int L1 = level + 1, N = 1 << logN;
        const int r = p % (2 * L1), t = r / L1, i = r % L1;
        const MDJob& J = jobs.j[p / (2 * L1)];
        u64 o[W];
#pragma unroll
        for (int w = 0; w < W; ++w) o[w] = mul_shoup(x.a[w] + 2 * q - v[w], K.m, K.ms, q);
        if ((J.mode & 1) && t == 0) add_vec(o, x.b, q);
        if (J.mode & 2) add_vec(o, x.c, q);
        st_vec(J.out + ((long long)t * J.out_cap + i) * N + k, o);
    }
};

// Rescale combine: poly p = (ct component bt, limb i) of the lifted last limb;
// out = (x - v) q_l^-1, then (mode 1) + the matching component of an addend ct, or
// (mode 2) doubled with cres_i subtracted from component 0 (2 T^2 - 1 of the Chebyshev powers).
struct EpiRescale {
    const u64* x;
    u64* out;
    const RescaleTab* tab;
    int x_cap, out_cap, l, N;
    int mode;
    const u64* add;     // mode 1: ct b at add + b add_bs, component t at + t add_cap N
    int add_cap;
    long long add_bs;
    const u64* cres;    // mode 2: [l] constants
    __device__ __forceinline__ EpiK consts(int p) const {
        const int bt = p / l, i = p % l;
        return EpiK{tab->qlinv[i], tab->qlinv_s[i], 0, 0, mode == 2 && (bt & 1) == 0 ? cres[i] : 0};
    }
    template <int W>
    __device__ __forceinline__ void load(EpiOps<W>& o, int p, int k) const {
        const int bt = p / l, i = p % l;
        ld_vec(o.a, x + ((long long)bt * x_cap + i) * N + k);
        if (mode == 1) ld_vec(o.b, add + (long long)(bt >> 1) * add_bs + ((long long)(bt & 1) * add_cap + i) * N + k);
    }
    template <int W>
    __device__ __forceinline__ void put(const EpiK& K, const EpiOps<W>& o, int p, int k, const u64 (&v)[W],
                                        const DevPrime& P) const {
        const u64 q = P.q;
        const int bt = p / l, i = p % l;
        u64 r[W];
#pragma unroll
        for (int w = 0; w < W; ++w) r[w] = mul_shoup(o.a[w] + 2 * q - v[w], K.m, K.ms, q);
        if (mode == 1) {
            add_vec(r, o.b, q);
        } else if (mode == 2) {
#pragma unroll
            for (int w = 0; w < W; ++w) {
                r[w] = sub_mod(add_mod(r[w], r[w], q), K.t, q);
            }
        }
        st_vec(out + ((long long)bt * out_cap + i) * N + k, r);
    }
};

// Rescale of the Chebyshev leaves Rescale(T1 cb_j + ca_j) without the leaves in memory: poly
// p = ((b nl + j) 2 + t) l + i of the lifted last limbs; the leaf's limb i,
// x_i cb_{j,i} (+ ca_{j,i} on component 0), is formed from T1 (query b at x + b x_bs) with the
// same operations as the leaf kernel that stores it, then out = (leaf_i - v) q_l^-1, leaf (b, j)
// at out + (b nl + j) 2 out_cap N. Bit for bit the leaves stored, then rescaled.
struct EpiLeafRescale {
    const u64* x;
    long long x_bs;
    int x_cap;
    const u64* cb;      // [nl][L1] residues of round(c1 Delta)
    const u64* cb_s;    // their Shoup quotients
    const u64* ca;      // [nl][L1] residues of round(c0 Delta) Delta
    int nl, L1;
    u64* out;
    int out_cap;
    const RescaleTab* tab;
    int l, N;
    __device__ __forceinline__ EpiK consts(int p) const {
        const int bjt = p / l, i = p % l, j = (bjt >> 1) % nl, e = j * L1 + i;
        return EpiK{cb[e], cb_s[e], tab->qlinv[i], tab->qlinv_s[i], (bjt & 1) == 0 ? ca[e] : 0};
    }
    template <int W>
    __device__ __forceinline__ void load(EpiOps<W>& o, int p, int k) const {
        const int bjt = p / l, i = p % l, t = bjt & 1, b = (bjt >> 1) / nl;
        ld_vec(o.a, x + (long long)b * x_bs + ((long long)t * x_cap + i) * N + k);
    }
    template <int W>
    __device__ __forceinline__ void put(const EpiK& K, const EpiOps<W>& o, int p, int k, const u64 (&v)[W],
                                        const DevPrime& P) const {
        const u64 q = P.q;
        const int bjt = p / l, i = p % l;
        const u64 lift = 2 * q + K.t;
        u64 r[W];
#pragma unroll
        for (int w = 0; w < W; ++w) {
            const u64 a = mul_shoup_lazy(o.a[w], K.m, K.ms, q);  // the sum is below 5q
            r[w] = mul_shoup(a + lift - v[w], K.n, K.ns, q);
        }
        st_vec(out + ((long long)bjt * out_cap + i) * N + k, r);
    }
};

// Relinearisation ModDown fused with the rescale after it (the product of two ciphertexts at
// level l, relinearised, then divided by q_l): poly p = (job j, component t, limb i < l) of
// y = conv P^-1 + lift, where conv is the ModDown's P -> Q conversion and lift the centered last
// limb of the ModDown's output. out = (acc_i P^-1 + d_i - v) q_l^-1 with acc the job's key-switch
// inner product [2][npos][N] and d its tensor product [3][l+1][N] (d0, d1 the addend; null: no
// addend, a plain ModDown then rescale); then the modes of EpiRescale. Each step is exact modular
// arithmetic and the NTT is linear, so this equals ModDown, the addition of (d0, d1) and the
// rescale one after the other, bit for bit.
struct EpiRelinRescale {
    const u64* acc;
    const u64* d;
    u64* out;          // job j at out + j out_bs, component t at + t out_cap N
    const RescaleTab* tab;
    const u64* pinv;
    const u64* pinv_s;
    int npos, l, N, out_cap, mode;
    long long out_bs;
    const u64* add;    // mode 1: job j's addend at add + j add_bs, component t at + t add_cap N
    int add_cap;
    long long add_bs;
    const u64* cres;   // mode 2: [l] constants
    __device__ __forceinline__ EpiK consts(int p) const {
        const int jt = p / l, i = p % l;
        return EpiK{pinv[i], pinv_s[i], tab->qlinv[i], tab->qlinv_s[i], mode == 2 && (jt & 1) == 0 ? cres[i] : 0};
    }
    template <int W>
    __device__ __forceinline__ void load(EpiOps<W>& o, int p, int k) const {
        const int jt = p / l, i = p % l, j = jt >> 1, t = jt & 1;
        ld_vec(o.a, acc + ((long long)jt * npos + i) * N + k);
        if (d) ld_vec(o.b, d + (((long long)j * 3 + t) * (l + 1) + i) * N + k);
        if (mode == 1) ld_vec(o.c, add + (long long)j * add_bs + ((long long)t * add_cap + i) * N + k);
    }
    template <int W>
    __device__ __forceinline__ void put(const EpiK& K, const EpiOps<W>& o, int p, int k, const u64 (&v)[W],
                                        const DevPrime& P) const {
        const u64 q = P.q;
        const int jt = p / l, i = p % l, j = jt >> 1, t = jt & 1;
        u64 r[W];
#pragma unroll
        for (int w = 0; w < W; ++w) {
            u64 m = mul_shoup_lazy(o.a[w], K.m, K.ms, q) + 2 * q - v[w];  // below 4q
            if (d) m += o.b[w];
            r[w] = mul_shoup(m, K.n, K.ns, q);
        }
        if (mode == 1) {
            add_vec(r, o.c, q);
        } else if (mode == 2) {
#pragma unroll
            for (int w = 0; w < W; ++w) {
                r[w] = sub_mod(add_mod(r[w], r[w], q), K.t, q);
            }
        }
        st_vec(out + (long long)j * out_bs + ((long long)t * out_cap + i) * N + k, r);
    }
};

// Constants of a pass and where its twiddles lie. SRC 0: staged in shared memory, natural
// order; 1: the table itself, natural order; 2: a row's twiddles in the order of row_tw_index.
template <int CLS, int SRC, int LOG>
struct Ctx {
    int Jbase, M;    // global index of the tile's element 0; M = R (column pass) or N (row pass)
    const uint4* tw;
    u64 q, qm, off, big;
    u32 bsh, c;
    __device__ __forceinline__ Ctx(int jb, int m, const uint4* t, const DevPrime& P)
        : Jbase(jb), M(m), tw(t), q(P.q), qm(CLS == 2 ? P.q : P.c2), off(P.off), big(P.big), bsh(P.bsh), c(P.c) {}
    template <int RB, int LO, int B>
    __device__ __forceinline__ void load(uint4* w, int tau) const {
        constexpr int lb = B - LO, NT = (1 << (RB - 1)) >> lb;
        const int base = (M + Jbase + ((tau >> LO) << (LO + RB))) >> (B + 1);
#pragma unroll
        for (int u = 0; u < NT; ++u) {
            if constexpr (SRC == 0) w[u] = tw[base + u];
            else if constexpr (SRC == 1) w[u] = __ldg(tw + base + u);
            else w[u] = __ldg(tw + row_tw_index(LOG, LO != 0, lb, u, tau));
        }
    }

};

// What a pass that ends in epilogue E keeps of v: canonical residues, or for the epilogues
// values below 2q. C2: the prime is of class 2 (classes 0 and 1 end alike).
template <class E, bool C2>
__device__ __forceinline__ u64 finish(u64 v, const DevPrime& P) {
    if constexpr (std::is_same<E, EpiDiag>::value) return v;  // to_mont takes any value
    const u64 f = C2 ? min(v, v - 2 * P.q) : fold_top(v, P.bsh, P.c);
    return std::is_same<E, EpiStore>::value ? min(f, f - P.q) : f;
}

// One radix-2 stage on bit B of the registers of a phase with base bit LO. The butterfly of
// registers e and e + 2^lb (lb = B - LO) takes twiddle (M + J + x) >> (B + 1), x its element
// index: M + J and the thread's bits of x above LO + RB are multiples of 2^(B+1), and x's bits
// below B + 1 are e's bits up to lb and the thread's bits below LO, so the twiddle is
// base + (e >> (lb + 1)): the stage needs 2^(RB-1) >> lb distinct twiddles, loaded before its
// butterflies run. T: stages of this phase run before this one (inverse, class 0: operands are
// below off 2^T).
template <bool INV, int CLS, int RB, int LO, int B, int T, class C>
__device__ __forceinline__ void stage(u64 (&v)[1 << RB], int tau, const C& c) {
    constexpr int lb = B - LO;
    uint4 w[(1 << (RB - 1)) >> lb];
    c.template load<RB, LO, B>(w, tau);
#pragma unroll
    for (int e = 0; e < (1 << RB); ++e) {
        if (e & (1 << lb)) continue;
        const int e1 = e | (1 << lb);
        const uint4& t = w[e >> (lb + 1)];
        if constexpr (!INV) {
            u64 X = v[e];
            if constexpr (CLS == 1) X = min(X, X - c.big);  // X - big wraps when X is below
            if constexpr (CLS == 2) X = min(X, X - 2 * c.q);
            const u64 Tw = mul_tw<CLS>(v[e1], t, c.qm);
            v[e] = X + Tw;
            v[e1] = X + (CLS == 2 ? 2 * c.q : c.off) - Tw;
        } else {
            const u64 X = v[e], Y = v[e1];
            const u64 lift = CLS == 0 ? c.off << T : CLS == 1 ? c.big : 2 * c.q;
            u64 S = X + Y;
            if constexpr (CLS != 0) S = min(S, S - lift);
            v[e] = S;
            v[e1] = mul_tw<CLS>(X - Y + lift, t, c.qm);
        }
    }
}

template <bool INV, int CLS, int RB, int LO, int BFROM, int BTO, int K, class C>
__device__ __forceinline__ void stages(u64 (&v)[1 << RB], int tau, const C& c) {
    // forward: bits BTO-1 down to BFROM; inverse: BFROM up to BTO-1
    if constexpr (K < BTO - BFROM) {
        constexpr int B = INV ? BFROM + K : BTO - 1 - K;
        stage<INV, CLS, RB, LO, B, K>(v, tau, c);
        stages<INV, CLS, RB, LO, BFROM, BTO, K + 1>(v, tau, c);
    }
}

// The phases of a pass, PH .. P - 1, exchanging through ex between them. An inverse column pass
// ends with its last stage (twiddle 1 of the table) and the product by N^-1 in one: the sums are
// multiplied by N^-1, the differences by N^-1 times the twiddle (FIN), or by the batch's own
// constants in their place (post).
template <int CLS, int RB, int LOG, bool INV, bool FIN, int PH, class Ex, class C>
__device__ __forceinline__ void phases(u64 (&v)[1 << RB], int tau, const C& c, Ex& ex, const DevPrime& P,
                                       const uint4* post = nullptr) {
    using I = PhaseInfo<RB, LOG, INV, PH>;
    constexpr bool last = PH == I::P - 1;
    if constexpr (PH > 0) {
        using Prev = PhaseInfo<RB, LOG, INV, PH - 1>;
        ex.template exchange<RB, Prev::LO, I::LO>(v, tau);
    }
    constexpr int BTO = I::BTO - (FIN && last ? 1 : 0);
    stages<INV, CLS, RB, I::LO, I::BFROM, BTO, 0>(v, tau, c);
    if constexpr (FIN && last) {
        constexpr int lb = LOG - 1 - I::LO, T = BTO - I::BFROM;
        const uint4 wn = post ? __ldg(post) : P.tw_ninv, ww = post ? __ldg(post + 1) : P.tw_wninv;
        const u64 lift = CLS == 0 ? c.off << T : CLS == 1 ? c.big : 2 * c.q;
#pragma unroll
        for (int e = 0; e < (1 << RB); ++e) {
            if (e & (1 << lb)) continue;
            const int e1 = e | (1 << lb);
            const u64 X = v[e], Y = v[e1];
            v[e] = mul_tw<CLS>(X + Y, wn, c.qm);
            v[e1] = mul_tw<CLS>(X - Y + lift, ww, c.qm);
        }
    } else if constexpr (INV && CLS == 0) {
        constexpr int lb = BTO - 1 - I::LO;  // the sums of the phase's last stage
#pragma unroll
        for (int e = 0; e < (1 << RB); ++e)
            if (!(e & (1 << lb))) v[e] = fold_top(v[e], c.bsh, c.c);
    }
    if constexpr (!last) phases<CLS, RB, LOG, INV, FIN, PH + 1>(v, tau, c, ex, P, post);
}

// exchange through shared memory, column layout s[x'][KTC]. With 4 columns x' = x ^ x3 ^
// (x4 << 1), with 8 columns x' = x ^ x3 (x4 when 16 elements are in registers): the rows a
// half-warp touches then fall on distinct bank groups in every phase layout. Wider tiles need no
// swizzle: a half-warp is one row.
template <int RB, int KTC>
__device__ __forceinline__ int col_row(int x) {
    if constexpr (KTC >= 16) return x;
    else if constexpr (RB == 4) return x ^ ((x >> 4) & 1);
    else return KTC == 4 ? x ^ ((x >> 3) & 1) ^ (((x >> 4) & 1) << 1) : x ^ ((x >> 3) & 1);
}

template <int KTC>
struct ColEx {
    u64* s;
    int col;
    template <int RB, int LA, int LB>
    __device__ __forceinline__ void exchange(u64 (&v)[1 << RB], int tau) {
#pragma unroll
        for (int e = 0; e < (1 << RB); ++e) s[col_row<RB, KTC>(phase_x<RB, LA>(tau, e)) * KTC + col] = v[e];
        __syncthreads();
#pragma unroll
        for (int e = 0; e < (1 << RB); ++e) v[e] = s[col_row<RB, KTC>(phase_x<RB, LB>(tau, e)) * KTC + col];
        if constexpr (RB == 3) __syncthreads();  // another exchange follows
    }
};

// Shared-memory word of element x of a row: the low 4 bits are XORed with bits 4..6
// (x4 -> bit 0, x5 -> bit 2, x6 -> bits 1 and 3). For 256-point rows this keeps every
// half-warp access of the forward (bits from 5, 2, 0) and inverse (0, 3, 5) phase layouts
// on 16 distinct 8-byte bank pairs.
__device__ __forceinline__ int row_swz(int x) {
    return x ^ ((x >> 4) & 1) ^ (((x >> 5) & 1) << 2) ^ (((x >> 6) & 1) * 10);
}

// exchange through shared memory, one row of 8 elements a thread
struct RowEx {
    u64* s;
    template <int RB, int LA, int LB>
    __device__ __forceinline__ void exchange(u64 (&v)[1 << RB], int tau) {
#pragma unroll
        for (int e = 0; e < (1 << RB); ++e) s[row_swz(phase_x<RB, LA>(tau, e))] = v[e];
        __syncthreads();
#pragma unroll
        for (int e = 0; e < (1 << RB); ++e) v[e] = s[row_swz(phase_x<RB, LB>(tau, e))];
        __syncthreads();
    }
};

// exchange through shared memory, one row of 16 elements a thread. A row's 2^LOG / 16 threads
// are 8 or 16 lanes of one warp, so the exchange needs no block barrier. Word x of a row lies at
// x ^ ((x >> 4) & 15): a half-warp then touches 16 distinct 8-byte bank pairs both when it
// stores elements e << LO | tau and when it loads tau << 4 | e; with 128-point rows (two rows a
// half-warp) odd rows flip bit 3 as well.
template <int LOG>
struct RowEx16 {
    u64* s;
    int odd;
    __device__ __forceinline__ int at(int x) const { return x ^ ((x >> 4) & 15) ^ (LOG == 7 ? odd << 3 : 0); }
    template <int RB, int LA, int LB>
    __device__ __forceinline__ void exchange(u64 (&v)[1 << RB], int tau) {
#pragma unroll
        for (int e = 0; e < (1 << RB); ++e) s[at(phase_x<RB, LA>(tau, e))] = v[e];
        __syncwarp();
#pragma unroll
        for (int e = 0; e < (1 << RB); ++e) v[e] = s[at(phase_x<RB, LB>(tau, e))];
        __syncwarp();
    }
};

// The twiddle class of prime pi, from the launch's parameters: the branch on it waits for no load.
__device__ __forceinline__ int prime_class(const RingDev& R, int pi) {
    return (int)(R.cls1 >> pi & 1) + 2 * (int)(R.cls2 >> pi & 1);
}

// column pass: one CTA = KTC columns x S rows; thread (tau, col) with col = threadIdx % KTC. The
// loads of the elements, the twiddles and the prime's constants are all issued before the first
// use of any of them: a small batch runs one or two CTAs an SM and waits for every dependent load.
template <int RB, int LOG, bool INV, int KTC, int CLS>
__device__ __forceinline__ void ntt_col_body(u64 (&v)[1 << RB], const DevPrime& P, const uint4* post, u64* sm) {
    constexpr int S = 1 << LOG;
    const int col = threadIdx.x & (KTC - 1), tau = threadIdx.x / KTC;
    const Ctx<CLS, 0, LOG> c(0, S, reinterpret_cast<const uint4*>(sm + S * KTC), P);
    ColEx<KTC> ex{sm, col};
    phases<CLS, RB, LOG, INV, INV, 0>(v, tau, c, ex, P, post);
    if constexpr (INV && CLS == 2) {
#pragma unroll
        for (int e = 0; e < (1 << RB); ++e) v[e] = finish<EpiStore, true>(v[e], P);
    }
}

template <int RB, int LOG, bool INV, int KTC, bool C2>
__device__ __forceinline__ void ntt_col(const RingDev& R, const PolyBatch& b, u64* sm) {
    constexpr int S = 1 << LOG, T = KTC * (S >> RB);
    const int p = blockIdx.y, N = R.N, C = N >> LOG;
    int pi;
    u64* x = poly_at(b, p, N, &pi);
    const uint4* tw = (INV ? R.itw : R.tw) + (size_t)pi * N;
    const u64* xin = INV ? x : poly_in(b, p, N, x);  // the column pass is the forward transform's first
    const int col = threadIdx.x & (KTC - 1), tau = threadIdx.x / KTC;
    constexpr int L0 = PhaseInfo<RB, LOG, INV, 0>::LO;
    u64 v[1 << RB];
#pragma unroll
    for (int e = 0; e < (1 << RB); ++e) v[e] = xin[phase_x<RB, L0>(tau, e) * C + (int)blockIdx.x * KTC + col];
    uint4* sw = reinterpret_cast<uint4*>(sm + S * KTC);  // twiddles [0, S)
#pragma unroll
    for (int i = 0; i < (S + T - 1) / T; ++i)
        if (i * T + (int)threadIdx.x < S) sw[i * T + threadIdx.x] = __ldg(tw + i * T + threadIdx.x);
    const DevPrime P = R.primes[pi];
    const uint4* post = poly_post(b, p);
    __syncthreads();
    const int cls = prime_class(R, pi);
    if (cls == 0) ntt_col_body<RB, LOG, INV, KTC, 0>(v, P, post, sm);
    else if (!C2 || cls == 1) ntt_col_body<RB, LOG, INV, KTC, 1>(v, P, post, sm);
    else if constexpr (C2) ntt_col_body<RB, LOG, INV, KTC, 2>(v, P, post, sm);
    constexpr int LL = LastLo<RB, LOG, INV>::v;
#pragma unroll
    for (int e = 0; e < (1 << RB); ++e)
        x[phase_x<RB, LL>(tau, e) * C + (int)blockIdx.x * KTC + col] =
            INV && !(C2 && cls == 2) ? finish<EpiStore, false>(v[e], P) : v[e];
}

template <int LOG, bool INV, int KTC>
__global__ void __launch_bounds__(KTC * (1 << LOG) / 8, 5) k_ntt_col(const __grid_constant__ RingDev R, const __grid_constant__ PolyBatch b) {
    pdl_wait();
    pdl_trigger();
    extern __shared__ __align__(16) u64 sm[];
    ntt_col<3, LOG, INV, KTC, true>(R, b, sm);
}

// row pass: one CTA = RPC rows of S contiguous elements (128 threads), S/8 threads per row
template <int LOG, bool INV, int CLS, class E>
__device__ __forceinline__ void ntt_row_body(u64 (&v)[8], const uint4* tw, const DevPrime& P, int Jbase, int N,
                                             u64* s) {
    const Ctx<CLS, 1, LOG> c(Jbase, N, tw, P);
    RowEx ex{s};
    phases<CLS, 3, LOG, INV, false, 0>(v, threadIdx.x % ((1 << LOG) / 8), c, ex, P);
    if constexpr (!INV) {
#pragma unroll
        for (int e = 0; e < 8; ++e) v[e] = finish<E, CLS == 2>(v[e], P);
    }
}

// a thread's finished values at consecutive places of its row (element e at k + e) to where the
// epilogue puts them
template <class E>
__device__ __forceinline__ void row_put(const u64 (&v)[8], u64* x, int p, int k, const E& epi, const EpiK& K,
                                        const DevPrime& P) {
    if constexpr (in_place<E>) {
#pragma unroll
        for (int e = 0; e < 8; ++e) x[k + e] = v[e];
    } else {
#pragma unroll
        for (int g = 0; g < 8; g += 4) {
            EpiOps<1> o[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) epi.load(o[e], p, k + g + e);
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const u64 w[1] = {v[g + e]};
                epi.put(K, o[e], p, k + g + e, w, P);
            }
        }
    }
}

constexpr int kRowThreads = 128;

template <int LOG, int LOGR, bool INV, class E>
__global__ void __launch_bounds__(kRowThreads, 9) k_ntt_row(const __grid_constant__ RingDev R, const __grid_constant__ PolyBatch b,
                                                                   const __grid_constant__ E epi) {
    pdl_wait();
    pdl_trigger();
    constexpr int S = 1 << LOG, TPR = S / 8;  // threads per row
    constexpr int RPC = (kRowThreads / TPR < (1 << LOGR)) ? kRowThreads / TPR : (1 << LOGR);  // rows per CTA
    extern __shared__ __align__(16) u64 sm[];
    const int p = blockIdx.y, N = R.N;
    int pi;
    u64* x = poly_at(b, p, N, &pi);
    const uint4* tw = (INV ? R.itw : R.tw) + (size_t)pi * N;
    const int rloc = threadIdx.x / TPR, tau = threadIdx.x % TPR;
    const int Jbase = (blockIdx.x * RPC + rloc) * S;
    const u64* xin = (INV ? poly_in(b, p, N, x) : x) + Jbase;  // the row pass is the inverse's first
    constexpr int L0 = PhaseInfo<3, LOG, INV, 0>::LO;
    const DevPrime P = R.primes[pi];
    u64 v[8];
    if (INV && rs_poly(b, p)) {
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            u64 t[1];
            rs_load(t, b, p, Jbase + phase_x<3, L0>(tau, e), N, P.q);
            v[e] = t[0];
        }
    } else {
#pragma unroll
        for (int e = 0; e < 8; ++e) v[e] = xin[phase_x<3, L0>(tau, e)];
    }
    const EpiK K = epi.consts(p);
    u64* s = sm + rloc * S;
    const int cls = prime_class(R, pi);
    if (cls == 0) ntt_row_body<LOG, INV, 0, E>(v, tw, P, Jbase, N, s);
    else if (cls == 1) ntt_row_body<LOG, INV, 1, E>(v, tw, P, Jbase, N, s);
    else ntt_row_body<LOG, INV, 2, E>(v, tw, P, Jbase, N, s);
    constexpr int LL = LastLo<3, LOG, INV>::v;
    if constexpr (INV) {
#pragma unroll
        for (int e = 0; e < 8; ++e) x[Jbase + phase_x<3, LL>(tau, e)] = v[e];
    } else {
        static_assert(LL == 0, "the last forward phase holds the low bits");
        row_put(v, x, p, Jbase + tau * 8, epi, K, P);
    }
}

// Single-launch transform for small batches (tile shape 4): a cluster of CL CTAs holds one
// polynomial, N / CL elements each, 8 a thread. Forward: a CTA transforms C / CL columns
// (exchanges in buffer A), then writes every result straight into the receive buffer B of the CTA
// that owns its row, through distributed shared memory; after the cluster barrier each CTA runs
// the row pass on its R / CL rows (exchanges in A) and stores them. Inverse: rows first, then
// columns. The intermediate never goes through global memory, and one launch with one wait for
// memory replaces two: a batch too small to fill the GPU is bound by that latency (about 3 us a
// pass), not by its arithmetic. Everything the kernel reads is asked for at its start: elements,
// both passes' twiddles and, before the cluster barrier, the epilogue's operands. For N <= 2^13 it
// is the faster form at every batch size (microseconds, forward / inverse, launches in a graph):
//   N = 2^13   8 polys 4.6/4.8 (two passes 5.8/5.8), 128: 13.4/14.5 (14.8/15.7), 1024: 76.8/83.6 (90.9/87.6)
//   N = 2^12   8 polys 4.7/4.5 (5.3/5.5), 128: 7.4/7.8 (9.7/9.9), 1024: 36.9/39.9 (45.6/44.0)
// At N = 2^16, 16 CTAs of 4096 elements, it took 15.7 us for 8 polynomials where two passes take
// 10.0: a cluster that large leaves most of the SMs' slots empty.
template <int LOGR, int LOGC, int CL>
struct ClusterShape {
    static constexpr int R = 1 << LOGR, C = 1 << LOGC, E = R * C / CL, T = E / 8, KTC = C / CL, RPC = R / CL;
    static constexpr size_t smem = (size_t)2 * E * 8 + (size_t)R * 16 + (size_t)E * 16;
};

__device__ __forceinline__ void ld_async16(void* dst, const void* src) {
    const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(src) : "memory");
}
__device__ __forceinline__ void ld_async_wait() {
    asm volatile("cp.async.commit_group;" ::: "memory");
    asm volatile("cp.async.wait_group 0;" ::: "memory");
}

// The shared memory of another CTA of the cluster may be written only once that CTA has started:
// every thread arrives as its kernel begins and waits before its first remote store, so the loads
// and the first pass lie between the two. Relaxed: nothing but the start is ordered by it. It costs
// 0 to 0.2 us a launch (times above; 8 polynomials without it: 4.6/4.7 at N = 2^13, 4.6/4.3 at 2^12).
__device__ __forceinline__ void cluster_arrive_started() { asm volatile("barrier.cluster.arrive.relaxed;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait_started() { asm volatile("barrier.cluster.wait;" ::: "memory"); }

template <int LOGR, int LOGC, int CL, bool INV, int CLS, class E>
__device__ __forceinline__ void ntt_cluster_body(u64 (&v)[8], const PolyBatch& b, u64* x, const DevPrime& P, int p, int rank, u64* sm, const E& epi) {
    namespace cg = cooperative_groups;
    using Sh = ClusterShape<LOGR, LOGC, CL>;
    constexpr int C = Sh::C, KTC = Sh::KTC, RPC = Sh::RPC;
    u64 *A = sm, *B = sm + Sh::E;
    const uint4* sw = reinterpret_cast<const uint4*>(sm + 2 * Sh::E);
    const uint4* srow = sw + Sh::R;  // the rows' twiddles as a table of their own: entry (RPC C + x) >> (bit + 1)
    cg::cluster_group cl = cg::this_cluster();
    const int col = threadIdx.x % KTC, tauc = threadIdx.x / KTC;
    const int rloc = threadIdx.x / (C / 8), taur = threadIdx.x % (C / 8);
    const int row0 = rank * RPC;
    const Ctx<CLS, 0, LOGR> cc(0, Sh::R, sw, P);
    const Ctx<CLS, 0, LOGC> cr(rloc * C, RPC * C, srow, P);
    constexpr int RL0 = PhaseInfo<3, LOGC, INV, 0>::LO, RLL = LastLo<3, LOGC, INV>::v;
    constexpr int CL0 = PhaseInfo<3, LOGR, INV, 0>::LO, CLL = LastLo<3, LOGR, INV>::v;
    if constexpr (!INV) {
        ColEx<KTC> exc{A, col};
        phases<CLS, 3, LOGR, false, false, 0>(v, tauc, cc, exc, P);
        cluster_wait_started();
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            const int row = phase_x<3, CLL>(tauc, e);
            cl.map_shared_rank(B, row / RPC)[(row % RPC) * C + rank * KTC + col] = v[e];
        }
        const int k = (row0 + rloc) * C + taur * 8;  // the thread's 8 results
        const EpiK K = epi.consts(p);
        EpiOps<2> ops[4];
        if constexpr (!in_place<E>) {
#pragma unroll
            for (int h = 0; h < 4; ++h) epi.load(ops[h], p, k + 2 * h);
        }
        cl.sync();
#pragma unroll
        for (int e = 0; e < 8; ++e) v[e] = B[rloc * C + phase_x<3, RL0>(taur, e)];
        RowEx exr{A + rloc * C};
        phases<CLS, 3, LOGC, false, false, 0>(v, taur, cr, exr, P);
        static_assert(RLL == 0, "the last forward phase holds the low bits");
#pragma unroll
        for (int h = 0; h < 4; ++h) {
            const u64 o[2] = {finish<E, false>(v[2 * h], P), finish<E, false>(v[2 * h + 1], P)};
            if constexpr (in_place<E>) st_vec(x + k + 2 * h, o);
            else epi.put(K, ops[h], p, k + 2 * h, o, P);
        }
    } else {
        RowEx exr{B + rloc * C};
        phases<CLS, 3, LOGC, true, false, 0>(v, taur, cr, exr, P);
        cluster_wait_started();
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            const int k = phase_x<3, RLL>(taur, e);
            cl.map_shared_rank(A, k / KTC)[(row0 + rloc) * KTC + k % KTC] = v[e];
        }
        cl.sync();
#pragma unroll
        for (int e = 0; e < 8; ++e) v[e] = A[phase_x<3, CL0>(tauc, e) * KTC + col];
        ColEx<KTC> exc{B, col};
        phases<CLS, 3, LOGR, true, true, 0>(v, tauc, cc, exc, P, poly_post(b, p));
#pragma unroll
        for (int e = 0; e < 8; ++e)
            x[phase_x<3, CLL>(tauc, e) * C + rank * KTC + col] = finish<EpiStore, false>(v[e], P);
    }
}

template <int LOGR, int LOGC, int CL, bool INV, class E>
__global__ void __launch_bounds__(ClusterShape<LOGR, LOGC, CL>::T)
    k_ntt_cluster(const __grid_constant__ RingDev R, const __grid_constant__ PolyBatch b,
                  const __grid_constant__ E epi) {
    cluster_arrive_started();
    pdl_wait();
    pdl_trigger();
    using Sh = ClusterShape<LOGR, LOGC, CL>;
    constexpr int N = Sh::R * Sh::C, C = Sh::C, KTC = Sh::KTC, RPC = Sh::RPC;
    extern __shared__ __align__(16) u64 sm[];
    const int p = blockIdx.y, rank = blockIdx.x;
    int pi;
    u64* x = poly_at(b, p, N, &pi);
    const uint4* tw = (INV ? R.itw : R.tw) + (size_t)pi * N;
    uint4* sw = reinterpret_cast<uint4*>(sm + 2 * Sh::E);
    for (int i = threadIdx.x; i < Sh::R; i += Sh::T) ld_async16(sw + i, tw + i);
    // entries RPC 2^lev .. of the rows' table are a stage's twiddles for this CTA's rows, which lie
    // together in the natural order
    for (int m = RPC + threadIdx.x; m < Sh::E; m += Sh::T) {
        const int lev = 31 - __clz(m / RPC);
        ld_async16(sw + Sh::R + m, tw + ((Sh::R + rank * RPC) << lev) + (m - (RPC << lev)));
    }
    u64 v[8];
    if constexpr (INV) {
        const int k = (rank * RPC + threadIdx.x / (C / 8)) * C + (threadIdx.x % (C / 8)) * 8;
        const u64* xin = poly_in(b, p, N, x) + k;
        const bool rs = rs_poly(b, p);
#pragma unroll
        for (int h = 0; h < 4; ++h) {
            u64 t[2];
            if (rs) rs_load(t, b, p, k + 2 * h, N, R.primes[pi].q);
            else ld_vec(t, xin + 2 * h);
            v[2 * h] = t[0];
            v[2 * h + 1] = t[1];
        }
    } else {
        const int col = threadIdx.x % KTC, tauc = threadIdx.x / KTC;
        const u64* xin = poly_in(b, p, N, x);
#pragma unroll
        for (int e = 0; e < 8; ++e)
            v[e] = xin[phase_x<3, PhaseInfo<3, LOGR, false, 0>::LO>(tauc, e) * C + rank * KTC + col];
    }
    const DevPrime P = R.primes[pi];  // class 0 or 1: the launcher checks
    ld_async_wait();
    __syncthreads();
    if (prime_class(R, pi) == 0) ntt_cluster_body<LOGR, LOGC, CL, INV, 0>(v, b, x, P, p, rank, sm, epi);
    else ntt_cluster_body<LOGR, LOGC, CL, INV, 1>(v, b, x, P, p, rank, sm, epi);
}

template <int LOGR, int LOGC, int CL, bool INV, class E>
void launch_cluster_k(const RingDev& R, const PolyBatch& b, cudaStream_t st, const E& epi) {
    using Sh = ClusterShape<LOGR, LOGC, CL>;
    auto* k = k_ntt_cluster<LOGR, LOGC, CL, INV, E>;
    static std::atomic<unsigned long long> lim{0};
    if (Sh::smem > 48 * 1024) smem_limit_once(k, (int)Sh::smem, lim);
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(CL, b.npolys);
    cfg.blockDim = dim3(Sh::T);
    cfg.dynamicSmemBytes = Sh::smem;
    cfg.stream = st;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = pdl_use(st) ? 1 : 0;
    at[1].id = cudaLaunchAttributeClusterDimension;
    at[1].val.clusterDim.x = CL;
    at[1].val.clusterDim.y = 1;
    at[1].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 2;
    cudaLaunchKernelEx(&cfg, k, R, b, epi);
}

template <int LOGR, int LOGC, class E>
void launch_ntt_cluster(const RingDev& R, const PolyBatch& b, bool inverse, cudaStream_t st, const E& epi) {
    // 1024 elements a CTA, 2048 at N = 2^14
    constexpr int CL = LOGR + LOGC >= 13 ? 8 : LOGR + LOGC == 12 ? 4 : LOGR + LOGC == 11 ? 2 : 1;
    if (inverse) launch_cluster_k<LOGR, LOGC, CL, true, EpiStore>(R, b, st, EpiStore{});
    else launch_cluster_k<LOGR, LOGC, CL, false, E>(R, b, st, epi);
}

// ---------------------------------------------------------------------------
// Radix-16 passes (tile shape 5, N = 2^14 .. 2^16, rings without class-2 primes): every thread
// keeps 16 residues and runs 4 stages (3 in the low phase of a 128-point pass) per shared-memory
// exchange, so a pass has one exchange (radix 8: two) and a stage on register bit lb loads
// 8 >> lb twiddles for its 8 butterflies.
// ---------------------------------------------------------------------------
constexpr int kCol16 = 8;  // columns of a column-pass CTA: 64-byte row segments

template <int LOG, bool INV>
__global__ void __launch_bounds__(kCol16 * (1 << LOG) / 16, (INV ? 6 : 5) * (256 >> LOG))
    k_ntt_col16(const __grid_constant__ RingDev R, const __grid_constant__ PolyBatch b) {
    pdl_wait();
    pdl_trigger();
    extern __shared__ __align__(16) u64 sm[];
    ntt_col<4, LOG, INV, kCol16, false>(R, b, sm);
}

// Row pass: 128 threads, each warp on its own 512 contiguous elements (2 rows of 256 points or 4
// of 128), so no block barrier. The phase on the low bits has a thread's 16 elements contiguous
// (128 bytes): they pass through shared memory in 16-byte chunks, chunk h of a thread at h ^
// (thread & 7), so that the global side moves 512 contiguous bytes per instruction and epilogues
// see consecutive elements in consecutive lanes. Reading and writing them thread by thread
// touches 32 cache lines per instruction, which bounded the pass (the epilogues above all).
template <int LOG, bool INV, int CLS>
__device__ __forceinline__ void ntt_row16_body(u64 (&v)[16], const uint4* tw, const DevPrime& P, int rho, int N,
                                               u64* ws) {
    constexpr int S = 1 << LOG, TPR = S / 16;
    const int lane = threadIdx.x & 31;
    const Ctx<CLS, 2, LOG> c(rho * S, N, tw + (size_t)rho * S, P);
    RowEx16<LOG> ex{ws + (lane / TPR) * S, rho & 1};
    phases<CLS, 4, LOG, INV, false, 0>(v, lane % TPR, c, ex, P);
}

template <int LOG, bool INV, class E>
__global__ void __launch_bounds__(128, 6) k_ntt_row16(const __grid_constant__ RingDev R,
                                                      const __grid_constant__ PolyBatch b,
                                                      const __grid_constant__ E epi) {
    pdl_wait();
    pdl_trigger();
    extern __shared__ __align__(16) u64 sm[];  // [4 warps][512]
    constexpr int S = 1 << LOG, TPR = S / 16;
    const int p = blockIdx.y, N = R.N;
    int pi;
    u64* x = poly_at(b, p, N, &pi);
    const uint4* tw = (INV ? R.irtw : R.rtw) + (size_t)pi * N;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int Wbase = (blockIdx.x * 4 + warp) * 512;  // the warp's first element
    const int rho = Wbase / S + lane / TPR;
    u64* ws = sm + warp * 512;
    u64 v[16];
    const DevPrime P = R.primes[pi];
    const EpiK K = epi.consts(p);
    if constexpr (INV) {
        ulonglong2* wc = reinterpret_cast<ulonglong2*>(ws);
        if (rs_poly(b, p)) {
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const int ch = j * 32 + lane;
                u64 t[2];
                rs_load(t, b, p, Wbase + 2 * ch, N, P.q);
                wc[ch ^ ((ch >> 3) & 7)] = make_ulonglong2(t[0], t[1]);
            }
        } else {
            const u64* xin = poly_in(b, p, N, x) + Wbase;
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const int ch = j * 32 + lane;
                ld_async16(wc + (ch ^ ((ch >> 3) & 7)), xin + 2 * ch);
            }
            ld_async_wait();
        }
        __syncwarp();
#pragma unroll
        for (int h = 0; h < 8; ++h) {
            const ulonglong2 t = wc[lane * 8 + (h ^ (lane & 7))];
            v[2 * h] = t.x;
            v[2 * h + 1] = t.y;
        }
        __syncwarp();
    } else {
        const u64* xr = x + (long long)rho * S;
#pragma unroll
        for (int e = 0; e < 16; ++e) v[e] = xr[phase_x<4, LOG - 4>(lane % TPR, e)];
    }
    if (prime_class(R, pi) == 0) ntt_row16_body<LOG, INV, 0>(v, tw, P, rho, N, ws);
    else ntt_row16_body<LOG, INV, 1>(v, tw, P, rho, N, ws);
    if constexpr (INV) {
        u64* xr = x + (long long)rho * S;
#pragma unroll
        for (int e = 0; e < 16; ++e) xr[phase_x<4, LOG - 4>(lane % TPR, e)] = v[e];
    } else {
        ulonglong2* wc = reinterpret_cast<ulonglong2*>(ws);
#pragma unroll
        for (int h = 0; h < 8; ++h)
            wc[lane * 8 + (h ^ (lane & 7))] =
                make_ulonglong2(finish<E, false>(v[2 * h], P), finish<E, false>(v[2 * h + 1], P));
        __syncwarp();
#pragma unroll
        for (int g = 0; g < 8; g += 4) {
            EpiOps<2> ops[4];
            if constexpr (!in_place<E>) {
#pragma unroll
                for (int j = 0; j < 4; ++j) epi.load(ops[j], p, Wbase + 2 * ((g + j) * 32 + lane));
            }
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int ch = (g + j) * 32 + lane;
                u64 o[2];
                ld_vec(o, ws + 2 * (ch ^ ((ch >> 3) & 7)));
                if constexpr (in_place<E>) st_vec(x + Wbase + 2 * ch, o);
                else epi.put(K, ops[j], p, Wbase + 2 * ch, o, P);
            }
        }
    }
}

template <int LOGR, int LOGC, class E>
void launch_ntt_r16(const RingDev& R, const PolyBatch& b, bool inverse, cudaStream_t st, const E& epi) {
    constexpr int SR = 1 << LOGR, SC = 1 << LOGC;
    const dim3 gc(SC / kCol16, b.npolys), gr(SR * SC / 2048, b.npolys);
    const int tc = kCol16 * SR / 16;
    const size_t smc = (size_t)(SR * kCol16 + 2 * SR) * sizeof(u64), smr = (size_t)2048 * sizeof(u64);
    if (!inverse) {
        launch_k(k_ntt_col16<LOGR, false>, gc, dim3(tc), smc, st, R, b);
        launch_k(k_ntt_row16<LOGC, false, E>, gr, dim3(128), smr, st, R, b, epi);
    } else {
        launch_k(k_ntt_row16<LOGC, true, EpiStore>, gr, dim3(128), smr, st, R, b, EpiStore{});
        launch_k(k_ntt_col16<LOGR, true>, gc, dim3(tc), smc, st, R, b);
    }
}

template <int LOGR, int LOGC, class E, int KTC>
void launch_ntt_t(const RingDev& R, const PolyBatch& b, bool inverse, cudaStream_t st, const E& epi) {
    constexpr int SR = 1 << LOGR, SC = 1 << LOGC;
    const int N = R.N;
    dim3 gc((N >> LOGR) / KTC, b.npolys);
    const int tc = KTC * SR / 8;
    const size_t smc = (size_t)(SR * KTC + 2 * SR) * sizeof(u64);
    constexpr int TPR = SC / 8, RPC = (kRowThreads / TPR < SR) ? kRowThreads / TPR : SR;
    dim3 gr(SR / RPC, b.npolys);
    const size_t smr = (size_t)RPC * SC * sizeof(u64);
    if (!inverse) {
        launch_k(k_ntt_col<LOGR, false, KTC>, dim3(gc), dim3(tc), smc, st, R, b);
        launch_k(k_ntt_row<LOGC, LOGR, false, E>, dim3(gr), dim3(RPC * TPR), smr, st, R, b, epi);
    } else {
        launch_k(k_ntt_row<LOGC, LOGR, true, EpiStore>, dim3(gr), dim3(RPC * TPR), smr, st, R, b, EpiStore{});
        launch_k(k_ntt_col<LOGR, true, KTC>, dim3(gc), dim3(tc), smc, st, R, b);
    }
}

// Tile shape of a launch: 0..3 are the radix-8 two-pass kernels, bit 0 set = 8 columns per
// column-pass CTA (else 4), bit 1 free; 4 is the cluster kernel (N <= 2^14) and 5 the radix-16
// two-pass kernels (N >= 2^14). Rings of N >= 2^14 choose per batch-size bucket by the tuner (RingDev
// holds the table); smaller ones run the cluster kernel. Measured at N = 2^16, forward / inverse, 9
// primes (1 of 60 bits, 8 of 50), microseconds, launches in a graph:
//   polys     4          8            16          64          256          1024
//   shape 0   8.0/7.8    11.6/11.2    16.6/16.9   51.5/52.3   189.5/191.6  734.4/740.0
//   shape 5   8.3/8.6    10.1/10.4    14.9/15.3   41.0/42.4   147.1/155.0  561.7/586.0
// (512 polys with Shoup products: shape 0 487.7/471.0, and 448.2/455.1 for 16 residues a thread
// that read and wrote their 128 contiguous bytes thread by thread; now 285.2/298.4.)
// Exceptions: shapes 4 and 5 have no code for class-2 primes and move 16-byte chunks, so a ring
// with such a prime or a batch at an address that is not a multiple of 16 bytes (a caller's own
// buffer) runs shape 0; so does a size that the shape does not have.
inline int ntt_shape_of(const RingDev& R, const PolyBatch& b) {
    const int shape = R.logN < 14 ? 4 : R.ntt_shape[ntt_bucket(b.npolys)];
    if (shape < 4) return shape;
    const uintptr_t a = (uintptr_t)b.base | (uintptr_t)b.src | (uintptr_t)b.base2 |
                        (uintptr_t)(8 * b.outer) | (uintptr_t)(8 * b.src_outer) | (uintptr_t)(8 * b.outer2);
    return !R.fast || (a & 15) || (shape == 4 && R.logN > 14) ? 0 : shape;
}

// Returns the number of kernels launched.
template <int LOGR, int LOGC, class E>
int launch_ntt_s(const RingDev& R, const PolyBatch& b, bool inverse, cudaStream_t st, const E& epi) {
    const int shape = ntt_shape_of(R, b);
    if constexpr (LOGR + LOGC <= 14) {
        if (shape == 4) {
            launch_ntt_cluster<LOGR, LOGC>(R, b, inverse, st, epi);
            return 1;
        }
    }
    if constexpr (LOGR + LOGC >= 14) {
        if (shape == 5) {
            launch_ntt_r16<LOGR, LOGC>(R, b, inverse, st, epi);
            return 2;
        }
    }
    if constexpr (LOGR + LOGC >= 15) {
        if (shape & 1) {
            launch_ntt_t<LOGR, LOGC, E, 8>(R, b, inverse, st, epi);
            return 2;
        }
    }
    launch_ntt_t<LOGR, LOGC, E, 4>(R, b, inverse, st, epi);
    return 2;
}

// The transform of a ring of N <= 2^14 (ntt_small.cu).
template <class E>
int launch_ntt_small(const RingDev& R, const PolyBatch& b, bool inverse, cudaStream_t s, const E& epi);

}  // namespace ntt_kernels
