// CKKS device kernels: base conversion (ModUp / ModDown), key-switch inner
// product with the slot automorphism fused into its gather, rescale, tensor
// product, the diagonal plaintext x ciphertext multiply-accumulate, Chebyshev
// scalar steps and the on-device slot encoder for template diagonals.
#include <algorithm>
#include <cstdio>

#include "ckks_kernels.h"
#include "bconv.cuh"

namespace {

constexpr int kThreads = 256;

__device__ __forceinline__ void fold(Acc128& a, u64 q) {
    if (a.hi >= q) a.hi -= q;
}

// ---------------------------------------------------------------------------
// Fast base conversions (ModUp, ModDown) as kernels of their own: a thread converts W = 2
// consecutive coefficients, 16-byte accesses, to every target in turn; the block's targets are
// staged in shared memory.
// ---------------------------------------------------------------------------
constexpr int kBcW = 2;          // 4 points a thread measured 84 us where 2 take 74 (k_modup, 15 inputs)
constexpr int kBcThreads = 128;  // 256: 74 us, 128: 70

// sources of a conversion: limb i of the thread's points at x + i N
template <int NS>
__device__ __forceinline__ void bconv_load(u64 (&y)[NS][kBcW], const u64* __restrict__ x, int N) {
#pragma unroll
    for (int i = 0; i < NS; ++i) {
#pragma unroll
        for (int w = 0; w < kBcW; w += 2) {
            const ulonglong2 t = *reinterpret_cast<const ulonglong2*>(x + (long long)i * N + w);
            y[i][w] = t.x;
            y[i][w + 1] = t.y;
        }
    }
}

__device__ __forceinline__ void bconv_store(u64* p, const u64 (&v)[kBcW]) {
#pragma unroll
    for (int w = 0; w < kBcW; w += 2) *reinterpret_cast<ulonglong2*>(p + w) = make_ulonglong2(v[w], v[w + 1]);
}

// n targets from global into shared memory
__device__ __forceinline__ void stage_targets(BconvTarget* s, const BconvTarget* __restrict__ g, int n) {
    static_assert(sizeof(BconvTarget) % 16 == 0, "copied in 16-byte words");
    const uint4* src = reinterpret_cast<const uint4*>(g);
    uint4* dst = reinterpret_cast<uint4*>(s);
    for (int e = threadIdx.x; e < n * (int)(sizeof(BconvTarget) / 16); e += blockDim.x) dst[e] = src[e];
    __syncthreads();
}

// ---------------------------------------------------------------------------
// ModUp: per digit, fast-convert the digit's limbs to every other position of Q_l u P
// (coefficient form). The digit's own positions are not written: the inner product reads them
// from the switched polynomial itself, in evaluation form.
// in: coefficient form, job j at in + j * in_job, already times inv_hat if SCALED;
// ext: [J][beta][npos][N]
// Bound by integer multiplies before (75 of 99 us in arithmetic for 15 inputs at level 7, 4 limbs a
// digit: 3 wide products a source, 80 cycles of reduction a target, and the products by inv_hat);
// now 4 wide products a source, 2 for the reduction, none for inv_hat, and a third of the traffic
// (the copies of the own positions) is gone. Block z = job, y = (digit, chunk of positions): one
// chunk when the jobs fill the GPU, up to npos of them for a single input.
// ---------------------------------------------------------------------------
template <int NS, bool SCALED>
__device__ __forceinline__ void modup_body(const ModUpTab& T, const BconvTarget* st, const u64* __restrict__ x,
                                           u64* __restrict__ out, int pos0, int pos1, int N, int k) {
    u64 y[NS][kBcW];
    bconv_load(y, x + (long long)T.lo * N + k, N);
    if constexpr (!SCALED) {
#pragma unroll
        for (int i = 0; i < NS; ++i)
#pragma unroll
            for (int w = 0; w < kBcW; ++w) y[i][w] = mul_shoup(y[i][w], T.inv_hat[i], T.inv_hat_s[i], T.src_q[i]);
    }
    const u64 zero[kBcW] = {};
    for (int pos = pos0; pos < pos1; ++pos) {
        if (pos >= T.lo && pos < T.lo + NS) continue;
        u64 v[kBcW];
        bconv<NS, kBcW>(st[pos - pos0], y, zero, v);
        bconv_store(out + (long long)pos * N + k, v);
    }
}

template <bool SCALED>
__global__ void __launch_bounds__(kBcThreads) k_modup(const u64* __restrict__ in, long long in_job,
                                                    u64* __restrict__ ext, const ModUpTab* __restrict__ tabs, int beta,
                                                    int npos, int N, int per) {
    pdl_wait();
    pdl_trigger();
    __shared__ BconvTarget st[FR_MAX_PRIMES];
    const int k = (blockIdx.x * blockDim.x + threadIdx.x) * kBcW;
    const int d = blockIdx.y % beta, pos0 = (blockIdx.y / beta) * per, pos1 = min(npos, pos0 + per);
    const int j = blockIdx.z;
    const ModUpTab& T = tabs[d];
    stage_targets(st, T.t + pos0, pos1 - pos0);
    if (k >= N) return;
    const u64* x = in + (long long)j * in_job;
    u64* out = ext + (((long long)j * beta + d) * npos) * N;
    switch (T.ns) {
        case 1: modup_body<1, SCALED>(T, st, x, out, pos0, pos1, N, k); break;
        case 2: modup_body<2, SCALED>(T, st, x, out, pos0, pos1, N, k); break;
        case 3: modup_body<3, SCALED>(T, st, x, out, pos0, pos1, N, k); break;
        case 4: modup_body<4, SCALED>(T, st, x, out, pos0, pos1, N, k); break;
        case 5: modup_body<5, SCALED>(T, st, x, out, pos0, pos1, N, k); break;
        case 6: modup_body<6, SCALED>(T, st, x, out, pos0, pos1, N, k); break;
        case 7: modup_body<7, SCALED>(T, st, x, out, pos0, pos1, N, k); break;
        default: modup_body<8, SCALED>(T, st, x, out, pos0, pos1, N, k); break;  // ns <= 8, checked on the host
    }
}

// ---------------------------------------------------------------------------
// Key-switch inner product: acc_t[pos] = sum_d sigma_g(ext_d[pos]) * key_d[t][limb(pos)]
// Keys are stored in Montgomery form, so one REDC of the 128-bit sum gives
// the canonical residue. The automorphism is a gather on the ext index. When
// all jobs of a launch use the same key (batched relinearisation), a thread
// reads its key words once and applies them to every job.
// A thread takes two consecutive points (16-byte loads, twice the bytes in flight of one: the
// kernel is bound by HBM latency). The automorphism keeps aligned pairs together: position k's
// source is src(k), and src(k + 1) = src(k) ^ 1 for even k, because the low bits of a position are
// the high bits of the exponent 2 brev(k) + 1, which an odd factor permutes among themselves. So a
// gathered pair is one aligned load, its halves swapped when src(k) is odd.
// Measured at the headline size, one point a thread -> two: the baby steps (31 keys, 3 digits, 13
// positions, 1.73 GB) 343 -> 264 us, 6.5 TB/s; k_ip_sum of the giant
// steps 148 -> 117 us, of the five hoisted steps of the slot sum 116 -> 104 us together.
// ---------------------------------------------------------------------------
constexpr int kIpThreads = 128;

struct U64x2 {
    u64 v[2];
};
__device__ __forceinline__ U64x2 ld2(const u64* p) {
    const ulonglong2 t = *reinterpret_cast<const ulonglong2*>(p);
    return U64x2{{t.x, t.y}};
}
// the pair gathered for the even position whose source is src
__device__ __forceinline__ U64x2 ld2_from(const u64* p, u32 src) {
    const U64x2 t = ld2(p + (src & ~1u));
    return (src & 1) ? U64x2{{t.v[1], t.v[0]}} : t;
}
__device__ __forceinline__ void st2(u64* p, u64 a, u64 b) { *reinterpret_cast<ulonglong2*>(p) = make_ulonglong2(a, b); }

// digit d's extension at position pos: its own limb of the switched polynomial, or ext
__device__ __forceinline__ const u64* ip_ext(const IPJob& J, int d, int npos, int pos, int owner, int N) {
    return d == owner ? J.own + (long long)pos * N : J.ext + ((long long)d * npos + pos) * N;
}

// key layout [digit][2][T][N]: Q limbs at positions 0.., P limbs from position kp. One
// instantiation per digit count, so the registers a launch needs follow its beta. One key group
// per blockIdx.y: its key words are read once and applied to every job of the group.
template <int BETA>
__global__ void __launch_bounds__(kIpThreads) k_ip(const __grid_constant__ IPJobs jobs, int npos, int level, int kp,
                                                   int T, const DevPrime* __restrict__ primes, int pbase, int logN,
                                                   const u64* __restrict__ pmod, const u64* __restrict__ pmod_s) {
    pdl_wait();
    pdl_trigger();
    const int N = 1 << logN;
    const int k = (blockIdx.x * kIpThreads + threadIdx.x) * 2;
    // position-major grid: the key groups of one position run back to back, so a ModUp
    // extension that several groups gather from (hoisted rotations) is read from L2
    const int pos = blockIdx.z, g = blockIdx.y;
    if (k >= N) return;
    // positions 0..level are Q limbs 0..level; the P limbs follow (prime indices from pbase)
    const int pi = pos <= level ? pos : pbase + (pos - (level + 1));
    const u64 q = primes[pi].q, qinv = primes[pi].qinv;
    const int klimb = pos <= level ? pos : kp + (pos - (level + 1));
    const int owner = jobs.owner[pos];
    const u64* key = jobs.gkey[g] + (long long)klimb * N + k;
    U64x2 k0[BETA], k1[BETA];
#pragma unroll
    for (int d = 0; d < BETA; ++d) {
        k0[d] = ld2(key + (long long)(2 * d) * T * N);
        k1[d] = ld2(key + (long long)(2 * d + 1) * T * N);
    }
    for (int jj = jobs.gstart[g]; jj < jobs.gstart[g + 1]; ++jj) {
        const IPJob& J = jobs.j[jj];
        const u32 src = J.galois != 1u ? galois_src_index((u32)k, J.galois, logN) : (u32)k;
        U64x2 e[BETA], badd{{0, 0}};
#pragma unroll
        for (int d = 0; d < BETA; ++d) e[d] = ld2_from(ip_ext(J, d, npos, pos, owner, N), src);
        const bool addb = J.addb && pos <= level;  // a rotation kept in Q_l u P: + P sigma(b) on the Q positions
        if (addb) badd = ld2_from(J.addb + (long long)pos * N, src);
        u64 r0[2], r1[2];
#pragma unroll
        for (int w = 0; w < 2; ++w) {
            Acc128 a0{0, 0}, a1{0, 0};
#pragma unroll
            for (int d = 0; d < BETA; ++d) {
                mac_full(a0, e[d].v[w], k0[d].v[w]);
                mac_full(a1, e[d].v[w], k1[d].v[w]);
            }
            fold(a0, q);
            fold(a1, q);
            r0[w] = redc(a0.hi, a0.lo, q, qinv);
            if (addb) r0[w] = add_mod(r0[w], mul_shoup(badd.v[w], pmod[pos], pmod_s[pos], q), q);
            r1[w] = redc(a1.hi, a1.lo, q, qinv);
        }
        st2(J.out + (long long)pos * N + k, r0[0], r0[1]);
        st2(J.out + ((long long)npos + pos) * N + k, r1[0], r1[1]);
    }
}

// Inner products summed into their accumulator (double-hoisted sums of rotations): thread
// (points k, k + 1, group g, position pos) runs the jobs of group g, each a key-switch inner product
// of its ext under its automorphism (the same products as k_ip), in one 128-bit sum per
// component, folded after every job: a product of two residues below q < 2^61 adds less than
// q/8 to the high word, so a job's beta <= 8 products leave it below 2q before the fold. Then
// it adds P sum_j sigma_j(addb_j) on the Q positions of component 0 (one product by P for all
// jobs) and, where an earlier launch started the sum (add), the value already in the accumulator. The words of U jobs are loaded together: the jobs' keys come from HBM one after the
// other otherwise. The grid is (points, groups, positions), groups fastest after the points:
// the key words of one position, which every group's job with that key reads, are L2 hits
// after the first group.
template <int BETA>
__global__ void __launch_bounds__(kIpThreads) k_ip_sum(const __grid_constant__ IPSumJobs jobs, int npos, int level,
                                                       int kp, int T, const DevPrime* __restrict__ primes, int pbase,
                                                       int logN, const u64* __restrict__ pmod,
                                                       const u64* __restrict__ pmod_s) {
    pdl_wait();
    pdl_trigger();
    constexpr int U = BETA == 1 ? 4 : BETA == 2 ? 2 : 1;
    const int N = 1 << logN;
    const int k = (blockIdx.x * kIpThreads + threadIdx.x) * 2;
    const int g = blockIdx.y;
    const int pos = blockIdx.z;
    if (k >= N) return;
    const int pi = pos <= level ? pos : pbase + (pos - (level + 1));
    const u64 q = primes[pi].q, qinv = primes[pi].qinv;
    const int klimb = pos <= level ? pos : kp + (pos - (level + 1));
    const int owner = jobs.owner[pos];
    Acc128 a0[2] = {}, a1[2] = {};
    u64 badd[2] = {0, 0};
    const int end = jobs.gstart[g + 1];
    for (int j0 = jobs.gstart[g]; j0 < end; j0 += U) {
        U64x2 e[U][BETA], k0[U][BETA], k1[U][BETA], bb[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const IPJob& J = jobs.j[min(j0 + u, end - 1)];
            const u32 src = J.galois != 1u ? galois_src_index((u32)k, J.galois, logN) : (u32)k;
            const u64* key = J.key + (long long)klimb * N + k;
#pragma unroll
            for (int d = 0; d < BETA; ++d) {
                e[u][d] = ld2_from(ip_ext(J, d, npos, pos, owner, N), src);
                k0[u][d] = ld2(key + (long long)(2 * d) * T * N);
                k1[u][d] = ld2(key + (long long)(2 * d + 1) * T * N);
            }
            if (J.addb && pos <= level) bb[u] = ld2_from(J.addb + (long long)pos * N, src);
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (j0 + u >= end) break;
            const bool addb = jobs.j[j0 + u].addb && pos <= level;
#pragma unroll
            for (int w = 0; w < 2; ++w) {
#pragma unroll
                for (int d = 0; d < BETA; ++d) {
                    mac_full(a0[w], e[u][d].v[w], k0[u][d].v[w]);
                    mac_full(a1[w], e[u][d].v[w], k1[u][d].v[w]);
                }
                fold(a0[w], q);
                fold(a1[w], q);
                if (addb) badd[w] = add_mod(badd[w], bb[u].v[w], q);
            }
        }
    }
    u64* O0 = jobs.j[jobs.gstart[g]].out + (long long)pos * N + k;
    u64* O1 = O0 + (long long)npos * N;
    U64x2 o0{{0, 0}}, o1{{0, 0}};
    if (jobs.add[g]) {
        o0 = ld2(O0);
        o1 = ld2(O1);
    }
    u64 r0[2], r1[2];
#pragma unroll
    for (int w = 0; w < 2; ++w) {
        const u64 pb = pos <= level ? mul_shoup(badd[w], pmod[pos], pmod_s[pos], q) : 0;
        r0[w] = add_mod(o0.v[w], add_mod(redc(a0[w].hi, a0[w].lo, q, qinv), pb, q), q);
        r1[w] = add_mod(o1.v[w], redc(a1[w].hi, a1[w].lo, q, qinv), q);
    }
    st2(O0, r0[0], r0[1]);
    st2(O1, r1[0], r1[1]);
}

// ---------------------------------------------------------------------------
// ModDown base conversion P -> Q_l: acc: job j's P limbs in coefficient form, times inv_hat; conv
// [J][2][level+1][N]
template <int NP>
__device__ __forceinline__ void p2q_body(const u64* __restrict__ x, u64* __restrict__ o, const BconvTarget* st,
                                         int level, int N, int k) {
    u64 y[NP][kBcW];
    bconv_load(y, x + (long long)(level + 1) * N + k, N);
    const u64 zero[kBcW] = {};
    for (int i = 0; i <= level; ++i) {
        u64 v[kBcW];
        bconv<NP, kBcW>(st[i], y, zero, v);
        bconv_store(o + (long long)i * N + k, v);
    }
}

__global__ void __launch_bounds__(kBcThreads) k_p2q(const u64* __restrict__ acc, long long acc_job, int npos,
                                                  int level, u64* __restrict__ conv, const P2QTab* __restrict__ tab,
                                                  int N) {
    pdl_wait();
    pdl_trigger();
    __shared__ BconvTarget st[FR_MAX_PRIMES];
    const int k = (blockIdx.x * blockDim.x + threadIdx.x) * kBcW;
    const int t = blockIdx.y;
    const int j = blockIdx.z;
    stage_targets(st, tab->t, level + 1);
    if (k >= N) return;
    const u64* x = acc + (long long)j * acc_job + (long long)t * npos * N;
    u64* o = conv + ((long long)j * 2 + t) * (level + 1) * N;
    switch (tab->np) {
        case 1: p2q_body<1>(x, o, st, level, N, k); break;
        case 2: p2q_body<2>(x, o, st, level, N, k); break;
        case 3: p2q_body<3>(x, o, st, level, N, k); break;
        case 4: p2q_body<4>(x, o, st, level, N, k); break;
        case 5: p2q_body<5>(x, o, st, level, N, k); break;
        case 6: p2q_body<6>(x, o, st, level, N, k); break;
        case 7: p2q_body<7>(x, o, st, level, N, k); break;
        default: p2q_body<8>(x, o, st, level, N, k); break;  // np <= 8, checked on the host
    }
}

// The same conversion followed by a rescale's lift (moddown_rescale): the P limbs come
// in coefficient form times inv_hat, and the table's targets carry [B/b_i]_t P^-1, so bconv gives
// conv_i P^-1. With zc = the last limb before the conversion's part
// is taken off (coefficient form), the last limb is m = zc - conv_l P^-1 (mod q_l), and
// y_i = conv_i P^-1 + [centered m]_{q_i} for i < l: m - q_l for m > half is added as m + (-q_l mod
// q_i), unreduced, before the conversion's own reduction. acc: job j's P limbs (inv_hat in them);
// zc [J][2][N]; y [J][2][l][N]. The conversions themselves no longer pass through memory.
template <int NP>
__device__ __forceinline__ void p2q_lift_body(const u64* __restrict__ x, const u64* __restrict__ zc,
                                              u64* __restrict__ o, const BconvTarget* st, const RescaleTab& R, u64 ql,
                                              int l, int N, int k) {
    u64 y[NP][kBcW];
    bconv_load(y, x + (long long)(l + 1) * N + k, N);
    u64 z[1][kBcW];
    bconv_load(z, zc + k, N);
    const u64 zero[kBcW] = {};
    u64 m[kBcW];
    bconv<NP, kBcW>(st[l], y, zero, m);
    bool neg[kBcW];
#pragma unroll
    for (int w = 0; w < kBcW; ++w) {
        m[w] = sub_mod(z[0][w], m[w], ql);
        neg[w] = m[w] > R.half;
    }
    for (int i = 0; i < l; ++i) {
        const u64 nq = R.q[i] - R.ql_mod[i];
        u64 add[kBcW], v[kBcW];
#pragma unroll
        for (int w = 0; w < kBcW; ++w) add[w] = m[w] + (neg[w] ? nq : 0);
        bconv<NP, kBcW>(st[i], y, add, v);
        bconv_store(o + (long long)i * N + k, v);
    }
}

__global__ void __launch_bounds__(kBcThreads) k_p2q_lift(const u64* __restrict__ acc, long long acc_job, int npos,
                                                       const u64* __restrict__ zc, u64* __restrict__ y,
                                                       const P2QTab* __restrict__ tab,
                                                       const RescaleTab* __restrict__ rtab, u64 ql, int l, int N) {
    pdl_wait();
    pdl_trigger();
    __shared__ BconvTarget st[FR_MAX_PRIMES];
    const int k = (blockIdx.x * blockDim.x + threadIdx.x) * kBcW;
    const int t = blockIdx.y;
    const int j = blockIdx.z;
    stage_targets(st, tab->t, l + 1);
    if (k >= N) return;
    const u64* x = acc + (long long)j * acc_job + (long long)t * npos * N;
    const u64* z = zc + ((long long)j * 2 + t) * N;
    u64* o = y + ((long long)j * 2 + t) * l * N;
    switch (tab->np) {
        case 1: p2q_lift_body<1>(x, z, o, st, *rtab, ql, l, N, k); break;
        case 2: p2q_lift_body<2>(x, z, o, st, *rtab, ql, l, N, k); break;
        case 3: p2q_lift_body<3>(x, z, o, st, *rtab, ql, l, N, k); break;
        case 4: p2q_lift_body<4>(x, z, o, st, *rtab, ql, l, N, k); break;
        case 5: p2q_lift_body<5>(x, z, o, st, *rtab, ql, l, N, k); break;
        case 6: p2q_lift_body<6>(x, z, o, st, *rtab, ql, l, N, k); break;
        case 7: p2q_lift_body<7>(x, z, o, st, *rtab, ql, l, N, k); break;
        default: p2q_lift_body<8>(x, z, o, st, *rtab, ql, l, N, k); break;
    }
}

// ---------------------------------------------------------------------------
// Rescale. lift: centered last limb (coefficient form) to each q_i, i < l.
// last: [B][2][N] ; lifted: [B][2][l][N]
// ---------------------------------------------------------------------------
// the centered lift of x < q_l (x, or x - q_l above half) mod q_i: x plus -q_l mod q_i, reduced once
__device__ __forceinline__ u64 centered_residue(u64 x, const RescaleTab& tab, const DevPrime& P, int i) {
    const u64 v = x + (x > tab.half ? P.q - tab.ql_mod[i] : 0);  // below 2^62
    if (P.fold63) {
        const u64 f = fold_top(v, P.bsh, P.c);
        return min(f, f - P.q);
    }
    return mul_shoup(v, 1, P.one_s, P.q);
}

__global__ void __launch_bounds__(kThreads) k_rescale_lift(const u64* __restrict__ last, u64* __restrict__ lifted,
                                                           const RescaleTab* __restrict__ tab,
                                                           const DevPrime* __restrict__ primes, int l, int N) {
    pdl_wait();
    pdl_trigger();
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    const int bt = blockIdx.y;
    if (k >= N) return;
    const u64 x = last[(long long)bt * N + k];
    u64* o = lifted + (long long)bt * l * N + k;
    for (int i = 0; i < l; ++i) o[(long long)i * N] = centered_residue(x, *tab, primes[i], i);
}

// Baby steps kept in Q_l u P (double hoisting of the baby steps): baby 0 of query b is P q_b on
// the Q positions and zero on the P positions (babies 1..n1-1 come from the inner-product
// kernel, which adds P sigma_i(q_b.b) itself). babies [B][n1][2][npos][N] (query b at babies +
// b baby_q); q_b at q + b q_bs, [2][q_cap][N], evaluation form. Grid (N / 256, npos, 2 B).
__global__ void __launch_bounds__(kThreads) k_baby0_pq(u64* __restrict__ babies, long long baby_q,
                                                       const u64* __restrict__ q, long long q_bs, int q_cap, int npos,
                                                       int level, const DevPrime* __restrict__ primes,
                                                       const u64* __restrict__ pmod, const u64* __restrict__ pmod_s,
                                                       int N) {
    pdl_wait();
    pdl_trigger();
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    const int pos = blockIdx.y;
    const int t = blockIdx.z & 1, b = blockIdx.z >> 1;
    if (k >= N) return;
    u64* o = babies + (long long)b * baby_q + ((long long)t * npos + pos) * N + k;
    if (pos > level) {
        *o = 0;
        return;
    }
    const u64 qp = primes[pos].q;
    *o = mul_shoup(q[(long long)b * q_bs + ((long long)t * q_cap + pos) * N + k], pmod[pos], pmod_s[pos], qp);
}

// ---------------------------------------------------------------------------
// Tensor product of ciphertext pairs (evaluation form):
// d0 = a0 b0, d1 = a0 b1 + a1 b0, d2 = a1 b1.  out: [B][3][level+1][N]
// Four 128-bit products and three reductions a point, two points a thread: 16 products of 7 limbs
// at N = 2^16 take 65 us, 4.6 TB/s (two Montgomery reductions per product, one point: 94 us).
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(kBcThreads) k_tensor(const TensorJobs jobs, int level,
                                                     const DevPrime* __restrict__ primes, int N) {
    pdl_wait();
    pdl_trigger();
    const int k = (blockIdx.x * blockDim.x + threadIdx.x) * 2;  // two points, 16-byte accesses
    const int i = blockIdx.y;
    const TensorJob& J = jobs.j[blockIdx.z];
    if (k >= N) return;
    const DevPrime P = primes[i];
    auto ld = [&](const u64* p) { return *reinterpret_cast<const ulonglong2*>(p + k); };
    const ulonglong2 a0 = ld(J.a + (long long)i * N), a1 = ld(J.a + ((long long)J.a_cap + i) * N);
    const ulonglong2 b0 = ld(J.b + (long long)i * N), b1 = ld(J.b + ((long long)J.b_cap + i) * N);
    u64 d0[2], d1[2], d2[2];
    auto point = [&](u64 x0, u64 x1, u64 y0, u64 y1, int w) {
        if (P.cls < 2) {
            Acc128 s0{0, 0}, s1{0, 0}, s2{0, 0};
            mac_full(s0, x0, y0);
            mac_full(s1, x0, y1);
            mac_full(s1, x1, y0);
            mac_full(s2, x1, y1);
            d0[w] = reduce_sum(s0, P);
            d1[w] = reduce_sum(s1, P);
            d2[w] = reduce_sum(s2, P);
        } else {
            d0[w] = mul_mod(x0, y0, P);
            d1[w] = add_mod(mul_mod(x0, y1, P), mul_mod(x1, y0, P), P.q);
            d2[w] = mul_mod(x1, y1, P);
        }
    };
    point(a0.x, a1.x, b0.x, b1.x, 0);
    point(a0.y, a1.y, b0.y, b1.y, 1);
    const long long ps = (long long)(level + 1) * N;
    u64* o = J.out + (long long)i * N + k;
    *reinterpret_cast<ulonglong2*>(o) = make_ulonglong2(d0[0], d0[1]);
    *reinterpret_cast<ulonglong2*>(o + ps) = make_ulonglong2(d1[0], d1[1]);
    *reinterpret_cast<ulonglong2*>(o + 2 * ps) = make_ulonglong2(d2[0], d2[1]);
}

// ---------------------------------------------------------------------------
// Diagonal MAC (on-demand BSGS, Eq. eq:prerotation) of one query:
//   P_j[t][i][k] = sum_{i' < n1, j n1 + i' < ell} baby_{i'}[t][i][k] * D'_{j n1 + i'}[i][k]
// A CTA owns TP evaluation points of one limb. The n1 baby words (both polys) of its points are
// staged in shared memory; JG thread groups split the n2 giant steps. The diagonals are streamed,
// U = 8 words a thread at a time (4 on chains with 61-bit primes, where only 4 products sum without
// a carry); when every batch is full (n1 a multiple of U dividing ell), a word's register is refilled
// with the next batch's word as soon as it has been multiplied, so the loads stay in flight.
// Bound by HBM: the diagonals lie in tiles (diag_word), so a CTA reads one contiguous run of ell
// kDiagTile words where rows 6.8 MB apart cost a fifth of the bandwidth, and already as 30-bit
// halves. At the headline size (512 diagonals of 13 limbs, N = 2^16, 4.14 GB) 888 us, 4.67 TB/s ->
// 637 us, 6.50 TB/s (tiles alone 668; 128 points x 4 rows 662; 64 x 8, two CTAs an SM, 666).
// ---------------------------------------------------------------------------
template <int TP, int U>
__global__ void __launch_bounds__(256, 4) k_mac(const u64* __restrict__ babies, int cap_b,
                                                const u64* __restrict__ diags, u64* __restrict__ out, int cap_o,
                                                int nl, int n1, int n2, int ell, int JG,
                                                const DevPrime* __restrict__ primes, int N) {
    pdl_wait();
    pdl_trigger();
    extern __shared__ u64 sb[];  // [n1][2][TP]
    const int pl = threadIdx.x % TP;
    const int jg = threadIdx.x / TP;
    const int k = blockIdx.x * TP + pl;
    const int i = blockIdx.y;
    const u64 q = primes[i].q, qinv = primes[i].qinv, one_s = primes[i].one_s;
    const bool fold_each = n1 > 64;
    // staging: thread (pl, jg) takes point pl of the rows r = 2 i' + t = jg, jg + JG, ... (no
    // index divisions)
    {
        const long long rstep = (long long)cap_b * N;
        const u64* src = babies + (long long)i * N + k;
#pragma unroll 8
        for (int r = jg; r < 2 * n1; r += JG) sb[r * TP + pl] = split30(src[r * rstep]);
    }
    __syncthreads();
    // the thread's work is a sequence of batches (giant step j, U diagonals from i0)
    int j = jg, i0 = 0;
    if (j >= n2) return;
    const u64* sbase = sb + pl;
    Acc128 acc[2] = {};
    // the products of one diagonal word d (both polys of the baby) into p
    auto mul_word = [&](AccK (&p)[2], u64 d, const u64* sq) {
        const u32 dsum = sum30(d);
        mack(p[0], d, dsum, sq[0]);
        mack(p[1], d, dsum, sq[TP]);
    };
    // after a batch of giant step j: add its sums (a product adds less than 2^58 to the high word, so
    // up to 64 per giant step need no fold and the high word is reduced once before the REDC); when
    // the giant step ends, store it
    auto close_batch = [&](AccK (&p)[2], int jc, bool last) {
#pragma unroll
        for (int t = 0; t < 2; ++t) {
            flushk(acc[t], p[t]);
            if (fold_each) fold(acc[t], q);
            if (last) {
                out[((long long)(2 * jc + t) * cap_o + i) * N + k] =
                    redc(mul_shoup(acc[t].hi, 1, one_s, q), acc[t].lo, q, qinv);
                acc[t] = Acc128{0, 0};
            }
        }
    };
    const u64* dbase = diags + diag_word(i, k, 0, ell, N);
    if (ell % n1 == 0 && n1 % U == 0) {
        // every batch is full: while a batch is multiplied, each word's register is refilled with
        // the same word of the next batch, so U loads per thread stay in flight throughout
        u64 d[U];
        {
            const u64* D = dbase + (long long)j * n1 * kDiagTile;
#pragma unroll
            for (int u = 0; u < U; ++u) d[u] = __ldcs(D + u * kDiagTile);
        }
        for (;;) {
            int jn = j, in = i0 + U;
            if (in == n1) {
                jn = j + JG;
                in = 0;
            }
            const bool more = jn < n2;
            const u64* Dn = dbase + (long long)((more ? jn : j) * n1 + (more ? in : i0)) * kDiagTile;
            const u64* s0 = sbase + i0 * 2 * TP;
            AccK p[2] = {};
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const u64 w = d[u];
                if (more) d[u] = __ldcs(Dn + u * kDiagTile);
                mul_word(p, w, s0 + u * 2 * TP);
            }
            close_batch(p, j, jn != j);
            if (!more) break;
            j = jn;
            i0 = in;
        }
        return;
    }
    for (;;) {
        const int cnt = min(n1, ell - j * n1);
        const u64* D = dbase + (long long)(j * n1 + i0) * kDiagTile;
        const u64* s0 = sbase + i0 * 2 * TP;
        AccK p[2] = {};
        if (i0 + U <= cnt) {
            // full batch: no bounds checks
            u64 d[U];
#pragma unroll
            for (int u = 0; u < U; ++u) d[u] = __ldcs(D + u * kDiagTile);
#pragma unroll
            for (int u = 0; u < U; ++u) mul_word(p, d[u], s0 + u * 2 * TP);
        } else {
            for (int u = 0; i0 + u < cnt; ++u) mul_word(p, __ldcs(D + u * kDiagTile), s0 + u * 2 * TP);
        }
        // next batch
        int jn = j, in = i0 + U;
        if (in >= cnt) {
            jn = j + JG;
            in = 0;
        }
        close_batch(p, j, jn != j);
        if (jn >= n2) break;
        j = jn;
        i0 = in;
    }
}

// ---------------------------------------------------------------------------
// Diagonal MAC with the diagonals streamed through shared memory (the on-demand schedule's S4
// for B = 2..4 queries against one database, when n1 is a multiple of SD = 8 and n2 of JG): the
// sums of k_mac, P_{b,j}[t][i][k] = sum_{i'} B_{b,i'}[t][i][k] * D'_{j n1 + i'}[i][k], every
// diagonal word read once for all B queries. A CTA owns TP points of one limb and JG giant-step
// rows: thread (jg, point) accumulates giant steps jb JG + jg for its point. The babies of the
// CTA's points are staged once (30-bit halves, every query); the diagonals flow through a ring of
// kMpNS stages, stage (jb, i0) holding diagonals (jb JG + jg) n1 + i0 + u for jg < JG, u < SD,
// filled by 16-byte asynchronous copies (cp.async, one commit group per stage, kMpNS - 1 stages
// in flight while one is multiplied). A warp reads TP consecutive words of one row: no bank
// conflicts, and no exchange between threads until a giant step's sums are complete.
// ---------------------------------------------------------------------------
constexpr int kMpNS = 4;  // ring stages
constexpr int kMpSD = 8;  // diagonals of one giant step per stage (8 products between carries)

__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
    const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int PENDING>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(PENDING) : "memory"); }

template <int B, int TP, int JG>
__global__ void __launch_bounds__(TP * JG) k_mac_pipe(const u64* __restrict__ babies, long long baby_q, int cap_b,
                                                      const u64* __restrict__ diags, u64* __restrict__ out,
                                                      long long out_q, int cap_o, int n1, int n2,
                                                      const DevPrime* __restrict__ primes, int N) {
    pdl_wait();
    pdl_trigger();
    constexpr int SD = kMpSD;
    const int ell = n1 * n2;
    constexpr int NT = TP * JG;                       // threads
    constexpr int ROWS = JG * SD;                     // diagonal rows per stage
    constexpr int CHUNKS = ROWS * TP / 2;             // 16-byte chunks per stage
    static_assert(CHUNKS % NT == 0, "whole chunks per thread");
    extern __shared__ __align__(16) u64 smp[];
    u64* sb = smp;                                    // babies [B][n1][2][TP], split
    u64* sd = sb + (size_t)B * n1 * 2 * TP;           // ring [NS][JG][SD][TP]
    const int i = blockIdx.y;
    const int k0 = blockIdx.x * TP;
    const int pl = threadIdx.x % TP, jg = threadIdx.x / TP;
    const u64 q = primes[i].q, qinv = primes[i].qinv;
    const int spb = n1 / SD;                          // stages per giant-step block
    const int nst = (n2 / JG) * spb;
    const int per_q = n1 * 2 * TP;
    auto issue = [&](int s) {
        if (s < nst) {
            const int jb = s / spb, i0 = (s % spb) * SD;
            u64* dst = sd + (size_t)(s % kMpNS) * ROWS * TP;
#pragma unroll
            for (int r = 0; r < CHUNKS / NT; ++r) {
                const int ch = threadIdx.x + r * NT;
                const int row = ch / (TP / 2), w = (ch % (TP / 2)) * 2;
                const int g = row / SD, u = row % SD;
                const long long d = (long long)(jb * JG + g) * n1 + i0 + u;
                cp_async16(dst + (size_t)row * TP + w, diags + diag_word(i, k0, d, ell, N) + w);
            }
        }
        cp_async_commit();  // an empty group past the last stage keeps the group count uniform
    };
#pragma unroll
    for (int s = 0; s < kMpNS - 1; ++s) issue(s);
    for (int e = threadIdx.x; e < B * per_q; e += NT) {
        const int qb = e / per_q, r = e % per_q;
        const int ib = r / (2 * TP), t = (r / TP) & 1, pp = r % TP;
        sb[e] = split30(babies[(long long)qb * baby_q + ((long long)ib * 2 + t) * cap_b * N + (long long)i * N + k0 + pp]);
    }
    Acc128 acc[B][2];
#pragma unroll
    for (int qb = 0; qb < B; ++qb) acc[qb][0] = acc[qb][1] = Acc128{0, 0};
    for (int s = 0; s < nst; ++s) {
        cp_async_wait<kMpNS - 2>();  // this thread's copies of stage s have landed
        __syncthreads();             // every thread's have; slot (s - 1) % NS is free again
        issue(s + kMpNS - 1);
        const int jb = s / spb, i0 = (s % spb) * SD;
        const u64* st = sd + (size_t)(s % kMpNS) * ROWS * TP + (size_t)jg * SD * TP + pl;
        AccK p[B][2];
#pragma unroll
        for (int qb = 0; qb < B; ++qb) p[qb][0] = p[qb][1] = AccK{0, 0, 0};
#pragma unroll
        for (int u = 0; u < SD; ++u) {
            const u64 ds = st[(size_t)u * TP];
            const u32 dsum = sum30(ds);
#pragma unroll
            for (int qb = 0; qb < B; ++qb) {
                const u64* sq = sb + (size_t)qb * per_q + ((size_t)(i0 + u) * 2) * TP + pl;
                mack(p[qb][0], ds, dsum, sq[0]);
                mack(p[qb][1], ds, dsum, sq[TP]);
            }
        }
#pragma unroll
        for (int qb = 0; qb < B; ++qb) {
            flushk(acc[qb][0], p[qb][0]);
            flushk(acc[qb][1], p[qb][1]);
            fold(acc[qb][0], q);
            fold(acc[qb][1], q);
        }
        if (i0 + SD == n1) {
            // giant step jb JG + jg complete for this point: reduce and store
            const int j = jb * JG + jg;
#pragma unroll
            for (int qb = 0; qb < B; ++qb) {
                u64* O = out + (long long)qb * out_q + (long long)j * 2 * cap_o * N;
                O[(long long)i * N + k0 + pl] = redc(acc[qb][0].hi, acc[qb][0].lo, q, qinv);
                O[((long long)cap_o + i) * N + k0 + pl] = redc(acc[qb][1].hi, acc[qb][1].lo, q, qinv);
                acc[qb][0] = acc[qb][1] = Acc128{0, 0};
            }
        }
    }
    cp_async_wait<0>();
}

// ---------------------------------------------------------------------------
// Diagonal MAC as a persistent pipeline (the on-demand schedule's S4 for B = 2..4 queries against
// one database): the sums of k_mac, P_{b,j}[t][i][k] = sum_{i'} B_{b,i'}[t][i][k] D'_{j n1 + i'}[i][k].
// A tile is TP = 16 points of one limb; each CTA runs the tiles blockIdx.x, blockIdx.x + gridDim.x,
// ... with 256 threads, thread (giant-step row jg, point) accumulating giant steps jb 16 + jg. One
// ring of kMrNS stages of 16-byte asynchronous copies carries everything: stage (tile, jb, i0)
// holds diagonals (jb 16 + g) n1 + i0 + u, g < 16, u < 8, and the last stage of a tile also
// carries the next tile's babies (every query, raw residues) into the other of two baby buffers.
// So the copies of the next tile overlap the products of this one, and a CTA never waits for a
// tile's start. The babies of a tile are split into 30-bit halves in shared memory once, after
// they land. Every diagonal word is read once for all B queries. Needs n1 % 8 == 0, n2 % 16 == 0
// and at least kMrNS stages per tile (checked by mac_ring_fits).
// ---------------------------------------------------------------------------
constexpr int kMrNS = 3;   // ring stages
constexpr int kMrTP = 16;  // points per tile
constexpr int kMrJG = 16;  // giant-step rows per CTA

// Cursor over a CTA's stages (tile m, stage sl of the tile), advanced without divisions.
struct MrCursor {
    int m, sl, slot, tile, i, k0;
};

template <int B, int N1>
__global__ void __launch_bounds__(kMrTP * kMrJG) k_mac_ring(const u64* __restrict__ babies, long long baby_q,
                                                            int cap_b, const u64* __restrict__ diags,
                                                            u64* __restrict__ out, long long out_q, int cap_o, int nl,
                                                            int n2, const DevPrime* __restrict__ primes,
                                                            int N) {
    pdl_wait();
    pdl_trigger();
    constexpr int TP = kMrTP, JG = kMrJG, SD = kMpSD, NT = TP * JG, NS = kMrNS;
    constexpr int ROWS = JG * SD;          // diagonal rows per stage
    constexpr int CHUNKS = ROWS * TP / 2;  // 16-byte chunks per stage
    static_assert(CHUNKS % NT == 0, "whole chunks per thread");
    extern __shared__ __align__(16) u64 smr[];
    constexpr int qw = N1 * 2 * TP;        // words of one query's babies in a tile
    constexpr int bw = B * qw;             // words of one tile's babies
    u64* bb = smr;                         // [2][B][N1][2][TP]
    u64* sd = bb + 2 * (size_t)bw;         // ring [NS][JG][SD][TP]
    const int pl = threadIdx.x % TP, jg = threadIdx.x / TP;
    const int tpl = N / TP;                // tiles per limb
    const int ntile = nl * tpl;
    const int mt = (int)blockIdx.x < ntile ? (ntile - 1 - (int)blockIdx.x) / (int)gridDim.x + 1 : 0;
    constexpr int spb = N1 / SD;           // stages per giant-step block
    const int nst = (n2 / JG) * spb;       // stages per tile
    const int ell = n2 * N1;
    auto at_tile = [&](MrCursor& c) {
        c.tile = (int)blockIdx.x + c.m * (int)gridDim.x;
        c.i = c.tile / tpl;
        c.k0 = (c.tile - c.i * tpl) * TP;
    };
    auto advance = [&](MrCursor& c) {
        c.slot = c.slot + 1 == NS ? 0 : c.slot + 1;
        if (++c.sl == nst) {
            c.sl = 0;
            ++c.m;
            at_tile(c);
        }
    };
    auto issue = [&](const MrCursor& c) {
        if (c.m < mt) {
            const int jb = c.sl / spb, i0 = (c.sl - jb * spb) * SD;
            u64* dst = sd + (size_t)c.slot * ROWS * TP;
            const u64* src = diags + diag_word(c.i, c.k0, jb * JG * N1 + i0, ell, N);
#pragma unroll
            for (int r = 0; r < CHUNKS / NT; ++r) {
                const int ch = threadIdx.x + r * NT;
                const int row = ch / (TP / 2), w = (ch % (TP / 2)) * 2;
                const int gg = row / SD, u = row % SD;
                cp_async16(dst + (size_t)row * TP + w, src + (gg * N1 + u) * kDiagTile + w);
            }
            // the babies of tile 0 ride on its first stage, those of tile m + 1 on tile m's last
            const int mb = (c.m == 0 && c.sl == 0) ? 0 : (c.sl == nst - 1 ? c.m + 1 : -1);
            if (mb >= 0 && mb < mt) {
                const int tb = (int)blockIdx.x + mb * (int)gridDim.x, il = tb / tpl, kb = (tb - il * tpl) * TP;
                u64* bd = bb + (size_t)(mb & 1) * bw;
                const u64* bs = babies + (long long)il * N + kb;
                for (int ch = threadIdx.x; ch < bw / 2; ch += NT) {
                    const int e = ch * 2;
                    const int qb = e / qw, r = e - qb * qw;
                    const int row = r / TP, pp = r - row * TP;  // row = 2 ib + t
                    cp_async16(bd + e, bs + (long long)qb * baby_q + (long long)row * cap_b * N + pp);
                }
            }
        }
        cp_async_commit();  // empty groups past the end keep the group count uniform
    };
    MrCursor ic{0, 0, 0, 0, 0, 0};  // issue cursor, NS - 1 stages ahead
    at_tile(ic);
#pragma unroll
    for (int s = 0; s < NS - 1; ++s) {
        issue(ic);
        advance(ic);
    }
    MrCursor cc{0, 0, 0, 0, 0, 0};  // compute cursor
    at_tile(cc);
    Acc128 acc[B][2];
#pragma unroll
    for (int qb = 0; qb < B; ++qb) acc[qb][0] = acc[qb][1] = Acc128{0, 0};
    for (; cc.m < mt; advance(cc)) {
        cp_async_wait<NS - 2>();  // this thread's copies of this stage (and earlier) have landed
        __syncthreads();          // everyone's have; the ring slot before this one is free again
        issue(ic);
        advance(ic);
        u64* bm = bb + (size_t)(cc.m & 1) * bw;
        if (cc.sl == 0) {
            // a new tile: its babies have landed; split them into 30-bit halves in place
            for (int e = threadIdx.x; e < bw; e += NT) bm[e] = split30(bm[e]);
            __syncthreads();
        }
        const int jb = cc.sl / spb, i0 = (cc.sl - jb * spb) * SD;
        const u64* st = sd + (size_t)cc.slot * ROWS * TP + jg * SD * TP + pl;
        const u64* sq = bm + i0 * 2 * TP + pl;
        AccK p[B][2];
#pragma unroll
        for (int qb = 0; qb < B; ++qb) p[qb][0] = p[qb][1] = AccK{0, 0, 0};
#pragma unroll
        for (int u = 0; u < SD; ++u) {
            const u64 ds = st[u * TP];
            const u32 dsum = sum30(ds);
#pragma unroll
            for (int qb = 0; qb < B; ++qb) {
                mack(p[qb][0], ds, dsum, sq[qb * qw + u * 2 * TP]);
                mack(p[qb][1], ds, dsum, sq[qb * qw + u * 2 * TP + TP]);
            }
        }
        // no fold here: a flush adds less than 2^60 to the high word, and a giant step has at
        // most 8 flushes (N1 <= 64), so the high word is reduced once, before the REDC
#pragma unroll
        for (int qb = 0; qb < B; ++qb) {
            flushk(acc[qb][0], p[qb][0]);
            flushk(acc[qb][1], p[qb][1]);
        }
        if (i0 + SD == N1) {
            // giant step jb JG + jg complete for this point: reduce and store
            const DevPrime P = primes[cc.i];
            const int j = jb * JG + jg;
#pragma unroll
            for (int qb = 0; qb < B; ++qb) {
                u64* O = out + (long long)qb * out_q + (long long)j * 2 * cap_o * N + (long long)cc.i * N + cc.k0 + pl;
                O[0] = redc(mul_shoup(acc[qb][0].hi, 1, P.one_s, P.q), acc[qb][0].lo, P.q, P.qinv);
                O[(long long)cap_o * N] = redc(mul_shoup(acc[qb][1].hi, 1, P.one_s, P.q), acc[qb][1].lo, P.q, P.qinv);
                acc[qb][0] = acc[qb][1] = Acc128{0, 0};
            }
        }
    }
    cp_async_wait<0>();
}

// ---------------------------------------------------------------------------
// Encrypted-database MAC (ct x ct with lazy relinearisation, the paper's setting of
// Section 5.3): for every giant step j, pointwise per limb,
//   (d0, d1, d2)_j = sum_{i < n1, j n1 + i < ell} B_i (x) E_{j n1 + i}
//   d0 += b0 e0,  d1 += b0 e1 + b1 e0,  d2 += b1 e1.
// The middle term takes one product (Karatsuba): d1 = sum (b0 + b1)(e0 + e1) - d0 - d2, the
// same residue mod q as the two products it replaces.
// babies: [n1][2][cap_b][N] evaluation form; diags: component t of ciphertext d is row 2 d + t
// of the tiles of diag_word, whole words in Montgomery form (e0 R + e1 R = (e0 + e1) R), so one
// REDC of each sum gives it in plain form;
// out: [n2][3][cap_o][N]. Tiling as k_mac: the babies of a point tile are staged in shared
// memory as 30-bit halves of b0, b1 and b0 + b1, giant steps run over the thread rows.
// Diagonals go in batches of 4 (one carry step per batch).
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(512, 2) k_mac_ct(const u64* __restrict__ babies, int cap_b,
                                                   const u64* __restrict__ diags, u64* __restrict__ out, int cap_o,
                                                   int nl, int n1, int n2, int ell, int TP, int JG,
                                                   const DevPrime* __restrict__ primes, int N) {
    pdl_wait();
    pdl_trigger();
    extern __shared__ u64 sb[];  // [n1][3][TP]: b0, b1, b0 + b1
    const int pl = threadIdx.x % TP;
    const int jg = threadIdx.x / TP;
    const int k = blockIdx.x * TP + pl;
    const int i = blockIdx.y;
    const u64 q = primes[i].q, qinv = primes[i].qinv;
    // staging: thread (pl, jg) takes point pl of babies jg, jg + JG, ... (no index divisions)
#pragma unroll 4
    for (int ib = jg; ib < n1; ib += JG) {
        const u64* src = babies + (long long)ib * 2 * cap_b * N + (long long)i * N + k;
        const u64 b0 = src[0], b1 = src[(long long)cap_b * N];
        u64* dst = sb + (size_t)ib * 3 * TP + pl;
        dst[0] = split30(b0);
        dst[TP] = split30(b1);
        dst[2 * TP] = split30(add_mod(b0, b1, q));
    }
    __syncthreads();
    constexpr int dstride = 2 * kDiagTile, cstride = kDiagTile;  // one diagonal ciphertext, one component
    for (int j = jg; j < n2; j += JG) {
        const int cnt = min(n1, ell - j * n1);
        const u64* D = diags + diag_word(i, k, 2LL * j * n1, 2 * ell, N);
        Acc128 a0{0, 0}, am{0, 0}, a2{0, 0};
        for (int i0 = 0; i0 < cnt; i0 += 4) {
            AccK p0{0, 0, 0}, pm{0, 0, 0}, p2{0, 0, 0};
            const u64* sq = sb + (size_t)i0 * 3 * TP + pl;
            if (i0 + 4 <= cnt) {
                u64 e0[4], e1[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    e0[u] = __ldcs(D + u * dstride);
                    e1[u] = __ldcs(D + u * dstride + cstride);
                }
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const u64* bq = sq + u * 3 * TP;
                    const u64 x0 = split30(e0[u]), x2 = split30(e1[u]), xm = split30(add_mod(e0[u], e1[u], q));
                    mack(p0, x0, sum30(x0), bq[0]);
                    mack(p2, x2, sum30(x2), bq[TP]);
                    mack(pm, xm, sum30(xm), bq[2 * TP]);
                }
            } else {
                for (int u = 0; i0 + u < cnt; ++u) {
                    const u64 f0 = __ldcs(D + u * dstride), f1 = __ldcs(D + u * dstride + cstride);
                    const u64* bq = sq + u * 3 * TP;
                    const u64 x0 = split30(f0), x2 = split30(f1), xm = split30(add_mod(f0, f1, q));
                    mack(p0, x0, sum30(x0), bq[0]);
                    mack(p2, x2, sum30(x2), bq[TP]);
                    mack(pm, xm, sum30(xm), bq[2 * TP]);
                }
            }
            flushk(a0, p0);
            flushk(am, pm);
            flushk(a2, p2);
            fold(a0, q);
            fold(am, q);
            fold(a2, q);
            D += 4 * dstride;
        }
        const u64 d0 = redc(a0.hi, a0.lo, q, qinv), d2 = redc(a2.hi, a2.lo, q, qinv);
        const u64 dm = redc(am.hi, am.lo, q, qinv);
        u64* O = out + (long long)j * 3 * cap_o * N + (long long)i * N + k;
        O[0] = d0;
        O[(long long)cap_o * N] = sub_mod(sub_mod(dm, d0, q), d2, q);
        O[2LL * cap_o * N] = d2;
    }
}

// ---------------------------------------------------------------------------
// Table-schedule MAC (Algorithm 1, step 4): S_g = sum_{m < ell} rotQ[m] (.) D_{g,m}
// for GG groups per CTA column. One thread per evaluation point of one limb; the two
// table words of a point are read once for the GG groups, the diagonal words streamed.
// table: [ell][2][cap_t][N]; diagonal m of group g at row m of the tiles at diags + g dgrp
// (diag_word; Montgomery form, 30-bit halves); output of group g at out + g og, [2][cap_o][N]. Products use the 30-bit
// split multiply-accumulate (four per carry step).
// ---------------------------------------------------------------------------
template <int GG>
__global__ void __launch_bounds__(256) k_mac_table(const u64* __restrict__ table, int cap_t,
                                                   const u64* __restrict__ diags, long long dgrp, int G,
                                                   u64* __restrict__ out, int cap_o, long long og, int nl, int ell,
                                                   const DevPrime* __restrict__ primes, int N) {
    pdl_wait();
    pdl_trigger();
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    const int i = blockIdx.y;
    const int g0 = blockIdx.z * GG;
    if (k >= N) return;
    const u64 q = primes[i].q, qinv = primes[i].qinv;
    const long long ts = 2ll * cap_t * N;
    const u64* t0 = table + (long long)i * N + k;
    const u64* t1 = t0 + (long long)cap_t * N;
    const u64* d0 = diags + (long long)g0 * dgrp + diag_word(i, k, 0, ell, N);
    Acc128 acc[GG][2];
#pragma unroll
    for (int gg = 0; gg < GG; ++gg) acc[gg][0] = acc[gg][1] = Acc128{0, 0};
    for (int m0 = 0; m0 < ell; m0 += 4) {
        u64 a[4], b[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const bool ok = m0 + u < ell;
            a[u] = split30(ok ? t0[(long long)(m0 + u) * ts] : 0ull);
            b[u] = split30(ok ? t1[(long long)(m0 + u) * ts] : 0ull);
        }
#pragma unroll
        for (int gg = 0; gg < GG; ++gg) {
            if (g0 + gg < G) {
                AccK p0{0, 0, 0}, p1{0, 0, 0};
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const u64 d = m0 + u < ell ? __ldcs(d0 + gg * dgrp + (long long)(m0 + u) * kDiagTile) : 0ull;
                    const u32 dsum = sum30(d);
                    mack(p0, d, dsum, a[u]);
                    mack(p1, d, dsum, b[u]);
                }
                flushk(acc[gg][0], p0);
                flushk(acc[gg][1], p1);
                fold(acc[gg][0], q);
                fold(acc[gg][1], q);
            }
        }
    }
#pragma unroll
    for (int gg = 0; gg < GG; ++gg) {
        if (g0 + gg < G) {
            u64* O = out + (long long)(g0 + gg) * og;
            O[(long long)i * N + k] = redc(acc[gg][0].hi, acc[gg][0].lo, q, qinv);
            O[((long long)cap_o + i) * N + k] = redc(acc[gg][1].hi, acc[gg][1].lo, q, qinv);
        }
    }
}

// ---------------------------------------------------------------------------
// Elementwise helpers on ciphertext batches [B][2][cap][N] (evaluation form).
// ---------------------------------------------------------------------------
// out = a + b over limbs 0..level of both polys
__global__ void k_add(const u64* a, int a_cap, long long a_bs, const u64* b, int b_cap, long long b_bs, u64* out,
                      int o_cap, long long o_bs, int level, const DevPrime* primes, int N) {
    pdl_wait();
    pdl_trigger();
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    const int i = blockIdx.y % (level + 1);
    const int t = blockIdx.y / (level + 1);
    const int bb = blockIdx.z;
    if (k >= N) return;
    const u64 q = primes[i].q;
    const u64 x = a[bb * a_bs + ((long long)t * a_cap + i) * N + k];
    const u64 y = b[bb * b_bs + ((long long)t * b_cap + i) * N + k];
    out[bb * o_bs + ((long long)t * o_cap + i) * N + k] = add_mod(x, y, q);
}

// sum of J ciphertexts (stride js) into out
__global__ void k_sum(const u64* a, int cap, long long js, int J, u64* out, int o_cap, int level,
                      const DevPrime* primes, int N) {
    pdl_wait();
    pdl_trigger();
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    const int i = blockIdx.y % (level + 1);
    const int t = blockIdx.y / (level + 1);
    if (k >= N) return;
    const u64 q = primes[i].q;
    u64 v = 0;
    for (int j = 0; j < J; ++j) v = add_mod(v, a[j * js + ((long long)t * cap + i) * N + k], q);
    out[((long long)t * o_cap + i) * N + k] = v;
}

// Lifted last limbs of the Chebyshev leaves, T1 cb_j + ca_j at limb l, from u, the coefficient
// form of T1's last limb ([B][2][N]): the INTT is linear and the constant ca_j is the constant
// polynomial, so the leaf's last limb in coefficient form is cb_{j,l} u + ca_{j,l} at coefficient 0
// of component 0; centered and reduced to q_i for i < l as in k_rescale_lift.
// lifted [B nl][2][l][N]; grid (N / 256, 2 nl, B).
__global__ void k_leaf_lift(const u64* __restrict__ u, const u64* __restrict__ cb, const u64* __restrict__ cb_s,
                            const u64* __restrict__ ca, int nl, int L1, u64* __restrict__ lifted,
                            const RescaleTab* __restrict__ tab, const DevPrime* __restrict__ primes, int l, int N) {
    pdl_wait();
    pdl_trigger();
    const u64 ql = primes[l].q;
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    const int j = blockIdx.y >> 1, t = blockIdx.y & 1, b = blockIdx.z;
    if (k >= N) return;
    u64 r = mul_shoup(u[((long long)b * 2 + t) * N + k], cb[j * L1 + l], cb_s[j * L1 + l], ql);
    if (t == 0 && k == 0) r = add_mod(r, ca[j * L1 + l], ql);
    u64* o = lifted + ((((long long)b * nl + j) * 2 + t) * l) * N + k;
    for (int i = 0; i < l; ++i) o[(long long)i * N] = centered_residue(r, *tab, primes[i], i);
}

// x to Montgomery form (evaluation keys)
__global__ void k_to_mont(u64* x, long long n_per_poly, PrimeMap pm, const DevPrime* primes, long long total) {
    pdl_wait();
    pdl_trigger();
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < total;
         e += (long long)gridDim.x * blockDim.x) {
        const int p = (int)(e / n_per_poly);
        const DevPrime P = primes[pm.idx[p % pm.period]];
        x[e] = to_mont(x[e], P);
    }
}

// ciphertext polynomials src [rows][nl][N] in Montgomery form into rows row0, row0 + 1, ... of the
// tiles of a database of `total` rows
__global__ void __launch_bounds__(kThreads) k_tile_mont(const u64* __restrict__ src, u64* __restrict__ diags,
                                                        long long row0, int total, int nl,
                                                        const DevPrime* __restrict__ primes, int N) {
    pdl_wait();
    pdl_trigger();
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    const int i = blockIdx.y, r = blockIdx.z;
    if (k >= N) return;
    diags[diag_word(i, k, row0 + r, total, N)] = to_mont(src[((long long)r * nl + i) * N + k], primes[i]);
}

// ---------------------------------------------------------------------------
// Device slot encoder for template diagonals (reading R5, same operations and
// order as the host encoder: inverse special FFT stages len = n..2, bit
// reversal, times 1/n and Delta, rounded half away from zero).
// Stage arithmetic uses explicitly rounded intrinsics (no contraction).
// ---------------------------------------------------------------------------
struct cplx {
    double r, i;
};

__device__ __forceinline__ void fft_inv_bfly(cplx& a, cplx& b, double wr, double wi) {
    const double sr = __dadd_rn(a.r, b.r), si = __dadd_rn(a.i, b.i);
    const double dr = __dsub_rn(a.r, b.r), di = __dsub_rn(a.i, b.i);
    a.r = sr;
    a.i = si;
    b.r = __dsub_rn(__dmul_rn(dr, wr), __dmul_rn(di, wi));
    b.i = __dadd_rn(__dmul_rn(dr, wi), __dmul_rn(di, wr));
}

// Gather of the pre-rotated diagonals into slot vectors:
// z[x] = diag_d(M_k)[(x - shift) mod n], diag_d(M_k)[b ell + r] = T[(k B + b) ell + r][(r + d) mod ell]
__global__ void k_diag_gather(const float* __restrict__ T, long long K, int ell, int n, long long grp, int d0, int nd,
                              int n1, cplx* __restrict__ z) {
    pdl_wait();
    pdl_trigger();
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int di = blockIdx.y;
    if (x >= n || di >= nd) return;
    const int d = d0 + di;
    const long long shift = (long long)(d / n1) * n1;
    long long y = ((long long)x - shift) % n;
    if (y < 0) y += n;
    const long long B = n / ell;
    const long long b = y / ell, r = y % ell;
    const long long row = (grp * B + b) * ell + r;
    const double v = row < K ? (double)T[row * ell + (r + d) % ell] : 0.0;
    z[(long long)di * n + x] = cplx{v, 0.0};
}

// first log2(R) stages (len = n .. 2n/R): columns of stride n/R; one tile of 16 columns
__global__ void __launch_bounds__(256) k_fft_col(cplx* z, int logn, int logR, const unsigned* rot, const double* zr,
                                                 const double* zi) {
    pdl_wait();
    pdl_trigger();
    extern __shared__ cplx sc[];
    const int n = 1 << logn, Rr = 1 << logR, C = n >> logR;
    const int TC = 16;
    const long long M = 4ll * n;
    cplx* x = z + (long long)blockIdx.y * n;
    const int col0 = blockIdx.x * TC;
    for (int e = threadIdx.x; e < Rr * TC; e += blockDim.x) {
        int r = e / TC, c = e % TC;
        sc[e] = x[(long long)r * C + col0 + c];
    }
    __syncthreads();
    for (int len = n; len >= 2 * C; len >>= 1) {
        const int hrow = (len >> 1) / C;  // half block in rows
        const long long lq = (long long)len << 2, gap = M / lq;  // powers of two
        for (int bf = threadIdx.x; bf < (Rr >> 1) * TC; bf += blockDim.x) {
            int c = bf % TC, pr = bf / TC;
            int blk = pr / hrow, u = pr - blk * hrow;
            int ra = blk * 2 * hrow + u, rb = ra + hrow;
            const int j = (col0 + c) + u * C;  // position inside the len-block
            const long long idx = (lq - (long long)(rot[j] & (unsigned)(lq - 1))) * gap;
            fft_inv_bfly(sc[ra * TC + c], sc[rb * TC + c], zr[idx], zi[idx]);
        }
        __syncthreads();
    }
    for (int e = threadIdx.x; e < Rr * TC; e += blockDim.x) {
        int r = e / TC, c = e % TC;
        x[(long long)r * C + col0 + c] = sc[e];
    }
}

// remaining stages (len = C .. 2) inside contiguous blocks of C
__global__ void __launch_bounds__(256) k_fft_row(cplx* z, int logn, int logR, int bpc, const unsigned* rot,
                                                 const double* zr, const double* zi) {
    pdl_wait();
    pdl_trigger();
    extern __shared__ cplx sc[];
    const int n = 1 << logn, C = n >> logR;
    const long long M = 4ll * n;
    cplx* x = z + (long long)blockIdx.y * n + (long long)blockIdx.x * bpc * C;
    const int tile = bpc * C;
    for (int e = threadIdx.x; e < tile; e += blockDim.x) sc[e] = x[e];
    __syncthreads();
    for (int len = C; len >= 2; len >>= 1) {
        const int h = len >> 1;
        const long long lq = (long long)len << 2, gap = M / lq;
        for (int bf = threadIdx.x; bf < tile / 2; bf += blockDim.x) {
            int blk = bf / h, u = bf - blk * h;
            int a = blk * len + u, b = a + h;
            const long long idx = (lq - (long long)(rot[u] & (unsigned)(lq - 1))) * gap;
            fft_inv_bfly(sc[a], sc[b], zr[idx], zi[idx]);
        }
        __syncthreads();
    }
    for (int e = threadIdx.x; e < tile; e += blockDim.x) x[e] = sc[e];
}

// v 2^shift rounded half away from zero. Both factors of the encoder (1/n and Delta) are powers
// of two, so the product is exact and the rounding is a shift of the mantissa: GB300 has two FP64
// lanes an SM, and two multiplications and llround per coefficient cost more than the
// rest of the kernel. Values that do not fit go through the FP64 form.
__device__ __forceinline__ long long scale_round(double v, int shift) {
    const u64 b = (u64)__double_as_longlong(v);
    const int ex = (int)(b >> 52) & 0x7ff, s = ex - 1075 + shift;  // |v| = m 2^(ex - 1075)
    if (ex == 0x7ff || s > 9) return llround(ldexp(v, shift));
    if (ex == 0 || s < -63) return 0;
    const u64 m = (b & 0xfffffffffffffull) | (1ull << 52);
    const u64 r = s >= 0 ? m << s : (m + (1ull << (-s - 1))) >> -s;
    return (b >> 63) ? -(long long)r : (long long)r;
}

// coefficient c of the encoded diagonal di: bit reversal, times 1/n and Delta, rounded half
// away from zero
__device__ __forceinline__ long long fft_coef(const cplx* __restrict__ z, int logn, int di, int c, int scale_bits) {
    const int n = 1 << logn;
    const int cc = c < n ? c : c - n;
    const int src = __brev(cc) >> (32 - logn);
    const cplx w = z[(long long)di * n + src];
    return scale_round(c < n ? w.r : w.i, scale_bits - logn);
}

// m mod q for a signed coefficient: |m| < 2^63 reduced by its bits from bits(q) up where that is
// enough for the prime (13 issue cycles a warp against 44), else with the Shoup quotient of 1
__device__ __forceinline__ u64 coef_residue(long long m, const DevPrime& P) {
    const bool neg = m < 0;
    const u64 a = neg ? (u64)(-(m + 1)) : (u64)m;
    u64 ra;
    if (P.fold63) {
        const u64 f = fold_top(a, P.bsh, P.c);
        ra = min(f, f - P.q);
    } else {
        ra = mul_shoup(a, 1, P.one_s, P.q);
    }
    return neg ? P.q - 1 - ra : ra;
}

// rounding and residues: out [nd][nl][N] (coefficient form)
__global__ void k_fft_finish(const cplx* __restrict__ z, int logn, int nd, u64* __restrict__ out, int nl,
                             const DevPrime* __restrict__ primes, int scale_bits) {
    pdl_wait();
    pdl_trigger();
    const int N = 2 << logn;
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    const int di = blockIdx.y;
    if (c >= N || di >= nd) return;
    const long long m = fft_coef(z, logn, di, c, scale_bits);
    u64* o = out + (long long)di * nl * N;
    for (int i = 0; i < nl; ++i) o[(long long)i * N + c] = coef_residue(m, primes[i]);
}

// rounding only: the integer coefficients m [nd][N] (storage tier B)
__global__ void k_fft_round(const cplx* __restrict__ z, int logn, int nd, long long* __restrict__ out,
                            int scale_bits) {
    pdl_wait();
    pdl_trigger();
    const int N = 2 << logn;
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    const int di = blockIdx.y;
    if (c >= N || di >= nd) return;
    out[(long long)di * N + c] = fft_coef(z, logn, di, c, scale_bits);
}

// residues of stored integer coefficients: m [nd][N] -> out [nd][nl][N]
__global__ void k_coef_residues(const long long* __restrict__ m, int nd, u64* __restrict__ out, int nl,
                                const DevPrime* __restrict__ primes, int N) {
    pdl_wait();
    pdl_trigger();
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    const int di = blockIdx.y;
    if (c >= N || di >= nd) return;
    const long long v = m[(long long)di * N + c];
    u64* o = out + (long long)di * nl * N;
    for (int i = 0; i < nl; ++i) o[(long long)i * N + c] = coef_residue(v, primes[i]);
}

}  // namespace

// ===========================================================================
// launchers
// ===========================================================================

// blocks of the base conversions: 2 points a thread
static unsigned bconv_blocks(int N) { return (unsigned)((N + kBcThreads * kBcW - 1) / (kBcThreads * kBcW)); }

void launch_modup(const u64* in, long long in_job, u64* ext, const ModUpTab* tabs, int beta, int npos, int N, int J,
                  bool scaled, cudaStream_t s) {
    // positions a block: all of them once the (job, digit) blocks alone give every SM 16 blocks,
    // fewer for small batches (each chunk re-reads the digit's limbs)
    const long long blocks = (long long)bconv_blocks(N) * beta * J;
    int chunks = 1;
    while (chunks < npos && blocks * chunks < 152 * 16) ++chunks;
    const int per = (npos + chunks - 1) / chunks;
    dim3 g(bconv_blocks(N), beta * ((npos + per - 1) / per), J);
    if (scaled) launch_k(k_modup<true>, dim3(g), dim3(kBcThreads), 0, s, in, in_job, ext, tabs, beta, npos, N, per);
    else launch_k(k_modup<false>, dim3(g), dim3(kBcThreads), 0, s, in, in_job, ext, tabs, beta, npos, N, per);
}

void launch_ip(const IPJobs& jobs, int beta, int npos, int level, int kp, int T, const DevPrime* primes,
               const PrimeMap& pos_prime, int logN, cudaStream_t s, const u64* pmod, const u64* pmod_s) {
    const int N = 1 << logN;
    dim3 g((N / 2 + kIpThreads - 1) / kIpThreads, jobs.ngroups, npos);
    const int pbase = npos > level + 1 ? pos_prime.idx[level + 1] : 0;
    switch (beta) {
#define FR_IP_CASE(B) \
    case B: launch_k(k_ip<B>, g, dim3(kIpThreads), 0, s, jobs, npos, level, kp, T, primes, pbase, logN, pmod, pmod_s); \
        break;
        FR_IP_CASE(1) FR_IP_CASE(2) FR_IP_CASE(3) FR_IP_CASE(4) FR_IP_CASE(5) FR_IP_CASE(6) FR_IP_CASE(7)
        default: launch_k(k_ip<8>, g, dim3(kIpThreads), 0, s, jobs, npos, level, kp, T, primes, pbase, logN, pmod, pmod_s);
            break;
#undef FR_IP_CASE
    }
}

void launch_ip_sum(const IPSumJobs& jobs, int beta, int npos, int level, int kp, int T, const DevPrime* primes,
                   const PrimeMap& pos_prime, int logN, const u64* pmod, const u64* pmod_s, cudaStream_t s) {
    const int N = 1 << logN;
    dim3 g((N / 2 + kIpThreads - 1) / kIpThreads, jobs.ngroups, npos);
    const int pbase = npos > level + 1 ? pos_prime.idx[level + 1] : 0;
    switch (beta) {
#define FR_IPS_CASE(B) \
    case B: launch_k(k_ip_sum<B>, g, dim3(kIpThreads), 0, s, jobs, npos, level, kp, T, primes, pbase, logN, pmod, pmod_s); \
        break;
        FR_IPS_CASE(1) FR_IPS_CASE(2) FR_IPS_CASE(3) FR_IPS_CASE(4) FR_IPS_CASE(5) FR_IPS_CASE(6) FR_IPS_CASE(7)
        default: launch_k(k_ip_sum<8>, g, dim3(kIpThreads), 0, s, jobs, npos, level, kp, T, primes, pbase, logN, pmod,
                          pmod_s);
            break;
#undef FR_IPS_CASE
    }
}

void launch_p2q(const u64* acc, long long acc_job, int npos, int level, u64* conv, const P2QTab* tab, int N, int J,
                cudaStream_t s) {
    dim3 g(bconv_blocks(N), 2, J);
    launch_k(k_p2q, dim3(g), dim3(kBcThreads), 0, s, acc, acc_job, npos, level, conv, tab, N);
}

void launch_p2q_lift(const u64* acc, long long acc_job, int npos, const u64* zc, u64* y, const P2QTab* tab_rs,
                     const RescaleTab* rtab, u64 ql, int l, int N, int J, cudaStream_t s) {
    dim3 g(bconv_blocks(N), 2, J);
    launch_k(k_p2q_lift, dim3(g), dim3(kBcThreads), 0, s, acc, acc_job, npos, zc, y, tab_rs, rtab, ql, l, N);
}

void launch_baby0_pq(u64* babies, long long baby_q, const u64* q, long long q_bs, int q_cap, int B, int npos,
                     int level, const DevPrime* primes, const u64* pmod, const u64* pmod_s, int N, cudaStream_t s) {
    dim3 g((N + kThreads - 1) / kThreads, npos, 2 * B);
    launch_k(k_baby0_pq, g, dim3(kThreads), 0, s, babies, baby_q, q, q_bs, q_cap, npos, level, primes, pmod, pmod_s, N);
}

void launch_rescale_lift(const u64* last, u64* lifted, const RescaleTab* tab, const DevPrime* primes, int l, int N,
                         int BT, cudaStream_t s) {
    dim3 g((N + kThreads - 1) / kThreads, BT);
    launch_k(k_rescale_lift, dim3(g), dim3(kThreads), 0, s, last, lifted, tab, primes, l, N);
}

void launch_tensor(const TensorJobs& jobs, int J, int level, const DevPrime* primes, int N, cudaStream_t s) {
    dim3 g((N / 2 + kBcThreads - 1) / kBcThreads, level + 1, J);
    launch_k(k_tensor, dim3(g), dim3(kBcThreads), 0, s, jobs, level, primes, N);
}

template <int TP, int U>
static void launch_mac_t(const u64* babies, int cap_b, const u64* diags, u64* out, int cap_o, int nl, int n1, int n2,
                         int ell, const DevPrime* primes, int N, cudaStream_t s) {
    const int JG = std::max(1, std::min(256 / TP, n2));
    const size_t sm = (size_t)n1 * 2 * TP * sizeof(u64);
    static std::atomic<unsigned long long> attr{0};
    smem_limit_once(k_mac<TP, U>, 200 * 1024, attr);
    launch_k(k_mac<TP, U>, dim3(N / TP, nl), dim3(TP * JG), sm, s, babies, cap_b, diags, out, cap_o, nl, n1, n2, ell, JG,
             primes, N);
}

static size_t mac_ring_smem(int B, int n1) {
    return ((size_t)2 * B * n1 * 2 * kMrTP + (size_t)kMrNS * kMrJG * kMpSD * kMrTP) * sizeof(u64);
}

bool mac_ring_fits(int n1, int ell, int N, int B, bool wide) {
    if (wide) return false;  // it sums eight products between carries
    // instantiated for n1 = 32 (the headline BSGS split); other splits take k_mac_pipe or k_mac
    if (n1 != 32 || ell % n1 != 0 || N % kMrTP != 0 || B < 2 || B > 4) return false;
    const int n2 = ell / n1;
    if (n1 > 64 || n2 % kMrJG != 0 || (n2 / kMrJG) * (n1 / kMpSD) < kMrNS) return false;
    return mac_ring_smem(B, n1) <= 200u * 1024;
}

template <int B>
static void launch_mac_ring_t(const u64* babies, long long baby_q, int cap_b, const u64* diags, u64* out,
                              long long out_q, int cap_o, int nl, int n1, int n2, const DevPrime* primes, int N,
                              cudaStream_t s) {
    const size_t sm = mac_ring_smem(B, n1);
    static std::atomic<unsigned long long> attr{0};
    smem_limit_once(k_mac_ring<B, 32>, 200 * 1024, attr);
    // persistent grid: as many CTAs as fit on the GPU at once, capped by the tile count
    int dev = 0, sms = 0, per = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_mac_ring<B, 32>, kMrTP * kMrJG, sm);
    const long long ntile = (long long)nl * (N / kMrTP);
    const int grid = (int)std::min<long long>(ntile, (long long)std::max(1, per) * std::max(1, sms));
    launch_k(k_mac_ring<B, 32>, dim3(grid), dim3(kMrTP * kMrJG), sm, s, babies, baby_q, cap_b, diags, out, out_q,
             cap_o, nl, n2, primes, N);
}

void launch_mac_ring(const u64* babies, long long baby_q, int cap_b, const u64* diags, u64* out, long long out_q,
                     int cap_o, int nl, int n1, int ell, int B, const DevPrime* primes, int N, cudaStream_t s) {
    const int n2 = ell / n1;
    switch (B) {
        case 2: launch_mac_ring_t<2>(babies, baby_q, cap_b, diags, out, out_q, cap_o, nl, n1, n2, primes, N, s); break;
        case 3: launch_mac_ring_t<3>(babies, baby_q, cap_b, diags, out, out_q, cap_o, nl, n1, n2, primes, N, s); break;
        case 4: launch_mac_ring_t<4>(babies, baby_q, cap_b, diags, out, out_q, cap_o, nl, n1, n2, primes, N, s); break;
        default: break;  // the engine splits larger batches
    }
}

bool mac_pipe_fits(int n1, int ell, int N, bool wide) {
    if (wide) return false;  // as the ring
    const int n2 = n1 > 0 ? ell / n1 : 0;
    return n1 % kMpSD == 0 && n1 <= 64 && ell % n1 == 0 && n2 % 4 == 0 && N % 64 == 0;
}

// TP points x JG giant-step rows per CTA:
// 16 points x 16 rows when the giant steps come in blocks of 16 (256 threads; 8 B KiB of staged
// babies and a 64 KiB ring, so two CTAs, 16 warps, share an SM), else 32 points x 4 rows.
template <int B, int TP, int JG>
static void launch_mac_pipe_s(const u64* babies, long long baby_q, int cap_b, const u64* diags, u64* out,
                              long long out_q, int cap_o, int nl, int n1, int n2, const DevPrime* primes, int N,
                              cudaStream_t s) {
    const size_t sm = ((size_t)B * n1 * 2 * TP + (size_t)kMpNS * JG * kMpSD * TP) * sizeof(u64);
    // the limit is raised once per device, so to the most any n1 <= 64 needs (200 KiB)
    static std::atomic<unsigned long long> attr{0};
    smem_limit_once(k_mac_pipe<B, TP, JG>, 200 * 1024, attr);
    dim3 g(N / TP, nl);
    launch_k(k_mac_pipe<B, TP, JG>, g, dim3(TP * JG), sm, s, babies, baby_q, cap_b, diags, out, out_q, cap_o, n1, n2,
             primes, N);
}

template <int B>
static void launch_mac_pipe_t(const u64* babies, long long baby_q, int cap_b, const u64* diags, u64* out,
                              long long out_q, int cap_o, int nl, int n1, int n2, const DevPrime* primes, int N,
                              cudaStream_t s) {
    if (n2 % 16 == 0 && N % 16 == 0)
        launch_mac_pipe_s<B, 16, 16>(babies, baby_q, cap_b, diags, out, out_q, cap_o, nl, n1, n2, primes, N, s);
    else
        launch_mac_pipe_s<B, 32, 4>(babies, baby_q, cap_b, diags, out, out_q, cap_o, nl, n1, n2, primes, N, s);
}

void launch_mac_pipe(const u64* babies, long long baby_q, int cap_b, const u64* diags, u64* out, long long out_q,
                     int cap_o, int nl, int n1, int ell, int B, const DevPrime* primes, int N, cudaStream_t s) {
    const int n2 = ell / n1;
    switch (B) {
        case 2: launch_mac_pipe_t<2>(babies, baby_q, cap_b, diags, out, out_q, cap_o, nl, n1, n2, primes, N, s); break;
        case 3: launch_mac_pipe_t<3>(babies, baby_q, cap_b, diags, out, out_q, cap_o, nl, n1, n2, primes, N, s); break;
        case 4: launch_mac_pipe_t<4>(babies, baby_q, cap_b, diags, out, out_q, cap_o, nl, n1, n2, primes, N, s); break;
        default: break;  // the engine splits larger batches
    }
}

template <int U>
static void launch_mac_u(const u64* babies, int cap_b, const u64* diags, u64* out, int cap_o, int nl, int n1, int n2,
                         int ell, const DevPrime* primes, int N, cudaStream_t s) {
    // points per CTA: a whole tile unless its staged babies (n1 2 TP words) exceed 128 KiB
    const int TP = n1 <= 128 ? 64 : n1 <= 256 ? 32 : 16;
    if (TP == 64) launch_mac_t<64, U>(babies, cap_b, diags, out, cap_o, nl, n1, n2, ell, primes, N, s);
    else if (TP == 32) launch_mac_t<32, U>(babies, cap_b, diags, out, cap_o, nl, n1, n2, ell, primes, N, s);
    else launch_mac_t<16, U>(babies, cap_b, diags, out, cap_o, nl, n1, n2, ell, primes, N, s);
}

void launch_mac(const u64* babies, int cap_b, const u64* diags, u64* out, int cap_o, int nl, int n1, int n2, int ell,
                bool wide, const DevPrime* primes, int N, cudaStream_t s) {
    if (wide) launch_mac_u<4>(babies, cap_b, diags, out, cap_o, nl, n1, n2, ell, primes, N, s);
    else launch_mac_u<8>(babies, cap_b, diags, out, cap_o, nl, n1, n2, ell, primes, N, s);
}

void launch_mac_ct(const u64* babies, int cap_b, const u64* diags, u64* out, int cap_o, int nl, int n1, int n2, int ell,
                   const DevPrime* primes, int N, cudaStream_t s) {
    // points per CTA: staged babies (n1 3 TP words) within 128 KiB; giant-step rows up to 512 threads
    int TP = 128;
    while (TP > 16 && (size_t)n1 * 3 * TP * 8 > (128u << 10)) TP >>= 1;
    int JG = 512 / TP;
    if (JG > n2) JG = n2;
    if (JG < 1) JG = 1;
    const size_t sm = (size_t)n1 * 3 * TP * sizeof(u64);
    static std::atomic<unsigned long long> attr{0};
    smem_limit_once(k_mac_ct, 200 * 1024, attr);
    dim3 g(N / TP, nl);
    launch_k(k_mac_ct, dim3(g), dim3(TP * JG), sm, s, babies, cap_b, diags, out, cap_o, nl, n1, n2, ell, TP, JG, primes, N);
}

void launch_mac_table(const u64* table, int cap_t, const u64* diags, long long dgrp, int G, u64* out, int cap_o,
                      long long og, int nl, int ell, const DevPrime* primes, int N, cudaStream_t s) {
    const int GG = G >= 8 ? 8 : G >= 4 ? 4 : G >= 2 ? 2 : 1;
    dim3 g((N + kThreads - 1) / kThreads, nl, (G + GG - 1) / GG);
    switch (GG) {
        case 8: launch_k(k_mac_table<8>, dim3(g), dim3(kThreads), 0, s, table, cap_t, diags, dgrp, G, out, cap_o, og, nl, ell, primes, N); break;
        case 4: launch_k(k_mac_table<4>, dim3(g), dim3(kThreads), 0, s, table, cap_t, diags, dgrp, G, out, cap_o, og, nl, ell, primes, N); break;
        case 2: launch_k(k_mac_table<2>, dim3(g), dim3(kThreads), 0, s, table, cap_t, diags, dgrp, G, out, cap_o, og, nl, ell, primes, N); break;
        default: launch_k(k_mac_table<1>, dim3(g), dim3(kThreads), 0, s, table, cap_t, diags, dgrp, G, out, cap_o, og, nl, ell, primes, N); break;
    }
}

void launch_add(const u64* a, int a_cap, long long a_bs, const u64* b, int b_cap, long long b_bs, u64* out, int o_cap,
                long long o_bs, int level, int B, const DevPrime* primes, int N, cudaStream_t s) {
    dim3 g((N + kThreads - 1) / kThreads, 2 * (level + 1), B);
    launch_k(k_add, dim3(g), dim3(kThreads), 0, s, a, a_cap, a_bs, b, b_cap, b_bs, out, o_cap, o_bs, level, primes, N);
}

void launch_sum(const u64* a, int cap, long long js, int J, u64* out, int o_cap, int level, const DevPrime* primes,
                int N, cudaStream_t s) {
    dim3 g((N + kThreads - 1) / kThreads, 2 * (level + 1));
    launch_k(k_sum, dim3(g), dim3(kThreads), 0, s, a, cap, js, J, out, o_cap, level, primes, N);
}

void launch_leaf_lift(const u64* u, const u64* cb, const u64* cb_s, const u64* ca, int nl, int L1, u64* lifted,
                      const RescaleTab* tab, const DevPrime* primes, int l, int N, int B, cudaStream_t s) {
    dim3 g((N + kThreads - 1) / kThreads, 2 * nl, B);
    launch_k(k_leaf_lift, dim3(g), dim3(kThreads), 0, s, u, cb, cb_s, ca, nl, L1, lifted, tab, primes, l, N);
}

void launch_to_mont(u64* x, long long n_per_poly, const PrimeMap& pm, const DevPrime* primes, long long total,
                    cudaStream_t s) {
    long long blocks = (total + kThreads - 1) / kThreads;
    if (blocks > 152 * 32) blocks = 152 * 32;
    launch_k(k_to_mont, dim3((unsigned)blocks), dim3(kThreads), 0, s, x, n_per_poly, pm, primes, total);
}

void launch_tile_mont(const u64* src, int rows, u64* diags, long long row0, int total, int nl, const DevPrime* primes,
                      int N, cudaStream_t s) {
    dim3 g((N + kThreads - 1) / kThreads, nl, rows);
    launch_k(k_tile_mont, g, dim3(kThreads), 0, s, src, diags, row0, total, nl, primes, N);
}

void launch_encode_fft(const float* T, long long K, int ell, int logn, long long grp, int d0, int nd, int n1, void* zbuf,
                       const unsigned* rot, const double* zr, const double* zi, cudaStream_t s) {
    cplx* z = (cplx*)zbuf;
    const int n = 1 << logn;
    {
        dim3 g((n + kThreads - 1) / kThreads, nd);
        launch_k(k_diag_gather, dim3(g), dim3(kThreads), 0, s, T, K, ell, n, grp, d0, nd, n1, z);
    }
    const int logR = logn / 2;
    const int Rr = 1 << logR, C = n >> logR;
    {
        dim3 g(C / 16, nd);
        const size_t sm = (size_t)Rr * 16 * sizeof(cplx);
        launch_k(k_fft_col, dim3(g), dim3(256), sm, s, z, logn, logR, rot, zr, zi);
    }
    {
        int bpc = 1024 / C;
        if (bpc < 1) bpc = 1;
        if (bpc > Rr) bpc = Rr;
        dim3 g(Rr / bpc, nd);
        const size_t sm = (size_t)bpc * C * sizeof(cplx);
        launch_k(k_fft_row, dim3(g), dim3(256), sm, s, z, logn, logR, bpc, rot, zr, zi);
    }
}

void launch_fft_residues(const void* zbuf, int z0, int logn, int nd, u64* out_coeff, int nl, const DevPrime* primes,
                         int scale_bits, cudaStream_t s) {
    const int n = 1 << logn;
    dim3 g((2 * n + kThreads - 1) / kThreads, nd);
    launch_k(k_fft_finish, dim3(g), dim3(kThreads), 0, s, (const cplx*)zbuf + (size_t)z0 * n, logn, nd, out_coeff, nl,
             primes, scale_bits);
}

void launch_fft_round(const void* zbuf, int logn, int nd, long long* out_int, int scale_bits, cudaStream_t s) {
    dim3 g(((2 << logn) + kThreads - 1) / kThreads, nd);
    launch_k(k_fft_round, dim3(g), dim3(kThreads), 0, s, (const cplx*)zbuf, logn, nd, out_int, scale_bits);
}

void launch_coef_residues(const long long* m, int nd, u64* out, int nl, const DevPrime* primes, int N,
                          cudaStream_t s) {
    dim3 g((N + kThreads - 1) / kThreads, nd);
    launch_k(k_coef_residues, dim3(g), dim3(kThreads), 0, s, m, nd, out, nl, primes, N);
}

namespace {

// Register-only FP64 fused multiply-add throughput (the ceiling of the encoder's FFT): eight
// independent chains per thread, x <- x a + b, with a slightly below 1 so values stay finite.
__global__ void __launch_bounds__(256) k_fp64_peak(double a, double b, int iters, double* sink) {
    double x[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) x[e] = 1.0 + 1e-3 * (threadIdx.x * 8 + e);
    for (int it = 0; it < iters; ++it) {
#pragma unroll
        for (int e = 0; e < 8; ++e) x[e] = __fma_rn(x[e], a, b);
    }
    double acc = 0;
#pragma unroll
    for (int e = 0; e < 8; ++e) acc += x[e];
    if (acc == -1.0) sink[0] = acc;  // keeps the loop live
}

}  // namespace

double measure_fp64_peak(int device) {
    int nsm = 0;
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, device);
    const int blocks = nsm * 8, threads = 256, iters = 4096;
    double* sink = nullptr;
    if (cudaMalloc(&sink, 8) != cudaSuccess) return 0;
    cudaEvent_t a, b;
    cudaEventCreate(&a);
    cudaEventCreate(&b);
    k_fp64_peak<<<blocks, threads>>>(0.999999, 1e-9, 64, sink);  // warm-up
    cudaEventRecord(a);
    k_fp64_peak<<<blocks, threads>>>(0.999999, 1e-9, iters, sink);
    cudaEventRecord(b);
    cudaEventSynchronize(b);
    float ms = 0;
    cudaEventElapsedTime(&ms, a, b);
    cudaEventDestroy(a);
    cudaEventDestroy(b);
    cudaFree(sink);
    if (ms <= 0) return 0;
    return 2.0 * blocks * threads * 8.0 * iters / (ms * 1e-3);  // an FMA is two operations
}
