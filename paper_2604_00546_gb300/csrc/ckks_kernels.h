// Tables and launchers of the CKKS device kernels.
#pragma once
#include "kernels.h"

// Fast base conversion, one target: sum_i y_i [B/b_i]_t mod t over at most 8 sources y_i < 2^61,
// without a quotient per product (the scheme of mul_tw, dev_arith.cuh). hat[i] = (w mod 2^S, w >> S,
// v mod 2^S, v >> S) with w = [B/b_i]_t and v = w 2^32 mod t; the products of several sources share
// the two 64-bit sums a0, a1 and one reduction a0 + (a1 mod 2^32) 2^S + (a1 >> 32) c2.
//   mode 0  all sources in one pair of sums (S = bits(t) - 28, targets of at most about 55 bits);
//   mode 1  two sources at a time (S = 30), the reduced pairs folded and added (60-bit targets);
//   mode 2  any target: hat[i].xy = w 2^64 mod t in 30-bit halves (mack), one Montgomery
//           reduction with qinv and one_s.
// The host picks the first mode whose sums provably fit (bconv_target).
struct BconvTarget {
    u64 q, qinv, one_s;
    u32 mode, mul, c2, bsh, c, pad;  // mul = 2^S; bsh, c as in DevPrime
    uint4 hat[8];
};

// ModUp constants of one digit at one level: sources are the digit's Q limbs
// [lo, lo + ns); targets are the other positions of Q_l u P. inv_hat = [(B/b_i)^-1]_{b_i}; the
// inverse transforms before a conversion multiply it in (PolyBatch::post).
struct ModUpTab {
    int ns, lo;
    u64 src_q[8], inv_hat[8], inv_hat_s[8];
    BconvTarget t[FR_MAX_PRIMES];
};

// ModDown constants: sources are the P limbs, targets Q limbs 0..l
struct P2QTab {
    int np;
    BconvTarget t[FR_MAX_PRIMES];
};

// Rescale constants at level l (divide by q_l)
struct RescaleTab {
    u64 half;  // (q_l - 1) / 2
    u64 q[FR_MAX_PRIMES];
    u64 ql_mod[FR_MAX_PRIMES];
    u64 qlinv[FR_MAX_PRIMES], qlinv_s[FR_MAX_PRIMES];
};

struct IPJob {
    const u64* ext;  // [beta][npos][N]; a digit's own positions are not in it
    const u64* own;  // the switched polynomial, limbs 0..level, stride N: the digits' own positions
    const u64* key;  // [digits][2][T][N], Montgomery form: Q limbs 0..kp-1, then P limbs
    u64* out;        // [2][npos][N]
    u32 galois;      // 1: no automorphism
    const u64* addb = nullptr;  // non-null: add P sigma_galois(addb) to component 0 on the Q positions
                                // (addb: limbs 0..level, stride N, evaluation form)
};

struct MDJob {
    const u64* acc;   // [2][npos][N]
    const u64* add;   // modes 1, 3: c0 limbs (stride N); mode 2: ct with add_cap
    u64* out;         // ct with out_cap
    int out_cap;
    int add_cap;
    int mode;         // 0 none, 1 rotation addend sigma_g(c0), 2 ct addend, 3 rotation + ct addend
    u32 galois;
    const u64* add2;  // mode 3: ct with add_cap added to both components
};

struct TensorJob {
    const u64* a;
    const u64* b;
    u64* out;  // [3][level+1][N]
    int a_cap, b_cap;
};

// job lists travel as kernel parameters (no descriptor copies, capturable in graphs)
#define FR_MAX_JOBS 64
// jobs grouped by key: group g uses gkey[g] for jobs gstart[g] .. gstart[g+1]-1
struct IPJobs {
    IPJob j[FR_MAX_JOBS];
    signed char owner[FR_MAX_PRIMES];  // digit that holds position pos (-1: none, the P limbs)
    const u64* gkey[FR_MAX_JOBS];
    int gstart[FR_MAX_JOBS + 1];
    int ngroups;
};
struct MDJobs { MDJob j[FR_MAX_JOBS]; };
// Inner products summed straight into the accumulators of their sums of rotations: group g
// (jobs gstart[g] .. gstart[g+1]-1) writes, or with add[g] adds into, j[gstart[g]].out. Each job's ext, key, galois and
// addb (its rotated ciphertext's c0) are used as in IPJobs.
struct IPSumJobs {
    IPJob j[FR_MAX_JOBS];
    signed char owner[FR_MAX_PRIMES];
    bool add[FR_MAX_JOBS];  // group g continues a sum (else it starts one)
    int gstart[FR_MAX_JOBS + 1];
    int ngroups;
};
struct TensorJobs { TensorJob j[FR_MAX_JOBS]; };

// Layout of a database's diagonals in evaluation form: tiles of kDiagTile points, [limb][N /
// kDiagTile][row][kDiagTile], so that a CTA of the MAC, which takes all rows at a few points of one
// limb, reads one contiguous run. Rows are the diagonals (or, encrypted, the two components of
// each). Offset of point k of limb i of row r among `rows` rows of N points:
constexpr int kDiagTile = 64;
__host__ __device__ __forceinline__ long long diag_word(int i, int k, long long r, int rows, int N) {
    return (((long long)i * (N / kDiagTile) + k / kDiagTile) * rows + r) * kDiagTile + k % kDiagTile;
}
// Forward NTT of encoded diagonals into a database: poly p of b is limb p % nl of diagonal d0 +
// p / nl; the values go to diags (ell rows) in Montgomery form (x 2^64 mod q), as 30-bit halves
// (split30).
int launch_ntt_diags(const RingDev& R, const PolyBatch& b, u64* diags, int d0, int ell, int nl, cudaStream_t s);
// src [rows][nl][N] (evaluation form) into rows row0.. of a database of total rows, Montgomery form
void launch_tile_mont(const u64* src, int rows, u64* diags, long long row0, int total, int nl, const DevPrime* primes,
                      int N, cudaStream_t s);
// Forward NTT of the P -> Q conversions of a ModDown fused with its combine:
// poly p of b is (job p / (2(level+1)), component, limb); the transformed values never reach
// memory, the jobs' outputs do.
int launch_ntt_moddown(const RingDev& R, const PolyBatch& b, const MDJobs& jobs, int npos, int level,
                        const u64* pinv, const u64* pinv_s, cudaStream_t s);
// Forward NTT of a rescale's lifted last limb fused with its combine: poly p of b is
// (ct component p / l, limb p % l); writes out = (x - NTT(lifted)) q_l^-1, then mode 1 adds
// the matching component of the ct at add + (p / l / 2) add_bs (cap add_cap), mode 2 doubles
// and subtracts cres[i] from component 0.
// Chebyshev leaves Rescale(T1 cb_j + ca_j) in two launches and one transform, without the
// leaves in memory: launch_leaf_lift forms the lifted last limbs [B nl][2][l][N] from u, the
// coefficient form of T1's last limb ([B][2][N]); launch_ntt_leaf_rescale transforms them
// (b: poly ((b nl + j) 2 + t) l + i) and writes leaf (b, j) at out + (b nl + j) 2 out_cap N.
// T1 of query b at x + b x_bs (cap x_cap); constants [nl][L1] each.
void launch_leaf_lift(const u64* u, const u64* cb, const u64* cb_s, const u64* ca, int nl, int L1, u64* lifted,
                      const RescaleTab* tab, const DevPrime* primes, int l, int N, int B, cudaStream_t s);
int launch_ntt_leaf_rescale(const RingDev& R, const PolyBatch& b, const u64* x, long long x_bs, int x_cap,
                             const u64* cb, const u64* cb_s, const u64* ca, int nl, int L1, u64* out, int out_cap,
                             const RescaleTab* tab, int l, cudaStream_t s);
int launch_ntt_rescale(const RingDev& R, const PolyBatch& b, const u64* x, int x_cap, u64* out, int out_cap,
                        const RescaleTab* tab, int l, int mode, const u64* add, int add_cap, long long add_bs,
                        const u64* cres, cudaStream_t s);
// Baby steps kept in Q_l u P: baby 0 = P q (zero on the P positions) of each of B queries,
// babies [B][n1][2][npos][N]; babies 1..n1-1 are inner products with IPJob::addb set.
void launch_baby0_pq(u64* babies, long long baby_q, const u64* q, long long q_bs, int q_cap, int B, int npos,
                     int level, const DevPrime* primes, const u64* pmod, const u64* pmod_s, int N, cudaStream_t s);
// Relinearisation fused with the rescale after it (J products at level l): z = acc_l P^-1 + d_l
// [J][2][N] is formed by its inverse NTT (PolyBatch::rs); after that and the P limbs', launch_p2q_lift
// forms y = conv P^-1 + centered lift [J][2][l][N]; the forward NTT of y with launch_ntt_relin_rescale writes
// out_j = (acc P^-1 + d - NTT(y)) q_l^-1 (+ the EpiRescale modes) at level l - 1.
void launch_p2q_lift(const u64* acc, long long acc_job, int npos, const u64* zc, u64* y, const P2QTab* tab_rs,
                     const RescaleTab* rtab, u64 ql, int l, int N, int J, cudaStream_t s);
int launch_ntt_relin_rescale(const RingDev& R, const PolyBatch& b, const u64* acc, const u64* d, int npos, int l,
                              const u64* pinv, const u64* pinv_s, const RescaleTab* tab, u64* out, int out_cap,
                              long long out_bs, int mode, const u64* add, int add_cap, long long add_bs,
                              const u64* cres, cudaStream_t s);
// ModUp of J inputs: coefficient form of input j at in + j in_job (scaled: already multiplied by
// the digits' inv_hat); writes the positions of ext that are not the digit's own
void launch_modup(const u64* in, long long in_job, u64* ext, const ModUpTab* tabs, int beta, int npos, int N, int J,
                  bool scaled, cudaStream_t s);
void launch_ip(const IPJobs& jobs, int beta, int npos, int level, int kp, int T, const DevPrime* primes,
               const PrimeMap& pos_prime, int logN, cudaStream_t s, const u64* pmod = nullptr,
               const u64* pmod_s = nullptr);
// ModDown conversions of the P limbs (coefficient form, times inv_hat) of J accumulators
void launch_p2q(const u64* acc, long long acc_job, int npos, int level, u64* conv, const P2QTab* tab, int N, int J,
                cudaStream_t s);
void launch_rescale_lift(const u64* last, u64* lifted, const RescaleTab* tab, const DevPrime* primes, int l, int N,
                         int BT, cudaStream_t s);
void launch_tensor(const TensorJobs& jobs, int J, int level, const DevPrime* primes, int N, cudaStream_t s);
// Sums of rotations with one ModDown (double hoisting), without the per-job inner products in
// memory: for each group g and position,
// out_g (+)= sum_{jobs of g} (IP_j + P sigma_j(addb_j) on the Q positions of component 0), the
// inner products as launch_ip computes them. out_g: [2][npos][N].
void launch_ip_sum(const IPSumJobs& jobs, int beta, int npos, int level, int kp, int T, const DevPrime* primes,
                   const PrimeMap& pos_prime, int logN, const u64* pmod, const u64* pmod_s, cudaStream_t s);
// Encrypted-database MAC: (d0, d1, d2)_j = sum_i B_i (x) E_{j n1 + i} for every giant step j.
// babies [n1][2][cap_b][N]; diags: 2 ell rows (evaluation form, Montgomery); out [n2][3][cap_o][N].
void launch_mac_ct(const u64* babies, int cap_b, const u64* diags, u64* out, int cap_o, int nl, int n1, int n2, int ell,
                   const DevPrime* primes, int N, cudaStream_t s);
// The diagonal MAC of B = 2..4 queries against one database with the diagonals streamed
// through a shared-memory ring of asynchronous copies, every diagonal word read once for all B
// queries (the sums of launch_mac: babies of query b at babies + b baby_q, [n1][2][cap_b][N];
// outputs at out + b out_q, [n2][2][cap_o][N]); usable when mac_pipe_fits.
bool mac_pipe_fits(int n1, int ell, int N, bool wide);
// The same sums as a persistent pipeline (k_mac_ring): one CTA per GPU slot runs point tiles in
// turn, the next tile's diagonals and babies in flight while this one is multiplied; B = 2..4
// queries, each diagonal word read once for all of them. Usable when mac_ring_fits.
bool mac_ring_fits(int n1, int ell, int N, int B, bool wide);
void launch_mac_ring(const u64* babies, long long baby_q, int cap_b, const u64* diags, u64* out, long long out_q,
                     int cap_o, int nl, int n1, int ell, int B, const DevPrime* primes, int N, cudaStream_t s);
void launch_mac_pipe(const u64* babies, long long baby_q, int cap_b, const u64* diags, u64* out, long long out_q,
                     int cap_o, int nl, int n1, int ell, int B, const DevPrime* primes, int N, cudaStream_t s);
// The diagonal MAC of one query: babies [n1][2][cap_b][N], outputs [n2][2][cap_o][N]. wide: some
// prime has 61 bits (the batched forms above then do not fit).
void launch_mac(const u64* babies, int cap_b, const u64* diags, u64* out, int cap_o, int nl, int n1, int n2, int ell,
                bool wide, const DevPrime* primes, int N, cudaStream_t s);
// Table schedule (Algorithm 1): out_g = sum_{m < ell} table[m] (.) D_{g,m} for g < G (evaluation form,
// not rescaled); table [ell][2][cap_t][N], group g's diagonals at diags + g * dgrp.
void launch_mac_table(const u64* table, int cap_t, const u64* diags, long long dgrp, int G, u64* out, int cap_o,
                      long long og, int nl, int ell, const DevPrime* primes, int N, cudaStream_t s);
void launch_add(const u64* a, int a_cap, long long a_bs, const u64* b, int b_cap, long long b_bs, u64* out, int o_cap,
                long long o_bs, int level, int B, const DevPrime* primes, int N, cudaStream_t s);
void launch_sum(const u64* a, int cap, long long js, int J, u64* out, int o_cap, int level, const DevPrime* primes,
                int N, cudaStream_t s);
void launch_to_mont(u64* x, long long n_per_poly, const PrimeMap& pm, const DevPrime* primes, long long total,
                    cudaStream_t s);
// Slot encoding of diagonals d0 .. d0 + nd - 1 of template group grp, up to the rounding: z [nd][n]
// complex doubles
void launch_encode_fft(const float* T, long long K, int ell, int logn, long long grp, int d0, int nd, int n1, void* zbuf,
                       const unsigned* rot, const double* zr, const double* zi, cudaStream_t s);
// The rounded coefficients of diagonals z0 .. z0 + nd - 1 of z as residues, out_coeff [nd][nl][N], or
// (storage tier B) of all nd of z as integers, out_int [nd][N]
void launch_fft_residues(const void* zbuf, int z0, int logn, int nd, u64* out_coeff, int nl, const DevPrime* primes,
                         int scale_bits, cudaStream_t s);
void launch_fft_round(const void* zbuf, int logn, int nd, long long* out_int, int scale_bits, cudaStream_t s);
// Residues of stored integer coefficients: m [nd][N] -> out [nd][nl][N] (coefficient form).
void launch_coef_residues(const long long* m, int nd, u64* out, int nl, const DevPrime* primes, int N,
                          cudaStream_t s);
