// Transforms: the entry points, the rings of N = 2^15 and 2^16, the tuner of their tile shapes and
// the butterfly's arithmetic ceiling.
#include <cstdlib>

#include "ntt_kernels.cuh"

using namespace ntt_kernels;

namespace {

// Register-only throughput of the forward butterfly used above (a class-0 prime's, the cheapest
// product): the arithmetic ceiling of the NTT on this GPU, no memory traffic.
__global__ void __launch_bounds__(256) k_butterfly_peak(uint4 w, u64 c2, u64 off, int iters, u64* sink) {
    u64 x[8], y[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) {
        x[e] = threadIdx.x * 8 + e;
        y[e] = blockIdx.x * 8 + e + 1;
    }
    for (int it = 0; it < iters; ++it) {
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            const u64 T = mul_tw<0>(y[e], w, c2);
            y[e] = x[e] - T + off;
            x[e] = x[e] + T;
        }
    }
    u64 acc = 0;
#pragma unroll
    for (int e = 0; e < 8; ++e) acc ^= x[e] ^ y[e];
    if (acc == 0x5a5a5a5a5a5a5a5aull) sink[0] = acc;  // keeps the loop live
}

}  // namespace

int pdl_mode() {
    static const int m = [] {
        const char* e = std::getenv("FR_PDL");
        return e && e[0] == '0' ? 0 : e && e[0] == '1' ? 1 : 2;
    }();
    return m;
}

double measure_butterfly_peak(int device) {
    // 50-bit prime; any twiddle works for a throughput measurement
    const u64 q = 1125899904679937ull, off = q << 9;
    const uint4 w = make_uint4(0x54321, 0x2badcafe, 0xabcde, 0x1234567);
    int nsm = 0;
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, device);
    const int blocks = nsm * 8, threads = 256, iters = 4096;
    u64* sink = nullptr;
    if (cudaMalloc(&sink, 8) != cudaSuccess) return 0;
    cudaEvent_t a, b;
    cudaEventCreate(&a);
    cudaEventCreate(&b);
    k_butterfly_peak<<<blocks, threads>>>(w, (1ull << 52) - 4 * q, off, 64, sink);  // warm-up
    cudaEventRecord(a);
    k_butterfly_peak<<<blocks, threads>>>(w, (1ull << 52) - 4 * q, off, iters, sink);
    cudaEventRecord(b);
    cudaEventSynchronize(b);
    float ms = 0;
    cudaEventElapsedTime(&ms, a, b);
    cudaEventDestroy(a);
    cudaEventDestroy(b);
    cudaFree(sink);
    if (ms <= 0) return 0;
    return (double)blocks * threads * 8.0 * iters / (ms * 1e-3);
}

template <class E>
int launch_ntt_e(const RingDev& R, const PolyBatch& b, bool inverse, cudaStream_t s, const E& epi) {
    if (b.npolys <= 0) return 0;
    switch (R.logN) {
        case 15: return launch_ntt_s<7, 8>(R, b, inverse, s, epi);
        case 16: return launch_ntt_s<8, 8>(R, b, inverse, s, epi);
        default: return launch_ntt_small(R, b, inverse, s, epi);
    }
}

int launch_ntt(const RingDev& R, const PolyBatch& b, bool inverse, cudaStream_t s) {
    return launch_ntt_e(R, b, inverse, s, EpiStore{});
}

// Times every tile shape of the forward + inverse transform for one batch size per bucket
// (CUDA events, best of `reps`) on a scratch buffer of zero residues and keeps the fastest
// shape per bucket in R.ntt_shape; us[bucket * FR_NTT_SHAPES + shape] receives the times.
void tune_ntt(RingDev& R, cudaStream_t s, double* us, int reps) {
    if (us)
        for (int i = 0; i < FR_NTT_BUCKETS * FR_NTT_SHAPES; ++i) us[i] = 0;
    if (R.logN < 14) return;
    const int sizes[FR_NTT_BUCKETS] = {4, 16, 64, 256};
    const int maxp = sizes[FR_NTT_BUCKETS - 1];
    u64* buf = nullptr;
    if (cudaMallocAsync(&buf, (size_t)maxp * R.N * 8, s) != cudaSuccess) { cudaGetLastError(); return; }
    cudaMemsetAsync(buf, 0, (size_t)maxp * R.N * 8, s);
    cudaEvent_t a, e;
    cudaEventCreate(&a);
    cudaEventCreate(&e);
    auto timed = [&](int bk, int sh) {
        PolyBatch pb{buf, 0, sizes[bk], sizes[bk], PrimeMap{}};
        pb.pm.period = R.nprimes;
        for (int i = 0; i < R.nprimes; ++i) pb.pm.idx[i] = (unsigned char)i;
        R.ntt_shape[bk] = (unsigned char)sh;
        cudaEventRecord(a, s);
        launch_ntt(R, pb, false, s);
        launch_ntt(R, pb, true, s);
        cudaEventRecord(e, s);
        cudaEventSynchronize(e);
        float ms = 0;
        cudaEventElapsedTime(&ms, a, e);
        if (cudaGetLastError() != cudaSuccess) return 1e30;  // a shape this GPU cannot launch
        return ms * 1000.0;
    };
    unsigned char best[FR_NTT_BUCKETS];
    for (int bk = 0; bk < FR_NTT_BUCKETS; ++bk) {
        double t[FR_NTT_SHAPES];
        for (int sh = 0; sh < FR_NTT_SHAPES; ++sh) t[sh] = 1e30;
        for (int r = 0; r <= reps; ++r)  // the first round warms up; the shapes take turns
            for (int sh = 0; sh < FR_NTT_SHAPES; ++sh) {
                // shapes that would run another's kernels (2 and 3 are 0 and 1, and take their times)
                if (sh == 2 || sh == 3 || (sh == 1 && R.logN < 15) || (sh >= 4 && !R.fast) || (sh == 4 && R.logN > 14))
                    continue;
                const double now = timed(bk, sh);
                if (r > 0 && now < t[sh]) t[sh] = now;
            }
        if (R.logN >= 15) {
            t[2] = t[0];
            t[3] = t[1];
        }
        best[bk] = 0;
        double tbest = t[0];
        for (int sh = 0; sh < FR_NTT_SHAPES; ++sh) {
            if (us) us[bk * FR_NTT_SHAPES + sh] = t[sh] < 1e29 ? t[sh] : -1.0;
            // another shape replaces the default only when at least 3% faster (timing noise)
            if (t[sh] < tbest && t[sh] < 0.97 * t[0]) {
                tbest = t[sh];
                best[bk] = (unsigned char)sh;
            }
        }
    }
    for (int bk = 0; bk < FR_NTT_BUCKETS; ++bk) R.ntt_shape[bk] = best[bk];
    cudaEventDestroy(a);
    cudaEventDestroy(e);
    cudaFreeAsync(buf, s);
    cudaStreamSynchronize(s);
}

int launch_ntt_diags(const RingDev& R, const PolyBatch& b, u64* diags, int d0, int ell, int nl, cudaStream_t s) {
    return launch_ntt_e(R, b, false, s, EpiDiag{diags, d0, ell, nl, R.N});
}

int launch_ntt_moddown(const RingDev& R, const PolyBatch& b, const MDJobs& jobs, int npos, int level,
                        const u64* pinv, const u64* pinv_s, cudaStream_t s) {
    EpiModDown e{jobs, npos, level, R.logN, pinv, pinv_s};
    return launch_ntt_e(R, b, false, s, e);
}

int launch_ntt_relin_rescale(const RingDev& R, const PolyBatch& b, const u64* acc, const u64* d, int npos, int l,
                              const u64* pinv, const u64* pinv_s, const RescaleTab* tab, u64* out, int out_cap,
                              long long out_bs, int mode, const u64* add, int add_cap, long long add_bs,
                              const u64* cres, cudaStream_t s) {
    EpiRelinRescale e{acc, d, out, tab, pinv, pinv_s, npos, l, R.N, out_cap, mode, out_bs, add, add_cap, add_bs, cres};
    return launch_ntt_e(R, b, false, s, e);
}

int launch_ntt_leaf_rescale(const RingDev& R, const PolyBatch& b, const u64* x, long long x_bs, int x_cap,
                             const u64* cb, const u64* cb_s, const u64* ca, int nl, int L1, u64* out, int out_cap,
                             const RescaleTab* tab, int l, cudaStream_t s) {
    EpiLeafRescale e{x, x_bs, x_cap, cb, cb_s, ca, nl, L1, out, out_cap, tab, l, R.N};
    return launch_ntt_e(R, b, false, s, e);
}

int launch_ntt_rescale(const RingDev& R, const PolyBatch& b, const u64* x, int x_cap, u64* out, int out_cap,
                        const RescaleTab* tab, int l, int mode, const u64* add, int add_cap, long long add_bs,
                        const u64* cres, cudaStream_t s) {
    EpiRescale e{x, out, tab, x_cap, out_cap, l, R.N, mode, add, add_cap, add_bs, cres};
    return launch_ntt_e(R, b, false, s, e);
}
