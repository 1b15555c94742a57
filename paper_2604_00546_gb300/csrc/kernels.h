// Kernel launchers shared by the engine (host-callable, device pointers only).
#pragma once
#include <cuda_runtime.h>
#include <atomic>
#include <cstdint>

#include "dev_arith.cuh"

// Programmatic dependent launch. Every kernel of the library starts with pdl_wait(), so it
// touches no memory before the kernel ahead of it in the stream has completed and flushed;
// launched with programmatic stream serialisation, only its launch and CTA scheduling
// overlap the tail of the previous kernel. pdl_trigger() lets the next kernel be scheduled
// once every CTA of this one has started.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// When launches carry the programmatic-serialisation attribute: FR_PDL=0 never, FR_PDL=1
// always, unset (mode 2) for launches outside stream capture only. Measured on the membership
// match: launched one by one it is about 4% faster with the attribute; replayed as a CUDA graph,
// about 2.5% slower with it.
int pdl_mode();
inline bool pdl_use(cudaStream_t s) {
    const int m = pdl_mode();
    if (m != 2) return m == 1;
    cudaStreamCaptureStatus st = cudaStreamCaptureStatusNone;
    return cudaStreamIsCapturing(s, &st) == cudaSuccess && st == cudaStreamCaptureStatusNone;
}

template <typename... KP, typename... A>
inline void launch_k(void (*k)(KP...), dim3 g, dim3 b, size_t smem, cudaStream_t s, A... args) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = g;
    cfg.blockDim = b;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = pdl_use(s) ? 1 : 0;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, k, static_cast<KP>(args)...);
}

// cudaFuncSetAttribute acts on the current device only: raise kernel k's dynamic shared memory
// limit once per device (bit d of `done` marks device d). A device is marked only once the
// call has succeeded, so a failed call is retried by the next launch; ordinals 64 and above
// are not cached and set the limit on every launch.
template <class K>
inline void smem_limit_once(K* k, int bytes, std::atomic<unsigned long long>& done) {
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev < 0 || dev >= 64) {
        cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
        return;
    }
    const unsigned long long bit = 1ull << dev;
    if (done.load(std::memory_order_acquire) & bit) return;
    if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes) == cudaSuccess)
        done.fetch_or(bit, std::memory_order_release);
}

#define FR_MAX_PRIMES 64

// Periodic prime assignment of a batch of polynomials: poly p uses prime idx[p % period].
struct PrimeMap {
    int period;
    unsigned char idx[FR_MAX_PRIMES];
};

// The polynomials of a ModUp extension [ndig][npos][N] that a digit does not own: of digit d's
// npos positions all but [lo[d], lo[d] + ns[d]). n of them in all; position pos uses prime pos up to
// limbs - 1, then pbase, pbase + 1, ...
struct ExtMap {
    int n = 0, ndig = 0, npos = 0, limbs = 0, pbase = 0;
    unsigned char lo[8] = {}, ns[8] = {};
};

// A batch of N-point polynomials: poly p lives at base + (p / inner) * outer + (p % inner) * N
// and uses prime pm.idx[p % pm.period]. With an extension map (ext.n > 0) poly p is polynomial
// p % ext.n of the extension at base + (p / ext.n) * outer. Everything is in the launch's
// parameters, so a pass starts its loads without waiting for another.
struct PolyBatch {
    u64* base;
    long long outer;
    int inner;
    int npolys;
    PrimeMap pm;
    ExtMap ext{};
    // optional source of the first pass (out of place): poly p read from
    // src + (p / inner) src_outer + (p % inner) N and written to its place in base
    const u64* src = nullptr;
    long long src_outer = 0;
    // optional second segment (no source, no extension map): polys split .. npolys - 1 live at
    // base2 + (q / inner2) outer2 + (q % inner2) N, q = p - split, with primes pm2, so the
    // transforms of two buffers share one launch
    int split = 0;
    u64* base2 = nullptr;
    long long outer2 = 0;
    int inner2 = 1;
    PrimeMap pm2{};
    // optional (inverse, first segment): poly p ends with the constants post[2e], post[2e + 1], e =
    // p % pm.period, instead of its prime's N^-1 and N^-1 itw[1] (tw_ninv, tw_wninv): a constant
    // factor on the coefficients costs nothing
    const uint4* post = nullptr;
    // optional (inverse, second segment): its poly (job j, component t) = 2 j + t starts from acc_l P^-1
    // + d_l, limb l of acc [J][2][npos][N] and of d [J][3][l+1][N] (null: no addend), instead of its
    // memory
    struct {
        const u64* acc = nullptr;
        const u64* d = nullptr;
        const u64 *pinv = nullptr, *pinv_s = nullptr;
        int npos = 0, l = 0;
    } rs{};
};

// NTT batch-size buckets for the tuned tile shapes: <= 4, <= 16, <= 64, larger.
#define FR_NTT_BUCKETS 4
#define FR_NTT_SHAPES 6
__host__ __device__ inline int ntt_bucket(int npolys) {
    return npolys <= 4 ? 0 : npolys <= 16 ? 1 : npolys <= 64 ? 2 : 3;
}

// Order of a row's twiddles for the radix-16 row pass of 2^LOG points (TPR = 2^LOG / 16 threads):
// 2^LOG entries a row. The 15 of the phase on the high bits are the row's own, (8 >> lb) - 1 + u
// for register bit lb; the low phase's follow as [(8 >> lb) - 1 + u][thread], so that the lanes of
// a warp read consecutive entries. In the natural order the threads' 8, 4, 2 entries of a stage
// lie 128, 64, 32 bytes apart, one cache line each. LOG = 7 runs three low stages (lb <= 2).
__host__ __device__ constexpr int row_tw_index(int LOG, bool high, int lb, int u, int tau) {
    return high ? (8 >> lb) - 1 + u : 16 + ((8 >> lb) - 1 + u - (LOG == 7 ? 1 : 0)) * ((1 << LOG) / 16) + tau;
}

// Ring tables resident on the device for one parameter set.
struct RingDev {
    int logN;
    int N;
    int nprimes;
    const DevPrime* primes;  // [nprimes]
    const uint4* tw;         // [nprimes][N] psi^brev(k) in the prime's twiddle format
    const uint4* itw;        // [nprimes][N] psi^-brev(k), likewise
    const uint4* rtw;        // [nprimes][N] the same twiddles in the order of the radix-16 row pass
    const uint4* irtw;       // (row_tw_index; N >= 2^14, null otherwise)
    bool fast;               // no prime of twiddle class 2
    unsigned long long cls1, cls2;  // bit i: prime i is of twiddle class 1, of class 2
    unsigned char ntt_shape[FR_NTT_BUCKETS];  // tile shape per batch-size bucket (see launch_ntt)
};

// Batched negacyclic NTT (evaluation order: position k = value at psi^(2 brev(k)+1)). This and every
// launch_ntt_* return the number of kernels launched: 1 for the cluster transform, 2 for two passes.
int launch_ntt(const RingDev& R, const PolyBatch& b, bool inverse, cudaStream_t s);
// Autotuner of the NTT tile shapes (see ntt.cu); us: FR_NTT_BUCKETS x FR_NTT_SHAPES times in
// microseconds (-1: shape not available), or null.
void tune_ntt(RingDev& R, cudaStream_t s, double* us, int reps);
// Butterflies per second of the NTT's forward butterfly with operands in registers.
double measure_butterfly_peak(int device);
// FP64 operations per second of fused multiply-adds with operands in registers.
double measure_fp64_peak(int device);
