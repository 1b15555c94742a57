// The transforms of rings of N = 2^10 .. 2^14 (a translation unit of its own: they compile beside
// the larger ones).
#include "ntt_kernels.cuh"

namespace ntt_kernels {

template <class E>
int launch_ntt_small(const RingDev& R, const PolyBatch& b, bool inverse, cudaStream_t s, const E& epi) {
    switch (R.logN) {
        case 10: return launch_ntt_s<5, 5>(R, b, inverse, s, epi);
        case 11: return launch_ntt_s<5, 6>(R, b, inverse, s, epi);
        case 12: return launch_ntt_s<6, 6>(R, b, inverse, s, epi);
        case 13: return launch_ntt_s<6, 7>(R, b, inverse, s, epi);
        case 14: return launch_ntt_s<7, 7>(R, b, inverse, s, epi);
        default: return 0;
    }
}

template int launch_ntt_small(const RingDev&, const PolyBatch&, bool, cudaStream_t, const EpiStore&);
template int launch_ntt_small(const RingDev&, const PolyBatch&, bool, cudaStream_t, const EpiDiag&);
template int launch_ntt_small(const RingDev&, const PolyBatch&, bool, cudaStream_t, const EpiModDown&);
template int launch_ntt_small(const RingDev&, const PolyBatch&, bool, cudaStream_t, const EpiRescale&);
template int launch_ntt_small(const RingDev&, const PolyBatch&, bool, cudaStream_t, const EpiLeafRescale&);
template int launch_ntt_small(const RingDev&, const PolyBatch&, bool, cudaStream_t, const EpiRelinRescale&);

}  // namespace ntt_kernels
