// The transforms of rings of N = 2^10 .. 2^14 (a translation unit of its own: they compile beside
// the larger ones).
#include "ntt_kernels.cuh"

namespace ntt_kernels {

template <class E>
void launch_ntt_small(const RingDev& R, const PolyBatch& b, bool inverse, cudaStream_t s, const E& epi) {
    switch (R.logN) {
        case 10: launch_ntt_s<5, 5>(R, b, inverse, s, epi); break;
        case 11: launch_ntt_s<5, 6>(R, b, inverse, s, epi); break;
        case 12: launch_ntt_s<6, 6>(R, b, inverse, s, epi); break;
        case 13: launch_ntt_s<6, 7>(R, b, inverse, s, epi); break;
        case 14: launch_ntt_s<7, 7>(R, b, inverse, s, epi); break;
        default: break;
    }
}

template void launch_ntt_small(const RingDev&, const PolyBatch&, bool, cudaStream_t, const EpiStore&);
template void launch_ntt_small(const RingDev&, const PolyBatch&, bool, cudaStream_t, const EpiDiag&);
template void launch_ntt_small(const RingDev&, const PolyBatch&, bool, cudaStream_t, const EpiModDown&);
template void launch_ntt_small(const RingDev&, const PolyBatch&, bool, cudaStream_t, const EpiRescale&);
template void launch_ntt_small(const RingDev&, const PolyBatch&, bool, cudaStream_t, const EpiLeafRescale&);
template void launch_ntt_small(const RingDev&, const PolyBatch&, bool, cudaStream_t, const EpiRelinRescale&);

}  // namespace ntt_kernels
