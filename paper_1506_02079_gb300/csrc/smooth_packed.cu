// smooth_tma_kernel with smooth_fused_kernel's operations and order, for packed copies of stacks
// whose rows TMA cannot read (smooth.cu): one instance per type, xy radius and number of z taps.
#include "emfuse_internal.cuh"
#include "smooth_tma.cuh"

namespace emfuse {
namespace smooth_detail {
namespace {

template <class Tin, int R>
int launch_r(const SmoothTmaCall& c, bool robust, cudaStream_t st) {
    const bool few = c.prm.Rz <= 3;  // the taps of smooth_fused_kernel's instances: 7 or 19
    if (robust) return few ? smooth_tma_launch<Tin, R, true, true, 7>(c, st) : smooth_tma_launch<Tin, R, true, true, 19>(c, st);
    return few ? smooth_tma_launch<Tin, R, false, true, 7>(c, st) : smooth_tma_launch<Tin, R, false, true, 19>(c, st);
}

template <class Tin>
int launch_t(const SmoothTmaCall& c, bool robust, cudaStream_t st) {
    switch (c.prm.Rxy) {
        case 1: return launch_r<Tin, 1>(c, robust, st);
        case 2: return launch_r<Tin, 2>(c, robust, st);
        case 3: return launch_r<Tin, 3>(c, robust, st);
        default: return launch_r<Tin, 4>(c, robust, st);
    }
}

}  // namespace

int smooth_tma_packed(const SmoothTmaCall& c, int dt, bool robust, cudaStream_t st) {
    return dt == EMFUSE_U8 ? launch_t<uint8_t>(c, robust, st) : launch_t<float>(c, robust, st);
}

}  // namespace smooth_detail
}  // namespace emfuse
