// mp_mixed.cu - mixed-precision tracking kernels (FP32 in-cell coordinates
// and velocities, the cumulative travel time as an FP32 pair; the engine is
// in mp_mixed.cuh).  Compiled with FMA contraction on.
#include "mp_mixed.cuh"

namespace mp {

// Launches of up to this many particles take three lanes each: 20 warps an SM
// on 152 SMs (endpoints, 200x200x20 cells, 329 steps the longest: 4864
// particles 137 us against 268, 19456: 190 / 274, 29184: 229 / 292, 38912:
// 328 / 294; the FP64 form's line is lower, its warps wait for one FP64 unit).
constexpr long long MIXED_AXES_MAX = 20 * 152 * AXES_PARTICLES;

cudaError_t launch_track_mixed(const DevField& f, const Batch& b, unsigned modes, int schedule, int block, cudaStream_t s)
{
    if (b.n_total <= 0) return cudaSuccess;
    const bool few = b.n_total <= MIXED_AXES_MAX;
    if (b.n_reqs == 1) {
        const MixEngine<false, true> e{f, b};
        return few ? launch_axes_mixed(e, modes, s) : launch_tracking(e, modes, schedule, block, s);
    }
    const MixEngine<false, false> e{f, b};
    return few ? launch_axes_mixed(e, modes, s) : launch_tracking(e, modes, schedule, block, s);
}

}  // namespace mp
