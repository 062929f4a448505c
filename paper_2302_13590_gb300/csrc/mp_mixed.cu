// mp_mixed.cu - mixed-precision tracking kernels (FP32 in-cell coordinates
// and velocities, the cumulative travel time as an FP32 pair; the engine is
// in mp_mixed.cuh).  Compiled with FMA contraction on.
#include "mp_mixed.cuh"

namespace mp {

// Launches of up to this many warps of ten particles on each SM take three
// lanes a particle (30,400 particles on 152 SMs; endpoints, 200x200x20 cells,
// 329 steps the longest: 4864 particles 137 us against 268, 19456: 190 / 274,
// 29184: 229 / 292, 38912: 328 / 294; the FP64 form's line is lower, its warps
// wait for one FP64 unit).
constexpr int MIXED_AXES_WARPS = 20;

cudaError_t form_mixed(long long n, LaunchForm* out) { return form_of<MixEngine<false, true>>(n, MIXED_AXES_WARPS, out); }

cudaError_t launch_track_mixed(const DevField& f, const Batch& b, unsigned modes, int schedule, int block, cudaStream_t s)
{
    if (b.n_total <= 0) return cudaSuccess;
    int sms = 0;
    const cudaError_t err = sm_count(&sms);
    if (err != cudaSuccess) return err;
    const bool few = few_particles(b.n_total, MIXED_AXES_WARPS, sms);
    if (b.n_reqs == 1) {
        const MixEngine<false, true> e{f, b};
        return few ? launch_axes_mixed(e, modes, s) : launch_tracking(e, modes, schedule, block, s);
    }
    const MixEngine<false, false> e{f, b};
    return few ? launch_axes_mixed(e, modes, s) : launch_tracking(e, modes, schedule, block, s);
}

}  // namespace mp
