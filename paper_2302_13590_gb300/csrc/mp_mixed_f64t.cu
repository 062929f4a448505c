// mp_mixed_f64t.cu - the mixed-precision engine with FP64 kept for the
// cumulative travel time and for the near-zero branch of the exit time
// (MP_PREC_MIXED_F64T): the accuracy reference for the FP32 pair and the
// FP32 series of the default mixed form.
#include "mp_mixed.cuh"

namespace mp {

cudaError_t form_mixed_f64t(long long n, LaunchForm* out) { return form_of<MixEngine<true, true>>(n, 0, out); }

cudaError_t launch_track_mixed_f64t(const DevField& f, const Batch& b, unsigned modes, int schedule, int block, cudaStream_t s)
{
    if (b.n_reqs == 1)
        return launch_tracking(MixEngine<true, true>{f, b}, modes, schedule, block, s);
    return launch_tracking(MixEngine<true, false>{f, b}, modes, schedule, block, s);
}

}  // namespace mp
