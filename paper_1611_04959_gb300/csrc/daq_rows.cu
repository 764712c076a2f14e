// The two-pass form for rows that share no 16-byte alignment (an n_samples that
// is not a multiple of 8, or an input that starts between 16-byte boundaries):
// tiles come in row by row (row_load).  A file of
// its own so that its kernels compile beside the others.
#include "daq_launch.cuh"

namespace daq {

cudaError_t launch_twopass_rows(const KArgs &a, const Plan &pl, int grid, int sms, bool skip_isl, cudaEvent_t const *ev,
                                cudaStream_t s)
{
    return launch_twopass_any<true>(a, pl, grid, sms, skip_isl, ev, s);
}

}  // namespace daq
