// The screening launches over rows of uneven norms, where bounds are kept per candidate
// (k > 1, or an exclusion radius): the bound takes the row's own norm.
#include "tc_scan_kernel.cuh"

namespace osann {

int launch_tc_scan_uneven(const void* maps, const TcArgs& a, int k, bool excl, cudaStream_t st, int num_sms)
{
    return excl ? launch_tc_dp<true, false, true>(maps, a, k, st, num_sms)
                : launch_tc_dp<false, false, true>(maps, a, k, st, num_sms);
}

}  // namespace osann
