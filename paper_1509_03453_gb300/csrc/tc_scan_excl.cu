// The screening launches with an exclusion radius, bound check out or in.
#include "tc_scan_kernel.cuh"

namespace osann {

int launch_tc_scan_excl(const void* maps, const TcArgs& a, int k, bool debug, cudaStream_t st, int num_sms)
{
    return debug ? launch_tc_dp<true, true>(maps, a, k, st, num_sms) : launch_tc_dp<true, false>(maps, a, k, st, num_sms);
}

}  // namespace osann
