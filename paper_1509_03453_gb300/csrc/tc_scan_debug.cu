// The screening launch with the bound check compiled in (OSANN_DEBUG_CHECKS=1):
// every screened value is compared with an fp32 evaluation of the folded
// product, and a violation sets OSANN_STATUS_BOUND.
#include "tc_scan_kernel.cuh"

namespace osann {

int launch_tc_scan_debug(const void* maps, const TcArgs& a, int k, cudaStream_t st, int num_sms)
{
    return launch_tc_dp<false, true>(maps, a, k, st, num_sms);
}

}  // namespace osann
