// The instantiations of us_spmm_tc_kernel.
#include "us_launch.h"
#include "us_spmm_tc.cuh"

namespace us {
namespace {

template <int OCT>
const void* pick(bool fold, bool w2, bool am)
{
    if (w2) return am ? nullptr : (const void*)us_spmm_tc_kernel<OCT, 2, true, false>;
    if (fold) return am ? nullptr : (const void*)us_spmm_tc_kernel<OCT, 2, false, false>;
    return am ? (const void*)us_spmm_tc_kernel<OCT, 1, false, true> : (const void*)us_spmm_tc_kernel<OCT, 1, false, false>;
}

}  // namespace

const void* kernel_tc(int octets, bool fold, bool w2, bool am)
{
    return octets == 3 ? pick<3>(fold, w2, am) : pick<2>(fold, w2, am);
}

}  // namespace us
