// The instantiations of us_spmm_tc_kernel.
#include "us_launch.h"
#include "us_spmm_tc.cuh"

namespace us {
namespace {

template <int OCT, bool ANY>
const void* pick(bool fold, bool w2, bool am)
{
    if (w2) return am ? nullptr : (const void*)us_spmm_tc_kernel<OCT, 2, true, false, ANY>;
    if (fold) return am ? nullptr : (const void*)us_spmm_tc_kernel<OCT, 2, false, false, ANY>;
    return am ? (const void*)us_spmm_tc_kernel<OCT, 1, false, true, ANY> : (const void*)us_spmm_tc_kernel<OCT, 1, false, false, ANY>;
}

}  // namespace

const void* kernel_tc(int octets, bool any_k, bool fold, bool w2, bool am)
{
    if (any_k) return octets == 3 ? pick<3, true>(fold, w2, am) : pick<2, true>(fold, w2, am);
    return octets == 3 ? pick<3, false>(fold, w2, am) : pick<2, false>(fold, w2, am);
}

}  // namespace us
