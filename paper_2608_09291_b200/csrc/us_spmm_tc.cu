// The instantiations of us_spmm_tc_kernel.
#include "us_launch.h"
#include "us_spmm_tc.cuh"

namespace us {

const void* kernel_tc(bool fold, bool w2, bool am)
{
    if (w2) return am ? nullptr : (const void*)us_spmm_tc_kernel<2, true, false>;
    if (fold) return am ? nullptr : (const void*)us_spmm_tc_kernel<2, false, false>;
    return am ? (const void*)us_spmm_tc_kernel<1, false, true> : (const void*)us_spmm_tc_kernel<1, false, false>;
}

}  // namespace us
