// The instantiations of us_spmm_kernel for one N class: compiled once per class with -DUS_NT=1, 2, 4, 8.
#include "us_launch.h"
#include "us_spmm_kernel.cuh"

#ifndef US_NT
#error "compile with -DUS_NT=1, 2, 4 or 8"
#endif

namespace us {
namespace {

template <bool ANY, int ST, bool LA>
const void* pick(const KernelKey& k)
{
    constexpr int NT = US_NT;
    constexpr bool kPacked = NT <= 4 && LA;   // packed X: planned for these classes and local mode only
    if (k.w2) {          // INT2 weights in folded tiles: plain kernels only
        if (k.timed || k.xp || k.am || k.dp) return nullptr;
        return (const void*)us_spmm_kernel<ANY, NT, ST, LA, false, false, false, 2, true>;
    }
    if (k.fold) {        // folded tiles; stage timers for the N <= 8 kernels only
        if (k.am || k.dp) return nullptr;
        if constexpr (NT == 1)
            if (k.timed && !k.xp) return (const void*)us_spmm_kernel<ANY, NT, ST, LA, true, false, false, 2>;
        if (k.timed) return nullptr;
        if constexpr (kPacked)
            if (k.xp) return (const void*)us_spmm_kernel<ANY, NT, ST, LA, false, true, false, 2>;
        return k.xp ? nullptr : (const void*)us_spmm_kernel<ANY, NT, ST, LA, false, false, false, 2>;
    }
    if (k.am) {          // chained call
        if (k.timed || k.dp) return nullptr;
        if constexpr (kPacked)
            if (k.xp) return (const void*)us_spmm_kernel<ANY, NT, ST, LA, false, true, true>;
        return k.xp ? nullptr : (const void*)us_spmm_kernel<ANY, NT, ST, LA, false, false, true>;
    }
    if (k.dp) {
        if constexpr (NT == 1)
            if (!k.timed && !k.xp) return (const void*)us_spmm_kernel<ANY, NT, ST, LA, false, false, false, 1, false, true>;
        return nullptr;
    }
    if constexpr (kPacked)
        if (k.xp) return k.timed ? (const void*)us_spmm_kernel<ANY, NT, ST, LA, true, true> : (const void*)us_spmm_kernel<ANY, NT, ST, LA, false, true>;
    if (k.xp) return nullptr;
    return k.timed ? (const void*)us_spmm_kernel<ANY, NT, ST, LA, true> : (const void*)us_spmm_kernel<ANY, NT, ST, LA, false>;
}

template <bool ANY>
const void* pick_mode(const KernelKey& k)
{
    if (k.stages == 1) return k.local ? pick<ANY, 1, true>(k) : pick<ANY, 1, false>(k);
    return k.local ? pick<ANY, 2, true>(k) : pick<ANY, 2, false>(k);
}

const void* pick_kernel(const KernelKey& k) { return k.any_k ? pick_mode<true>(k) : pick_mode<false>(k); }

}  // namespace

#if US_NT == 1
const void* kernel_nt1(const KernelKey& k) { return pick_kernel(k); }
#elif US_NT == 2
const void* kernel_nt2(const KernelKey& k) { return pick_kernel(k); }
#elif US_NT == 4
const void* kernel_nt4(const KernelKey& k) { return pick_kernel(k); }
#else
const void* kernel_nt8(const KernelKey& k) { return pick_kernel(k); }
#endif

}  // namespace us
