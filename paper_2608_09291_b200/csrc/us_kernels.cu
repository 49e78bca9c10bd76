// The instantiations of us_spmm_kernel and us_spmm_ahead_kernel for one N class and one kind of K: compiled with -DUS_NT=1, 2, 4, 8 and -DUS_ANY=0, 1.
#include "us_launch.h"
#include "us_spmm_ahead.cuh"
#include "us_spmm_kernel.cuh"

#if !defined(US_NT) || !defined(US_ANY)
#error "compile with -DUS_NT=1, 2, 4 or 8 and -DUS_ANY=0 or 1"
#endif

namespace us {
namespace {

template <int ST, bool LA>
const void* pick(const KernelKey& k)
{
    constexpr int NT = US_NT;
    constexpr bool ANY = US_ANY;
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

}  // namespace

template <>
const void* kernel_nt<US_NT, US_ANY>(const KernelKey& k)
{
    if (k.stages == 1) return k.local ? pick<1, true>(k) : pick<1, false>(k);
    return k.local ? pick<2, true>(k) : pick<2, false>(k);
}

#if US_NT <= 4
template <>
const void* kernel_ahead<US_NT, US_ANY>(int warps, int threads, bool fold, bool w2, bool am)
{
    constexpr int NT = US_NT;
    constexpr bool ANY = US_ANY;
    if (!fold) {
        if constexpr (NT == 1)
            if (warps == 8 && threads == 32 * 12)
                return am ? (const void*)us_spmm_ahead_kernel<NT, 1, false, true, ANY, 8, 12> : (const void*)us_spmm_ahead_kernel<NT, 1, false, false, ANY, 8, 12>;
        if constexpr (NT <= 2)
            if (warps == 12 && threads == 32 * 16)
                return am ? (const void*)us_spmm_ahead_kernel<NT, 1, false, true, ANY, 12, 16> : (const void*)us_spmm_ahead_kernel<NT, 1, false, false, ANY, 12, 16>;
        if constexpr (NT > 2)
            if (warps == 8 && threads == 32 * 10)
                return am ? (const void*)us_spmm_ahead_kernel<NT, 1, false, true, ANY, 8, 10> : (const void*)us_spmm_ahead_kernel<NT, 1, false, false, ANY, 8, 10>;
        return nullptr;
    }
    if (warps != 8 || am) return nullptr;
    if constexpr (NT <= 2)
        if (threads == 32 * 12)
            return w2 ? (const void*)us_spmm_ahead_kernel<NT, 2, true, false, ANY, 8, 12> : (const void*)us_spmm_ahead_kernel<NT, 2, false, false, ANY, 8, 12>;
    if (threads != 32 * 10) return nullptr;
    return w2 ? (const void*)us_spmm_ahead_kernel<NT, 2, true, false, ANY, 8, 10> : (const void*)us_spmm_ahead_kernel<NT, 2, false, false, ANY, 8, 10>;
}
#endif

}  // namespace us
