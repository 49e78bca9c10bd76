// Which instantiation of us_spmm_kernel a launch needs. The kernels are compiled in one translation unit
// per N class and kind of K (us_kernels.cu with US_NT = 1, 2, 4, 8 and US_ANY = 0, 1): they build in parallel, and a
// program loads only the units that it uses.
#pragma once

namespace us {

struct KernelKey {
    int stages;        // ring slots per warp, 1 or 2
    bool local;        // shared-memory strip sums
    bool timed;        // stage-timer build
    bool xp;           // activations staged packed
    bool am;           // absmax of the output
    bool fold;         // two column areas
    bool w2;           // INT2 weights
    bool dp;           // dp4a (a single token)
};

// The kernel for a key, or nullptr where no such variant is built.
template <int NT, bool ANY>   // ANY: K is not a multiple of 32
const void* kernel_nt(const KernelKey& k);
template <> const void* kernel_nt<1, false>(const KernelKey& k);
template <> const void* kernel_nt<2, false>(const KernelKey& k);
template <> const void* kernel_nt<4, false>(const KernelKey& k);
template <> const void* kernel_nt<8, false>(const KernelKey& k);
template <> const void* kernel_nt<1, true>(const KernelKey& k);
template <> const void* kernel_nt<2, true>(const KernelKey& k);
template <> const void* kernel_nt<4, true>(const KernelKey& k);
template <> const void* kernel_nt<8, true>(const KernelKey& k);

// us_spmm_ahead_kernel for N <= 8 NT (NT = 1, 2, 4) with so many decode warps and threads, in the same units; am = absmax of the output (default format only).
template <int NT, bool ANY>
const void* kernel_ahead(int warps, int threads, bool fold, bool w2, bool am);
template <> const void* kernel_ahead<1, false>(int warps, int threads, bool fold, bool w2, bool am);
template <> const void* kernel_ahead<2, false>(int warps, int threads, bool fold, bool w2, bool am);
template <> const void* kernel_ahead<4, false>(int warps, int threads, bool fold, bool w2, bool am);
template <> const void* kernel_ahead<1, true>(int warps, int threads, bool fold, bool w2, bool am);
template <> const void* kernel_ahead<2, true>(int warps, int threads, bool fold, bool w2, bool am);
template <> const void* kernel_ahead<4, true>(int warps, int threads, bool fold, bool w2, bool am);

// us_spmm_tc_kernel (us_spmm_tc.cu) with two or three octets: any_k = K is not a multiple of 32; fold = two column areas; am = absmax of the output (default format only).
const void* kernel_tc(int octets, bool any_k, bool fold, bool w2, bool am);

}  // namespace us
