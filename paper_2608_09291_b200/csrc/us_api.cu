// C ABI of the library (declared in include/unionsparse.h): handle management, upload, launch.
#include <algorithm>
#include <atomic>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <exception>
#include <map>
#include <memory>
#include <mutex>
#include <new>
#include <utility>
#include <vector>

#include <cuda.h>

#include "us_host.h"
#include "us_launch.h"
#include "us_load.h"
#include "us_spmm_kernel.cuh"
#include "us_spmm_tc.cuh"
#include "us_spmm_ahead.cuh"
#include "us_quant_kernels.cuh"

// How one N class is launched: fixed when the handle is made, so that a call is left with filling in its
// pointers and launching.
struct LaunchGeom {
    int nt, cls, warps, stages, smem, lut_rep;
    uint32_t slot_bytes;
    bool xp;
};
struct Kernel {
    const void* symbol = nullptr;      // nullptr where no such kernel is built
    cudaFunction_t fn = nullptr;       // on the handle's device, once it is loaded (load_kernel)
};
struct KernelForms {
    Kernel plain, chained, single, timed;
};
struct ClassPlan {
    bool ok = false;
    LaunchGeom g{};
    KernelForms fn;
    us::SpmmParams p{};   // everything but the call's pointers, N and the absmax range
};

// The same for us_spmm_tc_kernel, per number of 8-token groups.
struct TcPlan {
    bool ok = false;
    int octets = 2, threads = 0, smem = 0;
    Kernel plain, chained;
    us::TcParams p{};
};

// The same for us_spmm_ahead_kernel, per N class.
struct AheadPlan {
    bool ok = false;
    bool always = false;                 // whatever ran before; otherwise only behind a call of half an SM (ahead_plan)
    bool chain_ok = false;               // chained calls, too
    int threads = 0, smem = 0;
    Kernel plain, chained;
    us::AheadParams p{};
};

// A split of the tiles over the CTAs (make_schedule), for one length of K ranges.
struct Schedule {
    std::vector<uint32_t> begin;
    int strips = 1;
};

struct us_handle {
    us::HostMatrix host;
    std::map<int, Schedule> schedules;   // by segments of a K range, while the plans are laid
    AheadPlan ahead[3];              // NT = 1, 2, 4
    TcPlan tc[9];                    // index: 8-token groups of the call
    ClassPlan plan[4];               // per N class (NT = 1, 2, 4, 8)
    bool on_device = false;
    int device = -1;
    int sm_count = 148;               // (host-only handles plan for a 148-SM part)
    int max_N = 0;
    int max_smem = 227 * 1024;
    uint8_t* d_blob = nullptr;
    uint32_t* d_item_off = nullptr;
    std::vector<uint32_t> cta_begin[4];  // schedule per N class (NT = 1, 2, 4, 8)
    int G[4] = {1, 1, 1, 1};          // segments per K range, per class
    int s_local[4] = {0, 0, 0, 0};    // strips held in shared memory (0 = direct mode), per class
    bool xp[4] = {false, false, false, false};   // X staged packed (half the shared memory), per class
    int32_t* d_row_order = nullptr;
    uint16_t* d_w_scale = nullptr;
    int32_t* d_acc = nullptr;
    uint32_t* d_cnt = nullptr;
    uint32_t* d_err = nullptr;
    uint8_t* d_xq = nullptr;          // chained calls: packed INT4 codes of the activations, then their scales
    size_t xq_bytes = 0;              // bytes of the codes (the fp16 scales follow, 256-byte aligned)
    unsigned long long* d_timers = nullptr;
    bool timers_on = false;
    size_t acc_bytes = 0, cnt_bytes = 0;
    uint32_t withhold = 0xFFFFFFFFu;   // test hook (us_debug_withhold_copy)
    uint32_t wait_ns_hi = 2000000u;    // bounded waits: ~2 s
    cudaError_t sticky = cudaSuccess;
};

namespace {


int nt_for(int N) { return N <= 8 ? 1 : N <= 16 ? 2 : N <= 32 ? 4 : 8; }
int class_of(int nt) { return nt == 1 ? 0 : nt == 2 ? 1 : nt == 4 ? 2 : 3; }

// Experiment knobs, overridable from the environment (read once per process). Everything else the
// plan decides from the shape.
int env_int(const char* name, int fallback)
{
    const char* v = std::getenv(name);
    return (v && *v) ? std::atoi(v) : fallback;
}
int pdl_knob() { static int v = env_int("US_PDL", 1); return v; }          // programmatic dependent launch
int stages_knob() { static int v = env_int("US_STAGES", 0); return v; }    // ring slots per warp, 0 = automatic
// (up to 20 for the N <= 8 kernels; the other kernels are compiled for 16)
int max_warps() { static int v = std::min(20, std::max(2, env_int("US_MAX_WARPS", 16))); return v; }
int tc_knob() { static int v = env_int("US_TC", 1); return v; }   // tensor-memory kernel: 0 never, 1 by rule, 2 wherever it can run
int tc_oct_knob() { static int v = env_int("US_TC_OCT", 0); return v; }   // its octets: 0 by rule
int ahead_knob() { static int v = env_int("US_AHEAD", 1); return v; }   // decode-ahead kernel: 0 never, 1 by rule, 2 wherever it can run
int coresident_knob() { static int v = env_int("US_CORESIDENT", 1); return v; }  // small problems: half an SM per CTA
constexpr int kLocalAccBudget = 32 * 1024;   // local strip sums a K-range width is chosen with
constexpr int kLocalAccCap = 48 * 1024;      // ... and what is taken if nothing fits that
constexpr int kMinWarps = 12;                // warps the automatic K-range choice keeps room for
constexpr int kCoresidentTiles = 16;         // most tiles per CTA for the half-SM plan
constexpr int kCoresidentK = 5120;           // ... and widest K: its few threads stage all of X (N = 8, half SM / whole: 2304 x 8192 6.8 / 5.9 us,
                                             // 2304 x 6144 6.4 / 5.6, 4096 x 4096 4.6 / 5.6)
// The same where K is not a multiple of 32 and staging takes a thread one unit at a time (half SM / whole: N = 8
// 1500 x 4500 6.7 / 5.8 (N = 1, which shares the plan, loses by it, 5.3 / 5.6), 2304 x 4500 7.3 / 6.5, 2304 x 3000 5.5 / 5.4; N = 1 there 4.4 / 5.2).
int64_t coresident_K(int64_t K) { return K % 32 == 0 ? kCoresidentK : 3072; }
constexpr int kHalfSmBytes = 228 * 1024 / 2 - 1024 - 512;   // shared memory of a half-SM CTA: 228 KB per SM, 1 KB reserved per CTA

// Segments per K range for an N class. The int8 activations of one K range live in shared memory
// next to the warps' tile slots, so fewer, longer ranges (fewer partial-sum flushes) cost warps.
// Returns the range length of the split into the fewest equal ranges, not fewer than min_ranges,
// that still leaves room for min_warps one-slot warps (measured: 15 warps and one range beat
// 16 warps and two ranges by 25 % on a 13824 x 5120 matrix at N = 16).
// Shared memory of one K range's activations: int8 (one byte per token and k, 32 bytes of pad per
// token row) or packed (half of that).
// Ring slot: the largest tile plus the two payload rows the decode's window loads may read past a
// stream's end (rows are 128 bytes per column area).
uint32_t slot_bytes_for(const us::HostMatrix& hm)
{
    const uint32_t streams = hm.w2 ? 1u : (uint32_t)hm.fmt.C_A;
    return (hm.max_item_bytes + 256u * streams + 127u) & ~127u;
}

int64_t x_bytes(int nt, int64_t G, int K_L, bool xp)
{
    return (int64_t)nt * 8 * us::x_row_bytes((int)(G * K_L), xp);
}

// The schedule for K ranges of G segments: the classes and both kernels ask for the same ones.
const Schedule& schedule(us_handle* h, int G)
{
    const auto it = h->schedules.find(G);
    if (it != h->schedules.end()) return it->second;
    Schedule& s = h->schedules[G];
    us::make_schedule(h->host, h->sm_count, G, &s.begin, &s.strips);
    return s;
}

int segs_per_range(const us::HostMatrix& hm, int nt, int limit, int64_t min_ranges, bool xp)
{
    const int64_t n_segs = hm.n_segs;
    const int slot = (int)slot_bytes_for(hm);
    const int acc = nt * 512 * 2 <= kLocalAccBudget ? kLocalAccBudget : 0;
    const int other = 256 * 8 * 4 + (int)us::kLutScratchBytes + acc + 2 * us::kOffTable * 4 + 1280;
    for (int64_t r = std::max<int64_t>(1, min_ranges); r <= n_segs; ++r) {
        // A single range is worth more (no partial sums leave the CTA when the cuts fall on strip
        // boundaries): it may cost two more warps. Measured on 4096 x 11008, N = 8: one range with
        // 15 warps 9.8 us, two ranges with 16 warps 14.7 us.
        const int want = std::min(max_warps(), r == 1 ? std::min(10, kMinWarps) : kMinWarps);
        const int64_t G = (n_segs + r - 1) / r;
        const int64_t xb = x_bytes(nt, G, hm.fmt.K_L, xp) + G * nt * 32;
        if ((limit - other - xb) / slot >= want) return (int)G;
    }
    return 1;
}

const void* kernel_for(int cls, bool any_k, const us::KernelKey& k)
{
    switch (cls) {
        case 0: return any_k ? us::kernel_nt<1, true>(k) : us::kernel_nt<1, false>(k);
        case 1: return any_k ? us::kernel_nt<2, true>(k) : us::kernel_nt<2, false>(k);
        case 2: return any_k ? us::kernel_nt<4, true>(k) : us::kernel_nt<4, false>(k);
        default: return any_k ? us::kernel_nt<8, true>(k) : us::kernel_nt<8, false>(k);
    }
}

// The kernels that calls on this handle launch under a plan.
KernelForms kernel_forms(const us_handle* h, int cls, int stages, bool local, bool xp)
{
    us::KernelKey k{stages, local, false, xp, false, h->host.fmt.C_A == 2, h->host.w2, false};
    const bool any_k = h->host.K % 32 != 0;
    KernelForms f;
    f.plain.symbol = kernel_for(cls, any_k, k);
    k.am = true;
    f.chained.symbol = kernel_for(cls, any_k, k);
    k.am = false; k.dp = true;   // a single token: dp4a beats the MMA (measured 2-3 %)
    f.single.symbol = kernel_for(cls, any_k, k);
    k.dp = false; k.timed = true;
    f.timed.symbol = kernel_for(cls, any_k, k);
    return f;
}

// The most warps with which two CTAs of each of them share an SM's registers: 16384 to a scheduler, allocated 8 a thread
// at a time. (The stage-timer builds need more and do not share one.)
int half_sm_warps(const us_handle* h, int cls, bool local, bool xp)
{
    if (h->device < 0) return (cls == 0 ? 12 : 10) - (h->host.fmt.C_A == 2 ? 2 : 0);   // host-only handle: what it comes to today
    const KernelForms f = kernel_forms(h, cls, 1, local, xp);
    int regs = 0;
    for (const void* fn : {f.plain.symbol, f.chained.symbol, f.single.symbol}) {
        if (!fn) continue;
        cudaFuncAttributes fa;
        if (cudaFuncGetAttributes(&fa, fn) != cudaSuccess) { cudaGetLastError(); return 0; }
        regs = std::max(regs, fa.numRegs);
    }
    return regs ? 2 * (16384 / (32 * ((regs + 7) / 8 * 8))) : 0;
}

// Shared-memory layout of us_spmm_kernel: selector table, int8 X of one K range, per-(segment,
// token) sums, mbarriers, claim counter, local strip accumulators + counters, per-warp rings.
bool plan_launch(const us_handle* h, int N, LaunchGeom* g)
{
    g->nt = nt_for(N);
    g->cls = class_of(g->nt);
    const int G = h->G[g->cls], s_local = h->s_local[g->cls];
    g->xp = h->xp[g->cls];
    g->slot_bytes = slot_bytes_for(h->host);
    // selector table copies: 32 (conflict-free lookups) when that costs no warp, else 8
    int lut_rep = 32;
    auto fixed_for = [&](int rep) {
        return 256 * rep * 4 + (int)us::kLutScratchBytes + (int)x_bytes(g->nt, G, h->host.fmt.K_L, g->xp) + G * g->nt * 8 * 4 +
                           us::kClaimWords * 4 + s_local * (g->nt * 128 + 1) * 4 + 2 * us::kOffTable * 4 + 128;
    };
    int fixed_base = fixed_for(lut_rep);
    const int limit = h->max_smem;
    // Ring depth: two slots per warp when that still gives (nearly) all the warps; else one slot per
    // warp and more warps -- measured on the 70B-shaped FFN: 16 warps x 1 slot beat 9 warps x 2.
    auto warps_for = [&](int stages) {
        const int fixed = fixed_base + 32 * stages * 8;
        return std::min((limit - fixed) / (int)(stages * g->slot_bytes),
                        (g->nt == 1 && h->host.fmt.C_A == 1) ? max_warps() : std::min(16, max_warps()));
    };
    {
        const int w32 = std::max(warps_for(1), warps_for(2));
        fixed_base = fixed_for(8);
        const int w8 = std::max(warps_for(1), warps_for(2));
        // 32 copies only for long-running CTAs (measured: 1 % faster on the 70B-shaped FFN, but the
        // 4096 x 4096 case -- about one tile per warp -- loses 5 % to the bigger table)
        const int64_t n_cta = h->sm_count;
        const bool long_run = (h->host.n_items + n_cta - 1) / n_cta >= 4 * (int64_t)w8;
        if (w32 >= w8 && long_run) { lut_rep = 32; fixed_base = fixed_for(32); } else { lut_rep = 8; }
    }
    int stages = stages_knob() > 0 ? stages_knob() : (warps_for(1) >= warps_for(2) + 3 ? 1 : 2);
    int warps = warps_for(stages);
    if (warps < 2) return false;
    // Small problems at N <= 8 (a CTA sees about a tile per warp): take at most half an SM -- shared
    // memory and registers -- with one slot per warp, so that the next launch's CTA moves in beside
    // this one and runs its latency-bound prologue (parameters, offsets, first tile copies, table)
    // under this one's work; with one CTA per SM, programmatic dependent launch alone hides only the
    // launch latency, because all CTAs of a launch end at about the same time.
    // Measured on 4096 x 4096, N = 8: 6.6 -> 5.7 us; not worth it from ~20 tiles per CTA on.
    const int64_t n_cta = h->sm_count;
    const int64_t per_cta = (h->host.n_items + n_cta - 1) / n_cta;
    // the most tiles a CTA has: cuts fall on strip boundaries, so it can be more than the average (5008 x 3008, 3 tiles to a
    // strip: most CTAs have two strips, some three, and eight warps would need a second round for the ninth tile: 5.7 us
    // against 5.2 with 16 warps on the whole SM; 3000 x 6000 11.7 against 8.7; 512 x 8192, where 32 CTAs have a strip of 32
    // tiles each and the others none: 8.9 against 5.8)
    int64_t most = per_cta;
    for (size_t c = 0; c + 1 < h->cta_begin[g->cls].size(); ++c)
        most = std::max<int64_t>(most, (int64_t)h->cta_begin[g->cls][c + 1] - h->cta_begin[g->cls][c]);
    int fixed = fixed_base + 32 * stages * 8;
    // (us_spmm_ahead_kernel takes nearly all of these calls; what is left for this plan is said at build_ahead_plan, and tiles of
    // 2048 columns and more. At N = 9 .. 16 those leave too few slots, but at 90 % sparsity, and there half an SM is no better: 4096 x 4096
    // 7.3 / 7.6, 2048 x 4096 8.7 / 7.2, 3072 x 4096 9.1 / 7.4.)
    if (coresident_knob() && g->nt == 1 && most <= kCoresidentTiles && stages_knob() == 0 && h->host.Kp <= coresident_K(h->host.K)) {
        const int half = kHalfSmBytes;
        const int fixed8 = fixed_for(8) + 32 * 8;
        // (two column areas: 10 at most; 3001 x 2000, N = 8 4.10 us with 10, 4.18 with 12)
        int w = std::min({half_sm_warps(h, g->cls, s_local > 0, g->xp && s_local > 0), h->host.fmt.C_A == 2 ? 10 : 16, max_warps()});
        while (w >= 8 && fixed8 + w * (int)g->slot_bytes > half) --w;
        // (only if every tile of the CTA finds a warp at once: 1500 x 6000 has 12 and room for 10: N = 8 8.6 us against 6.0 with
        // 16 warps on the whole SM)
        if (w >= 8 && w >= most) { stages = 1; lut_rep = 8; warps = w; fixed = fixed8; }
    }
    g->stages = stages;
    g->lut_rep = lut_rep;
    g->warps = warps;
    g->smem = fixed + warps * stages * (int)g->slot_bytes;
    return true;
}

// Chooses, per N class, the K-range width, whether strips are summed in shared memory, and whether
// X is staged packed.
void plan_classes(us_handle* h)
{
    const int n_cta = h->sm_count;
    std::vector<uint32_t> (&sched)[4] = h->cta_begin;
    const int limit = h->max_smem;
    for (int c = 0; c < 4; ++c) {
        const int nt = 1 << c;
        // Local mode needs the strip sums of a CTA's share of one K range in shared memory; a short
        // last range spreads a CTA over more strips, so shorter ranges are tried before giving up.
        // Returns the range length found (0 = none) and leaves the schedule in `out`.
        auto local_plan = [&](bool xp, std::vector<uint32_t>* out, int* s_local) -> int {
            // second pass: a little more than the budget the range length was chosen with is taken
            // if nothing fits the budget and at least 11 warps remain -- the alternative is the global
            // split-K path for every tile (N = 32: 5120 x 13824 30.2 -> 22.4 us, 4096 x 11008 18.7 ->
            // 16.2 us; N = 64 on 5120 x 5120 25.3 -> 19.5 us)
            for (int pass = 0; pass < 2; ++pass) {
                int G = 0, worst = 1;
                for (int64_t r = 1; r <= h->host.n_segs; ++r) {
                    const int Gr = segs_per_range(h->host, nt, limit, r, xp);
                    if (Gr == G) continue;
                    G = Gr;
                    if (G <= 1) break;
                    const Schedule& sc = schedule(h, G);
                    *out = sc.begin;
                    worst = sc.strips;
                    const int need = worst * nt * 512;
                    if (pass == 0 && need <= kLocalAccBudget) { *s_local = worst; return G; }
                    if (pass == 1 && need <= kLocalAccCap) {
                        const int slot = (int)slot_bytes_for(h->host);
                        const int64_t fixed = 256 * 8 * 4 + (int64_t)us::kLutScratchBytes + need + 2 * us::kOffTable * 4 + 1280 +
                                              x_bytes(nt, G, h->host.fmt.K_L, xp) + (int64_t)G * nt * 32;
                        if ((limit - fixed) / slot >= 11) { *s_local = worst; return G; }
                    }
                }
            }
            return 0;
        };
        h->G[c] = 1;
        h->s_local[c] = 0;
        h->xp[c] = false;
        int sl = 0;
        const int G = local_plan(false, &sched[c], &sl);
        if (G > 0) { h->G[c] = G; h->s_local[c] = sl; }
        // Packed X (N <= 32: the kernel exists for those classes) halves the shared memory of a K
        // range at the price of three more integer instructions per n-tile and k-block. Worth it
        // when it turns several K ranges into one (then no partial sum leaves the CTA; N = 8 on
        // 5120 x 13824: 18.2 -> 15.1 us; where one range was enough already it costs 2-6 %).
        // Measured at N = 16: 28672 x 8192 38.4 -> 34.8 us and 4096 x 11008 17.9 -> 14.4 us (two
        // ranges become one); 5120 x 5120 12.0 -> 9.4 us (one range either way, but a CTA's share is
        // small and the staging pass and the freed shared memory count for more than the decode);
        // 13824 x 5120 15.7 -> 16.0 us (one range either way, long decode): not taken there.
        if (nt <= 4 && !h->host.w2) {   // (no packed-X kernel for INT2 weights)
            const int64_t n_segs = h->host.n_segs;
            const int64_t ranges = h->s_local[c] > 0 ? (n_segs + h->G[c] - 1) / h->G[c] : n_segs + 1;
            const bool small_share = nt >= 2 && (int64_t)h->host.blob_bytes / n_cta < 128 * 1024;
            if (ranges > 1 || small_share) {
                std::vector<uint32_t> alt;
                int sl2 = 0;
                const int G2 = local_plan(true, &alt, &sl2);
                const int64_t ranges2 = G2 > 0 ? (n_segs + G2 - 1) / G2 : 0;
                // (N = 32, packed against plain: 11008 x 4096 21.4 -> 18.5 us, 13824 x 5120 24.9 -> 23.6 us,
                // 5120 x 5120 17.3 -> 18.2 us with one range; three ranges instead of eleven one-segment
                // ranges on 4096 x 11008 were slower, 19.3 -> 26.4 us: only a single range pays)
                if (G2 > 0 && ranges2 == 1) {
                    h->G[c] = G2; h->s_local[c] = sl2; h->xp[c] = true;
                    sched[c] = alt;
                }
            }
        }
        // direct mode: one segment per range, every tile goes to the global workspace (longer ranges
        // and runs were measured: no gain at N = 32, the bigger X costs more than the adds it saves)
        if (h->s_local[c] == 0) sched[c] = schedule(h, 1).begin;
    }
}

// Gives the handle's device memory back, with its device current. Work that still uses it may be in flight on any
// stream: wait for it first, as cudaFree did.
void free_device(us_handle* h)
{
    int dev = -1;
    cudaGetDevice(&dev);
    if (dev != h->device) cudaSetDevice(h->device);
    cudaDeviceSynchronize();
    for (void* p : {(void*)h->d_blob, (void*)h->d_item_off, (void*)h->d_row_order, (void*)h->d_w_scale, (void*)h->d_acc,
                    (void*)h->d_cnt, (void*)h->d_err, (void*)h->d_xq})
        us::pool_free(h->device, p);
    cudaFree(h->d_timers);
    if (dev != h->device && dev >= 0) cudaSetDevice(dev);
}

// Argument checks shared by the two SpMM entry points.
us_status check_spmm_args(const us_handle* h, const void* X, int32_t N, const void* x_scale, const void* Y)
{
    if (!h || !X || !Y || N < 1 || N > h->max_N) return US_ERR_INVALID_ARG;
    if (!h->on_device) return US_ERR_UNSUPPORTED;
    if (x_scale && !h->d_w_scale) return US_ERR_INVALID_ARG;
    if (reinterpret_cast<uintptr_t>(X) % 16) return US_ERR_INVALID_ARG;
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess) return US_ERR_CUDA;
    if (dev != h->device) return US_ERR_INVALID_ARG;   // the handle's arrays live on another GPU
    return US_OK;
}

// Lays a class's launch down: geometry and every kernel parameter that no call changes.
void build_plan(us_handle* h, int cls)
{
    ClassPlan& pl = h->plan[cls];
    LaunchGeom& g = pl.g;
    pl.ok = plan_launch(h, 8 << cls, &g);
    if (!pl.ok) return;
    pl.fn = kernel_forms(h, cls, g.stages, h->s_local[cls] > 0, g.xp && h->s_local[cls] > 0);
    const us::HostMatrix& hm = h->host;
    us::SpmmParams& p = pl.p;
    std::memset(&p, 0, sizeof(p));
    p.blob = h->d_blob; p.item_off = h->d_item_off;
    std::memcpy(p.cta_begin, h->cta_begin[cls].data(), h->cta_begin[cls].size() * sizeof(uint32_t));
    p.G = h->G[cls]; p.s_local = h->s_local[cls]; p.lut_rep = g.lut_rep;
    {
        const int64_t n_kr = (hm.n_segs + p.G - 1) / p.G;
        const int64_t g_last = hm.n_segs - (n_kr - 1) * p.G;
        auto magic = [](uint64_t d) { return ((1ull << 40) / d) + 1ull; };
        p.mg_g = magic((uint64_t)p.G);
        p.mg_glast = magic((uint64_t)g_last);
        p.mg_krs = magic((uint64_t)hm.n_strips * (uint64_t)p.G);
        // Claim runs of up to a whole strip's segments of the range (the partial sums of a run stay
        // in registers; the kernel shortens the runs towards the end of a CTA's range), but never
        // so long that a CTA's warps run out of runs to share.
        const int64_t per_cta = std::max<int64_t>(1, hm.n_items / h->sm_count);
        const int balanced = (int)std::max<int64_t>(1, per_cta / (4 * (int64_t)g.warps));
        p.run_len = std::max(1, std::min(std::min(p.G, 2 * balanced), p.G));
        // Fewer tiles than warps: one tile per warp, all at once (1024 x 1024, N = 8: 4.1 -> 3.1 us); with more
        // tiles than warps, runs of two keep a run's sums in registers and win (4096 x 4096: 5.7 against 6.3 us).
        if ((hm.n_items + h->sm_count - 1) / h->sm_count <= g.warps) p.run_len = 1;
    }
    p.row_order = h->d_row_order; p.w_scale = h->d_w_scale;
    p.err = h->d_err;
    p.M = (int32_t)hm.M; p.K = (int32_t)hm.K;
    p.n_strips = (int32_t)hm.n_strips; p.n_segs = (int32_t)hm.n_segs;
    p.mask_rows = hm.mask_rows; p.K_L = hm.fmt.K_L;
    p.fold_kb = hm.fmt.C_A == 2 ? hm.nkb / 2 : 0;
    p.w2 = hm.w2 ? 1 : 0;
    p.slot_bytes = g.slot_bytes;
}

// Lays a launch of us_spmm_tc_kernel down for calls of `ng` 8-token groups.
void build_tc_plan(us_handle* h, int ng)
{
    TcPlan& pl = h->tc[ng];
    pl.ok = false;
    const us::HostMatrix& hm = h->host;
    if (ng < 2) return;
    us::TcParams& p = pl.p;
    std::memset(&p, 0, sizeof(p));
    const int64_t n_cta = h->sm_count;
    const int n_stage = hm.fmt.C_A == 1 ? (hm.mask_rows + 1) / 2 : hm.mask_rows;   // 256-column stages per tile
    const int64_t block_stages = hm.n_segs * n_stage;
    int64_t stages = (hm.n_strips + 15) / 16 * block_stages;
    if (block_stages >= (1 << 16) || stages >= (1 << 24)) return;   // exact division by multiplication
    // Where it is chosen. The kernel saves the X fragments, MMAs and split-K adds of every tile and gives all CTAs the same
    // number of stages; it pays a longer prologue and a flush through the workspace per CTA (4 to 5 us together at N = 64).
    // Where us_spmm_ahead_kernel takes the calls it is the better one. Against a plan of us_spmm_kernel that sums strips in
    // shared memory, whose time follows the largest share of a CTA (cuts fall on strip boundaries), straight lines in us
    // fit what was measured at s = .5 and .6, `share` and `mean` being the largest and the average CTA share in stages:
    //   N <= 16: that plan 5.9 + 1.08 share, this kernel 7.8 + 0.9 mean (20480 x 5120 17.6 / 17.5, 18432 x 6144 18.8 / 17.9, 27648 x 5120
    //            21.6 / 21.0, 20480 x 8192 26.0 / 23.3), from 10 stages on and with 1.6 us of margin: among other launches its code
    //            comes from L2 each time (a 13B-shaped chain with 27648 x 5120 on this kernel 74.3, on the other 72.2).
    //   N <= 32: 5.5 + 1.76 share, 7.5 + 1.1 mean (11008 x 4096 13.6 / 13.1, 4096 x 11008 14.7 / 12.3, 13824 x 5120 19.2 / 15.9,
    //            2048 x 8192 8.2 / 8.8), a us of margin, with INT2 weights 2.5 (11008 x 4096 11.8 / 12.4, 13824 x 5120 16.2 / 14.8). Where the
    //            order of the rows was changed its stores scatter, 7 us more here and 3 on a plan with one K range: 4 us of margin against those, 1.2 in ranges
    //            (rows sorted, densities .3 to .7: 11008 x 4096 16.2 / 20.9, 12288 x 4096 18.0 / 21.2, 16384 x 4096 21.7 / 23.3; in ranges 4096 x
    //            11008 19.5 / 19.5, with the weights in L2 15.3 / 15.7, at N = 20 17.0 / 15.5, 8192 x 8192 26.8 / 22.2; with .4 to .6 and .2 to .5 the same).
    //   N <= 64: from 2048 columns on (2048 x 2048 10.3 / 9.6, 4096 x 4096 16.6 / 14.2, 11008 x 4096 35 / 17.4), below that where
    //            CTAs have most of a stage (16384 x 512 19.3 / 16.0; 4096 x 1024, 0.4 stages, 8.8 / 9.7).
    // Against the direct mode it wins nearly always (N = 64 28672 x 8192 92 / 38).
    const int cls = class_of(nt_for(8 * ng));
    uint32_t most = 0;
    for (size_t c = 0; c + 1 < h->cta_begin[cls].size(); ++c) most = std::max(most, h->cta_begin[cls][c + 1] - h->cta_begin[cls][c]);
    const double mean = (double)stages / (double)n_cta, share = (double)most * n_stage / 16;
    bool scattered = false;   // a strip's rows are not one run of output rows
    for (int64_t i = 0; i + 16 <= hm.M && !scattered; i += 16)
        for (int64_t j = i; j < i + 16; ++j) scattered = scattered || hm.row_order[j] < i || hm.row_order[j] >= i + 16;
    const double margin = !scattered ? 0.0 : h->s_local[cls] > 0 && h->G[cls] == hm.n_segs ? 4.0 : 1.2;
    const bool better = cls <= 2 && h->ahead[cls].always ? false
                        : ng > 4                     ? hm.Kp >= 2048 || mean >= 0.8
                        : h->s_local[cls] == 0       ? mean >= 1.5
                        : ng <= 2                    ? mean >= 10 && 5.9 + 1.08 * share > 9.4 + 0.9 * mean
                                                     : 5.5 + 1.76 * share > (hm.w2 ? 10.0 : 8.5) + 1.1 * mean + margin;
    if (tc_knob() == 0 || (tc_knob() == 1 && !better)) return;
    p.slot_bytes = slot_bytes_for(hm);
    const int limit = h->max_smem;
    auto fixed_for = [&](int x_stages, int lut_rep) { return 256 * lut_rep * 4 + x_stages * ng * 2048 + 2048 + us::kTcFixedSmem; };
    auto slots_for = [&](int x_stages, int lut_rep) {
        return std::min(us::kTcMaxSlots, (limit - fixed_for(x_stages, lut_rep)) / (int)p.slot_bytes);
    };
    p.x_stages = 4;
    // Three octets (a kernel for N <= 16) where shares are long: two / three on 28672 x 8192, N = 16 29.3 / 28.0, with INT2
    // weights 25.7 / 24.7; 13824 x 5120, 7 stages, INT2 12.75 / 12.86.
    const int64_t stages3 = (hm.n_strips + 23) / 24 * block_stages;
    pl.octets = slots_for(3, 8) >= 24 && ng <= 2 && (tc_oct_knob() ? tc_oct_knob() == 3 : stages3 >= 8 * n_cta) ? 3 : 2;
    if (pl.octets == 3) { stages = stages3; p.x_stages = slots_for(4, 8) >= 24 ? 4 : 3; }
    const int warps = 8 * pl.octets;
    pl.threads = pl.octets == 3 ? us::TcShape<3>::kThreads : us::TcShape<2>::kThreads;
    // tiles of a warp: a CTA's stages may begin and end inside a tile
    const int64_t per_cta = (stages + n_cta - 1) / n_cta, tiles = (per_cta + n_stage - 1) / n_stage + (n_stage > 1 ? 1 : 0);
    if (std::min(per_cta, block_stages) > us::tc_max_run(hm.w2)) return;   // (from 5 * 10^9 weights on: the other kernel sums tile by tile)
    const int want = (int)std::min<int64_t>(3 * warps / 2, warps * tiles);   // slots worth having before the table gets its 32 copies
    while (p.x_stages > 2 && slots_for(p.x_stages, 8) < warps) --p.x_stages;
    p.lut_rep = slots_for(p.x_stages, 32) >= want && per_cta >= 16 ? 32 : 8;
    p.n_slots = std::min<int>(slots_for(p.x_stages, p.lut_rep), (int)(warps * tiles));
    if (p.n_slots < warps) return;
    pl.smem = fixed_for(p.x_stages, p.lut_rep) + p.n_slots * (int)p.slot_bytes;
    for (int64_t c = 0; c <= n_cta; ++c) p.cta_begin[c] = (uint32_t)(stages * c / n_cta);
    p.n_stage = n_stage; p.block_stages = (int32_t)block_stages;
    p.mg_block = ((1ull << 40) / (uint64_t)block_stages) + 1ull;
    p.blob = h->d_blob; p.item_off = h->d_item_off; p.row_order = h->d_row_order; p.w_scale = h->d_w_scale;
    p.err = h->d_err;
    p.M = (int32_t)hm.M; p.K = (int32_t)hm.K;
    p.n_strips = (int32_t)hm.n_strips; p.n_segs = (int32_t)hm.n_segs;
    p.mg_segs = ((1ull << 40) / (uint64_t)hm.n_segs) + 1ull;
    p.mask_rows = hm.mask_rows; p.K_L = hm.fmt.K_L;
    p.acc_nt = nt_for(8 * ng);
    pl.plain.symbol = us::kernel_tc(pl.octets, hm.K % 32 != 0, hm.fmt.C_A == 2, hm.w2, false);
    pl.chained.symbol = us::kernel_tc(pl.octets, hm.K % 32 != 0, hm.fmt.C_A == 2, hm.w2, true);
    pl.ok = true;
}

// Lays a launch of us_spmm_ahead_kernel down for the calls of an N class.
//
// Where it is chosen (us per call, us_spmm_kernel's plan / this, replayed graph; s = .5 unless it says; tiles: of 1024 columns,
// the largest CTA's share):
//   N <= 8: up to 64 tiles (1024 x 1024 3.1 / 2.2, 4096 x 4096 4.75 / 3.8, 11008 x 4096 8.8 / 6.6, 15360 x 5120, 33 tiles, 13.7 / 11.3,
//     27648 x 5120, 60 tiles, 19.0 / 18.7; 28672 x 8192 at .6, 97 tiles, 26.4 / 31.2: the other kernel's 16 warps on one CTA count from
//     there on), 46 with two column areas (20480 x 5120, 45 tiles, 14.6 / 14.6), 40 where K is cut in ranges or fewer than eight
//     slots are left (5120 x 13824, 31 tiles, 14.7 / 12.5; 11136 x 9388, 50 tiles and seven slots, 17.9 / 19.5).
//   N <= 16: up to 42 tiles (5120 x 5120 7.9 / 6.6, 11008 x 4096 10.1 / 8.2, 13824 x 5120, 30 tiles, 13.0 / 12.9, 22016 x 4096, 40 tiles,
//     16.7 / 15.9; 20480 x 5120, 45 tiles, 17.6 / 18.5). It is taken where alone it is no better, too: a CTA of the whole SM and one of
//     half an SM cannot overlap, and a change between the two kinds costs 3 to 8 us (the seven projections of a 13B-shaped
//     layer, four of 5120 x 5120, two of 13824 x 5120, one of 5120 x 13824: all whole 74, the first four half 73.5, all half 65).
//     Cut in ranges where the other plan has one range: 24 (4096 x 11008 13.4 / 10.7; 8192 x 8192, 28 tiles, 13.0 / 14.4). Two column areas: 28
//     and 24 (13824 x 5120 INT2 10.5 / 11.4, 5120 x 13824 16.2 / 17.7, 16384 x 4096, 28 tiles, INT2 12.7 / 11.2).
//   N <= 32: where all tiles are parked (4096 x 4096 8.7 / 6.4, 5120 x 5120 11.6 / 9.3; 11008 x 4096, 20 tiles, 13.7 / 16.9).
//   One segment to a strip and more than 8 tiles at N <= 8: not (24000 x 1024, 11 tiles, 4.9 / 5.6: the other half-SM plan has a warp
//     for every tile).
//   Otherwise, up to 64 tiles and with five slots at least: only behind calls of half an SM (ahead_plan), but at N = 9 .. 16 with two
//     column areas. Alone these calls are slower so (27648 x 5120, N = 16 20.0 / 21.3 at .7, with five slots 21.1 / 25.8 at .5; 8192 x 8192
//     12.9 / 13.5), among others the change of kind costs more: 13B-shaped layer, [Q;K;V] and [gate;up] stacked, N = 16, s = .3, .5, .6, .7,
//     all as they are alone / these behind the others: 72.4, 69.4, 68.4, 65.5 / 64.3, 60.8, 56.5, 53.8; seven products at .7 77.3 / 61.4; N = 8
//     stacked at .6, .7 57.4, 55.3 / 46.1, 44.6, 2 x 2 format at .5 54.0 / 45.7, INT2 50.6 / 42.0 (N = 16: 59.5 / 77.1, 50.5 / 68.4). With a
//     foreign kernel between all of these, which the library cannot know, .5 77.9 / 83.9, .7 76.1 / 74.7.
//   Chained calls: where all tiles are parked. The quantiser between two products takes the time in which later tiles would
//     have been decoded (13B-shaped chain, all half 80, like this 72, all whole 74).
void build_ahead_plan(us_handle* h, int cls)
{
    if (cls > 2 || ahead_knob() == 0) return;
    AheadPlan& pl = h->ahead[cls];
    const us::HostMatrix& hm = h->host;
    const int nt = 1 << cls;
    const bool plain = hm.fmt.C_A == 1;
    us::AheadParams& p = pl.p;
    std::memset(&p, 0, sizeof(p));
    p.slot_bytes = slot_bytes_for(hm);
    p.tile_cols = hm.mask_rows * hm.fmt.C_A * 8;
    const int places = us::kAheadCols / p.tile_cols;   // of parked tiles in each quarter of the tensor memory
    // The fewest K ranges whose X leaves room for six tile slots (5120 x 13824, N = 8: one range with five 16.3 us, two with
    // eight 12.5; N = 16: two with four 16.2, three with six 15.1).
    if (hm.n_items > (int64_t)us::kAheadMaxTiles * h->sm_count || hm.n_items * hm.fmt.K_L > 64 * 1024 * (int64_t)h->sm_count) return;
    int64_t most = 0;
    int warps = 8;
    int least = 6;   // tile slots
    auto lay = [&](int64_t r) {
        const int64_t G = (hm.n_segs + r - 1) / r;
        if ((hm.n_segs + G - 1) / G != r) return;
        const int64_t x = (int64_t)nt * 8 * us::ahead_x_row((int)std::min<int64_t>(G * hm.fmt.K_L, 1 << 20), hm.K % 32 != 0);
        // (no schedule is laid for ranges that cannot do: where not all can be parked, X and six slots beside it)
        const bool all_parked = hm.n_items <= 4 * places * (int64_t)h->sm_count;
        if (us::ahead_fixed_smem(nt, 1) + x + (all_parked ? 0 : least * (int64_t)p.slot_bytes) > kHalfSmBytes) return;
        const Schedule& sc = schedule(h, (int)G);
        const std::vector<uint32_t>& begin = sc.begin;
        const int strips = sc.strips;
        most = 1;
        bool one_range = true;   // to every CTA
        for (int c = 0; c < h->sm_count; ++c) {
            if (begin[c + 1] <= begin[c]) continue;
            most = std::max<int64_t>(most, (int64_t)begin[c + 1] - begin[c]);
            one_range = one_range && begin[c] / (hm.n_strips * G) == (begin[c + 1] - 1) / (hm.n_strips * G);
        }
        if (!one_range || most > us::kAheadMaxTiles) return;
        // Twelve decode warps and three that copy where 64 registers a thread do and there is work for them (with eight: 11008 x 4096,
        // N = 8 7.05, with twelve 6.6; 13824 x 5120, N = 16 13.5 / 12.9; 2048 x 2048, N = 8 the other way, 2.5 / 2.6). One copying warp less
        // is slower (20480 x 5120, N = 16 20.5 with one, 18.5 with three): each copy takes the issuing warp some 500 cycles.
        const bool wide = plain && (nt == 1 ? hm.K > kCoresidentK || most > 16 : nt == 2);
        warps = wide ? 12 : 8;
        pl.threads = 32 * (wide ? 16 : nt == 1 && plain ? 12 : nt <= 2 && most > 16 ? 12 : 10);
        if (4 * places < warps) return;
        const int64_t fixed = us::ahead_fixed_smem(nt, strips);
        auto slots_in = [&](int64_t bytes) { return (int32_t)std::min<int64_t>(most, std::max<int64_t>(0, bytes) / (int64_t)p.slot_bytes); };
        p.parked = (int32_t)std::min<int64_t>(most, 4 * places);
        p.n_slots = slots_in(kHalfSmBytes - fixed - x);
        p.x_over = p.parked == most && p.n_slots < std::min<int64_t>(most, warps) && fixed + x <= kHalfSmBytes ? 1 : 0;
        if (p.x_over) p.n_slots = slots_in(kHalfSmBytes - fixed);
        if (p.n_slots < std::min<int64_t>(most, least)) return;
        pl.smem = (int)(fixed + (p.x_over ? std::max<int64_t>(x, (int64_t)p.n_slots * p.slot_bytes) : x + (int64_t)p.n_slots * p.slot_bytes));
        std::copy(begin.begin(), begin.end(), p.cta_begin);
        p.n_ranges = (int32_t)r; p.G = (int32_t)G; p.s_local = strips;
    };
    auto fewest = [&](int slots, int ranges) {
        least = slots;
        for (int64_t r = 1; r <= ranges && p.n_ranges == 0; ++r) lay(r);
        return p.n_ranges > 0;
    };
    const bool six = fewest(6, 8);
    if (!six && !fewest(5, 8)) return;
    const int64_t share = most * hm.fmt.K_L / 1024;
    const bool more_ranges = p.n_ranges > 1 && h->s_local[cls] > 0 && h->G[cls] == hm.n_segs;   // than the other plan's one
    const bool better = !six       ? false
                        : cls == 0 ? share <= (p.n_ranges > 1 || p.n_slots < 8 ? 40 : plain ? 64 : 46) && (hm.n_segs > 1 || most <= 8)
                        : cls == 1 ? share <= (more_ranges || (!plain && p.n_ranges > 1) ? 24 : plain ? 42 : 28)
                                   : p.parked == most;
    const bool behind = (cls == 0 || (cls == 1 && plain)) && share <= 64 && h->plan[cls].g.smem > kHalfSmBytes && tc_knob() < 2;
    if (ahead_knob() == 1 && !better && !behind) return;
    if (!better && p.n_ranges > 1) {   // one range with five slots rather than more ranges
        const int ranges = p.n_ranges, slots = least;
        p.n_ranges = 0;
        if (!fewest(5, 1)) { least = slots; lay(ranges); }
    }
    pl.always = better || ahead_knob() == 2;
    p.tm_cols = 32;
    while (p.tm_cols < (p.parked + 3) / 4 * p.tile_cols) p.tm_cols *= 2;
    p.blob = h->d_blob; p.item_off = h->d_item_off; p.row_order = h->d_row_order; p.w_scale = h->d_w_scale;
    p.err = h->d_err;
    p.M = (int32_t)hm.M; p.K = (int32_t)hm.K;
    p.n_strips = (int32_t)hm.n_strips; p.n_segs = (int32_t)hm.n_segs;
    auto magic = [](int64_t d) { return ((1ull << 40) / (uint64_t)d) + 1ull; };
    p.mg_g = magic(p.G); p.mg_last = magic(hm.n_segs - (int64_t)(p.n_ranges - 1) * p.G); p.mg_range = magic(hm.n_strips * p.G);
    p.mask_rows = hm.mask_rows; p.K_L = hm.fmt.K_L;
    auto symbol = [&](bool am) {
        const bool any = hm.K % 32 != 0, fold = !plain;
        if (cls == 0) return any ? us::kernel_ahead<1, true>(warps, pl.threads, fold, hm.w2, am) : us::kernel_ahead<1, false>(warps, pl.threads, fold, hm.w2, am);
        if (cls == 1) return any ? us::kernel_ahead<2, true>(warps, pl.threads, fold, hm.w2, am) : us::kernel_ahead<2, false>(warps, pl.threads, fold, hm.w2, am);
        return any ? us::kernel_ahead<4, true>(warps, pl.threads, fold, hm.w2, am) : us::kernel_ahead<4, false>(warps, pl.threads, fold, hm.w2, am);
    };
    pl.plain.symbol = symbol(false);
    pl.chained.symbol = symbol(true);
    pl.ok = true;
    pl.chain_ok = pl.always && p.parked == most;
}

// Loads a kernel, opted in to the device's full dynamic shared memory (once per device, with that device current), so that
// us_spmm itself is nothing but a launch. Only what a handle's plans launch is loaded: a program's first handle takes 37 ms,
// 62 when it loaded every kernel of the aligned K.
cudaError_t load_kernel(int device, int smem_bytes, Kernel* k)
{
    static std::mutex mu;
    static std::map<std::pair<int, const void*>, cudaFunction_t> loaded;
    if (!k->symbol) return cudaSuccess;
    std::lock_guard<std::mutex> lock(mu);
    const auto it = loaded.find({device, k->symbol});
    if (it != loaded.end()) {
        k->fn = it->second;
        return cudaSuccess;
    }
    cudaError_t e = cudaFuncSetAttribute(k->symbol, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_bytes);
    if (e == cudaSuccess) e = cudaGetFuncBySymbol(&k->fn, k->symbol);
    if (e == cudaSuccess) loaded[{device, k->symbol}] = k->fn;
    return e;
}

// What a chained call adds to the plain one: the per-token absmax of a range of output rows, left
// for the quantiser of the next call.
struct ChainArgs {
    void* y_amax = nullptr;
    int64_t m0 = 0, m1 = 0;
};

// The driver's launch call, or nullptr. The runtime's looks the kernel up by its symbol on every call, among all that the
// library holds. 1024 x 1024, N = 8 into a new output, us of host time on two machines: 3.5 and 3.35 with the 128 kernels
// that there were before ragged K had its own, 3.9 with 240, 3.65 and 3.2 with the function in hand.
using DriverLaunch = CUresult (*)(const CUlaunchConfig*, CUfunction, void**, void**);
DriverLaunch driver_launch()
{
    static const DriverLaunch f = [] {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult r;
        if (cudaGetDriverEntryPointByVersion("cuLaunchKernelEx", &p, 12000, cudaEnableDefault, &r) != cudaSuccess) cudaGetLastError();
        return reinterpret_cast<DriverLaunch>(p);
    }();
    return f;
}

us_status launch(us_handle* h, const Kernel& kernel, void* params, int threads, int smem, cudaStream_t st)
{
    // Launched with programmatic stream serialization: the kernel may start while its predecessor
    // in the stream is still running; it waits (griddepcontrol.wait) before it touches anything
    // an earlier kernel could produce or still use.
    void* args[1] = {params};
    if (const DriverLaunch f = driver_launch()) {
        CUlaunchAttribute attr[1];
        attr[0].id = CU_LAUNCH_ATTRIBUTE_PROGRAMMATIC_STREAM_SERIALIZATION;
        attr[0].value.programmaticStreamSerializationAllowed = pdl_knob() ? 1 : 0;
        CUlaunchConfig cfg = {};
        cfg.gridDimX = (unsigned)h->sm_count;
        cfg.blockDimX = (unsigned)threads;
        cfg.gridDimY = cfg.gridDimZ = cfg.blockDimY = cfg.blockDimZ = 1;
        cfg.sharedMemBytes = (unsigned)smem;
        cfg.hStream = st;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        const CUresult r = f(&cfg, kernel.fn, args, nullptr);
        if (r == CUDA_SUCCESS) return US_OK;
        if (r != CUDA_ERROR_INVALID_CONTEXT) {   // (a thread that has made no runtime call yet has none: the runtime makes it current)
            h->sticky = (cudaError_t)r;          // (the codes are the runtime's)
            return US_ERR_CUDA;
        }
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)h->sm_count);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = (size_t)smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = pdl_knob() ? 1 : 0;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    const cudaError_t e = cudaLaunchKernelExC(&cfg, kernel.symbol, args);
    if (e != cudaSuccess) { h->sticky = e; return US_ERR_CUDA; }
    return US_OK;
}

// The calling thread's last call: how many calls behind it on the stream take half an SM where they otherwise would not.
// Two behind a call whose CTAs take half an SM anyhow, so that theirs can start beside them (a stacked [gate; up] and the down
// projection behind it); such calls again and again go back to the whole SM. None where another kernel of the library, or a
// clear, comes in between.
struct LastCall {
    int device = -1;
    cudaStream_t stream = nullptr;
    int beside = 0;
};
thread_local LastCall t_last;

// The plan of us_spmm_ahead_kernel that a call on that stream takes, if any (see build_ahead_plan). timed: on the other
// kernel's timer build.
const AheadPlan* ahead_plan(const us_handle* h, int N, cudaStream_t st, bool chain, bool timed)
{
    const int cls = class_of(nt_for(N));
    if (cls > 2 || !h->ahead[cls].ok) return nullptr;
    const AheadPlan& a = h->ahead[cls];
    if (chain) return a.chain_ok ? &a : nullptr;
    if (timed && h->plan[cls].fn.timed.fn) return nullptr;
    if (a.always) return h->tc[(N + 7) / 8].ok ? nullptr : &a;
    return t_last.beside > 0 && t_last.stream == st && t_last.device == h->device ? &a : nullptr;
}

// The one launch path behind us_spmm, us_spmm_static_scratch and us_spmm_requant: fills the call's own
// parameters into a copy of the class's plan and launches.
us_status enqueue_spmm(us_handle* h, const void* X, int32_t N, const void* x_scale, void* Y, cudaStream_t st,
                       int32_t* acc, uint32_t* cnt, bool timers, const ChainArgs* chain = nullptr)
{
    const int cls = class_of(nt_for(N));
    const ClassPlan& pl = h->plan[cls];
    const AheadPlan* const ahead = ahead_plan(h, N, st, chain != nullptr, timers);
    const bool half = ahead ? ahead->always : !h->tc[(N + 7) / 8].ok && pl.g.smem <= kHalfSmBytes;
    t_last = {h->device, st, chain ? 0 : half ? 2 : ahead ? t_last.beside - 1 : 0};   // (behind a chained call a quantiser runs first)
    const TcPlan& tc = h->tc[(N + 7) / 8];
    if (tc.ok && !ahead) {
        us::TcParams p = tc.p;
        p.X = static_cast<const uint8_t*>(X);
        p.x_scale = static_cast<const uint16_t*>(x_scale);
        p.Y = Y; p.acc = acc; p.cnt = cnt;
        p.N = N;
        p.fp16_out = x_scale ? 1 : 0;
        if (chain) {
            p.y_amax = static_cast<uint32_t*>(chain->y_amax);
            p.amax_m0 = (int32_t)chain->m0; p.amax_m1 = (int32_t)chain->m1;
        }
        p.wait_ns_hi = h->wait_ns_hi;
        p.withhold = h->withhold;
        const Kernel& k = p.y_amax ? tc.chained : tc.plain;
        if (!k.fn) return US_ERR_UNSUPPORTED;
        return launch(h, k, &p, tc.threads, tc.smem, st);
    }
    if (ahead) {
        const AheadPlan& ah = *ahead;
        us::AheadParams p = ah.p;
        p.X = static_cast<const uint8_t*>(X);
        p.x_scale = static_cast<const uint16_t*>(x_scale);
        p.Y = Y; p.acc = acc; p.cnt = cnt;
        p.N = N;
        p.fp16_out = x_scale ? 1 : 0;
        if (chain) {
            p.y_amax = static_cast<uint32_t*>(chain->y_amax);
            p.amax_m0 = (int32_t)chain->m0; p.amax_m1 = (int32_t)chain->m1;
        }
        p.wait_ns_hi = h->wait_ns_hi;
        p.withhold = h->withhold;
        const Kernel& k = p.y_amax ? ah.chained : ah.plain;
        if (!k.fn) return US_ERR_UNSUPPORTED;
        return launch(h, k, &p, ah.threads, ah.smem, st);
    }
    if (!pl.ok) return US_ERR_UNSUPPORTED;
    const LaunchGeom& g = pl.g;
    us::SpmmParams p = pl.p;
    p.X = static_cast<const uint8_t*>(X);
    p.x_scale = static_cast<const uint16_t*>(x_scale);
    p.Y = Y; p.acc = acc; p.cnt = cnt;
    p.N = N;
    p.fp16_out = x_scale ? 1 : 0;
    if (chain) {
        p.y_amax = static_cast<uint32_t*>(chain->y_amax);
        p.amax_m0 = (int32_t)chain->m0; p.amax_m1 = (int32_t)chain->m1;
    }
    p.wait_ns_hi = h->wait_ns_hi;
    p.withhold = h->withhold;

    // (a variant without a timer build runs untimed)
    const bool timed = timers && !p.y_amax && pl.fn.timed.fn;
    const Kernel& k = p.y_amax ? pl.fn.chained : timed ? pl.fn.timed : N == 1 && !timers && pl.fn.single.fn ? pl.fn.single : pl.fn.plain;
    if (!k.fn) return US_ERR_UNSUPPORTED;
    p.timers = timed ? h->d_timers : nullptr;

    return launch(h, k, &p, g.warps * 32, g.smem, st);
}

// A 256-thread kernel, launched with programmatic stream serialization like the SpMM.
template <class... P, class... A>
cudaError_t launch_small(void (*kernel)(P...), dim3 grid, cudaStream_t st, A... args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(256);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = pdl_knob() ? 1 : 0;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}

// Frees a handle, whole or in the making.
struct DeleteHandle {
    void operator()(us_handle* h) const
    {
        if (h->d_blob) free_device(h);
        delete h;
    }
};
using HandlePtr = std::unique_ptr<us_handle, DeleteHandle>;

// us_encode after the checks of its arguments. May throw.
us_status encode(const int8_t* W, int64_t M, int64_t K, const uint16_t* w_scale, const us_format* fmt, int32_t max_N, uint32_t flags,
                 HandlePtr* out)
{
    HandlePtr owner(new us_handle());
    us_handle* h = owner.get();
    h->max_N = max_N;
    const bool host_only = (flags & US_ENCODE_HOST_ONLY) != 0;
    cudaError_t e = cudaSuccess;
    if (!host_only) {
        e = cudaGetDevice(&h->device);
        if (e == cudaSuccess) e = cudaDeviceGetAttribute(&h->sm_count, cudaDevAttrMultiProcessorCount, h->device);
        if (e == cudaSuccess) e = cudaDeviceGetAttribute(&h->max_smem, cudaDevAttrMaxSharedMemoryPerBlockOptin, h->device);
        if (e != cudaSuccess) return US_ERR_CUDA;
        if (h->sm_count > us::kMaxCtas) h->sm_count = us::kMaxCtas;
    }
    us_format f = fmt ? *fmt : us_format{16, us::default_K_L(M, K, h->sm_count), 2, 1};
    us_status s;
    // the kernel's index arithmetic (exact division by multiplication) needs u * d < 2^40 for every
    // position u < n_items and divisor d <= n_items
    auto too_many = [&] { return h->host.n_items >= (1 << 20) || h->host.n_segs >= (1 << 16); };
    if (host_only) {
        s = us::encode_host(W, M, K, w_scale, f, flags, 0, &h->host);
    } else {
        us::DeviceMatrix dm;
        s = us::encode_layout(W, M, K, w_scale, f, flags, 0, true, &h->host);
        if (s == US_OK && too_many()) s = US_ERR_UNSUPPORTED;
        if (s == US_OK) s = us::encode_device(W, h->device, flags, &h->host, &dm);
        h->d_blob = dm.blob; h->d_item_off = dm.item_off; h->d_row_order = dm.row_order;
    }
    if (s != US_OK) return s;
    const us::HostMatrix& hm = h->host;
    if (!hm.kernel_layout) {   // a format without a kernel: statistics and decoding only
        *out = std::move(owner);
        return US_OK;
    }
    if (too_many()) return US_ERR_UNSUPPORTED;
    const int nt_max = nt_for(max_N);
    auto lay_plans = [&] {
        for (int c = 0; c <= class_of(nt_max); ++c) { build_plan(h, c); build_ahead_plan(h, c); }
        for (int ng = 1; ng <= (max_N + 7) / 8; ++ng) build_tc_plan(h, ng);
        h->schedules.clear();
    };
    plan_classes(h);
    if (host_only) {
        lay_plans();   // (for us_launch_info)
        *out = std::move(owner);
        return US_OK;
    }

    h->acc_bytes = (size_t)hm.n_strips * nt_max * 128 * sizeof(int32_t);
    h->cnt_bytes = (size_t)hm.n_strips * sizeof(uint32_t);
    cudaStream_t ps = us::pool_stream(h->device);
    auto alloc = [&](auto** p, size_t bytes) {
        if (e == cudaSuccess) e = us::pool_alloc(h->device, (void**)p, bytes);
    };
    auto clear = [&](void* p, size_t bytes) {
        if (e == cudaSuccess) e = cudaMemsetAsync(p, 0, bytes, ps);
    };
    if (!hm.w_scale.empty()) {
        alloc(&h->d_w_scale, hm.w_scale.size() * 2);
        if (e == cudaSuccess) e = cudaMemcpyAsync(h->d_w_scale, hm.w_scale.data(), hm.w_scale.size() * 2, cudaMemcpyHostToDevice, ps);
        // chained calls need fp16 output, hence weight scales
        h->xq_bytes = (((size_t)max_N * (size_t)((hm.K + 1) / 2)) + 255) & ~(size_t)255;
        alloc(&h->d_xq, h->xq_bytes + 256);
    }
    alloc(&h->d_acc, h->acc_bytes); clear(h->d_acc, h->acc_bytes);
    alloc(&h->d_cnt, h->cnt_bytes); clear(h->d_cnt, h->cnt_bytes);
    alloc(&h->d_err, 16); clear(h->d_err, 16);
    if (e == cudaSuccess) e = cudaStreamSynchronize(ps);
    if (e != cudaSuccess) {
        cudaGetLastError();
        return e == cudaErrorMemoryAllocation ? US_ERR_ALLOC : US_ERR_CUDA;
    }
    h->on_device = true;
    lay_plans();
    if (!h->plan[class_of(nt_max)].ok) return US_ERR_UNSUPPORTED;   // a tile does not fit the shared-memory ring
    for (int c = 0; c < 4; ++c)
        if (c < 3 && h->ahead[c].ok) {
            for (Kernel* k : {&h->ahead[c].plain, &h->ahead[c].chained})
                if (e == cudaSuccess) e = load_kernel(h->device, h->max_smem, k);
            if (!h->ahead[c].chain_ok)
                for (Kernel* k : {&h->plan[c].fn.plain, &h->plan[c].fn.chained, &h->plan[c].fn.single})
                    if (e == cudaSuccess) e = load_kernel(h->device, h->max_smem, k);
        } else {
            for (Kernel* k : {&h->plan[c].fn.plain, &h->plan[c].fn.chained, &h->plan[c].fn.single})
                if (e == cudaSuccess) e = load_kernel(h->device, h->max_smem, k);
        }
    for (TcPlan& pl : h->tc)
        for (Kernel* k : {&pl.plain, &pl.chained})
            if (e == cudaSuccess) e = load_kernel(h->device, h->max_smem, k);
    if (e != cudaSuccess) return US_ERR_CUDA;
    *out = std::move(owner);
    return US_OK;
}

}  // namespace

extern "C" {

us_status us_encode(const int8_t* W, int64_t M, int64_t K, const uint16_t* w_scale,
                    const us_format* fmt, int32_t max_N, uint32_t flags, us_handle** out)
{
    if (out) *out = nullptr;
    if (!W || !out || M <= 0 || K <= 0 || max_N < 1 || max_N > 64) return US_ERR_INVALID_ARG;
    if (M > 0x7FFFFFF0ll || K > 0x7FFFFFF0ll) return US_ERR_INVALID_ARG;
    try {
        HandlePtr h;
        const us_status s = encode(W, M, K, w_scale, fmt, max_N, flags, &h);
        *out = h.release();
        return s;
    } catch (const std::exception&) {   // no host memory
        return US_ERR_ALLOC;
    }
}

us_status us_get_stats(const us_handle* h, us_stats* out)
{
    if (!h || !out) return US_ERR_INVALID_ARG;
    us::fill_stats(h->host, out);
    return US_OK;
}

us_status us_decode(const us_handle* h, int8_t* W_out)
{
    if (!h || !W_out) return US_ERR_INVALID_ARG;
    std::vector<uint8_t> fetched;   // (the handle is read only: several threads may decode it at once)
    const uint8_t* blob = h->host.blob.data();
    if (h->on_device) {
        try {
            fetched.resize((size_t)h->host.blob_bytes);
        } catch (const std::bad_alloc&) {
            return US_ERR_ALLOC;
        }
        if (cudaMemcpy(fetched.data(), h->d_blob, fetched.size(), cudaMemcpyDeviceToHost) != cudaSuccess) return US_ERR_CUDA;
        blob = fetched.data();
    }
    us::decode_host(h->host, blob, W_out);
    return US_OK;
}

us_status us_get_row_order(const us_handle* h, int32_t* perm_out)
{
    if (!h || !perm_out) return US_ERR_INVALID_ARG;
    if (!h->host.kernel_layout) {   // the paper's layout keeps the rows where they are
        for (int64_t r = 0; r < h->host.Mp; ++r) perm_out[r] = r < h->host.M ? (int32_t)r : -1;
        return US_OK;
    }
    std::memcpy(perm_out, h->host.row_order.data(), h->host.row_order.size() * sizeof(int32_t));
    return US_OK;
}

us_status us_launch_info(const us_handle* h, int32_t N, int32_t* grid, int32_t* block,
                         int32_t* smem_bytes)
{
    if (!h || N < 1 || N > h->max_N) return US_ERR_INVALID_ARG;
    if (!h->host.kernel_layout) return US_ERR_UNSUPPORTED;
    const TcPlan& tc = h->tc[(N + 7) / 8];
    const int cls = class_of(nt_for(N));
    const ClassPlan& pl = h->plan[cls];
    const AheadPlan* ah = cls <= 2 && h->ahead[cls].always ? &h->ahead[cls] : nullptr;
    if (!tc.ok && !ah && !pl.ok) return US_ERR_UNSUPPORTED;
    if (grid) *grid = h->sm_count;
    if (block) *block = tc.ok ? tc.threads : ah ? ah->threads : pl.g.warps * 32;
    if (smem_bytes) *smem_bytes = tc.ok ? tc.smem : ah ? ah->smem : pl.g.smem;
    return US_OK;
}

const char* us_launch_kernel(const us_handle* h, int32_t N, void* stream)
{
    if (us_launch_info(h, N, nullptr, nullptr, nullptr) != US_OK) return nullptr;
    return ahead_plan(h, N, static_cast<cudaStream_t>(stream), false, false) ? "us_spmm_ahead_kernel"
           : h->tc[(N + 7) / 8].ok                                             ? "us_spmm_tc_kernel"
                                                                               : "us_spmm_kernel";
}

us_status us_spmm(us_handle* h, const void* X, int32_t N, const void* x_scale, void* Y, void* stream)
{
    const us_status s = check_spmm_args(h, X, N, x_scale, Y);
    if (s != US_OK) return s;
    return enqueue_spmm(h, X, N, x_scale, Y, static_cast<cudaStream_t>(stream), h->d_acc, h->d_cnt, h->timers_on);
}

// ---- us_spmm_static_scratch: the SpMM with its scratch in a fixed device array ------------------
// The array lives in the library image: every GPU that loads the library holds it until exit.
// In host code `g_static_scratch` is only a stand-in for the symbol; the device address is looked
// up once per device with cudaGetSymbolAddress and that pointer is what the kernel receives.
static __device__ __align__(256) unsigned char g_static_scratch[US_STATIC_SCRATCH_BYTES];

namespace {
constexpr int kMaxDevices = 64;
std::atomic<void*> g_scratch_addr[kMaxDevices];   // zero-initialised; one look-up per device
}  // namespace

us_status us_spmm_static_scratch(us_handle* h, const void* X, int32_t N, const void* x_scale, void* Y,
                                 void* stream)
{
    const us_status s = check_spmm_args(h, X, N, x_scale, Y);
    if (s != US_OK) return s;
    const us::HostMatrix& hm = h->host;
    // scratch the kernel needs: INT32 strip sums, then one arrival counter per strip
    const size_t acc_bytes = (size_t)hm.n_strips * nt_for(N) * 128 * sizeof(int32_t);
    const size_t cnt_bytes = (size_t)hm.n_strips * sizeof(uint32_t);
    if (acc_bytes + cnt_bytes > (size_t)US_STATIC_SCRATCH_BYTES) return US_ERR_SCRATCH_TOO_SMALL;

    const int dev = h->device;   // checked above: it is the current device
    if (dev < 0 || dev >= kMaxDevices) return US_ERR_INVALID_ARG;
    void* ptr = g_scratch_addr[dev].load(std::memory_order_acquire);
    if (!ptr) {  // set-up, once per device, with that device current (threads racing here all
                 // look up the same address)
        const cudaError_t e = cudaGetSymbolAddress(&ptr, g_static_scratch);
        if (e != cudaSuccess || !ptr) { h->sticky = e; return US_ERR_CUDA; }
        g_scratch_addr[dev].store(ptr, std::memory_order_release);
    }
    unsigned char* scratch = static_cast<unsigned char*>(ptr);
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    // The array keeps the previous call's contents: sums and counters must start at zero.
    const cudaError_t e = cudaMemsetAsync(scratch, 0, acc_bytes + cnt_bytes, st);
    if (e != cudaSuccess) { h->sticky = e; return US_ERR_CUDA; }
    t_last.beside = 0;
    return enqueue_spmm(h, X, N, x_scale, Y, st, reinterpret_cast<int32_t*>(scratch),
                        reinterpret_cast<uint32_t*>(scratch + acc_bytes), false);
}

// ---- chained calls: fp16 in, INT4 inside, fp16 out ---------------------------------------------
namespace {
cudaError_t launch_quantize(const uint16_t* X16, int64_t ldx, int32_t N, int64_t K, const uint32_t* amax, uint8_t* Xq,
                            uint16_t* x_scale, cudaStream_t st)
{
    const int64_t units = (K + 7) / 8;
    t_last.beside = 0;
    const dim3 grid((unsigned)std::max<int64_t>(1, std::min<int64_t>(64, (units + 255) / 256)), (unsigned)N);
    return launch_small(us::us_quantize_f16_kernel, grid, st, X16, ldx, K, amax, Xq, x_scale);
}
}  // namespace

us_status us_spmm_requant(us_handle* h, const void* X16, int64_t ldx, const void* x_amax, int32_t N, void* Y16,
                          void* y_amax, int64_t amax_m0, int64_t amax_m1, void* stream)
{
    if (!h || !X16 || !x_amax || !Y16 || N < 1 || N > h->max_N) return US_ERR_INVALID_ARG;
    if (!h->on_device) return US_ERR_UNSUPPORTED;
    if (!h->d_w_scale) return US_ERR_INVALID_ARG;   // fp16 output needs the weight scales
    if (y_amax && h->host.fmt.C_A != 1) return US_ERR_UNSUPPORTED;   // no absmax-tracking kernel for folded tiles
    if (ldx < h->host.K) return US_ERR_INVALID_ARG;
    if (reinterpret_cast<uintptr_t>(X16) % 2 || reinterpret_cast<uintptr_t>(Y16) % 2 ||
        reinterpret_cast<uintptr_t>(x_amax) % 4 || reinterpret_cast<uintptr_t>(y_amax) % 4) return US_ERR_INVALID_ARG;
    if (y_amax && (amax_m0 < 0 || amax_m1 > h->host.M || amax_m0 > amax_m1)) return US_ERR_INVALID_ARG;
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess) return US_ERR_CUDA;
    if (dev != h->device) return US_ERR_INVALID_ARG;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (y_amax == x_amax) return US_ERR_INVALID_ARG;
    ChainArgs c;
    c.y_amax = y_amax; c.m0 = amax_m0; c.m1 = amax_m1;
    // One small kernel quantises the activations once into the handle's buffer; it is launched like
    // the SpMM kernels, so the SpMM's weight copies start while it runs. (Quantising inside the SpMM's
    // own staging was measured: every one of the 148 CTAs then pulls the fp16 activations through L2
    // and converts them -- 5 us more than this at N = 1, 8 to 15 us more at N = 16 and 32.)
    uint16_t* xs = reinterpret_cast<uint16_t*>(h->d_xq + h->xq_bytes);
    const cudaError_t e = launch_quantize(static_cast<const uint16_t*>(X16), ldx, N, h->host.K,
                                          static_cast<const uint32_t*>(x_amax), h->d_xq, xs, st);
    if (e != cudaSuccess) { h->sticky = e; return US_ERR_CUDA; }
    return enqueue_spmm(h, h->d_xq, N, xs, Y16, st, h->d_acc, h->d_cnt, h->timers_on, &c);
}

us_status us_absmax_f16(const void* X16, int64_t ldx, int32_t N, int64_t K, void* amax, void* stream)
{
    if (!X16 || !amax || N < 1 || N > 64 || K < 1 || ldx < K) return US_ERR_INVALID_ARG;
    if (reinterpret_cast<uintptr_t>(X16) % 2 || reinterpret_cast<uintptr_t>(amax) % 4) return US_ERR_INVALID_ARG;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const int64_t units = (K + 7) / 8;
    const unsigned gx = (unsigned)std::max<int64_t>(1, std::min<int64_t>(16, (units + 255) / 256));
    t_last.beside = 0;
    const cudaError_t e = launch_small(us::us_absmax_f16_kernel, dim3(gx, (unsigned)N), st, static_cast<const uint16_t*>(X16), ldx, K,
                                       (int)N, static_cast<uint32_t*>(amax));
    if (e != cudaSuccess) { cudaGetLastError(); return US_ERR_CUDA; }
    return US_OK;
}

us_status us_quantize_f16(const void* X16, int64_t ldx, int32_t N, int64_t K, const void* amax, void* Xq,
                          void* x_scale, void* stream)
{
    if (!X16 || !amax || !Xq || N < 1 || N > 64 || K < 1 || ldx < K) return US_ERR_INVALID_ARG;
    if (reinterpret_cast<uintptr_t>(X16) % 2 || reinterpret_cast<uintptr_t>(amax) % 4 ||
        reinterpret_cast<uintptr_t>(x_scale) % 2) return US_ERR_INVALID_ARG;
    const cudaError_t e = launch_quantize(static_cast<const uint16_t*>(X16), ldx, N, K, static_cast<const uint32_t*>(amax),
                                          static_cast<uint8_t*>(Xq), static_cast<uint16_t*>(x_scale),
                                          static_cast<cudaStream_t>(stream));
    if (e != cudaSuccess) { cudaGetLastError(); return US_ERR_CUDA; }
    return US_OK;
}

us_status us_last_error(us_handle* h)
{
    if (!h) return US_ERR_INVALID_ARG;
    if (!h->on_device) return US_OK;
    cudaError_t e = cudaDeviceSynchronize();
    uint32_t flag = 0;
    if (e == cudaSuccess) e = cudaMemcpy(&flag, h->d_err, 4, cudaMemcpyDeviceToHost);
    const bool failed = flag != 0 || h->sticky != cudaSuccess || e != cudaSuccess;
    if (failed) {
        // A call that gave up leaves partial sums and arrival counts behind: clear them, so that the
        // next call on this handle starts from the zeroed workspace it relies on.
        cudaMemset(h->d_err, 0, 4);
        cudaMemset(h->d_acc, 0, h->acc_bytes);
        cudaMemset(h->d_cnt, 0, h->cnt_bytes);
        cudaDeviceSynchronize();
    }
    if (h->sticky != cudaSuccess) { e = h->sticky; h->sticky = cudaSuccess; }
    if (e != cudaSuccess) { cudaGetLastError(); return US_ERR_CUDA; }
    if (flag == us::kErrTimeout) return US_ERR_DEVICE_TIMEOUT;
    return flag ? US_ERR_CUDA : US_OK;
}

us_status us_debug_withhold_copy(us_handle* h, int64_t position, int64_t wait_us)
{
    if (!h) return US_ERR_INVALID_ARG;
    if (!h->on_device) return US_ERR_UNSUPPORTED;
    if (position < 0) {
        h->withhold = 0xFFFFFFFFu;
        h->wait_ns_hi = 2000000u;
        return US_OK;
    }
    if (position >= h->host.n_items || wait_us < 1 || wait_us > 2000000) return US_ERR_INVALID_ARG;
    h->withhold = (uint32_t)position;
    h->wait_ns_hi = (uint32_t)std::max<int64_t>(1, wait_us * 1000 / 1024);
    return US_OK;
}

us_status us_stage_timers(us_handle* h, int32_t enable, uint64_t* out, int32_t n_out)
try {
    if (!h || (out && n_out < 8)) return US_ERR_INVALID_ARG;
    if (!h->on_device) return US_ERR_UNSUPPORTED;
    const size_t bytes = us::kTimerWords * sizeof(unsigned long long);
    if (!h->d_timers) {
        int dev = -1;
        cudaGetDevice(&dev);
        if (dev != h->device) cudaSetDevice(h->device);
        cudaError_t e = cudaSuccess;
        for (ClassPlan& pl : h->plan)
            if (e == cudaSuccess) e = load_kernel(h->device, h->max_smem, &pl.fn.timed);
        if (e == cudaSuccess) e = cudaMalloc((void**)&h->d_timers, bytes);
        if (e == cudaSuccess) e = cudaMemset(h->d_timers, 0, bytes);
        if (dev != h->device && dev >= 0) cudaSetDevice(dev);
        if (e != cudaSuccess) {
            cudaGetLastError();
            return e == cudaErrorMemoryAllocation ? US_ERR_ALLOC : US_ERR_CUDA;
        }
    }
    if (out) {
        if (cudaDeviceSynchronize() != cudaSuccess) return US_ERR_CUDA;
        std::vector<uint64_t> t((size_t)us::kTimerWords);
        if (cudaMemcpy(t.data(), h->d_timers, bytes, cudaMemcpyDeviceToHost) != cudaSuccess) return US_ERR_CUDA;
        // reduce the per-warp records
        uint64_t sum[6] = {0, 0, 0, 0, 0, 0}, ck[4] = {0, 0, 0, 0}, max_life = 0, t_min = ~0ull, t_max = 0;
        std::vector<uint64_t> cta((size_t)5 * us::kMaxCtas, 0);   // per CTA: start, first warp end, X staged, end, past the dependency wait
        for (int c = 0; c < us::kMaxCtas; ++c) {
            uint64_t st = ~0ull, first_end = ~0ull, xs = 0, en = 0, pw = 0;
            for (int w = 0; w < us::kMaxWarpsPerCta; ++w) {
                const uint64_t* R = t.data() + (size_t)us::kWarpRec * ((size_t)c * us::kMaxWarpsPerCta + w);
                if (!R[0]) continue;
                for (int i = 0; i < 4; ++i) sum[i] += R[1 + i];
                sum[4] += 1;
                sum[5] += R[5];
                max_life = std::max(max_life, R[4]);
                for (int i = 0; i < 4; ++i) ck[i] += R[9 + i];
                st = std::min(st, R[6]); first_end = std::min(first_end, R[8]); xs = std::max(xs, R[7]);
                en = std::max(en, R[8]); pw = std::max(pw, R[13]);
            }
            if (en) {
                t_min = std::min(t_min, st); t_max = std::max(t_max, en);
                cta[5 * c] = st; cta[5 * c + 1] = first_end; cta[5 * c + 2] = xs; cta[5 * c + 3] = en; cta[5 * c + 4] = pw;
            }
        }
        for (int i = 0; i < 6; ++i) out[i] = sum[i];
        out[6] = max_life;
        out[7] = t_max > t_min ? t_max - t_min : 0;   // first warp start to last warp end, ns
        // optional tail: prologue checkpoints, then five time stamps per CTA
        for (int i = 8; i < n_out; ++i) {
            const int j = i - 8;
            uint64_t v = 0;
            if (j < 4) v = ck[j];
            else if (j - 4 < 5 * us::kMaxCtas) v = cta[j - 4] ? cta[j - 4] - t_min : 0;
            out[i] = v;
        }
        cudaMemset(h->d_timers, 0, bytes);
    }
    if (enable >= 0) h->timers_on = enable != 0;
    return US_OK;
} catch (const std::exception&) {   // no host memory
    return US_ERR_ALLOC;
}

us_status us_destroy(us_handle* h)
{
    if (h) DeleteHandle()(h);
    return US_OK;
}

int64_t us_spmm_bytes(const us_handle* h, int32_t N, int32_t fp16_out)
{
    if (!h || N < 1) return -1;
    us_stats st;
    us::fill_stats(h->host, &st);
    const int64_t x = (int64_t)N * ((h->host.K + 1) / 2);
    const int64_t y = (int64_t)N * h->host.M * (fp16_out ? 2 : 4);
    const int64_t sc = fp16_out ? 2 * (h->host.M + N) : 0;
    return st.bytes_total + x + y + sc;
}

const char* us_status_string(us_status s)
{
    switch (s) {
        case US_OK: return "ok";
        case US_ERR_INVALID_ARG: return "invalid argument";
        case US_ERR_VALUE_RANGE: return "weight value outside [-8, 7]";
        case US_ERR_SHAPE: return "format parameters do not fit the tile";
        case US_ERR_UNSUPPORTED: return "format or call not supported";
        case US_ERR_ALLOC: return "allocation failed";
        case US_ERR_CUDA: return "CUDA error";
        case US_ERR_DEVICE_TIMEOUT: return "bounded device wait ran out";
        case US_ERR_SCRATCH_TOO_SMALL: return "problem needs more scratch than the fixed device array holds";
    }
    return "unknown status";
}

}  // extern "C"
