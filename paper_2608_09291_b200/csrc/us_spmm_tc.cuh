// sm_100a SpMM on the 5th-generation tensor cores: the same tiles and the same decode as us_spmm_kernel, but the
// decoded weights go to tensor memory as the A operand of tcgen05.mma instead of through mma.sync in registers.
//
// Why: with mma.sync a warp loads the X fragments of every 8 tokens for every 16 x 32 weights it decodes, so from
// N = 16 on those loads, the MMAs and the split-K adds of every tile cost more than the decode (28672 x 8192 at 60 %
// sparsity: 24 us at N = 8, 32 at 16, 50 at 32, 87 at 64). Here a decoded k-block leaves the registers once,
// whatever N is; X is read from shared memory by the tensor core; partial sums stay in tensor memory over all of K.
//
//   decode    warps 0..15 in two octets (or 0..23 in three). A warp decodes 16-row tiles; the 8 tiles of an octet (same K segment) fill
//             the 128 lanes of one A operand: tcgen05.st.16x256b puts the lane's fragment bytes (rows g and g + 8,
//             columns 8t .. 8t + 7) where the MMA expects them, so the lane-stream layout needs no change.
//   MMA       one warp, one thread of it issues m128 nN k32 kind::i8 MMAs, 8 per 256-column stage, A from tensor memory.
//   X         the last warps expand the packed INT4 activations 256 columns at a time into a ring of operand-layout
//             stages (8-token groups x 16-byte k-columns), and sum them for the excess-8 correction.
//   flush     when an octet's run of K segments of one 128-row group ends, its warps read the sums back
//             (tcgen05.ld.16x256b gives mma.sync's accumulator layout) and store Y, or add to the split-K workspace.
//
// Work is cut in stages: 256 (384) rows x 256 columns (the octets share the stage's activations). A CTA owns a
// contiguous range of the (row block, column stage) order, the same number of stages for every CTA whatever the
// tile width: a warp enters a tile at any mask word by counting the set bits of the words before it.
// Tile copies form one ring of slots over the CTA's tiles in processing order; the warp that empties a slot refills
// it for whichever warp comes next, so any number of slots from one per warp on can be used.
#pragma once
#include "us_spmm_kernel.cuh"

namespace us {

// The CTA by number of octets: two, or three for N <= 16 (see the kernel).
template <int OCT>
struct TcShape {
    static constexpr int kDecode = 8 * OCT;              // decode warps
    static constexpr int kX = OCT == 2 ? 8 : 3;          // X warps
    static constexpr int kPair = OCT == 2 ? 2 : 1;       // X warps that share a stage
    static constexpr int kThreads = 32 * (kDecode + 1 + kX);
    static constexpr int kA = OCT == 2 ? 3 : 2;          // A stages per octet, 64 tensor-memory columns (256 of K) each
    static constexpr int kD = OCT == 2 ? 64 : 32;        // tensor-memory columns of an octet's sums, one a token
    static_assert(OCT * (kA * 64 + kD) <= 512, "tensor memory");
};
constexpr int kTcMaxOct = 3, kTcMaxA = 3;
constexpr int kTcMaxSlots = 64;
constexpr int kTcMaxXStages = 4;
constexpr int kTcSxRing = 16;         // row blocks whose activation sums are kept (see the X warps)
constexpr int kTcBars = kTcMaxSlots + 2 * kTcMaxOct * kTcMaxA + 2 * kTcMaxXStages + kTcMaxOct + 1;
constexpr int kTcMiscWords = 96 + kTcMaxSlots;
constexpr int kTcFixedSmem = kTcSxRing * 64 * 4 + kTcBars * 8 + kTcMiscWords * 4 + 1024;

// The most stages a run of one row block may have: its sums of 256 products per stage stay in tensor memory as INT32.
// INT4: raw byte (-128 .. 127) x 16 x (-128 .. 112), 2^14 at most -> 511; INT2: 4-bit field x 16 x, 15 * 128 -> 4369.
constexpr int64_t tc_max_run(bool w2) { return 0x7FFFFFFFll / (256 * (w2 ? 15 * 128 : 128 * 128)); }

struct TcParams {
    const uint8_t* blob;
    const uint32_t* item_off;
    const int32_t* row_order;
    const uint16_t* w_scale;
    const uint8_t* X;
    const uint16_t* x_scale;
    void* Y;
    int32_t* acc;
    uint32_t* cnt;
    uint32_t* err;
    int32_t M, K, N;
    int32_t n_strips, n_segs;
    unsigned long long mg_segs, mg_block;   // floor(2^40 / d) + 1 for d = n_segs, stages per row block
    int32_t n_stage, block_stages;          // stages per tile, per row block
    int32_t mask_rows, K_L;
    uint32_t slot_bytes;
    int32_t n_slots;              // ring slots, one per decode warp .. kTcMaxSlots
    int32_t x_stages;             // X stages in the ring
    int32_t lut_rep;
    int32_t acc_nt;               // n-tiles of the workspace's strip layout
    int32_t fp16_out;
    uint32_t* y_amax;
    int32_t amax_m0, amax_m1;
    uint32_t wait_ns_hi;
    uint32_t withhold;
    uint32_t cta_begin[kMaxCtas + 1];   // in stages
};

__device__ __forceinline__ void mbar_arrive(uint32_t bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
// Bounded wait for a whole warp, with one verdict for all its lanes (warp-wide tcgen05 instructions follow); gives up
// too when another warp of the CTA did. after: the wait cannot end before the stream's earlier work has, whose time is not
// counted, however long it runs with this kernel resident.
__device__ __forceinline__ bool tc_wait_warp(uint32_t bar, uint32_t parity, uint32_t limit_hi, volatile uint32_t* dead, bool after = false)
{
    if (__all_sync(0xffffffffu, mbar_try_wait(bar, parity))) return true;
    if (after) asm volatile("griddepcontrol.wait;" ::: "memory");
    const uint64_t t0 = global_timer_ns();
    const uint32_t nap = limit_hi < 64u ? 1000u : 20000u;
#pragma unroll 1
    for (uint32_t it = 0; it < (1u << 22); ++it) {
        if (__all_sync(0xffffffffu, mbar_try_wait_sleep(bar, parity, nap))) return true;
        if (__any_sync(0xffffffffu, *dead || ((global_timer_ns() - t0) >> 10) > limit_hi)) break;
    }
    return false;
}
// Waits, bounded, until a counter in shared memory has reached n.
__device__ __forceinline__ bool tc_wait_count(volatile uint32_t* count, uint32_t n, uint32_t limit_hi, volatile uint32_t* dead, bool after)
{
    if (__all_sync(0xffffffffu, *count >= n)) return true;
    if (after) asm volatile("griddepcontrol.wait;" ::: "memory");
    const uint64_t t0 = global_timer_ns();
#pragma unroll 1
    for (uint32_t it = 0; it < (1u << 24); ++it) {
        __nanosleep(100);
        if (__all_sync(0xffffffffu, *count >= n)) return true;
        if (__any_sync(0xffffffffu, *dead || ((global_timer_ns() - t0) >> 10) > limit_hi)) break;
    }
    return false;
}
__device__ __forceinline__ uint32_t tc_elect()
{
    uint32_t ok;
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xFFFFFFFF;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(ok));
    return ok;
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
// (issued by the elected lane only, as a predicate of the instruction: the code around it stays free of divergent
// branches, which keeps addresses and descriptors in uniform registers; from a divergent branch one MMA took 115 to
// 145 cycles to issue, like this 10)
__device__ __forceinline__ void tc_commit(uint32_t elected, uint32_t bar)
{
    asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %1, 0;\n\t"
                 "@q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n\t}" ::"r"(bar), "r"(elected) : "memory");
}
__device__ __forceinline__ void tc_st16(uint32_t addr, const uint32_t (&r)[16])
{
    asm volatile("tcgen05.st.sync.aligned.16x256b.x4.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};"
                 ::"r"(addr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]),
                 "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]) : "memory");
}
__device__ __forceinline__ void tc_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
// 16 lanes x 8 columns: an 8-token block in mma.sync accumulator order
__device__ __forceinline__ void tc_ld4(uint32_t addr, int (&c)[4])
{
    asm volatile("tcgen05.ld.sync.aligned.16x256b.x1.b32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(c[0]), "=r"(c[1]), "=r"(c[2]), "=r"(c[3]) : "r"(addr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tc_mma_i8(uint32_t elected, uint32_t d, uint32_t a, uint64_t b, uint32_t idesc, uint32_t accumulate)
{
    asm volatile("{\n\t.reg .pred p, q;\n\tsetp.ne.u32 q, %5, 0;\n\tsetp.ne.u32 p, %4, 0;\n\t"
                 "@q tcgen05.mma.cta_group::1.kind::i8 [%0], [%1], %2, %3, p;\n\t}"
                 ::"r"(d), "r"(a), "l"(b), "r"(idesc), "r"(accumulate), "r"(elected) : "memory");
}

// ---- decode of one mask word (four k-blocks of the lane) into A-operand registers -------------------
// As in process_tile; r[ca][4 * i ..] = {row g: columns 0..3, 4..7; row g + 8: the same} of k-block i in column area ca.
template <int CA, bool W2>
__device__ __forceinline__ void decode_word(uint32_t mw, uint32_t pay_a, uint32_t lut_a, uint32_t lut_stride, uint32_t& b8,
                                            uint32_t (&cw0)[W2 ? 1 : CA], uint32_t (&cw1)[W2 ? 1 : CA], uint32_t (&r)[CA][16])
{
    constexpr int SR = W2 ? 1 : CA;
    constexpr int kRow = 128 * SR;
    uint32_t pos[5], wm1[SR][4], w0[SR][4], w1[SR][4], e[4];
    pos[0] = b8;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const uint32_t cum = (i == 3) ? mw : (mw & ((1u << (8 * i + 8)) - 1u));
        pos[i + 1] = b8 + 8u * (uint32_t)__popc(cum);
        e[i] = lut_a + prmt(mw, 0u, 0x4440u + i) * lut_stride;
    }
    b8 = pos[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const uint32_t a = pay_a + (pos[i + 1] >> 5) * (uint32_t)kRow;
        wm1[0][i] = lds32_at<-kRow>(a);
        w0[0][i] = lds32_at<0>(a);
        w1[0][i] = lds32_at<kRow>(a);
        if (SR == 2) {
            wm1[SR - 1][i] = lds32_at<128 - kRow>(a);
            w0[SR - 1][i] = lds32_at<128>(a);
            w1[SR - 1][i] = lds32_at<128 + kRow>(a);
        }
        e[i] = lds32(e[i]);
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
#pragma unroll
        for (int s = 0; s < SR; ++s) {
            const uint32_t s0 = (i == 0) ? cw0[s] : w0[s][i == 0 ? 0 : i - 1];
            const uint32_t s1 = (i == 0) ? cw1[s] : w1[s][i == 0 ? 0 : i - 1];
            const uint32_t lo = __funnelshift_r(s0, s1, pos[i]);
            const uint32_t hi = __funnelshift_r(wm1[s][i], w0[s][i], pos[i + 1]);
            const uint32_t g0 = prmt(lo, W2 ? kFillW2 : kFill, e[i]);
            const uint32_t g1 = prmt(hi, W2 ? kFillW2 : kFill, e[i] >> 16);
            if (W2) {
#pragma unroll
                for (int ca = 0; ca < CA; ++ca) {
                    const uint32_t d0 = (ca ? g0 >> 4 : g0) & 0x0F0F0F0Fu, d1 = (ca ? g1 >> 4 : g1) & 0x0F0F0F0Fu;
                    r[ca][4 * i] = d0; r[ca][4 * i + 1] = d1;
                    r[ca][4 * i + 2] = d0 & 0x03030303u; r[ca][4 * i + 3] = d1 & 0x03030303u;
                }
            } else {
                r[s][4 * i] = g0; r[s][4 * i + 1] = g1;
                r[s][4 * i + 2] = g0 & 0x0F0F0F0Fu; r[s][4 * i + 3] = g1 & 0x0F0F0F0Fu;
            }
        }
    }
#pragma unroll
    for (int s = 0; s < SR; ++s) { cw0[s] = w0[s][3]; cw1[s] = w1[s][3]; }
}

// 32 packed activations of token n from column k (a multiple of 32) on; columns from K on are zero. Where K is not a
// multiple of 32 rows start at any byte: two aligned 16-byte loads hold the unit (in flight from here on: volatile, not
// sunk to their use), and unit_x shifts it into place. The end of a row, or of X, is fetched byte by byte out of line.
struct UnitX {
    uint4 lo, hi;
};
inline __device__ __noinline__ uint4 load_x_tail(const uint8_t* src, int left)
{
    uint32_t o[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        o[i] = 0;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int c = left - 8 * i - 2 * j;   // columns left at this byte
            if (c > 0) o[i] |= (src[4 * i + j] & (c > 1 ? 255u : 15u)) << (8 * j);
        }
    }
    return make_uint4(o[0], o[1], o[2], o[3]);
}
__device__ __forceinline__ uint4 ld_now(const uint8_t* a)
{
    uint4 v;
    asm volatile("ld.global.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(a));
    return v;
}
template <bool ANY>
__device__ __forceinline__ UnitX load_x32(const TcParams& p, int64_t ldx, int n, int k)
{
    UnitX u;
    u.lo = u.hi = make_uint4(0, 0, 0, 0);
    if (n >= p.N || k >= p.K) return u;
    const int64_t b = (int64_t)n * ldx + (k >> 1);
    if (!ANY) {
        u.lo = ld_now(p.X + b);
    } else if (p.K - k >= 32 && (b & ~(int64_t)15) + 32 <= (int64_t)p.N * ldx) {
        u.lo = ld_now(p.X + (b & ~(int64_t)15));
        u.hi = ld_now(p.X + (b & ~(int64_t)15) + 16);
    } else {
        u.lo = load_x_tail(p.X + b, p.K - k);
    }
    return u;
}
template <bool ANY>
__device__ __forceinline__ uint4 unit_x(const TcParams& p, int64_t ldx, int n, int k, const UnitX& u)
{
    if (!ANY) return u.lo;
    const int64_t b = (int64_t)n * ldx + (k >> 1);
    if (p.K - k < 32 || (b & ~(int64_t)15) + 32 > (int64_t)p.N * ldx) return u.lo;
    uint32_t w[7] = {u.lo.x, u.lo.y, u.lo.z, u.lo.w, u.hi.x, u.hi.y, u.hi.z};
    if (b & 8) { w[0] = w[2]; w[1] = w[3]; w[2] = w[4]; w[3] = w[5]; w[4] = w[6]; w[5] = u.hi.w; }
    if (b & 4) { w[0] = w[1]; w[1] = w[2]; w[2] = w[3]; w[3] = w[4]; w[4] = w[5]; }
    const uint32_t sh = 8u * (uint32_t)(b & 3);
    return make_uint4(__funnelshift_r(w[0], w[1], sh), __funnelshift_r(w[1], w[2], sh), __funnelshift_r(w[2], w[3], sh),
                      __funnelshift_r(w[3], w[4], sh));
}

// Stores the 16 x 8 results of one 8-token block (store_rows). Out of line, like everything that runs once or twice per
// CTA: such code is fetched line by line from L2 while the weight stream keeps that busy, and a line costs hundreds of
// cycles then.
template <bool AM>
__device__ __noinline__ void store_block_tc(const StoreCtx& p, int v0, int v1, int v2, int v3, int lane, int m_lo, int m_hi, int n_base)
{
    const int v[1][4] = {{v0, v1, v2, v3}};
    store_rows<1, AM>(p, v, lane, m_lo, m_hi, nullptr, -2, n_base);
}

// A strip is complete: take its sums from the workspace, two 8-token blocks ahead, leave that zeroed, store. The weight scales are
// fetched once and the activation scales come from shared memory. (Not unrolled further: this code is cold, its lines come from
// L2 one by one, and where strips complete in the middle of the weight stream that costs more than it saves.)
template <bool AM>
__device__ __noinline__ void finish_strip_tc(const StoreCtx p, const float* xsc_s, int32_t* accp, int ng, int lane, int m_lo, int m_hi)
{
    float sw_lo = 0.f, sw_hi = 0.f;
    if (p.fp16_out) {
        if (m_lo >= 0) sw_lo = __half2float(__ushort_as_half(__ldg(p.w_scale + m_lo)));
        if (m_hi >= 0) sw_hi = __half2float(__ushort_as_half(__ldg(p.w_scale + m_hi)));
    }
    int v[3][4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        v[0][j] = __ldcg(accp + j * 32);
        v[1][j] = ng > 1 ? __ldcg(accp + 128 + j * 32) : 0;
    }
    int n = 2 * (lane & 3);
#pragma unroll 1
    for (int nt = 0; nt < ng; ++nt, n += 8) {
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            v[2][j] = nt + 2 < ng ? __ldcg(accp + 256 + j * 32) : 0;
            __stcg(accp + j * 32, 0);
        }
        accp += 128;
        const float2 sx = *reinterpret_cast<const float2*>(xsc_s + n);
        uint32_t big[2] = {0u, 0u};
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int m = j < 2 ? m_lo : m_hi;
            if (n + (j & 1) < p.N && m >= 0) {
                const size_t o = (size_t)(n + (j & 1)) * p.M + m;
                if (p.fp16_out) {
                    const __half h = __float2half_rn((float)v[0][j] * (j < 2 ? sw_lo : sw_hi) * (j & 1 ? sx.y : sx.x));
                    reinterpret_cast<__half*>(p.Y)[o] = h;
                    if (AM && m >= p.amax_m0 && m < p.amax_m1) big[j & 1] = max(big[j & 1], (uint32_t)(__half_as_ushort(h) & 0x7FFFu));
                } else {
                    reinterpret_cast<int32_t*>(p.Y)[o] = v[0][j];
                }
            }
        }
        if (AM) {   // the eight lanes that hold a token combine
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                uint32_t m = big[k];
                m = max(m, __shfl_xor_sync(0xffffffffu, m, 4));
                m = max(m, __shfl_xor_sync(0xffffffffu, m, 8));
                m = max(m, __shfl_xor_sync(0xffffffffu, m, 16));
                if (lane < 4 && m) atomicMax(p.amax_s + n + k, m);
            }
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) { v[0][j] = v[1][j]; v[1][j] = v[2][j]; }
    }
}

// ANY: K is not a multiple of 32 (load_x32).
// OCT = 3: 24 decode warps, 384 rows to a stage, for N <= 16. With 16 decode warps 0.59 instructions issue per cycle and
// scheduler; eight more warps hide more of the decode's latency (28672 x 8192, N = 16: 29.3 -> 28.0 us, with INT2 weights
// 25.7 -> 24.7). Their A operands leave an octet two stages and the CTA three X warps: at N = 32 33.4 us against 33.1.
template <int OCT, int CA, bool W2, bool AM, bool ANY>
__global__ void __launch_bounds__(TcShape<OCT>::kThreads, 1) us_spmm_tc_kernel(const __grid_constant__ TcParams p)
{
    extern __shared__ __align__(1024) uint8_t smem[];
    using S = TcShape<OCT>;
    constexpr int kTcDecodeWarps = S::kDecode, kTcXWarps = S::kX, kTcAStages = S::kA;
    constexpr uint32_t kDW = (uint32_t)S::kDecode;
    // (the warp number through a shuffle: the compiler then knows it to be the same in all lanes)
    const int lane = threadIdx.x & 31, warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0);
    const int ng = (p.N + 7) >> 3;                       // 8-token groups
    const uint32_t x_stage_bytes = (uint32_t)ng * 2048u;

    // ---- shared memory (mirrored by build_tc_plan on the host) ---------------------------------------
    uint32_t* lut = reinterpret_cast<uint32_t*>(smem);                              // [256][lut_rep]
    uint8_t* xs = reinterpret_cast<uint8_t*>(lut + 256 * p.lut_rep);                // [x_stages][ng][16][8][16]
    // (an odd number of token groups: the MMA's last block reads on into the next stage, or these 2 KB; those sums are never used)
    float* xsc_s = reinterpret_cast<float*>(xs + (size_t)p.x_stages * x_stage_bytes);           // [64] activation scales, in those 2 KB
    int32_t* sx = reinterpret_cast<int32_t*>(xs + (size_t)p.x_stages * x_stage_bytes + 2048);   // [kTcSxRing][64]
    uint64_t* bars = reinterpret_cast<uint64_t*>(sx + kTcSxRing * 64);
    uint32_t* misc = reinterpret_cast<uint32_t*>(bars + kTcBars);   // [0] tensor memory, [1] dead, [2] finished warps, [32..95] absmax
    uint32_t* issued = misc + 96;                                   // phases started per slot
    uint8_t* ring = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(issued + kTcMaxSlots) + 127) & ~uintptr_t(127));
    const uint32_t bar0 = smem_u32(bars);
    const uint32_t b_w = bar0, b_af = bar0 + 8 * kTcMaxSlots, b_ae = b_af + 8 * OCT * kTcAStages,
                   b_xf = b_ae + 8 * OCT * kTcAStages, b_xe = b_xf + 8 * kTcMaxXStages, b_d = b_xe + 8 * kTcMaxXStages,
                   b_drain = b_d + 8 * OCT;
    volatile uint32_t* dead = misc + 1;

    const uint32_t beg = p.cta_begin[blockIdx.x], end = p.cta_begin[blockIdx.x + 1];
    if (beg >= end) {
        asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
        if (AM && threadIdx.x < 64) {
            asm volatile("griddepcontrol.wait;" ::: "memory");
            p.y_amax[64 + 64 * blockIdx.x + threadIdx.x] = 0;
            if (blockIdx.x == 0 && threadIdx.x == 0) p.y_amax[0] = gridDim.x;
        }
        return;
    }
    // first stage of the range: row block q0 of 16 kDW rows, segment seg0, stage st0 of its tiles; then stage by stage
    const int n_stage = p.n_stage, total = (int)(end - beg);
    const int q0 = (int)fdiv(beg, p.mg_block), in_block = (int)beg - q0 * p.block_stages;
    const int seg0 = in_block / n_stage, st0 = in_block - seg0 * n_stage;
    const uint32_t tile0 = (uint32_t)(q0 * p.n_segs + seg0);                        // in (block, segment) order
    const uint32_t n_tile = (uint32_t)((st0 + total + n_stage - 1) / n_stage);      // tiles of a warp

    const uint64_t w_policy = l2_evict_first_policy();
    // Tile t of the CTA: warp t % kDW, that warp's t / kDW-th. Returns the tile index, kNull for a strip past the matrix
    // (its slot's phase is completed without a copy), kNone past the CTA's last tile.
    constexpr uint32_t kNone = 0xFFFFFFFFu, kNull = 0xFFFFFFFEu;
    auto tile_at = [&](uint32_t t) -> uint32_t {
        if (t / kDW >= n_tile) return kNone;
        const uint32_t u = tile0 + t / kDW, q = fdiv(u, p.mg_segs), seg = u - q * (uint32_t)p.n_segs;
        const uint32_t strip = kDW * q + t % kDW;
        return strip < (uint32_t)p.n_strips ? strip * (uint32_t)p.n_segs + seg : kNull;
    };
    auto copy_tile = [&](uint32_t tile, uint32_t o0, uint32_t o1, uint32_t slot) {   // one lane
        const uint32_t bytes = (o1 - o0) * 16u, bar = b_w + 8u * slot;
        if (tile == p.withhold) return;
        *(volatile uint32_t*)(issued + slot) = issued[slot] + 1u;
        if (tile == kNull) { mbar_arrive(bar); return; }
        mbar_expect_tx(bar, bytes);
        bulk_g2s(smem_u32(ring + (size_t)slot * p.slot_bytes), p.blob + (size_t)o0 * 16u, bytes, bar, w_policy);
    };

    // ---- prologue: first copies, barriers, tensor memory, selector table --------------------------------
    // lane j of a decode warp: the first copy into the warp's j-th slot. Only the warps' first tiles are requested at
    // once (they would otherwise arrive no sooner than everything the ring holds), the rest when those have arrived.
    const uint32_t t_first = (uint32_t)warp + kDW * (uint32_t)lane;
    uint32_t tile_first = kNone, of0 = 0, of1 = 0;
    if (warp < kTcDecodeWarps) {
        if (t_first < (uint32_t)p.n_slots) {
            tile_first = tile_at(t_first);
            if (tile_first < kNull) { of0 = __ldg(p.item_off + tile_first); of1 = __ldg(p.item_off + tile_first + 1); }
            mbar_init(b_w + 8u * t_first, 1);
            issued[t_first] = 0;
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        if (tile_first != kNone && lane == 0) copy_tile(tile_first, of0, of1, t_first);
        // selector table: entry e by two threads, each writing half of its copies (conflict-free rotation)
        const int e = threadIdx.x & 255, part = threadIdx.x >> 8;
        if (part < 2) {
            const int n_half = p.lut_rep / 2;
            const uint32_t v = lut_entry(e);
            const int rot = p.lut_rep == 32 ? lane : lane >> 2;
#pragma unroll 1
            for (int i = 0; i < n_half; ++i) lut[e * p.lut_rep + ((rot + i + part * n_half) & (p.lut_rep - 1))] = v;
        }
    } else if (warp == kTcDecodeWarps) {
        if (lane < OCT * kTcAStages) { mbar_init(b_af + 8u * lane, 8); mbar_init(b_ae + 8u * lane, 1); }
        if (lane < kTcMaxXStages) { mbar_init(b_xf + 8u * lane, S::kPair); mbar_init(b_xe + 8u * lane, 1); }
        if (lane <= OCT) mbar_init(b_d + 8u * lane, 1);   // (and b_drain)
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        if (lane == 0) { misc[1] = 0; misc[2] = 0; }
        __syncwarp();
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(misc)) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
        // Only now: a dependent's CTA that fits beside this one takes tensor memory of its own, and then waits for this kernel.
        asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    } else {
        const int x = threadIdx.x - 32 * (kTcDecodeWarps + 1);
        for (int i = x; i < kTcSxRing * 64; i += 32 * kTcXWarps) sx[i] = 0;
        if (AM && x < 64) misc[32 + x] = 0;
    }
    // The X warps need the barriers only, not the decode warps' table and offsets (about 2000 cycles later).
    tc_fence_before();
    if (warp >= kTcDecodeWarps) asm volatile("bar.sync 1, %0;" ::"n"(32 * (1 + kTcXWarps)) : "memory");
    if (warp <= kTcDecodeWarps) asm volatile("bar.sync 2, %0;" ::"n"(32 * (1 + kTcDecodeWarps)) : "memory");
    tc_fence_after();
    const uint32_t tm = *(volatile uint32_t*)misc;
    const uint32_t n16 = (uint32_t)(p.N + 15) / 16u;        // 16-token blocks
    // tensor-memory columns: the A stages of the octets, then their sums
    const uint32_t tm_d = tm + OCT * kTcAStages * 64u;      // + o * S::kD

    bool ok = true;
    if (warp < kTcDecodeWarps) {
        // ================= decode warps =================
        const int o = warp >> 3;
        const uint32_t lane_base = (uint32_t)(32 * (warp & 3) + 16 * ((warp >> 2) & 1)) << 16;
        const uint32_t tm_a = tm + (uint32_t)o * kTcAStages * 64u + lane_base;
        const uint32_t lut_a = smem_u32(lut) + 4u * (uint32_t)(lane & (p.lut_rep - 1)), lut_stride = 4u * (uint32_t)p.lut_rep;
        const StoreCtx sctx{p.Y, p.w_scale, p.x_scale, p.acc, p.cnt, p.M, p.N, p.fp16_out, AM ? misc + 32 : nullptr, p.amax_m0, p.amax_m1};
        uint32_t as = 0, a_par = 1;           // A stage in turn, parity of its "empty" wait
        uint32_t d_par = 0;
        uint32_t slot = (uint32_t)warp, pass = 0;   // ring slot of this warp's next tile, its pass of the ring
        bool waited = false;                  // griddepcontrol.wait executed
        int left = total, q = q0, seg = seg0, st = st0, run_stages = 0;
        auto announce = [&](uint32_t bar) {   // the warp's part of an A stage is in tensor memory
            tc_wait_st();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar);
        };
        constexpr int SR = W2 ? 1 : CA;
        constexpr int WPS = CA == 1 ? 2 : 1;  // mask words per stage

        // The warp's i-th tile is in its slot: another warp may not even have had its own tile there yet, and the barrier's
        // parity alone could not tell, so wait for the pass to begin, then for its copy. (From the second pass on that may take MMAs
        // in another warp's way, and those X.)
        auto wait_tile = [&](uint32_t i) {
            ok = tc_wait_count(issued + slot, pass + 1u, p.wait_ns_hi, dead, pass > 0) && tc_wait_warp(b_w + 8u * slot, pass & 1u, p.wait_ns_hi, dead);
            if (ok && i == 0 && lane > 0 && tile_first != kNone) copy_tile(tile_first, of0, of1, t_first);
            return ok;
        };
        // offsets of the tile that will take over that slot, fetched behind the decode
        uint32_t tile_next, no0 = 0, no1 = 0;
        auto look_ahead = [&](uint32_t i) {
            tile_next = tile_at(kDW * i + (uint32_t)warp + (uint32_t)p.n_slots);
            if (lane == 0 && tile_next < kNull) { no0 = __ldg(p.item_off + tile_next); no1 = __ldg(p.item_off + tile_next + 1); }
        };
        auto refill = [&]() {   // the slot is free: refill it for the tile that comes n_slots later, go to the next
            if (lane == 0 && tile_next != kNone) {
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                copy_tile(tile_next, no0, no1, slot);
            }
            slot += kDW;
            while (slot >= (uint32_t)p.n_slots) { slot -= (uint32_t)p.n_slots; ++pass; }
        };

        // The loop ends where the warp's strip lies past the matrix. (Two forms of one condition, because the compiler lays the
        // whole loop out differently for them. Second form against the first on 28672 x 8192, N = 16: INT2 weights 24.2 us
        // against 23.9, default format 28.3 against 28.7, folded 26.7 against 27.4.)
        const int q_end = (p.n_strips - warp + (int)kDW - 1) / (int)kDW;
        uint32_t i = 0;
        for (; left > 0; ++i) {
            const uint32_t strip = kDW * (uint32_t)q + (uint32_t)warp;
            if (W2 ? q >= q_end : strip >= (uint32_t)p.n_strips) break;
            look_ahead(i);
            const uint32_t slot_a = smem_u32(ring + (size_t)slot * p.slot_bytes) + 4u * lane;
            uint32_t b8 = 0, cw0[SR], cw1[SR], mw = 0;
            int words = p.mask_rows - WPS * st;       // mask words of the tile from here on
            if (!wait_tile(i)) break;
            const uint32_t pay_a = slot_a + 128u * p.mask_rows;
            uint32_t mask_a = slot_a;
#pragma unroll 1
            for (int w = WPS * st; w > 0; --w) {  // entered in its middle: the stream position there
                b8 += 8u * (uint32_t)__popc(lds32(mask_a));
                mask_a += 128u;
            }
            mw = lds32(mask_a);
            const uint32_t a0 = pay_a + (b8 >> 5) * (uint32_t)(128 * SR);
#pragma unroll
            for (int s = 0; s < SR; ++s) { cw0[s] = lds32(a0 + 128u * s); cw1[s] = lds32(a0 + 128u * (SR + s)); }
            const int n_here = min(n_stage - st, left);
            for (int j = 0; j < n_here; ++j) {
                ok = tc_wait_warp(b_ae + 8u * (o * kTcAStages + as), a_par, p.wait_ns_hi, dead, true);
                if (!ok) break;
                tc_fence_after();
                const uint32_t dst = tm_a + 64u * as;
#pragma unroll
                for (int h = 0; h < WPS; ++h) {
                    if (h == 1 && words <= 0) break;   // (an odd number of mask words: the last stage is half a stage)
                    const uint32_t m = mw;
                    mask_a += 128u;
                    if (--words > 0) mw = lds32(mask_a);
                    uint32_t r[CA][16];
                    decode_word<CA, W2>(m, pay_a, lut_a, lut_stride, b8, cw0, cw1, r);
                    tc_st16(dst + 32u * h, r[0]);
                    if (CA == 2) tc_st16(dst + 32u, r[CA - 1]);
                }
                announce(b_af + 8u * (o * kTcAStages + as));
                if (++as == kTcAStages) { as = 0; a_par ^= 1u; }
            }
            if (!ok) break;
            refill();
            left -= n_here;
            run_stages += n_here;
            st = 0;
            if (++seg < p.n_segs && left > 0) continue;

            // ---- the run of this row block ends: read the sums back ----
            const int m_lo = __ldg(p.row_order + strip * 16 + (lane >> 2)), m_hi = __ldg(p.row_order + strip * 16 + (lane >> 2) + 8);
            ok = tc_wait_warp(b_d + 8u * o, d_par, p.wait_ns_hi, dead);
            if (!ok) break;
            d_par ^= 1u;
            if (!waited) {   // Y and the workspace may still be in use by the stream's earlier work
                asm volatile("griddepcontrol.wait;" ::: "memory");
                waited = true;
            }
            tc_fence_after();
            const int32_t* sxp = sx + ((q - q0) % kTcSxRing) * 64 + 2 * (lane & 3);
            const bool whole = run_stages == p.block_stages;
            int32_t* accp = p.acc + (size_t)strip * (p.acc_nt * 128) + lane;
#pragma unroll 1
            for (int nt = 0; nt < ng; ++nt) {
                int c[4], y[4];
                tc_ld4(tm_d + (uint32_t)(S::kD * o) + 8u * nt + lane_base, c);
                const int s0 = sxp[8 * nt] >> 4, s1 = sxp[8 * nt + 1] >> 4;
                if (W2) {
                    y[0] = (c[2] >> 4) - 2 * s0;
                    y[1] = (c[3] >> 4) - 2 * s1;
                    y[2] = ((c[0] - c[2]) >> 6) - 2 * s0;
                    y[3] = ((c[1] - c[3]) >> 6) - 2 * s1;
                } else {
                    y[0] = (c[2] >> 4) - 8 * s0;
                    y[1] = (c[3] >> 4) - 8 * s1;
                    y[2] = (c[0] - c[2]) >> 8;
                    y[3] = (c[1] - c[3]) >> 8;
                }
                if (whole) {
                    store_block_tc<AM>(sctx, y[0], y[1], y[2], y[3], lane, m_lo, m_hi, 8 * nt);
                } else {
#pragma unroll
                    for (int j = 0; j < 4; ++j) atomicAdd(accp + nt * 128 + j * 32, y[j]);
                }
            }
            tc_fence_before();
            if (!whole) {
                __syncwarp();
                uint32_t old = 0;
                if (lane == 0)
                    asm volatile("atom.acq_rel.gpu.global.add.u32 %0, [%1], %2;" : "=r"(old) : "l"(p.cnt + strip), "r"(run_stages) : "memory");
                old = __shfl_sync(0xffffffffu, old, 0);
                if (old + (uint32_t)run_stages == (uint32_t)p.block_stages) {
                    __syncwarp();
                    finish_strip_tc<AM>(sctx, xsc_s, accp, ng, lane, m_lo, m_hi);
                    if (lane == 0) p.cnt[strip] = 0;
                }
            }
            run_stages = 0;
            seg = 0;
            ++q;
        }
        // In the last row block a warp's strip may lie past the matrix. Such a warp announces its part of every stage as it
        // is, and passes its ring slots on: not before they are filled, the warp before it may still be decoding from them.
#pragma unroll 1
        for (; ok && left > 0; ++i) {
            look_ahead(i);
            if (!wait_tile(i)) break;
            const int n_here = min(n_stage - st, left);
#pragma unroll 1
            for (int j = 0; j < n_here && ok; ++j) {
                ok = tc_wait_warp(b_ae + 8u * (o * kTcAStages + as), a_par, p.wait_ns_hi, dead, true);
                if (!ok) break;
                if (lane == 0) mbar_arrive(b_af + 8u * (o * kTcAStages + as));
                if (++as == kTcAStages) { as = 0; a_par ^= 1u; }
            }
            if (!ok) break;
            refill();
            left -= n_here;
            st = 0;
        }
        if (!waited) asm volatile("griddepcontrol.wait;" ::: "memory");
    } else if (warp == kTcDecodeWarps) {
        // ================= MMA issue =================
        // The whole warp walks the loop; one elected lane issues.
        const uint32_t leader = tc_elect();
        // D = INT32, A and B = signed 8 bit, both K-major, N = 16 n16, M = 128
        const uint32_t idesc = (2u << 4) | (1u << 7) | (1u << 10) | ((2u * n16) << 17) | (8u << 24);
        // B descriptor: no swizzle, 128 bytes between 16-byte k-columns, 2048 between 8-token groups
        const uint64_t bd0 = ((uint64_t)(128u >> 4) << 16) | ((uint64_t)(2048u >> 4) << 32) | (1ull << 46) | (uint64_t)(smem_u32(xs) >> 4);
        uint32_t as = 0, a_par = 0, xst = 0, x_par = 0, more = 0;   // more: the run has begun (accumulate)
        int left_block = p.block_stages - in_block, st = st0;
        const bool odd = CA == 1 && (p.mask_rows & 1);
        for (int s = 0; s < total && ok; ++s) {
            const bool half = odd && st == n_stage - 1;   // the tile's last stage holds one mask word only
            const bool last = --left_block == 0 || s == total - 1;   // end of the run of this row block
            ok = tc_wait_warp(b_xf + 8u * xst, x_par, p.wait_ns_hi, dead, true);
            const uint64_t b = bd0 + (uint64_t)((xst * x_stage_bytes) >> 4);
#pragma unroll
            for (int o = 0; o < OCT; ++o) {
                if (ok) ok = tc_wait_warp(b_af + 8u * (o * kTcAStages + as), a_par, p.wait_ns_hi, dead);
                if (!ok) break;
                tc_fence_after();
                const uint32_t a = tm + (uint32_t)o * kTcAStages * 64u + 64u * as, d = tm_d + (uint32_t)(S::kD * o);
#pragma unroll
                for (uint32_t j = 0; j < 4; ++j) tc_mma_i8(leader, d, a + 8u * j, b + 16u * j, idesc, j == 0 ? more : 1u);
                if (!half)
#pragma unroll
                    for (uint32_t j = 4; j < 8; ++j) tc_mma_i8(leader, d, a + 8u * j, b + 16u * j, idesc, 1u);
                tc_commit(leader, b_ae + 8u * (o * kTcAStages + as));
                if (last) tc_commit(leader, b_d + 8u * o);
            }
            tc_commit(leader, b_xe + 8u * xst);
            more = last ? 0u : 1u;
            if (left_block == 0) left_block = p.block_stages;
            if (++st == n_stage) st = 0;
            if (++as == kTcAStages) { as = 0; a_par ^= 1u; }
            if (++xst == (uint32_t)p.x_stages) { xst = 0; x_par ^= 1u; }
        }
        if (!ok) *dead = 1;
        tc_commit(leader, b_drain);   // nothing is in flight when the tensor memory is given back
        mbar_wait_bounded(b_drain, 0, p.wait_ns_hi);
        __syncwarp();
    } else {
        // ================= X warps =================
        // Whole stages in turn, so that the loads of several stages are in flight at once; with two octets two warps share a stage
        // (even and odd token groups). (No more stages at once than the ring has: a warp one pass of the ring ahead could not tell the
        // barrier's phases apart.)
        constexpr int P = S::kPair;
        const int xw = warp - kTcDecodeWarps - 1, c0 = xw / P, W = min(kTcXWarps / P, p.x_stages), g0 = xw % P;
        const int64_t ldx = ((int64_t)p.K + 1) / 2;
        const int r = lane & 7, qq = lane >> 3;
        int xst = c0, q = q0, seg = seg0, st = st0 + c0;
        uint32_t x_par = 1;
        const int k_second = CA == 1 ? 128 : p.K_L / 2;
        asm volatile("griddepcontrol.wait;" ::: "memory");
        // (by the warps of the first stage: its barriers hand the scales on to the decode warps, as they do the sums)
        if (p.fp16_out && c0 == 0)
            for (int i = lane + 32 * g0; i < p.N; i += 32 * P) xsc_s[i] = __half2float(__ushort_as_half(p.x_scale[i]));
        if (c0 < W)
        for (int c = c0; c < total; c += W) {
            while (st >= n_stage) {
                st -= n_stage;
                if (++seg == p.n_segs) { seg = 0; ++q; }
            }
            // columns of this lane's two 32-column units: CA = 1 consecutive; CA = 2 half of the stage from each column area
            const int k0 = seg * p.K_L + (CA == 1 ? 256 : 128) * st + 32 * qq;
            const int k1 = CA == 1 && 2 * st + 1 >= p.mask_rows ? p.K : k0 + k_second;
            // (the lane's 32 columns are lane t = qq of a fragment: 8 of them in each of the unit's four k-blocks)
            uint8_t* dst0 = xs + (size_t)xst * x_stage_bytes + g0 * 2048 + (qq >> 1) * 128 + r * 16 + (qq & 1) * 8;
            int32_t* sxr = sx + ((q - q0) % kTcSxRing) * 64;
            UnitX v0 = load_x32<ANY>(p, ldx, 8 * g0 + r, k0), v1 = load_x32<ANY>(p, ldx, 8 * g0 + r, k1);
            UnitX n0, n1;   // a group ahead
            if (!ANY) { n0 = load_x32<ANY>(p, ldx, 8 * (g0 + P) + r, k0); n1 = load_x32<ANY>(p, ldx, 8 * (g0 + P) + r, k1); }
            ok = tc_wait_warp(b_xe + 8u * xst, x_par, p.wait_ns_hi, dead);
            if (!ok) break;
#pragma unroll 1
            for (int g = g0; g < ng; g += P) {
                // the group after next, or (any K: twice the registers) the next
                constexpr int kAhead = ANY ? 1 : 2;
                UnitX f0, f1;
                f0.lo = f0.hi = f1.lo = f1.hi = make_uint4(0, 0, 0, 0);
                if (g + kAhead * P < ng) {
                    f0 = load_x32<ANY>(p, ldx, (g + kAhead * P) * 8 + r, k0);
                    f1 = load_x32<ANY>(p, ldx, (g + kAhead * P) * 8 + r, k1);
                }
                int s = 0;
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const uint4 v = unit_x<ANY>(p, ldx, 8 * g + r, h ? k1 : k0, h ? v1 : v0);
                    uint8_t* dst = dst0 + h * 1024;
                    *reinterpret_cast<uint2*>(dst) = expand8(v.x, s);
                    *reinterpret_cast<uint2*>(dst + 256) = expand8(v.y, s);
                    *reinterpret_cast<uint2*>(dst + 512) = expand8(v.z, s);
                    *reinterpret_cast<uint2*>(dst + 768) = expand8(v.w, s);
                }
                dst0 += 2048 * P;
                s += __shfl_xor_sync(0xffffffffu, s, 8);
                s += __shfl_xor_sync(0xffffffffu, s, 16);
                if (lane < 8) atomicAdd(sxr + g * 8 + lane, s);
                if (ANY) { v0 = f0; v1 = f1; }
                else { v0 = n0; v1 = n1; n0 = f0; n1 = f1; }
            }
            // the row block's last stage: clear the sums of the block eight further on (those of the block eight back, which
            // shared their place, were read long ago)
            if (g0 == 0 && seg == p.n_segs - 1 && st == n_stage - 1) {
                int32_t* z = sx + ((q - q0 + kTcSxRing / 2) % kTcSxRing) * 64;
                z[lane] = 0; z[lane + 32] = 0;
            }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            __syncwarp();
            if (lane == 0) mbar_arrive(b_xf + 8u * xst);
            st += W;
            xst += W;
            if (xst >= p.x_stages) { xst -= p.x_stages; x_par ^= 1u; }
        }
    }
    if (!ok && lane == 0) {
        *dead = 1;
        atomicExch(p.err, kErrTimeout);
    }
    // Chained call: the last decode warp to finish publishes the CTA's per-token absmax.
    if (AM && warp < kTcDecodeWarps) {
        __syncwarp();
        uint32_t old = 0;
        if (lane == 0)
            asm volatile("atom.acq_rel.cta.shared.add.u32 %0, [%1], 1;" : "=r"(old) : "r"(smem_u32(misc + 2)) : "memory");
        old = __shfl_sync(0xffffffffu, old, 0);
        if (old == (uint32_t)kTcDecodeWarps - 1u) {
            for (int n = lane; n < 64; n += 32) p.y_amax[64 + 64 * blockIdx.x + n] = *(volatile uint32_t*)(misc + 32 + n);
            if (blockIdx.x == 0 && lane == 0) p.y_amax[0] = gridDim.x;
        }
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == kTcDecodeWarps) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tm));
    // After a wait ran out: the copies that were issued must land before the CTA exits.
    if (*dead && warp == 0 && lane == 0)
        for (int s = 0; s < p.n_slots; ++s)
            if (issued[s]) mbar_wait_bounded(b_w + 8u * s, (issued[s] - 1u) & 1u, p.wait_ns_hi);
}

}  // namespace us
