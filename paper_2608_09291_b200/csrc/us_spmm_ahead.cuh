// sm_100a SpMM kernel for calls that give an SM about a tile or two per warp: the weights are decoded ahead of the
// activations, while the stream's earlier work still runs, and wait in tensor memory.
//
// What bounds such a call is the chain between the end of the kernel before it and its own stores: staging X, decoding one
// tile per warp, adding up, storing (4096 x 4096, N = 8: 1.4, 1.2 and 0.5 us of a period of 4.5). Only X has to wait for
// the kernel before. A CTA takes at most half an SM (shared memory, registers and tensor memory), so that it is resident
// beside the CTA of the launch before; there it copies and decodes its first tiles and leaves the gathered payload bytes
// in tensor memory, 64 columns of the warp's 32 lanes for a tile of 1024 columns (registers would hold one tile only, and
// cost the warps that hide the decode's latency). When X may be read, what is left is a copy of X into shared memory, as
// it is, and the MMAs: per k-block two masks, the two halves of a word of X per 8 tokens and the MMA.
//
//   decode    W warps; tile j of the CTA belongs to warp j % W. The first tiles are parked ahead, later ones when their turn
//             comes, in the place of the warp's first. Tile j is copied to slot j % n_slots; every tile has a barrier of its
//             own, used once, and one that says that it is decoded.
//   helpers   the last T - W warps. All: row numbers and scales of the CTA's strips. The first: tensor memory, X (one bulk copy per
//             token; ragged rows are shifted into place by everyone) and its scales. The others: copies into slots that
//             come free (a copy takes the warp that issues it some 500 cycles: 20480 x 5120, N = 16 20.5 us with one of them, 18.5 with three).
//
// 4096 x 4096, N = 8: 4.75 us a call with us_spmm_kernel's half-SM plan, 3.8 so (7.4 MB: 1.95 TB/s); 13824 x 5120, N = 8: 11.2, 10.0; what is left
// of the former is the end of one kernel up to the end of the next one's wait (2), X (0.7), MMAs and stores (1).
//
// A CTA sums its part of each strip in shared memory. With one K range the cuts fall on strip boundaries: it stores its strips,
// and nothing goes through the split-K workspace. Where X does not leave room (N = 16 from K = 6000 or so), K is cut in ranges as
// in us_spmm_kernel, every CTA works on one of them, and the sums meet in the workspace.
#pragma once
#include "us_spmm_tc.cuh"

namespace us {

constexpr int kAheadMaxTiles = 64;    // tiles a CTA may have
constexpr int kAheadCols = 256;       // tensor-memory columns a CTA may have (two share an SM)

struct AheadParams {
    const uint8_t* blob;
    const uint32_t* item_off;
    const int32_t* row_order;
    const uint16_t* w_scale;
    const uint8_t* X;
    const uint16_t* x_scale;
    void* Y;
    int32_t* acc;                   // split-K workspace, zero between calls (several K ranges)
    uint32_t* cnt;
    uint32_t* err;
    int32_t M, K, N;
    int32_t n_strips, n_segs;
    int32_t n_ranges, G;            // K ranges, segments of each (the last may have fewer)
    unsigned long long mg_g, mg_last, mg_range;   // floor(2^40 / d) + 1 for d = G, the last range's segments, n_strips * G
    int32_t mask_rows, K_L;
    uint32_t slot_bytes;
    int32_t n_slots;
    int32_t x_over;                 // X takes the place of the slots once every tile is parked
    int32_t s_local;                // most strips of a CTA
    int32_t parked;                 // tiles that wait in tensor memory
    int32_t tile_cols;              // tensor-memory columns of a parked tile
    int32_t tm_cols;                // allocated by a CTA
    int32_t fp16_out;
    uint32_t* y_amax;
    int32_t amax_m0, amax_m1;
    uint32_t wait_ns_hi;
    uint32_t withhold;
    uint32_t cta_begin[kMaxCtas + 1];   // in tiles
};

// Shared memory before X and the ring (mirrored by the kernel's carve-up; both start on 128 bytes), and that of X.
__host__ __device__ constexpr int ahead_fixed_smem(int nt, int s_local)
{
    return 256 * 8 * 4 + nt * 8 * 4 + (2 * kAheadMaxTiles + 2) * 8 + (96 + kAheadMaxTiles) * 4 + s_local * (nt * 128 + 32) * 4 + 128;
}
// A token's row of X. (any: room for the 16-byte units that hold a row of any first byte)
__host__ __device__ constexpr int ahead_x_row(int cols, bool any) { return x_row_bytes(cols, true) + (any && cols / 2 % 128 ? 128 : 0); }

__device__ __forceinline__ void tc_st8(uint32_t addr, const uint32_t (&r)[8])
{
    asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};"
                 ::"r"(addr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]) : "memory");
}
__device__ __forceinline__ void tc_ld8(uint32_t addr, uint32_t (&r)[8])
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]) : "r"(addr) : "memory");
}
// (the registers pass through the wait, so that nothing that reads them moves above it)
__device__ __forceinline__ void tc_wait_ld8(uint32_t (&r)[8])
{
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7])::"memory");
}

// Decodes a staged tile into tensor memory: per mask word and column area the gathered bytes of its four k-blocks, two
// registers each.
template <int CA, bool W2>
__device__ __forceinline__ void park_tile(uint32_t slot_a, uint32_t lut_a, int mask_rows, uint32_t tm_a)
{
    constexpr int SR = W2 ? 1 : CA;
    uint32_t mask_a = slot_a;
    const uint32_t pay_a = slot_a + 128u * mask_rows;
    uint32_t b8 = 0, cw0[SR], cw1[SR];
#pragma unroll
    for (int s = 0; s < SR; ++s) { cw0[s] = lds32(pay_a + 128u * s); cw1[s] = lds32(pay_a + 128u * (SR + s)); }
    uint32_t mw = lds32(mask_a);
#pragma unroll 1
    for (int w = mask_rows; w > 0; --w) {
        const uint32_t m = mw;
        mask_a += 128u;
        if (w > 1) mw = lds32(mask_a);
        uint32_t r[CA][16];
        decode_word<CA, W2>(m, pay_a, lut_a, 32u, b8, cw0, cw1, r);
#pragma unroll
        for (int ca = 0; ca < CA; ++ca) {
            const uint32_t d[8] = {r[ca][0], r[ca][1], r[ca][4], r[ca][5], r[ca][8], r[ca][9], r[ca][12], r[ca][13]};
            tc_st8(tm_a, d);
            tm_a += 8u;
        }
    }
}

// MMAs of a parked tile with packed activations (process_tile's second half), step by step: a mask word in a column area,
// 8 registers of gathered bytes and 4 of activations per token group, the next step's on their way.
template <int NT, int CA, bool W2>
struct Parked {
    static constexpr uint32_t kLow = W2 ? 0x03030303u : 0x0F0F0F0Fu;
    uint32_t d[2][8];
    uint32_t tm_a;
    int steps;

    __device__ __forceinline__ void load(uint32_t tm, int mask_rows)   // the first step
    {
        tm_a = tm;
        steps = mask_rows * CA;
        tc_ld8(tm_a, d[0]);
    }
    __device__ __forceinline__ static void load_x(uint32_t xb_a, int xstride, uint32_t x_fold, int s, uint4 (&x)[NT])
    {
        const uint32_t xa = xb_a + 64u * (uint32_t)(CA == 2 ? s >> 1 : s) + (CA == 2 && (s & 1) ? x_fold : 0u);
#pragma unroll
        for (int nt = 0; nt < NT; ++nt) x[nt] = lds128(xa + nt * 8 * xstride);
    }
    __device__ __forceinline__ static void step(const uint32_t (&v)[8], const uint4 (&x)[NT], int (&c)[NT][4], int (&c2)[4], int (&sum)[NT])
    {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const uint32_t d0 = v[2 * i], d1 = v[2 * i + 1], e0 = d0 & kLow, e1 = d1 & kLow;
#pragma unroll
            for (int nt = 0; nt < NT; ++nt) {
                const uint2 b = expand8(i == 0 ? x[nt].x : i == 1 ? x[nt].y : i == 2 ? x[nt].z : x[nt].w, sum[nt]);
                // (one token group: two sums in turn, so that the MMAs do not all wait for one another)
                mma_s8(NT == 1 && (i & 1) ? c2 : c[nt], d0, e0, d1, e1, b.x, b.y);
            }
        }
    }
    __device__ __forceinline__ void run(uint32_t xb_a, int xstride, uint32_t x_fold, int (&c)[NT][4], int (&sum)[NT])
    {
        int c2[4] = {0, 0, 0, 0};
        uint4 x[2][NT];
        load_x(xb_a, xstride, x_fold, 0, x[0]);
#pragma unroll 1
        for (int s = 0; s < steps; s += 2) {
            tc_wait_ld8(d[0]);
            if (s + 1 < steps) {
                tc_ld8(tm_a + 8u * (s + 1), d[1]);
                load_x(xb_a, xstride, x_fold, s + 1, x[1]);
            }
            step(d[0], x[0], c, c2, sum);
            if (s + 1 >= steps) break;
            tc_wait_ld8(d[1]);
            if (s + 2 < steps) {
                tc_ld8(tm_a + 8u * (s + 2), d[0]);
                load_x(xb_a, xstride, x_fold, s + 2, x[0]);
            }
            step(d[1], x[1], c, c2, sum);
        }
        if (NT == 1)
#pragma unroll
            for (int j = 0; j < 4; ++j) c[0][j] += c2[j];
    }
};

// X to shared memory, one copy per token, and the activation scales: lane h's part. What can be computed before the
// stream's earlier work is done is (the copies are the head of the chain that bounds a call).
template <bool ANY>
struct AheadX {
    const uint8_t* from;
    const uint16_t* scale;
    const uint8_t* tail;   // ANY: a byte past the last 16-byte unit of X, lane h's if it is one of these columns
    uint8_t* tail_dst;
    uint32_t dst, bytes;

    // (of columns k0 .. k0 + cols, k0 a multiple of 128)
    __device__ __forceinline__ void prepare(const AheadParams& p, int k0, int cols, uint8_t* xs, int xstride, uint32_t b_x, int h)
    {
        bytes = 0;
        from = nullptr;
        scale = nullptr;
        tail = nullptr;
        tail_dst = xs;
        dst = 0;
        const int64_t ldx = ((int64_t)p.K + 1) / 2, whole = (int64_t)p.N * ldx & ~(int64_t)15;   // 16-byte units of X
        const int64_t row_bytes = min((int64_t)cols / 2, ldx - k0 / 2);
        if (h < p.N) {
            const int64_t begin = h * ldx + k0 / 2, end = begin + row_bytes;
            const int64_t b = ANY ? begin & ~(int64_t)15 : begin, e = ANY ? min((end + 15) & ~(int64_t)15, whole) : end;
            from = p.X + b;
            dst = smem_u32(xs + h * xstride);
            if (e > b) {
                bytes = (uint32_t)(e - b);
                mbar_expect_tx_only(b_x, bytes);
            }
        }
        if (p.fp16_out && h < p.N) scale = p.x_scale + h;
        if (ANY && whole + h < (int64_t)p.N * ldx) {   // (15 bytes at most)
            const int64_t at = whole + h;
            const int row = (int)((uint32_t)at / (uint32_t)ldx);   // (eight ranges at most, each of which fits shared memory: 32 bits hold it)
            const int64_t begin = row * ldx + k0 / 2;
            if (at >= begin && at < begin + row_bytes) {
                tail = p.X + at;
                tail_dst = xs + row * xstride + (at - (begin & ~(int64_t)15));
            }
        }
        // columns past K, which the copies do not write: they meet zero weights, and the sums count them
        if (!ANY && k0 + cols > p.K) {
            const int rest = (k0 + cols - p.K) / 32;   // 16-byte units
            for (int i = h; i < p.N * rest; i += 32)
                *reinterpret_cast<uint4*>(xs + (i / rest) * xstride + (p.K - k0) / 2 + 16 * (i % rest)) = make_uint4(0, 0, 0, 0);
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    __device__ __forceinline__ void fetch(float* xsc_s, uint32_t b_x, int h)
    {
        asm volatile("griddepcontrol.wait;" ::: "memory");
        if (bytes) bulk_g2s(dst, from, bytes, b_x);
        const unsigned short s = ld16_if(scale, scale != nullptr);
        const uint8_t last = ANY ? ld8_if(tail, tail != nullptr) : (uint8_t)0;
        if (scale) xsc_s[h] = __half2float(__ushort_as_half(s));
        if (ANY && tail) *tail_dst = last;
        __syncwarp();
        if (h == 0) mbar_arrive(b_x);
    }
};

// Ragged rows (K no multiple of 32) start at any byte: the copies bring the 16-byte units that hold a row, and a warp shifts a
// row down to where it belongs, 512 bytes at a time. (What lies past column K meets zero weights, and the sums count it.)
inline __device__ __noinline__ void ahead_shift_rows(uint8_t* xs, int xstride, int K, int N, int units, int warp, int warps, int lane)
{
    const int64_t ldx = ((int64_t)K + 1) / 2;
#pragma unroll 1
    for (int t = warp; t < N; t += warps) {
        const uint32_t by = (uint32_t)(t * ldx) & 15u, sh = 8u * (by & 3u);
        if (by == 0) continue;
        const uint32_t row = smem_u32(xs + t * xstride);
#pragma unroll 1
        for (int u0 = 0; u0 < units; u0 += 32) {
            const int u = u0 + lane;
            uint4 lo = make_uint4(0, 0, 0, 0), hi = lo;
            if (u < units) { lo = lds128(row + 16 * u); hi = lds128(row + 16 * u + 16); }
            uint32_t w[8] = {lo.x, lo.y, lo.z, lo.w, hi.x, hi.y, hi.z, hi.w};
            if (by & 8u) { w[0] = w[2]; w[1] = w[3]; w[2] = w[4]; w[3] = w[5]; w[4] = w[6]; w[5] = w[7]; }
            if (by & 4u) { w[0] = w[1]; w[1] = w[2]; w[2] = w[3]; w[3] = w[4]; w[4] = w[5]; }
            __syncwarp();   // (before the first unit of the next lane is overwritten)
            if (u < units)
                *reinterpret_cast<uint4*>(xs + t * xstride + 16 * u) =
                    make_uint4(__funnelshift_r(w[0], w[1], sh), __funnelshift_r(w[1], w[2], sh), __funnelshift_r(w[2], w[3], sh),
                               __funnelshift_r(w[3], w[4], sh));
            __syncwarp();
        }
    }
}

// ANY: K is not a multiple of 32. AM: chained call that leaves the absmax of its outputs.
template <int NT, int CA, bool W2, bool AM, bool ANY, int W, int T>
__global__ void __launch_bounds__(32 * T, 2) us_spmm_ahead_kernel(const __grid_constant__ AheadParams p)
{
    extern __shared__ __align__(1024) uint8_t smem[];
    constexpr int H = T - W;
    static_assert(W % 4 == 0 && H >= 2, "parked tile j is of quarter j % 4 of the tensor memory; two helpers for X and the scales");
    const int lane = threadIdx.x & 31, warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0);
    const int h = (int)threadIdx.x - 32 * W;   // helper thread, from 0 on
    const int xstride = ahead_x_row(p.G * p.K_L, ANY);

    // ---- shared memory (ahead_fixed_smem) ---------------------------------------------------------------
    uint32_t* lut = reinterpret_cast<uint32_t*>(smem);                            // [256][8]
    float* xsc_s = reinterpret_cast<float*>(lut + 256 * 8);                       // [NT * 8] activation scales
    uint64_t* bars = reinterpret_cast<uint64_t*>(xsc_s + NT * 8);                 // [kAheadMaxTiles] tiles; X; [kAheadMaxTiles] decoded
    uint32_t* misc = reinterpret_cast<uint32_t*>(bars + 2 * kAheadMaxTiles + 2);      // [0] tensor memory, [1] dead, [32..95] absmax
    uint32_t* issued = misc + 96;                                                 // [kAheadMaxTiles] copy issued
    int32_t* acc_l = reinterpret_cast<int32_t*>(issued + kAheadMaxTiles);         // [s_local][NT * 128]
    int32_t* rows_s = acc_l + p.s_local * NT * 128;                               // [s_local][16] output rows
    float* wsc_s = reinterpret_cast<float*>(rows_s + p.s_local * 16);             // [s_local][16] weight scales
    uint8_t* xs = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(wsc_s + p.s_local * 16) + 127) & ~uintptr_t(127));   // [NT * 8][xstride], packed
    uint8_t* ring = p.x_over ? xs : xs + NT * 8 * xstride;
    const uint32_t bar0 = smem_u32(bars), b_x = bar0 + 8u * kAheadMaxTiles, b_e = b_x + 16u;
    volatile uint32_t* dead = misc + 1;

    const uint32_t beg = p.cta_begin[blockIdx.x], n = p.cta_begin[blockIdx.x + 1] - beg;   // the CTA's tiles
    if (n == 0) {   // no work: a chained call still owes its part of the absmax buffer
        asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
        if (AM && threadIdx.x < 64) {
            asm volatile("griddepcontrol.wait;" ::: "memory");
            p.y_amax[64 + 64 * blockIdx.x + threadIdx.x] = 0;
            if (blockIdx.x == 0 && threadIdx.x == 0) p.y_amax[0] = gridDim.x;
        }
        return;
    }
    // The CTA's tile j is position q0 + j of its K range (kr: g segments), in (strip, segment) order.
    const int kr = p.n_ranges == 1 ? 0 : (int)fdiv(beg, p.mg_range);
    const bool last_range = kr == p.n_ranges - 1;
    const uint32_t g = last_range ? (uint32_t)(p.n_segs - kr * p.G) : (uint32_t)p.G;
    const unsigned long long mg = last_range ? p.mg_last : p.mg_g;
    const uint32_t q0 = beg - (uint32_t)kr * (uint32_t)p.n_strips * (uint32_t)p.G;
    const uint32_t rb_first = fdiv(q0, mg), n_strips = fdiv(q0 + n - 1, mg) - rb_first + 1;
    auto tile_index = [&](uint32_t j) -> uint32_t {
        if (p.n_ranges == 1) return beg + j;
        const uint32_t rb = fdiv(q0 + j, mg);
        return rb * (uint32_t)p.n_segs + (uint32_t)(kr * p.G) + (q0 + j - rb * g);
    };
    const uint64_t w_policy = l2_evict_first_policy();
    auto copy_tile = [&](uint32_t j, uint32_t o0, uint32_t o1) {   // one lane
        const uint32_t bytes = (o1 - o0) * 16u, bar = bar0 + 8u * j;
        if (beg + j == p.withhold) return;
        *(volatile uint32_t*)(issued + j) = 1u;
        mbar_expect_tx(bar, bytes);
        bulk_g2s(smem_u32(ring + (size_t)(j % (uint32_t)p.n_slots) * p.slot_bytes), p.blob + (size_t)o0 * 16u, bytes, bar, w_policy);
    };

    // ---- prologue: first copies, selector table, tensor memory -------------------------------------------
    if (warp < W) {
        const uint32_t j = (uint32_t)warp + (uint32_t)W * (uint32_t)lane;   // lane l: the warp's l-th tile
        if (j < n) {
            uint32_t o0 = 0, o1 = 0;
            if (j < (uint32_t)p.n_slots) {
                const uint32_t t = tile_index(j);
                o0 = __ldg(p.item_off + t); o1 = __ldg(p.item_off + t + 1);
            }
            mbar_init(bar0 + 8u * j, 1);
            mbar_init(b_e + 8u * j, 1);
            *(volatile uint32_t*)(issued + j) = 0u;
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            if (j < (uint32_t)p.n_slots) copy_tile(j, o0, o1);
        }
        if (threadIdx.x < 256) {   // 256 entries, one a thread, eight copies
            const uint32_t v = lut_entry(threadIdx.x);
            uint4* e = reinterpret_cast<uint4*>(lut + 8 * threadIdx.x);
            e[0] = make_uint4(v, v, v, v);
            e[1] = make_uint4(v, v, v, v);
        }
    } else {
        if (warp == W) {
            if (lane == 0) {
                mbar_init(b_x, 1);
                misc[1] = 0;
            }
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            __syncwarp();
            asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(misc)), "r"((uint32_t)p.tm_cols) : "memory");
            asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
            // Only now: a dependent's CTA on this SM takes its tensor memory after this one has its own, and may then wait for it.
            asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
        }
        for (int i = h; i < p.s_local * NT * 128; i += 32 * H) acc_l[i] = 0;
        if (AM && h < 64) misc[32 + h] = 0;
        for (int i = h; i < (int)n_strips * 16; i += 32 * H) {
            const int m = __ldg(p.row_order + rb_first * 16 + i);
            rows_s[i] = m;
            wsc_s[i] = p.fp16_out && m >= 0 ? __half2float(__ushort_as_half(__ldg(p.w_scale + m))) : 0.f;
        }
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tm = *(volatile uint32_t*)misc;

    bool ok = true;
    if (warp < W) {
        // ================= decode warps =================
        const uint32_t lut_a = smem_u32(lut) + 4u * (uint32_t)(lane & 7);
        // parked tile j: the lanes of its warp's quarter of the tensor memory, and the j / 4-th place there
        auto place = [&](uint32_t j) { return tm + (j >> 2) * (uint32_t)p.tile_cols + ((uint32_t)(32 * (warp & 3)) << 16); };
        auto slot_of = [&](uint32_t j) { return smem_u32(ring + (size_t)(j % (uint32_t)p.n_slots) * p.slot_bytes) + 4u * lane; };
        auto park = [&](uint32_t j, uint32_t at) {   // decodes tile j to a place in tensor memory
            if (!tc_wait_warp(bar0 + 8u * j, 0u, p.wait_ns_hi, dead)) return false;
            park_tile<CA, W2>(slot_of(j), lut_a, p.mask_rows, at);
            __syncwarp();
            if (lane == 0) mbar_arrive(b_e + 8u * j);   // the slot may be refilled
            return true;
        };
        const uint32_t parked_end = min(n, (uint32_t)p.parked);
        for (uint32_t j = (uint32_t)warp; j < parked_end; j += W) {
            ok = park(j, place(j));
            if (!ok) break;
        }
        tc_wait_st();

        // From here on the stream's earlier work must be done: X is read and Y written.
        if (p.x_over) asm volatile("bar.arrive 2, %0;" ::"n"(32 * (W + 1)) : "memory");   // the slots are X's now
        asm volatile("griddepcontrol.wait;" ::: "memory");
        Parked<NT, CA, W2> parked;
        if (ok && (uint32_t)warp < parked_end) parked.load(place(warp), p.mask_rows);
        if (ok) ok = tc_wait_warp(b_x, 0u, p.wait_ns_hi, dead);
        if (ANY) {
            if (ok) ahead_shift_rows(xs, xstride, p.K, p.N, (int)g * (p.K_L / 32), warp, W + 1, lane);
            asm volatile("bar.sync 3, %0;" ::"n"(32 * (W + 1)) : "memory");
        }
        const uint32_t x_fold = CA == 2 ? (uint32_t)p.K_L / 4u : 0u;   // bytes of packed X to the second column area
        const uint32_t xb0 = smem_u32(xs) + (uint32_t)((lane >> 2) * xstride + 16 * (lane & 3));
        for (uint32_t j = (uint32_t)warp; ok && j < n; j += W) {
            const uint32_t rb = fdiv(q0 + j, mg), ls = rb - rb_first, sgl = q0 + j - rb * g;
            int c[NT][4], sum[NT];
#pragma unroll
            for (int nt = 0; nt < NT; ++nt) c[nt][0] = c[nt][1] = c[nt][2] = c[nt][3] = sum[nt] = 0;
            const uint32_t xb_a = xb0 + sgl * (uint32_t)(p.K_L / 2);
            if (j >= parked_end) {   // (in the place of the warp's first tile, which is done with)
                ok = park(j, place(warp));
                if (!ok) break;
                tc_wait_st();
            }
            if (j >= W) parked.load(place(j < parked_end ? j : (uint32_t)warp), p.mask_rows);
            parked.run(xb_a, xstride, x_fold, c, sum);
            int y[NT][4];
#pragma unroll
            for (int nt = 0; nt < NT; ++nt) {
                // a row group's four lanes hold the parts of a token's sum; the accumulators are those of tokens 2t, 2t + 1
                int s = sum[nt];
                s += __shfl_xor_sync(0xffffffffu, s, 1);
                s += __shfl_xor_sync(0xffffffffu, s, 2);
                const int s0 = __shfl_sync(0xffffffffu, s, 8 * (lane & 3)) >> 4, s1 = __shfl_sync(0xffffffffu, s, 8 * (lane & 3) + 4) >> 4;
                if (W2) {
                    y[nt][0] = (c[nt][2] >> 4) - 2 * s0;
                    y[nt][1] = (c[nt][3] >> 4) - 2 * s1;
                    y[nt][2] = ((c[nt][0] - c[nt][2]) >> 6) - 2 * s0;
                    y[nt][3] = ((c[nt][1] - c[nt][3]) >> 6) - 2 * s1;
                } else {
                    y[nt][0] = (c[nt][2] >> 4) - 8 * s0;
                    y[nt][1] = (c[nt][3] >> 4) - 8 * s1;
                    y[nt][2] = (c[nt][0] - c[nt][2]) >> 8;
                    y[nt][3] = (c[nt][1] - c[nt][3]) >> 8;
                }
            }
            int32_t* al = acc_l + ls * (NT * 128) + lane;
#pragma unroll
            for (int nt = 0; nt < NT; ++nt)
#pragma unroll
                for (int i = 0; i < 4; ++i) atomicAdd(al + nt * 128 + i * 32, y[nt][i]);
        }
        if (!ok) {
            *dead = 1;
            asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");   // (the first step of a tile that is not multiplied)
        }
        // All decode warps together store the CTA's strips, 32 results of a strip and token group at a time. (With a counter per
        // strip, as where warps end at different times, its last warp stored all of it: 1024 x 1024, N = 8 2.37 us, like this 2.29.)
        asm volatile("bar.sync 1, %0;" ::"n"(32 * W) : "memory");
        // (a result: fragment value i of token group nt of the CTA's strip ls)
        auto store = [&](int ls, int nt, int i, int v) {
            const int tok = nt * 8 + 2 * (lane & 3) + (i & 1), at = 16 * ls + (lane >> 2) + 8 * (i >> 1), row = rows_s[at];
            uint32_t big = 0;
            if (tok < p.N && row >= 0) {
                const size_t o = (size_t)tok * p.M + row;
                if (p.fp16_out) {
                    const __half f = __float2half_rn((float)v * wsc_s[at] * xsc_s[tok]);
                    reinterpret_cast<__half*>(p.Y)[o] = f;
                    if (AM && row >= p.amax_m0 && row < p.amax_m1) big = __half_as_ushort(f) & 0x7FFFu;
                } else {
                    reinterpret_cast<int32_t*>(p.Y)[o] = v;
                }
            }
            if (AM) {   // the eight lanes that hold a token combine
                big = max(big, __shfl_xor_sync(0xffffffffu, big, 4));
                big = max(big, __shfl_xor_sync(0xffffffffu, big, 8));
                big = max(big, __shfl_xor_sync(0xffffffffu, big, 16));
                if (lane < 4 && big) atomicMax(misc + 32 + tok, big);
            }
        };
        const int n_part = *dead ? 0 : (int)n_strips * NT * 4;   // of 32 results each
        if (p.n_ranges == 1) {
            for (int k = warp; k < n_part; k += W) store((k >> 2) / NT, (k >> 2) % NT, k & 3, acc_l[k * 32 + lane]);
        } else {
            int32_t* acc = p.acc + (size_t)rb_first * (NT * 128) + lane;
            for (int k = warp; k < n_part; k += W) atomicAdd(acc + k * 32, acc_l[k * 32 + lane]);
            asm volatile("bar.sync 1, %0;" ::"n"(32 * W) : "memory");
            for (uint32_t ls = (uint32_t)warp; n_part && ls < n_strips; ls += W) {
                // announce the CTA's tiles of the strip; the arrival that completes it takes the sums and leaves the workspace zeroed
                const uint32_t a = max((rb_first + ls) * g, q0), b = min((rb_first + ls + 1) * g, q0 + n);
                uint32_t old = 0;
                if (lane == 0)
                    asm volatile("atom.acq_rel.gpu.global.add.u32 %0, [%1], %2;" : "=r"(old) : "l"(p.cnt + rb_first + ls), "r"(b - a) : "memory");
                old = __shfl_sync(0xffffffffu, old, 0);
                if (old + (b - a) != (uint32_t)p.n_segs) continue;
                __syncwarp();
                int32_t* al = acc + ls * (NT * 128);
                int v[NT][4];
#pragma unroll
                for (int nt = 0; nt < NT; ++nt)
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        v[nt][i] = __ldcg(al + nt * 128 + i * 32);
                        __stcg(al + nt * 128 + i * 32, 0);
                    }
                if (lane == 0) p.cnt[rb_first + ls] = 0;
#pragma unroll
                for (int nt = 0; nt < NT; ++nt)
#pragma unroll
                    for (int i = 0; i < 4; ++i) store((int)ls, nt, i, v[nt][i]);
            }
        }
    } else {
        // ================= helpers =================
        if (warp == W) {
            if (p.x_over) asm volatile("bar.sync 2, %0;" ::"n"(32 * (W + 1)) : "memory");
            AheadX<ANY> x;
            x.prepare(p, kr * p.G * p.K_L, (int)g * p.K_L, xs, xstride, b_x, lane);
            x.fetch(xsc_s, b_x, lane);
            if (ANY) {
                ok = tc_wait_warp(b_x, 0u, p.wait_ns_hi, dead);
                if (ok) ahead_shift_rows(xs, xstride, p.K, p.N, (int)g * (p.K_L / 32), warp, W + 1, lane);
                asm volatile("bar.sync 3, %0;" ::"n"(32 * (W + 1)) : "memory");
            }
        } else {
            // tiles into slots that come free: a copy costs the warp that issues it some 500 cycles
            for (uint32_t j = (uint32_t)(p.n_slots + warp - W - 1); j < n; j += H - 1) {
                uint32_t o0 = 0, o1 = 0;
                if (lane == 0) {
                    const uint32_t t = tile_index(j);
                    o0 = __ldg(p.item_off + t); o1 = __ldg(p.item_off + t + 1);
                }
                // (the slot of a tile that is not parked comes free behind the MMAs)
                ok = tc_wait_warp(b_e + 8u * (j - (uint32_t)p.n_slots), 0u, p.wait_ns_hi, dead, j >= (uint32_t)(p.n_slots + p.parked));
                if (!ok) break;
                if (lane == 0) {
                    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                    copy_tile(j, o0, o1);
                }
                __syncwarp();
            }
        }
    }
    if (!ok && lane == 0) {
        *dead = 1;
        atomicExch(p.err, kErrTimeout);
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == W) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tm), "r"((uint32_t)p.tm_cols));
    if (AM && threadIdx.x < 64) {   // chained call: the CTA's per-token absmax
        p.y_amax[64 + 64 * blockIdx.x + threadIdx.x] = threadIdx.x < NT * 8 ? misc[32 + threadIdx.x] : 0u;
        if (blockIdx.x == 0 && threadIdx.x == 0) p.y_amax[0] = gridDim.x;
    }
    // After a wait ran out: the copies that were issued must land before the CTA exits, those of X among them (the first
    // helper warp has issued them, whatever became of the others): the next CTA here has its own data in this memory.
    if (*dead && warp == 0 && lane == 0) {
        for (uint32_t j = 0; j < n; ++j)
            if (issued[j]) mbar_wait_bounded(bar0 + 8u * j, 0u, p.wait_ns_hi);
        mbar_wait_bounded(b_x, 0u, p.wait_ns_hi);
    }
}

}  // namespace us
