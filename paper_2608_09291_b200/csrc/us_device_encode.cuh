// Encoder kernels: the lane-stream layout of us_host.h built on the GPU from the weight as packed INT4 (two columns a
// byte, even column in the low nibble; W2: the same nibbles), rows of `ld` bytes, zero beyond K.
//
// One warp per tile; lane 4g + t reads what it will own: for every mask word w (four k-blocks) the 32 columns 128 w + 32 t ..
// of strip rows g and g + 8, one 16-byte load per row (and column area). Two passes over the 22 MB of an 11008 x 4096 matrix,
// sizes then bytes, about 20 us each; the host encoder needed 13 ms on 16 threads for the same, most of it byte by byte.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace us {

struct EncodeParams {
    const uint8_t* W;           // M rows of ld bytes
    const int32_t* row_order;
    int64_t ld;
    int32_t n_segs, n_items, K_L, mask_rows;
    int32_t fold, w2;           // two column areas; INT2 weights
    uint32_t* size16;           // per tile: size in units of 16 bytes
    uint32_t* item_off;         // n_items + 1
    unsigned long long* sum_P;
    uint8_t* blob;
};

// nibbles of v that are not zero -> one bit each, in slot order: nibbles 0, 2, 4, 6, then 1, 3, 5, 7
__device__ __forceinline__ uint32_t nonzero_nibbles(uint32_t v)
{
    uint32_t n = v | (v >> 1);
    n |= n >> 2;                 // bits 4 i
    // four bits 8 apart to bits 24 .. 27 by one multiplication (no two of its terms share a bit)
    const uint32_t even = ((n & 0x01010101u) * 0x01020408u) >> 24, odd = (((n >> 4) & 0x01010101u) * 0x01020408u) >> 24;
    return (even & 15u) | ((odd & 15u) << 4);
}

// The lane's weights of a mask word, a 32-bit word per k-block: v[area][row half][k-block].
struct EncodeLane {
    const uint8_t *a, *b;   // rows g and g + 8 at the tile's first column, nullptr = padding row
    int64_t second;         // bytes to the second column area
    bool fold;
    __device__ __forceinline__ EncodeLane(const EncodeParams& p, int item, int lane)
    {
        const int rb = item / p.n_segs, sg = item - rb * p.n_segs;
        const int ra = p.row_order[rb * 16 + (lane >> 2)], rw = p.row_order[rb * 16 + (lane >> 2) + 8];
        const int64_t col = (int64_t)sg * (p.K_L / 2) + 16 * (lane & 3);
        a = ra < 0 ? nullptr : p.W + (int64_t)ra * p.ld + col;
        b = rw < 0 ? nullptr : p.W + (int64_t)rw * p.ld + col;
        second = p.K_L / 4;
        fold = p.fold != 0;
    }
    __device__ __forceinline__ static void load16(const uint8_t* s, uint32_t (&v)[4])
    {
        const uint4 q = s ? __ldg(reinterpret_cast<const uint4*>(s)) : make_uint4(0, 0, 0, 0);
        v[0] = q.x; v[1] = q.y; v[2] = q.z; v[3] = q.w;
    }
    __device__ __forceinline__ void load(int w, uint32_t (&v)[2][2][4]) const
    {
        const int64_t o = 64 * (int64_t)w;
        load16(a ? a + o : nullptr, v[0][0]);
        load16(b ? b + o : nullptr, v[0][1]);
        load16(fold && a ? a + o + second : nullptr, v[1][0]);
        load16(fold && b ? b + o + second : nullptr, v[1][1]);
    }
};

__global__ void __launch_bounds__(256) us_encode_size_kernel(const EncodeParams p)
{
    const int lane = threadIdx.x & 31, item = (int)(((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5);
    if (item >= p.n_items) return;
    const EncodeLane l(p, item, lane);
    int len = 0;
#pragma unroll 2
    for (int w = 0; w < p.mask_rows; ++w) {
        uint32_t v[2][2][4];
        l.load(w, v);
#pragma unroll
        for (int i = 0; i < 4; ++i) len += __popc(nonzero_nibbles(v[0][0][i] | v[0][1][i] | v[1][0][i] | v[1][1][i]));
    }
    const int longest = __reduce_max_sync(0xffffffffu, len), sum = __reduce_add_sync(0xffffffffu, len);
    if (lane == 0) {
        const int streams = p.fold && !p.w2 ? 2 : 1;
        p.size16[item] = (uint32_t)(p.mask_rows + (longest + 3) / 4 * streams) * 8u;   // 128-byte rows
        atomicAdd(p.sum_P, (unsigned long long)sum);
    }
}

// Exclusive prefix sum of the tile sizes: one block. item_off[n_items] = the total; out[0] = the total as 64 bits,
// out[1] = the largest size.
__global__ void __launch_bounds__(1024) us_encode_scan_kernel(const uint32_t* size16, uint32_t* item_off, int n, unsigned long long* out)
{
    __shared__ unsigned long long part[32];
    __shared__ unsigned long long carry_s;
    __shared__ uint32_t big_s;
    if (threadIdx.x == 0) { carry_s = 0; big_s = 0; }
    __syncthreads();
    uint32_t big = 0;
    for (int i0 = 0; i0 < n; i0 += 1024) {
        const int i = i0 + (int)threadIdx.x;
        const uint32_t mine = i < n ? size16[i] : 0u;
        big = max(big, mine);
        unsigned long long s = mine;
        for (int d = 1; d < 32; d <<= 1) {
            const unsigned long long t = __shfl_up_sync(0xffffffffu, s, d);
            if ((int)(threadIdx.x & 31) >= d) s += t;
        }
        if ((threadIdx.x & 31) == 31) part[threadIdx.x >> 5] = s;
        __syncthreads();
        if (threadIdx.x < 32) {
            unsigned long long t = part[threadIdx.x];
            for (int d = 1; d < 32; d <<= 1) {
                const unsigned long long q = __shfl_up_sync(0xffffffffu, t, d);
                if ((int)threadIdx.x >= d) t += q;
            }
            part[threadIdx.x] = t;
        }
        __syncthreads();
        const unsigned long long before = carry_s + (threadIdx.x >= 32 ? part[(threadIdx.x >> 5) - 1] : 0ull) + s - mine;
        if (i < n) item_off[i] = (uint32_t)before;
        __syncthreads();
        if (threadIdx.x == 0) carry_s += part[31];
        __syncthreads();
    }
    big = __reduce_max_sync(0xffffffffu, big);
    if ((threadIdx.x & 31) == 0) atomicMax(&big_s, big);
    __syncthreads();
    if (threadIdx.x == 0) { item_off[n] = (uint32_t)carry_s; out[0] = carry_s; out[1] = big_s; }
}

__global__ void __launch_bounds__(256) us_encode_write_kernel(const EncodeParams p)
{
    const int lane = threadIdx.x & 31, item = (int)(((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5);
    if (item >= p.n_items) return;
    const EncodeLane l(p, item, lane);
    const uint32_t off = p.item_off[item], size = p.item_off[item + 1] - off;
    uint32_t* mask = reinterpret_cast<uint32_t*>(p.blob + (size_t)off * 16) + lane;
    uint32_t* pay = mask + 32 * p.mask_rows;
    const int streams = p.fold && !p.w2 ? 2 : 1, row = 32 * streams;
    const int rows = (int)(size / 8u - (uint32_t)p.mask_rows) / streams;   // payload rows of a stream
    unsigned long long acc[2] = {0, 0};   // bytes not yet stored, per stream
    int n = 0, at = 0;                    // how many; payload row they go to
    for (int w = 0; w < p.mask_rows; ++w) {
        uint32_t mw = 0, v[2][2][4];
        l.load(w, v);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const uint32_t m = nonzero_nibbles(v[0][0][i] | v[0][1][i] | v[1][0][i] | v[1][1][i]);
            mw |= m << (8 * i);
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const int c = 4 * (2 * (j & 3) + (j >> 2));   // (slot_column)
                const uint32_t a0 = (v[0][0][i] >> c) & 15u, b0 = (v[0][1][i] >> c) & 15u;
                const uint32_t a1 = (v[1][0][i] >> c) & 15u, b1 = (v[1][1][i] >> c) & 15u;
                if ((m >> j) & 1u) {
                    if (p.w2) {
                        acc[0] |= (unsigned long long)(((a0 + 2u) & 3u) | (((b0 + 2u) & 3u) << 2) | (((a1 + 2u) & 3u) << 4) | (((b1 + 2u) & 3u) << 6)) << (8 * n);
                    } else {
                        acc[0] |= (unsigned long long)((b0 << 4) | (a0 ^ 8u)) << (8 * n);
                        acc[1] |= (unsigned long long)((b1 << 4) | (a1 ^ 8u)) << (8 * n);
                    }
                    ++n;
                }
                if (j == 3 || j == 7) {   // at most three and four bytes wait here
                    if (n >= 4) {
                        pay[at * row] = (uint32_t)acc[0];
                        if (streams == 2) pay[at * row + 32] = (uint32_t)acc[1];
                        acc[0] >>= 32; acc[1] >>= 32;
                        n -= 4;
                        ++at;
                    }
                }
            }
        }
        mask[32 * w] = mw;
    }
    for (; at < rows; ++at) {   // the partial last word, then zeros up to the tile's longest stream
        pay[at * row] = (uint32_t)acc[0];
        if (streams == 2) pay[at * row + 32] = (uint32_t)acc[1];
        acc[0] = acc[1] = 0;
    }
}

}  // namespace us
