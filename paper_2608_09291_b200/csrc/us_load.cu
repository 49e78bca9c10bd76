// Bringing a weight onto the GPU: packing on the host's cores, upload and encoding overlapped, device memory from a pool.
#include <algorithm>
#include <atomic>
#include <exception>
#include <mutex>
#include <thread>

#include "us_device_encode.cuh"
#include "us_load.h"

namespace us {
namespace {

// ---- per-device memory pool, upload stream and pinned staging ------------------------------------------------------
// A cudaMalloc costs 340 us on the machines measured, a cudaFree 290, and a handle has eight arrays: 5 ms per weight
// loaded. Allocations from a CUDA memory pool cost 2 us. The pool keeps at most kPoolKeep bytes beyond what live handles
// hold and gives the rest back at the next synchronisation; the staging buffer is of fixed size. All operations on the
// pool go through its own stream, under a lock.
constexpr int kMaxThreads = 16;
constexpr size_t kChunk = 512 * 1024;       // bytes of a staging buffer, two per thread: copies of this size run at 37 GB/s,
                                            // of 128 KB at 20
constexpr uint64_t kPoolKeep = 64ull << 20;

struct Device {
    std::mutex mu;
    bool ready = false;
    cudaMemPool_t pool = nullptr;
    cudaStream_t stream = nullptr;
    uint8_t* staging = nullptr;
    cudaEvent_t copied[2 * kMaxThreads] = {};
};
constexpr int kMaxDevices = 64;
Device g_dev[kMaxDevices];

cudaError_t open_device(int device, Device** out)
{
    if (device < 0 || device >= kMaxDevices) return cudaErrorInvalidDevice;
    Device& d = g_dev[device];
    *out = &d;
    if (d.ready) return cudaSuccess;
    cudaMemPoolProps props = {};
    props.allocType = cudaMemAllocationTypePinned;
    props.location.type = cudaMemLocationTypeDevice;
    props.location.id = device;
    cudaError_t e = d.pool ? cudaSuccess : cudaMemPoolCreate(&d.pool, &props);
    uint64_t keep = kPoolKeep;
    if (e == cudaSuccess) e = cudaMemPoolSetAttribute(d.pool, cudaMemPoolAttrReleaseThreshold, &keep);
    if (e == cudaSuccess && !d.stream) e = cudaStreamCreateWithFlags(&d.stream, cudaStreamNonBlocking);
    if (e == cudaSuccess && !d.staging) e = cudaHostAlloc((void**)&d.staging, 2 * kMaxThreads * kChunk, cudaHostAllocDefault);
    for (int i = 0; i < 2 * kMaxThreads && e == cudaSuccess; ++i)
        if (!d.copied[i]) e = cudaEventCreateWithFlags(&d.copied[i], cudaEventDisableTiming);
    d.ready = e == cudaSuccess;
    return e;
}

// What encode_device holds, given back on every way out: its temporaries in stream order, the matrix too unless it is done.
struct Scratch {
    cudaStream_t st;
    DeviceMatrix* out;
    uint8_t* dense = nullptr;
    uint32_t* size16 = nullptr;
    unsigned long long* sums = nullptr;   // total size, largest size, sum of P
    bool done = false;
    ~Scratch()
    {
        if (!done) cudaStreamSynchronize(st);
        for (void* p : {(void*)dense, (void*)size16, (void*)sums}) if (p) cudaFreeAsync(p, st);
        if (done) return;
        for (void* p : {(void*)out->blob, (void*)out->item_off, (void*)out->row_order}) if (p) cudaFreeAsync(p, st);
        *out = DeviceMatrix();
        cudaGetLastError();
    }
};

}  // namespace

cudaError_t pool_alloc(int device, void** p, size_t bytes)
{
    *p = nullptr;
    if (device < 0 || device >= kMaxDevices) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lock(g_dev[device].mu);
    Device* d;
    const cudaError_t e = open_device(device, &d);
    return e == cudaSuccess ? cudaMallocFromPoolAsync(p, std::max<size_t>(bytes, 16), d->pool, d->stream) : e;
}

void pool_free(int device, void* p)
{
    if (!p || device < 0 || device >= kMaxDevices) return;
    std::lock_guard<std::mutex> lock(g_dev[device].mu);
    cudaFreeAsync(p, g_dev[device].stream);
}

cudaStream_t pool_stream(int device) { return g_dev[device].stream; }

us_status encode_device(const int8_t* W, int device, uint32_t flags, HostMatrix* hp, DeviceMatrix* out)
{
    HostMatrix& h = *hp;
    const int64_t M = h.M, K = h.K, ld = h.Kp / 2, total = M * ld;
    const bool sort = (flags & US_ENCODE_SORT_ROWS) && !(flags & US_ENCODE_PAIR_ROWS);   // (with pairing: ordered already)
    if (device < 0 || device >= kMaxDevices) return US_ERR_CUDA;
    std::lock_guard<std::mutex> lock(g_dev[device].mu);
    Device* d;
    if (open_device(device, &d) != cudaSuccess) return US_ERR_CUDA;
    cudaStream_t st = d->stream;

    Scratch t{st, out};
    auto alloc = [&](auto** p, size_t bytes) { return cudaMallocFromPoolAsync((void**)p, std::max<size_t>(bytes, 16), d->pool, st); };
    if (alloc(&t.dense, (size_t)total) != cudaSuccess || alloc(&t.size16, (size_t)h.n_items * 4) != cudaSuccess ||
        alloc(&t.sums, 24) != cudaSuccess || alloc(&out->item_off, (size_t)(h.n_items + 1) * 4) != cudaSuccess ||
        alloc(&out->row_order, (size_t)h.Mp * 4) != cudaSuccess)
        return US_ERR_ALLOC;

    // ---- pack to INT4 (range check, nonzeros per row) and upload, chunk by chunk on all cores ----------------------
    const size_t chunk = (size_t)std::min<int64_t>(kChunk, std::max<int64_t>(32 * 1024, (total / (2 * kMaxThreads) + 4095) / 4096 * 4096));
    const int64_t n_chunks = (total + (int64_t)chunk - 1) / (int64_t)chunk;
    const int n_thr = (int)std::min<int64_t>({kMaxThreads, std::max(1u, std::thread::hardware_concurrency()), n_chunks});
    std::vector<std::atomic<int32_t>> row_nnz((size_t)M);
    for (auto& c : row_nnz) c.store(0, std::memory_order_relaxed);
    std::atomic<int64_t> next{0};
    std::atomic<int> bad{0}, failed{0};
    auto work = [&](int i) {
        if (i > 0 && cudaSetDevice(device) != cudaSuccess) { failed = 1; return; }
        for (int k = 0;; ++k) {
            const int64_t c = next.fetch_add(1);
            if (c >= n_chunks || bad.load(std::memory_order_relaxed)) break;
            const int b = 2 * i + (k & 1);
            uint8_t* buf = d->staging + (size_t)b * kChunk;
            if (k >= 2 && cudaEventSynchronize(d->copied[b]) != cudaSuccess) { failed = 1; break; }
            const int64_t o0 = c * (int64_t)chunk, o1 = std::min<int64_t>(total, o0 + (int64_t)chunk);
            if (!pack_int4(W, K, ld, o0, o1, buf, h.w2, row_nnz.data())) { bad = 1; break; }
            if (cudaMemcpyAsync(t.dense + o0, buf, (size_t)(o1 - o0), cudaMemcpyHostToDevice, st) != cudaSuccess ||
                cudaEventRecord(d->copied[b], st) != cudaSuccess) { failed = 1; break; }
        }
    };
    {
        std::vector<std::thread> pool;
        pool.reserve((size_t)n_thr);
        try {
            for (int i = 1; i < n_thr; ++i) pool.emplace_back(work, i);
        } catch (const std::exception&) {   // fewer threads do it too
        }
        work(0);
        for (auto& th : pool) th.join();
    }
    if (bad) return US_ERR_VALUE_RANGE;
    if (failed) return US_ERR_CUDA;
    if (sort) {
        std::vector<int64_t> cnt((size_t)M);
        for (int64_t r = 0; r < M; ++r) cnt[r] = row_nnz[r].load(std::memory_order_relaxed);
        sort_rows(cnt, &h);
    }
    h.nnz = 0;
    for (auto& c : row_nnz) h.nnz += c.load(std::memory_order_relaxed);

    // ---- tile sizes, offsets, tiles ---------------------------------------------------------------------------------
    EncodeParams p = {};
    p.W = t.dense; p.row_order = out->row_order; p.ld = ld;
    p.n_segs = (int32_t)h.n_segs; p.n_items = (int32_t)h.n_items; p.K_L = h.fmt.K_L; p.mask_rows = h.mask_rows;
    p.fold = h.fmt.C_A == 2; p.w2 = h.w2;
    p.size16 = t.size16; p.item_off = out->item_off; p.sum_P = t.sums + 2;
    cudaMemsetAsync(t.sums, 0, 24, st);
    cudaMemcpyAsync(out->row_order, h.row_order.data(), (size_t)h.Mp * 4, cudaMemcpyHostToDevice, st);
    const unsigned blocks = (unsigned)((h.n_items + 7) / 8);
    us_encode_size_kernel<<<blocks, 256, 0, st>>>(p);
    us_encode_scan_kernel<<<1, 1024, 0, st>>>(t.size16, out->item_off, p.n_items, t.sums);
    unsigned long long got[3] = {0, 0, 0};
    h.item_off.resize((size_t)h.n_items + 1);
    cudaMemcpyAsync(got, t.sums, sizeof(got), cudaMemcpyDeviceToHost, st);
    cudaMemcpyAsync(h.item_off.data(), out->item_off, h.item_off.size() * 4, cudaMemcpyDeviceToHost, st);
    if (cudaGetLastError() != cudaSuccess || cudaStreamSynchronize(st) != cudaSuccess) return US_ERR_CUDA;
    if (got[0] > 0xFFFFFFFFull) return US_ERR_ALLOC;
    h.blob_bytes = got[0] * 16;
    h.max_item_bytes = (uint32_t)got[1] * 16u;
    h.sum_P = (int64_t)got[2];
    h.bytes_payload_padded = (int64_t)h.blob_bytes - h.n_items * (int64_t)h.mask_rows * 128;
    if (alloc(&out->blob, (size_t)h.blob_bytes) != cudaSuccess) return US_ERR_ALLOC;
    p.blob = out->blob;
    us_encode_write_kernel<<<blocks, 256, 0, st>>>(p);
    if (cudaGetLastError() != cudaSuccess) return US_ERR_CUDA;
    t.done = true;
    return US_OK;
}

}  // namespace us
