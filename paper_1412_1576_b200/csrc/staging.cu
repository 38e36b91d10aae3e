// Copies between device memory and host memory that is not page-locked.  The runtime's own copy of such memory
// runs at the speed of one host thread (8-12 GB/s here, the link takes 55); these go through small page-locked
// buffers by several threads at once, each moving every LANES-th piece: while one thread's piece is on the link,
// the others copy theirs between its buffer and the caller's memory.
// The buffers and their streams are made at the first large copy and shared by all contexts of the process
// (LANES x 2 x PIECE bytes, one copy at a time; a second copy at the same moment takes the runtime's way).
#include <algorithm>
#include <cstring>
#include <mutex>
#include <thread>

#include <cuda.h>

#include "lda_internal.cuh"

namespace lda {

// Every piece costs calls into the driver, which take turns: 160 MB to the device and 320 MB back took 10.0 and 17.5 ms
// in pieces of 512 KiB, 7.2 and 12.4 in pieces of 2 MiB.  Shorter copies go in shorter pieces, four per lane as long as
// those are not below PIECE_MIN (16 MiB; a copy of 2 MiB is four pieces, and four lanes have nothing to do).
constexpr int LANES = 8;
constexpr size_t PIECE = 2 << 20, PIECE_MIN = 512 << 10;
// Below this a copy is over before the threads have started.
constexpr size_t STAGED_MIN = 2 << 20;

struct Lane {
    char* pinned = nullptr;  // two pieces
    cudaStream_t stream = nullptr;
    cudaEvent_t done[2] = {};
};
struct StagingPool {
    std::mutex lock;
    int device = -1;
    Lane lane[LANES];
    void release()
    {
        for (Lane& l : lane) {
            for (cudaEvent_t& e : l.done)
                if (e) cudaEventDestroy(e);
            if (l.stream) cudaStreamDestroy(l.stream);
            if (l.pinned) cudaFreeHost(l.pinned);
            l = Lane{};
        }
        device = -1;
        cudaGetLastError();
    }
    bool ready(int dev)  // under the lock
    {
        if (device == dev) return true;
        if (device >= 0) release();
        bool ok = true;
        for (Lane& l : lane) {
            ok = ok && cudaHostAlloc(reinterpret_cast<void**>(&l.pinned), 2 * PIECE, cudaHostAllocPortable) == cudaSuccess;
            ok = ok && cudaStreamCreateWithFlags(&l.stream, cudaStreamNonBlocking) == cudaSuccess;
            for (cudaEvent_t& e : l.done) ok = ok && cudaEventCreateWithFlags(&e, cudaEventDisableTiming) == cudaSuccess;
        }
        if (!ok) {
            release();
            return false;
        }
        device = dev;
        return true;
    }
    static StagingPool& pool()
    {
        static StagingPool* p = new StagingPool;  // never destroyed: the process's end releases what it holds
        return *p;
    }
};

bool page_locked(const void* p)
{
    cudaPointerAttributes a{};
    if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return a.type != cudaMemoryTypeUnregistered;
}

// Of the driver's interface, which is not linked: the runtime's own query says nothing about how far page-locked memory
// reaches.  (Its first and last byte are not enough: two registrations may have other memory between them, and device
// addresses are host addresses.)
void* device_view(const void* p, size_t bytes)
{
    using Query = CUresult (*)(unsigned int, CUpointer_attribute*, void**, CUdeviceptr);
    static const Query query = [] {
        void* f = nullptr;
        cudaDriverEntryPointQueryResult found{};
        if (cudaGetDriverEntryPointByVersion("cuPointerGetAttributes", &f, 7000, cudaEnableDefault, &found) != cudaSuccess ||
            found != cudaDriverEntryPointSuccess) {
            cudaGetLastError();
            f = nullptr;
        }
        return reinterpret_cast<Query>(f);
    }();
    if (!query) return nullptr;
    // what a pointer has no value for stays as it is
    unsigned int type = 0;
    unsigned long long at = 0, start = 0, size = 0, access = 0;
    CUpointer_attribute names[] = {CU_POINTER_ATTRIBUTE_MEMORY_TYPE, CU_POINTER_ATTRIBUTE_DEVICE_POINTER,
                                   CU_POINTER_ATTRIBUTE_RANGE_START_ADDR, CU_POINTER_ATTRIBUTE_RANGE_SIZE, CU_POINTER_ATTRIBUTE_ACCESS_FLAGS};
    void* values[] = {&type, &at, &start, &size, &access};
    if (query(5, names, values, (CUdeviceptr)(uintptr_t)p) != CUDA_SUCCESS) return nullptr;
    if (type != CU_MEMORYTYPE_HOST || access != CU_POINTER_ATTRIBUTE_ACCESS_FLAG_READWRITE) return nullptr;
    const bool inside = at >= start && at - start <= size && bytes <= size - (at - start);
    return inside ? reinterpret_cast<void*>((uintptr_t)at) : nullptr;
}

template <bool TO_HOST>
static cudaError_t move_lane(Lane& l, int device, int first, char* host, char* dev, size_t bytes, size_t piece)
{
    cudaError_t e = cudaSetDevice(device);
    size_t pending_at[2] = {0, 0}, pending_n[2] = {0, 0};
    int b = 0;
    auto finish = [&](int i) {  // the piece in half i is on its way: wait for it, and pass it on
        if (!pending_n[i]) return;
        const cudaError_t w = cudaEventSynchronize(l.done[i]);
        if (e == cudaSuccess) e = w;
        if (TO_HOST && w == cudaSuccess) std::memcpy(host + pending_at[i], l.pinned + i * PIECE, pending_n[i]);
        pending_n[i] = 0;
    };
    for (size_t at = (size_t)first * piece; at < bytes && e == cudaSuccess; at += (size_t)LANES * piece, b ^= 1) {
        const size_t n = bytes - at < piece ? bytes - at : piece;
        char* half = l.pinned + b * PIECE;
        finish(b);
        if (e != cudaSuccess) break;
        if (!TO_HOST) std::memcpy(half, host + at, n);
        e = TO_HOST ? cudaMemcpyAsync(half, dev + at, n, cudaMemcpyDeviceToHost, l.stream)
                    : cudaMemcpyAsync(dev + at, half, n, cudaMemcpyHostToDevice, l.stream);
        if (e == cudaSuccess) e = cudaEventRecord(l.done[b], l.stream);
        if (e == cudaSuccess) {
            pending_at[b] = at;
            pending_n[b] = n;
        }
    }
    finish(b);
    finish(b ^ 1);
    cudaStreamSynchronize(l.stream);  // after an error: nothing of this copy stays on its way
    return e;
}

template <bool TO_HOST>
static cudaError_t move_bytes(Ctx& c, void* host, void* dev, size_t bytes)
{
    // what was queued so far comes first; the lanes have streams of their own
    cudaError_t e = cudaStreamSynchronize(c.stream);
    if (e != cudaSuccess || bytes == 0) return e;
    if (bytes >= STAGED_MIN && !page_locked(host)) {
        StagingPool& p = StagingPool::pool();
        std::unique_lock<std::mutex> g(p.lock, std::try_to_lock);
        if (g.owns_lock() && p.ready(c.device)) {
            cudaError_t err[LANES];
            std::thread t[LANES];
            int started = 0;
            const size_t piece = std::min(PIECE, std::max(PIECE_MIN, bytes / (4 * LANES) / 4096 * 4096));
            char *h = static_cast<char*>(host), *d = static_cast<char*>(dev);
            auto lane = [&](int i) { err[i] = move_lane<TO_HOST>(p.lane[i], c.device, i, h, d, bytes, piece); };
            try {
                for (; started < LANES - 1; ++started) t[started] = std::thread(lane, started);
            } catch (...) {  // no more threads to be had: this one does the rest
            }
            for (int i = started; i < LANES; ++i) lane(i);
            for (int i = 0; i < started; ++i) t[i].join();
            for (cudaError_t x : err)
                if (x != cudaSuccess) e = x;
            return e;
        }
    }
    // on the context's stream: a copy on the default stream may return before the data has arrived, and nothing orders
    // a non-blocking stream behind that
    e = TO_HOST ? cudaMemcpyAsync(host, dev, bytes, cudaMemcpyDeviceToHost, c.stream)
                : cudaMemcpyAsync(dev, host, bytes, cudaMemcpyHostToDevice, c.stream);
    const cudaError_t done = cudaStreamSynchronize(c.stream);
    return e != cudaSuccess ? e : done;
}

cudaError_t copy_to_host(Ctx& c, void* host, const void* dev, size_t bytes)
{
    return move_bytes<true>(c, host, const_cast<void*>(dev), bytes);
}
cudaError_t copy_to_device(Ctx& c, void* dev, const void* host, size_t bytes)
{
    return move_bytes<false>(c, const_cast<void*>(host), dev, bytes);
}

}  // namespace lda
