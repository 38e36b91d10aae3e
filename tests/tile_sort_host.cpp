// tile_sort.cuh on the host: the threads of the CTA are contexts of one host thread, a warp runs as far as the next barrier
// before the next warp is let go, and the caller says in which order.  What one warp writes before another has read it shows.
#include <ucontext.h>

#include <algorithm>
#include <cstdint>
#include <cstring>
#include <vector>

struct uint4 {
    uint32_t x, y, z, w;
};
static uint4 make_uint4(uint32_t x, uint32_t y, uint32_t z, uint32_t w) { return uint4{x, y, z, w}; }
using std::max;
using std::min;
static struct {
    int x;
} threadIdx;
static void __syncthreads();
static uint32_t __shfl_xor_sync(uint32_t mask, uint32_t value, int distance);
#define __device__
#define __forceinline__ inline
#include "../paper_1412_1576_b200/csrc/tile_sort.cuh"

namespace {

constexpr int THREADS = lda::SORT_THREADS, WARPS = THREADS / 32, KEYS = THREADS * lda::SORT_PER;
enum Wait { RUNS, AT_SHUFFLE, AT_BARRIER, DONE };
struct Thread {
    ucontext_t context;
    std::vector<char> stack = std::vector<char>(64 << 10);
    Wait wait;
    uint32_t given;
} threads[THREADS];
ucontext_t scheduler;
alignas(16) uint32_t keys[KEYS];
struct {
    const uint32_t* z;
    const int32_t* off;
    int32_t segments, cnt, K;
    int topic_bits;
    uint32_t* in_registers;
    int* in_range;
} job;

void pause(Wait why)
{
    const int me = threadIdx.x;
    threads[me].wait = why;
    swapcontext(&threads[me].context, &scheduler);
}

void body()
{
    uint32_t x[lda::SORT_PER];
    if (!lda::tile_keys(x, keys, job.off, job.segments, job.z, job.cnt, job.topic_bits, job.K)) *job.in_range = 0;
    lda::sort_tile(x, keys, job.cnt);
    std::memcpy(job.in_registers + threadIdx.x * lda::SORT_PER, x, sizeof x);
    threads[threadIdx.x].wait = DONE;
}

bool all(int first, int n, Wait w)
{
    return std::all_of(threads + first, threads + first + n, [=](const Thread& t) { return t.wait == w; });
}

// A warp as far as it gets without the others: all its threads at a barrier, or through.
bool run_warp(int warp)
{
    for (;;) {
        for (int t = 32 * warp; t < 32 * warp + 32; ++t) {
            if (threads[t].wait != RUNS) continue;
            threadIdx.x = t;
            swapcontext(&scheduler, &threads[t].context);
        }
        if (!all(32 * warp, 32, AT_SHUFFLE)) break;
        for (int t = 32 * warp; t < 32 * warp + 32; ++t) threads[t].wait = RUNS;
    }
    return all(32 * warp, 32, AT_BARRIER) || all(32 * warp, 32, DONE);
}

}  // namespace

static void __syncthreads() { pause(AT_BARRIER); }
static uint32_t __shfl_xor_sync(uint32_t, uint32_t value, int distance)
{
    const int me = threadIdx.x;
    threads[me].given = value;
    pause(AT_SHUFFLE);
    const uint32_t got = threads[me ^ distance].given;
    pause(AT_SHUFFLE);  // nobody gives the next value before all have this one
    return got;
}

// Both copies of the sorted keys; `in_range`: no thread saw a topic outside [0, K).  0, or -1 if threads of a warp part.
extern "C" int tile_sort_host(const uint32_t* z, const int32_t* off, int32_t segments, int32_t topic_bits, int32_t K,
                              const int32_t* warp_order, uint32_t* in_registers, uint32_t* in_shared, int* in_range)
{
    *in_range = 1;
    job = {z, off, segments, off[segments], K, topic_bits, in_registers, in_range};
    for (Thread& t : threads) {
        getcontext(&t.context);
        t.context.uc_stack.ss_sp = t.stack.data();
        t.context.uc_stack.ss_size = t.stack.size();
        t.context.uc_link = &scheduler;
        makecontext(&t.context, body, 0);
        t.wait = RUNS;
    }
    while (!all(0, THREADS, DONE)) {
        for (int w = 0; w < WARPS; ++w)
            if (!run_warp(warp_order[w])) return -1;
        if (all(0, THREADS, AT_BARRIER))
            for (Thread& t : threads) t.wait = RUNS;
        else if (!all(0, THREADS, DONE)) return -1;
    }
    std::memcpy(in_shared, keys, sizeof keys);
    return 0;
}
