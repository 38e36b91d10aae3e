// Sort of a tile's (segment, topic) keys by one CTA of SORT_THREADS threads, for k_seg_count_sorted (counts.cu).  A header of
// its own without CUDA headers: its barriers are tested on the host, warp by warp in any order (tests/tile_sort_host.cpp).
#pragma once
#include <cstdint>

namespace lda {

constexpr int SORT_THREADS = 256, SORT_PER = 8;  // keys of a thread: two 16-byte words

// Keys (segment << topic_bits | topic) of a tile's tokens [0, cnt), eight consecutive ones in every thread's registers; past
// `cnt` the largest value.  `off` [segments + 1]: first token of each segment.  The topics are read from `z` in order, then picked
// up from `keys` [SORT_THREADS * SORT_PER], which is shared memory like `off`.  False on a thread that saw a topic outside [0, K).
// Starts after a barrier behind `off`; ends WITHOUT one behind its reads of `keys`.
template <typename T>
__device__ __forceinline__ bool tile_keys(uint32_t (&x)[SORT_PER], uint32_t* keys, const int32_t* off, int32_t segments,
                                          const T* z, int32_t cnt, int topic_bits, int32_t K)
{
    const int tid = threadIdx.x;
    for (int j = tid; j < SORT_THREADS * SORT_PER; j += SORT_THREADS) keys[j] = j < cnt ? (uint32_t)z[j] : 0xFFFFFFFFu;
    __syncthreads();
    const uint4 lo4 = reinterpret_cast<const uint4*>(keys)[2 * tid], hi4 = reinterpret_cast<const uint4*>(keys)[2 * tid + 1];
    const uint32_t k[SORT_PER] = {lo4.x, lo4.y, lo4.z, lo4.w, hi4.x, hi4.y, hi4.z, hi4.w};
    int seg = 0, hi = segments;  // last segment with off[seg] <= j
    while (hi - seg > 1) {
        const int mid = (seg + hi) >> 1;
        if (off[mid] <= tid * SORT_PER) seg = mid; else hi = mid;
    }
    bool in_range = true;
#pragma unroll
    for (int q = 0; q < SORT_PER; ++q) {
        const int j = tid * SORT_PER + q;
        x[q] = 0xFFFFFFFFu;
        if (j >= cnt) continue;
        while (off[seg + 1] <= j) ++seg;
        in_range = in_range && k[q] < (uint32_t)K;
        x[q] = ((uint32_t)seg << topic_bits) | k[q];
    }
    return in_range;
}

// Ascending sort of what tile_keys() left.  Leaves the keys in `keys` as well.  A bitonic network, its steps by the distance of the
// two keys that they compare: in a thread's registers, in a warp by shuffles, and only the six widest through shared memory.
// (All 66 steps there, a barrier after each: n_kw of 200 M tokens, V = 10^6, K = 10^5, 3.69 ms; so 2.55.)
// All threads call it.  Its first barrier stands between other threads' last reads of `keys` and its first stores there: the
// exchanges between warps write all over `keys`, and the steps before them order a warp's threads only.  Ends with one.
__device__ __forceinline__ void sort_tile(uint32_t (&x)[SORT_PER], uint32_t* keys, int32_t cnt)
{
    constexpr uint32_t FULL = 0xFFFFFFFFu;
    const int tid = threadIdx.x;
    auto order = [](uint32_t& a, uint32_t& b, bool up) {
        const uint32_t lo = min(a, b), hi = max(a, b);
        a = up ? lo : hi;
        b = up ? hi : lo;
    };
    auto in_thread = [&](bool up) {  // steps of 4, 2 and 1 in one direction
#pragma unroll
        for (int stride = 4; stride > 0; stride >>= 1)
#pragma unroll
            for (int q = 0; q < SORT_PER; ++q)
                if (!(q & stride)) order(x[q], x[q | stride], up);
    };
    uint4* area = reinterpret_cast<uint4*>(keys);  // a thread's two words SORT_THREADS apart: no bank conflicts
    auto store = [&](int at0, int at1) {
        area[at0] = make_uint4(x[0], x[1], x[2], x[3]);
        area[at1] = make_uint4(x[4], x[5], x[6], x[7]);
    };
    __syncthreads();
#pragma unroll
    for (int q = 0; q < SORT_PER; q += 2) order(x[q], x[q + 1], !(q & 2));
#pragma unroll
    for (int q = 0; q < SORT_PER; ++q)
        if (!(q & 2)) order(x[q], x[q | 2], !(q & 4));
#pragma unroll
    for (int q = 0; q < SORT_PER; q += 2) order(x[q], x[q + 1], !(q & 4));
    in_thread(!(tid & 1));
    // `size`: keys of a sorted run, in threads; a tile of few keys needs only the first of them
    for (int size = 2; size <= SORT_THREADS && size * SORT_PER < 2 * cnt; size <<= 1) {
        const bool up = !(tid & size);
        for (int stride = size >> 1; stride > 0; stride >>= 1) {
            const bool keep_low = !(tid & stride) == up;
            uint32_t y[SORT_PER];
            if (stride >= 32) {
                store(tid, tid + SORT_THREADS);
                __syncthreads();
                const uint4 a = area[tid ^ stride], b = area[(tid ^ stride) + SORT_THREADS];
                __syncthreads();
                y[0] = a.x; y[1] = a.y; y[2] = a.z; y[3] = a.w;
                y[4] = b.x; y[5] = b.y; y[6] = b.z; y[7] = b.w;
            } else {
#pragma unroll
                for (int q = 0; q < SORT_PER; ++q) y[q] = __shfl_xor_sync(FULL, x[q], stride);
            }
#pragma unroll
            for (int q = 0; q < SORT_PER; ++q) x[q] = keep_low ? min(x[q], y[q]) : max(x[q], y[q]);
        }
        in_thread(up);
    }
    store(2 * tid, 2 * tid + 1);
    __syncthreads();
}

}  // namespace lda
