// Device-side helpers: Philox4x32-10, range scaling, block/warp scans.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace lda {

// Philox4x32 with 10 rounds (Salmon et al., SC'11): counter-based, so a random
// word depends only on (seed, token, sweep, step) and not on which thread asks.
// Its ten rounds' keys come in one of two forms.  (The products of a round, 32 bits by 32, run at a quarter of the rate of other
// operations and bound the generator: 85 cycles per warp and scheduler.)
// PhiloxKey: worked out on the host, a round's exclusive-or takes them from the constant bank.  Keys added up in the kernel
// take issue slots beside the products: document pass of 738 M tokens, two steps, 9.97 ms, 9.81 so.
struct PhiloxKey {
    uint32_t k[20];
    PhiloxKey() = default;
    explicit __host__ __device__ PhiloxKey(unsigned long long seed)
    {
        for (int r = 0; r < 10; ++r) {
            k[2 * r] = (uint32_t)seed + (uint32_t)r * 0x9E3779B9u;
            k[2 * r + 1] = (uint32_t)(seed >> 32) + (uint32_t)r * 0xBB67AE85u;
        }
    }
    __device__ __forceinline__ uint2 round(int r) const { return make_uint2(k[2 * r], k[2 * r + 1]); }
};
// PhiloxSeed: added up in the kernel.  For loops over steps (document pass of doc-proposals alone, four steps, 24 M tokens,
// V = 10^6, K = 10^5: 1.121 ms with keys from the constant bank, 1.074 so; three steps of the cycle, 16 M: 394 us and 387), and
// where one block per token is little beside the rest (exact conditional, 2.6 M tokens, K = 1000: 1.298 ms and 1.293).
struct PhiloxSeed {
    uint32_t lo, hi;
    explicit __host__ __device__ PhiloxSeed(unsigned long long seed) : lo((uint32_t)seed), hi((uint32_t)(seed >> 32)) {}
    explicit __device__ __forceinline__ PhiloxSeed(const PhiloxKey& key) : lo(key.k[0]), hi(key.k[1]) {}
    __device__ __forceinline__ uint2 round(int r) const
    {
        return make_uint2(lo + (uint32_t)r * 0x9E3779B9u, hi + (uint32_t)r * 0xBB67AE85u);
    }
};

template <class Key>
__device__ __forceinline__ uint4 philox4x32_10(uint4 c, const Key& key)
{
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        // (the two halves of a product as two instructions: a wide multiplication ties up register pairs, which
        // costs the kernels at their register limit more than it saves)
        const uint32_t hi0 = __umulhi(0xD2511F53u, c.x), lo0 = 0xD2511F53u * c.x;
        const uint32_t hi1 = __umulhi(0xCD9E8D57u, c.z), lo1 = 0xCD9E8D57u * c.z;
        const uint2 k = key.round(r);
        c = make_uint4(hi1 ^ c.y ^ k.x, lo1, hi0 ^ c.w ^ k.y, lo0);
    }
    return c;
}

// (double)x for an unsigned 32-bit x, exactly, without the (slow) integer-to-double conversion
// instruction: x placed in the low mantissa bits of 2^52, then 2^52 subtracted.
__device__ __forceinline__ double u32_to_double(uint32_t x)
{
    return __dsub_rn(__hiloint2double(0x43300000, (int)x), 4503599627370496.0);
}

// floor(r * n / 2^32): a 32-bit random word mapped to {0..n-1}.
__device__ __forceinline__ uint32_t scale_to_range(uint32_t r, uint32_t n) { return __umulhi(r, n); }

__device__ __forceinline__ int bit_length(unsigned long long x) { return 64 - __clzll((long long)x); }

// Quotients part/whole <= 1 as 32-bit fractions (split points and mixture thresholds of Section 4.2),
// min(2^32 - 1, floor((part >> sh) * 2^32 / (whole >> sh))) with whole >> sh < 2^32, for many parts of one
// whole: from a double reciprocal of the (shifted) whole, set right with the exact integer remainder.  The
// estimate is within 2^-20 of the true quotient (two roundings of 2^-53 on a value <= 2^32), so
// its integer part is off by one at most.  A 64-bit integer division costs several times as much.
struct Frac32 {
    int sh;
    uint32_t w;  // whole >> sh, < 2^32
    double inv;  // 1 / w
    __device__ __forceinline__ explicit Frac32(unsigned long long whole)
    {
        sh = bit_length(whole) - 32;
        if (sh < 0) sh = 0;
        w = (uint32_t)(whole >> sh);
        inv = __ddiv_rn(1.0, u32_to_double(w));
    }
    __device__ __forceinline__ uint32_t operator()(unsigned long long part) const
    {
        const uint32_t p = (uint32_t)(part >> sh);  // part <= whole
        const unsigned long long x = (unsigned long long)p << 32;
        unsigned long long q = __double2ull_rz(__dmul_rn(__dmul_rn(u32_to_double(p), 4294967296.0), inv));
        const long long r = (long long)(x - q * (unsigned long long)w);
        if (r < 0) --q;
        else if (r >= (long long)w) ++q;
        return q > 0xFFFFFFFFull ? 0xFFFFFFFFu : (uint32_t)q;
    }
};

// Share of a word's sparse term (mass S) in its proposal, the dense term having mass B.
__device__ __forceinline__ uint32_t mixture_threshold(unsigned long long S, unsigned long long B)
{
    return S == 0 ? 0u : Frac32(S + B)(S);
}

// --- n_kd tables --------------------------------------------------------------------------------
// Section 5's hashed rows (fn. 5 asks for at least twice as many slots as entries), one table per
// document: `cap` = DK_SLOTS_PER_TOKEN * (document length) slots, so the load factor stays <= 0.25 (some document tiles have
// more: tile_slots() in docside.cu).  A slot is
// (topic << count_bits) | count, or DK_EMPTY_SLOT.  Open addressing with linear probing: topic k
// starts at slot floor(k * DK_HASH_MULT mod 2^32 * cap / 2^32) and moves up one slot at a time,
// wrapping; an empty slot met on the way means "absent".  At this load a search takes about 1.2
// probes (found) or 1.4 (absent).
constexpr uint32_t DK_EMPTY_SLOT = 0xFFFFFFFFu;
constexpr uint32_t DK_HASH_MULT = 0x9E3779B1u;
constexpr int DK_SLOTS_PER_TOKEN = 4;

__device__ __forceinline__ uint32_t dk_home(uint32_t k, uint32_t cap) { return __umulhi(k * DK_HASH_MULT, cap); }

// Adds one occurrence of topic k to the table `tab[0..cap)`: claims an empty slot with one
// compare-and-swap that also sets the count to 1, or finds the topic's slot and adds one to its
// count bits.  Safe against concurrent insertions into the same table.  Returns the slot, or
// DK_EMPTY_SLOT if the table had no room (which the load factor rules out).
__device__ __forceinline__ uint32_t dk_insert(uint32_t* tab, uint32_t cap, uint32_t k, int count_bits)
{
    const uint32_t first = (k << count_bits) | 1u;
    uint32_t h = dk_home(k, cap);
    for (uint32_t n = 0; n < cap; ++n) {
        const uint32_t prev = atomicCAS(&tab[h], DK_EMPTY_SLOT, first);
        if (prev == DK_EMPTY_SLOT) return h;
        if ((prev >> count_bits) == k) {
            atomicAdd(&tab[h], 1u);
            return h;
        }
        if (++h == cap) h = 0;
    }
    return DK_EMPTY_SLOT;
}

// n_kd[k] as a packed entry (0 when absent).
__device__ __forceinline__ uint32_t dk_lookup(const uint32_t* tab, uint32_t cap, uint32_t k, int count_bits)
{
    uint32_t h = dk_home(k, cap);
    for (uint32_t n = 0; n < cap; ++n) {
        const uint32_t e = tab[h];
        if (e == DK_EMPTY_SLOT) return 0u;
        if ((e >> count_bits) == k) return e;
        if (++h == cap) h = 0;
    }
    return 0u;
}

// 32 bytes to an address that is a multiple of 32: a whole sector in one access.  L2 takes scattered whole sectors at a higher
// rate than halves: records written in random order within 2^20, 2^21 and 2^22 of them 148, 100 and 62 G/s, as two 16-byte
// stores 61, 52 and 44.
__device__ __forceinline__ void store_32(void* p, uint4 a, uint4 b)
{
    asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "r"(a.x), "r"(a.y), "r"(a.z), "r"(a.w),
                 "r"(b.x), "r"(b.y), "r"(b.z), "r"(b.w)
                 : "memory");
}
__device__ __forceinline__ void load_32(const void* p, uint4& a, uint4& b)
{
    asm volatile("ld.global.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(a.x), "=r"(a.y), "=r"(a.z), "=r"(a.w), "=r"(b.x), "=r"(b.y), "=r"(b.z), "=r"(b.w)
                 : "l"(p));
}

template <typename T>
__device__ __forceinline__ T warp_reduce_sum(T v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Inclusive scan across the 32 lanes of a warp.
template <typename T>
__device__ __forceinline__ T warp_scan_incl(T v)
{
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        T u = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += u;
    }
    return v;
}

// Block-wide sum; `smem` holds at least 32 T; result returned to every thread.
template <typename T>
__device__ __forceinline__ T block_reduce_sum(T v, T* smem)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
    v = warp_reduce_sum(v);
    __syncthreads();
    if (lane == 0) smem[warp] = v;
    __syncthreads();
    T t = (lane < nw) ? smem[lane] : T(0);
    t = warp_reduce_sum(t);
    return t;
}

// Block-wide exclusive scan of one value per thread; returns the exclusive
// prefix and writes the block total to `total`.  `smem` holds at least 33 T.
template <typename T>
__device__ __forceinline__ T block_scan_excl(T v, T* smem, T& total)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
    T incl = warp_scan_incl(v);
    __syncthreads();
    if (lane == 31) smem[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        T w = (lane < nw) ? smem[lane] : T(0);
        T wi = warp_scan_incl(w);
        smem[lane] = wi - w;
        if (lane == 31) smem[32] = wi;
    }
    __syncthreads();
    total = smem[32];
    return smem[warp] + incl - v;
}

}  // namespace lda
