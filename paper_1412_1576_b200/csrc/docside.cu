// Document side of the MH step (pass 2), one tile of whole documents per CTA.
//
// The sweep-start n_kd of a document (Eq. 12) is a function of that document's assignments
// alone, so the tile's tables are built where they are used: in shared memory, by insertion
// (Section 5's hashed rows: claim a slot with compare-and-swap, then add one to its count), and
// thrown away afterwards.  Every token then gathers what the accept/reject pass needs from this
// side:
//   - the token's own (topic, n_kd) record,
//   - for every word-proposal (drawn by pass 1): n_kd at the proposed topic,
//   - for every doc-proposal (Eq. 9, Eq. 12): the Philox block of the step, the proposed topic
//     -- the topic of a random token of the document, or a uniform topic with probability
//     K*alpha / (n_d + K*alpha) -- its n_kd, and the step's acceptance uniform.
// The current assignments and the word-proposals arrive in block-major order and the results go
// back in block-major order: a tile's documents lie in one block of that order (two at a block
// border), so these scattered reads and writes stay in L2.
#include <type_traits>

#include "lda_device.cuh"
#include "lda_internal.cuh"

namespace lda {

constexpr double INV_2_32 = 1.0 / 4294967296.0;

// A token's current topic and its first word-proposal sit side by side at its block-major index:
// one read brings both.
__device__ __forceinline__ void load_topic_pair(const uint16_t* zbm, uint32_t bm, uint32_t& z, uint32_t& t1)
{
    const uint32_t w = __ldcg(reinterpret_cast<const uint32_t*>(zbm) + bm);
    z = w & 0xFFFFu;
    t1 = w >> 16;
}
__device__ __forceinline__ void load_topic_pair(const int32_t* zbm, uint32_t bm, uint32_t& z, uint32_t& t1)
{
    const uint2 w = __ldcg(reinterpret_cast<const uint2*>(zbm) + bm);
    z = w.x;
    t1 = w.y;
}

// --- n_kd of a document in a tile, in shared memory ----------------------------------------------
// Two forms, chosen per corpus (load_common()):
//   DENSE   a 16-bit counter per topic (K even or padded): an addition, a read;
//   hashed  tile_slots() slots per token, as dk_insert in lda_device.cuh has it.  (Probing aligned pairs of slots by
//           8-byte reads: fewer turns of the loop, more instructions each; 10.6 ms per sweep instead of 10.1 at 738 M
//           tokens.)
// Both give (topic << count_bits) | n_kd.
template <bool DENSE>
struct TileTable {
    const uint32_t* tab;      // the document's counters, or its slots
    const uint32_t* tok;      // DENSE: topic of the document's j-th token; hashed: its slot
    uint32_t cap;             // hashed: slots
    int cb;
    __device__ __forceinline__ uint32_t counted(uint32_t k) const
    {
        return k << cb | reinterpret_cast<const uint16_t*>(tab)[k];
    }
    __device__ __forceinline__ uint32_t of_topic(uint32_t k) const
    {
        if (DENSE) return counted(k);
        const uint32_t e = dk_lookup(tab, cap, k, cb);
        return e ? e : k << cb;
    }
    // the j-th token's topic (copy), or topic j
    __device__ __forceinline__ uint32_t drawn(bool copy, uint32_t j) const
    {
        if (DENSE) return counted(copy ? tok[j] : j);
        // the slot to look at first is the token's or the topic's home: one read serves both
        uint32_t h = copy ? tok[j] : dk_home(j, cap);
        uint32_t e = tab[h];
        if (copy) return e;
        const uint32_t want = j << cb;
        for (uint32_t n = 0; n < cap; ++n) {
            if (e == DK_EMPTY) break;
            if ((e >> cb) == j) return e;
            if (++h == cap) h = 0;
            e = tab[h];
        }
        return want;
    }
};

// Adds one occurrence of topic k; returns what TileTable::tok keeps, or ~0 if there was no room.
template <bool DENSE>
__device__ __forceinline__ uint32_t tile_insert(uint32_t* tab, uint32_t cap, uint32_t k, int cb)
{
    if (DENSE) {
        atomicAdd(&tab[k >> 1], (k & 1u) ? 0x10000u : 1u);
        return k;
    }
    return dk_insert(tab, cap, k, cb);
}

// The table of a document longer than a tile, in device memory or staged: a counter per topic (DENSE) or hashed.
template <bool DENSE>
struct LongTable {
    const uint32_t* tab;
    const uint32_t* topic_of;  // topics of the document's tokens, in document order
    uint32_t cap;
    int cb;
    __device__ __forceinline__ uint32_t of_topic(uint32_t k) const
    {
        if (DENSE) return k << cb | tab[k];
        const uint32_t e = dk_lookup(tab, cap, k, cb);
        return e ? e : k << cb;
    }
    __device__ __forceinline__ uint32_t drawn(bool copy, uint32_t j) const { return of_topic(copy ? topic_of[j] : j); }
};

// Everything pass 3 needs from the document side for one token, written at the token's
// block-major index `bm`.
template <typename T, int MODE, int FIXED, class Table>
__device__ __forceinline__ void doc_side_token(const View& v, const Table& table, uint32_t tok, uint32_t doc_len,
                                               uint32_t own, uint32_t t_first, uint32_t bm,
                                               const PhiloxKey& key, uint32_t sweep, int32_t mh_steps)
{
    const T* prop = reinterpret_cast<const T*>(v.prop);
    const size_t N = (size_t)v.N;
    uint32_t* out = v.dside + (size_t)bm * v.side_stride;
    const double n_d = u32_to_double(doc_len);
    // The record's words come in order (step_record_at()).  With the step count fixed at compile time they are all
    // collected in registers; else four at a time, which then go out as one 16-byte store.
    constexpr int REGW = (FIXED > 0 && step_record_words<MODE>(FIXED) > 4) ? 8 : 4;
    static_assert(FIXED == 0 || step_record_words<MODE>(FIXED) <= 8, "the record is kept in eight registers");
    uint32_t wr[REGW];
#pragma unroll
    for (int q = 0; q < REGW; ++q) wr[q] = 0u;
    wr[0] = own;
    auto put = [&](int at, uint32_t val) {
        if (FIXED > 0) {
            wr[at] = val;  // the step loops are unrolled: `at` is a constant
        } else {
            const int q = at & 3;
            wr[0] = q == 0 ? val : wr[0];
            wr[1] = q == 1 ? val : wr[1];
            wr[2] = q == 2 ? val : wr[2];
            wr[3] = q == 3 ? val : wr[3];
            if (q == 3) __stcs(reinterpret_cast<uint4*>(out + at - 3), make_uint4(wr[0], wr[1], wr[2], wr[3]));
        }
    };
    // word-proposal of step st, the wi-th of its kind: n_kd at the topic pass 1 drew
    auto word_step = [&](int32_t st, int32_t wi) {
        const uint32_t t1 = wi == 0 ? t_first : (uint32_t)__ldcg(prop + (size_t)wi * N + bm);
        put(step_record_at<MODE>(st), table.of_topic(t1));
    };
    // doc-proposal of step st
    auto doc_step = [&](int32_t st) {
        const uint4 at = make_uint4(v.tok_base + tok, sweep, (uint32_t)st, 0u);
        const uint4 r = FIXED > 0 ? philox4x32_10(at, key) : philox4x32_10(at, PhiloxSeed(key));
        const bool copy = __dmul_rn(__dmul_rn(u32_to_double(r.x), INV_2_32), __dadd_rn(n_d, v.Kalpha)) < n_d;
        const uint32_t o2 = table.drawn(copy, scale_to_range(r.y, copy ? doc_len : (uint32_t)v.K));
        put(step_record_at<MODE>(st), o2);
        put(step_record_at<MODE>(st) + 1, r.w);  // the step's acceptance uniform
    };
    if (MODE == LDA_PROPOSALS_CYCLE) {
#pragma unroll
        for (int32_t st = 0; st < mh_steps; st += 2) {
            word_step(st, st >> 1);
            if (st + 1 < mh_steps) doc_step(st + 1);
        }
    } else if (MODE == LDA_PROPOSALS_WORD) {
#pragma unroll
        for (int32_t st = 0; st < mh_steps; ++st) word_step(st, st);
    } else {
#pragma unroll
        for (int32_t st = 0; st < mh_steps; ++st) doc_step(st);
    }
    if (FIXED == 0) {
        const int words = step_record_words<MODE>(mh_steps);
        if (words & 3) __stcs(reinterpret_cast<uint4*>(out + (words & ~3)), make_uint4(wr[0], wr[1], wr[2], wr[3]));
        return;
    }
    if (REGW == 8) {
        store_32(out, make_uint4(wr[0], wr[1], wr[2], wr[3]), make_uint4(wr[4], wr[5], wr[6], wr[7]));
    } else {
        __stcs(reinterpret_cast<uint4*>(out), make_uint4(wr[0], wr[1], wr[2], wr[3]));
    }
}

// array[first, first + count) of n elements towards L2, in the 16-byte units that hold it.
template <typename E>
__device__ __forceinline__ void prefetch_l2(const E* array, int64_t first, int32_t count, int32_t n)
{
    constexpr int64_t UNIT = 16 / sizeof(E);
    const int64_t a = first & ~(UNIT - 1), b = min((first + count + UNIT - 1) & ~(UNIT - 1), (int64_t)n & ~(UNIT - 1));
    if (a < b)
        asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(array + a), "r"((uint32_t)((b - a) * sizeof(E))) : "memory");
}
template <typename T>
using PairWord = std::conditional_t<sizeof(T) == 2, uint32_t, uint2>;
constexpr int64_t PREFETCH_AHEAD = 1 << 20;

// `cap` = tokens a tile can hold (the shared-memory carve-up) = DOC_TILE_ROUNDS x blockDim.x: a
// thread owns at most DOC_TILE_ROUNDS tokens and keeps what it read about them in registers across
// the phases.  Small tiles keep many CTAs per SM, which is what hides the gathers of the first phase.
// FIXED > 0: the number of steps is this compile-time constant (the argument is ignored).
// Threads the compiler must leave room for per SM: the two-step kernels with a word step need few
// enough registers to fill the SM (16 CTAs of 128 threads), the others three quarters of it.
__host__ __device__ constexpr int doc_resident_threads(int mode, int fixed)
{
    return (fixed == 2 && mode != LDA_PROPOSALS_DOC) ? 2048 : 1536;
}
// Slots per token of the hashed tables.  More of them mean shorter searches, but what shared memory takes L1 lacks, and its lines
// are what the gathers in flight wait in: with 16 CTAs per SM five slots take 10.5 ms and six 13.4 instead of 9.72 (738 M
// tokens, K = 10 000, two steps); with the twelve of the other forms with a fixed step count six are ahead (74 M, four steps:
// 1.509 -> 1.447 ms; doc-proposals alone, two steps, 16 M, K = 3000 and 12 000, documents of 40 and 700: 0.319 -> 0.263 ms,
// 0.330 -> 0.271).  Loops over any number of steps wait for other things, and lose by six: 24 M, V = 10^6, K = 10^5, four steps of
// word-proposals 0.805 ms with four slots, 0.834 with six, of doc-proposals 1.121 and 1.139.  `few_tiles`: a multiprocessor has so
// few that L1 is no matter; with word-proposals six are ahead (65 000 tokens, K = 1812, eight steps of them: 15.2 us with four,
// 14.4 with six; of the cycle: 12.5 and 12.3; without: 7.6 and 7.8).  As a parameter of the kernel the number costs more than that.
__host__ __device__ constexpr int tile_slots(int mode, int fixed, bool dense, bool few_tiles)
{
    if (dense || doc_resident_threads(mode, fixed) == 2048) return DOC_TILE_SLOTS;
    return fixed > 0 || (few_tiles && mode != LDA_PROPOSALS_DOC) ? DOC_TILE_SLOTS_MOST : DOC_TILE_SLOTS;
}
constexpr int64_t FEW_TILES_TOKENS = (int64_t)1 << 21;
template <typename T, int THREADS, int MODE, int FIXED, bool DENSE, int SLOTS>
__global__ void __launch_bounds__(THREADS, doc_resident_threads(MODE, FIXED) / THREADS)
k_doc_tile(View v, const int32_t* __restrict__ tiles, PhiloxKey key, int32_t mh_steps_arg)
{
    stamp(v, STAMP_DOC_TILES);
    const int32_t mh_steps = FIXED > 0 ? FIXED : mh_steps_arg;
    constexpr int cap = DOC_TILE_ROUNDS * THREADS;
    extern __shared__ __align__(16) uint32_t doc_smem[];
    uint32_t* area = doc_smem;                                           // [SLOTS * cap] the tile's tables
    int32_t* soff = reinterpret_cast<int32_t*>(area + SLOTS * cap);  // [cap + 1] document offsets
    uint32_t* tok_s = reinterpret_cast<uint32_t*>(soff + cap + 1);        // [cap] see TileTable::tok
    const int tid = threadIdx.x;
    const int32_t s0 = tiles[2 * blockIdx.x], s1 = tiles[2 * blockIdx.x + 1];
    const int32_t nseg = s1 - s0;
    const int32_t base = v.doc_off[s0];
    const int32_t cnt = v.doc_off[s1] - base;
    if (cnt == 0) return;
    const int32_t half_k = DENSE ? (v.K + 1) >> 1 : 0;  // words of a document's counters
    const T* zbm = reinterpret_cast<const T*>(v.zbm);
    // One thread asks for what later tiles read first: the index of the tokens PREFETCH_AHEAD further on, which is more than the
    // tiles in flight hold, and the same stretch of the next block's topic pairs (a block's pairs are read all over its
    // tokens).  A warp's gather is as slow as its slowest read: 738 M tokens, K = 10 000: 9.81 -> 9.71 ms; 99 M, K = 1000:
    // 1.058 -> 1.038.
    if (tid == THREADS - 32) {
        prefetch_l2(v.bm_of_tok, (int64_t)base + PREFETCH_AHEAD, cnt, v.N);
        prefetch_l2(reinterpret_cast<const PairWord<T>*>(v.zbm), (int64_t)base + ((int64_t)1 << v.block_shift), cnt, v.N);
    }
    uint32_t bm[DOC_TILE_ROUNDS], z[DOC_TILE_ROUNDS], t1[DOC_TILE_ROUNDS];
#pragma unroll
    for (int r = 0; r < DOC_TILE_ROUNDS; ++r) {
        const int j = tid + r * THREADS;
        bm[r] = z[r] = t1[r] = 0;
        if (j < cnt) {
            bm[r] = __ldcs(v.bm_of_tok + base + j);
            load_topic_pair(zbm, bm[r], z[r], t1[r]);
        }
    }
    uint32_t doc[DOC_TILE_ROUNDS];  // first token of the token's document | its length << 16: every register counts here
    for (int j = tid; j <= nseg; j += THREADS) soff[j] = v.doc_off[s0 + j] - base;
    const uint32_t none = DENSE ? 0u : DK_EMPTY;
    const int quads = DENSE ? (nseg * half_k + 3) >> 2 : (cnt * SLOTS + 3) >> 2;
    for (int j = tid; j < quads; j += THREADS) reinterpret_cast<uint4*>(area)[j] = make_uint4(none, none, none, none);
    __syncthreads();
    // every token finds its document and adds itself to the document's table
#pragma unroll
    for (int r = 0; r < DOC_TILE_ROUNDS; ++r) {
        const int j = tid + r * THREADS;
        doc[r] = 0;
        if (j < cnt) {
            int lo = 0, hi = nseg;  // last document with soff[doc] <= j
            while (hi - lo > 1) {
                const int mid = (lo + hi) >> 1;
                if (soff[mid] <= j) lo = mid; else hi = mid;
            }
            const int32_t f = soff[lo], n = soff[lo + 1] - f;
            doc[r] = (uint32_t)n << 16 | (uint32_t)f;
            uint32_t at = 0xFFFFFFFFu;
            if (z[r] < (uint32_t)v.K)
                at = tile_insert<DENSE>(area + (DENSE ? lo * half_k : SLOTS * f), SLOTS * (uint32_t)n, z[r], v.count_bits);
            if (at == 0xFFFFFFFFu) {
                atomicOr(v.err, z[r] < (uint32_t)v.K ? ERR_ROW_OVERFLOW : ERR_TOPIC_RANGE);
                at = 0;
            }
            tok_s[j] = at;
            z[r] = DENSE ? (uint32_t)lo << 16 | at : at;  // from here on: the slot, or the topic with its document
        }
    }
    __syncthreads();
    // the tables are complete: every token gathers its share
    const uint32_t sweep = running_sweep(v);
#pragma unroll
    for (int r = 0; r < DOC_TILE_ROUNDS; ++r) {
        const int j = tid + r * THREADS;
        if (j < cnt) {
            const uint32_t f = doc[r] & 0xFFFFu, n = doc[r] >> 16;
            const TileTable<DENSE> table{area + (DENSE ? (z[r] >> 16) * half_k : SLOTS * f), tok_s + f, SLOTS * n, v.count_bits};
            const uint32_t own = DENSE ? table.counted(z[r] & 0xFFFFu) : table.tab[z[r]];
            doc_side_token<T, MODE, FIXED>(v, table, (uint32_t)(base + j), n, own, t1[r], bm[r], key, sweep, mh_steps);
        }
    }
}

// Documents longer than a tile are cut into chunks of LONG_CHUNK tokens, a CTA each, in two kernels: the first
// adds the chunk's topics to the document's table in device memory (cleared before) and leaves them in document order, the
// second gathers the tokens' records.  A table is a counter per topic where that takes no more room than
// hashing, else hashed like a tile's; counters of up to LONG_STAGE_MAX_K topics go through shared memory.
// (One CTA per document, as the tiles have it, lasts as long as the longest document: 12 M tokens in
// 3000 documents of log-normal length, K = 777, took 523 us per sweep, the two kernels take 230.)
template <typename T, bool DENSE>
__device__ __forceinline__ void long_count(const View& v, uint32_t* tab, uint32_t cap, int32_t first, int32_t cnt, uint32_t* bins,
                                           bool keep_topics)
{
    const T* zbm = reinterpret_cast<const T*>(v.zbm);
    const bool staged = DENSE && v.K <= LONG_STAGE_MAX_K;
    if (staged) {
        for (int32_t k = threadIdx.x; k < v.K; k += LONG_THREADS) bins[k] = 0;
        __syncthreads();
    }
    for (int32_t j0 = threadIdx.x; j0 < cnt; j0 += LONG_AT_ONCE * LONG_THREADS) {
        uint32_t k[LONG_AT_ONCE];
#pragma unroll
        for (int u = 0; u < LONG_AT_ONCE; ++u) {
            const int32_t j = j0 + u * LONG_THREADS;
            k[u] = j < cnt ? __ldcs(v.bm_of_tok + first + j) : 0u;
        }
#pragma unroll
        for (int u = 0; u < LONG_AT_ONCE; ++u) k[u] = j0 + u * LONG_THREADS < cnt ? (uint32_t)__ldcg(zbm + 2 * (size_t)k[u]) : 0u;
#pragma unroll
        for (int u = 0; u < LONG_AT_ONCE; ++u) {
            const int32_t j = j0 + u * LONG_THREADS;
            if (j >= cnt) continue;
            if (keep_topics) v.rec[first + j] = min(k[u], (uint32_t)v.K - 1u);
            if (k[u] >= (uint32_t)v.K) {
                atomicOr(v.err, ERR_TOPIC_RANGE);
            } else if (staged) {
                atomicAdd(&bins[k[u]], 1u);
            } else if (DENSE) {
                atomicAdd(&tab[k[u]], 1u);
            } else if (dk_insert(tab, cap, k[u], v.count_bits) == 0xFFFFFFFFu) {
                atomicOr(v.err, ERR_ROW_OVERFLOW);
            }
        }
    }
    if (staged) {
        __syncthreads();
        for (int32_t k = threadIdx.x; k < v.K; k += LONG_THREADS) {
            const uint32_t n = bins[k];
            if (n) atomicAdd(&tab[k], n);
        }
    }
}

template <typename T>
__global__ void __launch_bounds__(LONG_THREADS)
k_long_count(View v, const int4* __restrict__ chunks, bool keep_topics, int stamp_id)
{
    stamp(v, stamp_id);
    extern __shared__ __align__(16) uint32_t long_bins[];
    const int4 c = __ldg(chunks + blockIdx.x);
    const LongDoc d = v.long_docs[c.x];
    uint32_t* tab = v.dk_slots + d.slot;
    if (d.dense) long_count<T, true>(v, tab, 0u, c.y, c.z, long_bins, keep_topics);
    else long_count<T, false>(v, tab, DK_SLOTS_PER_TOKEN * (uint32_t)d.len, c.y, c.z, long_bins, keep_topics);
}

template <typename T, int MODE, int FIXED, bool DENSE>
__device__ __forceinline__ void long_gather(const View& v, const LongDoc& d, const uint32_t* tab, int32_t first, int32_t cnt,
                                            const PhiloxKey& key, int32_t mh_steps)
{
    const T* zbm = reinterpret_cast<const T*>(v.zbm);
    const uint32_t sweep = running_sweep(v);
    const LongTable<DENSE> table{tab, v.rec + d.first, DK_SLOTS_PER_TOKEN * (uint32_t)d.len, v.count_bits};
    for (int32_t j0 = threadIdx.x; j0 < cnt; j0 += LONG_AT_ONCE * LONG_THREADS) {
        uint32_t bm[LONG_AT_ONCE], z[LONG_AT_ONCE], t1[LONG_AT_ONCE];
#pragma unroll
        for (int u = 0; u < LONG_AT_ONCE; ++u) {
            const int32_t j = j0 + u * LONG_THREADS;
            bm[u] = z[u] = t1[u] = 0;
            if (j < cnt) bm[u] = __ldcs(v.bm_of_tok + first + j);
        }
#pragma unroll
        for (int u = 0; u < LONG_AT_ONCE; ++u)
            if (j0 + u * LONG_THREADS < cnt) load_topic_pair(zbm, bm[u], z[u], t1[u]);
#pragma unroll
        for (int u = 0; u < LONG_AT_ONCE; ++u) {
            const int32_t j = j0 + u * LONG_THREADS;
            if (j < cnt)
                doc_side_token<T, MODE, FIXED>(v, table, (uint32_t)(first + j), (uint32_t)d.len, table.of_topic(z[u]), t1[u], bm[u], key,
                                               sweep, mh_steps);
        }
    }
}

template <typename T, int MODE, int FIXED>
__global__ void __launch_bounds__(LONG_THREADS, LONG_MIN_CTAS)
k_long_gather(View v, const int4* __restrict__ chunks, PhiloxKey key, int32_t mh_steps_arg)
{
    const int32_t mh_steps = FIXED > 0 ? FIXED : mh_steps_arg;
    extern __shared__ __align__(16) uint32_t long_bins[];
    const int4 c = __ldg(chunks + blockIdx.x);
    const LongDoc d = v.long_docs[c.x];
    const uint32_t* tab = v.dk_slots + d.slot;
    if (!d.dense) {
        long_gather<T, MODE, FIXED, false>(v, d, tab, c.y, c.z, key, mh_steps);
        return;
    }
    if (v.K <= LONG_STAGE_MAX_K) {
        for (int32_t k = threadIdx.x; k < v.K; k += LONG_THREADS) long_bins[k] = __ldcg(tab + k);
        __syncthreads();
        tab = long_bins;
    }
    long_gather<T, MODE, FIXED, true>(v, d, tab, c.y, c.z, key, mh_steps);
}

static size_t long_smem_bytes(const Ctx& c) { return c.K <= LONG_STAGE_MAX_K ? (size_t)c.K * 4 : 0; }

// Tables of the documents longer than a tile; keep_topics: and their topics in document order in View::rec
// (which an export in flight may be reading).
int launch_long_tables(Ctx& c, cudaStream_t stream, bool keep_topics, int stamp_id)
{
    if (!c.n_long_chunks) return 0;
    if (c.long_hashed_slots) cudaMemsetAsync(c.v.dk_slots, 0xFF, (size_t)c.long_hashed_slots * 4, stream);
    if (c.long_slots > c.long_hashed_slots)
        cudaMemsetAsync(c.v.dk_slots + c.long_hashed_slots, 0, (size_t)(c.long_slots - c.long_hashed_slots) * 4, stream);
    const int4* chunks = reinterpret_cast<const int4*>(c.long_chunks);
    if (c.wide_topics)
        k_long_count<int32_t><<<c.n_long_chunks, LONG_THREADS, long_smem_bytes(c), stream>>>(c.v, chunks, keep_topics, stamp_id);
    else
        k_long_count<uint16_t><<<c.n_long_chunks, LONG_THREADS, long_smem_bytes(c), stream>>>(c.v, chunks, keep_topics, stamp_id);
    return 1;
}

size_t doc_tile_smem_bytes(int tile_tokens, int slots) { return (size_t)tile_tokens * (4 * slots + 4 + 4) + 16; }

// (A limit that is set loads the kernel: only for what needs more than the 48 KB that every kernel has.)
template <typename T, int MODE, int FIXED, bool DENSE, int SLOTS>
static void set_tile_limit()
{
    constexpr auto most = cudaFuncAttributeMaxDynamicSharedMemorySize;
    if constexpr (SLOTS > DOC_TILE_SLOTS)
        cudaFuncSetAttribute(k_doc_tile<T, 512, MODE, FIXED, DENSE, SLOTS>, most, (int)doc_tile_smem_bytes(DOC_TILE_ROUNDS * 512, SLOTS));
    static_assert(DOC_TILE_ROUNDS * 512 * (4 * DOC_TILE_SLOTS + 8) + 16 <= 48 << 10, "tiles of 512 threads with the fewest slots");
    cudaFuncSetAttribute(k_doc_tile<T, 1024, MODE, FIXED, DENSE, SLOTS>, most, (int)doc_tile_smem_bytes(DOC_TILE_MAX, SLOTS));
}

template <typename T, int MODE, int FIXED>
static void set_doc_limit()
{
    constexpr int many = tile_slots(MODE, FIXED, false, false), few = tile_slots(MODE, FIXED, false, true);
    set_tile_limit<T, MODE, FIXED, false, many>();
    if constexpr (few != many) set_tile_limit<T, MODE, FIXED, false, few>();
    if constexpr (sizeof(T) == 2) set_tile_limit<T, MODE, FIXED, true, tile_slots(MODE, FIXED, true, false)>();
}

void set_doc_smem_limits()
{
    set_doc_limit<uint16_t, LDA_PROPOSALS_CYCLE, 0>();
    set_doc_limit<uint16_t, LDA_PROPOSALS_CYCLE, 2>();
    set_doc_limit<uint16_t, LDA_PROPOSALS_CYCLE, 4>();
    set_doc_limit<uint16_t, LDA_PROPOSALS_WORD, 0>();
    set_doc_limit<uint16_t, LDA_PROPOSALS_WORD, 2>();
    set_doc_limit<uint16_t, LDA_PROPOSALS_DOC, 0>();
    set_doc_limit<uint16_t, LDA_PROPOSALS_DOC, 2>();
    set_doc_limit<int32_t, LDA_PROPOSALS_CYCLE, 0>();
    set_doc_limit<int32_t, LDA_PROPOSALS_CYCLE, 2>();
    set_doc_limit<int32_t, LDA_PROPOSALS_CYCLE, 4>();
    set_doc_limit<int32_t, LDA_PROPOSALS_WORD, 0>();
    set_doc_limit<int32_t, LDA_PROPOSALS_WORD, 2>();
    set_doc_limit<int32_t, LDA_PROPOSALS_DOC, 0>();
    set_doc_limit<int32_t, LDA_PROPOSALS_DOC, 2>();
}

template <typename T, int MODE, int FIXED>
static int doc_side_tm(Ctx& c, int mh_steps)
{
    const PhiloxKey key(c.seed);
    const PassStreams on(c, (c.n_doc_tiles > 0) + (c.n_long_chunks > 0));
    int launches = 0;
    if (c.n_doc_tiles) {
        auto tiles = [&](auto dense, auto few) {
            constexpr bool DENSE = decltype(dense)::value;
            constexpr int SLOTS = tile_slots(MODE, FIXED, DENSE, decltype(few)::value);
            const size_t smem = doc_tile_smem_bytes(c.doc_tile, SLOTS);
            const auto kernel = c.doc_threads == 128   ? k_doc_tile<T, 128, MODE, FIXED, DENSE, SLOTS>
                                : c.doc_threads == 256 ? k_doc_tile<T, 256, MODE, FIXED, DENSE, SLOTS>
                                : c.doc_threads == 512 ? k_doc_tile<T, 512, MODE, FIXED, DENSE, SLOTS>
                                                       : k_doc_tile<T, 1024, MODE, FIXED, DENSE, SLOTS>;
            kernel<<<c.n_doc_tiles, c.doc_threads, smem, on[1]>>>(c.v, c.doc_tiles, key, mh_steps);
        };
        if (c.doc_dense) tiles(std::integral_constant<bool, sizeof(T) == 2>{}, std::false_type{});  // never with 32-bit topics
        else if (c.N <= FEW_TILES_TOKENS) tiles(std::false_type{}, std::true_type{});
        else tiles(std::false_type{}, std::false_type{});
        ++launches;
    }
    if (c.n_long_chunks) {
        launches += launch_long_tables(c, on[0], true, STAMP_DOC_LONG);
        k_long_gather<T, MODE, FIXED><<<c.n_long_chunks, LONG_THREADS, long_smem_bytes(c), on[0]>>>(
            c.v, reinterpret_cast<const int4*>(c.long_chunks), key, mh_steps);
        ++launches;
    }
    return launches;
}

template <typename T>
static int doc_side_t(Ctx& c, int mh_steps)
{
    switch (c.proposals) {
        // chains of two steps (and the cycle with four) have kernels of their own
        case LDA_PROPOSALS_WORD:
            return mh_steps == 2 ? doc_side_tm<T, LDA_PROPOSALS_WORD, 2>(c, mh_steps)
                                 : doc_side_tm<T, LDA_PROPOSALS_WORD, 0>(c, mh_steps);
        case LDA_PROPOSALS_DOC:
            return mh_steps == 2 ? doc_side_tm<T, LDA_PROPOSALS_DOC, 2>(c, mh_steps)
                                 : doc_side_tm<T, LDA_PROPOSALS_DOC, 0>(c, mh_steps);
        default:
            return mh_steps == 2   ? doc_side_tm<T, LDA_PROPOSALS_CYCLE, 2>(c, mh_steps)
                   : mh_steps == 4 ? doc_side_tm<T, LDA_PROPOSALS_CYCLE, 4>(c, mh_steps)
                                   : doc_side_tm<T, LDA_PROPOSALS_CYCLE, 0>(c, mh_steps);
    }
}

int launch_doc_side(Ctx& c, int mh_steps)
{
    if (c.N == 0) return 0;
    return c.wide_topics ? doc_side_t<int32_t>(c, mh_steps) : doc_side_t<uint16_t>(c, mh_steps);
}

}  // namespace lda
