// Count-table rebuild from the assignments (Section 3: n_kw, n_k; Eq. 12: n_kd).
//
// n_kw (segments = words over the word-sorted z): per word, the sorted list of
// (topic, count).  Two paths, chosen per word at load time:
//   - tail words: whole words are packed into tiles of <= SORT_TILE tokens; the
//     warps of a CTA count each word's topics in shared-memory hash tables and read them
//     back in topic order through a bitmap over the topics (K <= 16384), or the CTA sorts
//     the tile's (word, topic) keys (larger K);
//   - hot words: shared-memory histogram over a window of topics, written out as
//     dense row and sorted row.
// n_k: column sums, added up by the kernels that write the rows when K and the number of CTAs are small
// enough for that (choose_nk_mode()), else taken from the rows just written.
// n_kd (segments = documents): the MH step builds every document's table itself, per tile, in
// shared memory (docside.cu), and so does the log-likelihood (loglik.cu); lda_get_counts gets
// sorted rows from export.cu.
// No per-token global atomics: a CTA touches global counters once per bin it
// actually filled (documents longer than a tile are the one exception).
#include <algorithm>

#include "lda_device.cuh"
#include "lda_internal.cuh"
#include "tile_sort.cuh"

namespace lda {

static_assert(SORT_TILE == SORT_THREADS * SORT_PER, "tiles of documents and of tail words are as large as what is sorted at once");

struct EmitWord {
    const int32_t* row_start;
    uint32_t* topic;
    uint32_t* count;
    int32_t* nnz;
    int32_t* nk;  // null: n_k is not added up here
    __device__ __forceinline__ void entry(int32_t seg, int32_t rank, uint32_t k, uint32_t n) const
    {
        const int32_t slot = row_start[seg] + rank;
        topic[slot] = k;
        count[slot] = n;
        if (nk) atomicAdd(&nk[k], (int32_t)n);
    }
    __device__ __forceinline__ void rows(int32_t seg, int32_t n) const { nnz[seg] = n; }
};

// Tail words when K is large (the bitmap of k_word_rows would cost more than the sort): one CTA per
// tile of whole words [s0, s1) holding <= SORT_TILE tokens and <= SORT_TILE words sorts the tile's
// (word, topic) keys (tile_sort.cuh) and run-length encodes them.
template <typename T, class Emit>
__global__ void __launch_bounds__(256)
k_seg_count_sorted(const int32_t* __restrict__ tiles, const int32_t* __restrict__ seg_off,
                   const T* __restrict__ z, int topic_bits, int32_t K, Emit emit, SweepState* state, int stamp_id)
{
    stamp(state, stamp_id);
    int* const err = &state->err;
    __shared__ __align__(16) uint32_t keys[SORT_TILE];
    __shared__ int32_t soff[SORT_TILE + 1];
    __shared__ int32_t hidx[SORT_TILE + 1];
    __shared__ int32_t headpos[SORT_TILE + 1];
    __shared__ int32_t scan_tmp[33];

    const int tid = threadIdx.x;
    const int32_t s0 = tiles[2 * blockIdx.x], s1 = tiles[2 * blockIdx.x + 1];
    const int32_t nseg = s1 - s0;
    const int32_t base = seg_off[s0];
    const int32_t cnt = seg_off[s1] - base;
    for (int j = tid; j <= nseg; j += blockDim.x) soff[j] = seg_off[s0 + j] - base;
    __syncthreads();
    if (cnt == 0) {
        for (int j = tid; j < nseg; j += blockDim.x) emit.rows(s0 + j, 0);
        return;
    }
    uint32_t x[SORT_PER];
    if (!tile_keys(x, keys, soff, nseg, z + base, cnt, topic_bits, K)) atomicOr(err, ERR_TOPIC_RANGE);
    sort_tile(x, keys, cnt);
    // head flags -> exclusive scan
    uint32_t flags = 0;
#pragma unroll
    for (int q = 0; q < SORT_PER; ++q) {
        const int j = tid * SORT_PER + q;
        const uint32_t before = q > 0 ? x[q - 1] : j > 0 ? keys[j - 1] : ~x[0];
        if (j < cnt && x[q] != before) flags |= 1u << q;
    }
    int32_t total;
    int32_t run = block_scan_excl<int32_t>(__popc(flags), scan_tmp, total);
#pragma unroll
    for (int q = 0; q < SORT_PER; ++q) {
        const int j = tid * SORT_PER + q;
        if (j < cnt) {
            hidx[j] = run;
            if (flags >> q & 1u) headpos[run++] = j;
        }
    }
    if (tid == 0) { hidx[cnt] = total; headpos[total] = cnt; }
    __syncthreads();
    const uint32_t kmask = (1u << topic_bits) - 1u;
    for (int h = tid; h < total; h += blockDim.x) {
        const int j = headpos[h];
        const uint32_t key = keys[j];
        const int32_t seg = (int32_t)(key >> topic_bits);
        const int32_t rank = h - hidx[soff[seg]];
        emit.entry(s0 + seg, rank, key & kmask, (uint32_t)(headpos[h + 1] - j));
    }
    for (int j = tid; j < nseg; j += blockDim.x) emit.rows(s0 + j, hidx[soff[j + 1]] - hidx[soff[j]]);
}

// Tail words (K <= WORD_ROWS_BITMAP_MAX_K): one CTA per tile of whole words [s0, s1) holding at most
// SORT_TILE tokens and ROW_TILE_WORDS words.  The tile's topics are read once, into shared memory; words of
// up to ROW_WARP_TOKENS are then handed to the CTA's warps a few at a time, without a barrier between them:
//   - up to 2 tokens (in a large vocabulary most words): a lane's work;
//   - up to 32 tokens: a lane holds a token, lanes with the same topic find each other, the lowest of
//     them writes the entry at the rank of its topic among the word's distinct topics;
//   - longer: counted in a hash table of the warp's own (load <= 1/2); the token that claims a topic's
//     slot marks the topic in a bitmap, and writes its entry once the bitmap's running popcounts tell the
//     topic's rank.
// Words longer than that take the whole CTA, one after the other, in the same way.
// What bounds it is latency (a word is a chain of a dozen dependent shared-memory steps): hence many words in
// flight per multiprocessor, little shared memory per CTA, and no CTA-wide steps for short words.
// NK: the tile's column sums go to n_k too (NkMode).
constexpr int ROW_WARP_TOKENS = 128;
constexpr int ROW_WARP_SLOTS = 2 * ROW_WARP_TOKENS;
constexpr int ROW_CTA_SLOTS = 2 * SORT_TILE;
constexpr int ROW_COUNT_BITS = 12;  // of a table entry: a tail word has at most SORT_TILE = 2048 tokens
static_assert(SORT_TILE < (1 << ROW_COUNT_BITS), "count bits");

// How the kernels that write rows add up n_k: not at all (a pass over the rows follows), through bins in shared
// memory with one global add per bin and CTA, or with one global add per row entry.  Which: choose_nk_mode().
enum NkMode { NK_NONE, NK_BINS, NK_DIRECT };

struct RowTables {
    const int32_t* row_start;
    uint32_t* topic;
    uint32_t* count;
    int32_t* nnz;
    int32_t* nk;  // column sums are added here (NK kernels)
    SweepState* state;
};

// Words of 32 bits of a bitmap over K topics such that each lane of a warp owns an odd number of them (no
// two lanes on the same shared-memory bank).
__host__ __device__ constexpr int row_bitmap_lane_words(int K) { return (((K + 31) / 32 + 31) / 32) | 1; }
// Bytes of a warp's (table, bitmap, running popcounts) times eight, or of the CTA's, whichever is more.
static size_t row_area_bytes(int K)
{
    const size_t bitmap = (size_t)row_bitmap_lane_words(K) * 32;
    const size_t warps = 8 * (ROW_WARP_SLOTS * 4 + bitmap * 6), cta = ROW_CTA_SLOTS * 4 + bitmap * 6;
    return ((warps > cta ? warps : cta) + 15) / 16 * 16;
}

// Counts one token of topic k in a table of 2^log2_slots slots (never full: load <= 1/2).  Returns the slot
// if this token claimed it, else ~0.
__device__ __forceinline__ uint32_t row_count(uint32_t* table, int log2_slots, uint32_t k)
{
    const uint32_t mask = (1u << log2_slots) - 1u, fresh = (k << ROW_COUNT_BITS) | 1u;
    uint32_t h = (k * DK_HASH_MULT) >> (32 - log2_slots);
    for (uint32_t tries = 0; tries <= mask; ++tries, h = (h + 1) & mask) {
        const uint32_t prev = atomicCAS(&table[h], DK_EMPTY, fresh);
        if (prev == DK_EMPTY) return h;
        if ((prev >> ROW_COUNT_BITS) == k) {
            atomicAdd(&table[h], 1u);
            break;
        }
    }
    return 0xFFFFFFFFu;
}

template <NkMode NK>
__global__ void __launch_bounds__(256, 6)
k_word_rows(const int32_t* __restrict__ tiles, const int32_t* __restrict__ word_off, const uint16_t* __restrict__ z,
            RowTables out, int32_t K, int32_t area_words, int stamp_id)
{
    stamp(out.state, stamp_id);
    extern __shared__ __align__(16) uint32_t row_area[];  // the warps' tables and bitmaps, then the CTA's; NK: bins behind
    __shared__ int32_t soff[ROW_TILE_WORDS + 1];
    __shared__ uint16_t zs[SORT_TILE];
    __shared__ uint16_t long_words[SORT_TILE / ROW_WARP_TOKENS];
    __shared__ int32_t warp_total[8];
    __shared__ int32_t next_word, n_long;
    int* const err = &out.state->err;
    int32_t* bins = reinterpret_cast<int32_t*>(row_area + area_words);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int32_t s0 = tiles[2 * blockIdx.x], nw = tiles[2 * blockIdx.x + 1] - s0;
    const int32_t base = __ldg(word_off + s0), cnt = __ldg(word_off + s0 + nw) - base;
    if (tid == 0) {
        next_word = 0;
        n_long = 0;
    }
    for (int32_t j = tid; j <= nw; j += 256) soff[j] = __ldg(word_off + s0 + j) - base;
    for (int32_t j = tid; j < cnt; j += 256) {
        const uint16_t k = __ldcs(z + base + j);
        if ((uint32_t)k >= (uint32_t)K) atomicOr(err, ERR_TOPIC_RANGE);
        zs[j] = (uint32_t)k < (uint32_t)K ? k : (uint16_t)0;
    }
    if (NK == NK_BINS)
        for (int32_t k = tid; k < K; k += 256) bins[k] = 0;
    __syncthreads();
    auto emit = [&](int32_t at, uint32_t k, uint32_t n) {
        out.topic[at] = k;
        out.count[at] = n;
        if (NK == NK_BINS) atomicAdd(&bins[k], (int32_t)n);
        if (NK == NK_DIRECT) atomicAdd(&out.nk[k], (int32_t)n);
    };
    const int32_t lane_words = row_bitmap_lane_words(K);
    const uint4 empty = make_uint4(DK_EMPTY, DK_EMPTY, DK_EMPTY, DK_EMPTY), zero = make_uint4(0u, 0u, 0u, 0u);
    {
        uint32_t* table = row_area + warp * ROW_WARP_SLOTS;
        uint32_t* bitmap = row_area + 8 * ROW_WARP_SLOTS + warp * 32 * lane_words;
        uint16_t* before = reinterpret_cast<uint16_t*>(row_area + 8 * ROW_WARP_SLOTS + 8 * 32 * lane_words) + warp * 32 * lane_words;
        const int32_t batch = min(32, max(1, nw >> 4));
        int32_t wb = 0;
        uint32_t todo = 0;  // words of the batch that are left for the whole warp
        for (;;) {
            if (!todo) {
                if (lane == 0) wb = atomicAdd(&next_word, batch);
                wb = __shfl_sync(0xFFFFFFFFu, wb, 0);
                if (wb >= nw) break;
                const int32_t w = wb + lane;
                const bool mine = lane < batch && w < nw;
                const int32_t first = mine ? soff[w] : 0, n = mine ? soff[w + 1] - first : 0;
                if (mine && n <= 2) {
                    const uint32_t a = n > 0 ? (uint32_t)zs[first] : 0u, b = n > 1 ? (uint32_t)zs[first + 1] : a;
                    if (n > 0) {
                        const int32_t out0 = __ldg(out.row_start + s0 + w);
                        emit(out0, min(a, b), a == b ? (uint32_t)n : 1u);
                        if (a != b) emit(out0 + 1, max(a, b), 1u);
                    }
                    out.nnz[s0 + w] = n == 0 ? 0 : a == b ? 1 : 2;
                }
                todo = __ballot_sync(0xFFFFFFFFu, n > 2);
                continue;
            }
            const int32_t w = wb + __ffs((int)todo) - 1;
            todo &= todo - 1u;
            const int32_t first = soff[w], n = soff[w + 1] - first;
            const int32_t out0 = __ldg(out.row_start + s0 + w);
            if (n <= 32) {
                const uint32_t k = lane < n ? (uint32_t)zs[first + lane] : 0xFFFFFFFFu;
                const uint32_t same = __match_any_sync(0xFFFFFFFFu, k);
                const bool lead = lane < n && (uint32_t)(__ffs((int)same) - 1) == (uint32_t)lane;
                const uint32_t leaders = __ballot_sync(0xFFFFFFFFu, lead);
                int32_t rank = 0;
                for (uint32_t m = leaders; m; m &= m - 1u) {
                    const uint32_t other = __shfl_sync(0xFFFFFFFFu, k, __ffs((int)m) - 1);
                    rank += other < k ? 1 : 0;
                }
                if (lead) emit(out0 + rank, k, (uint32_t)__popc(same));
                if (lane == 0) out.nnz[s0 + w] = __popc(leaders);
            } else if (n <= ROW_WARP_TOKENS) {
                const int log2_slots = n <= 64 ? 7 : 8;
                static_assert(ROW_WARP_SLOTS == 256, "table sizes above");
                for (uint32_t i = lane; i < (1u << log2_slots) / 4; i += 32) reinterpret_cast<uint4*>(table)[i] = empty;
                for (int32_t i = lane; i < 8 * lane_words; i += 32) reinterpret_cast<uint4*>(bitmap)[i] = zero;
                __syncwarp();
                uint32_t slot[ROW_WARP_TOKENS / 32], topic[ROW_WARP_TOKENS / 32];
#pragma unroll
                for (int r = 0; r < ROW_WARP_TOKENS / 32; ++r) {
                    const int32_t j = lane + 32 * r;
                    slot[r] = 0xFFFFFFFFu;
                    topic[r] = 0;
                    if (j < n) {
                        topic[r] = (uint32_t)zs[first + j];
                        slot[r] = row_count(table, log2_slots, topic[r]);
                        if (slot[r] != 0xFFFFFFFFu) atomicOr(&bitmap[topic[r] >> 5], 1u << (topic[r] & 31u));
                    }
                }
                __syncwarp();
                int32_t c = 0;
                for (int32_t i = lane * lane_words; i < (lane + 1) * lane_words; ++i) {
                    before[i] = (uint16_t)c;
                    c += __popc(bitmap[i]);
                }
                const int32_t incl = warp_scan_incl<int32_t>(c);
                for (int32_t i = lane * lane_words; i < (lane + 1) * lane_words; ++i) before[i] += (uint16_t)(incl - c);
                __syncwarp();
#pragma unroll
                for (int r = 0; r < ROW_WARP_TOKENS / 32; ++r) {
                    if (slot[r] == 0xFFFFFFFFu) continue;
                    const uint32_t k = topic[r], below = (1u << (k & 31u)) - 1u;
                    emit(out0 + (int32_t)before[k >> 5] + __popc(bitmap[k >> 5] & below), k,
                         table[slot[r]] & ((1u << ROW_COUNT_BITS) - 1u));
                }
                if (lane == 31) out.nnz[s0 + w] = incl;
                __syncwarp();
            } else if (lane == 0) {
                long_words[atomicAdd(&n_long, 1)] = (uint16_t)w;  // at most SORT_TILE / ROW_WARP_TOKENS of them
            }
        }
    }
    __syncthreads();
    uint32_t* table = row_area;
    uint32_t* bitmap = row_area + ROW_CTA_SLOTS;
    uint16_t* before = reinterpret_cast<uint16_t*>(bitmap + 32 * lane_words);
    const int32_t per = (32 * lane_words + 255) / 256;  // bitmap words per thread
    for (int32_t q = 0; q < n_long; ++q) {
        const int32_t w = long_words[q], first = soff[w], n = soff[w + 1] - first;
        const int32_t out0 = __ldg(out.row_start + s0 + w);
        const int log2_slots = 33 - __clz(n - 1);  // at least 2 n slots
        for (uint32_t i = tid; i < (1u << log2_slots) / 4; i += 256) reinterpret_cast<uint4*>(table)[i] = empty;
        for (int32_t i = tid; i < 8 * lane_words; i += 256) reinterpret_cast<uint4*>(bitmap)[i] = zero;
        __syncthreads();
        uint32_t slot[SORT_TILE / 256];
#pragma unroll
        for (int r = 0; r < SORT_TILE / 256; ++r) {
            const int32_t j = tid + 256 * r;
            slot[r] = 0xFFFFFFFFu;
            if (j < n) {
                const uint32_t k = (uint32_t)zs[first + j];
                slot[r] = row_count(table, log2_slots, k);
                if (slot[r] != 0xFFFFFFFFu) atomicOr(&bitmap[k >> 5], 1u << (k & 31u));
            }
        }
        __syncthreads();
        const int32_t i0 = min(32 * lane_words, tid * per), i1 = min(32 * lane_words, i0 + per);
        int32_t c = 0;
        for (int32_t i = i0; i < i1; ++i) c += __popc(bitmap[i]);
        const int32_t incl = warp_scan_incl<int32_t>(c);
        if (lane == 31) warp_total[warp] = incl;
        __syncthreads();
        int32_t lower = 0, all = 0;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int32_t t = warp_total[i];
            if (i < warp) lower += t;
            all += t;
        }
        c = lower + incl - c;
        for (int32_t i = i0; i < i1; ++i) {
            before[i] = (uint16_t)c;
            c += __popc(bitmap[i]);
        }
        __syncthreads();
#pragma unroll
        for (int r = 0; r < SORT_TILE / 256; ++r) {
            if (slot[r] == 0xFFFFFFFFu) continue;
            const uint32_t k = (uint32_t)zs[first + tid + 256 * r], below = (1u << (k & 31u)) - 1u;
            emit(out0 + (int32_t)before[k >> 5] + __popc(bitmap[k >> 5] & below), k,
                 table[slot[r]] & ((1u << ROW_COUNT_BITS) - 1u));
        }
        if (tid == 0) out.nnz[s0 + w] = all;
        __syncthreads();
    }
    if (NK == NK_BINS) {
        __syncthreads();
        for (int32_t k = tid; k < K; k += 256) {
            const int32_t n = bins[k];
            if (n) atomicAdd(&out.nk[k], n);
        }
    }
}

// Warm words (more tokens than a tail tile holds, no dense row): one CTA per word.  The word's
// tokens are counted in 16-bit bins over a window of topics in shared memory (two bins per word of
// shared memory; a warm word has fewer than 65536 tokens), and the nonzero bins, read in order,
// are the sorted row: every warp owns a run of consecutive bin pairs, counts its nonzero bins, the
// warps' totals are scanned, and a second walk writes the entries.
template <typename T>
__global__ void __launch_bounds__(1024)
k_warm_rows(const int32_t* __restrict__ words, const int32_t* __restrict__ word_off, const T* __restrict__ z,
            const int32_t* __restrict__ row_start, uint32_t* __restrict__ wk_topic, uint32_t* __restrict__ wk_count,
            int32_t* __restrict__ wk_nnz, int32_t* __restrict__ nk, int32_t K, int32_t window, SweepState* state)
{
    // nk: null if n_k is not added up here
    stamp(state, STAMP_WARM_ROWS);
    int* const err = &state->err;
    extern __shared__ __align__(16) uint32_t bins2[];
    __shared__ int32_t warp_total[33];
    const int32_t w = words[blockIdx.x];
    const int32_t first = word_off[w], cnt = word_off[w + 1] - first;
    const int32_t out0 = row_start[w], cap = row_start[w + 1] - out0;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    int32_t done = 0;
    for (int32_t k0 = 0; k0 < K; k0 += window) {
        const int32_t nb = min(window, K - k0), nw = (nb + 1) >> 1;
        const int32_t nw4 = (nw + 3) >> 2;
        for (int b = threadIdx.x; b < nw4; b += blockDim.x) reinterpret_cast<uint4*>(bins2)[b] = make_uint4(0u, 0u, 0u, 0u);
        __syncthreads();
        for (int32_t j = threadIdx.x; j < cnt; j += blockDim.x) {
            const uint32_t k = (uint32_t)__ldcs(z + first + j);
            if (k >= (uint32_t)K) { atomicOr(err, ERR_TOPIC_RANGE); continue; }
            const uint32_t b = k - (uint32_t)k0;
            if (b < (uint32_t)nb) atomicAdd(&bins2[b >> 1], (b & 1u) ? 0x10000u : 1u);
        }
        __syncthreads();
        // a warp's run of bin pairs
        const int32_t per_warp = ((nw + nwarps - 1) / nwarps + 31) & ~31;
        const int32_t q0 = min(nw, warp * per_warp), q1 = min(nw, q0 + per_warp);
        int32_t mine = 0;
        for (int32_t q = q0 + lane; q < q1; q += 32) {
            const uint32_t n2 = bins2[q];
            mine += ((n2 & 0xFFFFu) != 0u) + ((n2 >> 16) != 0u);
        }
        mine = warp_reduce_sum<int32_t>(mine);
        if (lane == 0) warp_total[warp] = mine;
        __syncthreads();
        if (threadIdx.x == 0) {
            int32_t run = 0;
            for (int i = 0; i < nwarps; ++i) { const int32_t t = warp_total[i]; warp_total[i] = run; run += t; }
            warp_total[32] = run;
        }
        __syncthreads();
        int32_t at = done + warp_total[warp];
        const int32_t total = warp_total[32];
        if (done + total > cap) {
            if (threadIdx.x == 0) atomicOr(err, ERR_ROW_OVERFLOW);
        } else {
            const uint32_t below = (1u << lane) - 1u;
            for (int32_t q = q0 + lane; q - lane < q1; q += 32) {
                const uint32_t n2 = q < q1 ? bins2[q] : 0u;
                const bool lo = (n2 & 0xFFFFu) != 0u, hi = (n2 >> 16) != 0u;
                const uint32_t m_lo = __ballot_sync(0xffffffffu, lo), m_hi = __ballot_sync(0xffffffffu, hi);
                int32_t pos = at + __popc(m_lo & below) + __popc(m_hi & below);
                if (lo) {
                    wk_topic[out0 + pos] = (uint32_t)(k0 + 2 * q);
                    wk_count[out0 + pos] = n2 & 0xFFFFu;
                    if (nk) atomicAdd(&nk[k0 + 2 * q], (int32_t)(n2 & 0xFFFFu));
                    ++pos;
                }
                if (hi) {
                    wk_topic[out0 + pos] = (uint32_t)(k0 + 2 * q + 1);
                    wk_count[out0 + pos] = n2 >> 16;
                    if (nk) atomicAdd(&nk[k0 + 2 * q + 1], (int32_t)(n2 >> 16));
                }
                at += __popc(m_lo) + __popc(m_hi);
            }
        }
        done += total;
        __syncthreads();
    }
    if (threadIdx.x == 0) wk_nnz[w] = done;
}

// Hot words: one CTA per run of a word's tokens; histogram of a window of topics in shared memory
// (32-bit bins).  A word of one run (nearly all of them: runs are long) has its whole row in the bins, and the
// CTA writes it out in both forms -- the dense row, zeros included, and the sorted one -- and, NK, adds it to
// n_k.  The runs of a longer word add their nonzero bins to the word's line of `acc`; the last of them to
// finish takes the line's contents the same way and leaves it zero for the next rebuild.
// How the tokens are cut: load_common() in api.cu.
// windows of more topics leave room for one CTA per multiprocessor: it gets twice the threads
constexpr int HIST_WIDE = 24576;
struct HotRuns {
    const int4* runs;      // (word, first token, tokens, index of the word among those with several runs or -1)
    const int32_t* dense_slot;
    int32_t* dense_rows;
    int32_t stride;
    int32_t* acc;          // [words with several runs][stride], all zero between rebuilds
    int32_t* acc_done;     // [...] runs that have added theirs
    const int32_t* acc_runs;  // [...] runs in all
};

// Bins [0, nb) of topics k0.. -> dense row and sorted entries from position `done` of the word's row on;
// returns how many there were.  Every warp owns a run of bins: one walk to count, one to write.
template <NkMode NK, class Bin>
__device__ __forceinline__ int32_t emit_bins(const Bin& bin, int32_t k0, int32_t nb, int32_t* dense, int32_t out0,
                                             int32_t cap, int32_t done, const RowTables& out, int32_t* warp_total)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    const int32_t per_warp = ((nb + nwarps - 1) / nwarps + 31) & ~31;
    const int32_t q0 = min(nb, warp * per_warp), q1 = min(nb, q0 + per_warp);
    int32_t mine = 0;
    for (int32_t q = q0 + lane; q - lane < q1; q += 32) mine += __popc(__ballot_sync(0xFFFFFFFFu, q < q1 && bin(q) != 0));
    if (lane == 0) warp_total[warp] = mine;
    __syncthreads();
    const int32_t t = lane < nwarps ? warp_total[lane] : 0;
    const int32_t incl = warp_scan_incl<int32_t>(t);
    const int32_t total = __shfl_sync(0xFFFFFFFFu, incl, 31);
    int32_t at = done + __shfl_sync(0xFFFFFFFFu, incl - t, warp);
    const bool fits = done + total <= cap;
    if (!fits && threadIdx.x == 0) atomicOr(&out.state->err, ERR_ROW_OVERFLOW);
    for (int32_t q = q0 + lane; q - lane < q1; q += 32) {
        const int32_t n = q < q1 ? bin(q) : 0;
        const uint32_t some = __ballot_sync(0xFFFFFFFFu, n != 0);
        if (q < q1) dense[k0 + q] = n;
        if (n && fits) {
            const int32_t slot = out0 + at + __popc(some & ((1u << lane) - 1u));
            out.topic[slot] = (uint32_t)(k0 + q);
            out.count[slot] = (uint32_t)n;
            if (NK != NK_NONE) atomicAdd(&out.nk[k0 + q], n);
        }
        at += __popc(some);
    }
    __syncthreads();
    return total;
}

template <typename T, NkMode NK, bool NARROW>
__global__ void __launch_bounds__(1024, 2)
k_hot_rows(HotRuns h, const T* __restrict__ z, RowTables out, int32_t K, int32_t window)
{
    stamp(out.state, STAMP_HIST);
    extern __shared__ __align__(16) int32_t hist_bins[];
    __shared__ int32_t warp_total[32];
    __shared__ bool last;
    int* const err = &out.state->err;
    const int4 run = h.runs[blockIdx.x];
    const int32_t w = run.x, first = run.y, cnt = run.z, multi = run.w;
    int32_t* dense = h.dense_rows + (size_t)h.dense_slot[w] * h.stride;
    int32_t* acc = h.acc + (size_t)max(multi, 0) * h.stride;
    const int32_t out0 = out.row_start[w], cap = out.row_start[w + 1] - out0;
    int32_t done = 0;
    // More topics than a window has: a run whose counts fit 16 bits takes twice as many at once.  Each window is a pass over the
    // run's tokens (n_kw of 200 M tokens, K = 10^5: 2.55 ms with three windows for every run, 2.43 with two and with one).
    const bool narrow = NARROW && cnt < 65536;
    uint32_t* bins2 = reinterpret_cast<uint32_t*>(hist_bins);
    const int32_t step = narrow ? 2 * window : window;
    for (int32_t k0 = 0; k0 < K; k0 += step) {
        const int32_t nb = min(step, K - k0), words = narrow ? (nb + 1) / 2 : nb;
        for (int b = threadIdx.x; b < (words + 3) / 4; b += blockDim.x)
            reinterpret_cast<int4*>(hist_bins)[b] = make_int4(0, 0, 0, 0);
        __syncthreads();
        auto add = [&](uint32_t k) {
            if (k >= (uint32_t)K) { atomicOr(err, ERR_TOPIC_RANGE); return; }
            const uint32_t b = k - (uint32_t)k0;
            if (b >= (uint32_t)nb) return;
            if (narrow) atomicAdd(&bins2[b >> 1], (b & 1u) ? 0x10000u : 1u);
            else atomicAdd(&hist_bins[b], 1);
        };
        // the run's topics are read 16 bytes at a time; what lies before the first and after the
        // last 16-byte boundary one by one
        constexpr int E = 16 / (int)sizeof(T);
        const int32_t head = min(cnt, (int32_t)((E - (first & (E - 1))) & (E - 1)));
        const int32_t nvec = (cnt - head) / E;
        const uint4* zv = reinterpret_cast<const uint4*>(z + first + head);
        for (int q = threadIdx.x; q < nvec; q += blockDim.x) {
            const uint4 x = k0 == 0 ? __ldcs(zv + q) : __ldg(zv + q);
            const uint32_t xs[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                if (sizeof(T) == 2) {
                    add(xs[u] & 0xFFFFu);
                    add(xs[u] >> 16);
                } else {
                    add(xs[u]);
                }
            }
        }
        for (int j = threadIdx.x; j < cnt - nvec * E; j += blockDim.x)
            add((uint32_t)z[first + (j < head ? j : nvec * E + j)]);
        __syncthreads();
        const auto bin = [=](int32_t q) { return narrow ? (int32_t)(bins2[q >> 1] >> (16 * (q & 1)) & 0xFFFFu) : hist_bins[q]; };
        if (multi < 0) {
            done += emit_bins<NK>(bin, k0, nb, dense, out0, cap, done, out, warp_total);
        } else {
            for (int b = threadIdx.x; b < nb; b += blockDim.x) {
                const int32_t n = bin(b);
                if (n) atomicAdd(&acc[k0 + b], n);
            }
            __syncthreads();
        }
    }
    if (multi >= 0) {
        __threadfence();
        __syncthreads();
        if (threadIdx.x == 0) last = atomicAdd(&h.acc_done[multi], 1) == h.acc_runs[multi] - 1;
        __syncthreads();
        if (!last) return;
        __threadfence();
        done = emit_bins<NK>([acc](int32_t q) { return __ldcg(acc + q); }, 0, K, dense, out0, cap, 0, out, warp_total);
        for (int k = threadIdx.x; k < K; k += blockDim.x) acc[k] = 0;
        if (threadIdx.x == 0) h.acc_done[multi] = 0;
    }
    if (threadIdx.x == 0) out.nnz[w] = done;
}

// n_k = sum over words of n_kw (Section 3), taken from the rows the n_kw rebuild has just written
// instead of from another pass over the assignments:
//   - dense rows: column sums, one thread per topic and group of rows;
//   - sorted rows of the words without a dense row: CTA-private shared-memory bins over a chunk
//     of words, flushed with one global add per nonzero bin.
__global__ void __launch_bounds__(256)
k_nk_from_dense(const int32_t* __restrict__ dense_rows, int32_t n_dense, int32_t K, int32_t stride,
                int32_t* __restrict__ nk, SweepState* state)
{
    stamp(state, STAMP_NK_DENSE);
    // four consecutive topics per thread (rows are padded to a multiple of four and 16-byte aligned;
    // the padding is never written, so it reads as zero), a slice of the rows per blockIdx.y
    const int32_t k = 4 * (blockIdx.x * blockDim.x + threadIdx.x);
    if (k >= stride) return;
    int4 s = make_int4(0, 0, 0, 0);
#pragma unroll 4
    for (int32_t r = blockIdx.y; r < n_dense; r += gridDim.y) {
        const int4 x = __ldcs(reinterpret_cast<const int4*>(dense_rows + (size_t)r * stride + k));
        s.x += x.x; s.y += x.y; s.z += x.z; s.w += x.w;
    }
    if (s.x) atomicAdd(&nk[k], s.x);
    if (s.y && k + 1 < K) atomicAdd(&nk[k + 1], s.y);
    if (s.z && k + 2 < K) atomicAdd(&nk[k + 2], s.z);
    if (s.w && k + 3 < K) atomicAdd(&nk[k + 3], s.w);
}

__global__ void __launch_bounds__(512)
k_nk_from_sparse(const int32_t* __restrict__ row_start, const int32_t* __restrict__ wk_nnz,
                 const uint32_t* __restrict__ wk_topic, const uint32_t* __restrict__ wk_count,
                 const int32_t* __restrict__ dense_slot, int32_t V, int32_t* __restrict__ nk, int32_t K,
                 int32_t window, SweepState* state)
{
    stamp(state, STAMP_NK_SPARSE);
    extern __shared__ int32_t bins[];
    const int32_t per = (V + gridDim.x - 1) / gridDim.x;
    const int32_t w_lo = per * blockIdx.x, w_hi = min(V, w_lo + per);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    for (int32_t k0 = 0; k0 < K; k0 += window) {
        const int32_t nb = min(window, K - k0);
        for (int b = threadIdx.x; b < nb; b += blockDim.x) bins[b] = 0;
        __syncthreads();
        for (int32_t w = w_lo + warp; w < w_hi; w += nwarps) {
            if (dense_slot[w] >= 0) continue;
            const int32_t r0 = row_start[w], n = wk_nnz[w];
            for (int32_t j = lane; j < n; j += 32) {
                const uint32_t b = wk_topic[r0 + j] - (uint32_t)k0;
                if (b < (uint32_t)nb) atomicAdd(&bins[b], (int32_t)wk_count[r0 + j]);
            }
        }
        __syncthreads();
        for (int b = threadIdx.x; b < nb; b += blockDim.x) {
            const int32_t n = bins[b];
            if (n) atomicAdd(&nk[k0 + b], n);
        }
        __syncthreads();
    }
}

// The same sums when K is too large for bins in shared memory: one global add per row entry (the
// adds of one warp go to different topics: a row holds a topic once).
__global__ void __launch_bounds__(256)
k_nk_from_sparse_direct(const int32_t* __restrict__ row_start, const int32_t* __restrict__ wk_nnz,
                        const uint32_t* __restrict__ wk_topic, const uint32_t* __restrict__ wk_count,
                        const int32_t* __restrict__ dense_slot, int32_t V, int32_t* __restrict__ nk, SweepState* state)
{
    stamp(state, STAMP_NK_SPARSE);
    const int lane = threadIdx.x & 31;
    const int32_t warps = (gridDim.x * blockDim.x) >> 5;
    for (int32_t w = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; w < V; w += warps) {
        if (dense_slot[w] >= 0) continue;
        const int32_t r0 = row_start[w], n = wk_nnz[w];
        for (int32_t j = lane; j < n; j += 32) atomicAdd(&nk[__ldcs(wk_topic + r0 + j)], (int32_t)__ldcs(wk_count + r0 + j));
    }
}

struct EmitRowSizes {
    int32_t* nnz;
    __device__ __forceinline__ void entry(int32_t, int32_t, uint32_t, uint32_t) const {}
    __device__ __forceinline__ void rows(int32_t seg, int32_t n) const { nnz[seg] = n; }
};

struct EmitRowEntries {
    const long long* row_off;
    int32_t* topic;
    int32_t* count;
    __device__ __forceinline__ void entry(int32_t seg, int32_t rank, uint32_t k, uint32_t n) const
    {
        const long long at = row_off[seg] + rank;
        topic[at] = (int32_t)k;
        count[at] = (int32_t)n;
    }
    __device__ __forceinline__ void rows(int32_t, int32_t) const {}
};

// Sorted rows of the segments (documents) of `tiles` from z given in segment order: sizes only, or
// the entries at the row offsets (export.cu).
template <typename T>
void launch_doc_rows(Ctx& c, const int32_t* tiles, int32_t n_tiles, const T* z, int32_t* nnz, const long long* row_off,
                     int32_t* topic, int32_t* count)
{
    if (nnz)
        k_seg_count_sorted<T, EmitRowSizes><<<n_tiles, 256, 0, c.stream>>>(tiles, c.v.doc_off, z, c.v.topic_bits, c.K,
                                                                            EmitRowSizes{nnz}, c.v.state, -1);
    else
        k_seg_count_sorted<T, EmitRowEntries><<<n_tiles, 256, 0, c.stream>>>(
            tiles, c.v.doc_off, z, c.v.topic_bits, c.K, EmitRowEntries{row_off, topic, count}, c.v.state, -1);
}
// The same, single pass, for K <= WORD_ROWS_BITMAP_MAX_K: sizes, and entries from the documents' first tokens on (a row
// has at most as many entries as the document has tokens).
void launch_doc_rows_spread(Ctx& c, const int32_t* tiles, int32_t n_tiles, const uint16_t* z, int32_t* nnz, uint32_t* topic, uint32_t* count)
{
    const RowTables out{c.v.doc_off, topic, count, nnz, nullptr, c.v.state};
    const size_t area = row_area_bytes(c.K);
    k_word_rows<NK_NONE><<<n_tiles, 256, area, c.stream>>>(tiles, c.v.doc_off, z, out, c.K, (int32_t)(area / 4), -1);
}
template void launch_doc_rows<uint16_t>(Ctx&, const int32_t*, int32_t, const uint16_t*, int32_t*, const long long*, int32_t*, int32_t*);
template void launch_doc_rows<int32_t>(Ctx&, const int32_t*, int32_t, const int32_t*, int32_t*, const long long*, int32_t*, int32_t*);

static int hist_window(const Ctx& c) { return c.K < HIST_BINS ? c.K : HIST_BINS; }

template <typename T, NkMode NK>
static int count_wk_t(Ctx& c)
{
    View& v = c.v;
    int launches = 0;
    const T* z = (const T*)v.zw;
    const RowTables out{v.row_start, v.wk_topic, v.wk_count, v.wk_nnz, v.nk_next, v.state};
    // the tail words' rows and the hot words' rows are built side by side
    fork_streams(c);
    if (c.n_hot_runs) {
        const HotRuns h{reinterpret_cast<const int4*>(c.hot_runs), v.dense_slot, v.dense_rows, v.dense_stride, c.acc,
                        c.acc_done, c.acc_runs};
        const int win = c.K < HIST32_BINS ? c.K : HIST32_BINS;
        const auto kernel = NK != NK_BINS && c.K > HIST32_BINS ? k_hot_rows<T, NK, NK != NK_BINS> : k_hot_rows<T, NK, false>;
        kernel<<<c.n_hot_runs, win > HIST_WIDE ? 1024 : 512, (size_t)((win + 3) / 4) * 16, c.stream>>>(h, z, out, c.K, win);
        ++launches;
    }
    if (c.n_word_tiles) {
        if (c.K <= WORD_ROWS_BITMAP_MAX_K) {
            const size_t area = row_area_bytes(c.K);
            if constexpr (sizeof(T) == 2)  // 32-bit topics mean a larger K
                k_word_rows<NK><<<c.n_word_tiles, 256, area + (NK == NK_BINS ? (size_t)c.K * 4 : 0), c.side[0]>>>(
                    c.word_tiles, v.word_off, z, out, c.K, (int32_t)(area / 4), STAMP_ROWS);
        } else {
            EmitWord e{v.row_start, v.wk_topic, v.wk_count, v.wk_nnz, NK == NK_NONE ? nullptr : v.nk_next};
            k_seg_count_sorted<T, EmitWord><<<c.n_word_tiles, 256, 0, c.side[0]>>>(
                c.word_tiles, v.word_off, z, v.topic_bits, c.K, e, v.state, STAMP_ROWS);
        }
        ++launches;
    }
    if (c.n_warm) {
        const int win = c.K < HIST16_BINS ? c.K : HIST16_BINS;
        k_warm_rows<T><<<c.n_warm, 1024, (size_t)((win + 7) / 8) * 16, c.side[1]>>>(
            c.warm_words, v.word_off, z, v.row_start, v.wk_topic, v.wk_count, v.wk_nnz, NK == NK_NONE ? nullptr : v.nk_next, c.K, win,
            v.state);
        ++launches;
    }
    join_streams(c);
    return launches;
}

// Must follow launch_count_wk(): reads the rows it wrote and adds into View::nk_next, which the sweep's
// first kernel (or the caller) has cleared.
int launch_count_k_from_rows(Ctx& c)
{
    View& v = c.v;
    if (c.N == 0) return 0;
    int launches = 0;
    // both kernels add into n_k (integer adds: any order gives the same sums)
    fork_streams(c);
    if (c.n_dense) {
        const dim3 grid((unsigned)((v.dense_stride / 4 + 255) / 256), (unsigned)std::min(c.n_dense, 256));
        k_nk_from_dense<<<grid, 256, 0, c.stream>>>(v.dense_rows, c.n_dense, c.K, v.dense_stride, v.nk_next, v.state);
        ++launches;
    }
    if (c.n_dense < c.V) {
        if (c.K <= HIST_BINS) {
            const int win = hist_window(c);
            const int grid = std::min(148 * 4, (int)((c.V + 255) / 256));
            k_nk_from_sparse<<<grid, 512, (size_t)win * 4, c.side[0]>>>(v.row_start, v.wk_nnz, v.wk_topic, v.wk_count,
                                                                       v.dense_slot, c.V, v.nk_next, c.K, win, v.state);
        } else {
            const int grid = (int)std::min<int64_t>(148 * 16, ((int64_t)c.V * 32 + 255) / 256);
            k_nk_from_sparse_direct<<<grid, 256, 0, c.side[0]>>>(v.row_start, v.wk_nnz, v.wk_topic, v.wk_count,
                                                                v.dense_slot, c.V, v.nk_next, v.state);
        }
        ++launches;
    }
    join_streams(c);
    return launches;
}

int launch_count_wk(Ctx& c)
{
    if (c.wide_topics) return c.nk_mode == NK_NONE ? count_wk_t<int32_t, NK_NONE>(c) : count_wk_t<int32_t, NK_DIRECT>(c);
    return c.nk_mode == NK_NONE   ? count_wk_t<uint16_t, NK_NONE>(c)
           : c.nk_mode == NK_BINS ? count_wk_t<uint16_t, NK_BINS>(c)
                                  : count_wk_t<uint16_t, NK_DIRECT>(c);
}
int launch_count_k(Ctx& c) { return c.nk_mode != NK_NONE ? 0 : launch_count_k_from_rows(c); }

// n_k by the row kernels or by a pass of its own.  Bins: every CTA adds to every topic's counter once, and the adds
// to one counter queue, so K and the number of CTAs are bounded.  One add per entry: as many adds as nonzeros, fine
// while they are few (9 M tokens, K = 16 695: 0.36 ms less per rebuild); with more, the pass over the rows (bins again,
// fewer CTAs) is ahead.
void choose_nk_mode(Ctx& c)
{
    if (c.K <= NK_WITH_ROWS_MAX_K && c.n_hot_runs + c.n_word_tiles <= NK_WITH_ROWS_MAX_CTAS && c.N >= c.K) c.nk_mode = NK_BINS;
    else c.nk_mode = c.N <= NK_DIRECT_MAX_TOKENS ? NK_DIRECT : NK_NONE;
}

void set_hist_smem_limits()
{
    cudaFuncSetAttribute(k_warm_rows<uint16_t>, cudaFuncAttributeMaxDynamicSharedMemorySize, HIST16_BINS * 2 + 16);
    cudaFuncSetAttribute(k_warm_rows<int32_t>, cudaFuncAttributeMaxDynamicSharedMemorySize, HIST16_BINS * 2 + 16);
    const int hist = HIST32_BINS * 4, rows = (int)row_area_bytes(WORD_ROWS_BITMAP_MAX_K),
              rows_bins = (int)row_area_bytes(NK_WITH_ROWS_MAX_K) + NK_WITH_ROWS_MAX_K * 4;
    constexpr auto most = cudaFuncAttributeMaxDynamicSharedMemorySize;
    cudaFuncSetAttribute(k_hot_rows<uint16_t, NK_NONE, false>, most, hist);
    cudaFuncSetAttribute(k_hot_rows<uint16_t, NK_NONE, true>, most, hist);
    cudaFuncSetAttribute(k_hot_rows<uint16_t, NK_BINS, false>, most, hist);
    cudaFuncSetAttribute(k_hot_rows<uint16_t, NK_DIRECT, false>, most, hist);
    cudaFuncSetAttribute(k_hot_rows<uint16_t, NK_DIRECT, true>, most, hist);
    cudaFuncSetAttribute(k_hot_rows<int32_t, NK_NONE, false>, most, hist);
    cudaFuncSetAttribute(k_hot_rows<int32_t, NK_NONE, true>, most, hist);
    cudaFuncSetAttribute(k_hot_rows<int32_t, NK_DIRECT, false>, most, hist);
    cudaFuncSetAttribute(k_hot_rows<int32_t, NK_DIRECT, true>, most, hist);
    cudaFuncSetAttribute(k_word_rows<NK_NONE>, most, rows);
    cudaFuncSetAttribute(k_word_rows<NK_DIRECT>, most, rows);
    cudaFuncSetAttribute(k_word_rows<NK_BINS>, most, rows_bins);
    cudaFuncSetAttribute(k_nk_from_sparse, cudaFuncAttributeMaxDynamicSharedMemorySize, HIST_BINS * 4);
}

}  // namespace lda
