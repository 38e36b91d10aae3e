// One-time corpus layout (Section 6, item 3: token-topic pairs are sorted by
// word once, so that the tokens of a word -- and of a slice of words -- are
// contiguous).  Tokens are sorted stably by word id, so inside a word they
// stay in document order.  The sort itself uses CUB's device radix sort: it
// runs once per corpus, outside the per-sweep path.
#include <algorithm>

#include <cub/device/device_radix_sort.cuh>
#include <cub/device/device_scan.cuh>

#include "lda_device.cuh"
#include "lda_internal.cuh"

namespace lda {

__global__ void k_check_words_iota(const int32_t* __restrict__ words, uint32_t* __restrict__ iota,
                                   int32_t n, int32_t V, int* err)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        iota[i] = (uint32_t)i;
        const int32_t w = words[i];
        if (w < 0 || w >= V) atomicOr(err, ERR_WORD_RANGE);
    }
}

// word_off[w] = first position whose word is >= w (positions are word-sorted).
__global__ void k_word_offsets(const int32_t* __restrict__ sorted_words, int32_t n, int32_t V,
                               int32_t* __restrict__ word_off)
{
    const int32_t w = blockIdx.x * blockDim.x + threadIdx.x;
    if (w > V) return;
    int32_t lo = 0, hi = n;
    while (lo < hi) {
        const int32_t mid = lo + ((hi - lo) >> 1);
        if (sorted_words[mid] < w) lo = mid + 1; else hi = mid;
    }
    word_off[w] = lo;
}

// What the passes need of every word: room for its sparse row (row_len becomes row_start by a prefix sum), whether the
// MH step treats it as hot, no dense row yet.  `tf` gives the words' frequencies where they are not those of this corpus.
// (These lists are made here, not on the host: for 944 000 words and 110 000 tokens, the host's copies of
// them and their pages were 6 of the 12 ms of a load.)
__global__ void k_word_rooms(const int32_t* __restrict__ word_off, const int32_t* __restrict__ tf, int32_t V, int32_t K,
                             int32_t* __restrict__ row_len, uint8_t* __restrict__ hot_word, int32_t* __restrict__ dense_slot)
{
    const int32_t w = blockIdx.x * blockDim.x + threadIdx.x;
    if (w > V) return;
    int32_t n = 0;
    if (w < V) {
        n = word_off[w + 1] - word_off[w];
        if (tf) n = max(n, tf[w]);
        hot_word[w] = n > COLD_TILE;
        dense_slot[w] = -1;
    }
    row_len[w] = min(n, K);
}

__global__ void k_dense_slots(const int32_t* __restrict__ dense_words, int32_t n, int32_t* __restrict__ dense_slot)
{
    const int32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) dense_slot[dense_words[i]] = i;
}

void launch_dense_slots(Ctx& c, const int32_t* dense_words)
{
    if (c.n_dense) k_dense_slots<<<(c.n_dense + 255) / 256, 256, 0, c.stream>>>(dense_words, c.n_dense, const_cast<int32_t*>(c.v.dense_slot));
}

// Keys of the block-major order: the block of a token is the high part of its document-order index.
__global__ void k_block_keys(const uint32_t* __restrict__ tok_orig, int32_t n, int shift,
                             uint32_t* __restrict__ keys, uint32_t* __restrict__ iota)
{
    for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < n;
         p += (int64_t)gridDim.x * blockDim.x) {
        keys[p] = tok_orig[p] >> shift;
        iota[p] = (uint32_t)p;
    }
}

// The block-major index of every token, by word-sorted position and by document-order index.
__global__ void k_block_major_maps(const uint32_t* __restrict__ order, const uint32_t* __restrict__ tok_orig,
                                   int32_t n, uint32_t* __restrict__ inv, uint32_t* __restrict__ bm_of_tok)
{
    for (int64_t m = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; m < n;
         m += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t p = order[m];
        inv[p] = (uint32_t)m;
        bm_of_tok[tok_orig[p]] = (uint32_t)m;
    }
}

int build_layout(Ctx& c, const int32_t* word_ids_dev, const std::vector<int32_t>& doc_off_host, LayoutTemps& temps)
{
    const int32_t N = (int32_t)c.N, D = (int32_t)c.D, V = c.V;
    cudaStream_t st = c.stream;
    const size_t n1 = (size_t)(N > 0 ? N : 1);

    uint32_t* tok_orig = (uint32_t*)dev_alloc(c, n1 * 4);
    uint32_t* inv = (uint32_t*)dev_alloc(c, n1 * 4);
    uint32_t* bm_of_tok = (uint32_t*)dev_alloc(c, n1 * 4);
    int32_t* word_off = (int32_t*)dev_alloc(c, ((size_t)V + 1) * 4);
    int32_t* doc_off = (int32_t*)dev_alloc(c, ((size_t)D + 1) * 4);
    int32_t* row_start = (int32_t*)dev_alloc(c, ((size_t)V + 1) * 4);
    int32_t* dense_slot = (int32_t*)dev_alloc(c, (size_t)V * 4);
    uint8_t* hot_word = (uint8_t*)dev_alloc(c, (size_t)V);
    if (!tok_orig || !inv || !bm_of_tok || !word_off || !doc_off || !row_start || !dense_slot || !hot_word) return LDA_ENOMEM;
    c.v.row_start = row_start;
    c.v.dense_slot = dense_slot;
    c.v.hot_word = hot_word;
    c.v.inv = inv;
    c.v.bm_of_tok = bm_of_tok;
    c.v.tok_orig = tok_orig;
    c.v.word_off = word_off;
    c.v.doc_off = doc_off;
    if (copy_to_device(c, doc_off, doc_off_host.data(), ((size_t)D + 1) * 4) != cudaSuccess) return LDA_ECUDA;

    // transient buffers of the sorts; both sorts share the temporary storage
    int end_bit = 1, blk_bits = 1;
    while (end_bit < 31 && (1ll << end_bit) < (long long)V) ++end_bit;
    while (blk_bits < 32 && (((long long)N - 1) >> c.block_shift) >= (1ll << blk_bits)) ++blk_bits;
    size_t temp_bytes = 0, temp2_bytes = 0, scan_bytes = 0;
    const int32_t* no_keys = nullptr;
    const uint32_t* no_values = nullptr;
    if (N > 0 && (cub::DeviceRadixSort::SortPairs(nullptr, temp_bytes, no_keys, (int32_t*)nullptr, no_values, tok_orig, N, 0, end_bit,
                                                  st) != cudaSuccess ||
                  cub::DeviceRadixSort::SortPairs(nullptr, temp2_bytes, no_values, (uint32_t*)nullptr, no_values, tok_orig, N, 0,
                                                  blk_bits, st) != cudaSuccess))
        return LDA_ECUDA;
    if (cub::DeviceScan::ExclusiveSum(nullptr, scan_bytes, row_start, row_start, V + 1, st) != cudaSuccess) return LDA_ECUDA;
    auto transient = [&](size_t bytes) -> void* {
        void* p = nullptr;
        if (tmp_alloc(c, &p, bytes)) temps.held.push_back(p);
        return p;
    };
    int32_t* keys_out = (int32_t*)transient(n1 * 4);
    uint32_t* iota = (uint32_t*)transient(n1 * 4);
    uint32_t* keys_blk = (uint32_t*)transient(n1 * 4);
    uint32_t* order = (uint32_t*)transient(n1 * 4);
    void* temp = transient(std::max({temp_bytes, temp2_bytes, scan_bytes}));
    int32_t* tf = c.shard_global_tf.empty() ? nullptr : (int32_t*)transient((size_t)V * 4);
    if (!keys_out || !iota || !keys_blk || !order || !temp || (!tf && !c.shard_global_tf.empty())) return LDA_ENOMEM;
    bool ok = true;
    if (N > 0) {
        k_check_words_iota<<<1184, 256, 0, st>>>(word_ids_dev, iota, N, V, c.v.err);
        ok = cub::DeviceRadixSort::SortPairs(temp, temp_bytes, word_ids_dev, keys_out, iota, tok_orig, N, 0, end_bit, st) == cudaSuccess;
    }
    k_word_offsets<<<(V + 1 + 255) / 256, 256, 0, st>>>(keys_out, N, V, word_off);
    cudaEventRecord(c.ev_chunk, st);
    if (tf && copy_to_device(c, tf, c.shard_global_tf.data(), (size_t)V * 4) != cudaSuccess) return LDA_ECUDA;
    k_word_rooms<<<(V + 1 + 255) / 256, 256, 0, st>>>(word_off, tf, V, c.K, row_start, hot_word, dense_slot);
    ok = ok && cub::DeviceScan::ExclusiveSum(temp, scan_bytes, row_start, row_start, V + 1, st) == cudaSuccess;
    if (N > 0 && ok) {
        // block-major order: tokens sorted by (block of their document-order index, word-sorted
        // position); a stable sort of the positions by block (one block: the positions themselves)
        if (((long long)N - 1) >> c.block_shift) {
            k_block_keys<<<1184, 256, 0, st>>>(tok_orig, N, c.block_shift, keys_blk, iota);
            uint32_t* keys_tmp = reinterpret_cast<uint32_t*>(keys_out);  // the word keys are no longer needed
            ok = cub::DeviceRadixSort::SortPairs(temp, temp2_bytes, keys_blk, keys_tmp, iota, order, N, 0, blk_bits, st) == cudaSuccess;
        } else {
            order = iota;  // still 0, 1, 2, ...
        }
        if (ok) k_block_major_maps<<<1184, 256, 0, st>>>(order, tok_orig, N, inv, bm_of_tok);
    }
    return ok && cudaPeekAtLastError() == cudaSuccess ? LDA_OK : LDA_ECUDA;
}

}  // namespace lda
