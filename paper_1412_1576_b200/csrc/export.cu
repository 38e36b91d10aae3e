// n_kd (Eq. 12) as sorted rows in device memory: for every document the (topic, count) pairs of its
// nonzero counts, topics ascending.  The MH step never needs this form (its document pass builds
// hashed tables per tile and drops them); it is what lda_get_counts(LDA_NDK) hands out and what the
// exact-conditional sweep (gibbs.cu) walks.  Documents are packed whole into tiles of at most
// SORT_TILE tokens, sorted and run-length encoded by k_seg_count_sorted (counts.cu); a longer document
// gets a CTA of its own and a histogram over the topics.  Two passes: row sizes, a prefix sum for
// the row offsets (CUB's device scan: this path is off the sweep), then the entries.
#include <algorithm>

#include <cub/device/device_scan.cuh>

#include "lda_device.cuh"
#include "lda_internal.cuh"

namespace lda {

// A document longer than a sort tile: topics counted window by window in shared memory.
// EMIT false: nnz[d] = number of distinct topics; true: the row's entries at row_off[d].
template <typename T, bool EMIT>
__global__ void __launch_bounds__(512)
k_long_doc_rows(const int32_t* __restrict__ long_docs, const int32_t* __restrict__ doc_off, const T* __restrict__ z,
                int32_t K, int32_t window, int32_t* __restrict__ nnz, const long long* __restrict__ row_off,
                int32_t* __restrict__ topic, int32_t* __restrict__ count, int* err)
{
    extern __shared__ int32_t bins[];
    __shared__ int32_t scan_tmp[33];
    const int32_t d = long_docs[blockIdx.x];
    const int32_t first = doc_off[d], n = doc_off[d + 1] - first;
    int32_t done = 0;
    for (int32_t k0 = 0; k0 < K; k0 += window) {
        const int32_t nb = min(window, K - k0);
        for (int32_t b = threadIdx.x; b < nb; b += blockDim.x) bins[b] = 0;
        __syncthreads();
        for (int32_t j = threadIdx.x; j < n; j += blockDim.x) {
            const uint32_t k = (uint32_t)z[first + j];
            if (k >= (uint32_t)K) { atomicOr(err, ERR_TOPIC_RANGE); continue; }
            const uint32_t b = k - (uint32_t)k0;
            if (b < (uint32_t)nb) atomicAdd(&bins[b], 1);
        }
        __syncthreads();
        for (int32_t b0 = 0; b0 < nb; b0 += blockDim.x) {
            const int32_t b = b0 + (int32_t)threadIdx.x;
            const int32_t c = b < nb ? bins[b] : 0;
            int32_t total;
            const int32_t pos = block_scan_excl<int32_t>(c > 0 ? 1 : 0, scan_tmp, total);
            if (EMIT && c > 0) {
                const long long at = row_off[d] + done + pos;
                topic[at] = k0 + b;
                count[at] = c;
            }
            done += total;
        }
        __syncthreads();
    }
    if (!EMIT && threadIdx.x == 0) nnz[d] = done;
}

template <typename T>
void launch_doc_rows(Ctx& c, const int32_t* tiles, int32_t n_tiles, const T* z, int32_t* nnz, const long long* row_off,
                     int32_t* topic, int32_t* count);  // counts.cu

void free_dk_csr(Ctx& c, DkCsr& r)
{
    raw_free(c, r.row_off);
    raw_free(c, r.nnz);
    raw_free(c, r.topic);
    raw_free(c, r.count);
    r = DkCsr{};
}

// Rows from where they lie (row r at first[r]) to row_off[r].  A CTA takes COMPACT_RUN consecutive entries of the
// result, whatever rows they belong to: rows differ in length by four orders of magnitude, and a warp per row
// took 78 us for 370 000 entries where the longest row had 14 000.
constexpr int COMPACT_RUN = 2048;
__global__ void __launch_bounds__(256)
k_compact_rows(const int32_t* __restrict__ first, const long long* __restrict__ row_off, int32_t rows, long long total,
               const uint32_t* __restrict__ topic_in, const uint32_t* __restrict__ count_in, int32_t* __restrict__ topic,
               int32_t* __restrict__ count)
{
    __shared__ int32_t range[2];
    const long long o0 = (long long)blockIdx.x * COMPACT_RUN, o1 = min(total, o0 + COMPACT_RUN);
    auto row_of = [&](long long o, int32_t lo, int32_t hi) {  // last row in [lo, hi) that starts at or before o
        while (hi - lo > 1) {
            const int32_t mid = lo + ((hi - lo) >> 1);
            if (__ldg(row_off + mid) <= o) lo = mid; else hi = mid;
        }
        return lo;
    };
    if (threadIdx.x < 2) range[threadIdx.x] = row_of(threadIdx.x ? o1 - 1 : o0, 0, rows);
    __syncthreads();
    for (long long o = o0 + threadIdx.x; o < o1; o += 256) {
        const int32_t r = row_of(o, range[0], range[1] + 1);
        const long long at = first[r] + (o - __ldg(row_off + r));
        topic[o] = (int32_t)__ldcs(topic_in + at);
        count[o] = (int32_t)__ldcs(count_in + at);
    }
}

static void compact_rows(Ctx& c, const int32_t* first, const long long* row_off, int64_t rows, long long total,
                         const uint32_t* topic_in, const uint32_t* count_in, int32_t* topic, int32_t* count)
{
    const unsigned grid = (unsigned)((total + COMPACT_RUN - 1) / COMPACT_RUN);
    if (grid) k_compact_rows<<<grid, 256, 0, c.stream>>>(first, row_off, (int32_t)rows, total, topic_in, count_in, topic, count);
}

// Exclusive prefix sum of nnz[0..n) into row_off[0..n], its total to the host.  nnz[n] must be there (any value).
static int row_offsets(Ctx& c, const int32_t* nnz, long long* row_off, int64_t n, long long* total)
{
    void* temp = nullptr;
    size_t temp_bytes = 0;
    // nnz(n_kd), nnz(n_kw) <= n_tokens < 2^31: the 32-bit running sum cannot overflow
    if (cub::DeviceScan::ExclusiveSum(nullptr, temp_bytes, nnz, row_off, (int)(n + 1), c.stream) != cudaSuccess ||
        !tmp_alloc(c, &temp, temp_bytes)) {
        cudaGetLastError();
        return LDA_ENOMEM;
    }
    const cudaError_t e = cub::DeviceScan::ExclusiveSum(temp, temp_bytes, nnz, row_off, (int)(n + 1), c.stream);
    int rc = LDA_OK;
    if (e != cudaSuccess || cudaMemcpyAsync(total, row_off + n, 8, cudaMemcpyDeviceToHost, c.stream) != cudaSuccess ||
        cudaStreamSynchronize(c.stream) != cudaSuccess) {
        cudaGetLastError();
        rc = LDA_ECUDA;
    }
    raw_free(c, temp);
    return rc;
}

void launch_doc_rows_spread(Ctx& c, const int32_t* tiles, int32_t n_tiles, const uint16_t* z, int32_t* nnz, uint32_t* topic,
                            uint32_t* count);  // counts.cu

template <typename T>
static int build_dk_csr_t(Ctx& c, DkCsr& r, bool sizes_only)
{
    const View& v = c.v;
    const int32_t D = (int32_t)c.D;
    r = DkCsr{};
    if (!tmp_alloc(c, &r.row_off, ((size_t)D + 1) * 8) || !tmp_alloc(c, &r.nnz, ((size_t)D + 1) * 4)) {
        free_dk_csr(c, r);
        return LDA_ENOMEM;
    }
    cudaMemsetAsync(r.nnz, 0, ((size_t)D + 1) * 4, c.stream);
    // the assignments in document order, in the record array (scratch between calls)
    T* z = reinterpret_cast<T*>(v.rec);
    launch_export_assignments(c, z, sizeof(T) == 2);
    const int win = c.K < HIST_BINS ? c.K : HIST_BINS;
    // K small enough for the row kernel of the tail words: sizes and entries in one pass, the entries apart
    // first; else, or without room for that, the sorting kernel twice
    uint32_t *topic_at = nullptr, *count_at = nullptr;
    if (c.K <= WORD_ROWS_BITMAP_MAX_K && c.n_doc_sort_tiles && !sizes_only) {
        if (!tmp_alloc(c, &topic_at, (size_t)c.N * 4) || !tmp_alloc(c, &count_at, (size_t)c.N * 4)) {
            raw_free(c, topic_at);
            topic_at = nullptr;
        }
    }
    if (topic_at)  // (16-bit topics, by the limit on K)
        launch_doc_rows_spread(c, c.doc_sort_tiles, c.n_doc_sort_tiles, static_cast<const uint16_t*>(static_cast<void*>(v.rec)), r.nnz,
                               topic_at, count_at);
    else if (c.n_doc_sort_tiles) launch_doc_rows<T>(c, c.doc_sort_tiles, c.n_doc_sort_tiles, z, r.nnz, nullptr, nullptr, nullptr);
    if (c.n_doc_sort_long)
        k_long_doc_rows<T, false><<<c.n_doc_sort_long, 512, (size_t)win * 4, c.stream>>>(
            c.doc_sort_long, v.doc_off, z, c.K, win, r.nnz, nullptr, nullptr, nullptr, v.err);
    // the entries apart are a convenience: without the room for them beside the rest, the sorting kernel makes the rows
    const auto drop_entries = [&] {
        cudaStreamSynchronize(c.stream);
        raw_free(c, topic_at);
        raw_free(c, count_at);
        topic_at = count_at = nullptr;
    };
    int rc = row_offsets(c, r.nnz, r.row_off, D, &r.total);
    if (rc == LDA_ENOMEM && topic_at) {
        drop_entries();
        rc = row_offsets(c, r.nnz, r.row_off, D, &r.total);
    }
    const size_t cap = (size_t)(r.total > 0 ? r.total : 1);
    const auto room = [&] { return (r.topic || tmp_alloc(c, &r.topic, cap * 4)) && tmp_alloc(c, &r.count, cap * 4); };
    if (rc == LDA_OK && !sizes_only && !room()) {
        rc = LDA_ENOMEM;
        if (topic_at) {
            drop_entries();
            if (room()) rc = LDA_OK;
        }
    }
    if (rc == LDA_OK && !sizes_only) {
        if (topic_at) {
            // the rows of the documents longer than a tile are written over below
            compact_rows(c, v.doc_off, r.row_off, D, r.total, topic_at, count_at, r.topic, r.count);
        } else if (c.n_doc_sort_tiles) {
            launch_doc_rows<T>(c, c.doc_sort_tiles, c.n_doc_sort_tiles, z, nullptr, r.row_off, r.topic, r.count);
        }
        if (c.n_doc_sort_long)
            k_long_doc_rows<T, true><<<c.n_doc_sort_long, 512, (size_t)win * 4, c.stream>>>(
                c.doc_sort_long, v.doc_off, z, c.K, win, nullptr, r.row_off, r.topic, r.count, v.err);
    }
    if (topic_at) drop_entries();
    if (rc != LDA_OK) free_dk_csr(c, r);
    return rc;
}

int build_wk_csr(Ctx& c, WkCsr& r, bool sizes_only)
{
    const View& v = c.v;
    const int64_t V = c.V;
    r = WkCsr{};
    int rc = tmp_alloc(c, &r.row_off, ((size_t)V + 1) * 8) ? row_offsets(c, v.wk_nnz, r.row_off, V, &r.total) : LDA_ENOMEM;
    const size_t cap = (size_t)(r.total > 0 ? r.total : 1);
    if (rc == LDA_OK && !sizes_only) {
        if (tmp_alloc(c, &r.topic, cap * 4) && tmp_alloc(c, &r.count, cap * 4))
            compact_rows(c, v.row_start, r.row_off, V, r.total, v.wk_topic, v.wk_count, r.topic, r.count);
        else
            rc = LDA_ENOMEM;
    }
    if (rc != LDA_OK) free_wk_csr(c, r);
    return rc;
}

void free_wk_csr(Ctx& c, WkCsr& r)
{
    raw_free(c, r.row_off);
    raw_free(c, r.topic);
    raw_free(c, r.count);
    r = WkCsr{};
}

int build_dk_csr(Ctx& c, DkCsr& r, bool sizes_only)
{
    return c.wide_topics ? build_dk_csr_t<int32_t>(c, r, sizes_only) : build_dk_csr_t<uint16_t>(c, r, sizes_only);
}

void set_export_smem_limits()
{
    cudaFuncSetAttribute(k_long_doc_rows<uint16_t, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, HIST_BINS * 4);
    cudaFuncSetAttribute(k_long_doc_rows<uint16_t, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, HIST_BINS * 4);
    cudaFuncSetAttribute(k_long_doc_rows<int32_t, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, HIST_BINS * 4);
    cudaFuncSetAttribute(k_long_doc_rows<int32_t, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, HIST_BINS * 4);
}

}  // namespace lda
