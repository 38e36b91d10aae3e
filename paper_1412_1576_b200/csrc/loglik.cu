// Collapsed joint log-likelihood log p(w, z), split as in Figure 11 into a word
// part and a document part (Dirichlet-multinomial closed form):
//   word = K lgamma(V beta) + sum_{n_kw>0} [lgamma(n_kw+beta) - lgamma(beta)] - sum_k lgamma(n_k + V beta)
//   doc  = D lgamma(K alpha) + sum_{n_kd>0} [lgamma(n_kd+alpha) - lgamma(alpha)] - sum_d lgamma(n_d + K alpha)
// Each CTA writes one partial sum; a last kernel adds the partials in a fixed order.
#include <algorithm>
#include <cmath>
#include <type_traits>

#include "lda_device.cuh"
#include "lda_internal.cuh"

namespace lda {

constexpr int LL_BLOCKS = 592;  // of 256 threads and more
// Counts below this take lgamma(count + prior) - lgamma(prior) from a table filled with the same expression: same
// values as calling lgamma() per entry.
constexpr int LL_TABLE = 512;

// Word part.  A warp takes up to 32 consecutive words, its lanes their sizes at once (rows of a few entries, most of
// them, would otherwise cost a chain of reads each); rows of more than LL_ROW entries are left and taken in
// pieces of LL_ROW by all warps: `longer` lists the words that can have one.
constexpr int LL_ROW = ALIAS_MID_MAX;
struct LlWords {
    double lg_beta;
    int32_t per_warp;          // words a warp takes at a time
    const int32_t* longer;     // [n_longer]
    int32_t n_longer;
    const double* tab;         // [LL_TABLE] lgamma(c + beta) - lgamma(beta)
};
// The share of CTA `block` of `blocks`; the CTA's sum, on every thread.
__device__ __forceinline__ double ll_word_part(const View& v, const LlWords& a, int block, int blocks, double* small, double* tmp)
{
    for (int c = threadIdx.x; c < LL_TABLE; c += blockDim.x) small[c] = a.tab[c];
    __syncthreads();
    const int warps = (blocks * (int)blockDim.x) >> 5, lane = threadIdx.x & 31;
    const int thread = block * (int)blockDim.x + (int)threadIdx.x, warp = thread >> 5;
    double s = 0.0;
    auto add = [&](int32_t at) {
        const uint32_t c = v.wk_count[at];
        s += c < (uint32_t)LL_TABLE ? small[c] : lgamma((double)c + v.beta) - a.lg_beta;
    };
    for (int32_t wb = warp * a.per_warp; wb < v.V; wb += warps * a.per_warp) {
        int32_t n_mine = 0, r_mine = 0;
        if (lane < a.per_warp && wb + lane < v.V) {
            n_mine = v.wk_nnz[wb + lane];
            r_mine = v.row_start[wb + lane];
        }
        for (uint32_t some = __ballot_sync(0xFFFFFFFFu, n_mine > 0 && n_mine <= LL_ROW); some; some &= some - 1) {
            const int src = __ffs((int)some) - 1;
            const int32_t n = __shfl_sync(0xFFFFFFFFu, n_mine, src), r0 = __shfl_sync(0xFFFFFFFFu, r_mine, src);
            for (int32_t j = lane; j < n; j += 32) add(r0 + j);
        }
    }
    const int32_t pieces = (v.K + LL_ROW - 1) / LL_ROW;
    for (int64_t i = warp; i < (int64_t)a.n_longer * pieces; i += warps) {
        const int32_t w = a.longer[i / pieces], n = v.wk_nnz[w], j0 = (int32_t)(i % pieces) * LL_ROW;
        if (n <= LL_ROW || j0 >= n) continue;
        const int32_t r0 = v.row_start[w], j1 = min(n, j0 + LL_ROW);
        for (int32_t j = j0 + lane; j < j1; j += 32) add(r0 + j);
    }
    for (int32_t k = thread; k < v.K; k += blocks * (int)blockDim.x) s -= lgamma((double)v.nk[k] + v.Vbeta);
    return block_reduce_sum<double>(s, tmp);
}

__global__ void __launch_bounds__(256) k_ll_word(View v, LlWords a, double* __restrict__ out)
{
    __shared__ double tmp[32];
    __shared__ double small[LL_TABLE];
    const double s = ll_word_part(v, a, (int)blockIdx.x, (int)gridDim.x, small, tmp);
    if (threadIdx.x == 0) out[blockIdx.x] = s;
}

__global__ void k_sum_nnz(const int32_t* __restrict__ a, int64_t n, unsigned long long* out)
{
    __shared__ unsigned long long tmp[32];
    unsigned long long s = 0;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        s += (unsigned long long)a[i];
    s = block_reduce_sum<unsigned long long>(s, tmp);
    if (threadIdx.x == 0 && s) atomicAdd(out, s);
}

// Tables in device memory, filled once per corpus: [0, LL_TABLE) holds lgamma(c + alpha) - lgamma(alpha),
// [LL_TABLE, 2 LL_TABLE) lgamma(n + K alpha), [2 LL_TABLE, 3 LL_TABLE) lgamma(c + beta) - lgamma(beta).
__global__ void k_ll_fill_tables(View v, double lg_alpha, double lg_beta, double* __restrict__ tab)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x, c = i % LL_TABLE;
    if (i < LL_TABLE) tab[i] = lgamma((double)c + v.alpha) - lg_alpha;
    else if (i < 2 * LL_TABLE) tab[i] = lgamma((double)c + v.Kalpha);
    else if (i < 3 * LL_TABLE) tab[i] = lgamma((double)c + v.beta) - lg_beta;
}

// lgamma() for the rare count beyond the tables, kept out of line so that the kernel below fits the
// register budget of a full multiprocessor.
__device__ __noinline__ double lgamma_out_of_line(double x) { return lgamma(x); }

// Document part.  n_kd is not kept between sweeps (the MH step builds it per tile of documents
// and drops it), so it is built here the same way and by the same shape of kernel as pass 2 of the
// MH step: one CTA per tile of whole documents, a thread owns DOC_TILE_ROUNDS tokens, inserts their
// topics into the documents' hashed tables in shared memory, and the CTA then adds up
// lgamma(n_kd + alpha) - lgamma(alpha) over the filled slots and -lgamma(n_d + K alpha) per document.
// One partial sum per tile (a second kernel adds them in a fixed order) and the number of filled
// slots, nnz(n_kd).
template <typename T, int THREADS>
__device__ __forceinline__ void ll_doc_tile(const View& v, int tile, const int32_t* __restrict__ tiles, double lg_alpha,
                                            const double* __restrict__ tab, double* __restrict__ tile_part,
                                            uint32_t* __restrict__ tile_nnz, uint32_t* doc_smem, double* tmp)
{
    constexpr int cap = DOC_TILE_ROUNDS * THREADS;
    uint32_t* slots = doc_smem;                                                            // [DK_SLOTS_PER_TOKEN * cap]
    int32_t* soff = reinterpret_cast<int32_t*>(slots + DK_SLOTS_PER_TOKEN * cap);          // [cap + 1]
    const int tid = threadIdx.x;
    const int32_t s0 = tiles[2 * tile], s1 = tiles[2 * tile + 1];
    const int32_t nseg = s1 - s0;
    const int32_t base = v.doc_off[s0];
    const int32_t cnt = v.doc_off[s1] - base;
    const T* zbm = reinterpret_cast<const T*>(v.zbm);
    uint32_t z[DOC_TILE_ROUNDS];
#pragma unroll
    for (int r = 0; r < DOC_TILE_ROUNDS; ++r) {
        const int j = tid + r * THREADS;
        z[r] = 0;
        if (j < cnt) z[r] = (uint32_t)__ldcg(zbm + 2 * (size_t)__ldcs(v.bm_of_tok + base + j));
    }
    for (int j = tid; j <= nseg; j += THREADS) soff[j] = v.doc_off[s0 + j] - base;
    const uint4 empty4 = make_uint4(DK_EMPTY, DK_EMPTY, DK_EMPTY, DK_EMPTY);
    for (int j = tid; j < cnt * (DK_SLOTS_PER_TOKEN / 4); j += THREADS) reinterpret_cast<uint4*>(slots)[j] = empty4;
    __syncthreads();
#pragma unroll
    for (int r = 0; r < DOC_TILE_ROUNDS; ++r) {
        const int j = tid + r * THREADS;
        if (j < cnt) {
            int lo = 0, hi = nseg;  // last document with soff[doc] <= j
            while (hi - lo > 1) {
                const int mid = (lo + hi) >> 1;
                if (soff[mid] <= j) lo = mid; else hi = mid;
            }
            const int32_t first = soff[lo], len = soff[lo + 1] - first;
            if (z[r] >= (uint32_t)v.K) atomicOr(v.err, ERR_TOPIC_RANGE);
            else if (dk_insert(slots + DK_SLOTS_PER_TOKEN * first, DK_SLOTS_PER_TOKEN * (uint32_t)len, z[r],
                               v.count_bits) == DK_EMPTY)
                atomicOr(v.err, ERR_ROW_OVERFLOW);
        }
    }
    __syncthreads();
    const uint32_t cmask = (1u << v.count_bits) - 1u;
    double s = 0.0;
    uint32_t filled = 0;
    for (int j = tid; j < cnt; j += THREADS) {  // a token's worth of slots at a time
        const uint4 e4 = reinterpret_cast<const uint4*>(slots)[j];
        const uint32_t e[4] = {e4.x, e4.y, e4.z, e4.w};
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            if (e[q] != DK_EMPTY) {
                const uint32_t c = e[q] & cmask;
                s += c < (uint32_t)LL_TABLE ? __ldg(tab + c) : lgamma_out_of_line((double)c + v.alpha) - lg_alpha;
                ++filled;
            }
        }
    }
    for (int d = tid; d < nseg; d += THREADS) {
        const int32_t len = soff[d + 1] - soff[d];
        if (len > 0) s -= len < LL_TABLE ? __ldg(tab + LL_TABLE + len) : lgamma_out_of_line((double)len + v.Kalpha);
    }
    s = block_reduce_sum<double>(s, tmp);
    if (tid == 0) tile_part[tile] = s;
    __syncthreads();
    filled = block_reduce_sum<uint32_t>(filled, reinterpret_cast<uint32_t*>(tmp));
    if (tid == 0) tile_nnz[tile] = filled;
}

template <typename T, int THREADS>
__global__ void __launch_bounds__(THREADS, 1536 / THREADS)
k_ll_doc_tiles(View v, const int32_t* __restrict__ tiles, double lg_alpha, const double* __restrict__ tab,
               double* __restrict__ tile_part, uint32_t* __restrict__ tile_nnz)
{
    extern __shared__ __align__(16) uint32_t doc_smem[];
    __shared__ double tmp[32];
    ll_doc_tile<T, THREADS>(v, (int)blockIdx.x, tiles, lg_alpha, tab, tile_part, tile_nnz, doc_smem, tmp);
}

// Adds the tiles' partial sums: CTA b takes the b-th run of `per` consecutive tiles, always in the same order.
__global__ void __launch_bounds__(256) k_ll_sum_tiles(const double* __restrict__ tile_part,
                                                      const uint32_t* __restrict__ tile_nnz, int32_t n_tiles, int32_t per,
                                                      double* __restrict__ out, uint32_t* __restrict__ nnz_out)
{
    __shared__ double tmp[32];
    const int32_t t0 = blockIdx.x * per, t1 = min(n_tiles, t0 + per);
    double s = 0.0;
    unsigned long long filled = 0;
    for (int32_t t = t0 + threadIdx.x; t < t1; t += blockDim.x) {
        s += tile_part[t];
        filled += tile_nnz[t];
    }
    s = block_reduce_sum<double>(s, tmp);
    if (threadIdx.x == 0) out[blockIdx.x] = s;
    __syncthreads();
    filled = block_reduce_sum<unsigned long long>(filled, reinterpret_cast<unsigned long long*>(tmp));
    if (threadIdx.x == 0) nnz_out[blockIdx.x] = (uint32_t)filled;  // nnz(n_kd) <= n_tokens < 2^31
}

// Documents longer than a tile, from their tables in device memory (launch_long_tables()): CTAs take them in turns.
__global__ void __launch_bounds__(512)
k_ll_doc_long(View v, int32_t n_long, double lg_alpha, const double* __restrict__ tab_lg, double* __restrict__ out,
              uint32_t* __restrict__ nnz_out)
{
    __shared__ double tmp[32];
    __shared__ double small[LL_TABLE];
    for (int c = threadIdx.x; c < LL_TABLE; c += blockDim.x) small[c] = tab_lg[c];
    __syncthreads();
    const uint32_t cmask = (1u << v.count_bits) - 1u;
    double s = 0.0;
    unsigned long long filled = 0;
    for (int32_t i = blockIdx.x; i < n_long; i += gridDim.x) {
        const LongDoc d = v.long_docs[i];
        const uint32_t* tab = v.dk_slots + d.slot;
        const uint32_t slots = d.dense ? (uint32_t)v.K : DK_SLOTS_PER_TOKEN * (uint32_t)d.len;
        const uint32_t none = d.dense ? 0u : DK_EMPTY, mask = d.dense ? 0xFFFFFFFFu : cmask;
#pragma unroll 4
        for (uint32_t j = threadIdx.x; j < slots; j += blockDim.x) {
            const uint32_t e = __ldcg(tab + j);
            if (e != none) {
                const uint32_t c = e & mask;
                s += c < (uint32_t)LL_TABLE ? small[c] : lgamma((double)c + v.alpha) - lg_alpha;
                ++filled;
            }
        }
        if (threadIdx.x == 0) s -= lgamma((double)d.len + v.Kalpha);
    }
    s = block_reduce_sum<double>(s, tmp);
    if (threadIdx.x == 0) out[blockIdx.x] = s;
    __syncthreads();
    filled = block_reduce_sum<unsigned long long>(filled, reinterpret_cast<unsigned long long*>(tmp));
    if (threadIdx.x == 0) nnz_out[blockIdx.x] = (uint32_t)filled;
}

// The partial sums of both parts, always in the same order, and the error word, to host memory.  One CTA.
struct LlSums {
    const double* word;
    int32_t n_word;
    const double* doc_a;
    const uint32_t* nnz_a;
    int32_t n_a;
    const double* doc_b;
    const uint32_t* nnz_b;
    int32_t n_b;
    const int* err;
    SweepReport* rep;
};
__device__ __forceinline__ void ll_finish(const LlSums& p, double* tmp, unsigned long long* tmp_n)
{
    double w = 0.0, d = 0.0;
    unsigned long long nnz = 0;
    for (int32_t i = threadIdx.x; i < p.n_word; i += blockDim.x) w += __ldcg(p.word + i);
    for (int32_t i = threadIdx.x; i < p.n_a; i += blockDim.x) {
        d += __ldcg(p.doc_a + i);
        nnz += __ldcg(p.nnz_a + i);
    }
    for (int32_t i = threadIdx.x; i < p.n_b; i += blockDim.x) {
        d += __ldcg(p.doc_b + i);
        nnz += __ldcg(p.nnz_b + i);
    }
    w = block_reduce_sum<double>(w, tmp);
    __syncthreads();
    d = block_reduce_sum<double>(d, tmp);
    nnz = block_reduce_sum<unsigned long long>(nnz, tmp_n);
    if (threadIdx.x == 0) {
        p.rep->ll_word = w;
        p.rep->ll_doc = d;
        p.rep->nnz_dk = nnz;
        p.rep->err = __ldcg(p.err);
    }
}
__global__ void __launch_bounds__(512) k_ll_finish(LlSums p)
{
    __shared__ double tmp[32];
    __shared__ unsigned long long tmp_n[32];
    ll_finish(p, tmp, tmp_n);
}

// Small corpora: all of it as one kernel.  Some CTAs take a tile of documents each, the others the word part, and
// the last one to be done adds the partial sums up (`arrived` counts them and is zero between calls).  Three
// kernels on two streams take the host nine calls, which is longer than a corpus of 10 000 tokens takes the device.
// The part of fewer CTAs comes first: behind more CTAs of the other than fit the GPU at once it would start late and be alone at
// the end (10^6 tokens in documents of 800, V = 5000, K = 3000: 51 us with the tiles first, 43.5 so, three kernels 44; in documents
// of 1400, V = 20 000, K = 12 000: 45.8, 37.3 and 41.6).
// As many CTAs per multiprocessor as with the tiles first; without the bound the compiler takes registers for one less.
template <typename T, int THREADS>
__global__ void __launch_bounds__(THREADS, THREADS == 1024 ? 1 : THREADS == 512 ? 3 : 1280 / THREADS)
k_ll_all(View v, const int32_t* __restrict__ tiles, int32_t n_tiles, double lg_alpha, const double* __restrict__ tab,
         double* __restrict__ tile_part, uint32_t* __restrict__ tile_nnz, LlWords words, double* __restrict__ word_part,
         LlSums sums, unsigned int* __restrict__ arrived)
{
    extern __shared__ __align__(16) uint32_t doc_smem[];
    __shared__ double tmp[32];
    __shared__ unsigned long long tmp_n[32];
    __shared__ bool last;
    const int n_word = (int)gridDim.x - n_tiles, first_tile = n_word < n_tiles ? n_word : 0, first_word = n_word < n_tiles ? 0 : n_tiles;
    const int tile = (int)blockIdx.x - first_tile, word = (int)blockIdx.x - first_word;
    if (0 <= tile && tile < n_tiles) {
        ll_doc_tile<T, THREADS>(v, tile, tiles, lg_alpha, tab, tile_part, tile_nnz, doc_smem, tmp);
    } else {
        const double s = ll_word_part(v, words, word, n_word, reinterpret_cast<double*>(doc_smem), tmp);
        if (threadIdx.x == 0) word_part[word] = s;
    }
    if (threadIdx.x == 0) {  // the partial sums are this thread's stores
        __threadfence();
        last = atomicAdd(arrived, 1u) + 1u == gridDim.x;
        if (last) *arrived = 0u;
        __threadfence();
    }
    __syncthreads();
    if (last) ll_finish(sums, tmp, tmp_n);
}

constexpr int LL_TILE_SUMS = 1024;  // partial sums the tiles' sums are folded into
constexpr int LL_ONE_KERNEL_TILES = 1024;  // up to this many tiles everything is one kernel
constexpr int LL_TILE_DIRECT = 4096;  // up to this many tiles the last kernel adds them up itself

static int long_ll_grid(const Ctx& c) { return std::max(1, std::min<int>(c.n_long_docs, LL_BLOCKS)); }

template <typename T>
static void launch_ll_tiles_t(Ctx& c, size_t smem, double lg_alpha, cudaStream_t stream)
{
    switch (c.doc_threads) {
        case 128: k_ll_doc_tiles<T, 128><<<c.n_doc_tiles, 128, smem, stream>>>(c.v, c.doc_tiles, lg_alpha, c.ll_tab, c.ll_tile_part, c.ll_tile_nnz); break;
        case 256: k_ll_doc_tiles<T, 256><<<c.n_doc_tiles, 256, smem, stream>>>(c.v, c.doc_tiles, lg_alpha, c.ll_tab, c.ll_tile_part, c.ll_tile_nnz); break;
        case 512: k_ll_doc_tiles<T, 512><<<c.n_doc_tiles, 512, smem, stream>>>(c.v, c.doc_tiles, lg_alpha, c.ll_tab, c.ll_tile_part, c.ll_tile_nnz); break;
        default: k_ll_doc_tiles<T, 1024><<<c.n_doc_tiles, 1024, smem, stream>>>(c.v, c.doc_tiles, lg_alpha, c.ll_tab, c.ll_tile_part, c.ll_tile_nnz); break;
    }
}
static void launch_ll_tiles(Ctx& c, size_t smem, double lg_alpha, cudaStream_t stream)
{
    if (c.wide_topics) launch_ll_tiles_t<int32_t>(c, smem, lg_alpha, stream);
    else launch_ll_tiles_t<uint16_t>(c, smem, lg_alpha, stream);
}

template <typename T>
static void launch_ll_all_t(Ctx& c, const LlWords& words, int n_word, const LlSums& sums, double lg_alpha, double* word_part)
{
    const size_t smem = doc_tile_smem_bytes(c.doc_tile, DK_SLOTS_PER_TOKEN);
    const int grid = c.n_doc_tiles + n_word;
    auto go = [&](auto threads) {
        constexpr int THREADS = decltype(threads)::value;
        static_assert(LL_TABLE * 8 <= DOC_TILE_ROUNDS * THREADS * 4 * DK_SLOTS_PER_TOKEN, "the word part's table fits in a tile's room");
        k_ll_all<T, THREADS><<<grid, THREADS, smem, c.stream>>>(c.v, c.doc_tiles, c.n_doc_tiles, lg_alpha, c.ll_tab, c.ll_tile_part,
                                                                c.ll_tile_nnz, words, word_part, sums, reinterpret_cast<unsigned int*>(c.red_i + 1));
    };
    switch (c.doc_threads) {
        case 128: go(std::integral_constant<int, 128>{}); break;
        case 256: go(std::integral_constant<int, 256>{}); break;
        case 512: go(std::integral_constant<int, 512>{}); break;
        default: go(std::integral_constant<int, 1024>{}); break;
    }
}

// Queues the word part (if asked for) and the document part, side by side, and the kernel that reports their sums.
static void queue_loglik(Ctx& c, bool word_part)
{
    double* part = c.red;  // [LL_WORD_PARTIALS + LL_DOC_PARTIALS]
    uint32_t* nnz = c.red_nnz;  // [LL_DOC_PARTIALS]
    const double lg_alpha = std::lgamma(c.alpha);
    int n_word = 0, n_a = 0, n_b = 0;
    const double* doc_a = part + LL_WORD_PARTIALS;
    const uint32_t* nnz_a = nnz;
    double* doc_b = part + LL_WORD_PARTIALS + LL_TILE_SUMS;
    uint32_t* nnz_b = nnz + LL_TILE_SUMS;
    const double lg_beta = std::lgamma(c.beta);
    if (!c.ll_tables_ready) {
        cudaMemsetAsync(c.red_i + 1, 0, 8, c.stream);  // k_ll_all's count of CTAs
        k_ll_fill_tables<<<3 * LL_TABLE / 64, 64, 0, c.stream>>>(c.v, lg_alpha, lg_beta, c.ll_tab);
        c.ll_tables_ready = true;
    }
    LlWords words{lg_beta, 32, c.alias_words[2], c.n_alias_words[2], c.ll_tab + 2 * LL_TABLE};
    if (word_part) {
        while (words.per_warp > 1 && c.V / words.per_warp < c.n_sm * 16) words.per_warp /= 2;
        n_word = (int)std::min<int64_t>(LL_BLOCKS, (c.V + 8 * (int64_t)words.per_warp - 1) / (8 * (int64_t)words.per_warp));
        // a warp per piece of a long row, a thread per topic
        const int64_t pieces = (int64_t)c.n_alias_words[2] * ((c.K + LL_ROW - 1) / LL_ROW);
        n_word = (int)std::min<int64_t>(LL_BLOCKS, std::max<int64_t>({(int64_t)n_word, (pieces + 7) / 8, ((int64_t)c.K + 255) / 256}));
    }
    if (word_part && !c.n_long_docs && c.n_doc_tiles > 0 && c.n_doc_tiles <= LL_ONE_KERNEL_TILES) {
        // as many threads as the word part has by itself (43 000 tokens, V = 435 000, ten sweeps and a look, three kernels against
        // one: 549.3 and 553.0 us with half as many, on another GPU 554.4 and 552.9 so)
        n_word = std::min<int>(LL_WORD_PARTIALS, (n_word * 256 + c.doc_threads - 1) / c.doc_threads);
        const LlSums sums{part, n_word, c.ll_tile_part, c.ll_tile_nnz, c.n_doc_tiles, doc_b, nnz_b, 0, c.v.err, c.report};
        if (c.wide_topics) launch_ll_all_t<int32_t>(c, words, n_word, sums, lg_alpha, part);
        else launch_ll_all_t<uint16_t>(c, words, n_word, sums, lg_alpha, part);
        return;
    }
    fork_streams(c);
    if (word_part) k_ll_word<<<n_word, 256, 0, c.side[0]>>>(c.v, words, part);
    if (c.n_long_docs) {
        n_b = long_ll_grid(c);
        launch_long_tables(c, c.side[1], false, -1);
        k_ll_doc_long<<<n_b, 512, 0, c.side[1]>>>(c.v, c.n_long_docs, lg_alpha, c.ll_tab, doc_b, nnz_b);
    }
    if (c.n_doc_tiles) {
        launch_ll_tiles(c, doc_tile_smem_bytes(c.doc_tile, DK_SLOTS_PER_TOKEN), lg_alpha, c.stream);
        if (c.n_doc_tiles <= LL_TILE_DIRECT) {
            doc_a = c.ll_tile_part;
            nnz_a = c.ll_tile_nnz;
            n_a = c.n_doc_tiles;
        } else {
            const int per = (c.n_doc_tiles + LL_TILE_SUMS - 1) / LL_TILE_SUMS;
            n_a = (c.n_doc_tiles + per - 1) / per;
            k_ll_sum_tiles<<<n_a, 256, 0, c.stream>>>(c.ll_tile_part, c.ll_tile_nnz, c.n_doc_tiles, per, part + LL_WORD_PARTIALS, nnz);
        }
    }
    join_streams(c);
    k_ll_finish<<<1, 512, 0, c.stream>>>(LlSums{part, n_word, doc_a, nnz_a, n_a, doc_b, nnz_b, n_b, c.v.err, c.report});
}

int launch_loglik(Ctx& c, double* out3_host)
{
    queue_loglik(c, true);
    if (cudaStreamSynchronize(c.stream) != cudaSuccess) return -1;
    // every document with tokens contributes lgamma(K alpha) - lgamma(n_d + K alpha); an empty one nothing
    const double lw = (double)c.K * std::lgamma(c.v.Vbeta) + c.report->ll_word;
    const double ld = (double)c.n_nonempty_docs * std::lgamma(c.v.Kalpha) + c.report->ll_doc;
    out3_host[0] = lw + ld;
    out3_host[1] = lw;
    out3_host[2] = ld;
    return 0;
}

// nnz(n_kw) and nnz(n_kd) of the current assignments (the latter by the document part's kernels).
int launch_count_nnz(Ctx& c, int64_t* nnz_wk_host, int64_t* nnz_dk_host)
{
    unsigned long long* acc = (unsigned long long*)c.red_i;
    cudaMemsetAsync(acc, 0, 8, c.stream);
    k_sum_nnz<<<296, 256, 0, c.stream>>>(c.v.wk_nnz, c.V, acc);
    queue_loglik(c, false);
    unsigned long long h = 0;
    cudaMemcpyAsync(&h, acc, 8, cudaMemcpyDeviceToHost, c.stream);
    cudaStreamSynchronize(c.stream);
    *nnz_wk_host = (int64_t)h;
    *nnz_dk_host = (int64_t)c.report->nnz_dk;
    return 3;
}

void set_loglik_smem_limits()
{
    const int doc_bytes = (int)doc_tile_smem_bytes(DOC_TILE_MAX, DK_SLOTS_PER_TOKEN);
    cudaFuncSetAttribute(k_ll_doc_tiles<uint16_t, 1024>, cudaFuncAttributeMaxDynamicSharedMemorySize, doc_bytes);
    cudaFuncSetAttribute(k_ll_doc_tiles<int32_t, 1024>, cudaFuncAttributeMaxDynamicSharedMemorySize, doc_bytes);
    cudaFuncSetAttribute(k_ll_all<uint16_t, 1024>, cudaFuncAttributeMaxDynamicSharedMemorySize, doc_bytes);
    cudaFuncSetAttribute(k_ll_all<int32_t, 1024>, cudaFuncAttributeMaxDynamicSharedMemorySize, doc_bytes);
}

}  // namespace lda
