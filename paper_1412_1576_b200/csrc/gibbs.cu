// Exact-conditional yardstick (Section 3, Eq. 1; the split of Section 4, Eq. 3): a frozen sweep in
// which every token draws its new topic from the collapsed conditional itself instead of running a
// short MH chain towards it.  It is what the MH sweep is measured against (log-likelihood per sweep),
// not a fast path: a token costs O(K_d log K_w + log K).
//
//   p(k) ~ n_kd'(n_kw'+beta)/(n_k'+V beta)  +  alpha (n_kw'+beta)/(n_k'+V beta)      (primes: token removed)
//
// Every term is floored to a multiple of 2^-44 and the draw is the inverse CDF over these integer
// masses -- the document term's topics first (ascending), then all topics -- so the result does
// not depend on the order the terms are added in.  The second term differs between two tokens of
// a word only at the token's own topic, so its running sums over k are built once per word and
// sweep; the first term walks the document's sorted n_kd row (export.cu) and looks n_kw up in the
// word's sorted row.  One Philox word per token and sweep: counter (token, sweep, 0, 2).
#include <algorithm>
#include <type_traits>

#include "lda_device.cuh"
#include "lda_internal.cuh"

namespace lda {

typedef unsigned long long ull;
constexpr double GIBBS_FIXED_ONE = 17592186044416.0;  // 2^44

__device__ __forceinline__ ull gibbs_doc_term(double beta, double Vbeta, int32_t n_kd, int32_t n_kw, int32_t n_k)
{
    const double x = __ddiv_rn(__dmul_rn((double)n_kd, __dadd_rn((double)n_kw, beta)), __dadd_rn((double)n_k, Vbeta));
    return __double2ull_rz(__dmul_rn(x, GIBBS_FIXED_ONE));
}

__device__ __forceinline__ ull gibbs_prior_term(double alpha, double beta, double Vbeta, int32_t n_kw, int32_t n_k)
{
    const double x = __ddiv_rn(__dmul_rn(alpha, __dadd_rn((double)n_kw, beta)), __dadd_rn((double)n_k, Vbeta));
    return __double2ull_rz(__dmul_rn(x, GIBBS_FIXED_ONE));
}

constexpr int WORD_OF_RUN = 512;
// word_of[i] = word of the token with document-order index i (the layout keeps tokens by word).  A CTA finds
// the words of its run of tokens first; a token then searches among those.
__global__ void __launch_bounds__(256) k_word_of_tokens(View v, int32_t* __restrict__ word_of)
{
    constexpr int RUN = WORD_OF_RUN;
    __shared__ int32_t range[2];
    const int32_t p0 = blockIdx.x * RUN, p1 = min(v.N - p0, RUN) + p0;
    if (threadIdx.x < 2) {
        const int32_t p = threadIdx.x == 0 ? p0 : p1 - 1;
        int32_t lo = 0, hi = v.V;  // last word with word_off[word] <= p
        while (hi - lo > 1) {
            const int32_t mid = lo + ((hi - lo) >> 1);
            if (v.word_off[mid] <= p) lo = mid; else hi = mid;
        }
        range[threadIdx.x] = lo;
    }
    __syncthreads();
    for (int32_t p = p0 + (int32_t)threadIdx.x; p < p1; p += 256) {
        int32_t lo = range[0], hi = range[1] + 1;
        while (hi - lo > 1) {
            const int32_t mid = lo + ((hi - lo) >> 1);
            if (__ldg(v.word_off + mid) <= p) lo = mid; else hi = mid;
        }
        word_of[v.tok_orig[p]] = lo;
    }
}

// One CTA per word: running sums over k of the smoothing term under the frozen counts, and, where there is
// room for it, the word's n_kw as a dense row.
__global__ void __launch_bounds__(256) k_gibbs_prior_prefix(View v, ull* __restrict__ prefix, int32_t* __restrict__ matrix)
{
    extern __shared__ int32_t row_s[];  // [K] the word's n_kw as a dense row
    __shared__ ull scan_tmp[33];
    const int32_t w = blockIdx.x, K = v.K;
    for (int32_t k = threadIdx.x; k < K; k += blockDim.x) row_s[k] = 0;
    __syncthreads();
    const int32_t r0 = v.row_start[w], n = v.wk_nnz[w];
    for (int32_t j = threadIdx.x; j < n; j += blockDim.x) row_s[v.wk_topic[r0 + j]] = (int32_t)v.wk_count[r0 + j];
    __syncthreads();
    ull carry = 0;
    for (int32_t k0 = 0; k0 < K; k0 += blockDim.x) {
        const int32_t k = k0 + (int32_t)threadIdx.x;
        const ull term = k < K ? gibbs_prior_term(v.alpha, v.beta, v.Vbeta, row_s[k], v.nk[k]) : 0ull;
        ull total;
        const ull before = block_scan_excl<ull>(term, scan_tmp, total);
        if (k < K) {
            prefix[(size_t)w * K + k] = carry + before + term;
            if (matrix) matrix[(size_t)w * K + k] = row_s[k];
        }
        carry += total;
        __syncthreads();
    }
}

// n_kw[w][k] from the word's sorted row.
__device__ __forceinline__ int32_t word_count(const View& v, int32_t row0, int32_t nnz, uint32_t k)
{
    int32_t lo = 0, hi = nnz;
    while (lo < hi) {
        const int32_t mid = (lo + hi) >> 1;
        if (__ldg(v.wk_topic + row0 + mid) < k) lo = mid + 1; else hi = mid;
    }
    return (lo < nnz && __ldg(v.wk_topic + row0 + lo) == k) ? (int32_t)__ldg(v.wk_count + row0 + lo) : 0;
}

// One warp per `run_len` consecutive tokens (of one document or several).  What belongs to a token alone -- its
// Philox block, the smoothing term's correction and total, a draw from the smoothing term -- is a lane's work for
// 32 tokens at once; the document term of one token is the whole warp's, a lane per topic of the document: the
// document's row is read in order, the word's counts lie next to each other in `matrix`, and the running sums
// the draw needs are a warp scan.  (A lane per token, walking the document's row alone and searching the word's
// sorted row for every topic of it: 2.15 ms for 2 M tokens of 100-token documents, K = 100.)
// run_len: up to GIBBS_RUN, shorter where that would leave multiprocessors idle.
constexpr int GIBBS_RUN = 64;
template <typename T, bool MATRIX>
__global__ void __launch_bounds__(256)
k_gibbs_tokens(View v, const T* __restrict__ z, const int32_t* __restrict__ word_of, const long long* __restrict__ row_off,
               const int32_t* __restrict__ dk_topic, const int32_t* __restrict__ dk_count, const ull* __restrict__ prefix,
               const int32_t* __restrict__ matrix, int32_t* __restrict__ z_new, uint2 key, uint32_t sweep, int32_t run_len)
{
    constexpr uint32_t FULL = 0xFFFFFFFFu;
    const int lane = threadIdx.x & 31;
    const int64_t run = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int32_t K = v.K;
    int32_t i = (int32_t)min(run * run_len, (int64_t)v.N);
    const int32_t i_end = (int32_t)min((run + 1) * run_len, (int64_t)v.N);
    if (i >= i_end) return;
    int32_t d;
    {
        int32_t lo = 0, hi = v.D;  // last document with doc_off[document] <= i: it is not empty
        while (hi - lo > 1) {
            const int32_t mid = lo + ((hi - lo) >> 1);
            if (__ldg(v.doc_off + mid) <= i) lo = mid; else hi = mid;
        }
        d = lo;
    }
    while (i < i_end) {
        while (__ldg(v.doc_off + d + 1) <= i) ++d;
        const long long e0 = row_off[d];
        const int32_t rows = (int32_t)(row_off[d + 1] - e0);
        const int32_t n = min(32, min(i_end, __ldg(v.doc_off + d + 1)) - i);  // tokens of this turn, a lane each
        // the first 64 topics of the document stay in registers for all of them
        uint32_t k_r[2];
        int32_t c_r[2], n_r[2];
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const int32_t e = 32 * q + lane;
            k_r[q] = e < rows ? (uint32_t)__ldg(dk_topic + e0 + e) : 0u;
            c_r[q] = e < rows ? __ldg(dk_count + e0 + e) : 0;
            n_r[q] = __ldg(v.nk + k_r[q]);
        }
        uint32_t z_l = 0, r_l = 0, pick_l = (uint32_t)(K - 1);
        int32_t w_l = 0, row_l = 0, nnz_l = 0;
        long long delta_l = 0;
        ull prior_l = 0, x_l = 0;
        bool smooth_l = false;
        if (lane < n) {
            z_l = (uint32_t)z[i + lane];
            w_l = word_of[i + lane];
            int32_t n_zw;
            if (MATRIX) {
                n_zw = __ldg(matrix + (size_t)w_l * K + z_l);
            } else {
                row_l = v.row_start[w_l];
                nnz_l = v.wk_nnz[w_l];
                n_zw = word_count(v, row_l, nnz_l, z_l);
            }
            const int32_t n_z = __ldg(v.nk + z_l);
            delta_l = (long long)gibbs_prior_term(v.alpha, v.beta, v.Vbeta, n_zw - 1, n_z - 1) -
                      (long long)gibbs_prior_term(v.alpha, v.beta, v.Vbeta, n_zw, n_z);
            prior_l = (ull)((long long)__ldg(prefix + (size_t)w_l * K + K - 1) + delta_l);
            r_l = philox4x32_10(make_uint4(v.tok_base + (uint32_t)(i + lane), sweep, 0u, 2u), key).x;
        }
        for (int t = 0; t < n; ++t) {
            const uint32_t z0 = __shfl_sync(FULL, z_l, t);
            const int32_t w = __shfl_sync(FULL, w_l, t);
            const int32_t row0 = MATRIX ? 0 : __shfl_sync(FULL, row_l, t), nnz = MATRIX ? 0 : __shfl_sync(FULL, nnz_l, t);
            const int32_t* line = matrix + (size_t)w * K;
            // a topic's mass in the document term
            auto mass = [&](uint32_t k, int32_t c, int32_t n_k) -> ull {
                const int32_t own = (k == z0), n_kd = c - own;
                if (n_kd <= 0) return 0ull;
                const int32_t n_kw = MATRIX ? __ldg(line + k) : word_count(v, row0, nnz, k);
                return gibbs_doc_term(v.beta, v.Vbeta, n_kd, n_kw - own, n_k - own);
            };
            auto round_mass = [&](int32_t q) -> ull {
                const int32_t e = 32 * q + lane;
                if (e >= rows) return 0ull;
                const uint32_t k = (uint32_t)__ldg(dk_topic + e0 + e);
                return mass(k, __ldg(dk_count + e0 + e), __ldg(v.nk + k));
            };
            const ull m0 = mass(k_r[0], c_r[0], n_r[0]), m1 = rows > 32 ? mass(k_r[1], c_r[1], n_r[1]) : 0ull;
            ull mine = m0 + m1;
            for (int32_t q = 2; 32 * q < rows; ++q) mine += round_mass(q);
            const ull sum_doc = warp_reduce_sum<ull>(mine);
            const ull total = sum_doc + __shfl_sync(FULL, prior_l, t);
            const ull x = __umul64hi(total, (ull)__shfl_sync(FULL, r_l, t) << 32);  // floor(total * r / 2^32)
            if (x >= sum_doc) {  // from the smoothing term, later
                if (lane == t) {
                    smooth_l = true;
                    x_l = x - sum_doc;
                }
                continue;
            }
            ull before = 0;
            for (int32_t q = 0; 32 * q < rows; ++q) {
                const ull m = q == 0 ? m0 : q == 1 ? m1 : round_mass(q);
                const ull cum = before + warp_scan_incl<ull>(m);
                const uint32_t over = __ballot_sync(FULL, cum > x);
                if (over) {
                    const int src = __ffs((int)over) - 1;
                    const uint32_t k = q == 0 ? k_r[0] : q == 1 ? k_r[1] : (uint32_t)__ldg(dk_topic + e0 + 32 * q + src);
                    const uint32_t chosen = __shfl_sync(FULL, k, src);
                    if (lane == t) pick_l = chosen;
                    break;
                }
                before = __shfl_sync(FULL, cum, 31);
            }
        }
        if (smooth_l) {
            // running sums of the word, set right at the token's own topic: the first that exceeds x
            const ull* pre = prefix + (size_t)w_l * K;
            int32_t lo = 0, hi = K - 1;
            while (lo < hi) {
                const int32_t mid = (lo + hi) >> 1;
                const ull c = (ull)((long long)__ldg(pre + mid) + ((uint32_t)mid >= z_l ? delta_l : 0ll));
                if (c > x_l) hi = mid; else lo = mid + 1;
            }
            pick_l = (uint32_t)lo;
        }
        if (lane < n) z_new[i + lane] = (int32_t)pick_l;
        i += n;
    }
}

}  // namespace lda

using namespace lda;

int lda::gibbs_sweep(Ctx& c, int32_t iters)
{
    const View& v = c.v;
    const size_t n1 = (size_t)std::max<int64_t>(c.N, 1);
    int32_t* word_of = nullptr;
    int32_t* z_new = nullptr;
    ull* prefix = nullptr;
    int32_t* matrix = nullptr;
    int rc = LDA_OK;
    if (!tmp_alloc(c, &word_of, n1 * 4) || !tmp_alloc(c, &z_new, n1 * 4) || !tmp_alloc(c, &prefix, (size_t)c.V * c.K * 8))
        rc = LDA_ENOMEM;
    // half as much again for n_kw as a matrix; without it the counts are looked up in the sorted rows
    if (rc == LDA_OK && !tmp_alloc(c, &matrix, (size_t)c.V * c.K * 4)) matrix = nullptr;
    const uint2 key = make_uint2((uint32_t)c.seed, (uint32_t)(c.seed >> 32));
    if (rc == LDA_OK && c.N > 0) k_word_of_tokens<<<(unsigned)((c.N + WORD_OF_RUN - 1) / WORD_OF_RUN), 256, 0, c.stream>>>(v, word_of);
    for (int32_t it = 0; rc == LDA_OK && it < iters && c.N > 0; ++it) {
        DkCsr r;
        if ((rc = build_dk_csr(c, r, false))) break;  // also leaves z in document order in the record array
        k_gibbs_prior_prefix<<<c.V, 256, (size_t)c.K * 4, c.stream>>>(v, prefix, matrix);
        int32_t run_len = GIBBS_RUN;
        while (run_len > 4 && c.N / run_len < (int64_t)c.n_sm * 32) run_len /= 2;
        const unsigned grid = (unsigned)((c.N + 8 * run_len - 1) / (8 * run_len));
        auto tokens = [&](auto z) {
            using T = std::remove_const_t<std::remove_pointer_t<decltype(z)>>;
            const auto kernel = matrix ? k_gibbs_tokens<T, true> : k_gibbs_tokens<T, false>;
            kernel<<<grid, 256, 0, c.stream>>>(v, z, word_of, r.row_off, r.topic, r.count, prefix, matrix, z_new, key, c.sweep, run_len);
        };
        if (c.wide_topics) tokens(reinterpret_cast<const int32_t*>(v.rec));
        else tokens(reinterpret_cast<const uint16_t*>(v.rec));
        launch_spread_assignments(c, z_new, false);
        rebuild_counts(c);
        c.sweep += 1;
        if (cudaStreamSynchronize(c.stream) != cudaSuccess) rc = LDA_ECUDA;
        free_dk_csr(c, r);
    }
    if (iters > 0 && c.N == 0) c.sweep += (uint32_t)iters;
    launch_set_state(c);  // the device's sweep counter follows
    cudaStreamSynchronize(c.stream);
    raw_free(c, word_of);
    raw_free(c, z_new);
    raw_free(c, prefix);
    raw_free(c, matrix);
    if (rc == LDA_OK && cudaGetLastError() != cudaSuccess) rc = LDA_ECUDA;
    return rc;
}

void lda::set_gibbs_smem_limits()
{
    cudaFuncSetAttribute(k_gibbs_prior_prefix, cudaFuncAttributeMaxDynamicSharedMemorySize, GIBBS_MAX_K * 4);
}
