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

// a / b for one b and many a: y is 1/b rounded to nearest.  Two steps of Markstein's correction (IBM J. Res. Dev. 34(1),
// 1990): the first makes the quotient faithful, the second, from a faithful quotient and a correctly rounded
// reciprocal, the correctly rounded one -- the value of __ddiv_rn(a, b) where nothing over- or underflows.
__device__ __forceinline__ double div_by(double a, double b, double y)
{
    double q = __dmul_rn(a, y);
    q = __fma_rn(__fma_rn(-b, q, a), y, q);
    return __fma_rn(__fma_rn(-b, q, a), y, q);
}

// One warp per `run_len` consecutive tokens (of one document or several), at most 32 of a document at a time.  What
// belongs to a token alone -- its Philox block, its own topic's mass, the smoothing term's correction and total, a draw
// from the smoothing term -- is a lane's work for all of them at once.  The document term of a token is the work of LANES
// lanes, 32 / LANES tokens side by side: each lane adds up its part of the document's row (the first GIBBS_KEPT / LANES
// topics stay in registers, with the reciprocals of their denominators), a few shuffle steps make the running sums, and
// the lane in whose part the draw falls finds the topic there.  Bound by the latency of the counts' reads: more
// registers than three or four CTAs per multiprocessor leave cost more than they save.  16 lanes suit rows that stay in
// registers, 32 longer ones: 2 M tokens of 100-token documents, K = 100: 517 and 559 us; 1.1 M of 808, rows of
// 300 topics: 2141 and 1686 us (a warp per token that sums and then scans: 670 and 2199; eight lanes: 615 and 3100; the
// loads of several topics that are not kept in flight together: slower, by their registers).
// run_len: up to GIBBS_RUN, shorter where that would leave multiprocessors idle.
constexpr int GIBBS_RUN = 64;
constexpr int GIBBS_KEPT = 64;
template <bool MATRIX, int LANES>
__global__ void __launch_bounds__(256, LANES == 32 ? 4 : 3)
k_gibbs_tokens(View v, const uint16_t* __restrict__ z, const int32_t* __restrict__ word_of, const long long* __restrict__ row_off,
               const int32_t* __restrict__ dk_topic, const int32_t* __restrict__ dk_count, const ull* __restrict__ prefix,
               const int32_t* __restrict__ matrix, int32_t* __restrict__ z_new, PhiloxSeed key, uint32_t sweep, int32_t run_len)
{
    constexpr uint32_t FULL = 0xFFFFFFFFu;
    constexpr int TOKENS = 32 / LANES, KEPT = GIBBS_KEPT / LANES;
    constexpr ull NOT_SMOOTH = ~0ull;
    const int lane = threadIdx.x & 31, sub = lane % LANES, group = lane / LANES;
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
        const int32_t n = min(32, min(i_end, __ldg(v.doc_off + d + 1)) - i);  // tokens of this turn
        // this lane's part of the row: entries [e, e + part), fewer at its end
        const int32_t part = (rows + LANES - 1) / LANES, e = sub * part, mine_n = max(0, min(part, rows - e));
        uint32_t k_r[KEPT];
        int32_t c_r[KEPT];
        double b_r[KEPT], y_r[KEPT];  // denominator of a term in units of 2^-44, and its reciprocal
#pragma unroll
        for (int q = 0; q < KEPT; ++q) {
            if (q >= part) break;
            const bool in = q < mine_n;
            k_r[q] = in ? (uint32_t)__ldg(dk_topic + e0 + e + q) : 0u;
            c_r[q] = in ? __ldg(dk_count + e0 + e + q) : 0;
            b_r[q] = __dmul_rn(__dadd_rn((double)__ldg(v.nk + k_r[q]), v.Vbeta), 1.0 / GIBBS_FIXED_ONE);
            y_r[q] = __drcp_rn(b_r[q]);
        }
        uint32_t z_l = 0, r_l = 0;
        int32_t w_l = 0, row_l = 0, nnz_l = 0;
        long long delta_l = 0;
        ull prior_l = 0, own_l = 0, x_l = NOT_SMOOTH;
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
            // the token's own topic is in the row; its mass there, the token removed
            int32_t lo = 0, hi = rows - 1;
            while (lo < hi) {
                const int32_t mid = (lo + hi) >> 1;
                if ((uint32_t)__ldg(dk_topic + e0 + mid) < z_l) lo = mid + 1; else hi = mid;
            }
            const int32_t n_zd = __ldg(dk_count + e0 + lo) - 1;
            if (n_zd > 0) own_l = gibbs_doc_term(v.beta, v.Vbeta, n_zd, n_zw - 1, n_z - 1);
        }
        for (int t0 = 0; t0 < n; t0 += TOKENS) {
            const int t = min(t0 + group, n - 1);  // the groups past the last token repeat it
            const uint32_t z0 = __shfl_sync(FULL, z_l, t);
            const ull own = __shfl_sync(FULL, own_l, t), prior = __shfl_sync(FULL, prior_l, t);
            const uint32_t r = __shfl_sync(FULL, r_l, t);
            const int32_t w = __shfl_sync(FULL, w_l, t);
            const int32_t row0 = MATRIX ? 0 : __shfl_sync(FULL, row_l, t), nnz = MATRIX ? 0 : __shfl_sync(FULL, nnz_l, t);
            const int32_t* line = matrix + (size_t)w * K;
            auto count_of = [&](uint32_t k) { return MATRIX ? __ldg(line + k) : word_count(v, row0, nnz, k); };
            auto later = [&](int32_t q) -> ull {  // an entry that is not kept
                const uint32_t k = (uint32_t)__ldg(dk_topic + e0 + e + q);
                if (k == z0) return own;
                return gibbs_doc_term(v.beta, v.Vbeta, __ldg(dk_count + e0 + e + q), count_of(k), __ldg(v.nk + k));
            };
            ull m[KEPT];
            ull mine = 0;
#pragma unroll
            for (int q = 0; q < KEPT; ++q) {
                if (q >= part) break;
                const double a = __dmul_rn((double)c_r[q], __dadd_rn((double)count_of(k_r[q]), v.beta));
                const ull term = __double2ull_rz(div_by(a, b_r[q], y_r[q]));
                m[q] = q >= mine_n ? 0ull : k_r[q] == z0 ? own : term;
                mine += m[q];
            }
            for (int32_t q = KEPT; q < mine_n; ++q) mine += later(q);
            ull cum = mine;  // running sum over the group's lanes
#pragma unroll
            for (int o = 1; o < LANES; o *= 2) {
                const ull up = __shfl_up_sync(FULL, cum, o, LANES);
                if (sub >= o) cum += up;
            }
            const ull sum_doc = __shfl_sync(FULL, cum, LANES - 1, LANES);
            const ull total = sum_doc + prior;
            const ull x = __umul64hi(total, (ull)r << 32);  // floor(total * r / 2^32)
            // a draw from the smoothing term is left to the token's lane
            const ull rest = __shfl_sync(FULL, x >= sum_doc ? x - sum_doc : NOT_SMOOTH, lane % TOKENS * LANES);
            if (lane / TOKENS * TOKENS == t0) x_l = rest;
            if (cum > x && cum - mine <= x && t0 + group < n) {
                ull left = x - (cum - mine);  // the first entry whose running sum exceeds it
                uint32_t chosen = 0;
                bool found = false;
#pragma unroll
                for (int q = 0; q < KEPT; ++q) {
                    if (q >= part) break;
                    if (!found) {
                        chosen = k_r[q];
                        found = left < m[q];
                        left -= found ? 0ull : m[q];
                    }
                }
                for (int32_t q = KEPT; !found; ++q) {
                    const ull mass = later(q);
                    chosen = (uint32_t)__ldg(dk_topic + e0 + e + q);
                    found = left < mass || q + 1 >= mine_n;
                    left -= mass;
                }
                z_new[i + t] = (int32_t)chosen;
            }
        }
        if (lane < n && x_l != NOT_SMOOTH) {
            // running sums of the word, set right at the token's own topic: the first that exceeds x
            const ull* pre = prefix + (size_t)w_l * K;
            int32_t lo = 0, hi = K - 1;
            while (lo < hi) {
                const int32_t mid = (lo + hi) >> 1;
                const ull c = (ull)((long long)__ldg(pre + mid) + ((uint32_t)mid >= z_l ? delta_l : 0ll));
                if (c > x_l) hi = mid; else lo = mid + 1;
            }
            z_new[i + lane] = lo;
        }
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
    const PhiloxSeed key(c.seed);
    if (rc == LDA_OK && c.N > 0) k_word_of_tokens<<<(unsigned)((c.N + WORD_OF_RUN - 1) / WORD_OF_RUN), 256, 0, c.stream>>>(v, word_of);
    for (int32_t it = 0; rc == LDA_OK && it < iters && c.N > 0; ++it) {
        DkCsr r;
        rc = build_dk_csr(c, r, false);  // also leaves z in document order in the record array
        if (rc == LDA_ENOMEM && matrix) {  // the rows are needed, the matrix is not
            cudaStreamSynchronize(c.stream);
            raw_free(c, matrix);
            matrix = nullptr;
            rc = build_dk_csr(c, r, false);
        }
        if (rc) break;
        k_gibbs_prior_prefix<<<c.V, 256, (size_t)c.K * 4, c.stream>>>(v, prefix, matrix);
        int32_t run_len = GIBBS_RUN;
        while (run_len > 4 && c.N / run_len < (int64_t)c.n_sm * 32) run_len /= 2;
        const unsigned grid = (unsigned)((c.N + 8 * run_len - 1) / (8 * run_len));
        const bool long_rows = r.total > c.D * (long long)GIBBS_KEPT;
        const auto kernel = matrix ? (long_rows ? k_gibbs_tokens<true, 32> : k_gibbs_tokens<true, 16>)
                                   : (long_rows ? k_gibbs_tokens<false, 32> : k_gibbs_tokens<false, 16>);
        kernel<<<grid, 256, 0, c.stream>>>(v, reinterpret_cast<const uint16_t*>(v.rec), word_of, r.row_off, r.topic, r.count, prefix, matrix,
                                           z_new, key, c.sweep, run_len);
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
