// Word-proposal tables (Section 4.2): the word-proposal (n_kw + beta)/(n_k + V*beta)
// is sampled as a mixture of a sparse term over the word's nonzero n_kw (one alias
// table per word, O(K_w) to build) and a dense term beta/(n_k + V*beta) whose alias
// table is shared by all words.
//
// Alias construction is cooperative (a few lanes to a cluster of CTAs per row)
// and exact in integers, so the table is a function of the counts alone:
//   - fixed-point weights wt_i = floor(weight_i * 2^44), W44 = sum wt_i;
//   - pre-shift sh = max(0, bitlen(W44) + bitlen(n) - 62), w_i = wt_i >> sh, W = sum w_i;
//   - bin capacity W, item i brings a_i = n * w_i; a_i <= W is "light", else "heavy";
//   - with D_l = deficits of the lights before light l (ascending item order) and
//     E_m = surpluses of heavies 0..m, light l is filled by heavy #{m : E_m <= D_l};
//     heavy m keeps W + E_m - D_lam with lam = min{l : D_l >= E_m} and is filled by
//     heavy m+1 (or is full).
// This is the closed form of "fill lights in order from the current heavy item; an
// exhausted heavy item becomes a bin topped up by the next heavy item".
#include <cooperative_groups.h>

#include <algorithm>
#include <type_traits>

#include "lda_device.cuh"
#include "lda_internal.cuh"

namespace lda {

typedef unsigned long long ull;

// The threads that build one row together: a warp, a CTA, or a cluster of CTAs.
enum GroupKind { WARP, CTA, CLUSTER };
constexpr int GROUP_SMEM = 99 + 6 + 6;  // 64-bit words of shared memory a CTA of a group needs (none for WARP)

template <GroupKind KIND>
struct Group {
    ull* smem;  // [GROUP_SMEM]
    __device__ __forceinline__ int cluster_rank() const
    {
        return KIND == CLUSTER ? (int)cooperative_groups::this_cluster().block_rank() : 0;
    }
    __device__ __forceinline__ int cluster_size() const
    {
        return KIND == CLUSTER ? (int)cooperative_groups::this_cluster().num_blocks() : 1;
    }
    __device__ __forceinline__ int rank() const
    {
        return KIND == WARP ? (int)(threadIdx.x & 31) : cluster_rank() * (int)blockDim.x + (int)threadIdx.x;
    }
    __device__ __forceinline__ int size() const { return KIND == WARP ? 32 : cluster_size() * (int)blockDim.x; }
    __device__ __forceinline__ void sync() const
    {
        if (KIND == WARP) __syncwarp();
        else if (KIND == CTA) __syncthreads();
        else cooperative_groups::this_cluster().sync();  // orders global memory between the CTAs too
    }
    // Sums of three values over the CTAs of the cluster (each thread holds its CTA's values), and over the CTAs of
    // lower rank: one warp reads the other CTAs' shared memory, a lane per CTA.  Two calls in a row use different
    // slots (`turn` 0 and 1), so the barrier of the second says that everybody has read the first's.
    __device__ __forceinline__ void cluster_sums(const ull (&mine)[3], ull (&all)[3], ull (&lower)[3], int turn) const
    {
        ull* slot = smem + 99 + 3 * turn;
        ull* res = smem + 105;
        if (threadIdx.x == 0) {
#pragma unroll
            for (int q = 0; q < 3; ++q) slot[q] = mine[q];
        }
        cooperative_groups::cluster_group cl = cooperative_groups::this_cluster();
        cl.sync();
        if (threadIdx.x < 32) {
            const unsigned r = threadIdx.x;
            const ull* other = cl.map_shared_rank(slot, r < cl.num_blocks() ? r : 0u);
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                const ull x = r < cl.num_blocks() ? other[q] : 0ull;
                const ull sum = warp_reduce_sum<ull>(x), below = warp_reduce_sum<ull>(r < cl.block_rank() ? x : 0ull);
                if (r == 0) {
                    res[q] = sum;
                    res[3 + q] = below;
                }
            }
        }
        __syncthreads();
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            all[q] = res[q];
            lower[q] = res[3 + q];
        }
        __syncthreads();
    }
    __device__ __forceinline__ ull reduce(ull v, int turn) const
    {
        if (KIND == WARP) return warp_reduce_sum<ull>(v);
        const ull t = block_reduce_sum<ull>(v, smem);
        if (KIND == CTA) return t;
        const ull mine[3] = {t, 0, 0};
        ull all[3], lower[3];
        cluster_sums(mine, all, lower, turn);
        return all[0];
    }
    // Exclusive scans of three values at once (one pass, one set of barriers); v[] in, prefixes
    // out in v[], totals in tot[].
    __device__ __forceinline__ void scan_excl3(ull (&v)[3], ull (&tot)[3]) const
    {
        ull incl[3];
#pragma unroll
        for (int q = 0; q < 3; ++q) incl[q] = warp_scan_incl<ull>(v[q]);
        if (KIND == WARP) {
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                tot[q] = __shfl_sync(0xffffffffu, incl[q], 31);
                v[q] = incl[q] - v[q];
            }
            return;
        }
        const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
        __syncthreads();
        if (lane == 31) {
#pragma unroll
            for (int q = 0; q < 3; ++q) smem[33 * q + warp] = incl[q];
        }
        __syncthreads();
        if (warp == 0) {
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                const ull w = (lane < nw) ? smem[33 * q + lane] : 0ull;
                const ull wi = warp_scan_incl<ull>(w);
                smem[33 * q + lane] = wi - w;
                if (lane == 31) smem[33 * q + 32] = wi;
            }
        }
        __syncthreads();
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            tot[q] = smem[33 * q + 32];
            v[q] = smem[33 * q + warp] + incl[q] - v[q];
        }
        if (KIND == CLUSTER) {
            const ull mine[3] = {tot[0], tot[1], tot[2]};
            ull lower[3];
            cluster_sums(mine, tot, lower, 0);  // after reduce() with 0 and 1
#pragma unroll
            for (int q = 0; q < 3; ++q) v[q] += lower[q];
        }
    }
};

// What a kernel that finishes the bins needs to know of a row prepared by build_alias_row<.., false>.
struct RowSums {
    ull W, d_sum;
    uint32_t L, H;
};

// Builds one table of n items.  weight(i) gives the fixed-point weight of item i.
// sc_w, sc_de, sc_item: scratch of n entries each, private to this row.
// out.bin(i, split point, alias item) receives every bin.
// Returns W44 (the sum of the fixed-point weights) to every thread of the group.
template <GroupKind KIND, bool FINISH = true, class Weight, class Item, class Out>
__device__ ull build_alias_row(const Group<KIND>& g, int32_t n, Weight weight, ull* __restrict__ sc_w, ull* __restrict__ sc_de,
                               Item* __restrict__ sc_item, const Out& out, int* err, RowSums* sums = nullptr)
{
    const int r = g.rank(), gs = g.size();
    // Items are taken four (weights) or two (bins) at a time per thread, their loads issued side by
    // side: a row is built by one warp or one CTA, so what a pass costs is the latency of its chain of
    // dependent reads, not the number of instructions.
    ull s = 0;
    for (int32_t i0 = r; i0 < n; i0 += 4 * gs) {
        ull wt[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int32_t i = i0 + u * gs;
            wt[u] = i < n ? weight(i) : 0ull;
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int32_t i = i0 + u * gs;
            if (i < n) sc_w[i] = wt[u];
            s += wt[u];
        }
    }
    const ull W44 = g.reduce(s, 0);
    int sh = bit_length(W44) + bit_length((ull)n) - 62;
    if (sh < 0) sh = 0;
    s = 0;
#pragma unroll 4
    for (int32_t i = r; i < n; i += gs) s += sc_w[i] >> sh;
    const ull W = g.reduce(s, 1);
    if (W == 0) {
        if (r == 0) {
            atomicOr(err, ERR_ALIAS);
            if (!FINISH) *sums = RowSums{0, 0, 0, 0};
        }
        g.sync();  // no CTA of a cluster leaves while another may read its shared memory (reduce())
        return W44;
    }
    // Every thread takes a run of consecutive items (lights and heavies are numbered in ascending
    // item order): one pass to count them and add up their deficits and surpluses, one scan of the
    // threads' totals, one pass to write the prefix of every item.  An odd run length keeps the
    // threads of a warp on different shared-memory banks.
    g.sync();  // the weights were written item by item across the group
    const int32_t seg = ((n + gs - 1) / gs) | 1;
    const int32_t i_first = min(n, r * seg), i_last = min(n, i_first + seg);
    ull cnt = 0, d_mine = 0, e_mine = 0;
#pragma unroll 4
    for (int32_t i = i_first; i < i_last; ++i) {
        const ull a = (ull)n * (sc_w[i] >> sh);
        if (a <= W) { cnt += 1ull; d_mine += W - a; } else { cnt += 1ull << 32; e_mine += a - W; }
    }
    ull pre[3] = {cnt, d_mine, e_mine}, tot[3];
    g.scan_excl3(pre, tot);
    {
        uint32_t l = (uint32_t)pre[0], m = (uint32_t)(pre[0] >> 32);
        ull d_at = pre[1], e_at = pre[2];
#pragma unroll 2
        for (int32_t i = i_first; i < i_last; ++i) {
            const ull a = (ull)n * (sc_w[i] >> sh);
            sc_w[i] = a;
            if (a <= W) {
                sc_de[l] = d_at;  // deficits of the lights before this one
                sc_item[l] = (Item)i;
                ++l;
                d_at += W - a;
            } else {
                e_at += a - W;
                sc_de[n - 1 - m] = e_at;  // surpluses of the heavies up to and including this one
                sc_item[n - 1 - m] = (Item)i;
                ++m;
            }
        }
    }
    const uint32_t L = (uint32_t)tot[0], H = (uint32_t)(tot[0] >> 32);
    const ull d_sum = tot[1];
    if (!FINISH) {  // the bins are another kernel's work
        if (r == 0) *sums = RowSums{W, d_sum, L, H};
        g.sync();  // no CTA of a cluster leaves while another may read its shared memory
        return W44;
    }
    g.sync();
    const Frac32 frac(W);
    // The searches below count the entries of a sorted prefix array under a bound, one bit of the
    // answer per step from the top: the same number of steps for every item, so several items' searches
    // run in one loop (a CTA has more barriers to make up for than a warp, and fewer neighbours on its SM).
    constexpr int U = KIND == WARP ? 2 : 4;
    const uint32_t top_h = H ? 1u << (31 - __clz((int)H)) : 0u;
    const uint32_t top_l = L ? 1u << (31 - __clz((int)L)) : 0u;
    for (uint32_t l0 = r; l0 < L; l0 += U * gs) {
        uint32_t it[U], pos[U];
        ull a[U], D[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const uint32_t l = l0 + u * gs;
            it[u] = l < L ? sc_item[l] : 0u;
            D[u] = l < L ? sc_de[l] : 0ull;
            pos[u] = 0;
        }
#pragma unroll
        for (int u = 0; u < U; ++u) a[u] = l0 + u * gs < L ? sc_w[it[u]] : W;
        for (uint32_t step = top_h; step; step >>= 1) {  // number of heavies with E_m <= D
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const uint32_t q = pos[u] + step;
                if (q <= H && sc_de[n - q] <= D[u]) pos[u] = q;
            }
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (l0 + u * gs >= L) continue;
            const uint32_t i = it[u];
            uint32_t al = i;
            if (a[u] != W) {
                uint32_t lo = pos[u];
                if (lo >= H) { atomicOr(err, ERR_ALIAS); lo = H ? H - 1 : 0; }
                al = H ? sc_item[n - 1 - lo] : i;
            }
            const uint32_t thr32 = frac(a[u]);
            out.bin(i, thr32, al);
        }
    }
    for (uint32_t m0 = r; m0 < H; m0 += U * gs) {
        uint32_t it[U], pos[U];
        ull E[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const uint32_t m = m0 + u * gs;
            it[u] = m < H ? sc_item[n - 1 - m] : 0u;
            E[u] = m < H ? sc_de[n - 1 - m] : 0ull;
            pos[u] = 0;
        }
        for (uint32_t step = top_l; step; step >>= 1) {  // number of lights with D_l < E: the first light with D_l >= E
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const uint32_t q = pos[u] + step;
                if (q <= L && sc_de[q - 1] < E[u]) pos[u] = q;
            }
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const uint32_t m = m0 + u * gs;
            if (m >= H) continue;
            const uint32_t i = it[u], lo = pos[u];  // lo == L stands for the total deficit
            const ull Dl = lo < L ? sc_de[lo] : d_sum;
            const ull thr = W + E[u] - Dl;
            uint32_t al = i;
            if (thr != W) {
                if (m + 1 >= H) atomicOr(err, ERR_ALIAS);
                else al = sc_item[n - 1 - (m + 1)];
            }
            const uint32_t thr32 = frac(thr);
            out.bin(i, thr32, al);
        }
    }
    return W44;
}

constexpr double FIXED_ONE = 17592186044416.0;  // 2^44

struct DenseWeight {
    const int32_t* nk;
    double beta, Vbeta;
    __device__ __forceinline__ ull operator()(int32_t k) const
    {
        const double den = __dadd_rn((double)nk[k], Vbeta);
        return __double2ull_rz(__dmul_rn(__ddiv_rn(beta, den), FIXED_ONE));
    }
};

struct SparseWeight {
    const uint32_t* topic;
    const uint32_t* count;
    const int32_t* nk;
    double Vbeta;
    __device__ __forceinline__ ull operator()(int32_t i) const
    {
        const double den = __dadd_rn((double)nk[topic[i]], Vbeta);
        return __double2ull_rz(__dmul_rn(__ddiv_rn((double)count[i], den), FIXED_ONE));
    }
};

struct DenseOut {
    uint32_t* thr;
    uint32_t* idx;
    uint2* pk;  // both in one word pair, for the proposal pass; may be null
    __device__ __forceinline__ void bin(uint32_t i, uint32_t thr32, uint32_t al) const
    {
        thr[i] = thr32;
        idx[i] = al;
        if (pk) pk[i] = make_uint2(thr32, al);
    }
};

// What the first kernel of a sweep does besides its own work: the device's sweep counter moves on, the n_k
// buffer the sweep's rebuild will add into is cleared (nothing beside it reads either).
__device__ __forceinline__ void begin_sweep(const View& v, int rank, int size)
{
    if (v.state && rank == 0) {
        SweepState& st = *v.state;
        const uint32_t slot = st.next_slot;
        st.sweep = st.next;
        st.next += 1;
        st.slot = slot;
        st.next_slot = slot + 1;
        st.stamps[slot][STAMP_DENSE] = st.stamps[slot][STAMP_DENSE_END] = global_timer();
    }
    if (v.nk_next)
        for (int32_t k = rank; k < v.dense_stride; k += size) v.nk_next[k] = 0;
}

// Doc-proposal chains draw from no word's table: their sweeps begin with this and build none.
__global__ void __launch_bounds__(1024) k_begin_sweep(View v) { begin_sweep(v, (int)threadIdx.x, (int)blockDim.x); }

int launch_begin_sweep(Ctx& c)
{
    k_begin_sweep<<<1, 1024, 0, c.stream>>>(c.v);
    return 1;
}

// The dense smoothing table; first kernel of a sweep (unless v.state is null).
// One CTA builds a table of up to DENSE_CTA_MAX_K topics; a larger one takes a cluster of DENSE_CLUSTER
// CTAs, whose passes over the table meet at cluster barriers: what bounds the kernel is the
// latency of a few dependent passes over K items, so threads, not bytes, are what it is short of.
// The searches of a large table are scattered reads of device memory, too many for eight multiprocessors: its
// bins are finished by a second kernel, a thread per bin.
constexpr int DENSE_CTA_MAX_K = 2048;
constexpr int DENSE_CLUSTER = 8;
// behind the scratch arrays of K items (20 bytes each)
__device__ __forceinline__ RowSums* dense_sums(ull* sc, int32_t K)
{
    return reinterpret_cast<RowSums*>(sc + 2 * (size_t)K + (K + 1) / 2);
}
template <GroupKind KIND>
__global__ void __launch_bounds__(1024) k_alias_dense(View v, ull* sc)
{
    __shared__ ull smem[GROUP_SMEM];
    Group<KIND> g{smem};
    const int32_t K = v.K;
    begin_sweep(v, g.rank(), g.size());
    DenseWeight wf{v.nk, v.beta, v.Vbeta};
    const ull B = build_alias_row<KIND, KIND == CTA>(g, K, wf, sc, sc + K, (uint32_t*)(sc + 2 * (size_t)K),
                                                     DenseOut{v.dn_thr, v.dn_idx, v.dn_pk}, v.err, dense_sums(sc, K));
    // A table without mass (beta so small that every weight is floored to zero) raises the error word and gets no bins;
    // the proposals that are drawn all the same stay topics of the model.
    if (B == 0 && v.dn_pk)
        for (int32_t k = g.rank(); k < K; k += g.size()) v.dn_pk[k] = make_uint2(0xFFFFFFFFu, (uint32_t)k);
    if (g.rank() == 0) {
        *v.dense_mass = B;
        if (v.state) v.state->stamps[v.state->slot][STAMP_DENSE_END] = global_timer();
    }
}

__global__ void __launch_bounds__(256) k_alias_dense_bins(View v, ull* sc)
{
    const uint32_t K = (uint32_t)v.K, i = blockIdx.x * blockDim.x + threadIdx.x;
    const RowSums t = *dense_sums(sc, v.K);
    const ull *w = sc, *de = sc + K;
    const uint32_t* item = (const uint32_t*)(sc + 2 * (size_t)K);
    if (i >= K || t.W == 0) return;
    const DenseOut out{v.dn_thr, v.dn_idx, v.dn_pk};
    const Frac32 frac(t.W);
    uint32_t pos = 0;
    if (i < t.L) {
        const uint32_t k = item[i];
        const ull a = w[k], D = de[i];
        for (uint32_t step = t.H ? 1u << (31 - __clz((int)t.H)) : 0u; step; step >>= 1)
            if (pos + step <= t.H && de[K - pos - step] <= D) pos += step;
        uint32_t al = k;
        if (a != t.W) {
            if (pos < t.H) al = item[K - 1 - pos]; else atomicOr(v.err, ERR_ALIAS);
        }
        out.bin(k, frac(a), al);
    } else {
        const uint32_t m = i - t.L, k = item[K - 1 - m];
        const ull E = de[K - 1 - m];
        for (uint32_t step = t.L ? 1u << (31 - __clz((int)t.L)) : 0u; step; step >>= 1)
            if (pos + step <= t.L && de[pos + step - 1] < E) pos += step;
        const ull part = t.W + E - (pos < t.L ? de[pos] : t.d_sum);
        uint32_t al = k;
        if (part != t.W) {
            if (m + 1 < t.H) al = item[K - 2 - m]; else atomicOr(v.err, ERR_ALIAS);
        }
        out.bin(k, frac(part), al);
    }
    // all CTAs run at once: the last one's time is the table's
    if (v.state && blockIdx.x + 1 == gridDim.x && threadIdx.x == 0) v.state->stamps[v.state->slot][STAMP_DENSE_END] = global_timer();
}

static int dense_launches(int32_t K) { return K > DENSE_CTA_MAX_K ? 2 : 1; }
static cudaError_t run_alias_dense(const View& v, ull* scratch, cudaStream_t stream)
{
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    const int ctas = v.K > DENSE_CTA_MAX_K ? DENSE_CLUSTER : 1;
    int threads = 64;  // about an item per thread
    while (threads < 1024 && threads * ctas < v.K) threads <<= 1;
    cfg.gridDim = dim3((unsigned)ctas);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.stream = stream;
    if (ctas == 1) return cudaLaunchKernelEx(&cfg, k_alias_dense<CTA>, v, scratch);
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = DENSE_CLUSTER;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, k_alias_dense<CLUSTER>, v, scratch);
    if (e != cudaSuccess) return e;
    k_alias_dense_bins<<<(unsigned)((v.K + 255) / 256), 256, 0, stream>>>(v, scratch);
    return cudaGetLastError();
}

// Mixture thresholds as lda_get_tables() reports them (the proposal pass works its tiles' out itself).
__global__ void __launch_bounds__(256) k_mix_thresholds(View v, uint32_t* __restrict__ mix32)
{
    const int32_t w = blockIdx.x * blockDim.x + threadIdx.x;
    if (w < v.V) mix32[w] = mixture_threshold(v.sp_mass[w], *v.dense_mass);
}

void launch_mix_thresholds(Ctx& c, uint32_t* mix32)
{
    k_mix_thresholds<<<(c.V + 255) / 256, 256, 0, c.stream>>>(c.v, mix32);
}

// ---- per-word sparse tables ----------------------------------------------------------------------
// Rows differ in length by four orders of magnitude, and what a row costs is the latency of its chain
// of dependent steps (weights, two sums, one scan, one search per item), so a row gets as many threads as
// it has work for: a few lanes (up to 32 items, everything in registers), a warp (256, 512), a CTA of 256 threads (2048),
// one of 1024 (ALIAS_BIG_MAX), a cluster (longer).  Which kernel looks at a word depends on the
// row's capacity, which one builds it on its length in this sweep.
//
// Who reads a table decides what is written: hot words (with 16-bit topics) are drawn from through packed bins,
// all others through split points and alias items (lda_get_tables() wants those of all words: `all`).
struct RowOut {
    uint32_t* thr;
    uint32_t* idx;
    uint2* pk;               // null: not wanted
    const uint32_t* topic;   // of the row's items
    bool plain;              // thr, idx wanted
    __device__ __forceinline__ RowOut(const View& v, int32_t w, int32_t r0, bool all)
    {
        const bool hot = __ldg(v.hot_word + w) != 0;
        thr = v.al_thr + r0;
        idx = v.al_idx + r0;
        pk = (v.al_pk && (hot || all)) ? v.al_pk + r0 : nullptr;
        topic = v.wk_topic + r0;
        plain = all || !hot || !v.al_pk;
    }
    __device__ __forceinline__ void bin(int32_t i, uint32_t thr32, uint32_t al) const
    {
        if (plain) {
            thr[i] = thr32;
            idx[i] = al;
        }
        if (pk) pk[i] = make_uint2(thr32, topic[i] | (topic[al] << 16));
    }
};

__device__ __forceinline__ ull sparse_weight(uint32_t count, int32_t nk, double Vbeta)
{
    const double den = __dadd_rn(u32_to_double((uint32_t)nk), Vbeta);
    return __double2ull_rz(__dmul_rn(__ddiv_rn(u32_to_double(count), den), FIXED_ONE));
}

// Rows of at most WD items, one lane per item, 32 / WD rows per warp.  Every lane of the warp calls it
// (n = 0: no row).
template <int WD>
__device__ __forceinline__ void alias_row_lanes(const View& v, int32_t w, int32_t n, int32_t r0, bool all)
{
    constexpr uint32_t FULL = 0xFFFFFFFFu;
    const int lane = threadIdx.x & 31, l = lane & (WD - 1);
    const bool live = l < n;
    uint32_t k = 0;
    ull a = 0;
    if (live) {
        k = __ldg(v.wk_topic + r0 + l);
        a = sparse_weight(__ldg(v.wk_count + r0 + l), __ldg(v.nk + k), v.Vbeta);
    }
    ull W44 = a;
#pragma unroll
    for (int o = WD / 2; o > 0; o >>= 1) W44 += __shfl_xor_sync(FULL, W44, o);
    const int sh = max(0, bit_length(W44) + bit_length((ull)n) - 62);
    a >>= sh;
    ull W = a;
#pragma unroll
    for (int o = WD / 2; o > 0; o >>= 1) W += __shfl_xor_sync(FULL, W, o);
    a *= (ull)n;
    const bool heavy = live && a > W;
    const ull d = live && !heavy ? W - a : 0, e = heavy ? a - W : 0;
    ull D = d, E = e;  // inclusive prefixes over the row's lanes
#pragma unroll
    for (int o = 1; o < WD; o <<= 1) {
        const ull x = __shfl_up_sync(FULL, D, o, WD), y = __shfl_up_sync(FULL, E, o, WD);
        if (l >= o) {
            D += x;
            E += y;
        }
    }
    const ull d_sum = __shfl_sync(FULL, D, WD - 1, WD);
    D -= d;  // deficits of the lights before this lane
    // a light item looks for the first lane whose surpluses exceed D, a heavy one for the first lane with
    // deficits of at least E before it; both prefixes ascend over the lanes
    int pos = 0;
#pragma unroll
    for (int step = WD / 2; step > 0; step >>= 1) {
        const int q = pos + step;
        const ull x = __shfl_sync(FULL, E, q - 1, WD), y = __shfl_sync(FULL, D, q - 1, WD);
        if (heavy ? y < E : x <= D) pos = q;
    }
    {
        const ull x = __shfl_sync(FULL, E, pos, WD), y = __shfl_sync(FULL, D, pos, WD);
        if (heavy ? y < E : x <= D) ++pos;
    }
    const ull D_at = __shfl_sync(FULL, D, min(pos, WD - 1), WD);
    const uint32_t heavies = (__ballot_sync(FULL, heavy) >> (lane & ~(WD - 1))) & (WD == 32 ? FULL : (1u << WD) - 1u);
    const uint32_t above = heavies & ~((2u << l) - 1u);
    ull part = a;
    int al = l;
    bool bad = live && W == 0;
    if (heavy) {
        part = W + E - (pos < WD ? D_at : d_sum);
        if (part != W) {
            bad = bad || !above;
            if (above) al = __ffs((int)above) - 1;
        }
    } else if (live && a != W) {
        bad = bad || pos >= n;
        if (pos < n) al = pos;
    }
    if (bad) atomicOr(v.err, ERR_ALIAS);
    const uint32_t k_al = __shfl_sync(FULL, k, al, WD);
    if (live) {
        const uint32_t thr32 = Frac32(W)(part);
        const RowOut out(v, w, r0, all);
        if (out.plain) {
            out.thr[l] = thr32;
            out.idx[l] = (uint32_t)al;
        }
        if (out.pk) out.pk[l] = make_uint2(thr32, k | (k_al << 16));
        if (l == 0) v.sp_mass[w] = W44;
    }
}

constexpr int ALIAS_WARP_THREADS = 256;
constexpr int ALIAS_WARP_SMEM = ALIAS_WARP_THREADS / 32 * ALIAS_WARP_MAX * ALIAS_SCRATCH_PER_ITEM;
// Rows of up to ALIAS_WARP_MAX items: a warp takes `per_warp` consecutive words of the list, the short rows several at a
// time.  The list holds the words that occur (820 000 words, 300 000 tokens: 38 us over the whole vocabulary).
__global__ void __launch_bounds__(ALIAS_WARP_THREADS)
k_alias_sparse_warp(View v, const int32_t* __restrict__ list, int32_t n_list, int32_t per_warp, bool all)
{
    extern __shared__ __align__(16) unsigned char alias_scratch[];
    constexpr int WARPS = ALIAS_WARP_THREADS / 32;
    constexpr uint32_t FULL = 0xFFFFFFFFu;
    const int lane = threadIdx.x & 31, wic = threadIdx.x >> 5;
    const Group<WARP> g{nullptr};
    const int32_t stride = (int32_t)((gridDim.x * blockDim.x) >> 5) * per_warp;
    for (int32_t first = (int32_t)((blockIdx.x * blockDim.x + threadIdx.x) >> 5) * per_warp; first < n_list; first += stride) {
        int32_t n_mine = -1, r_mine = 0, mine = 0;
        if (lane < per_warp && first + lane < n_list) {
            mine = __ldg(list + first + lane);
            n_mine = v.wk_nnz[mine];
            r_mine = v.row_start[mine];
            if (n_mine == 0) v.sp_mass[mine] = 0;
        }
        // the lanes of `words` that hold a row of the class; `rows` of them are built at once
        auto several = [&](uint32_t words, auto width) {
            constexpr int WD = decltype(width)::value;
            while (words) {
                uint32_t rest = words;
                for (int i = 0; i < lane / WD; ++i) rest &= rest - 1;  // this lane's group takes the (lane / WD)-th
                const int src = rest ? __ffs((int)rest) - 1 : 0;
                const int32_t n = __shfl_sync(FULL, n_mine, src), r0 = __shfl_sync(FULL, r_mine, src);
                alias_row_lanes<WD>(v, __shfl_sync(FULL, mine, src), rest ? n : 0, r0, all);
                for (int i = 0; i < 32 / WD; ++i) words &= words - 1;
            }
        };
        several(__ballot_sync(FULL, n_mine > 0 && n_mine <= 8), std::integral_constant<int, 8>{});
        several(__ballot_sync(FULL, n_mine > 8 && n_mine <= 16), std::integral_constant<int, 16>{});
        several(__ballot_sync(FULL, n_mine > 16 && n_mine <= 32), std::integral_constant<int, 32>{});
        for (uint32_t words = __ballot_sync(FULL, n_mine > 32 && n_mine <= ALIAS_WARP_MAX); words; words &= words - 1) {
            const int src = __ffs((int)words) - 1;
            const int32_t n = __shfl_sync(FULL, n_mine, src), r0 = __shfl_sync(FULL, r_mine, src);
            const int32_t w = __shfl_sync(FULL, mine, src);
            ull* de = reinterpret_cast<ull*>(alias_scratch) + (size_t)wic * ALIAS_WARP_MAX;
            ull* wt = de + WARPS * ALIAS_WARP_MAX;
            uint16_t* item = reinterpret_cast<uint16_t*>(reinterpret_cast<ull*>(alias_scratch) + 2 * WARPS * ALIAS_WARP_MAX) +
                             (size_t)wic * ALIAS_WARP_MAX;
            const SparseWeight wf{v.wk_topic + r0, v.wk_count + r0, v.nk, v.Vbeta};
            const ull S = build_alias_row<WARP>(g, n, wf, wt, de, item, RowOut(v, w, r0, all), v.err);
            if (lane == 0) v.sp_mass[w] = S;
            __syncwarp();
        }
    }
}

// One warp per word of the list: rows of ALIAS_WARP_MAX < n <= ALIAS_LONG_WARP_MAX items.  Their weights stay in
// device memory: 18 bytes of shared memory per item would leave too few warps per multiprocessor (738 M tokens,
// K = 10 000, all kernels together: 1.6 ms so, 1.8 with these rows on CTAs of 256 threads).
__global__ void __launch_bounds__(128) k_alias_sparse_long_warp(View v, const int32_t* __restrict__ words, int32_t n_words, bool all,
                                                                ull* sc_w)
{
    __shared__ ull de_s[4][ALIAS_LONG_WARP_MAX];
    __shared__ uint16_t item_s[4][ALIAS_LONG_WARP_MAX];
    const int wic = threadIdx.x >> 5;
    const int32_t i = blockIdx.x * 4 + wic;
    if (i >= n_words) return;
    const int32_t w = words[i], n = v.wk_nnz[w];
    if (n <= ALIAS_WARP_MAX || n > ALIAS_LONG_WARP_MAX) return;
    const int32_t r0 = v.row_start[w];
    const SparseWeight wf{v.wk_topic + r0, v.wk_count + r0, v.nk, v.Vbeta};
    const ull S = build_alias_row<WARP>(Group<WARP>{nullptr}, n, wf, sc_w + r0, de_s[wic], item_s[wic], RowOut(v, w, r0, all), v.err);
    if ((threadIdx.x & 31) == 0) v.sp_mass[w] = S;
}

// One CTA per word: rows of LO < n <= HI items.
template <int THREADS, int LO, int HI>
__global__ void __launch_bounds__(THREADS)
k_alias_sparse_cta(View v, const int32_t* __restrict__ words, bool all)
{
    extern __shared__ __align__(16) unsigned char alias_scratch[];
    __shared__ ull smem[GROUP_SMEM];
    const Group<CTA> g{smem};
    const int32_t w = words[blockIdx.x];
    const int32_t n = v.wk_nnz[w];
    if (n <= LO || n > HI) return;
    const int32_t r0 = v.row_start[w];
    ull* wt = reinterpret_cast<ull*>(alias_scratch);
    const SparseWeight wf{v.wk_topic + r0, v.wk_count + r0, v.nk, v.Vbeta};
    const ull S = build_alias_row<CTA>(g, n, wf, wt, wt + HI, reinterpret_cast<uint16_t*>(wt + 2 * HI), RowOut(v, w, r0, all), v.err);
    if (threadIdx.x == 0) v.sp_mass[w] = S;
}

// Rows longer than ALIAS_BIG_MAX: a cluster of CTAs per word, scratch in the row's range of the arrays in device memory.
__global__ void __cluster_dims__(ALIAS_ROW_CLUSTER) __launch_bounds__(512)
k_alias_sparse_cluster(View v, const int32_t* __restrict__ words, ull* sc_w, ull* sc_de, uint32_t* sc_item, bool all)
{
    __shared__ ull smem[GROUP_SMEM];
    const Group<CLUSTER> g{smem};
    const int32_t w = words[blockIdx.x / ALIAS_ROW_CLUSTER];
    const int32_t n = v.wk_nnz[w];
    if (n <= ALIAS_BIG_MAX) return;
    const int32_t r0 = v.row_start[w];
    const SparseWeight wf{v.wk_topic + r0, v.wk_count + r0, v.nk, v.Vbeta};
    const ull S = build_alias_row<CLUSTER>(g, n, wf, sc_w + r0, sc_de + r0, sc_item + r0, RowOut(v, w, r0, all), v.err);
    if (g.rank() == 0) v.sp_mass[w] = S;
}

int launch_alias_dense(Ctx& c, bool in_sweep)
{
    View v = c.v;
    if (!in_sweep) {  // the table alone: no sweep begins
        v.state = nullptr;
        v.nk_next = nullptr;
    }
    run_alias_dense(v, c.sc_dense, c.stream);
    return dense_launches(c.K);
}

// The kernels build the tables of different words: they run side by side, the ones with the longest rows
// (and the longest tail) first.  begin_sweep: the sweep's first kernel, the dense table, runs beside them
// (nothing here reads what it writes).
int launch_alias_sparse(Ctx& c, bool all, bool begin_sweep)
{
    const Ctx::Slice& q = c.slices[(size_t)c.cur_slice];
    int launches = 0;
    fork_streams(c);
    if (begin_sweep) {
        run_alias_dense(c.v, c.sc_dense, c.side[0]);
        launches += dense_launches(c.K);
    }
    const auto words = [&](int cls) { return c.alias_words[cls] + q.alias_lo[cls]; };
    if (q.alias_n[3]) {
        k_alias_sparse_cluster<<<q.alias_n[3] * ALIAS_ROW_CLUSTER, 512, 0, c.stream>>>(c.v, words(3), c.sc_w, c.sc_de, c.sc_item, all);
        ++launches;
    }
    if (q.alias_n[2]) {
        k_alias_sparse_cta<1024, ALIAS_MID_MAX, ALIAS_BIG_MAX>
            <<<q.alias_n[2], 1024, ALIAS_BIG_MAX * ALIAS_SCRATCH_PER_ITEM, c.stream>>>(c.v, words(2), all);
        ++launches;
    }
    // a warp takes a row of 257..512 items at the least cost, a CTA in the least time: a CTA if all have room at once
    const bool few = q.alias_n[0] <= 4 * c.n_sm;
    if (few && q.alias_n[0]) {
        k_alias_sparse_cta<256, ALIAS_WARP_MAX, ALIAS_MID_MAX>
            <<<q.alias_n[0], 256, ALIAS_MID_MAX * ALIAS_SCRATCH_PER_ITEM, c.side[0]>>>(c.v, words(0), all);
        ++launches;
    }
    if (!few && q.alias_n[1]) {
        k_alias_sparse_cta<256, ALIAS_LONG_WARP_MAX, ALIAS_MID_MAX>
            <<<q.alias_n[1], 256, ALIAS_MID_MAX * ALIAS_SCRATCH_PER_ITEM, c.side[0]>>>(c.v, words(1), all);
        ++launches;
    }
    if (!few) {
        k_alias_sparse_long_warp<<<(q.alias_n[0] + 3) / 4, 128, 0, c.side[0]>>>(c.v, words(0), q.alias_n[0], all, c.sc_w);
        ++launches;
    }
    if (q.present_n <= 0) {
        join_streams(c);
        return launches;
    }
    // words per warp: as many as fill a warp's lanes with the words' sizes, as long as every multiprocessor gets two CTAs
    int per_warp = 32;
    while (per_warp > 1 && q.present_n / per_warp < c.n_sm * 16) per_warp /= 2;
    const int64_t warps = ((int64_t)q.present_n + per_warp - 1) / per_warp;
    constexpr int WARPS = ALIAS_WARP_THREADS / 32;
    k_alias_sparse_warp<<<(int)std::min<int64_t>((warps + WARPS - 1) / WARPS, (int64_t)c.n_sm * 16), ALIAS_WARP_THREADS,
                          ALIAS_WARP_SMEM, c.side[1]>>>(c.v, c.present + q.present_lo, q.present_n, per_warp, all);
    ++launches;
    join_streams(c);
    return launches;
}

void set_alias_smem_limits()
{
    cudaFuncSetAttribute(k_alias_sparse_warp, cudaFuncAttributeMaxDynamicSharedMemorySize, ALIAS_WARP_SMEM);
    cudaFuncSetAttribute(k_alias_sparse_cta<256, ALIAS_LONG_WARP_MAX, ALIAS_MID_MAX>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         ALIAS_MID_MAX * ALIAS_SCRATCH_PER_ITEM);
    cudaFuncSetAttribute(k_alias_sparse_cta<256, ALIAS_WARP_MAX, ALIAS_MID_MAX>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         ALIAS_MID_MAX * ALIAS_SCRATCH_PER_ITEM);
    cudaFuncSetAttribute(k_alias_sparse_cta<1024, ALIAS_MID_MAX, ALIAS_BIG_MAX>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         ALIAS_BIG_MAX * ALIAS_SCRATCH_PER_ITEM);
}

}  // namespace lda

// ---------------------------------------------------------------------------------------
// Allocation-free entry point.
//
// Some callers cannot allocate device memory at the moment they need a table: code that
// runs inside a framework's memory pool and must not touch cudaMalloc behind its back, a
// real-time loop where an allocation's implicit device synchronisation is not acceptable,
// or a process whose memory budget was fixed at start-up.  For them the dense smoothing
// table can be built with the construction scratch held in a file-scope device array.
// Every GPU that loads the library holds that array (20 bytes per topic of LDA_NOALLOC_MAX_K,
// about 2.6 MB) until exit.
// ---------------------------------------------------------------------------------------
namespace lda {

constexpr int NOALLOC_MAX_K = LDA_NOALLOC_MAX_K;
// per topic: one 64-bit mass, one 64-bit prefix sum, one 32-bit item index = 20 bytes
constexpr size_t NOALLOC_SCRATCH_WORDS = 2 * (size_t)NOALLOC_MAX_K + (size_t)NOALLOC_MAX_K / 2 + 4;  // + RowSums

static __device__ __align__(256) unsigned long long g_noalloc_scratch[NOALLOC_SCRATCH_WORDS];
static __device__ __align__(256) int g_noalloc_status[4];

// Device addresses of the two arrays above, looked up once per device.  In host code the
// array names are only handles for the runtime, not addresses a kernel could use.
struct NoallocAddr {
    bool ready = false;
    unsigned long long* scratch = nullptr;
    int* status = nullptr;
};
static NoallocAddr g_noalloc_addr[64];

static int noalloc_setup(int dev, NoallocAddr** out)
{
    if (dev < 0 || dev >= 64) return LDA_ERANGE;
    NoallocAddr& a = g_noalloc_addr[dev];
    if (!a.ready) {
        void* p = nullptr;
        void* q = nullptr;
        if (cudaGetSymbolAddress(&p, g_noalloc_scratch) != cudaSuccess ||
            cudaGetSymbolAddress(&q, g_noalloc_status) != cudaSuccess) {
            cudaGetLastError();
            return LDA_ECUDA;
        }
        a.scratch = (unsigned long long*)p;
        a.status = (int*)q;
        a.ready = true;
    }
    *out = &a;
    return LDA_OK;
}

}  // namespace lda

extern "C" int lda_dense_table_noalloc(const int32_t* n_k_dev, int32_t K, int32_t V, double beta,
                                       uint32_t* dn_thr32_dev, int32_t* dn_alias_dev,
                                       uint64_t* dense_mass_dev, int32_t* status_dev, void* cuda_stream)
{
    using namespace lda;
    if (!n_k_dev || !dn_thr32_dev || !dn_alias_dev || !dense_mass_dev) return LDA_EINVAL;
    if (K <= 0 || V <= 0 || !(beta > 0) || !isfinite(beta)) return LDA_EINVAL;
    if (K > NOALLOC_MAX_K) return LDA_ERANGE;  // the fixed scratch array holds LDA_NOALLOC_MAX_K topics
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) { cudaGetLastError(); return LDA_ECUDA; }
    NoallocAddr* addr = nullptr;
    int rc = noalloc_setup(dev, &addr);
    if (rc != LDA_OK) return rc;
    cudaStream_t st = (cudaStream_t)cuda_stream;
    int* status = status_dev ? (int*)status_dev : addr->status;
    // the status word must start at zero; the scratch itself is fully overwritten before it is read
    if (cudaMemsetAsync(status, 0, sizeof(int), st) != cudaSuccess) { cudaGetLastError(); return LDA_ECUDA; }
    View v{};
    v.V = V;
    v.K = K;
    v.beta = beta;
    v.Vbeta = (double)V * beta;
    v.nk = const_cast<int32_t*>(n_k_dev);
    v.dn_thr = dn_thr32_dev;
    v.dn_idx = (uint32_t*)dn_alias_dev;
    v.dense_mass = (unsigned long long*)dense_mass_dev;
    v.err = status;
    if (run_alias_dense(v, addr->scratch, st) != cudaSuccess || cudaGetLastError() != cudaSuccess) {
        cudaGetLastError();
        return LDA_ECUDA;
    }
    return LDA_OK;
}
