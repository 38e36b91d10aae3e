// C ABI of the library: argument checks, device memory, work lists, launch order.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <limits>
#include <memory>
#include <mutex>
#include <new>
#include <system_error>
#include <thread>
#include <utility>

#include "lda_internal.cuh"

namespace lda {
void set_hist_smem_limits();
void set_sample_smem_limits();
void set_doc_smem_limits();
void set_alias_smem_limits();
void set_export_smem_limits();
void set_loglik_smem_limits();

void* raw_alloc(Ctx& c, size_t bytes)
{
    if (c.alloc_fn) return c.alloc_fn(bytes, c.alloc_user);
    void* p = nullptr;
    if (cudaMalloc(&p, bytes) != cudaSuccess) {
        cudaGetLastError();
        return nullptr;
    }
    return p;
}

void raw_free(Ctx& c, void* p)
{
    if (!p) return;
    if (c.free_fn) c.free_fn(p, c.alloc_user);
    else cudaFree(p);
}

void* dev_alloc(Ctx& c, size_t bytes)
{
    if (bytes == 0) bytes = 16;
    void* p = raw_alloc(c, bytes);
    if (!p) return nullptr;
    c.allocs.push_back(p);
    c.alloc_bytes.push_back(bytes);
    c.alloc_own.push_back(c.alloc_fn ? 1 : 0);
    c.device_bytes += (int64_t)bytes;
    return p;
}

void dev_free(Ctx& c, void* p)
{
    if (!p) return;
    for (size_t i = 0; i < c.allocs.size(); ++i)
        if (c.allocs[i] == p) {
            c.device_bytes -= (int64_t)c.alloc_bytes[i];
            const bool own = c.alloc_own[i] != 0;
            c.allocs.erase(c.allocs.begin() + i);
            c.alloc_bytes.erase(c.alloc_bytes.begin() + i);
            c.alloc_own.erase(c.alloc_own.begin() + i);
            if (own && c.free_fn) c.free_fn(p, c.alloc_user);
            else cudaFree(p);
            return;
        }
}

void dev_free_all(Ctx& c)
{
    for (size_t i = 0; i < c.allocs.size(); ++i) {
        if (c.alloc_own[i] && c.free_fn) c.free_fn(c.allocs[i], c.alloc_user);
        else cudaFree(c.allocs[i]);
    }
    c.allocs.clear();
    c.alloc_bytes.clear();
    c.alloc_own.clear();
    c.device_bytes = 0;
}

// A context's sweep state (device memory) and the report the device writes for it (host memory), with the streams
// and events a context needs.  Sets are handed from one context to the next -- a new one costs more driver time
// than a small corpus takes to load -- and at most KEPT idle ones are kept.
struct ContextParts {
    int device = -1;
    SweepState* state = nullptr;
    SweepReport* report = nullptr;
    cudaStream_t side[2] = {}, copy = nullptr;
    cudaEvent_t ev[5] = {};
};
struct PartsPool {
    static constexpr size_t KEPT = 4;
    std::mutex lock;
    std::vector<ContextParts> idle;
    static PartsPool& pool()
    {
        static PartsPool* p = new PartsPool;  // never destroyed: contexts may outlive static objects
        return *p;
    }
    static void release(ContextParts& b)
    {
        for (cudaEvent_t e : b.ev)
            if (e) cudaEventDestroy(e);
        for (cudaStream_t s : {b.side[0], b.side[1], b.copy})
            if (s) cudaStreamDestroy(s);
        if (b.state) cudaFree(b.state);
        if (b.report) cudaFreeHost(b.report);
        cudaGetLastError();
    }
    bool take(Ctx& c)
    {
        ContextParts b;
        {
            std::lock_guard<std::mutex> g(lock);
            for (size_t i = 0; i < idle.size() && b.device < 0; ++i)
                if (idle[i].device == c.device) {
                    b = idle[i];
                    idle.erase(idle.begin() + (long)i);
                }
        }
        if (b.device < 0) {
            bool ok = cudaMalloc(reinterpret_cast<void**>(&b.state), sizeof(SweepState)) == cudaSuccess &&
                      cudaHostAlloc(reinterpret_cast<void**>(&b.report), sizeof(SweepReport),
                                    cudaHostAllocPortable | cudaHostAllocMapped) == cudaSuccess;
            for (cudaEvent_t& e : b.ev) ok = ok && cudaEventCreateWithFlags(&e, cudaEventDisableTiming) == cudaSuccess;
            for (cudaStream_t* s : {&b.side[0], &b.side[1], &b.copy})
                ok = ok && cudaStreamCreateWithFlags(s, cudaStreamNonBlocking) == cudaSuccess;
            if (!ok) {
                release(b);
                return false;
            }
            b.device = c.device;
        }
        c.v.state = b.state;
        c.v.err = &b.state->err;
        c.report = b.report;
        for (int i = 0; i < 2; ++i) {
            c.side[i] = b.side[i];
            c.ev_join[i] = b.ev[i];
        }
        c.copy = b.copy;
        c.ev_fork = b.ev[2];
        c.ev_chunk = b.ev[3];
        c.ev_export = b.ev[4];
        return true;
    }
    void give(Ctx& c)  // nothing of the context runs any more
    {
        if (!c.v.state) return;
        ContextParts b{c.device, c.v.state, c.report, {c.side[0], c.side[1]}, c.copy,
                       {c.ev_join[0], c.ev_join[1], c.ev_fork, c.ev_chunk, c.ev_export}};
        c.v.state = nullptr;
        {
            std::lock_guard<std::mutex> g(lock);
            if (idle.size() < KEPT) {
                idle.push_back(b);
                return;
            }
        }
        release(b);
    }
};

__global__ void k_set_state(SweepState* st, uint32_t sweep)
{
    unsigned long long* stamps = &st->stamps[0][0];
    for (int i = threadIdx.x; i < STAMP_RING * STAMPS; i += blockDim.x) stamps[i] = 0;
    if (threadIdx.x == 0) {
        st->moves[0] = st->moves[1] = 0;
        st->next = sweep;
        st->next_slot = 0;
    }
}

// After a batch of sweeps: what the host wants to know goes to host memory, the rest is made ready
// for the next batch.  One CTA; runs after the batch's last kernel.
__global__ void k_report(SweepState* st, SweepReport* rep)
{
    const uint32_t n = st->next_slot;
    __syncthreads();
    if (threadIdx.x == 0) {
        rep->end = global_timer();
        rep->moves[0] = st->moves[0];
        rep->moves[1] = st->moves[1];
        rep->err = st->err;
        st->moves[0] = st->moves[1] = 0;
        st->err = 0;
        st->next_slot = 0;
    }
    for (uint32_t i = threadIdx.x; i < n * STAMPS; i += blockDim.x) {
        (&rep->stamps[0][0])[i] = (&st->stamps[0][0])[i];
        (&st->stamps[0][0])[i] = 0;
    }
}

void launch_set_state(Ctx& c) { k_set_state<<<1, 128, 0, c.stream>>>(c.v.state, c.sweep); }
void launch_report(Ctx& c) { k_report<<<1, 128, 0, c.stream>>>(c.v.state, c.report); }

static void drop_graphs(Ctx& c)
{
    for (cudaGraphExec_t& g : c.graph) {
        if (g) cudaGraphExecDestroy(g);
        g = nullptr;
    }
    c.plain_sweeps = 0;
}

static int fail(Ctx* c, int code, const char* msg)
{
    if (c) c->err = msg;
    return code;
}

// Nothing leaves the C entries by an exception: `f` gives the status, or the host had no memory for it.
template <typename F>
static int guarded(Ctx& c, F f)
{
    try {
        return f();
    } catch (const std::bad_alloc&) {
        return fail(&c, LDA_ENOMEM, "host allocation failed");
    }
}

static int cuda_fail(Ctx* c, const char* where)
{
    cudaError_t e = cudaGetLastError();
    if (c) c->err = std::string(where) + ": " + cudaGetErrorString(e);
    return LDA_ECUDA;
}

// Reads and clears the device error word.
static int read_err(Ctx& c, int* bits)
{
    if (cudaMemcpyAsync(bits, c.v.err, sizeof(int), cudaMemcpyDeviceToHost, c.stream) != cudaSuccess ||
        cudaStreamSynchronize(c.stream) != cudaSuccess)
        return cuda_fail(&c, "reading the device error word");
    if (*bits) cudaMemsetAsync(c.v.err, 0, sizeof(int), c.stream);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) {
        c.err = std::string("kernel launch: ") + cudaGetErrorString(e);
        return LDA_ECUDA;
    }
    return LDA_OK;
}

static int check_device(Ctx& c)
{
    if (cudaSetDevice(c.device) != cudaSuccess) return cuda_fail(&c, "cudaSetDevice");
    return LDA_OK;
}

// An export started by lda_get_assignments*_async() may still be copying out of the staging buffer:
// whatever is queued on the context's stream from here on starts after it (no host wait).
static void order_after_export(Ctx& c)
{
    if (!c.export_pending) return;
    cudaStreamWaitEvent(c.stream, c.ev_export, 0);
    c.export_pending = false;
}

// Host wait for everything the context has queued, the copy stream included.
static int wait_all(Ctx& c)
{
    cudaError_t e = cudaStreamSynchronize(c.stream);
    if (e == cudaSuccess && c.copy) e = cudaStreamSynchronize(c.copy);
    c.export_pending = false;
    return e == cudaSuccess ? LDA_OK : cuda_fail(&c, "waiting for the context's streams");
}

static void free_corpus(Ctx& c)
{
    if (c.copy) cudaStreamSynchronize(c.copy);  // an export may still read the staging buffer
    c.export_pending = false;
    drop_graphs(c);
    dev_free_all(c);
    View nv{};
    nv.V = c.V; nv.K = c.K; nv.alpha = c.alpha; nv.beta = c.beta;
    nv.Vbeta = (double)c.V * c.beta;
    nv.Kalpha = (double)c.K * c.alpha;
    // What single precision gets wrong, in units of 2^-24 of the value: 2 for each of a side's three factors without the token
    // (count and prior as they are converted, then their sum), 3 for each of the two with it put back (one more sum), 4 for the products,
    // and 2 for the uniform's conversion and product: 18 on its side, 16 on the other, one of the difference.  64 are allowed.
    // Priors for which products might underflow leave every step to double precision (an overflow shows by itself).
    nv.alpha_f = (float)nv.alpha;
    nv.beta_f = (float)nv.beta;
    nv.Vbeta_f = (float)nv.Vbeta;
    const double low = std::min({nv.alpha, nv.beta, nv.Vbeta}), high = std::max({nv.alpha, nv.beta, nv.Vbeta});
    nv.filter_eps = low >= 0x1p-24 && high <= 0x1p60 ? 0x1p-18f : std::numeric_limits<float>::infinity();
    nv.dense_stride = (c.K + 3) & ~3;
    nv.state = c.v.state;
    nv.err = &nv.state->err;
    c.v = nv;
    c.loaded = c.inited = c.tables_valid = c.wide_counts = false;
    c.N = c.D = 0;
    c.side_steps = 0;
    c.slices.clear();
    c.cur_slice = 0;
    c.al_thr0 = c.al_idx0 = c.sc_item0 = c.sc_item = nullptr;
    c.al_pk0 = nullptr;
    c.sc_w0 = c.sc_de0 = c.sc_w = c.sc_de = nullptr;
}

// Row slot r of the running slice lives at entry r - row_lo of the slice-sized buffers: the pointers the
// kernels index with row slots are the buffers' moved back by row_lo entries (and only ever used with
// slots of that slice).
template <typename P>
static P* moved_back(P* base, int64_t entries)
{
    return base ? reinterpret_cast<P*>(reinterpret_cast<uintptr_t>(base) - (uintptr_t)entries * sizeof(P)) : nullptr;
}

void set_slice(Ctx& c, int slice)
{
    const Ctx::Slice& q = c.slices[(size_t)slice];
    c.cur_slice = slice;
    c.v.al_thr = moved_back(c.al_thr0, q.row_lo);
    c.v.al_idx = moved_back(c.al_idx0, q.row_lo);
    c.v.al_pk = moved_back(c.al_pk0, q.row_lo);
    c.sc_w = moved_back(c.sc_w0, q.row_lo);
    c.sc_de = moved_back(c.sc_de0, q.row_lo);
    c.sc_item = moved_back(c.sc_item0, q.row_lo);
}

}  // namespace lda

// Buffers the passes of the MH step hand results to each other in; sized by the number of steps.
int lda::ensure_exchange(Ctx& c, int mh_steps)
{
    if (c.N == 0) return LDA_OK;
    auto bytes_for = [&](int mode, int steps, size_t& prop_b, size_t& side_b, size_t& ua_b, int& stride) {
        const size_t zt = c.wide_topics ? 4 : 2, n = (size_t)c.N;
        const int n_word = mode == LDA_PROPOSALS_CYCLE ? (steps + 1) / 2 : mode == LDA_PROPOSALS_WORD ? steps : 0;
        const int n_doc = steps - n_word;
        const size_t planes = (size_t)(n_word > 0 ? n_word : 1);
        stride = (1 + steps + n_doc + 3) & ~3;  // own, one word per step, one uniform per doc step
        prop_b = zt * planes * n;
        side_b = 4 * (size_t)stride * n;
        ua_b = 4 * planes * n;
    };
    size_t pb = 0, sb = 0, ub = 0;
    int stride = 0;
    if (mh_steps <= c.side_steps && c.side_mode == c.proposals && c.v.dside) {
        // buffers laid out for more steps of the same schedule are large enough: only the record
        // stride follows the step count (a chain of two steps keeps its 16-byte records after a
        // chain of four has run)
        bytes_for(c.proposals, mh_steps, pb, sb, ub, stride);
        c.v.side_stride = stride;
        return LDA_OK;
    }
    cudaStreamSynchronize(c.stream);
    drop_graphs(c);
    dev_free(c, c.v.prop);
    dev_free(c, c.v.dside);
    dev_free(c, c.v.ua_w);
    c.v.prop = nullptr;
    c.v.dside = nullptr;
    c.v.ua_w = nullptr;
    c.side_steps = 0;
    bytes_for(c.proposals, mh_steps, pb, sb, ub, stride);
    c.v.prop = dev_alloc(c, pb);
    c.v.dside = (uint32_t*)dev_alloc(c, sb);
    c.v.ua_w = (uint32_t*)dev_alloc(c, ub);
    if (!c.v.prop || !c.v.dside || !c.v.ua_w) {
        c.err = "device allocation failed";
        return LDA_ENOMEM;
    }
    c.v.side_stride = stride;
    c.side_steps = mh_steps;
    c.side_mode = c.proposals;
    return LDA_OK;
}

namespace lda {

void set_wide_counts(Ctx& c, bool wide)
{
    if (c.wide_counts != wide && c.cold_direct) drop_graphs(c);  // the accept pass takes another kernel
    c.wide_counts = wide;
}

void rebuild_counts(Ctx& c)
{
    set_wide_counts(c, false);
    cudaMemsetAsync(c.v.nk_next, 0, (size_t)c.v.dense_stride * 4, c.stream);
    launch_count_wk(c);
    launch_count_k(c);
    exchange_nk(c);
    c.tables_valid = false;
}

// One sweep, kernel by kernel.  Returns the number of kernels.
static int queue_sweep(Ctx& c, int mh_steps)
{
    // several vocabulary slices: the sparse tables are built slice by slice inside pass 1.  The dense table beside
    // the sparse ones where its 5 to 80 us count (its cluster may have to wait for room among their CTAs).
    int n = 0;
    if (c.proposals == LDA_PROPOSALS_DOC) n += launch_begin_sweep(c);  // no word-proposal, no tables
    else if (c.slices.size() > 1) n += launch_alias_dense(c, true);
    else if (c.N <= SIDE_BY_SIDE_MAX_TOKENS) n += launch_alias_sparse(c, false, true);
    else n += launch_alias_dense(c, true) + launch_alias_sparse(c, false);
    n += launch_sample(c, mh_steps);
    n += launch_count_wk(c);
    n += launch_count_k(c);
    return n;
}

// The same as a graph: the launches of a sweep and the waits between its streams are worked out once
// and cost the host one call.  Worth it from the third sweep of a configuration on (building it takes
// as long as launching a handful of sweeps kernel by kernel).  False: launch it kernel by kernel.
constexpr int GRAPH_AFTER = 2;
static bool replay_sweep(Ctx& c, int mh_steps)
{
    if (c.graph_refused) return false;
    if (c.graph_steps != mh_steps || c.graph_mode != c.proposals || c.graph_seed != c.seed) {
        drop_graphs(c);
        c.graph_steps = mh_steps;
        c.graph_mode = c.proposals;
        c.graph_seed = c.seed;
    }
    if (c.plain_sweeps < GRAPH_AFTER) {
        ++c.plain_sweeps;
        return false;
    }
    cudaGraphExec_t& exec = c.graph[c.v.nk < c.v.nk_next ? 0 : 1];
    if (!exec) {
        cudaGraph_t graph = nullptr;
        if (!c.capture && cudaStreamCreateWithFlags(&c.capture, cudaStreamNonBlocking) != cudaSuccess) c.capture = nullptr;
        bool ok = c.capture && cudaStreamBeginCapture(c.capture, cudaStreamCaptureModeThreadLocal) == cudaSuccess;
        if (ok) {
            const cudaStream_t stream = c.stream;
            c.stream = c.capture;
            c.graph_launches = queue_sweep(c, mh_steps);
            c.stream = stream;
            ok = cudaStreamEndCapture(c.capture, &graph) == cudaSuccess && graph &&
                 cudaGraphInstantiate(&exec, graph, 0) == cudaSuccess;
        }
        if (graph) cudaGraphDestroy(graph);
        if (!ok) {
            cudaGetLastError();
            exec = nullptr;
            c.graph_refused = true;
            return false;
        }
    }
    return cudaGraphLaunch(exec, c.stream) == cudaSuccess;
}

// Phase times of a batch of sweeps from the start stamps of their kernels.
static void add_phase_times(const Ctx& c, const SweepReport& r, int batch, lda_stats& s)
{
    auto first_of = [](unsigned long long a, unsigned long long b, unsigned long long otherwise) {
        if (!a || (b && b < a)) a = b;
        return a ? a : otherwise;
    };
    for (int b = 0; b < batch; ++b) {
        const unsigned long long* t = r.stamps[b];
        const unsigned long long end = b + 1 < batch ? r.stamps[b + 1][STAMP_DENSE] : r.end;
        const unsigned long long begin = t[STAMP_DENSE];
        const unsigned long long nk = first_of(t[STAMP_NK_DENSE], t[STAMP_NK_SPARSE], end);
        const unsigned long long wk = first_of(first_of(t[STAMP_ROWS], t[STAMP_WARM_ROWS], 0), t[STAMP_HIST], nk);
        const unsigned long long acc = first_of(first_of(t[STAMP_ACCEPT_HOT], t[STAMP_ACCEPT_WARM], 0), t[STAMP_ACCEPT_COLD], wk);
        const unsigned long long doc = first_of(t[STAMP_DOC_TILES], t[STAMP_DOC_LONG], acc);
        const unsigned long long pro = first_of(t[STAMP_PROPOSE_HOT], t[STAMP_PROPOSE_COLD],
                                                c.slices.size() > 1 ? t[STAMP_DENSE_END] : doc);
        auto ms = [](unsigned long long from, unsigned long long to) { return to > from ? 1e-6f * (float)(to - from) : 0.f; };
        // the sparse tables are built beside the dense one
        const unsigned long long dense_end = std::min(t[STAMP_DENSE_END], pro);
        s.ms_alias_dense += ms(begin, dense_end);
        s.ms_alias_sparse += ms(dense_end, pro);
        s.ms_propose += ms(pro, doc);
        s.ms_doc_side += ms(doc, acc);
        s.ms_accept += ms(acc, wk);
        s.ms_sample += ms(pro, wk);
        s.ms_count_wk += ms(wk, nk);
        s.ms_count_k += ms(nk, end);
        s.ms_total += ms(begin, end);
    }
}

static int ensure_tables(Ctx& c)
{
    if (c.tables_valid) return LDA_OK;
    launch_alias_dense(c, false);
    launch_alias_sparse(c, true);  // the running slice's (lda_get_tables walks the slices itself)
    int bits = 0;
    int rc = read_err(c, &bits);
    if (rc) return rc;
    if (bits) return fail(&c, LDA_EINTERNAL, "alias construction raised the device error word");
    c.tables_valid = true;
    return LDA_OK;
}

// What one pass over the document offsets tells.
struct Documents {
    std::vector<int32_t> off;  // the offsets in 32 bits
    int64_t longest = 0, nonempty = 0;
};

static int scan_documents(Ctx* c, int64_t n_tokens, const int64_t* doc_off, int64_t n_docs, Documents& docs)
{
    if (n_tokens >= 2147483648ll || n_docs >= 2147483647ll) return fail(c, LDA_ERANGE, "n_tokens and n_docs must be below 2^31");
    if (doc_off[0] != 0 || doc_off[n_docs] != n_tokens)
        return fail(c, LDA_ERANGE, "doc_offsets must start at 0 and end at n_tokens");
    docs.off.resize((size_t)n_docs + 1);
    bool ordered = true;  // by comparison: the difference of two offsets that are not in order may wrap
    for (int64_t d = 0; d < n_docs; ++d) {
        const int64_t a = doc_off[d], b = doc_off[d + 1];
        ordered = ordered && a <= b;
        const int64_t len = (int64_t)((uint64_t)b - (uint64_t)a);
        docs.longest = std::max(docs.longest, len);
        docs.nonempty += len > 0;
        docs.off[(size_t)d + 1] = (int32_t)b;
    }
    if (!ordered) return fail(c, LDA_ERANGE, "doc_offsets must be non-decreasing");
    return LDA_OK;
}

// Work lists on their way to the device: one allocation and one copy for all of them.  The lists stay where they
// are until send().
struct ListPack {
    struct Entry {
        const void* list;
        size_t bytes, at;
        void** target;
    };
    std::vector<Entry> lists;
    size_t total = 0;
    std::unique_ptr<char[]> host;  // until the copy is done
    template <typename E, typename P>
    void add(const std::vector<E>& list, P** target)
    {
        lists.push_back({list.data(), list.size() * sizeof(E), total, const_cast<void**>(reinterpret_cast<const void* const*>(target))});
        total = (total + lists.back().bytes + 15) / 16 * 16;
    }
    bool send(Ctx& c)
    {
        char* dev = (char*)dev_alloc(c, total);
        host.reset(new char[total]);
        for (const Entry& l : lists) {
            if (l.bytes) std::memcpy(host.get() + l.at, l.list, l.bytes);
            *l.target = dev + l.at;
        }
        return dev && cudaMemcpyAsync(dev, host.get(), total, cudaMemcpyHostToDevice, c.stream) == cudaSuccess;
    }
};

// A task beside the caller, on a thread of its own where it is worth one (and one can be had).  join() says whether
// it had the memory it needed.
struct Beside {
    std::thread thread;
    bool ok = true;
    template <typename F>
    Beside(bool worth_it, F f)
    {
        const auto task = [this, f] {
            try {
                f();
            } catch (const std::bad_alloc&) {
                ok = false;
            }
        };
        if (worth_it) {
            try {
                thread = std::thread(task);
                return;
            } catch (const std::system_error&) {
            }
        }
        task();
    }
    bool join()
    {
        if (thread.joinable()) thread.join();
        return ok;
    }
    ~Beside() { join(); }
};

static int load_lists(Ctx& c, const int32_t* words_dev, int64_t n_tokens, const Documents& docs, int64_t n_docs)
{
    free_corpus(c);
    c.N = n_tokens;
    c.D = n_docs;
    View& v = c.v;
    v.N = (int32_t)n_tokens;
    v.D = (int32_t)n_docs;
    const int32_t V = c.V, K = c.K;
    const int32_t N = v.N, D = v.D;
    const std::vector<int32_t>& doc_off = docs.off;

    int tb = 1;
    while ((1ll << tb) < (long long)K) ++tb;
    int cb = 1;  // a count never has all bits set, so no entry equals the empty-slot marker
    while ((1ll << cb) <= docs.longest + 1) ++cb;
    if (tb + cb > 32) {
        free_corpus(c);
        return fail(&c, LDA_ERANGE, "bits(K-1) + bits(longest document) exceeds 32");
    }
    v.topic_bits = tb;
    v.count_bits = cb;
    v.tok_base = (uint32_t)c.shard_first_token;

    // shape and form of the document tiles
    int32_t dense_docs = 0;
    {
        // A document that does not fit a tile takes the long documents' kernels.  The tile shape is the one with the
        // least estimated time, the smaller of two unless the larger is a tenth better; the relative costs per token are
        // measured (12 M tokens of 4000-token documents at K = 777, 30-70 M of 300 to 1000 at K = 21 to 12 000, 200 M of
        // log-normal ones at K = 100 000): large tiles leave few CTAs per multiprocessor, a document alone in a tile
        // leaves part of it empty, a table in device memory is the slower the less shared memory can stand in for it.
        // Tables of tiles: a counter per topic when a tile holds enough documents' worth of them to be filled (two
        // counters take the room of a slot), hashed otherwise.
        constexpr double TILE_COST[2][DOC_TILE_SHAPES] = {{1.0, 1.0, 1.0, 1.05}, {1.0, 1.0, 1.1, 1.2}};
        const int32_t mean_len = N / std::max(1, D);
        const auto dense_of = [&](int32_t tile) { return 2 * DOC_TILE_SLOTS * tile / (K + 1); };
        const auto is_dense = [&](int32_t tile) {
            return D > 0 && dense_of(tile) > 0 && (int64_t)dense_of(tile) * mean_len >= tile - mean_len;
        };
        double cost[DOC_TILE_SHAPES] = {};
        int64_t inside[DOC_TILE_SHAPES] = {}, rest = N;
        for (int32_t d = 0; d < D && docs.longest > DOC_TILE_TOKENS[0] / 2; ++d) {
            const int32_t len = doc_off[d + 1] - doc_off[d];
            if (len <= DOC_TILE_TOKENS[0] / 2) continue;
            rest -= len;
            const double outside = K > DK_SLOTS_PER_TOKEN_HOST * (int64_t)len ? 3.7 : K > LONG_STAGE_MAX_K ? 2.8 : 2.6;
            for (int sft = 0; sft < DOC_TILE_SHAPES; ++sft) {
                const int32_t tile = DOC_TILE_TOKENS[sft];
                inside[sft] += len > tile ? 0 : len;
                cost[sft] += len > tile          ? outside * len
                             : 2 * len > tile    ? TILE_COST[is_dense(tile)][sft] * std::max((double)len, 0.75 * tile)
                                                 : TILE_COST[is_dense(tile)][sft] * len;
            }
        }
        int shape = 0;
        for (int sft = 0; sft < DOC_TILE_SHAPES; ++sft) {
            cost[sft] += TILE_COST[is_dense(DOC_TILE_TOKENS[sft])][sft] * (double)rest;
            // (where most tokens are in longer documents anyway, a few large tiles only make a tail: 4000-token documents,
            // 272 us per pass with the largest shape, 224 with the smallest)
            if (cost[sft] < 0.9 * cost[shape] && 3 * (inside[sft] + rest) >= N) shape = sft;
        }
        c.doc_tile = DOC_TILE_TOKENS[shape];
        c.doc_threads = DOC_TILE_THREADS[shape];
        c.doc_dense = is_dense(c.doc_tile);
        dense_docs = dense_of(c.doc_tile);
        // Tokens per block of the block-major order: small blocks keep the document pass's scattered accesses in L2, long
        // ones make the word-order passes' runs longer.  With hashed tables the document pass is bound by
        // its instructions and 2^22 is best (738 M tokens, K = 10 000: 23.2 ms per sweep, 24.0 with 2^20); with
        // counters by those accesses, and 2^20 is (99 M tokens, K = 1000: 3.08 ms, 3.35 with 2^22).
        c.block_shift = c.block_option ? c.block_option : c.doc_dense ? 20 : 22;
        v.block_shift = c.block_shift;
    }

    // The documents' lists are made on another thread; the sorts are queued, the words' lists made beside the second.
    LayoutTemps temps;
    struct Release {
        Ctx& c;
        LayoutTemps& t;
        void now()
        {
            cudaStreamSynchronize(c.stream);
            for (void* p : t.held) raw_free(c, p);
            t.held.clear();
        }
        ~Release() { now(); }
    } release{c, temps};
    // tiles of whole documents: for the MH step, and for the sorted n_kd rows (<= SORT_TILE tokens and <= ROW_TILE_WORDS
    // documents each); made beside all that follows (400 000 documents: 1.6 ms on one core)
    std::vector<int32_t> doc_tiles, long_docs, doc_sort_tiles, doc_sort_long;
    const int32_t tile = c.doc_tile, tile_docs = c.doc_dense ? std::min(dense_docs, tile) : tile;
    const auto pack = [&](int32_t tokens, int32_t documents, std::vector<int32_t>& tiles, std::vector<int32_t>& longer) {
        int32_t s0 = 0, tok = 0;
        auto close = [&](int32_t s1) {
            if (s1 > s0) { tiles.push_back(s0); tiles.push_back(s1); }
        };
        for (int32_t d = 0; d < D; ++d) {
            const int32_t len = doc_off[d + 1] - doc_off[d];
            if (len > tokens) { close(d); s0 = d + 1; tok = 0; longer.push_back(d); continue; }
            if (tok + len > tokens || d - s0 >= documents) { close(d); s0 = d; tok = 0; }
            tok += len;
        }
        close(D);
    };
    Beside doc_lists(D > 20000, [&, tile, tile_docs] { pack(tile, tile_docs, doc_tiles, long_docs); });
    Beside doc_sort_lists(D > 20000, [&] { pack(SORT_TILE, ROW_TILE_WORDS, doc_sort_tiles, doc_sort_long); });
    int rc = build_layout(c, words_dev, doc_off, temps);
    if (rc != LDA_OK) {
        cudaStreamSynchronize(c.stream);
        cudaGetLastError();
        free_corpus(c);
        return fail(&c, rc, "building the word-sorted layout failed");
    }
    std::unique_ptr<int32_t[]> word_off(new int32_t[(size_t)V + 1]);
    int bits = 0;
    cudaStreamWaitEvent(c.side[0], c.ev_chunk, 0);  // word_off is there
    if (cudaMemcpyAsync(word_off.get(), v.word_off, ((size_t)V + 1) * 4, cudaMemcpyDeviceToHost, c.side[0]) != cudaSuccess ||
        cudaMemcpyAsync(&bits, v.err, sizeof(int), cudaMemcpyDeviceToHost, c.side[0]) != cudaSuccess ||
        cudaStreamSynchronize(c.side[0]) != cudaSuccess) {
        cudaStreamSynchronize(c.stream);
        free_corpus(c);
        return cuda_fail(&c, "copying word offsets");
    }
    if (bits) {
        read_err(c, &bits);  // waits for the stream and clears the word
        free_corpus(c);
        return fail(&c, LDA_ERANGE, "word id outside [0,V)");
    }

    // --- dense / sparse class of every word (Section 5) ---------------------------------
    // tf_here: the word's tokens in this corpus (its token range); tf: what the word's row and class
    // are sized for -- the same, unless the corpus is one shard of a larger one (lda_set_shard), in
    // which case the row has to hold the counts of all shards
    // The host's lists go over the words present only: a vocabulary may have ten times as many as the corpus uses.
    const int32_t* global_tf = c.shard_global_tf.empty() ? nullptr : c.shard_global_tf.data();
    const int32_t* const off = word_off.get();
    const auto tf_here = [off](int32_t w) { return off[w + 1] - off[w]; };
    const auto tf = [=](int32_t w) { return global_tf ? std::max(tf_here(w), global_tf[w]) : tf_here(w); };
    std::vector<int32_t> present;
    present.reserve((size_t)std::min<int64_t>(V, global_tf ? V : (int64_t)N));
    for (int32_t w = 0; w < V; ++w)
        if (tf(w) > 0) present.push_back(w);
    int32_t tf_cut = INT32_MAX;
    const int64_t n_top = std::min<int64_t>((int64_t)std::floor(c.dense_frac * (double)V), V);
    if (n_top > 0) {
        // the n_top-th largest frequency -- but a dense row of K counters only pays for a word with a fair share of K
        // tokens.  By a count of each frequency, the few very large ones by themselves.
        constexpr int32_t COUNTED = 1 << 13;
        tf_cut = std::max((int32_t)std::max(1.0, c.dense_min_tf), K / 8);
        std::vector<int32_t> words_of(COUNTED), above;
        int32_t most = 0;
        for (const int32_t w : present) {
            const int32_t t = tf(w);
            if (t <= tf_cut) continue;
            if (t < COUNTED) { ++words_of[(size_t)t]; most = std::max(most, t); }
            else above.push_back(t);
        }
        if ((int64_t)above.size() >= n_top) {
            std::nth_element(above.begin(), above.begin() + (n_top - 1), above.end(), std::greater<int32_t>());
            tf_cut = above[(size_t)n_top - 1];
        } else {
            int64_t n = (int64_t)above.size();
            for (int32_t t = most; t > tf_cut; --t)
                if ((n += words_of[(size_t)t]) >= n_top) tf_cut = t;  // ends the loop
        }
    }
    // K above the staging limit: only words with more than WARM_MAX_TF tokens get a dense row, the
    // others with more tokens than a tail tile holds a sorted row built by a CTA of their own
    const bool warm_class = K > HOT_STAGE_MAX_K;
    std::vector<int32_t> warm_words;
    // How the words' tokens are cut into runs.  A run is staged, or counted, by one CTA, so long runs
    // cost the least work -- but the pass lasts as long as its longest CTA, and a corpus of a few million
    // tokens in the longest runs occupies a handful of multiprocessors.  So: the longest run that
    // still gives every multiprocessor `per_sm` CTAs, and no shorter than what its staging is worth
    // (measured on 2 M tokens, K = 100: histograms 56 -> 8 us, accept pass of the hot words 40 -> 9 us).
    const auto run_for = [&](int64_t tokens, int64_t per_sm, int32_t longest, int32_t shortest) {
        int32_t r = longest;
        while (r > shortest && tokens / r < per_sm * c.n_sm) r /= 2;
        return std::max(r, shortest);
    };
    const auto is_hot = [tf](int32_t w) { return tf(w) > COLD_TILE; };
    const auto has_warm_row = [=](int32_t w) { return warm_class && tf(w) > SORT_TILE && tf(w) <= WARM_MAX_TF; };
    const auto has_dense_row = [=](int32_t w) { return !has_warm_row(w) && (tf(w) > SORT_TILE || tf(w) >= tf_cut); };
    int64_t t_hot = 0, t_cold = 0, t_dense = 0, cap_total = 0;
    for (const int32_t w : present) {
        (is_hot(w) ? t_hot : t_cold) += tf_here(w);
        if (has_dense_row(w)) t_dense += tf_here(w);
        cap_total += std::min(tf(w), K);
    }
    int32_t k_pow2 = 1;  // a row of K counters: staged by the accept pass, added up by the histograms
    while (k_pow2 < K) k_pow2 *= 2;
    const int32_t hist_run = run_for(t_dense, 8, HIST_RUN_MAX, std::min(std::max(4 * k_pow2, 4096), HIST_RUN_MAX));
    // a staged row of K counters (and n_k) is worth a quarter of K tokens or more; rows that are not staged
    // (K > HOT_STAGE_MAX_K: left in device memory, or sorted and no longer than the word's token count) less
    const int32_t hot_tile = run_for(t_hot, 4, HOT_TILE_MAX, warm_class ? 1024 : std::min(std::max(k_pow2 / 4, 2048), 8192));
    int32_t propose_tile = run_for(t_hot, 4, HOT_TILE_PROPOSE_MAX, 2048);
    if (propose_tile == 2048) propose_tile = 1536;  // one turn of the two-step kernel
    const int32_t cold_tile = run_for(t_cold, 4, COLD_TILE, 256);
    // tail tiles of few enough words for a counter per word and topic, if they still hold a fair number of tokens
    const int32_t direct_words = std::min(COLD_DIRECT / K, COLD_WORDS);
    c.cold_direct = direct_words > 0 && t_cold / std::max(1, V) * direct_words >= cold_tile / 2;
    const int32_t cold_words = c.cold_direct ? direct_words : COLD_WORDS;
    const bool sorted_rows = K > WORD_ROWS_BITMAP_MAX_K;
    const int32_t row_tile = run_for(N - t_dense, 4, SORT_TILE, 256), row_tile_words = sorted_rows ? SORT_TILE : ROW_TILE_WORDS;

    std::vector<int32_t> dense_words, alias_words[ALIAS_CLASSES], hot_runs, acc_runs, word_tiles;
    // vocabulary slices of about equal row capacity; slice_w[s] = first word of slice s, slice_row[s] = room of the words before
    const int n_slices = std::max(1, c.alias_slices);
    std::vector<int32_t> slice_w((size_t)n_slices + 1, V);
    std::vector<int64_t> slice_row((size_t)n_slices + 1, cap_total);
    slice_w[0] = 0;
    slice_row[0] = 0;
    if (n_slices > 1) {
        int64_t cap_sum = 0;
        int32_t end = 0;  // one past the last word seen
        int sl = 1;
        for (const int32_t w : present) {
            // (the first word before which there is that much room)
            for (; sl < n_slices && cap_total * sl / n_slices <= cap_sum; ++sl) {
                slice_w[(size_t)sl] = cap_total * sl / n_slices > 0 ? end : 0;
                slice_row[(size_t)sl] = cap_sum;
            }
            end = w + 1;
            cap_sum += std::min(tf(w), K);
        }
    }
    // The lists of words do not depend on one another (580 000 words: 1 to 2 ms each on one core).
    const bool many_words = present.size() > 50000;
    Beside class_lists(many_words, [&, tf, tf_here, has_warm_row, has_dense_row] {
        for (const int32_t w : present) {
            const int32_t cap = std::min(tf(w), K);
            for (int i = 0; i < ALIAS_CLASSES && cap > ALIAS_CLASS_MAX[i]; ++i) alias_words[i].push_back(w);
            if (has_warm_row(w)) {
                warm_words.push_back(w);
            } else if (has_dense_row(w)) {
                dense_words.push_back(w);
                const int32_t runs = std::max(1, (tf_here(w) + hist_run - 1) / hist_run);
                for (int32_t i = 0; i < runs; ++i) {
                    const int32_t o = i * hist_run;
                    hot_runs.insert(hot_runs.end(), {w, word_off[w] + o, std::min(hist_run, tf_here(w) - o),
                                                     runs > 1 ? (int32_t)acc_runs.size() : -1});
                }
                if (runs > 1) acc_runs.push_back(runs);
            }
        }
    });
    // tiles of consecutive sparse words: <= row_tile tokens (or one longer word) and <= row_tile_words words each
    Beside word_tile_list(many_words, [&, tf, has_dense_row, row_tile, row_tile_words] {
        int32_t s0 = 0, s1 = 0, tok = 0;
        auto close = [&] {
            if (s1 > s0) { word_tiles.push_back(s0); word_tiles.push_back(s1); }
        };
        for (const int32_t w : present) {
            const bool other = has_dense_row(w) || tf(w) > SORT_TILE;
            if (other || tok + tf(w) > row_tile || w - s0 >= row_tile_words) { close(); s0 = s1 = w; tok = 0; }
            if (other) continue;
            if (!tok) s0 = w;
            s1 = w + 1;
            tok += tf(w);
        }
        close();
    });
    // MH kernel work lists: a hot word (more tokens than a tail tile holds; it has a dense row by
    // the rule above) is cut into runs, tail words are packed whole into tiles, one longer than a tile cut
    std::vector<int32_t> hot_tiles, hot_tiles_warm, hot_tiles_propose, cold_tiles;
    {
        static_assert(COLD_TILE >= SORT_TILE, "every word longer than a tail tile must have a dense row or a warm one");
        int32_t s0 = 0, s1 = 0, tok = 0;
        auto close = [&] {
            if (s1 > s0 && word_off[s1] > word_off[s0])
                cold_tiles.insert(cold_tiles.end(), {s0, s1, word_off[s0], word_off[s1] - word_off[s0]});
        };
        auto cut = [&](std::vector<int32_t>& list, int32_t w, int32_t run) {
            for (int32_t o = 0; o < tf_here(w); o += run)
                list.insert(list.end(), {w, word_off[w] + o, std::min(run, tf_here(w) - o)});
        };
        int sl = 1;
        for (const int32_t w : present) {
            bool fresh = false;  // no tile reaches across two slices
            for (; sl < n_slices && slice_w[(size_t)sl] <= w; ++sl) fresh = true;
            const bool alone = is_hot(w) || tf(w) > cold_tile;
            if (fresh || alone || tok + tf(w) > cold_tile || w - s0 >= cold_words) { close(); s0 = s1 = w; tok = 0; }
            if (is_hot(w)) {
                cut(has_dense_row(w) ? hot_tiles : hot_tiles_warm, w, hot_tile);
                cut(hot_tiles_propose, w, propose_tile);
            } else if (alone) {
                for (int32_t o = 0; o < tf_here(w); o += cold_tile)
                    cold_tiles.insert(cold_tiles.end(), {w, w + 1, word_off[w] + o, std::min(cold_tile, tf_here(w) - o)});
            } else {
                if (!tok) s0 = w;
                s1 = w + 1;
                tok += tf(w);
            }
        }
        close();
    }
    bool lists_ok = true;
    for (Beside* b : {&doc_lists, &doc_sort_lists, &word_tile_list, &class_lists}) lists_ok = b->join() && lists_ok;
    if (!lists_ok) { free_corpus(c); return fail(&c, LDA_ENOMEM, "host allocation failed"); }
    c.n_dense = (int32_t)dense_words.size();
    c.n_doc_sort_tiles = (int32_t)(doc_sort_tiles.size() / 2);
    c.n_doc_sort_long = (int32_t)doc_sort_long.size();
    c.n_word_tiles = (int32_t)(word_tiles.size() / 2);
    c.n_doc_tiles = (int32_t)(doc_tiles.size() / 2);
    c.n_hot_runs = (int32_t)(hot_runs.size() / 4);
    choose_nk_mode(c);
    c.n_long_docs = (int32_t)long_docs.size();
    for (int i = 0; i < ALIAS_CLASSES; ++i) c.n_alias_words[i] = (int32_t)alias_words[i].size();
    c.n_hot_tiles = (int32_t)(hot_tiles.size() / 3);
    c.n_hot_tiles_warm = (int32_t)(hot_tiles_warm.size() / 3);
    c.n_warm = (int32_t)warm_words.size();
    c.n_hot_tiles_propose = (int32_t)(hot_tiles_propose.size() / 3);
    c.n_cold_tiles = (int32_t)(cold_tiles.size() / 4);
    c.slices.assign((size_t)n_slices, Ctx::Slice{});
    int64_t slice_rows_max = 1;
    {
        // every list is in ascending word order: a slice's part is a run of it
        auto first_at = [](const std::vector<int32_t>& list, size_t lo, size_t hi, int stride, int32_t w) {
            size_t a = lo, b = hi;  // first entry of [lo, hi) whose word is >= w
            while (a < b) {
                const size_t m = (a + b) / 2;
                if (list[m * stride] < w) a = m + 1; else b = m;
            }
            return (int32_t)a;
        };
        for (int sl = 0; sl < n_slices; ++sl) {
            Ctx::Slice& q = c.slices[(size_t)sl];
            q.w_lo = slice_w[(size_t)sl];
            q.w_hi = slice_w[(size_t)sl + 1];
            q.row_lo = slice_row[(size_t)sl];
            q.row_n = slice_row[(size_t)sl + 1] - q.row_lo;
            slice_rows_max = std::max(slice_rows_max, q.row_n);
            for (int i = 0; i < ALIAS_CLASSES; ++i) {
                q.alias_lo[i] = first_at(alias_words[i], 0, alias_words[i].size(), 1, q.w_lo);
                q.alias_n[i] = first_at(alias_words[i], 0, alias_words[i].size(), 1, q.w_hi) - q.alias_lo[i];
            }
            q.present_lo = first_at(present, 0, present.size(), 1, q.w_lo);
            q.present_n = first_at(present, 0, present.size(), 1, q.w_hi) - q.present_lo;
            q.hotp_lo = first_at(hot_tiles_propose, 0, (size_t)c.n_hot_tiles_propose, 3, q.w_lo);
            q.hotp_n = first_at(hot_tiles_propose, 0, (size_t)c.n_hot_tiles_propose, 3, q.w_hi) - q.hotp_lo;
            q.cold_lo = first_at(cold_tiles, 0, (size_t)c.n_cold_tiles, 4, q.w_lo);
            q.cold_n = first_at(cold_tiles, 0, (size_t)c.n_cold_tiles, 4, q.w_hi) - q.cold_lo;
        }
    }
    const size_t cap_alias = (size_t)slice_rows_max;

    release.now();  // before the large buffers are allocated: they may take over its memory
    const size_t n1 = (size_t)std::max<int64_t>(N, 1), cap1 = (size_t)std::max<int64_t>(cap_total, 1);
    const size_t zt = c.wide_topics ? 4 : 2;
    bool ok = true;
    auto A = [&](size_t bytes) { void* p = dev_alloc(c, bytes); ok = ok && p; return p; };
    v.zw = A(n1 * zt);
    v.zbm = A(2 * n1 * zt);  // (topic, first word-proposal) pairs
    v.rec = (uint32_t*)A(n1 * 4 + 16);  // + one aligned group of four words past the last record
    ListPack lists;
    const int32_t* dense_words_dev = nullptr;
    lists.add(dense_words, &dense_words_dev);
    lists.add(present, &c.present);
    lists.add(word_tiles, &c.word_tiles);
    lists.add(doc_tiles, &c.doc_tiles);
    lists.add(hot_runs, &c.hot_runs);
    lists.add(acc_runs, &c.acc_runs);
    lists.add(doc_sort_tiles, &c.doc_sort_tiles);
    lists.add(doc_sort_long, &c.doc_sort_long);
    for (int i = 0; i < ALIAS_CLASSES; ++i) lists.add(alias_words[i], &c.alias_words[i]);
    lists.add(hot_tiles, &c.hot_tiles);
    lists.add(hot_tiles_warm, &c.hot_tiles_warm);
    lists.add(warm_words, &c.warm_words);
    lists.add(hot_tiles_propose, &c.hot_tiles_propose);
    lists.add(cold_tiles, &c.cold_tiles);
    c.acc = (int32_t*)A(acc_runs.size() * (size_t)v.dense_stride * 4);
    c.acc_done = (int32_t*)A(acc_runs.size() * 4);
    v.wk_nnz = (int32_t*)A(((size_t)V + 1) * 4);  // one past the end is read by the row offsets' scan
    v.wk_topic = (uint32_t*)A(cap1 * 4);
    v.wk_count = (uint32_t*)A(cap1 * 4);
    v.dense_rows = (int32_t*)A(std::max<size_t>((size_t)c.n_dense * v.dense_stride, 1) * 4);
    c.al_thr0 = (uint32_t*)A(cap_alias * 4);
    c.al_idx0 = (uint32_t*)A(cap_alias * 4);
    c.al_pk0 = c.wide_topics ? nullptr : (uint2*)A(cap_alias * 8);
    v.dn_pk = (uint2*)A((size_t)K * 8);
    v.sp_mass = (unsigned long long*)A((size_t)V * 8);
    c.mix32 = (uint32_t*)A((size_t)V * 4);
    v.dn_thr = (uint32_t*)A((size_t)K * 4);
    v.dn_idx = (uint32_t*)A((size_t)K * 4);
    v.dense_mass = (unsigned long long*)A(8);
    v.nk = (int32_t*)A((size_t)v.dense_stride * 8);  // two, padded like a dense row: copied in 16-byte units
    v.nk_next = v.nk ? v.nk + v.dense_stride : nullptr;
    // tables of the documents longer than a tile (hashed ones first), and their chunks
    std::vector<LongDoc> long_list;
    std::vector<int32_t> long_chunks;
    long long slots = 0;
    for (const bool dense : {false, true}) {
        for (const int32_t d : long_docs) {
            const int32_t first = doc_off[d], len = doc_off[d + 1] - doc_off[d];
            if ((K <= DK_SLOTS_PER_TOKEN_HOST * (int64_t)len) != dense) continue;
            for (int32_t o = 0; o < len; o += LONG_CHUNK)
                long_chunks.insert(long_chunks.end(), {(int32_t)long_list.size(), first + o, std::min(LONG_CHUNK, len - o), 0});
            long_list.push_back(LongDoc{slots, first, len, dense, 0});
            slots += dense ? (K + 3) / 4 * 4 : (long long)DK_SLOTS_PER_TOKEN_HOST * len;
        }
        if (!dense) c.long_hashed_slots = slots;
    }
    c.long_slots = slots;
    c.n_long_chunks = (int32_t)(long_chunks.size() / 4);
    v.dk_slots = (uint32_t*)A((size_t)slots * 4 + 32);
    lists.add(long_list, &v.long_docs);
    lists.add(long_chunks, &c.long_chunks);
    ok = lists.send(c) && ok;
    c.sc_w0 = (unsigned long long*)A(cap_alias * 8);
    c.sc_de0 = (unsigned long long*)A(cap_alias * 8);
    c.sc_item0 = (uint32_t*)A(cap_alias * 4);
    c.sc_dense = (unsigned long long*)A((size_t)K * 8 * 3);
    c.red = (double*)A(sizeof(double) * (LL_WORD_PARTIALS + LL_DOC_PARTIALS));
    c.red_nnz = (uint32_t*)A(4 * LL_DOC_PARTIALS);
    c.red_i = (int64_t*)A(16);
    c.ll_tab = (double*)A(sizeof(double) * 3 * 512);
    c.ll_tile_part = (double*)A(sizeof(double) * std::max<size_t>((size_t)c.n_doc_tiles, 1));
    c.ll_tile_nnz = (uint32_t*)A(4 * std::max<size_t>((size_t)c.n_doc_tiles, 1));
    c.ll_tables_ready = false;
    if (!ok) { free_corpus(c); return fail(&c, LDA_ENOMEM, "device allocation failed"); }
    set_slice(c, 0);
    launch_dense_slots(c, dense_words_dev);
    cudaMemsetAsync(v.wk_nnz, 0, ((size_t)V + 1) * 4, c.stream);
    cudaMemsetAsync(v.sp_mass, 0, (size_t)V * 8, c.stream);
    cudaMemsetAsync(c.acc, 0, acc_runs.size() * (size_t)v.dense_stride * 4, c.stream);
    cudaMemsetAsync(c.acc_done, 0, acc_runs.size() * 4, c.stream);
    cudaMemsetAsync(v.dense_rows, 0, (size_t)c.n_dense * v.dense_stride * 4, c.stream);  // the rows' padding stays zero
    cudaMemsetAsync(v.nk, 0, (size_t)v.dense_stride * 8, c.stream);
    if (cudaStreamSynchronize(c.stream) != cudaSuccess) { free_corpus(c); return cuda_fail(&c, "load"); }
    c.stats = lda_stats{};
    c.stats.n_tokens = N;
    c.stats.n_docs = D;
    c.stats.n_dense_words = c.n_dense;
    c.n_nonempty_docs = docs.nonempty;
    c.loaded = true;
    return LDA_OK;
}

static int load_common(Ctx& c, const int32_t* words_dev, int64_t n_tokens, const Documents& docs, int64_t n_docs)
{
    const int rc = guarded(c, [&] { return load_lists(c, words_dev, n_tokens, docs, n_docs); });
    if (rc != LDA_OK && !c.allocs.empty()) {  // left behind by an exception
        cudaStreamSynchronize(c.stream);
        free_corpus(c);
    }
    return rc;
}

}  // namespace lda

using namespace lda;

struct lda_ctx {
    Ctx c;
};

extern "C" {

int lda_create(int32_t V, int32_t K, double alpha, double beta, lda_ctx** out)
{
    if (!out) return LDA_EINVAL;
    *out = nullptr;
    if (V <= 0 || K <= 0 || !(alpha > 0) || !(beta > 0) || !std::isfinite(alpha) || !std::isfinite(beta))
        return LDA_EINVAL;
    if (K > 131072) return LDA_ERANGE;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) { cudaGetLastError(); return LDA_ECUDA; }
    lda_ctx* h = new (std::nothrow) lda_ctx();
    if (!h) return LDA_ENOMEM;
    Ctx& c = h->c;
    c.V = V; c.K = K; c.alpha = alpha; c.beta = beta; c.device = dev;
    if (cudaDeviceGetAttribute(&c.n_sm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || c.n_sm < 1) {
        cudaGetLastError();
        c.n_sm = 148;
    }
    c.wide_topics = K > 65536;
    c.v.V = V; c.v.K = K; c.v.alpha = alpha; c.v.beta = beta;
    c.v.Vbeta = (double)V * beta;
    c.v.Kalpha = (double)K * alpha;
    c.v.dense_stride = (K + 3) & ~3;
    if (!PartsPool::pool().take(c) || cudaMemset(c.v.state, 0, sizeof(SweepState)) != cudaSuccess) {
        PartsPool::pool().give(c);
        delete h;
        cudaGetLastError();
        return LDA_ECUDA;
    }
    static std::once_flag limits_set[64];  // the kernels' limits stay with the device
    auto set_limits = [] {
        set_hist_smem_limits();
        set_sample_smem_limits();
        set_doc_smem_limits();
        set_alias_smem_limits();
        set_export_smem_limits();
        set_loglik_smem_limits();
        set_gibbs_smem_limits();
    };
    if (dev < 64) std::call_once(limits_set[dev], set_limits);
    else set_limits();
    *out = h;
    return LDA_OK;
}

void lda_destroy(lda_ctx* h)
{
    if (!h) return;
    Ctx& c = h->c;
    cudaSetDevice(c.device);
    cudaStreamSynchronize(c.stream);
    for (cudaStream_t s : {c.side[0], c.side[1], c.copy}) cudaStreamSynchronize(s);
    drop_graphs(c);
    if (c.capture) cudaStreamDestroy(c.capture);
    dev_free_all(c);
    PartsPool::pool().give(c);
    cudaGetLastError();
    delete h;
}

const char* lda_last_error(const lda_ctx* h) { return h ? h->c.err.c_str() : "null context"; }

int lda_set_stream(lda_ctx* h, void* cuda_stream)
{
    if (!h) return LDA_EINVAL;
    cudaStreamSynchronize(h->c.stream);
    h->c.stream = (cudaStream_t)cuda_stream;
    return LDA_OK;
}

int lda_set_allocator(lda_ctx* h, lda_alloc_fn alloc_fn, lda_free_fn free_fn, void* user)
{
    if (!h || (alloc_fn == nullptr) != (free_fn == nullptr)) return LDA_EINVAL;
    Ctx& c = h->c;
    if (c.loaded) return fail(&c, LDA_ESTATE, "lda_set_allocator must come before lda_load_corpus");
    c.alloc_fn = alloc_fn;
    c.free_fn = free_fn;
    c.alloc_user = user;
    return LDA_OK;
}

int lda_set_option(lda_ctx* h, const char* key, double value)
{
    if (!h || !key) return LDA_EINVAL;
    Ctx& c = h->c;
    if (c.loaded) return fail(&c, LDA_ESTATE, "options must be set before lda_load_corpus");
    if (!std::strcmp(key, "dense_frac")) {
        if (!(value >= 0.0 && value <= 1.0)) return fail(&c, LDA_EINVAL, "dense_frac must be in [0,1]");
        c.dense_frac = value;
        return LDA_OK;
    }
    if (!std::strcmp(key, "alias_slices")) {
        if (!(value >= 1.0 && value <= 256.0) || value != std::floor(value))
            return fail(&c, LDA_EINVAL, "alias_slices must be a whole number in [1,256]");
        c.alias_slices = (int)value;
        return LDA_OK;
    }
    if (!std::strcmp(key, "copy_chunk_log2")) {
        if (!(value >= 10.0 && value <= 30.0) || value != std::floor(value))
            return fail(&c, LDA_EINVAL, "copy_chunk_log2 must be a whole number in [10,30]");
        c.copy_chunk = (int64_t)1 << (int)value;
        return LDA_OK;
    }
    if (!std::strcmp(key, "dense_min_tf")) {
        if (!(value >= 1.0)) return fail(&c, LDA_EINVAL, "dense_min_tf must be >= 1");
        c.dense_min_tf = value;
        return LDA_OK;
    }
    if (!std::strcmp(key, "block_log2")) {
        if (!(value >= 10.0 && value <= 30.0)) return fail(&c, LDA_EINVAL, "block_log2 must be in [10,30]");
        c.block_option = (int)value;
        return LDA_OK;
    }
    return fail(&c, LDA_EINVAL, "unknown option");
}

int lda_set_proposals(lda_ctx* h, int mode)
{
    if (!h) return LDA_EINVAL;
    Ctx& c = h->c;
    if (mode != LDA_PROPOSALS_CYCLE && mode != LDA_PROPOSALS_WORD && mode != LDA_PROPOSALS_DOC)
        return fail(&c, LDA_EINVAL, "unknown proposal mode");
    c.proposals = mode;  // the exchange buffers are laid out again by the next sweep
    return LDA_OK;
}

int lda_load_corpus(lda_ctx* h, const int32_t* word_ids, int64_t n_tokens, const int64_t* doc_offsets,
                    int64_t n_docs)
{
    if (!h) return LDA_EINVAL;
    Ctx& c = h->c;
    if (!doc_offsets || n_tokens < 0 || n_docs < 0 || (n_tokens > 0 && !word_ids))
        return fail(&c, LDA_EINVAL, "null pointer or negative size");
    Documents docs;
    int rc = guarded(c, [&] { return scan_documents(&c, n_tokens, doc_offsets, n_docs, docs); });
    if (rc) return rc;
    if ((rc = check_device(c))) return rc;
    int32_t* wd = nullptr;
    if (!tmp_alloc(c, &wd, (size_t)std::max<int64_t>(n_tokens, 1) * 4)) return fail(&c, LDA_ENOMEM, "device allocation failed");
    if (copy_to_device(c, wd, word_ids, (size_t)n_tokens * 4) != cudaSuccess) {
        raw_free(c, wd);
        return cuda_fail(&c, "copying word ids");
    }
    rc = load_common(c, wd, n_tokens, docs, n_docs);
    cudaStreamSynchronize(c.stream);
    raw_free(c, wd);
    return rc;
}

int lda_load_corpus_device(lda_ctx* h, const int32_t* word_ids_dev, int64_t n_tokens,
                           const int64_t* doc_offsets_dev, int64_t n_docs)
{
    if (!h) return LDA_EINVAL;
    Ctx& c = h->c;
    if (!doc_offsets_dev || n_tokens < 0 || n_docs < 0 || (n_tokens > 0 && !word_ids_dev))
        return fail(&c, LDA_EINVAL, "null pointer or negative size");
    if (n_docs >= 2147483647ll) return fail(&c, LDA_ERANGE, "n_docs must be below 2^31");
    int rc = check_device(c);
    if (rc) return rc;
    std::vector<int64_t> off;
    if ((rc = guarded(c, [&] { off.resize((size_t)n_docs + 1); return LDA_OK; }))) return rc;
    // the offsets come after what the default stream has queued, as a copy on that stream does, whatever the
    // context's stream is
    if (cudaEventRecord(c.ev_chunk, cudaStreamLegacy) != cudaSuccess || cudaStreamWaitEvent(c.stream, c.ev_chunk, 0) != cudaSuccess ||
        copy_to_host(c, off.data(), doc_offsets_dev, ((size_t)n_docs + 1) * 8) != cudaSuccess)
        return cuda_fail(&c, "copying doc offsets");
    Documents docs;
    if ((rc = guarded(c, [&] { return scan_documents(&c, n_tokens, off.data(), n_docs, docs); }))) return rc;
    return load_common(c, word_ids_dev, n_tokens, docs, n_docs);
}

int lda_init(lda_ctx* h, uint64_t seed)
{
    if (!h) return LDA_EINVAL;
    Ctx& c = h->c;
    if (!c.loaded) return fail(&c, LDA_ESTATE, "lda_init before lda_load_corpus");
    int rc = check_device(c);
    if (rc) return rc;
    order_after_export(c);
    c.seed = seed;
    c.sweep = 0;
    launch_set_state(c);
    launch_init(c);
    rebuild_counts(c);
    int bits = 0;
    if ((rc = read_err(c, &bits))) return rc;
    if (bits) return fail(&c, LDA_EINTERNAL, "count rebuild raised the device error word");
    c.inited = true;
    return LDA_OK;
}

// Tokens per chunk of a transfer: the kernel's part of the first (or last) chunk runs beside no copy, so chunks
// are short, but a sixteenth of the corpus is short enough and 2^20 tokens are worth a copy of their own.  Above 2^28
// tokens a sixteenth is no longer short: 738 M tokens to the device, one sweep and back took 84.2 ms in chunks of 46 M
// tokens, 82.0 with 2^25, 81.9 with 2^24, 82.7 with 2^22.
static int64_t transfer_chunk(const Ctx& c)
{
    return c.copy_chunk ? c.copy_chunk : std::min<int64_t>((int64_t)1 << 24, std::max<int64_t>((int64_t)1 << 20, c.N / 16));
}

static int set_assignments(lda_ctx* h, const void* z, bool narrow, uint64_t seed, uint32_t sweep)
{
    if (!h) return LDA_EINVAL;
    Ctx& c = h->c;
    if (!c.loaded) return fail(&c, LDA_ESTATE, "lda_set_assignments before lda_load_corpus");
    if (narrow && c.wide_topics) return fail(&c, LDA_ERANGE, "16-bit assignments need K <= 65536");
    if (c.N > 0 && !z) return fail(&c, LDA_EINVAL, "null assignments");
    int rc = check_device(c);
    if (rc) return rc;
    // the record array (one word per token, only meaningful while the exported n_kd is valid)
    // doubles as the staging buffer: no allocation here
    char* zdev = reinterpret_cast<char*>(c.v.rec);
    order_after_export(c);
    // chunk by chunk on the copy stream, each chunk spread into the block-major order (on the context's
    // stream) while the next one is on its way
    const size_t zt = narrow ? 2 : 4;
    const int64_t chunk = transfer_chunk(c);
    cudaEventRecord(c.ev_chunk, c.stream);
    cudaStreamWaitEvent(c.copy, c.ev_chunk, 0);  // the staging buffer's earlier users are done
    for (int64_t first = 0; first < c.N; first += chunk) {
        const int64_t count = std::min<int64_t>(chunk, c.N - first);
        if (cudaMemcpyAsync(zdev + (size_t)first * zt, reinterpret_cast<const char*>(z) + (size_t)first * zt,
                            (size_t)count * zt, cudaMemcpyHostToDevice, c.copy) != cudaSuccess)
            return cuda_fail(&c, "copying assignments");
        cudaEventRecord(c.ev_chunk, c.copy);
        cudaStreamWaitEvent(c.stream, c.ev_chunk, 0);
        launch_spread_chunk(c, zdev, narrow, first, count);
    }
    launch_word_order_topics(c);
    int bits = 0;
    rc = read_err(c, &bits);
    if (rc) return rc;
    if (bits & ERR_TOPIC_RANGE) { c.inited = false; return fail(&c, LDA_ERANGE, "assignment outside [0,K)"); }
    c.seed = seed;
    c.sweep = sweep;
    launch_set_state(c);
    rebuild_counts(c);
    if ((rc = read_err(c, &bits))) return rc;
    if (bits) return fail(&c, LDA_EINTERNAL, "count rebuild raised the device error word");
    c.inited = true;
    return LDA_OK;
}

int lda_set_assignments(lda_ctx* h, const int32_t* z, uint64_t seed, uint32_t sweep)
{
    return set_assignments(h, z, false, seed, sweep);
}

int lda_set_assignments_u16(lda_ctx* h, const uint16_t* z, uint64_t seed, uint32_t sweep)
{
    return set_assignments(h, z, true, seed, sweep);
}

int lda_sweep(lda_ctx* h, int32_t iters, int32_t mh_steps)
{
    if (!h) return LDA_EINVAL;
    Ctx& c = h->c;
    if (iters < 0 || mh_steps < 1 || mh_steps > 1024)
        return fail(&c, LDA_EINVAL, "iters must be >= 0 and mh_steps in 1..1024");
    if (!c.inited) return fail(&c, LDA_ESTATE, "lda_sweep before lda_init");
    int rc = check_device(c);
    if (rc) return rc;
    order_after_export(c);
    if ((rc = ensure_exchange(c, mh_steps))) return rc;
    lda_stats& s = c.stats;
    s.ms_alias_dense = s.ms_alias_sparse = s.ms_sample = s.ms_count_wk = s.ms_count_k = s.ms_count_dk =
        s.ms_total = s.ms_propose = s.ms_doc_side = s.ms_accept = 0.f;
    s.kernel_launches = 0;
    s.iters = iters;
    s.word_proposed = s.word_accepted = s.doc_proposed = s.doc_accepted = 0;
    // Iterations are queued without waiting for each other; the host waits once per STAMP_RING of them
    // (and after the last) for the error word, the move counters and the phase times.
    for (int32_t it0 = 0; it0 < iters; it0 += STAMP_RING) {
        const int32_t batch = std::min<int32_t>(STAMP_RING, iters - it0);
        for (int32_t b = 0; b < batch; ++b) {
            s.kernel_launches += replay_sweep(c, mh_steps) ? c.graph_launches : queue_sweep(c, mh_steps);
            exchange_nk(c);
            c.tables_valid = false;
            c.sweep += 1;
        }
        launch_report(c);
        ++s.kernel_launches;
        cudaError_t e = cudaStreamSynchronize(c.stream);
        if (e == cudaSuccess) e = cudaGetLastError();
        if (e != cudaSuccess) {
            c.inited = false;
            c.err = std::string("sweep: ") + cudaGetErrorString(e);
            return LDA_ECUDA;
        }
        const SweepReport& r = *c.report;
        if (r.err) {
            // some iteration of this batch met inconsistent tables: the state is not to be trusted
            c.inited = false;
            c.err = "a kernel raised the device error word: " + std::to_string(r.err) +
                    " (call lda_init or lda_set_assignments again)";
            return LDA_EINTERNAL;
        }
        add_phase_times(c, r, batch, s);
        s.word_accepted += (int64_t)r.moves[0];
        s.doc_accepted += (int64_t)r.moves[1];
    }
    const int64_t n_word = c.proposals == LDA_PROPOSALS_CYCLE  ? (mh_steps + 1) / 2
                           : c.proposals == LDA_PROPOSALS_WORD ? mh_steps
                                                               : 0;
    s.word_proposed = (int64_t)iters * c.N * n_word;
    s.doc_proposed = (int64_t)iters * c.N * (mh_steps - n_word);
    return LDA_OK;
}

int lda_set_shard(lda_ctx* h, int64_t first_token, const int32_t* global_term_freq)
{
    if (!h) return LDA_EINVAL;
    Ctx& c = h->c;
    if (c.loaded) return fail(&c, LDA_ESTATE, "lda_set_shard must come before lda_load_corpus");
    if (first_token < 0 || first_token >= 4294967296ll) return fail(&c, LDA_ERANGE, "first_token must be in [0, 2^32)");
    c.shard_first_token = first_token;
    c.shard_global_tf.clear();
    if (global_term_freq) {
        for (int32_t w = 0; w < c.V; ++w)
            if (global_term_freq[w] < 0) return fail(&c, LDA_ERANGE, "negative term frequency");
        return guarded(c, [&] { c.shard_global_tf.assign(global_term_freq, global_term_freq + c.V); return LDA_OK; });
    }
    return LDA_OK;
}

int lda_word_counts_to_dense(lda_ctx* h, int32_t* nwk_dev)
{
    if (!h) return LDA_EINVAL;
    Ctx& c = h->c;
    if (!nwk_dev) return fail(&c, LDA_EINVAL, "null matrix");
    if (!c.inited) return fail(&c, LDA_ESTATE, "lda_word_counts_to_dense before lda_init");
    int rc = check_device(c);
    if (rc) return rc;
    launch_word_counts_to_dense(c, nwk_dev);
    if (cudaStreamSynchronize(c.stream) != cudaSuccess || cudaGetLastError() != cudaSuccess)
        return cuda_fail(&c, "writing the count matrix");
    return LDA_OK;
}

int lda_word_counts_from_dense(lda_ctx* h, const int32_t* nwk_dev)
{
    if (!h) return LDA_EINVAL;
    Ctx& c = h->c;
    if (!nwk_dev) return fail(&c, LDA_EINVAL, "null matrix");
    if (!c.inited) return fail(&c, LDA_ESTATE, "lda_word_counts_from_dense before lda_init");
    int rc = check_device(c);
    if (rc) return rc;
    launch_word_counts_from_dense(c, nwk_dev);
    c.tables_valid = false;
    int bits = 0;
    if ((rc = read_err(c, &bits))) { c.inited = false; return rc; }
    set_wide_counts(c, (bits & NOTE_WIDE_COUNT) != 0);
    if (bits & ~NOTE_WIDE_COUNT) {
        c.inited = false;
        return fail(&c, LDA_ERANGE,
                    "the matrix has negative entries or more nonzeros in a row than the term frequencies given to lda_set_shard allow");
    }
    return LDA_OK;
}

int lda_gibbs_sweep(lda_ctx* h, int32_t iters)
{
    if (!h) return LDA_EINVAL;
    Ctx& c = h->c;
    if (iters < 0) return fail(&c, LDA_EINVAL, "iters must be >= 0");
    if (!c.inited) return fail(&c, LDA_ESTATE, "lda_gibbs_sweep before lda_init");
    if (c.K > GIBBS_MAX_K) return fail(&c, LDA_ERANGE, "the exact-conditional sweep takes K <= 16384");
    if ((long long)c.V * c.K * 8 > GIBBS_MAX_PREFIX_BYTES)
        return fail(&c, LDA_ERANGE, "the exact-conditional sweep keeps V*K running sums: V*K*8 bytes must stay below 24 GiB");
    if ((double)c.K * c.alpha >= 131072.0) return fail(&c, LDA_ERANGE, "the exact-conditional sweep needs K*alpha < 2^17");
    if (c.v.count_bits > 19) return fail(&c, LDA_ERANGE, "the exact-conditional sweep takes documents shorter than 2^19 tokens");
    int rc = check_device(c);
    if (rc) return rc;
    order_after_export(c);
    rc = gibbs_sweep(c, iters);
    if (rc) return fail(&c, rc, "the exact-conditional sweep failed");
    int bits = 0;
    if ((rc = read_err(c, &bits))) { c.inited = false; return rc; }
    if (bits) {
        c.inited = false;
        return fail(&c, LDA_EINTERNAL, "a kernel of the exact-conditional sweep raised the device error word");
    }
    return LDA_OK;
}

int lda_loglik(lda_ctx* h, double* total, double* word_ll, double* doc_ll)
{
    if (!h) return LDA_EINVAL;
    Ctx& c = h->c;
    if (!c.inited) return fail(&c, LDA_ESTATE, "lda_loglik before lda_init");
    int rc = check_device(c);
    if (rc) return rc;
    double out[3];
    if (launch_loglik(c, out) < 0 || cudaPeekAtLastError() != cudaSuccess) return cuda_fail(&c, "log-likelihood");
    if (c.report->err) {
        int bits = 0;
        if ((rc = read_err(c, &bits))) return rc;  // clears it
        return fail(&c, LDA_EINTERNAL, "the log-likelihood kernels raised the device error word");
    }
    if (total) *total = out[0];
    if (word_ll) *word_ll = out[1];
    if (doc_ll) *doc_ll = out[2];
    return LDA_OK;
}

// The n_kw rows without any device memory: they are copied as they lie, room behind them included, and put together here.
static int word_rows_by_host(Ctx& c, int64_t* row_offsets, int32_t* topics, int32_t* counts, int64_t capacity, int64_t* nnz_out)
{
    const View& v = c.v;
    const size_t V = (size_t)c.V;
    std::vector<int32_t> nnz(V), start(V + 1), entries;
    if (copy_to_host(c, nnz.data(), v.wk_nnz, V * 4) != cudaSuccess || copy_to_host(c, start.data(), v.row_start, (V + 1) * 4) != cudaSuccess)
        return cuda_fail(&c, "copying row sizes");
    int64_t total = 0;
    for (const int32_t n : nnz) total += n;
    if (nnz_out) *nnz_out = total;
    if (!row_offsets && !topics && !counts) return LDA_OK;
    if (capacity < total) return fail(&c, LDA_ERANGE, "capacity below the number of nonzeros");
    if (row_offsets) {
        row_offsets[0] = 0;
        for (size_t w = 0; w < V; ++w) row_offsets[w + 1] = row_offsets[w] + nnz[w];
    }
    const std::pair<int32_t*, const uint32_t*> columns[2] = {{topics, v.wk_topic}, {counts, v.wk_count}};
    for (const auto& [to, from] : columns) {
        if (!to || !total) continue;
        entries.resize((size_t)start[V]);
        if (copy_to_host(c, entries.data(), from, entries.size() * 4) != cudaSuccess) return cuda_fail(&c, "copying the n_kw rows");
        int32_t* out = to;
        for (size_t w = 0; w < V; ++w) out = std::copy_n(entries.begin() + start[w], nnz[w], out);
    }
    return LDA_OK;
}

int lda_get_counts(lda_ctx* h, int which, int64_t* row_offsets, int32_t* topics, int32_t* counts,
                   int64_t capacity, int64_t* nnz_out)
{
    if (!h) return LDA_EINVAL;
    Ctx& c = h->c;
    if (!c.inited) return fail(&c, LDA_ESTATE, "lda_get_counts before lda_init");
    int rc = check_device(c);
    if (rc) return rc;
    order_after_export(c);
    const View& v = c.v;
    cudaStreamSynchronize(c.stream);
    if (which == LDA_NK) {
        if (nnz_out) *nnz_out = c.K;
        if (counts) {
            if (capacity < c.K) return fail(&c, LDA_ERANGE, "capacity below K");
            if (cudaMemcpy(counts, v.nk, (size_t)c.K * 4, cudaMemcpyDeviceToHost) != cudaSuccess)
                return cuda_fail(&c, "copying n_k");
        }
        return LDA_OK;
    }
    if (which == LDA_NDK) {
        // sorted rows are built on the device; only the row offsets and the nonzeros cross to the host
        const bool sizes_only = !row_offsets && !topics && !counts;
        DkCsr r;
        if ((rc = build_dk_csr(c, r, sizes_only))) return fail(&c, rc, "building the n_kd rows failed");
        int bits = 0;
        if ((rc = read_err(c, &bits))) { free_dk_csr(c, r); return rc; }
        if (bits) { free_dk_csr(c, r); return fail(&c, LDA_EINTERNAL, "the n_kd rows raised the device error word"); }
        const int64_t total = (int64_t)r.total;
        if (nnz_out) *nnz_out = total;
        if (sizes_only) { free_dk_csr(c, r); return LDA_OK; }
        if (capacity < total) { free_dk_csr(c, r); return fail(&c, LDA_ERANGE, "capacity below the number of nonzeros"); }
        static_assert(sizeof(long long) == sizeof(int64_t), "row offsets are copied as they are");
        bool ok = true;
        if (row_offsets) ok = ok && copy_to_host(c, row_offsets, r.row_off, ((size_t)c.D + 1) * 8) == cudaSuccess;
        if (topics && total) ok = ok && copy_to_host(c, topics, r.topic, (size_t)total * 4) == cudaSuccess;
        if (counts && total) ok = ok && copy_to_host(c, counts, r.count, (size_t)total * 4) == cudaSuccess;
        free_dk_csr(c, r);
        if (!ok) return cuda_fail(&c, "copying the n_kd rows");
        return LDA_OK;
    }
    if (which != LDA_NWK) return fail(&c, LDA_EINVAL, "unknown table");
    const bool sizes_only = !row_offsets && !topics && !counts;
    WkCsr r;
    rc = build_wk_csr(c, r, sizes_only);
    if (rc == LDA_ENOMEM)
        return guarded(c, [&] { return word_rows_by_host(c, row_offsets, topics, counts, capacity, nnz_out); });
    if (rc) return fail(&c, rc, "building the n_kw rows failed");
    const int64_t total = (int64_t)r.total;
    if (nnz_out) *nnz_out = total;
    if (!sizes_only && capacity < total) {
        cudaStreamSynchronize(c.stream);
        free_wk_csr(c, r);
        return fail(&c, LDA_ERANGE, "capacity below the number of nonzeros");
    }
    bool ok = true;
    if (row_offsets) ok = ok && copy_to_host(c, row_offsets, r.row_off, ((size_t)c.V + 1) * 8) == cudaSuccess;
    if (topics && total) ok = ok && copy_to_host(c, topics, r.topic, (size_t)total * 4) == cudaSuccess;
    if (counts && total) ok = ok && copy_to_host(c, counts, r.count, (size_t)total * 4) == cudaSuccess;
    cudaStreamSynchronize(c.stream);
    free_wk_csr(c, r);
    if (!ok) return cuda_fail(&c, "copying the n_kw rows");
    return LDA_OK;
}

constexpr size_t EXPORT_ONE_STREAM_BYTES = 256 << 10;
constexpr int64_t EXPORT_PAGEABLE_CHUNK = (int64_t)1 << 25;  // tokens
static int get_assignments(lda_ctx* h, void* z_out, bool narrow, bool wait)
{
    if (!h) return LDA_EINVAL;
    Ctx& c = h->c;
    if (!c.inited) return fail(&c, LDA_ESTATE, "lda_get_assignments before lda_init");
    if (narrow && c.wide_topics) return fail(&c, LDA_ERANGE, "16-bit assignments need K <= 65536");
    if (c.N > 0 && !z_out) return fail(&c, LDA_EINVAL, "null output");
    if (c.N == 0) return LDA_OK;
    int rc = check_device(c);
    if (rc) return rc;
    order_after_export(c);
    char* zdev = reinterpret_cast<char*>(c.v.rec);  // staging, see set_assignments()
    // chunk by chunk: collected into document order on the context's stream, copied out on the copy
    // stream while the next chunk is collected
    const size_t zt = narrow ? 2 : 4;
    if ((size_t)c.N * zt <= EXPORT_ONE_STREAM_BYTES) {
        // One piece of page-locked memory is written by the kernel that collects the topics: a copy behind it takes as long as one of a
        // sweep's kernels, and what a caller queues next waits for it (a sweep, a snapshot and the log-likelihood of 10 000
        // tokens: 74 -> 71 us, of 60 000: 87 -> 78).
        void* const view = (uintptr_t)z_out % zt == 0 ? device_view(z_out, (size_t)c.N * zt) : nullptr;
        if (view) {
            launch_export_chunk(c, view, narrow, 0, c.N);
            return wait ? wait_all(c) : LDA_OK;
        }
        // a copy of a few microseconds is not worth the events that would order a second stream
        launch_export_chunk(c, zdev, narrow, 0, c.N);
        if (cudaMemcpyAsync(z_out, zdev, (size_t)c.N * zt, cudaMemcpyDeviceToHost, c.stream) != cudaSuccess)
            return cuda_fail(&c, "copying assignments");
        return wait ? wait_all(c) : LDA_OK;
    }
    // A copy into memory that is not page-locked returns when it is done, and each has a price of its own: 20 M tokens
    // of 16 bits took 2.8 ms in chunks of a sixteenth, 2.0 in one.
    const int64_t chunk = c.copy_chunk || page_locked(z_out) ? transfer_chunk(c) : EXPORT_PAGEABLE_CHUNK;
    for (int64_t first = 0; first < c.N; first += chunk) {
        const int64_t count = std::min<int64_t>(chunk, c.N - first);
        launch_export_chunk(c, zdev, narrow, first, count);
        cudaEventRecord(c.ev_chunk, c.stream);
        cudaStreamWaitEvent(c.copy, c.ev_chunk, 0);
        if (cudaMemcpyAsync(reinterpret_cast<char*>(z_out) + (size_t)first * zt, zdev + (size_t)first * zt,
                            (size_t)count * zt, cudaMemcpyDeviceToHost, c.copy) != cudaSuccess)
            return cuda_fail(&c, "copying assignments");
    }
    cudaEventRecord(c.ev_export, c.copy);
    c.export_pending = true;
    return wait ? wait_all(c) : LDA_OK;
}

int lda_get_assignments(lda_ctx* h, int32_t* z_out) { return get_assignments(h, z_out, false, true); }

int lda_get_assignments_u16(lda_ctx* h, uint16_t* z_out) { return get_assignments(h, z_out, true, true); }

int lda_get_assignments_async(lda_ctx* h, int32_t* z_out) { return get_assignments(h, z_out, false, false); }

int lda_get_assignments_u16_async(lda_ctx* h, uint16_t* z_out) { return get_assignments(h, z_out, true, false); }

int lda_wait(lda_ctx* h)
{
    if (!h) return LDA_EINVAL;
    Ctx& c = h->c;
    int rc = check_device(c);
    if (rc) return rc;
    return wait_all(c);
}

static int get_tables(Ctx& c, uint32_t* sp_thr32, int32_t* sp_alias, int64_t capacity, uint32_t* mix32, uint32_t* dn_thr32,
                      int32_t* dn_alias, uint64_t* dense_mass)
{
    int rc = LDA_OK;
    const View& v = c.v;
    const size_t V = (size_t)c.V, K = (size_t)c.K;
    const bool want_sparse = sp_thr32 || sp_alias;
    std::vector<int32_t> nnz(V), start(V + 1);
    std::vector<uint32_t> a, b;
    if (want_sparse) {
        if (cudaMemcpy(nnz.data(), v.wk_nnz, V * 4, cudaMemcpyDeviceToHost) != cudaSuccess ||
            cudaMemcpy(start.data(), v.row_start, (V + 1) * 4, cudaMemcpyDeviceToHost) != cudaSuccess)
            return cuda_fail(&c, "copy");
        int64_t total = 0;
        for (size_t w = 0; w < V; ++w) total += nnz[w];
        if (capacity < total) return fail(&c, LDA_ERANGE, "capacity below the number of nonzeros");
        a.resize(std::max<size_t>((size_t)start[V], 1));
        b.resize(a.size());
    }
    // The device holds the sparse tables of one vocabulary slice at a time: build slice after slice
    // (one slice: the whole vocabulary, built once and kept until the counts change).
    const bool one = c.slices.size() == 1;
    if (one) {
        if ((rc = ensure_tables(c))) return rc;
    } else {
        c.tables_valid = false;
        launch_alias_dense(c, false);
    }
    for (size_t sl = 0; sl < c.slices.size(); ++sl) {
        const Ctx::Slice& q = c.slices[sl];
        if (!one) {
            set_slice(c, (int)sl);
            launch_alias_sparse(c, true);
            int bits = 0;
            if ((rc = read_err(c, &bits))) return rc;
            if (bits) return fail(&c, LDA_EINTERNAL, "alias construction raised the device error word");
        }
        if (want_sparse && q.row_n &&
            (cudaMemcpy(a.data() + q.row_lo, c.al_thr0, (size_t)q.row_n * 4, cudaMemcpyDeviceToHost) != cudaSuccess ||
             cudaMemcpy(b.data() + q.row_lo, c.al_idx0, (size_t)q.row_n * 4, cudaMemcpyDeviceToHost) != cudaSuccess))
            return cuda_fail(&c, "copy");
    }
    if (mix32) {
        launch_mix_thresholds(c, c.mix32);
        if (cudaStreamSynchronize(c.stream) != cudaSuccess ||
            cudaMemcpy(mix32, c.mix32, V * 4, cudaMemcpyDeviceToHost) != cudaSuccess)
            return cuda_fail(&c, "copy");
    }
    if (dn_thr32 && cudaMemcpy(dn_thr32, v.dn_thr, K * 4, cudaMemcpyDeviceToHost) != cudaSuccess) return cuda_fail(&c, "copy");
    if (dn_alias && cudaMemcpy(dn_alias, v.dn_idx, K * 4, cudaMemcpyDeviceToHost) != cudaSuccess) return cuda_fail(&c, "copy");
    if (dense_mass && cudaMemcpy(dense_mass, v.dense_mass, 8, cudaMemcpyDeviceToHost) != cudaSuccess) return cuda_fail(&c, "copy");
    if (!want_sparse) return LDA_OK;
    int64_t o = 0;
    for (size_t w = 0; w < V; ++w)
        for (int32_t j = 0; j < nnz[w]; ++j, ++o) {
            if (sp_thr32) sp_thr32[o] = a[(size_t)start[w] + j];
            if (sp_alias) sp_alias[o] = (int32_t)b[(size_t)start[w] + j];
        }
    return LDA_OK;
}

int lda_get_tables(lda_ctx* h, uint32_t* sp_thr32, int32_t* sp_alias, int64_t capacity, uint32_t* mix32,
                   uint32_t* dn_thr32, int32_t* dn_alias, uint64_t* dense_mass)
{
    if (!h) return LDA_EINVAL;
    Ctx& c = h->c;
    if (!c.inited) return fail(&c, LDA_ESTATE, "lda_get_tables before lda_init");
    int rc = check_device(c);
    if (rc) return rc;
    return guarded(c, [&] { return get_tables(c, sp_thr32, sp_alias, capacity, mix32, dn_thr32, dn_alias, dense_mass); });
}

int lda_get_stats(lda_ctx* h, lda_stats* out)
{
    if (!h || !out) return LDA_EINVAL;
    Ctx& c = h->c;
    if (c.inited) {
        if (check_device(c)) return LDA_ECUDA;
        int64_t a = 0, b = 0;
        launch_count_nnz(c, &a, &b);
        c.stats.nnz_wk = a;
        c.stats.nnz_dk = b;
    }
    c.stats.device_bytes = c.device_bytes;
    c.stats.sweeps_done = (int32_t)c.sweep;
    *out = c.stats;
    return LDA_OK;
}

}  // extern "C"
