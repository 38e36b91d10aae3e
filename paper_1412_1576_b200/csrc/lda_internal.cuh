// Internal declarations shared by the library's translation units.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include <string>
#include <vector>

#include "../../include/lda_b200.h"

namespace lda {

// The proposal schedule of a chain (Section 4.3): whether step m draws the doc-proposal, and the
// running index of step m among the steps of its own kind.
template <int MODE>
__host__ __device__ constexpr bool step_is_doc(int m)
{
    return MODE == LDA_PROPOSALS_CYCLE ? (m & 1) != 0 : MODE == LDA_PROPOSALS_DOC;
}
template <int MODE>
__host__ __device__ constexpr int step_kind_index(int m)
{
    return MODE == LDA_PROPOSALS_CYCLE ? m >> 1 : m;
}

// The record the document side leaves per token, in the order it is made: the token's own (topic, n_kd) word, then per
// step a (topic, n_kd) word and, behind a doc step's, its acceptance uniform.  Words of a chain of m steps:
template <int MODE>
__host__ __device__ constexpr int step_record_words(int m)
{
    return 1 + m + (MODE == LDA_PROPOSALS_CYCLE ? m / 2 : MODE == LDA_PROPOSALS_DOC ? m : 0);
}

// Place of step m's (topic, n_kd) word in it.
template <int MODE>
__host__ __device__ constexpr int step_record_at(int m)
{
    return step_record_words<MODE>(m);
}

// Device error word bits (set by kernels, read by the host after a sweep).
enum : int {
    ERR_WORD_RANGE = 1,   // a word id outside [0,V) at load
    ERR_COUNT_ZERO = 2,   // a token's own topic has a zero count (tables inconsistent)
    ERR_ROW_OVERFLOW = 4, // a count row needed more entries than its capacity
    ERR_TOPIC_RANGE = 8,  // an assignment outside [0,K)
    ERR_ALIAS = 16,       // alias construction met an impossible state
    ERR_STAGE = 32,       // a bulk copy into shared memory did not complete within its wait limit
    NOTE_WIDE_COUNT = 64, // no error: an imported count of a tail word does not fit 16 bits (shard.cu)
};

constexpr uint32_t DK_EMPTY = 0xFFFFFFFFu;  // == DK_EMPTY_SLOT of the device helpers
constexpr int DK_SLOTS_PER_TOKEN_HOST = 4;   // == DK_SLOTS_PER_TOKEN of the device helpers
constexpr int SORT_TILE = 2048;      // tokens per segmented-sort tile (one CTA)
// Tiles of whole documents (one CTA each) of the document-side kernels: tokens per tile and
// threads per CTA, chosen per corpus from these shapes; longer documents are cut into chunks (LONG_CHUNK).
constexpr int DOC_TILE_SHAPES = 4;
constexpr int DOC_TILE_ROUNDS = 3;  // tokens per thread: every shape holds this many times its thread count
constexpr int DOC_TILE_THREADS[DOC_TILE_SHAPES] = {128, 256, 512, 1024};
constexpr int DOC_TILE_TOKENS[DOC_TILE_SHAPES] = {DOC_TILE_ROUNDS * 128, DOC_TILE_ROUNDS * 256, DOC_TILE_ROUNDS * 512,
                                                  DOC_TILE_ROUNDS * 1024};
constexpr int DOC_TILE_MAX = DOC_TILE_ROUNDS * 1024;
constexpr int DOC_TILE_SLOTS = 4;  // 32-bit words per token of a tile's counters, and of hashed tables at least
constexpr int DOC_TILE_SLOTS_MOST = 6;  // ... and at most (docside.cu: tile_slots())
// partial sums of the log-likelihood kernels: word part; document part (tiles + long documents)
constexpr int LL_WORD_PARTIALS = 1184;
constexpr int LL_DOC_PARTIALS = 148 * 16 + 592 + 1024;
constexpr int HIST_BINS = 32768;     // shared-memory histogram window (32-bit bins)
constexpr int WORD_ROWS_BITMAP_MAX_K = 16384;  // tail rows: topic bitmap up to this K, key sort above
constexpr int HIST16_BINS = 106496;  // window of a warm word's n_kw histogram (16-bit bins, 208 KB)
constexpr int HIST32_BINS = 53248;   // window of a hot word's n_kw histogram (32-bit bins, 208 KB)
constexpr int HIST_RUN_MAX = 262144;  // tokens per CTA (one run of a word) in the histogram path, at most
constexpr int ROW_TILE_WORDS = 512;   // words per tile of the tail words' row kernel
// n_k added up by the row kernels themselves (choose_nk_mode())
constexpr int NK_WITH_ROWS_MAX_K = 4096;
constexpr int NK_WITH_ROWS_MAX_CTAS = 16384;
constexpr int64_t NK_DIRECT_MAX_TOKENS = 1 << 24;
constexpr int HOT_TILE_MAX = 32768;  // accept pass: tokens of one hot word per CTA (the word's row is staged once per CTA), at most
constexpr int HOT_TILE_PROPOSE_MAX = 8192;  // propose pass: nothing is staged, shorter runs balance better
constexpr int COLD_TILE = 2048;      // MH kernel: tokens of a tile of tail words, at most
constexpr int COLD_WORDS = 512;      // MH kernel: words per tail tile
constexpr int COLD_DIRECT = 12288;   // MH kernel: 16-bit counters of a tail tile in shared memory
constexpr int HOT_STAGE_MAX_K = 16384;  // dense rows up to this many topics are staged in shared memory
// Beyond that K a dense row (4 K bytes) only pays for frequent words.  Words with more tokens than
// a tail tile holds but at most WARM_MAX_TF keep a sorted sparse row only ("warm" words): rebuilt by
// one CTA per word from a 16-bit histogram over the topics, and staged whole in shared memory by
// the accept pass (a row has at most as many entries as the word has tokens).
constexpr int WARM_MAX_TF = 12288;
// longest sparse alias row built by a warp (of either kernel), by a CTA of 256 and of 1024 threads; longer: a cluster
constexpr int ALIAS_WARP_MAX = 256, ALIAS_LONG_WARP_MAX = 512, ALIAS_MID_MAX = 2048, ALIAS_BIG_MAX = 10240;
constexpr int ALIAS_CLASSES = 4;
constexpr int ALIAS_CLASS_MAX[ALIAS_CLASSES] = {ALIAS_WARP_MAX, ALIAS_LONG_WARP_MAX, ALIAS_MID_MAX, ALIAS_BIG_MAX};
constexpr int ALIAS_ROW_CLUSTER = 8;         // CTAs of that cluster
constexpr int ALIAS_SCRATCH_PER_ITEM = 18;   // bytes of construction scratch per item

// Start times (nanoseconds of the device's global timer) a sweep's kernels leave for lda_stats.
enum : int {
    STAMP_DENSE = 0, STAMP_DENSE_END, STAMP_PROPOSE_HOT, STAMP_PROPOSE_COLD, STAMP_DOC_TILES, STAMP_DOC_LONG,
    STAMP_ACCEPT_HOT, STAMP_ACCEPT_WARM, STAMP_ACCEPT_COLD, STAMP_ROWS, STAMP_WARM_ROWS, STAMP_HIST,
    STAMP_NK_DENSE, STAMP_NK_SPARSE, STAMPS
};
constexpr int STAMP_RING = 32;  // sweeps queued before the host waits and reads their stamps

// What changes from sweep to sweep lives in device memory, so that a sweep is the same sequence of
// launches with the same arguments every time (and can be replayed as a CUDA graph).  One per context.
struct SweepState {
    unsigned long long moves[2];  // steps of the running lda_sweep() that moved a chain: word-, doc-proposals
    int32_t err;                  // device error word
    uint32_t sweep, next;         // Philox sweep counter of the running sweep; of the one after it
    uint32_t slot, next_slot;     // their rows of `stamps`
    uint32_t pad;
    unsigned long long stamps[STAMP_RING][STAMPS];
};
// The part of it the host reads after a batch of sweeps, in host memory the device writes to.
struct SweepReport {
    unsigned long long moves[2];
    unsigned long long end;  // time after the batch
    int32_t err, pad;
    unsigned long long stamps[STAMP_RING][STAMPS];
    // of the log-likelihood's last kernel (which writes `err` too)
    double ll_word, ll_doc;
    unsigned long long nnz_dk;
};

// A document longer than a tile: its tokens [first, first + len) and its table in View::dk_slots, from
// `slot` on -- K counters (dense) or 4 * len slots, probed as dk_insert in lda_device.cuh has it.
struct LongDoc {
    long long slot;
    int32_t first, len;
    int32_t dense, pad;
};
constexpr int LONG_CHUNK = 2048, LONG_THREADS = 256;
constexpr int LONG_MIN_CTAS = 5;
constexpr int LONG_AT_ONCE = 4;  // tokens of a thread whose reads are in flight together
constexpr int LONG_STAGE_MAX_K = 4096;  // counters of a long document staged in shared memory up to this K

// Everything a kernel needs, passed by value.
struct View {
    int32_t V, K, N, D;
    double alpha, beta, Vbeta, Kalpha;
    // for the first look at an acceptance (accept_tokens()): the priors in single precision, and how close its sides may come
    float alpha_f, beta_f, Vbeta_f, filter_eps;
    uint32_t tok_base;  // Philox token key of the corpus' first token (0 unless the corpus is a shard)
    int topic_bits;  // bits of K-1
    int block_shift; // log2 of the tokens per block of the block-major order
    int count_bits;  // low bits of a packed n_kd entry that hold the count
    // tokens in word-sorted order (position p)
    const uint32_t* tok_orig;  // index of the token in the caller's document order
    // block-major order (index m): the tokens sorted by (block of the document-order index,
    // word-sorted position).  Buffers in this order are reached from word order in runs of
    // consecutive positions and from document order within one L2-sized block at a time.
    const uint32_t* inv;        // [N] block-major index of the token at word-sorted position p
    const uint32_t* bm_of_tok;  // [N] block-major index of the token with document-order index i
    // per-sweep exchange buffers between the word-order and the document-order passes
    void* prop;        // [word steps][N] block-major: topics proposed by the word-proposals after the first
    uint32_t* ua_w;    // [word steps][N] word order: acceptance uniforms of the word-proposal steps
    uint32_t* dside;   // [N][side_stride] block-major: step_record_words(): own (topic << count_bits) | n_kd, per step the same,
                       // per doc step its acceptance uniform
    int32_t side_stride;  // words per token in dside, a multiple of 4
    // assignments (topic type: u16 or i32) after the last MH step or initialisation
    void* zw;   // word-sorted order: read by the n_kw / n_k rebuild
    void* zbm;  // block-major order, two entries per token: its topic, read (through bm_of_tok) by everything
                // that works per document, and beside it the first word-proposal of the running MH step
    // One word per token in document order: scratch (topics of long documents during the MH step,
    // staging of assignments on their way in and out, z in document order for export.cu).
    uint32_t* rec;
    const uint8_t* hot_word;  // [V] 1: the MH step treats the word as hot (more than COLD_TILE tokens)
    const int32_t* word_off;  // [V+1] token range of each word in word-sorted order
    const int32_t* doc_off;   // [D+1]
    // n_kw: every word has a sorted (topic, count) row of fixed capacity; hot words also a dense row
    const int32_t* row_start;  // [V+1] first slot of each word's row
    int32_t* wk_nnz;           // [V]
    uint32_t* wk_topic;        // [row_start[V]]
    uint32_t* wk_count;
    const int32_t* dense_slot;  // [V] index of the word's dense row or -1
    int32_t* dense_rows;        // [n_dense * dense_stride]
    int32_t dense_stride;       // K rounded up to a multiple of 4 (rows start 16-byte aligned)
    // word-proposal tables
    uint32_t* al_thr;  // split point of each sparse bin as a 32-bit fraction
    uint32_t* al_idx;  // alias item of each sparse bin
    uint2* al_pk;      // 16-bit topics only: bin as (split point, topic of the bin's item | topic of
                       // its alias item << 16), so a draw costs one read
    unsigned long long* sp_mass;  // [V] fixed-point mass of the word's sparse term
    uint32_t* dn_thr;  // [K]
    uint32_t* dn_idx;  // [K]
    uint2* dn_pk;      // [K] (split point, alias) of the dense table in one word pair
    unsigned long long* dense_mass;
    int32_t* nk;       // [K] column sums of n_kw: the counts frozen at sweep start
    int32_t* nk_next;  // [K] ... of the rebuild in progress; the host exchanges the two after a rebuild
    // n_kd of the documents longer than a tile (the others' tables only ever live in shared memory), built
    // by k_long_count: hashed ones first, then the ones with a counter per topic
    uint32_t* dk_slots;
    const LongDoc* long_docs;
    int* err;           // = &state->err
    SweepState* state;  // sweep counter, move counters, stamps
};

struct Ctx {
    int32_t V = 0, K = 0;
    double alpha = 0, beta = 0;
    int device = 0;
    int n_sm = 148;  // multiprocessors of the device
    cudaStream_t stream = nullptr;
    bool wide_topics = false;  // false: 16-bit topic storage, true: 32-bit
    int block_option = 0;  // option "block_log2", 0: chosen per corpus
    int block_shift = 22;  // log2 of the tokens per block of the block-major order
    int doc_tile = DOC_TILE_TOKENS[0], doc_threads = DOC_TILE_THREADS[0];  // shape of the document tiles
    bool doc_dense = false;  // their n_kd tables are a counter per topic
    int side_steps = 0;    // number of steps the exchange buffers are allocated for
    int side_mode = 0;     // ... and the proposal schedule they are laid out for
    int proposals = 0;     // LDA_PROPOSALS_*: which proposal each step of a chain draws
    int64_t shard_first_token = 0;        // lda_set_shard(): global index of this corpus' first token
    std::vector<int32_t> shard_global_tf;  // ... and the term frequencies over all shards (empty: this corpus alone)
    double dense_frac = 0.05;
    double dense_min_tf = 64;
    int alias_slices = 1;  // vocabulary slices whose word-proposal tables are alive one at a time
    bool loaded = false, inited = false, tables_valid = false;
    int64_t n_nonempty_docs = 0;
    uint64_t seed = 0;
    uint32_t sweep = 0;
    int64_t N = 0, D = 0;
    View v{};
    // host-side work lists (device copies below)
    int32_t n_word_tiles = 0, n_doc_tiles = 0, n_dense = 0, n_hot_runs = 0, n_long_docs = 0,
            n_hot_tiles = 0, n_hot_tiles_propose = 0, n_cold_tiles = 0;
    int32_t* word_tiles = nullptr;   // [n_word_tiles*2] word ranges sorted per CTA
    int32_t* doc_tiles = nullptr;    // [n_doc_tiles*2]
    int32_t* hot_runs = nullptr;     // [n_hot_runs*4] (word, first token, count, index of a word with several runs or -1)
    int32_t* acc = nullptr;          // [words with several runs][dense_stride], zero between rebuilds
    int32_t* acc_done = nullptr;     // [...] runs of the word that are done, zero between rebuilds
    int32_t* acc_runs = nullptr;     // [...] runs of the word
    bool cold_direct = false;        // the accept pass keeps the tail tiles' rows as 16-bit counters
    bool wide_counts = false;        // ... unless n_kw was imported with larger counts in tail words
    int nk_mode = 0;                 // how the row kernels add up n_k
    int32_t n_long_chunks = 0;
    int32_t* long_chunks = nullptr;  // [n_long_chunks*4] (index into View::long_docs, first token, count, 0)
    int64_t long_slots = 0, long_hashed_slots = 0;  // of View::dk_slots: in all, of the hashed tables
    // sorted n_kd rows (export.cu): tiles of whole documents of at most SORT_TILE tokens, and the longer documents
    int32_t n_doc_sort_tiles = 0, n_doc_sort_long = 0;
    int32_t* doc_sort_tiles = nullptr;
    int32_t* doc_sort_long = nullptr;
    // words whose row can exceed ALIAS_CLASS_MAX[i] (each list is part of the one before it)
    int32_t n_alias_words[ALIAS_CLASSES] = {};
    int32_t* present = nullptr;  // words that occur, ascending
    int32_t* alias_words[ALIAS_CLASSES] = {};
    int32_t n_warm = 0, n_hot_tiles_warm = 0;
    int32_t* warm_words = nullptr;      // [n_warm] words with a sorted row and more tokens than a tail tile holds
    int32_t* hot_tiles_warm = nullptr;  // [n_hot_tiles_warm*3] their runs for the accept pass
    int32_t* hot_tiles = nullptr;    // [n_hot_tiles*3] (word, first token, count): MH kernel, words with a dense row (accept pass)
    int32_t* hot_tiles_propose = nullptr;  // the same cut into the shorter runs of the propose passs
    int32_t* cold_tiles = nullptr;   // [n_cold_tiles*4] (first word, end word, first token, count): MH kernel, whole tail
                                     // words or a run of one
    // Vocabulary slices (Section 3, Fig. 1: the model is visited slice by slice): the words are cut into
    // runs of about equal row capacity; the sparse alias tables and their construction scratch hold one
    // slice at a time (entry of row slot r of the running slice: r - row_lo), so pass 1 goes slice by
    // slice: build the slice's tables, draw the word-proposals of its tokens.  One slice = everything.
    struct Slice {
        int32_t w_lo = 0, w_hi = 0;        // words [w_lo, w_hi)
        int64_t row_lo = 0, row_n = 0;     // their row slots [row_lo, row_lo + row_n)
        int32_t alias_lo[ALIAS_CLASSES] = {}, alias_n[ALIAS_CLASSES] = {};  // their part of the lists alias_words
        int32_t present_lo = 0, present_n = 0;  // ... of present
        int32_t hotp_lo = 0, hotp_n = 0;   // ... of hot_tiles_propose
        int32_t cold_lo = 0, cold_n = 0;   // ... of cold_tiles
    };
    std::vector<Slice> slices;
    int cur_slice = 0;
    uint32_t* al_thr0 = nullptr;  // the slice-sized buffers View::al_thr, al_idx, al_pk and sc_w, sc_de, sc_item
    uint32_t* al_idx0 = nullptr;  // point into, shifted by the running slice's row_lo
    uint2* al_pk0 = nullptr;
    unsigned long long* sc_w0 = nullptr;
    unsigned long long* sc_de0 = nullptr;
    uint32_t* sc_item0 = nullptr;
    // alias-construction scratch
    unsigned long long* sc_w = nullptr;   // [row capacity total] scaled masses
    unsigned long long* sc_de = nullptr;  // deficits prefix (front) / surpluses prefix (back)
    uint32_t* sc_item = nullptr;          // light items (front) / heavy items (back)
    unsigned long long* sc_dense = nullptr;  // same three for the dense table, [3*K]
    uint32_t* mix32 = nullptr;               // [V] mixture thresholds, for lda_get_tables()
    double* ll_tab = nullptr;        // [3 * 512] lgamma tables of the log-likelihood
    double* ll_tile_part = nullptr;  // [n_doc_tiles] its partial sums, one per tile of documents
    uint32_t* ll_tile_nnz = nullptr; // [n_doc_tiles] filled table slots of the tile: its share of nnz(n_kd)
    bool ll_tables_ready = false;
    double* red = nullptr;                   // reduction partials for the log-likelihood
    uint32_t* red_nnz = nullptr;             // [LL_DOC_PARTIALS] nnz(n_kd) beside the document part's partials
    int64_t* red_i = nullptr;
    // device memory comes from cudaMalloc / cudaFree unless lda_set_allocator() gave other routines
    lda_alloc_fn alloc_fn = nullptr;
    lda_free_fn free_fn = nullptr;
    void* alloc_user = nullptr;
    std::vector<void*> allocs;
    std::vector<size_t> alloc_bytes;  // size of every entry of `allocs`
    std::vector<char> alloc_own;      // 1: the entry came from the caller's allocator, 0: from cudaMalloc
    int64_t device_bytes = 0;
    lda_stats stats{};
    int64_t launches = 0;
    SweepReport* report = nullptr;  // host memory the device writes (one block of the process-wide pool)
    // A sweep as a CUDA graph, one per parity of the sweep counter (the two n_k buffers take turns).
    // Built once a configuration has run a few sweeps launch by launch; dropped whenever an argument of
    // its kernels changes.
    cudaGraphExec_t graph[2] = {};
    int graph_launches = 0;      // kernels in it
    int graph_steps = 0, graph_mode = 0;
    uint64_t graph_seed = 0;
    int plain_sweeps = 0;        // sweeps launched one kernel at a time since the last change
    bool graph_refused = false;  // capture failed once: this context launches kernel by kernel
    cudaStream_t capture = nullptr;
    // Two more streams for kernels of one phase that touch different words: fork_streams() makes them
    // wait for the work queued on `stream` so far, join_streams() makes `stream` wait for theirs.
    cudaStream_t side[2] = {};
    cudaEvent_t ev_fork = nullptr, ev_join[2] = {};
    // Assignments travel between host and device in chunks on a stream of their own, so that the copy
    // of one chunk runs beside the kernel that spreads (or collects) its neighbour.  ev_chunk orders a
    // chunk's two halves; ev_export completes when the last chunk of an export has reached the host:
    // whatever touches the staging buffer next waits for it on the device (order_after_export()).
    int64_t copy_chunk = 0;  // tokens per chunk (option "copy_chunk_log2"; 0: by the size of the corpus)
    cudaStream_t copy = nullptr;
    cudaEvent_t ev_chunk = nullptr, ev_export = nullptr;
    bool export_pending = false;
    std::string err;
};

// The running sweep's counter.  Read where it is used (a cache hit after a CTA's first read): kept in a
// register across a kernel it costs the register-bound passes a spill.  Constant while its readers run.
__device__ __forceinline__ uint32_t running_sweep(const View& v)
{
    uint32_t s;
    asm volatile("ld.global.ca.u32 %0, [%1];" : "=r"(s) : "l"(&v.state->sweep));
    return s;
}

__device__ __forceinline__ unsigned long long global_timer()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
    return t;
}

// First instruction of a kernel: one thread of the grid notes the time (`id` < 0: not noted).
__device__ __forceinline__ void stamp(SweepState* state, int id)
{
    if (id >= 0 && blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0)
        state->stamps[state->slot][id] = global_timer();
}
__device__ __forceinline__ void stamp(const View& v, int id) { stamp(v.state, id); }

inline void fork_streams(Ctx& c)
{
    cudaEventRecord(c.ev_fork, c.stream);
    for (int i = 0; i < 2; ++i) cudaStreamWaitEvent(c.side[i], c.ev_fork, 0);
}

inline void join_streams(Ctx& c)
{
    for (int i = 0; i < 2; ++i) {
        cudaEventRecord(c.ev_join[i], c.side[i]);
        cudaStreamWaitEvent(c.stream, c.ev_join[i], 0);
    }
}

// The kernels of one pass of the MH step touch different tokens and could always run side by side.  With
// few tokens none of them fills the GPU and the pass lasts as long as the slower one; with many
// (738 M tokens: accept pass 6.7 ms side by side, 6.1 one after the other) they only compete for L2.
constexpr int64_t SIDE_BY_SIDE_MAX_TOKENS = (int64_t)1 << 24;
struct PassStreams {
    Ctx& c;
    bool side;
    PassStreams(Ctx& ctx, int kernels) : c(ctx), side(kernels > 1 && ctx.N <= SIDE_BY_SIDE_MAX_TOKENS)
    {
        if (side) fork_streams(c);
    }
    ~PassStreams()
    {
        if (side) join_streams(c);
    }
    cudaStream_t operator[](int i) const { return side && i > 0 ? c.side[i - 1] : c.stream; }
};

// --- launchers (each returns the number of kernels it launched) -----------------
int launch_init(Ctx& c);
void launch_set_state(Ctx& c);   // the device's copy of the sweep counter := the host's; move counters and stamps cleared
void launch_report(Ctx& c);      // state -> c.report, move counters and stamps cleared
int launch_spread_assignments(Ctx& c, const void* z_dev, bool narrow);  // z (doc order; u16 if narrow, else i32) -> both layouts
int launch_spread_chunk(Ctx& c, const void* z_dev, bool narrow, int64_t first, int64_t count);  // ... tokens [first, first+count) -> block-major
int launch_word_order_topics(Ctx& c);                                  // block-major -> word order, all tokens
int launch_export_assignments(Ctx& c, void* z_dev, bool narrow);
int launch_export_chunk(Ctx& c, void* z_dev, bool narrow, int64_t first, int64_t count);
int launch_count_wk(Ctx& c);
int launch_count_k(Ctx& c);      // n_k of the rows just rebuilt, added to View::nk_next (cleared before), unless the
                                 // row kernels have done it
int launch_count_k_from_rows(Ctx& c);  // ... in any case
void rebuild_counts(Ctx& c);     // n_kw and n_k from the assignments, outside a sweep
void set_wide_counts(Ctx& c, bool wide);
void choose_nk_mode(Ctx& c);     // after the work lists are made
inline void exchange_nk(Ctx& c) { int32_t* t = c.v.nk; c.v.nk = c.v.nk_next; c.v.nk_next = t; }
int launch_begin_sweep(Ctx& c);  // first kernel of a sweep that needs no tables
int launch_alias_dense(Ctx& c, bool in_sweep);  // in_sweep: as the first kernel of a sweep, see there
void launch_mix_thresholds(Ctx& c, uint32_t* mix32);  // of the tables last built
int launch_alias_sparse(Ctx& c, bool all, bool begin_sweep = false);  // the running slice's tables (all: in every form, for lda_get_tables)
void set_slice(Ctx& c, int slice);          // makes `slice` the running one (moves the table pointers)
int launch_sample(Ctx& c, int mh_steps);   // all passes of the MH step; needs ensure_exchange()
int launch_doc_side(Ctx& c, int mh_steps);  // pass 2 of the MH step
int launch_long_tables(Ctx& c, cudaStream_t stream, bool keep_topics, int stamp_id);  // n_kd tables of the documents longer than a tile
size_t doc_tile_smem_bytes(int tile_tokens, int slots);  // dynamic shared memory of the document-tile kernels, `slots` a token
int ensure_exchange(Ctx& c, int mh_steps);  // (re)allocates View::prop / View::dside; LDA_* status
int launch_loglik(Ctx& c, double* out3_host);
int launch_count_nnz(Ctx& c, int64_t* nnz_wk_host, int64_t* nnz_dk_host);

// n_kd as sorted rows in device memory (export.cu): row_off[D+1], and unless sizes_only the entries.
// The caller releases the arrays with free_dk_csr().
struct DkCsr {
    long long* row_off = nullptr;
    int32_t* nnz = nullptr;
    int32_t* topic = nullptr;
    int32_t* count = nullptr;
    long long total = 0;
};
int build_dk_csr(Ctx& c, DkCsr& r, bool sizes_only);  // LDA_* status; queued on c.stream, rows complete after a sync
void free_dk_csr(Ctx& c, DkCsr& r);

// n_kw as a dense V x K matrix in device memory and back (shard.cu): the exchange format of the
// document-sharded mode.  Return the number of kernels launched.
int launch_word_counts_to_dense(Ctx& c, int32_t* nwk_dev);
int launch_word_counts_from_dense(Ctx& c, const int32_t* nwk_dev);

// Exact-conditional yardstick (gibbs.cu): `iters` frozen sweeps drawing from Eq. 1.  LDA_* status.
constexpr int GIBBS_MAX_K = 16384;              // a word's dense n_kw row is staged in shared memory
constexpr long long GIBBS_MAX_PREFIX_BYTES = 24ll << 30;  // V * K running sums of 8 bytes
int gibbs_sweep(Ctx& c, int32_t iters);
void set_gibbs_smem_limits();

// Blocking copies that are fast for host memory that is not page-locked, too (staging.cu); after everything
// queued on the context's stream.
cudaError_t copy_to_host(Ctx& c, void* host, const void* dev, size_t bytes);
cudaError_t copy_to_device(Ctx& c, void* dev, const void* host, size_t bytes);
bool page_locked(const void* host);
// Address that kernels may write [host, host + bytes) by, or null: it has to lie in one allocation or registration of page-locked
// memory that is not read-only.
void* device_view(const void* host, size_t bytes);

// n_kw as compact rows in device memory: row offsets [V+1] and the entries (export.cu).  LDA_* status.
struct WkCsr {
    long long* row_off = nullptr;
    int32_t* topic = nullptr;
    int32_t* count = nullptr;
    long long total = 0;
};
int build_wk_csr(Ctx& c, WkCsr& r, bool sizes_only);
void free_wk_csr(Ctx& c, WkCsr& r);

// load-time layout (sort + offsets), queued; fills c.v token arrays and records ev_chunk when word_off is there.
// The transient buffers are the caller's to release once the stream is done with them.  LDA_* status.
struct LayoutTemps {
    std::vector<void*> held;
};
void launch_dense_slots(Ctx& c, const int32_t* dense_words);  // slot i to dense_words[i], i < n_dense
int build_layout(Ctx& c, const int32_t* word_ids_dev, const std::vector<int32_t>& doc_off, LayoutTemps& temps);

void* raw_alloc(Ctx& c, size_t bytes);  // the context's allocator (cudaMalloc by default); nullptr on failure
void raw_free(Ctx& c, void* p);
template <typename P>
inline bool tmp_alloc(Ctx& c, P** p, size_t bytes)  // transient buffer, released with raw_free()
{
    *p = static_cast<P*>(raw_alloc(c, bytes ? bytes : 1));
    return *p != nullptr;
}
void* dev_alloc(Ctx& c, size_t bytes);  // tracked allocation held by the context; nullptr on failure
void dev_free(Ctx& c, void* p);         // releases one tracked allocation (nullptr: nothing)
void dev_free_all(Ctx& c);

}  // namespace lda
