"""Branches of the sweep that depend on sizes: the oracle's assignments, counts and tables on both sides of
each of them."""
import numpy as np
import pytest

from oracle import ldaref
from paper_1412_1576_b200 import binding, synth

pytestmark = pytest.mark.gpu


def _pair(c, seed=77):
    w, off = c.word_ids.numpy(), c.doc_offsets.numpy()
    g = binding.LightLDA(c.V, c.K, c.alpha, c.beta)
    o = ldaref.Oracle(c.V, c.K, c.alpha, c.beta)
    for e in (g, o):
        e.load_corpus(w, off)
        e.init(seed)
    return g, o


def _same(g, o):
    assert np.array_equal(g.get_assignments(), o.get_assignments())
    assert np.array_equal(g.get_nk(), o.get_nk())
    for which in (binding.LDA_NWK, binding.LDA_NDK):
        for a, b in zip(g.get_csr(which), o.get_csr(which)):
            assert np.array_equal(a, b)
    a, b = g.get_tables(), o.get_tables()
    for k in a:
        assert np.array_equal(a[k], b[k]), k


@pytest.mark.parametrize("K", [1, 63, 65, 2048, 2049, 8193, 100_003])
def test_dense_table_by_one_cta_and_by_a_cluster(K):
    c = synth.generate(V=300, K=K, D=150, length=("poisson", 40.0), zipf_s=1.1, alpha=0.05, beta=0.01, seed=5)
    g, o = _pair(c)
    _same(g, o)
    g.sweep(4, 2)  # the last ones replayed as a graph
    o.sweep(4, 2)
    _same(g, o)


def test_replayed_sweeps_follow_changes_of_their_arguments(tiny_corpus):
    """Step count, schedule, seed and state change between sweeps that are otherwise replayed."""
    g, o = _pair(tiny_corpus)
    z = None
    for iters, steps, mode, seed in ((5, 2, 0, None), (1, 2, 0, None), (4, 4, 0, None), (4, 2, 1, None), (35, 2, 0, None),
                                     (4, 2, 0, 123), (3, 2, 2, 124)):
        if seed is not None:
            z = o.get_assignments()
            g.set_assignments(z, seed, 9)
            o.set_assignments(z, seed, 9)
        g.set_proposals(mode)
        o.set_proposals(mode)
        g.sweep(iters, steps)
        o.sweep(iters, steps)
        assert np.array_equal(g.get_assignments(), o.get_assignments()), (iters, steps, mode, seed)
    _same(g, o)


@pytest.mark.parametrize("K,V", [(10_500, 3), (2_500, 40), (600, 400), (40, 3_000)])
def test_rows_of_every_length(K, V):
    """Count rows and runs of words from one token to a few thousand, lengths around powers of two among them (the alias
    rows' classes go by topics: test_alias_rows_at_the_borders_of_their_classes)."""
    rng = np.random.default_rng(K)
    edges = [1, 2, 7, 8, 9, 15, 16, 17, 31, 32, 33, 63, 64, 65, 96, 97, 127, 128, 129, 255, 256, 257, 511, 512, 513, 1023, 2047,
             2048, 2049, 4095, 6000]
    tf = np.array([edges[i % len(edges)] if V > 3 else [11_500, 10_241, 2_100][i] for i in range(V)])
    while tf.sum() > 150_000:
        tf[rng.integers(V)] = 3
    words = rng.permutation(np.repeat(np.arange(V), tf)).astype(np.int32)
    cuts = np.sort(rng.integers(0, words.size + 1, words.size // 60))
    offsets = np.concatenate([[0], cuts, [words.size]]).astype(np.int64)
    g = binding.LightLDA(V, K, 0.05, 0.01)
    o = ldaref.Oracle(V, K, 0.05, 0.01)
    for e in (g, o):
        e.load_corpus(words, offsets)
        e.init(3)
    _same(g, o)
    g.sweep(3, 2)
    o.sweep(3, 2)
    _same(g, o)


EDGES = [1, 2, 8, 9, 16, 17, 32, 33, 255, 256, 257, 511, 512, 513, 2_047, 2_048, 2_049]


@pytest.mark.parametrize("K,rows", [(10_500, EDGES + [10_239, 10_240, 10_241, 10_500]), (20_000, EDGES + [10_240, 10_241, 15_000]),
                                    (2_100, EDGES * 45)])
def test_alias_rows_at_the_borders_of_their_classes(K, rows):
    """Rows with exactly as many topics as the borders between the kernels that build them, by assignments made for it;
    and more rows that may be long (765 words, 315 of them above 256 topics) than CTAs are given to at once."""
    rng = np.random.default_rng(K)
    many = len(rows) > 100
    words, z = [], []
    for w, n in enumerate(rows):
        topics = rng.permutation(K)[:n]
        more = rng.choice(topics, max(3, 300 - n if many else 0))     # a word's tokens bound its row
        words.append(np.full(n + more.size, w))
        z.append(np.concatenate([topics, more]))
    mixed = rng.permutation(sum(x.size for x in z))
    words, z = np.concatenate(words)[mixed].astype(np.int32), np.concatenate(z)[mixed].astype(np.int32)
    offsets = np.concatenate([[0], np.sort(rng.integers(0, z.size + 1, z.size // 60)), [z.size]]).astype(np.int64)
    g, o = binding.LightLDA(len(rows), K, 0.05, 0.01), ldaref.Oracle(len(rows), K, 0.05, 0.01)
    for e in (g, o):
        e.load_corpus(words, offsets)
        e.set_assignments(z, 17, 0)
    assert np.array_equal(np.diff(g.get_csr(binding.LDA_NWK)[0]), rows)
    _same(g, o)
    for e in (g, o):
        e.sweep(3, 2)
    _same(g, o)


@pytest.mark.parametrize("K", [37, 3_000, 4_096, 4_097, 20_000])
@pytest.mark.parametrize("mode", [0, 2])
def test_long_documents_by_chunks(K, mode):
    """Documents around the tile sizes and the chunk size, long ones with a counter per topic (staged or not) and
    hashed ones, beside short ones."""
    lengths = np.array([1, 383, 384, 385, 768, 769, 1537, 2047, 2048, 2049, 4097, 0, 9_001, 30, 30, 0, 3_073, 5_200])
    rng = np.random.default_rng(K + mode)
    words = rng.integers(0, 700, lengths.sum()).astype(np.int32)
    offsets = np.concatenate([[0], np.cumsum(lengths)]).astype(np.int64)
    g = binding.LightLDA(700, K, 0.05, 0.01)
    o = ldaref.Oracle(700, K, 0.05, 0.01)
    for e in (g, o):
        e.load_corpus(words, offsets)
        e.init(11)
        e.set_proposals(mode)
        e.sweep(4, 2)
    _same(g, o)
    for a, b in zip(g.loglik(), o.loglik()):
        assert a == pytest.approx(b, rel=1e-10)
    assert g.stats()["nnz_dk"] == g.get_csr(binding.LDA_NDK)[1].size


@pytest.mark.parametrize("K,length", [(191, 24), (193, 24), (767, 96), (769, 96), (1023, 330), (3_071, 384), (3_073, 384), (3_100, 500)])
def test_document_tiles_with_counters_and_with_hashed_tables(K, length):
    """Topic counts on both sides of what a tile's counters hold, odd ones among them."""
    c = synth.generate(V=900, K=K, D=70, length=("poisson", float(length)), zipf_s=1.05, alpha=0.3, beta=0.01, seed=K)
    g, o = _pair(c)
    for steps, mode in ((2, 0), (3, 0), (2, 2), (4, 0)):
        for e in (g, o):
            e.set_proposals(mode)
            e.sweep(2, steps)
        assert np.array_equal(g.get_assignments(), o.get_assignments()), (steps, mode)
    _same(g, o)


@pytest.mark.parametrize("K,slices", [(40, 1), (40, 5), (3_000, 1), (9_000, 4)])
def test_vocabularies_mostly_empty(K, slices):
    """Words far apart, gaps wider than any tile, none at the first and last ids; a frequent one among them; gaps in which
    a slice begins.  20 500 documents, so that their lists are made on another thread."""
    V = 60_000
    rng = np.random.default_rng(K)
    used = np.unique(np.concatenate([rng.integers(5, V - 5, 900), np.arange(30_000, 30_300), [29_000]]))
    words = rng.permutation(np.concatenate([rng.choice(used, 41_000), np.full(2_500, 29_000)])).astype(np.int32)
    offsets = np.concatenate([[0], np.sort(rng.integers(0, words.size + 1, 20_500)), [words.size]]).astype(np.int64)
    g = binding.LightLDA(V, K, 0.05, 0.01)
    binding.lda_set_option(g._h, "alias_slices", slices)
    o = ldaref.Oracle(V, K, 0.05, 0.01)
    for e in (g, o):
        e.load_corpus(words, offsets)
        e.init(4)
        e.sweep(2, 2)
    for a, b in zip(g.loglik(), o.loglik()):
        assert a == pytest.approx(b, rel=1e-10)
    if slices == 1:
        _same(g, o)
    else:
        assert np.array_equal(g.get_assignments(), o.get_assignments())


@pytest.mark.parametrize("K,short", [(1, 0), (9, 0), (64, 0), (65, 0), (500, 0), (500, 40)])
def test_exact_conditional_rows_of_every_length(K, short):
    """Document rows of one topic to hundreds: parts of a row that are kept in registers and parts that are not, turns
    of one token and of 32; long rows and, with many short documents, rows that are short on average."""
    lengths = np.array([1, 2, 3, 7, 8, 9, 31, 32, 33, 63, 64, 65, 66, 127, 0, 200, 700, 1_500, 5] + [1] * short)
    rng = np.random.default_rng(K)
    words = rng.integers(0, 80, lengths.sum()).astype(np.int32)
    offsets = np.concatenate([[0], np.cumsum(lengths)]).astype(np.int64)
    g = binding.LightLDA(80, K, 0.07, 0.013)
    o = ldaref.Oracle(80, K, 0.07, 0.013)
    for e in (g, o):
        e.load_corpus(words, offsets)
        e.init(6)
    for _ in range(3):
        g.gibbs_sweep(1)
        o.gibbs_sweep(1)
        assert np.array_equal(g.get_assignments(), o.get_assignments())


@pytest.mark.parametrize("alpha,beta", [(0.05, 1e-9), (1e-9, 0.01), (2.0, 2.0 ** -24), (2.0 ** -25, 3.0), (1e9, 1e9), (0.05, 1e6)])
@pytest.mark.parametrize("steps,mode", [(2, 0), (3, 0), (4, 0), (2, 1), (2, 2)])
def test_acceptances_under_extreme_priors(alpha, beta, steps, mode):
    """Priors on both sides of those that leave every acceptance to double precision, and such as let single-precision
    products overflow."""
    c = synth.generate(V=300, K=40, D=150, length=("poisson", 60.0), zipf_s=1.1, alpha=0.05, beta=0.01, seed=8)
    w, off = c.word_ids.numpy(), c.doc_offsets.numpy()
    g, o = binding.LightLDA(c.V, c.K, alpha, beta), ldaref.Oracle(c.V, c.K, alpha, beta)
    for e in (g, o):
        e.load_corpus(w, off)
        e.init(21)
        e.set_proposals(mode)
        e.sweep(4, steps)
    assert np.array_equal(g.get_assignments(), o.get_assignments())


@pytest.mark.parametrize("K", [16_384, 16_385, 53_248, 53_249, 106_496, 106_497])
@pytest.mark.parametrize("steps,mode", [(2, 0), (3, 0), (4, 0), (2, 1)])
def test_long_words_at_large_topic_counts(K, steps, mode):
    """Words around the lengths at which a word's rows change their form, and one with more tokens of a topic than 16 bits
    count, at topic counts around the limits of what shared memory holds of a word, once or twice over."""
    tf = [66_500, 12_289, 12_288, 2_049, 2_048, 2_047, 300, 1]
    rng = np.random.default_rng(K)
    words = np.repeat(np.arange(len(tf)), tf)
    z = rng.integers(0, K, words.size)
    z[:66_000] = K - 1                  # of the first word: 65 535 and more
    z[66_500:68_000] = 0
    mixed = rng.permutation(words.size)
    words, z = words[mixed].astype(np.int32), z[mixed].astype(np.int32)
    offsets = np.concatenate([[0], np.sort(rng.integers(0, z.size + 1, z.size // 80)), [z.size]]).astype(np.int64)
    g, o = binding.LightLDA(len(tf), K, 0.01, 0.01), ldaref.Oracle(len(tf), K, 0.01, 0.01)
    for e in (g, o):
        e.load_corpus(words, offsets)
        e.set_proposals(mode)
        e.set_assignments(z, 5, 0)
        e.sweep(2, steps)
    assert np.array_equal(g.get_assignments(), o.get_assignments())
    assert np.array_equal(g.get_nk(), o.get_nk())


@pytest.mark.parametrize("K", [53_248, 53_249, 106_497])
@pytest.mark.parametrize("rest", [1, 300, 65_535, 65_536])
def test_words_of_several_runs_at_large_topic_counts(K, rest):
    """A word that is counted in two runs, of 262 144 tokens and of `rest`: below 65 536 the second counts in 16 bits where K asks
    for it, in windows of twice the width, and both add to one line.  Two rebuilds, so that the line is cleared between."""
    n = 262_144 + rest
    rng = np.random.default_rng(rest)
    words = np.zeros(n + 500, np.int32)
    words[n:] = rng.integers(1, 4, 500)
    z = rng.integers(0, K, words.size).astype(np.int32)
    z[:70_000], z[n - rest:n] = K - 1, rng.choice([0, 53_247, K - 1], rest)
    offsets = np.concatenate([[0], np.sort(rng.integers(0, z.size + 1, z.size // 80)), [z.size]]).astype(np.int64)
    g, o = binding.LightLDA(4, K, 0.01, 0.01), ldaref.Oracle(4, K, 0.01, 0.01)
    for e in (g, o):
        e.load_corpus(words, offsets)
        e.set_assignments(z, 5, 0)
    for again in range(2):
        assert np.array_equal(g.get_nk(), o.get_nk()), again
        for a, b in zip(g.get_csr(binding.LDA_NWK), o.get_csr(binding.LDA_NWK)):
            assert np.array_equal(a, b), again
        for e in (g, o):
            e.sweep(1, 2)
        assert np.array_equal(g.get_assignments(), o.get_assignments()), again


@pytest.mark.parametrize("tokens", [1 << 21, (1 << 21) + 1])
def test_corpora_around_two_million_tokens(tokens):
    """As many tokens as let the tail words' kernel have six CTAs per multiprocessor, and loops over steps six slots per token, and
    one more."""
    rng = np.random.default_rng(tokens)
    words = (2_500 * rng.random(tokens) ** 2).astype(np.int32)
    offsets = np.concatenate([[0], np.sort(rng.integers(0, tokens + 1, tokens // 50)), [tokens]]).astype(np.int64)
    g, o = binding.LightLDA(2_500, 2_000, 0.05, 0.01), ldaref.Oracle(2_500, 2_000, 0.05, 0.01)
    for e in (g, o):
        e.load_corpus(words, offsets)
        e.init(9)
    for steps, mode in ((2, 0), (3, 0), (3, 1), (1, 2)):
        for e in (g, o):
            e.set_proposals(mode)
            e.sweep(1, steps)
        assert np.array_equal(g.get_assignments(), o.get_assignments()), (steps, mode)


@pytest.mark.parametrize("tokens", [1, 7, 8, 9, 15, 16, 17, 255, 256, 257, 1_023, 1_024, 1_025, 2_047, 2_048])
def test_sorted_rows_of_tiles_of_every_length(tokens):
    """Rows of words and of documents at a topic count too large for a bitmap: one word and one document of just so many
    tokens, then 30 words of about a hundredth as many."""
    K = 20_000
    rng = np.random.default_rng(tokens)
    words = np.concatenate([np.zeros(tokens, np.int32), rng.integers(1, 31, max(tokens // 4, 1)).astype(np.int32)])
    z = np.where(rng.random(words.size) < 0.5, rng.integers(0, 9, words.size), rng.integers(0, K, words.size)).astype(np.int32)
    offsets = np.array([0, tokens, tokens, words.size], np.int64)
    g, o = binding.LightLDA(40, K, 0.05, 0.01), ldaref.Oracle(40, K, 0.05, 0.01)
    for e in (g, o):
        e.load_corpus(words, offsets)
        e.set_assignments(z, 3, 0)
    _same(g, o)
    for e in (g, o):
        e.sweep(2, 2)
    _same(g, o)


@pytest.mark.parametrize("docs,V,K", [(1, 3, 1), (7, 40_000, 50), (1_024, 300, 40), (1_025, 300, 40), (40, 2, 9_000), (40, 50, 70_000)])
def test_log_likelihood_by_one_kernel_and_by_several(docs, V, K):
    """As many tiles of documents as one kernel takes and one more; rows longer than a warp's, large vocabularies.  Sums of
    at most 4 10^5 terms: 1e-10 covers their order."""
    rng = np.random.default_rng(docs)
    words = rng.integers(0, V, docs * 384).astype(np.int32)
    offsets = (np.arange(docs + 1) * 384).astype(np.int64)
    g, o = binding.LightLDA(V, K, 0.05, 0.01), ldaref.Oracle(V, K, 0.05, 0.01)
    for e in (g, o):
        e.load_corpus(words, offsets)
        e.init(2)
    first = g.loglik()
    for a, b in zip(first, o.loglik()):
        assert a == pytest.approx(b, rel=1e-10)
    assert g.loglik() == first      # and again
    for e in (g, o):
        e.sweep(1, 2)
    for a, b in zip(g.loglik(), o.loglik()):
        assert a == pytest.approx(b, rel=1e-10)
