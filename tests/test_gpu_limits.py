"""Calls at the limits of what the library accepts: priors that leave a table without mass."""
import numpy as np
import pytest

from oracle import ldaref
from paper_1412_1576_b200 import binding, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K", [16, 2_048, 2_049])
def test_dense_table_without_mass(K):
    """beta / (n_k + V beta) below 2^-44 for every topic, on one CTA and on a cluster: an error, and the context can be
    used again; so can others."""
    import torch
    c = synth.generate(V=40, K=K, D=60, length=("fixed", 1_000), zipf_s=None, alpha=0.1, beta=0.01, seed=K)
    w, off = c.word_ids.numpy(), c.doc_offsets.numpy()
    g = binding.LightLDA(c.V, c.K, c.alpha, 1e-300)
    g.load_corpus(w, off)
    for _ in range(2):
        g.init(3)
        assert g.get_nk().min() > 0          # else that topic would have a mass
        with pytest.raises(binding.LdaError) as e:
            g.sweep(3, 2)
        assert e.value.status == binding.LDA_EINTERNAL
        with pytest.raises(binding.LdaError) as e:
            g.sweep(1, 2)
        assert e.value.status == binding.LDA_ESTATE
    g.init(3)
    nk = torch.from_numpy(g.get_nk()).cuda()
    thr, al = torch.zeros(K, dtype=torch.int32, device="cuda"), torch.zeros(K, dtype=torch.int32, device="cuda")
    mass, status = torch.ones(1, dtype=torch.int64, device="cuda"), torch.zeros(1, dtype=torch.int32, device="cuda")
    torch.cuda.synchronize()
    assert binding.lda_dense_table_noalloc(nk.data_ptr(), K, c.V, 1e-300, thr.data_ptr(), al.data_ptr(), mass.data_ptr(),
                                           status.data_ptr()) == binding.LDA_OK
    torch.cuda.synchronize()
    assert int(status) != 0 and int(mass) == 0
    h, o = binding.LightLDA(c.V, c.K, c.alpha, 0.01), ldaref.Oracle(c.V, c.K, c.alpha, 0.01)
    for e in (h, o):
        e.load_corpus(w, off)
        e.init(3)
        e.sweep(2, 2)
    assert np.array_equal(h.get_assignments(), o.get_assignments())


def _loaded(c, stream):
    g = binding.LightLDA(c.V, c.K, c.alpha, c.beta, stream=stream)
    g.load_corpus(c.word_ids.numpy(), c.doc_offsets.numpy())
    g.init(5)
    g.sweep(1, 2)
    return g


def test_host_corpora_on_streams_of_their_own(small_corpus, tiny_corpus):
    """Loading on a stream that no other is ordered with: corpora small enough for one copy, and larger ones by several
    threads at once, of which one has the page-locked buffers."""
    import threading

    import torch
    want = {}
    for c in (tiny_corpus, small_corpus):
        o = ldaref.Oracle(c.V, c.K, c.alpha, c.beta)
        o.load_corpus(c.word_ids.numpy(), c.doc_offsets.numpy())
        o.init(5)
        o.sweep(1, 2)
        want[id(c)] = o.get_assignments()
    torch.cuda.synchronize()
    for _ in range(10):
        g = _loaded(tiny_corpus, torch.cuda.Stream().cuda_stream)
        assert np.array_equal(g.get_assignments(), want[id(tiny_corpus)])
    got, streams = [None] * 4, [torch.cuda.Stream() for _ in range(4)]

    def load(i):
        torch.cuda.set_device(0)
        got[i] = [_loaded(small_corpus, streams[i].cuda_stream).get_assignments() for _ in range(3)]
    threads = [threading.Thread(target=load, args=(i,)) for i in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for z in [z for zs in got for z in zs]:
        assert np.array_equal(z, want[id(small_corpus)])


@pytest.mark.parametrize("n_docs", [2_000, 400_000])
def test_device_offsets_still_on_their_way(n_docs):
    """Offsets that the default stream is about to write, read by a context on a stream that is not ordered with it."""
    import torch
    words = torch.randint(0, 50, (2 * n_docs,), dtype=torch.int32, device="cuda")
    offsets = torch.zeros(n_docs + 1, dtype=torch.int64, device="cuda")
    ready = torch.arange(0, 2 * n_docs + 1, 2, dtype=torch.int64, device="cuda")
    g = binding.LightLDA(50, 20, 0.1, 0.01, stream=torch.cuda.Stream().cuda_stream)
    torch.cuda.synchronize()
    torch.cuda._sleep(100_000_000)   # some 50 ms
    offsets.copy_(ready)
    assert binding.lda_load_corpus_device(g._h, words.data_ptr(), 2 * n_docs, offsets.data_ptr(), n_docs) == binding.LDA_OK
    g.N, g.D = 2 * n_docs, n_docs
    g.init(1)
    assert int(g.get_nk().sum()) == 2 * n_docs


def test_imported_counts_beyond_16_bits():
    """Counts of tail words that lda_word_counts_from_dense brings in may be larger than any corpus's: tiles whose rows are
    otherwise 16-bit counters, sweeps on both sides of the import, replayed ones among them."""
    import torch
    c = synth.generate(V=50, K=100, D=60, length=("fixed", 25), zipf_s=None, alpha=0.1, beta=0.01, seed=2)
    g, o = binding.LightLDA(c.V, c.K, c.alpha, c.beta), ldaref.Oracle(c.V, c.K, c.alpha, c.beta)
    for e in (g, o):
        e.load_corpus(c.word_ids.numpy(), c.doc_offsets.numpy())
        e.init(9)
    m, m_host = torch.zeros(c.V * c.K, dtype=torch.int32, device="cuda"), np.zeros(c.V * c.K, np.int32)
    for times in (1, 70_001, 1, 65_535, 70_001):
        for e in (g, o):
            e.sweep(4, 2)
        g.word_counts_to_dense(m)
        o.word_counts_to_dense(m_host)
        assert np.array_equal(m.cpu().numpy(), m_host)
        m *= times
        m_host *= times
        torch.cuda.synchronize()
        g.word_counts_from_dense(m)
        o.word_counts_from_dense(m_host)
        assert np.array_equal(g.get_nk(), o.get_nk())
        for iters in (1, 3):
            for e in (g, o):
                e.sweep(iters, 2)
            assert np.array_equal(g.get_assignments(), o.get_assignments()), (times, iters)


@pytest.mark.parametrize("K,n", [(16, 1), (16, 131_072), (16, 131_073), (70_000, 65_536), (70_000, 65_537)])
@pytest.mark.parametrize("place", ["pinned", "pinned, behind others", "pageable", "pinned, odd address"])
def test_snapshots_into_any_host_memory(K, n, place):
    """As many tokens as the kernel writes to page-locked memory itself, and one more; nothing beside them is touched."""
    import torch
    words = (np.arange(n) % 7).astype(np.int32)
    g, o = binding.LightLDA(7, K, 0.1, 0.01), ldaref.Oracle(7, K, 0.1, 0.01)
    offsets = np.minimum(np.arange(n // 64 + 2) * 64, n).astype(np.int64)
    for e in (g, o):
        e.load_corpus(words, offsets)
        e.init(3)
    size = 2 if K <= 65_536 else 4
    first = {"pinned": 0, "pageable": 0, "pinned, behind others": 6 * size, "pinned, odd address": 6 * size + 1}[place]
    held = torch.full((first + n * size + 32,), 0x5A, dtype=torch.uint8, pin_memory=place != "pageable")
    export = binding.lda_get_assignments_u16_async_ptr if size == 2 else binding.lda_get_assignments_async_ptr
    assert export(g._h, held.data_ptr() + first) == binding.LDA_OK
    g.wait()
    raw = held.numpy()
    z = np.frombuffer(raw[first:first + n * size].tobytes(), np.uint16 if size == 2 else np.int32)
    assert np.array_equal(z, o.get_assignments())
    assert (raw[:first] == 0x5A).all() and (raw[first + n * size:] == 0x5A).all()


def test_which_host_memory_kernels_write():
    """The look at a snapshot's destination alone, nothing is launched: only what lies in one page-locked piece."""
    import ctypes
    import mmap

    import torch
    torch.cuda.init()
    view = binding.load_library()._ZN3lda11device_viewEPKvm
    view.restype, view.argtypes = ctypes.c_void_p, [ctypes.c_void_p, ctypes.c_size_t]
    page, rt = mmap.PAGESIZE, torch.cuda.cudart()
    held = mmap.mmap(-1, 12 * page)
    p = ctypes.addressof(ctypes.c_char.from_buffer(held))
    pieces = [(p, page), (p + 3 * page, page), (p + 4 * page, page), (p + 6 * page + 100, 5_000)]
    for at, size in pieces:
        assert int(rt.cudaHostRegister(at, size, 0)) == 0
    read_only = p + 10 * page
    refused = int(rt.cudaHostRegister(read_only, page, 8))  # cudaHostRegisterReadOnly
    try:
        for at, size in pieces:
            assert view(at, size) == at and view(at + 64, size - 64) == at + 64 and view(at + size - 1, 1) == at + size - 1
            assert view(at, size + 1) is None and view(at + 64, size - 63) is None and view(at + size - 1, 2) is None
        assert view(p, 4 * page) is None               # first and last page, two between them are not page-locked
        assert view(p + 3 * page, 2 * page) is None    # two pieces side by side: the copy decides
        assert view(p + 2 * page, 4) is None and view(p + 2 * page, 2 * page) is None
        assert view(read_only, 4) is None
        pinned, on_device = torch.empty(1_000, dtype=torch.int16, pin_memory=True), torch.empty(10, device="cuda")
        assert view(pinned.data_ptr(), 2_000) == pinned.data_ptr()
        assert view(on_device.data_ptr(), 4) is None
    finally:
        for at, _ in pieces + ([(read_only, 0)] if refused == 0 else []):
            assert int(rt.cudaHostUnregister(at)) == 0


@pytest.mark.parametrize("offsets", [[0, 2, 1, 4], [0, -1, 4], [0, 5, 4], [0, 2 ** 63 - 1, -2 ** 63, -2 ** 62, 4],
                                     [0, 2 ** 62, 2 ** 63 - 1, -2 ** 63, -2 ** 62, 0, 4]])
def test_offsets_out_of_order_are_refused(offsets):
    """Also those whose differences, taken in 64 bits, are all positive."""
    words = np.zeros(4, np.int32)
    g = binding.LightLDA(3, 2, 0.1, 0.01)
    assert binding.lda_load_corpus(g._h, words, np.array(offsets, np.int64)) == binding.LDA_ERANGE
    assert "non-decreasing" in binding.lda_last_error(g._h)
    assert binding.lda_load_corpus(g._h, words, np.array([0, 0, 3, 4, 4], np.int64)) == binding.LDA_OK


class _Budget:
    """A context's device memory from PyTorch's pool, refused beyond `left` bytes once that is set."""

    def __init__(self):
        self.left, self.sizes = None, {}
        alloc, free = binding.torch_caching_allocator(None)

        def take(n, user):
            if self.left is not None and n > self.left:
                return None
            p = alloc(n, user)
            if p and self.left is not None:
                self.left -= n
                self.sizes[p] = n
            return p

        def give(p, user):
            if self.left is not None and p:
                self.left += self.sizes.pop(p, 0)
            free(p, user)
        self.functions = binding.ALLOC_FN(take), binding.FREE_FN(give)

    def context(self, c, seed):
        g = binding.LightLDA(c.V, c.K, c.alpha, c.beta, allocator="cuda")
        g._allocator = self.functions     # alive as long as the context
        assert binding.lda_set_allocator(g._h, *self.functions) == 0
        g.load_corpus(c.word_ids.numpy(), c.doc_offsets.numpy())
        g.init(seed)
        return g


def _pair_with_budget(K=100, D=1_000):
    c = synth.generate(V=2_000, K=K, D=D, length=("fixed", 100), zipf_s=1.0, alpha=0.1, beta=0.01, seed=4)
    b, o = _Budget(), ldaref.Oracle(c.V, c.K, c.alpha, c.beta)
    o.load_corpus(c.word_ids.numpy(), c.doc_offsets.numpy())
    o.init(8)
    return c, b, b.context(c, 8), o


SPARE = 64 << 10   # scans' temporary storage


def test_document_rows_in_the_room_they_need():
    """Offsets, sizes and entries are all the device memory that the n_kd rows may insist on."""
    c, b, g, o = _pair_with_budget()
    want = o.get_csr(ldaref.NDK)
    for left in (12 * (c.n_docs + 1) + 8 * want[1].size + SPARE, 12 * (c.n_docs + 1) + 8 * c.n_tokens + SPARE, 1 << 40):
        b.left = left
        for x, y in zip(g.get_csr(binding.LDA_NDK), want):
            assert np.array_equal(x, y)
        assert b.left == left      # all of it went back
    b.left = 4 * want[1].size
    with pytest.raises(binding.LdaError) as e:
        g.get_csr(binding.LDA_NDK)
    assert e.value.status == binding.LDA_ENOMEM and b.left == 4 * want[1].size
    b.left = None


def test_word_rows_without_device_memory():
    """The n_kw rows lie in device memory already: to read them takes no more of it, if there is none."""
    c, b, g, o = _pair_with_budget()
    for sweep in range(2):
        want = o.get_csr(ldaref.NWK)
        nnz = want[1].size
        for left in (0, 8 * (c.V + 1), 8 * (c.V + 1) + SPARE + 4 * nnz, 1 << 40):
            b.left = left
            for x, y in zip(g.get_csr(binding.LDA_NWK), want):
                assert np.array_equal(x, y)
            assert b.left == left
        b.left = 0
        column = np.zeros(nnz, np.int32)
        assert binding.lda_get_counts(g._h, binding.LDA_NWK, None, None, column) == (binding.LDA_OK, nnz)
        assert np.array_equal(column, want[2])
        assert binding.lda_get_counts(g._h, binding.LDA_NWK, None, column[1:], None) == (binding.LDA_ERANGE, nnz)
        b.left = None
        for e in (g, o):
            e.sweep(1, 2)


def test_exact_conditional_sweep_without_room_for_the_matrix():
    """Beside the running sums the sweep insists on the documents' rows, not on n_kw as a matrix."""
    c, b, g, o = _pair_with_budget()
    rows = 12 * (c.n_docs + 1) + 8 * c.n_tokens
    matrix = 4 * c.V * c.K
    assert rows > SPARE and matrix > SPARE
    needed = 8 * c.n_tokens + 8 * c.V * c.K
    for left in (needed + max(rows, matrix) + SPARE, needed + rows + matrix + 8 * c.n_tokens + SPARE, 1 << 40):
        b.left = left
        g.gibbs_sweep(2)
        assert b.left == left
        o.gibbs_sweep(2)
        assert np.array_equal(g.get_assignments(), o.get_assignments())
    b.left = needed + rows // 4
    with pytest.raises(binding.LdaError) as e:
        g.gibbs_sweep(1)
    assert e.value.status == binding.LDA_ENOMEM
    b.left = None


HOST_MEMORY = """
import resource
import numpy as np
from paper_1412_1576_b200 import binding
g = binding.LightLDA(5, 4, 0.1, 0.01, allocator="cuda")
words, few = np.arange(40, dtype=np.int32) % 5, np.array([0, 10, 40], np.int64)
g.load_corpus(words, few)
g.init(1)
g.sweep(1, 2)
offsets, none = np.zeros(30_000_001, np.int64), np.zeros(0, np.int32)   # documents without a token
with open("/proc/self/statm") as f:
    now = int(f.read().split()[0]) * resource.getpagesize()
soft, hard = resource.getrlimit(resource.RLIMIT_AS)
resource.setrlimit(resource.RLIMIT_AS, (now + (48 << 20), hard))
rc = binding.lda_load_corpus(g._h, none, offsets)
resource.setrlimit(resource.RLIMIT_AS, (soft, hard))
assert rc == binding.LDA_ENOMEM, rc
g.sweep(1, 2)                                # the corpus it had is still there
assert int(g.get_nk().sum()) == 40
g.load_corpus(none, offsets)
print("done")
"""


def test_host_memory_that_cannot_be_had_is_an_error():
    """No exception leaves the library: a list of 120 MB under a limit that does not allow it."""
    import os
    import subprocess
    import sys
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", HOST_MEMORY], cwd=root, capture_output=True, text=True, timeout=120)
    assert r.returncode == 0 and r.stdout.strip() == "done", r.stdout + r.stderr
