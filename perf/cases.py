"""What this library is asked to do in real use, as measurable cases.

Kinds of work (field "kind"):

train    `iters` sweeps of an ongoing run, then what a training loop looks at between two stretches of
         sweeps: the log-likelihood and a snapshot of every assignment (queued with
         get_assignments_async, read beside it, complete after wait()).
resume   one step through host buffers: assignments in from pinned memory (counts and tables rebuilt),
         one sweep, assignments out, log-likelihood.  Checkpoint/restart, and samplers whose state
         lives on the host.
start    from a corpus in host arrays to a first look: new context, token layout, initial assignments and
         counts, one sweep, log-likelihood and snapshot.
export   the trained model and the documents' topic counts as CSR arrays (get_nk, lda_get_counts).
gibbs    sweeps of the exact-conditional yardstick and their log-likelihood.

Sizes of the listed cases are the five workloads of synth.CONFIGS (some with fewer documents, so that a
state fits a card several times over), beside a corpus of long documents and odd sizes.
"""
import math

import numpy as np
import torch

from paper_1412_1576_b200 import synth
from paper_1412_1576_b200.binding import (LDA_NDK, LDA_NWK, PROPOSALS_CYCLE, PROPOSALS_DOC,
                                          PROPOSALS_WORD, LightLDA, lda_get_counts)

MODES = {"cycle": PROPOSALS_CYCLE, "word": PROPOSALS_WORD, "doc": PROPOSALS_DOC}
# sweeps a state has behind it before it is measured: a run is past its uniform random start most of the time
BURN_IN = 8


def _case(name, kind, V, K, D, law, mean, sigma, zipf, alpha, iters=1, mh=2, mode="cycle"):
    c = dict(kind=kind, V=V, K=K, D=D, law=law, mean=mean, sigma=sigma, zipf=zipf, alpha=alpha,
             beta=0.01, iters=iters, mh=mh, mode=mode)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # "tiny": 10 000 tokens, one sweep at a time with a look at the likelihood after each -- all latency
        _case("tiny_monitor", "train", 500, 16, 200, "fixed", 50, 0.0, 0.0, 0.1, iters=1),
        # "small": 2 M tokens, K = 100
        _case("small_train", "train", 10_000, 100, 20_000, "poisson", 100, 0.0, 1.05, 0.5, iters=10),
        # "mid": 99 M tokens, K = 1000 (NYTimes shape)
        _case("mid_train", "train", 100_000, 1_000, 300_000, "poisson", 330, 0.0, 1.05, 0.1, iters=10),
        # "large": 738 M tokens, K = 10 000 (PubMed shape), the workload the headline figure is quoted on
        _case("large_train", "train", 141_000, 10_000, 8_200_000, "poisson", 90, 0.0, 1.1, 0.01, iters=5),
        # the same shape at a tenth of the documents with the four proposals per token its configuration names
        _case("large_tenth_mh4", "train", 141_000, 10_000, 820_000, "poisson", 90, 0.0, 1.1, 0.01, iters=5, mh=4),
        # "big" at a fifth of the documents: V = 10^6, K = 10^5, 32-bit topics, ragged (log-normal) documents
        _case("big_fifth_train", "train", 1_000_000, 100_000, 2_000_000, "lognormal", 100, 1.0, 1.0, 0.01, iters=3),
        # books: documents of thousands to a hundred thousand tokens, odd vocabulary and topic count
        _case("books_train", "train", 30_011, 777, 3_001, "lognormal", 4_000, 0.8, 1.05, 0.1, iters=5),
        # the word-proposal alone (the ablation of Figure 11), odd sizes
        _case("word_only_train", "train", 20_011, 333, 33_331, "poisson", 151, 0.0, 1.05, 0.15, iters=5, mode="word"),
        # host round trip of a tenth of "large" (74 M tokens)
        _case("large_tenth_resume", "resume", 141_000, 10_000, 820_000, "poisson", 90, 0.0, 1.1, 0.01),
        # start-up on a fifth of "mid" (20 M tokens)
        _case("mid_fifth_start", "start", 100_000, 1_000, 60_000, "poisson", 330, 0.0, 1.05, 0.1),
        # model and document rows out, a tenth of "mid" (10 M tokens)
        _case("mid_tenth_export", "export", 100_000, 1_000, 30_000, "poisson", 330, 0.0, 1.05, 0.1),
        # exact-conditional sweep on "small"
        _case("small_gibbs", "gibbs", 10_000, 100, 20_000, "poisson", 100, 0.0, 1.05, 0.5, iters=1),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: tokens, topics, vocabulary and document lengths over their logarithms."""
    kind = rng.choices(["train", "resume", "start", "export", "gibbs"], [11, 3, 2, 2, 2])[0]
    n_max = {"train": 300e6, "resume": 100e6, "start": 50e6, "export": 20e6, "gibbs": 4e6}[kind]
    N = _log_uniform(rng, 10_000, n_max)
    if kind == "gibbs":  # the yardstick keeps V*K running sums
        K, V = _log_uniform(rng, 16, 1_000), _log_uniform(rng, 500, 20_000)
    else:
        K, V = _log_uniform(rng, 16, 100_000), _log_uniform(rng, 500, 1_000_000)
    # topic bits + bits of the longest document's length stay within 32
    mean = _log_uniform(rng, 10, 150 if K > 16_384 else 1_500)
    law = rng.choice(["fixed", "poisson", "lognormal"])
    mode, mh, iters = "cycle", 2, 1
    if kind in ("train", "resume", "start"):
        mode = rng.choices(["cycle", "word", "doc"], [8, 1, 1])[0]
        mh = rng.choices([1, 2, 3, 4, 8], [1, 6, 1, 3, 1])[0]
    if kind == "train":  # no more work than the largest listed case; a sweep costs more at large K
        most = (1.8e9 if K > 16_384 else 5e9) / (N * max(mh, 2))
        iters = max(1, min(rng.randint(1, 10), int(most)))
    return _case("", kind, V, K, max(1, N // mean), law, mean, round(rng.uniform(0.5, 1.0), 3) if law == "lognormal" else 0.0,
                 rng.choice([0.0, 1.0, 1.05, 1.1]), rng.choice([0.01, 0.1, 0.5]), iters, mh, mode)


def _corpus(case, seed):
    """(word ids, document offsets) on the GPU.  Lengths follow the case's law; their sum is D * mean for
    every seed: the corpus is drawn a little longer and every document shortened in proportion."""
    D, mean, sigma = case["D"], case["mean"], case["sigma"]
    gen = dict(V=case["V"], K=case["K"], D=D, zipf_s=case["zipf"] or None, alpha=case["alpha"], beta=case["beta"],
               seed=seed, device="cuda")
    n = D * mean
    if case["law"] == "fixed":
        c = synth.generate(length=("fixed", mean), **gen)
        return c.word_ids, c.doc_offsets
    spread = mean ** -0.5 if case["law"] == "poisson" else math.sqrt(math.expm1(sigma * sigma))
    longer = 1.0 + 6.0 * spread / math.sqrt(D)
    while True:
        c = synth.generate(length=(case["law"], mean * longer, sigma), **gen)
        if c.n_tokens >= n:
            break
        longer *= 2.0
    lengths = c.doc_offsets.diff()
    short = (lengths.double() * (n / c.n_tokens)).floor().long()
    room = torch.nonzero(short < lengths).flatten()[:n - int(short.sum())]
    short[room] += 1
    place = torch.arange(c.n_tokens, device="cuda") - torch.repeat_interleave(c.doc_offsets[:-1], lengths)
    words = c.word_ids[place < torch.repeat_interleave(short, lengths)]
    offsets = torch.zeros_like(c.doc_offsets)
    torch.cumsum(short, 0, out=offsets[1:])
    return words, offsets


def _pinned_assignments(case, n):
    # 16-bit topics cross the host link whenever the library stores them in 16 bits
    return torch.empty(n, dtype=torch.int16 if case["K"] <= 65_536 else torch.int32, pin_memory=True)


def prepare(case, seed):
    words, offsets = _corpus(case, seed)
    n = words.numel()
    if case["kind"] == "start":  # the corpus as a program has it after reading it: host arrays
        return dict(case=case, seed=seed, words=words.cpu().numpy(), offsets=offsets.cpu().numpy(),
                    z=_pinned_assignments(case, n))
    lda = LightLDA(case["V"], case["K"], case["alpha"], case["beta"])
    lda.load_corpus(words, offsets)
    lda.init(seed)
    lda.set_proposals(MODES[case["mode"]])
    lda.sweep(BURN_IN, case["mh"])
    state = dict(case=case, seed=seed, lda=lda)
    if case["kind"] in ("train", "resume", "gibbs"):
        state["z"] = _pinned_assignments(case, n)
    if case["kind"] == "resume":
        state["z_in"] = _pinned_assignments(case, n)
        lda.get_assignments_async(state["z_in"])
        lda.wait()
    if case["kind"] == "export":  # the caller's buffers: a row has at most as many entries as it has tokens
        for which, rows in (("n_kw", case["V"]), ("n_kd", case["D"])):
            state[which] = (np.zeros(rows + 1, np.int64), np.zeros(n, np.int32), np.zeros(n, np.int32))
    return state


def _look(lda, z):
    """Snapshot of the assignments and the log-likelihood, the one on its way while the other is computed."""
    lda.get_assignments_async(z)
    total, word, doc = lda.loglik()
    lda.wait()
    return {"loglik": total, "loglik_words": word, "loglik_docs": doc, "z": z}


def run(state):
    case, kind = state["case"], state["case"]["kind"]
    if kind == "start":
        lda = LightLDA(case["V"], case["K"], case["alpha"], case["beta"])
        lda.load_corpus(state["words"], state["offsets"])
        lda.init(state["seed"])
        lda.set_proposals(MODES[case["mode"]])
        lda.sweep(1, case["mh"])
        first = _look(lda, state["z"])
        lda.close()
        return first
    lda = state["lda"]
    if kind == "train":
        lda.sweep(case["iters"], case["mh"])
        return _look(lda, state["z"])
    if kind == "resume":
        z = state["z_in"].numpy()
        if z.dtype == np.int16:
            lda.set_assignments_u16(z.view(np.uint16), state["seed"], BURN_IN)
        else:
            lda.set_assignments(z, state["seed"], BURN_IN)
        lda.sweep(1, case["mh"])
        return _look(lda, state["z"])
    if kind == "export":
        out = {"n_k": lda.get_nk()}
        for which, name in ((LDA_NWK, "n_kw"), (LDA_NDK, "n_kd")):
            status, entries = lda_get_counts(lda._h, which, *state[name])
            if status:
                raise RuntimeError(f"lda_get_counts: status {status}")
            out[name], out[name + "_entries"] = state[name], entries
        return out
    lda.gibbs_sweep(case["iters"])
    return _look(lda, state["z"])


def work(case):
    """Per sweep every token's word and topic are read and its topic written; a snapshot writes every topic."""
    n = float(case["D"]) * case["mean"]
    t = 2.0 if case["K"] <= 65_536 else 4.0
    sweep, snapshot = n * (4.0 + 2.0 * t), n * t
    kind = case["kind"]
    if kind == "export":  # topics in; (topic, count) entries out, most topics of a document occurring once
        return {"bytes": t * n + 8.0 * 0.75 * n, "flops": 0.0}
    if kind == "gibbs":  # one term per topic of the document, a handful of operations each
        terms = min(case["K"], 0.75 * case["mean"])
        return {"bytes": case["iters"] * sweep + snapshot, "flops": case["iters"] * n * terms * 8.0}
    # topics in, or word ids and offsets
    extra = {"resume": snapshot, "start": 4.0 * n + 8.0 * case["D"]}.get(kind, 0.0)
    # about a dozen double-precision operations per proposal
    return {"bytes": case["iters"] * sweep + snapshot + extra, "flops": case["iters"] * n * case["mh"] * 12.0}


def tolerance(case):
    if case["kind"] == "export":
        return "exact"
    # topics and counts are whole numbers and stay the same; the log-likelihood is a sum of up to 10^9
    # double-precision terms of both signs, taken in any order
    return {"rel": 1e-9, "max": 1e-9, "differ": 0.0}
