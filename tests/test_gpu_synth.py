"""Inputs made on the GPU depend on the configuration and the seed alone."""
import pytest

from paper_1412_1576_b200 import synth

pytestmark = pytest.mark.gpu


def test_word_distribution_is_the_same_every_time(monkeypatch):
    """The cumulative distribution the words are drawn from, bit for bit: a difference in its last bits shows in one draw
    of some 10^9, which comparing small corpora would never meet."""
    import torch
    seen = []
    search = torch.searchsorted
    monkeypatch.setattr(torch, "searchsorted", lambda cdf, u: (seen.append(cdf.clone()), search(cdf, u))[1])
    corpora = [synth.generate(V=1_000_000, K=50, D=2_000, length=("poisson", 50.0), zipf_s=1.0, alpha=0.1, beta=0.01, seed=3,
                              device="cuda") for _ in range(12)]
    assert len(seen) == 12
    for cdf, c in zip(seen, corpora):
        assert torch.equal(cdf, seen[0])
        assert torch.equal(c.word_ids, corpora[0].word_ids) and torch.equal(c.doc_offsets, corpora[0].doc_offsets)
    exact = torch.arange(1, 1_000_001, dtype=torch.float64).reciprocal().cumsum(0)
    assert torch.allclose(seen[0].cpu(), exact / exact[-1], rtol=1e-12, atol=0)
