"""kvr_margin, whose two answers run in one pass where that gives the same bits:
exactly the difference of the two kvr_answer_logprob calls, the document's
cache untouched -- with n on a page boundary and inside a page, a last page
that the longer answer crosses, answers of one and of different lengths, and
row counts that fall back to two passes."""
import numpy as np
import pytest

from paper_2609_17983_gb300 import synth

try:
    from paper_2609_17983_gb300 import kvrepair as kv
except ImportError as _e:  # pragma: no cover
    kv, _IMPORT_ERROR = None, _e

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [200, 256, 250])
def test_margin_is_the_difference_of_two_log_probabilities(n):
    cfg = synth.preset("qwen7b", n_layers=2)
    model = kv.Model(cfg, None, seed=0, max_context=512, max_rows=256)
    cache = model.prefill(synth.document(1, n, cfg["vocab"]))
    k0, v0 = cache.read_raw(np.arange(n))
    launches = []
    for mp, m_new, m_old in ((24, 6, 6), (5, 3, 7), (1, 1, 1), (9, 5, 5), (40, 20, 2)):
        prompt, a_new, a_old = (synth.fill_tokens(7 + i, c, cfg["vocab"], 13)
                                for i, c in enumerate((mp, m_new, m_old)))
        l0 = model.launches()
        got = model.margin(cache, prompt, a_new, a_old)
        l1 = model.launches()
        want = (model.answer_logprob(cache, prompt, a_new)
                - model.answer_logprob(cache, prompt, a_old))
        assert got == want, (mp, m_new, m_old)
        launches.append((l1 - l0) / (model.launches() - l1))
    assert min(launches) < 0.7  # one pass where it can be
    k1, v1 = cache.read_raw(np.arange(n))
    assert np.array_equal(k0, k1) and np.array_equal(v0, v1)
    model.close()
