"""kvr_margin, whose two answers run in one pass where that gives the same bits:
exactly the difference of the two kvr_answer_logprob calls, the document's
cache untouched -- with n on a page boundary and inside a page, a last page
that the longer answer crosses, answers of one and of different lengths, and
row counts that fall back to two passes."""
import ctypes

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


class Allocator:
    """The library's allocator hook over PyTorch's: bytes asked for, and refusals."""

    def __init__(self):
        import torch
        self.asked, self.refuse = 0, False

        def alloc(nbytes, ctx):
            if self.refuse:
                return None
            self.asked += int(nbytes)
            return torch.cuda.caching_allocator_alloc(int(nbytes))

        def free(ptr, ctx):
            if ptr:
                torch.cuda.caching_allocator_delete(ptr)

        self.hooks = (kv._ALLOC(alloc), kv._FREE(free))
        assert kv._lib.kvr_set_allocator(*(ctypes.cast(h, ctypes.c_void_p) for h in self.hooks),
                                         None) == 0


def test_margin_memory_is_the_models():
    # a cache holds the pages of its positions and the reserve, no more; the second
    # answer's pages come with the first margin, once for all documents; where they
    # cannot be had the margin runs in two passes and is the same
    mem, model = Allocator(), None
    try:
        cfg = synth.preset("qwen7b", n_layers=2)
        page = 64 * cfg["n_layers"] * 2 * cfg["n_kv_heads"] * cfg["head_dim"] * 2
        model = kv.Model(cfg, None, seed=0, max_context=512, max_rows=256)
        caches = []
        for n, pages in ((10, 2), (200, 5), (256, 5)):
            a0 = mem.asked
            caches.append(model.prefill(synth.document(1, n, cfg["vocab"])))
            assert pages * page <= mem.asked - a0 < pages * page + 65536, n
        ask = [synth.fill_tokens(7 + i, c, cfg["vocab"], 13) for i, c in enumerate((24, 6, 6))]
        mem.refuse = True
        l0 = model.launches()
        two = [model.margin(c, *ask) for c in caches]
        l1 = model.launches()
        mem.refuse = False
        a0 = mem.asked
        one = [model.margin(c, *ask) for c in caches]
        assert one == two and model.launches() - l1 < 0.7 * (l1 - l0)
        assert 2 * page <= mem.asked - a0 < 2 * page + 65536
        a0 = mem.asked
        assert [model.margin(c, *ask) for c in reversed(caches)] == two[::-1]
        assert mem.asked == a0
    finally:
        if model is not None:
            model.close()
        kv.use_cuda_allocator()
