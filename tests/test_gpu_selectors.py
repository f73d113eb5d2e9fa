"""The Attention selector's scoring kernels over long pools: CTAs that take
several key chunks each (two, three, and a last CTA with fewer), two query
tiles per kv group with the second one ragged, pool lengths that leave a logit
row's last quad and the last chunk ragged -- against the oracle's scores on the
same stale cache, within the tie band that the other selector tests use."""
import numpy as np
import pytest

import oracle
from paper_2609_17983_gb300 import synth
from tests.test_gpu_margin import Allocator

try:
    from paper_2609_17983_gb300 import kvrepair as kv
except ImportError as _e:  # pragma: no cover
    kv, _IMPORT_ERROR = None, _e

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,dh,n", [("bf16", 128, 4299), ("bf16", 64, 3001), ("fp32", 128, 3002),
                                        ("fp32", 64, 4301)])
def test_attention_selector_of_long_pools(dtype, dh, n):
    cfg = synth.preset("tiny", dtype=dtype, d_model=512, ffn=512, n_heads=32, n_kv_heads=8,
                       head_dim=dh)
    W = synth.weights(cfg, 0)
    s, L, K = 100, 11, 32  # 44 queries a kv group
    doc = synth.document(17, n, cfg["vocab"])
    new = synth.edit_tokens(18, doc[s:s + L], cfg["vocab"], cfg["delim_id"])
    bits = synth.kv_rows(19, n, cfg["n_layers"], 8, dh, "bf16", std=0.45)
    k, v = (synth.bf16_bits_to_f32(x) for x in bits)
    model = kv.Model(cfg, None, seed=0, max_context=4608, max_rows=256)
    cache = model.load_cache(doc, *(bits if dtype == "bf16" else (k, v)))
    got = model.select(cache, "attention", K, s, new)
    to = lambda x: np.ascontiguousarray(x.transpose(1, 0, 2, 3))  # noqa: E731
    sc, D = oracle.scores(cfg, W, oracle.Cache(to(k), to(v), doc.copy()), "attention", s, new)
    ref = oracle.topk(sc, D, K)
    band = (1e-4 if dtype == "fp32" else 2e-2) * np.abs(sc[D]).max()
    kth = sc[ref].min()
    assert len(got) == K
    assert all(sc[j] >= kth - band for j in got)
    assert all(j in got for j in ref if sc[j] > kth + band)
    model.close()


# The radix select of the K largest keys: pools around a thread's share (1024
# keys) and of several keys a thread, up to the longest context; K from one to
# the whole pool; delimiters that are many, few and absent.  The keys are whole numbers: exactly the oracle's set.
@pytest.mark.parametrize("n", [40, 1055, 1056, 1057, 5000, 16384])
def test_simple_policies_match_the_oracle(n):
    cfg = synth.preset("tiny", n_layers=1)
    model = kv.Model(cfg, None, seed=0, max_context=16384, max_rows=1024)
    rng = np.random.default_rng(n)
    s, L = 28, 4  # the pool: n - 32 positions
    for every in (3, 700, None):
        doc = synth.document(n, n, cfg["vocab"])
        if every:
            at = np.arange(s + L + every - 1, n, every)
            doc[at[rng.random(len(at)) < 0.9]] = cfg["delim_id"]
        new = synth.edit_tokens(2, doc[s:s + L], cfg["vocab"], cfg["delim_id"])
        cache = model.prefill(doc)
        ref = oracle.empty_cache(cfg, n)
        ref.tokens[:] = doc
        for policy, seed in (("random", 0), ("random", n), ("structural", 0),
                             ("editlocal_boundary", 0), ("editlocal", 0)):
            for K in (1, 32, n // 2, n - s - L):
                got = model.select(cache, policy, K, s, new, seed)
                want = oracle.select(cfg, None, ref, policy, K, s, new, seed)
                assert got.tolist() == want.tolist(), (policy, every, K)
        cache.close()
    model.close()


def test_attention_selector_scratch_of_a_long_span():
    # 1000 span rows of 24 layers over a pool of 24: the queries kept are one
    # group's (64 MB, as its logits), not all layers' (197 MB)
    mem, model = Allocator(), None
    try:
        cfg = synth.preset("tiny", dtype="bf16", d_model=512, ffn=512, n_heads=32, n_kv_heads=8,
                           head_dim=64, n_layers=24)
        model = kv.Model(cfg, None, seed=0, max_context=1100, max_rows=1024)
        cache = model.prefill(synth.document(3, 1034, cfg["vocab"]))
        a0 = mem.asked
        model.select(cache, "attention", 8, 10, synth.fill_tokens(4, 1000, cfg["vocab"], 13))
        saved_rows = 1000 * 24 * 2 * 8 * 64 * 2
        assert mem.asked - a0 < saved_rows + 2 * (64 << 20) + (1 << 20)
    finally:
        if model is not None:
            model.close()
        kv.use_cuda_allocator()
