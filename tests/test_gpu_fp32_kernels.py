"""The fp32 model's kernels at the edges of their tiles: the FFMA GEMM against
float64 products (row and feature remainders, depths that are no multiple of
a chunk, each tile size), the attention against the oracle (each number of
queries per CTA, query groups that do not divide it, several documents)."""
import numpy as np
import pytest

import oracle
from paper_2609_17983_gb300 import synth

try:
    from paper_2609_17983_gb300 import kvrepair as kv
except ImportError as _e:  # pragma: no cover
    kv, _IMPORT_ERROR = None, _e

pytestmark = pytest.mark.gpu


def rel(a, b):
    return float(np.abs(a - b).max() / np.abs(b).max())


@pytest.mark.parametrize("dtype", ["fp32", "bf16"])
@pytest.mark.parametrize("M", [1, 17, 40, 257, 1500])
def test_ffma_gemm_edges(dtype, M):
    # depths of 260 and 688, which the tensor-core GEMM does not take, features
    # 512, 260, 1376 and 1021: sums of at most 688 fp32 products, whose
    # rounding is about sqrt(688) 2^-24 = 2e-6 of the largest result (the wo of
    # a bf16 model, 256 deep and 260 wide, too; SwiGLU there rounds to bf16)
    cfg = synth.preset("tiny", dtype=dtype, d_model=260, vocab=1021)
    m = kv.Model(cfg, synth.weights(cfg, 0), max_context=256, max_rows=1536)
    val = (lambda a: synth.bf16_bits_to_f32(a).astype(np.float64)) if dtype == "bf16" else \
        (lambda a: a.astype(np.float64))
    W = {n: val(m.read_tensor(n, 0)) for n in ("wq", "wk", "wv", "wo", "wg", "wu", "wd")}
    W["wqkv"] = np.concatenate([W["wq"], W["wk"], W["wv"]])
    W["lm_head"] = val(m.read_tensor("lm_head"))
    for name in ("wqkv", "wo", "wd", "lm_head"):
        n_out, k = W[name].shape
        x = synth.tensor(M, 5, (M, k), dtype, std=1.0)
        assert rel(kv.kvr_linear(m.h, name, 0, x, n_out), val(x) @ W[name].T) <= 1e-5, name
    x = synth.tensor(M, 6, (M, 260), dtype, std=1.0)
    g, u = val(x) @ W["wg"].T, val(x) @ W["wu"].T
    got = kv.kvr_linear(m.h, "wgu", 0, x, 688)
    assert rel(got, g / (1 + np.exp(-g)) * u) <= (1e-5 if dtype == "fp32" else 4e-3)
    m.close()


def loaded(model, cfg, n, seed):
    doc = synth.document(seed, n, cfg["vocab"])
    k, v = synth.kv_rows(seed, n, cfg["n_layers"], cfg["n_kv_heads"], cfg["head_dim"], "fp32",
                         std=0.45)
    to = lambda x: np.ascontiguousarray(x.transpose(1, 0, 2, 3))  # noqa: E731
    return model.load_cache(doc, k, v), oracle.Cache(to(k), to(v), doc.copy())


def check_rows(cfg, cache, ref, P):
    gk, gv = cache.read(P)
    for l in range(cfg["n_layers"]):
        assert rel(gk[:, l], ref.k[l, P]) <= 1e-4 and rel(gv[:, l], ref.v[l, P]) <= 1e-4, l


@pytest.mark.parametrize("H,G,dh,rows", [(6, 2, 128, 1), (6, 2, 128, 33), (6, 2, 128, 250),
                                         (6, 2, 64, 500), (4, 4, 64, 690)])
def test_fp32_attention(H, G, dh, rows):
    cfg = synth.preset("tiny", n_heads=H, n_kv_heads=G, head_dim=dh)
    W = synth.weights(cfg, 0)
    model = kv.Model(cfg, W, max_context=1024, max_rows=1024)
    cache, ref = loaded(model, cfg, 700, 4)
    A = np.sort(np.random.default_rng(rows).permutation(700)[:rows])
    none = np.zeros(0, np.int32)
    cache.repair(none, 0, A)
    check_rows(cfg, cache, oracle.repair(cfg, W, ref, none, 0, A), A)
    model.close()


@pytest.mark.parametrize("H,G,rows", [(6, 2, 40), (8, 1, 200), (10, 2, 200)])
def test_fp32_attention_of_several_documents(H, G, rows):
    cfg = synth.preset("tiny", n_heads=H, n_kv_heads=G)
    W = synth.weights(cfg, 0)
    model = kv.Model(cfg, W, max_context=1024, max_rows=1024)
    docs = [loaded(model, cfg, n, n) for n in (500, 333)]
    rng = np.random.default_rng(0)
    reqs, want = [], []
    for cache, ref in docs:
        new = synth.edit_tokens(3, ref.tokens[7:10], cfg["vocab"])
        A = np.sort(rng.permutation(np.arange(10, cache.n))[:rows])
        reqs.append((cache, [(7, new)], A))
        want.append(oracle.repair(cfg, W, ref, new, 7, A))
    model.repair_batch(reqs)
    for (cache, _, A), ref in zip(reqs, want):
        check_rows(cfg, cache, ref, np.concatenate([np.arange(7, 10), A]))
    model.close()


@pytest.mark.parametrize("rows", [1, 60, 120])
def test_attention_keeps_a_lone_nan(rows):
    # fresh keys are NaN (their projection holds one), stale keys are finite: a row at
    # the start of a block of 32 keys sees no other key of that block, and its output,
    # so the next layer's values, is NaN; rows for each number of queries per CTA
    cfg = synth.preset("tiny", n_layers=2)
    W = synth.weights(cfg, 0)
    W["layers"][0]["wk"] = W["layers"][0]["wk"].copy()
    W["layers"][0]["wk"][:, 3] = np.nan
    model = kv.Model(cfg, W, max_context=4096, max_rows=512)
    n = 32 * 121
    cache, _ = loaded(model, cfg, n, 5)
    at = 32 * np.arange(1, rows + 1)
    cache.repair(np.zeros(0, np.int32), 0, at)
    k, v = cache.read(at)
    assert np.isnan(k[:, 0]).all() and np.isnan(v[0, 1]).all()
    assert np.isnan(v[:, 1]).all() and np.isfinite(v[:, 0]).all()
    model.close()
