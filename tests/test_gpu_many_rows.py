"""The kernels of passes with many rows at the sizes where they can go wrong,
against the oracle and float64 products: two query tiles per CTA in the
attention (odd tile counts, ragged tiles, split and unsplit key ranges,
several documents), pairs of CTAs per tile in the GEMM (ragged token tiles, a
feature count that is an odd multiple of 128, few K blocks), vector row
kernels."""
from fractions import Fraction

import numpy as np
import pytest

import oracle
from paper_2609_17983_gb300 import synth

try:
    from paper_2609_17983_gb300 import kvrepair as kv
except ImportError as _e:  # pragma: no cover
    kv, _IMPORT_ERROR = None, _e

pytestmark = pytest.mark.gpu
TOL = 2e-2  # bf16 path, as everywhere


def rel(a, b):
    return float(np.abs(a - b).max() / np.abs(b).max())


def small_cfg(**over):
    return synth.preset("tiny", dtype="bf16", d_model=512, ffn=512, **over)


def loaded(model, cfg, n, seed):
    doc = synth.document(seed, n, cfg["vocab"])
    k, v = synth.kv_rows(seed, n, cfg["n_layers"], cfg["n_kv_heads"], cfg["head_dim"], "bf16",
                         std=0.45)
    to = lambda x: np.ascontiguousarray(synth.bf16_bits_to_f32(x).transpose(1, 0, 2, 3))  # noqa: E731
    return model.load_cache(doc, k, v), oracle.Cache(to(k), to(v), doc.copy())


def check_rows(cfg, cache, ref, P):
    gk, gv = cache.read(P)
    for l in range(cfg["n_layers"]):
        assert rel(gk[:, l], ref.k[l, P]) <= TOL and rel(gv[:, l], ref.v[l, P]) <= TOL, l


# (heads, kv heads, head_dim, n, rows, how): a key range split over CTAs with
# whole and with odd pairs of ragged tiles (7 heads a kv head: tiles of 126
# vectors), and one CTA per pair over many waves
@pytest.mark.parametrize("H,G,dh,n,rows,how", [(8, 2, 128, 2300, 1100, "window"),
                                               (14, 2, 64, 2300, 701, "scatter"),
                                               (32, 8, 64, 2400, 2400, "window")])
def test_attention_pairs_of_tiles(H, G, dh, n, rows, how):
    cfg = small_cfg(n_heads=H, n_kv_heads=G, head_dim=dh)
    W = synth.weights(cfg, 0)
    model = kv.Model(cfg, None, seed=0, max_context=4096, max_rows=4096)
    cache, ref = loaded(model, cfg, n, 11)
    A = (np.arange(n - rows, n) if how == "window" else
         np.sort(np.random.default_rng(1).permutation(np.arange(200, n))[:rows]))
    none = np.zeros(0, np.int32)
    cache.repair(none, 0, A)
    ref = oracle.repair(cfg, W, ref, none, 0, A)
    check_rows(cfg, cache, ref, A)
    model.close()


def test_attention_pairs_of_several_documents():
    cfg = small_cfg(n_heads=8, n_kv_heads=2, head_dim=128)
    W = synth.weights(cfg, 0)
    model = kv.Model(cfg, None, seed=0, max_context=4096, max_rows=4096)
    docs = [loaded(model, cfg, n, 20 + n) for n in (2300, 1501, 700)]
    rng = np.random.default_rng(2)
    reqs, want = [], []
    for (cache, ref), rows in zip(docs, (900, 601, 20)):  # odd tile counts, a lone tile
        s = 100
        new = synth.edit_tokens(3, ref.tokens[s:s + 5], cfg["vocab"])
        A = np.sort(rng.permutation(np.arange(s + 5, cache.n))[:rows])
        reqs.append((cache, [(s, new)], A))
        want.append(oracle.repair(cfg, W, ref, new, s, A))
    model.repair_batch(reqs)
    for (cache, edits, A), ref in zip(reqs, want):
        check_rows(cfg, cache, ref, np.concatenate([np.arange(100, 105), A]))
    model.close()


@pytest.mark.parametrize("rows", [20, 500])
def test_batches_of_other_documents_in_turn(rows):
    # every batch, and a margin, puts its documents' tensor maps where the last one's
    # were: documents of other lengths and in another order, without a pause between
    cfg = small_cfg(n_heads=8, n_kv_heads=2, head_dim=128)
    W = synth.weights(cfg, 0)
    model = kv.Model(cfg, None, seed=0, max_context=4096, max_rows=4096)
    docs = [loaded(model, cfg, n, 30 + n) for n in (2300, 1501, 700, 1100)]
    rng = np.random.default_rng(rows)
    done = []
    for pick in ((0, 1), (2, 3, 0), (1, 0), (3, 2)):
        reqs = []
        for i in pick:
            cache, ref = docs[i]
            s = int(rng.integers(0, 100))
            new = synth.edit_tokens(3 + s, ref.tokens[s:s + 5], cfg["vocab"])
            A = np.sort(rng.permutation(np.arange(s + 5, cache.n))[:rows])
            reqs.append((cache, [(s, new)], A))
            docs[i] = (cache, oracle.repair(cfg, W, ref, new, s, A))
            done.append((i, np.concatenate([np.arange(s, s + 5), A])))
        model.repair_batch(reqs)
    prompt, a, b = (synth.fill_tokens(7 + i, c, cfg["vocab"], 13) for i, c in enumerate((9, 5, 3)))
    for i in (1, 2):
        got = model.margin(docs[i][0], prompt, a, b)
        want = (oracle.answer_logprob(cfg, W, docs[i][1], prompt, a)
                - oracle.answer_logprob(cfg, W, docs[i][1], prompt, b))
        assert abs(got - want) <= TOL * max(1.0, abs(want))
    for i, P in done:
        check_rows(cfg, *docs[i], P)
    model.close()


@pytest.mark.parametrize("M", [961, 1537])
def test_gemm_pairs_of_ctas(M):
    # 7040, 4224 and 8576 output features: odd multiples of 128, so the last
    # feature tile is half empty; 66 and 67 K blocks (the last unit of two is
    # short), ragged token tiles, tiles split over clusters; a sample of rows
    cfg = synth.preset("llama8b", n_layers=1, d_model=4224, n_heads=33, n_kv_heads=11, ffn=4288,
                       vocab=1024)
    m = kv.Model(cfg, None, seed=0, max_context=256, max_rows=2048)
    f64 = lambda b: synth.bf16_bits_to_f32(b).astype(np.float64)  # noqa: E731
    x, xd = (synth.tensor(M, t, (M, k), "bf16", std=1.0) for t, k in ((5, 4224), (6, 4288)))
    at = np.unique(np.concatenate([np.arange(0, M, 61), np.arange(M - 5, M)]))
    wqkv = np.concatenate([m.read_tensor(n, 0) for n in ("wq", "wk", "wv")])
    # fp32 sums of exact products: 1e-3 as for the other GEMMs; SwiGLU rounds to bf16
    for name, w, y in (("wqkv", wqkv, x), ("wo", m.read_tensor("wo", 0), x),
                       ("wd", m.read_tensor("wd", 0), xd)):
        got = kv.kvr_linear(m.h, name, 0, y, w.shape[0])[at]
        assert rel(got, f64(y[at]) @ f64(w).T) <= 1e-3, name
    g = f64(x[at]) @ f64(m.read_tensor("wg", 0)).T
    u = f64(x[at]) @ f64(m.read_tensor("wu", 0)).T
    got = kv.kvr_linear(m.h, "wgu", 0, x, 4288)[at]
    assert rel(got, g / (1.0 + np.exp(-g)) * u) <= 1e-2
    m.close()


@pytest.mark.parametrize("vocab", [1024, 1021, 20, 18])
def test_answer_logprob_row_widths(vocab):
    # rows on 16-byte boundaries and rows that are not, and rows with fewer
    # entries than a cluster's CTAs have slices
    cfg = synth.preset("tiny", vocab=vocab)
    W = synth.weights(cfg, 0)
    model = kv.Model(cfg, None, seed=0, max_context=256, max_rows=256)
    doc = synth.document(5, 100, vocab)
    prompt, answer = synth.fill_tokens(6, 7, vocab, 13), synth.fill_tokens(7, 5, vocab, 13)
    got = model.answer_logprob(model.prefill(doc), prompt, answer)
    want = oracle.answer_logprob(cfg, W, oracle.prefill(cfg, W, doc), prompt, answer)
    assert abs(got - want) <= 1e-4 * abs(want)  # the fp32 path's tolerance
    model.close()


@pytest.mark.parametrize("vocab,ids", [(1021, [0]), (1021, [1020]), (1024, [8, 9, 10, 11]),
                                       (1024, [700]), (18, [17])])
def test_answer_logprob_of_a_nan(vocab, ids):
    # a NaN among the logits, also where a thread sees nothing else: the
    # log-softmax of the row is NaN
    cfg = synth.preset("tiny", vocab=vocab)
    W = synth.weights(cfg, 0)
    W["lm_head"] = W["lm_head"].copy()
    W["lm_head"][ids] = np.nan
    model = kv.Model(cfg, W, max_context=256, max_rows=256)
    cache = model.prefill(np.arange(2, 82, dtype=np.int32) % vocab)
    prompt, answer = np.array([3, 4], np.int32), np.array([5], np.int32)
    assert np.isnan(model.answer_logprob(cache, prompt, answer))
    model.close()


@pytest.mark.parametrize("policy,edit,n", [("attention", 3, 1500), ("attention", 220, 1500),
                                           ("attention", 700, 1110),
                                           ("cacheblend", 3, 1500), ("cacheblend", 3, 700)])
def test_model_selectors_over_layer_groups(policy, edit, n):
    # Attention: 220 span rows' logits of 14 layers are more than one launch takes
    # (groups of 6, 6 and 2 layers), 700 rows' queries (13 and 1), 3 rows' are one
    # launch; CacheBlend:
    # head-wise projections of many and of fewer rows
    cfg = small_cfg(n_heads=14, n_kv_heads=2, head_dim=128, n_layers=14)
    W = synth.weights(cfg, 0)
    model = kv.Model(cfg, None, seed=0, max_context=2048, max_rows=2048)
    doc = synth.document(6, n, cfg["vocab"])
    cache = model.prefill(doc)
    k, v = cache.read(np.arange(n))
    ref = oracle.Cache(*(np.ascontiguousarray(x.transpose(1, 0, 2, 3)) for x in (k, v)), doc.copy())
    s = n // 3
    new = synth.edit_tokens(8, doc[s:s + edit], cfg["vocab"])
    got = model.select(cache, policy, 32, s, new)
    sc, D = oracle.scores(cfg, W, ref, policy, s, new)
    sc, at = np.asarray(sc)[s + edit:n], got - s - edit
    # the 32 highest, but for scores within the rounding of the 32nd
    kth, band = np.sort(sc)[-32], TOL * np.abs(sc).max()
    assert len(got) == 32 and np.all(np.diff(got) > 0) and np.all(sc[at] >= kth - band)
    assert set(np.flatnonzero(sc > kth + band)) <= set(at.tolist())
    k1, v1 = cache.read(np.arange(n))
    assert np.array_equal(k, k1) and np.array_equal(v, v1)
    model.close()


@pytest.mark.parametrize("rows", [1, 512, 513])
def test_read_into_page_locked_memory(rows):
    # by the kernel's stores (16-byte aligned; up to 512 positions come with the
    # launch, more from device memory), and by copies (off the alignment): the same
    # rows as into pageable memory
    import torch
    cfg = small_cfg(n_heads=8, n_kv_heads=2, head_dim=64)
    model = kv.Model(cfg, None, seed=0, max_context=1024, max_rows=1024)
    cache, _ = loaded(model, cfg, 700, 3)
    P = np.sort(np.random.default_rng(rows).permutation(700)[:rows])
    want = cache.read_raw(P)
    shape, count = want[0].shape, want[0].size
    for off in (0, 4):
        buf = [torch.zeros(count + 8, dtype=torch.int16, pin_memory=True).numpy().view(np.uint16)
               for _ in range(2)]
        out = [b[off:off + count].reshape(shape) for b in buf]
        cache.read_raw(P, k_out=out[0], v_out=out[1])
        assert all(np.array_equal(o, w) for o, w in zip(out, want))
        assert all(not b[:off].any() and not b[off + count:].any() for b in buf)
    model.close()


# rows 1, 2 and 3 to a CTA, and a last CTA with one fewer; a float4, two and
# four a thread, the last ones ragged.  Layer 0's V is W_v times the norm of the
# embedding rows, here in float64; the bound is that of two fp32 sums of d terms
# relative to the largest entry (absolute sums stay below four of them).
@pytest.mark.parametrize("d", [256, 1280, 3584])
def test_norm_of_many_rows(d):
    cfg = synth.preset("tiny", n_layers=2, d_model=d, ffn=256)
    W = synth.weights(cfg, 0)
    model = kv.Model(cfg, None, seed=0, max_context=2048, max_rows=2048)
    for n in (257, 609, 1217, 1823):
        doc = synth.document(n, n, cfg["vocab"])
        x = W["embed"][doc].astype(np.float64)
        x /= np.sqrt((x * x).mean(axis=1, keepdims=True) + cfg["rms_eps"])
        want = (x * W["layers"][0]["attn_norm"]) @ W["layers"][0]["wv"].astype(np.float64).T
        _, v = model.prefill(doc).read(np.arange(n))
        err = np.abs(v[:, 0].reshape(n, -1) - want).max()
        assert err <= 8 * d * 2.0 ** -24 * np.abs(want).max(), n
    model.close()


def test_rope_rounding():
    # The rotation's rounding is part of what a cache holds (saved rows are compared
    # bit by bit): each half with one product rounded and one fused.  A document of
    # one repeated token has the same unrotated K row everywhere, and position 0
    # shows it; few rows, and the kernel of many
    # (exact sums go to fp32 through float64: a double rounding would need 29 bits
    # that happen to be a tie).
    cfg = synth.preset("tiny", n_layers=2)
    model = kv.Model(cfg, None, seed=0, max_context=1024, max_rows=512)
    half = cfg["head_dim"] // 2
    F = lambda v: Fraction(float(v))  # noqa: E731
    for n in (40, 200):
        k, _ = model.prefill(np.full(n, 17, np.int32)).read(np.arange(n))
        x = k[0, 0]
        for p in (1, 13, n - 1):
            for t in range(0, half, 5):
                a = p * cfg["rope_theta"] ** (-2.0 * t / cfg["head_dim"])
                c, s = np.float32(np.cos(a)), np.float32(np.sin(a))
                for g in range(cfg["n_kv_heads"]):
                    x1, x2 = x[g, t], x[g, t + half]
                    y1 = np.float32(float(F(x1) * F(c) - F(x2 * s)))
                    y2 = np.float32(float(F(x1) * F(s) + F(x2 * c)))
                    assert (k[p, 0, g, t], k[p, 0, g, t + half]) == (y1, y2), (n, p, t, g)
    model.close()
