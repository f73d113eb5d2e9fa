"""The upload of a call's small arrays where it can go wrong: array lengths
around one CTA's share (1024 words), more segments than one launch takes (128),
and the staging buffer starting over between calls.  Layer-0 K/V depend on a
row's token and position alone, so they show which tokens and positions the
device has: against a fresh prefill of the edited document, within fp32
rounding of sums in another order (another token's entry differs by O(1))."""
import numpy as np
import pytest

from paper_2609_17983_gb300 import synth

try:
    from paper_2609_17983_gb300 import kvrepair as kv
except ImportError as _e:  # pragma: no cover
    kv, _IMPORT_ERROR = None, _e

pytestmark = pytest.mark.gpu


def check_layer0(model, caches, docs, d):
    for cache, doc in zip(caches, docs):
        fresh = model.prefill(doc)
        pos = np.arange(len(doc))
        for got, want in zip(cache.read(pos), fresh.read(pos)):
            # two sums of d products; their absolute sum is below 4 largest entries
            bound = 8 * d * 2.0 ** -24 * np.abs(want[:, 0]).max()
            assert np.abs(got[:, 0] - want[:, 0]).max() <= bound
        fresh.close()


@pytest.mark.parametrize("lengths,edits", [((1023, 1024, 1025, 2049), 1), ((300, 257), 100),
                                           ((64,) * 32, 4)])
def test_uploads_reach_every_document(lengths, edits):
    cfg = synth.preset("tiny", n_layers=2)
    model = kv.Model(cfg, None, seed=0, max_context=4096, max_rows=1024)
    rng = np.random.default_rng(5)
    docs = [synth.document(3 + i, n, cfg["vocab"]) for i, n in enumerate(lengths)]
    caches = [model.prefill(d) for d in docs]
    for _ in range(6):  # about 20 K words staged: the buffer starts over
        reqs = []
        for doc, cache in zip(docs, caches):
            at = np.sort(rng.permutation(len(doc) // 2)[:edits]) * 2
            new = [np.array([(doc[a] + 1 + rng.integers(500)) % cfg["vocab"]], np.int32) for a in at]
            for a, t in zip(at, new):
                doc[a] = t[0]
            reqs.append((cache, [(int(a), t) for a, t in zip(at, new)], np.zeros(0, np.int32)))
        model.repair_batch(reqs)
    check_layer0(model, caches, docs, cfg["d_model"])
    model.close()


def test_single_repairs_reach_the_device_in_order():
    cfg = synth.preset("tiny", n_layers=2)
    model = kv.Model(cfg, None, seed=0, max_context=2048, max_rows=256)
    doc = synth.document(9, 1500, cfg["vocab"])
    cache = model.prefill(doc)
    for i in range(60):  # the same and neighbouring spans, again and again
        s, new = 700 + i % 3, np.arange(4, dtype=np.int32) + 11 * i
        cache.repair(new, s, np.arange(s + 4, s + 4 + i % 130))
        doc[s:s + 4] = new
    check_layer0(model, [cache], [doc], cfg["d_model"])
    model.close()


@pytest.mark.parametrize("read", [False, True])
def test_every_pass_of_a_document_runs_once(read):
    # the second pass of a row count is captured behind its own launches: it runs
    # once (its edit lands, its launches count once), as the first and the replays
    import torch
    cfg = synth.preset("tiny", n_layers=9)
    model = kv.Model(cfg, None, seed=0, max_context=2048, max_rows=256)
    stream = torch.cuda.Stream()
    model.set_stream(stream.cuda_stream)
    doc = synth.document(9, 300, cfg["vocab"])
    cache = model.prefill(doc)
    used = []
    for i in range(5):
        new, A = np.arange(4, dtype=np.int32) + 11 * i, np.arange(104, 130 - i % 2)
        l0 = model.launches()
        rows = cache.repair_read(new, 100, A) if read else cache.repair(new, 100, A)
        used.append(model.launches() - l0)
        doc[100:104] = new
        check_layer0(model, [cache], [doc], cfg["d_model"])
        if read:
            assert np.array_equal(rows[0], cache.read_raw(np.arange(100, 130 - i % 2))[0])
    assert len(set(used)) == 1
    model.close()


@pytest.mark.parametrize("dtype", ["bf16", "fp32"])
def test_rows_read_into_page_locked_memory(dtype):
    # the positions that a launch's arguments hold (512), one fewer and more, in
    # any order and with repeats: exactly what pageable arrays get
    import torch
    cfg = synth.preset("tiny", n_layers=3, dtype=dtype)
    model = kv.Model(cfg, None, seed=0, max_context=2048, max_rows=1024)
    cache = model.prefill(synth.document(4, 1700, cfg["vocab"]))
    for n in (511, 512, 513, 2300):
        pos = np.random.default_rng(n).integers(0, 1700, n).astype(np.int32)
        want = cache.read_raw(pos)
        t = torch.int16 if dtype == "bf16" else torch.float32
        got = [torch.zeros(want[0].shape, dtype=t, pin_memory=True).numpy().view(want[0].dtype)
               for _ in range(2)]
        cache.read_raw(pos, k_out=got[0], v_out=got[1])
        assert np.array_equal(got[0], want[0]) and np.array_equal(got[1], want[1]), n
    model.close()
