"""The grouping of a batch (host side) and the tuning cache that is keyed by it: an
entry timed on another grouping of the same instances is not restored."""
import hashlib
import json

import pytest

from paper_1808_04473_gb300 import build as fbuild
from paper_1808_04473_gb300 import ffeq, tuning


@pytest.fixture(scope="module", autouse=True)
def lib():
    fbuild.build()
    return ffeq.lib()


def _batch(n, sizes=((64, 8, 2), (128, 16, 4), (256, 31, 8)), precision=ffeq.BF16X3):
    cfg, inst = ffeq.pack_batch([(*sizes[i % len(sizes)], 1, 7, 0.5, 1.0) for i in range(n)], arch=ffeq.FD,
                                precision=precision)
    return ffeq.ffeq_batch_create(cfg, inst)


def test_layout_of_few_and_many_units():
    few, many = (ffeq.ffeq_batch_group_layout(_batch(n)) for n in (30, 600))
    assert [g[0] for g in few] == [8, 16, 32] and all(g[1] == 1 for g in few)
    assert {g[1] for g in many} == {2} and sum(g[3] for g in many) == 600
    assert all(g[1] == 1 for g in ffeq.ffeq_batch_group_layout(_batch(600, precision=ffeq.FP16X3)))
    assert ffeq.lib().ffeq_batch_group_layout(None, None, 0) == 1


def test_entry_of_another_grouping_is_not_restored(tmp_path, monkeypatch):
    batch, path = _batch(600), str(tmp_path / "cache.json")
    c = batch.config
    shapes = sorted((i.B, i.U, i.C, i.n_sc, i.n_sym) for i in batch.instances)
    old = [list(t) for t in ffeq.ffeq_batch_get_tuning(batch)]
    kept = [[t[0], 1, *t[2:]] for t in old]
    # As stored before the grouping was part of the key, and by a library that groups them otherwise.
    text = json.dumps(["GPU", c.arch, c.precision, c.estimate, c.llr_bits, c.equalizer, c.lama_iters, shapes])
    entries = {hashlib.sha256(text.encode()).hexdigest()[:32]: kept}
    layout = ffeq.ffeq_batch_group_layout(batch)
    monkeypatch.setattr(ffeq, "ffeq_batch_group_layout", lambda b: [(g[0], 1, *g[2:]) for g in layout])
    entries[tuning.batch_key(batch, "GPU")] = kept
    monkeypatch.undo()
    json.dump(entries, open(path, "w"))
    timed = []
    monkeypatch.setattr(ffeq, "ffeq_batch_autotune", lambda *a, **k: timed.append(1))
    t, cached = tuning.autotune_cached(batch, None, None, None, None, path=path, device_name="GPU")
    assert not cached and timed == [1] and [list(v) for v in t] == old
    t, cached = tuning.autotune_cached(batch, None, None, None, None, path=path, device_name="GPU")
    assert cached and timed == [1]
