"""The autotuner times the launch that its caller will make: one batch, or a list
of batches that together are the sample."""
import types

import pytest
import torch

from paper_2510_08695_gb300 import _bpdc, autotune


@pytest.mark.parametrize("shots,batches,lists", [(10, 1, 0), (10, 3, 3), (10, 10, 10), (2, 5, 2), (1, 4, 0)])
def test_timed_launch(monkeypatch, shots, batches, lists):
    calls = []
    graph = types.SimpleNamespace(decode=lambda syn, off, out, persistent: calls.append((syn, off, out, persistent)))
    monkeypatch.setattr(_bpdc, "decode_multi", lambda items: calls.append(items))
    syn = torch.arange(shots, dtype=torch.int32)[:, None]
    out = dict(status=torch.arange(shots), corrections=syn.clone())
    autotune.launcher(graph, syn, 100, out, False, batches)()
    assert len(calls) == 1
    if lists == 0:
        assert calls[0] == (syn, 100, out, False)
        return
    items = calls[0]
    assert len(items) == lists and all(it["graph"] is graph for it in items)
    at = 0
    for it in items:
        n = it["syndromes"].shape[0]
        assert n > 0 and it["shot_offset"] == 100 + at
        for whole, part in ((syn, it["syndromes"]), (out["status"], it["out"]["status"]),
                            (out["corrections"], it["out"]["corrections"])):
            assert part.data_ptr() == whole[at:at + n].data_ptr() and part.shape[0] == n
        at += n
    assert at == shots
