"""LocalModel on batches that it does not take: an empty batch is an IndexError
before anything is launched for it (no image to take the outputs' device and
sizes from)."""
import pytest
import torch

from paper_2201_05213_gb300 import codec as CD
from paper_2201_05213_gb300 import nlc as N


class _Codec(CD.Codec):
    def __init__(self):
        self.ctx, self.cfg, self.n_weights = None, (1, 16, 0, 1, N.NLC_FP32), 8


def test_an_empty_batch_is_refused(monkeypatch):
    calls = []
    monkeypatch.setattr(N, "nlc_load_weights", lambda *a, **k: None)
    monkeypatch.setattr(N, "nlc_forward", lambda *a, **k: calls.append(a))
    monkeypatch.setattr(CD, "_raise_status", lambda *a, **k: None)
    w = torch.zeros(8, requires_grad=True)
    for shape in ((0, 4, 4, 3), (0, 0, 0, 3)):
        with pytest.raises(IndexError):
            CD.LocalModel.apply(w, _Codec(), torch.zeros(shape, dtype=torch.uint8))
    assert not calls
    CD.LocalModel.apply(w, _Codec(), torch.zeros((2, 4, 4, 3), dtype=torch.uint8))
    assert len(calls) == 1
