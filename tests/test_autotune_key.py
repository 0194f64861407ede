"""The autotuner's cache tells apart what its choice depends on (no GPU: the key alone)."""
from types import SimpleNamespace

import pytest

from paper_1902_10432_gb300 import autotune


def _sim(prec="fp32", tau=1.0, q=19, nb=2):
    return SimpleNamespace(shape=(64, 48, 40), params=dict(prec=prec, tau=tau, q=q), q=q, nb=nb)


@pytest.mark.parametrize("other", [dict(tau=1.0000001), dict(q=27), dict(prec="fp16dev"), dict(nb=0)])
def test_key_tells_apart(other, monkeypatch):
    import torch

    monkeypatch.setattr(torch.cuda, "get_device_name", lambda: "GPU")
    # a choice made at tau = 1 exactly (the moment pass) must not be applied to a tau beside it
    assert autotune._key(_sim()) != autotune._key(_sim(**other))
    assert autotune._key(_sim(tau=1)) == autotune._key(_sim())
