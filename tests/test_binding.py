"""Argument checks of the Python entry points (made before any CUDA call, so they run without a GPU)."""
import pytest
import torch

import paper_2608_13076_gb300 as spade
from paper_2608_13076_gb300 import _build


@pytest.fixture(scope="module", autouse=True)
def library():
    spade.build()


def test_extension_is_rebuilt_for_another_torch(monkeypatch):
    assert _build.up_to_date()
    monkeypatch.setattr(torch, "__version__", "0.0.0")
    assert not _build.up_to_date()


def _args():
    b = lambda *s: torch.zeros(s, dtype=torch.bfloat16)
    i = lambda n: torch.zeros(n, dtype=torch.int32)
    return dict(k_cache=b(1, 1, 8, 64), v_cache=b(1, 1, 8, 64), ctx_lens=i(1), accepted_len=i(1), n_draft=i(1),
                status=i(1))


@pytest.mark.parametrize("name,value,error,text", [
    ("k_cache", None, ValueError, "k_cache is required"),
    ("k_cache", torch.zeros(1, 1, 8, 64), TypeError, "k_cache must be torch.bfloat16, got torch.float32"),
    ("k_cache", torch.zeros(1, 1, 8, 64, dtype=torch.bfloat16), ValueError, "k_cache must be a CUDA tensor"),
    ("k_cache", 3, AttributeError, "dtype"),
])
def test_tensor_checks(name, value, error, text):
    args = {**_args(), name: value}
    status = args.pop("status")
    with pytest.raises(error, match=text):
        spade.spade_kv_commit(*args.values(), status=status)
