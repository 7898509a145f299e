"""Host side of the binning (no GPU): what becomes of the device error word."""
from types import SimpleNamespace

import pytest
import torch

from paper_2507_20239_gb300 import _abi
from paper_2507_20239_gb300 import rasterizer as R


def _stub(monkeypatch, words, count=5000):
    """R.bin_sort over stand-in buffers, whose sorts end with the given error words in turn."""
    calls = dict(sizes=[], sorts=0)

    def alloc(frame, n_records, capacity, want_keys=False):
        calls["sizes"].append(capacity)
        return SimpleNamespace(error=torch.zeros(1, dtype=torch.int32), count=torch.tensor([count]))

    def sort(proj, frame, bins, stream=None):
        bins.error |= words[calls["sorts"]]
        calls["sorts"] += 1

    monkeypatch.setattr(R, "alloc_bins", alloc)
    monkeypatch.setattr(R, "bin_sort_into", sort)
    return calls, SimpleNamespace(mean2d=torch.zeros(10, 2))


def test_bin_sort_grows_on_capacity_only(monkeypatch):
    calls, proj = _stub(monkeypatch, [2, 0])
    R.bin_sort(proj, None, capacity=100)
    assert calls == dict(sizes=[100, int(5000 * 1.1) + 1024], sorts=2)
    calls, proj = _stub(monkeypatch, [2, 2, 2])
    with pytest.raises(_abi.GsError, match="GS_ERR_CAPACITY"):
        R.bin_sort(proj, None, capacity=100)
    assert calls["sorts"] == 3


@pytest.mark.parametrize("word", [4, 6])
def test_bin_sort_raises_a_timeout_as_one(monkeypatch, word):
    calls, proj = _stub(monkeypatch, [word, 0, 0])
    with pytest.raises(_abi.GsError, match="GS_ERR_TIMEOUT") as e:
        R.bin_sort(proj, None, capacity=100)
    assert e.value.code == 4 and calls == dict(sizes=[100], sorts=1)


def test_a_callers_bins_are_kept_on_a_timeout(monkeypatch):
    calls, proj = _stub(monkeypatch, [4])
    mine = SimpleNamespace(error=torch.tensor([2], dtype=torch.int32), count=torch.tensor([7]))
    with pytest.raises(_abi.GsError, match="GS_ERR_TIMEOUT"):
        R.bin_sort(proj, None, bins=mine)
    assert calls == dict(sizes=[], sorts=1)


def test_error_words():
    assert _abi.check_error_word(0, "x") is None
    for word, code in ((2, 2), (4, 4), (6, 4), (3, 2), (1, 1)):
        with pytest.raises(_abi.GsError) as e:
            _abi.check_error_word(word, "here")
        assert e.value.code == code and "here" in str(e.value)
