"""What the Python binding takes and refuses, through the CPython module and through ctypes where that module is missing: the same
arguments, the same statuses, the same exceptions.  Host side only: every call fails its host checks before a launch."""
import ctypes

import numpy as np
import pytest
import torch

import paper_2210_00129_b200 as sbp
from paper_2210_00129_b200 import build as sbp_build

FAKE = 0x1000          # never dereferenced


@pytest.fixture(params=["module", "ctypes"])
def calls(request, monkeypatch, tmp_path):
    sbp_build.build()
    monkeypatch.setattr(sbp, "_call", None)
    if request.param == "ctypes":
        monkeypatch.setattr(sbp, "CALLS_PATH", str(tmp_path / "_calls.so"))
    return request.param


def _sample(mode=0, B=2, H=4, ratio=0.5, rows=FAKE, step=2 ** 32):       # (a step of 2^32 is refused by the library)
    return sbp.sbp_sample_keep(mode, B, H, 4, ratio, 0, step, 0, 0, rows, FAKE, stream=0, check=False)


def test_the_expected_path_is_taken(calls):
    _sample()
    assert isinstance(sbp._call, sbp._CtypesCalls) == (calls == "ctypes")


def test_accepted(calls):
    t = torch.zeros(8, dtype=torch.int32)
    for call in (_sample, lambda: _sample(mode=True), lambda: _sample(ratio="0.5"), lambda: _sample(ratio=np.float32(0.5)),
                 lambda: _sample(ratio=torch.tensor(0.5)), lambda: _sample(ratio=1), lambda: _sample(B=np.int64(2)),
                 lambda: _sample(B=torch.tensor(2)), lambda: _sample(rows=t), lambda: _sample(rows=None)):
        assert call() == sbp.SBP_ERR_INVALID_ARG
    assert _sample(mode=1, ratio="0.6", step=0) == sbp.SBP_ERR_UNSUPPORTED


@pytest.mark.parametrize("bad", [2.0, "2", None, np.float64(2), torch.tensor(2.0)])
def test_sizes_are_whole_numbers(calls, bad):
    with pytest.raises(ctypes.ArgumentError):
        _sample(B=bad)
    with pytest.raises(ctypes.ArgumentError):
        _sample(step=bad)


def test_refused_pointers_and_ratios(calls):
    with pytest.raises(AttributeError):
        _sample(rows="0x1000")
    with pytest.raises(AttributeError):
        _sample(rows=np.zeros(4, dtype=np.int32))
    with pytest.raises(ValueError):
        _sample(ratio="half")
    with pytest.raises(TypeError):
        _sample(ratio=None)


def test_build_without_python_headers(monkeypatch, tmp_path):
    """Only the library is wanted then, and the calls go through ctypes."""
    sbp_build.build()
    monkeypatch.setattr(sbp_build, "CALLS_PATH", str(tmp_path / "_calls.so"))
    monkeypatch.setattr(sbp_build.sysconfig, "get_paths", lambda: {"include": str(tmp_path)})
    assert sbp_build.build() == sbp_build.LIB_PATH
    assert not (tmp_path / "_calls.so").exists()
