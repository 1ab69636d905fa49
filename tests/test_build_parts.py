"""The library and the extension module are built apart: what the module needs is no condition for the library, and a tree without the
module still runs, by ctypes."""
import sys
import warnings

import pytest
import torch

import paper_2605_23258_b200 as vec
from paper_2605_23258_b200 import binding as B
from paper_2605_23258_b200 import build as build_module
from paper_2605_23258_b200.pipeline import Compressor


def test_the_library_is_built_first_and_without_the_module(monkeypatch):
    order = []

    def no_compiler(force=False):
        order.append("module")
        raise FileNotFoundError("g++")
    monkeypatch.setattr(build_module, "_stale", lambda: order.append("library") or False)
    monkeypatch.setattr(build_module, "build_marshal", no_compiler)
    with pytest.warns(RuntimeWarning, match="g\\+\\+.*ctypes"):
        assert build_module.build() == build_module.LIB
    assert order == ["library", "module"]


def test_without_the_module_calls_go_through_ctypes(monkeypatch):
    sh, budget = vec.Shape(1, 1, 4, 2, 64, vec.VECTOR_F32, 16), vec.vector_plan_budget(200, 60, 10, 16)
    q, k, s = torch.zeros(2, 2, 16, 64), torch.zeros(2, 200, 64), torch.zeros(2, 200)
    monkeypatch.setattr(B, "_marshal_module", None)
    monkeypatch.setitem(sys.modules, "paper_2605_23258_b200._marshal", None)
    monkeypatch.delattr(vec, "_marshal", raising=False)
    with pytest.warns(RuntimeWarning, match="python -m paper_2605_23258_b200.build"):
        with pytest.raises(ValueError, match="must be a CUDA tensor"):
            vec.vector_score(sh, q, k, 200, s)
    with warnings.catch_warnings():
        warnings.simplefilter("error")                                  # said once
        with pytest.raises(vec.VectorError) as e:
            vec.vector_score(sh, None, None, 200, None, None, None, 0)
        assert e.value.status == -1
        c = Compressor(sh, budget, extra_rows=1, device="cpu")
        c.append(k[:, 0], k[:, 1], 3)
        assert c.cache.n_ret == budget.n_ret + 1
