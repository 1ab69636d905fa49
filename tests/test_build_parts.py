"""The library and the extension module are built apart: what the module needs is no condition for the library, and a tree without the
module still runs, by ctypes."""
import sysconfig
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


def test_without_the_module_calls_go_through_ctypes(monkeypatch, tmp_path):
    sh, budget = vec.Shape(1, 1, 4, 2, 64, vec.VECTOR_F32, 16), vec.vector_plan_budget(200, 60, 10, 16)
    q, k, s = torch.zeros(2, 2, 16, 64), torch.zeros(2, 200, 64), torch.zeros(2, 200)
    monkeypatch.setattr(B, "_marshal_module", None)
    monkeypatch.setattr(B, "marshal_path", lambda: str(tmp_path / "none.so"))
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


def test_the_module_belongs_to_one_torch_and_one_python(monkeypatch, tmp_path):
    """After a change of either the file that was there is neither fresh nor loaded."""
    here = build_module.marshal_path()
    assert torch.__version__ in here and here.endswith(sysconfig.get_config_var("EXT_SUFFIX"))
    assert build_module.build_marshal() == here
    made = []

    def compiler(args):
        made.append(args)
        raise RuntimeError("compiled again")
    monkeypatch.setattr(build_module.subprocess, "check_call", compiler)
    assert build_module.build_marshal() == here and not made
    monkeypatch.setattr(torch, "__version__", "99.0")
    with pytest.raises(RuntimeError, match="compiled again"):
        build_module.build_marshal()
    assert f"-D_GLIBCXX_USE_CXX11_ABI={int(torch.compiled_with_cxx11_abi())}" in made[0]
    monkeypatch.setattr(B, "_marshal_module", None)
    with pytest.warns(RuntimeWarning, match="torch99.0"):
        assert B._marshal().score() is None


def test_a_file_that_cannot_be_loaded(monkeypatch, tmp_path):
    (tmp_path / "no_module.so").write_bytes(b"no module")
    monkeypatch.setattr(B, "_marshal_module", None)
    monkeypatch.setattr(B, "marshal_path", lambda: str(tmp_path / "no_module.so"))
    with pytest.warns(RuntimeWarning, match="no_module.so cannot be used"):
        assert B._marshal().score() is None
