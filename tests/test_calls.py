"""The module that makes the plain calls of the sampling entry points: what it takes, what it leaves to binding.py, and what it
passes on.  Stand-ins with null addresses for the tensors, so that the library answers without a GPU."""
import sysconfig

import pytest
import torch

import __graft_entry__ as entry
from paper_2211_17192_b200 import binding, build


class StandIn:
    is_cuda = True

    def __init__(self, shape, dtype, contiguous=True):
        self.shape, self.dtype, self.contiguous = torch.Size(shape), dtype, contiguous

    def is_contiguous(self):
        return self.contiguous

    def data_ptr(self):
        return 0

    def numel(self):
        return 0


def plain():
    f, i, u = torch.float32, torch.int32, torch.uint8
    return [StandIn((4, 4, 100), f), StandIn((4, 3, 100), f), StandIn((4, 3), i), StandIn((4, 4), f), StandIn((4,), i), StandIn((4,), i),
            StandIn((9,), u)]


@pytest.fixture(scope="module")
def calls():
    entry.build()
    binding.lib()
    return binding._calls


def test_plain_calls_reach_the_library(calls):
    assert calls.verify(*plain(), 1.0, 1.0, 0, 1.0, 0) == -1 and b"null pointer" in binding.lib().spec_last_error()
    assert calls.verify(*plain(), -1, 1.0, 0, 1.0, 0) == -1 and b"temperature" in binding.lib().spec_last_error()
    assert calls.verify(*plain(), 1.0, 2.0, 0, 1.0, 0) == -1 and b"lenience" in binding.lib().spec_last_error()
    assert calls.verify(*plain(), 1.0, 1.0, -3, 1.0, 0) == -1 and b"top_k" in binding.lib().spec_last_error()
    assert calls.sample(StandIn((3, 0), torch.float32), plain()[3], 1.0, plain()[4], 0) == -1


@pytest.mark.parametrize("change", [
    (0, None), (1, None), (2, torch.zeros(4, 3, dtype=torch.int32)), (0, StandIn((4, 4, 100), torch.bfloat16)), (0, StandIn((4, 400), torch.float32)),
    (1, StandIn((4, 4, 100), torch.float32)), (2, StandIn((4, 3), torch.int64)), (2, StandIn((3, 3), torch.int32)), (3, StandIn((4, 3), torch.float32)),
    (4, StandIn((4,), torch.int32, contiguous=False)), (6, StandIn((9,), torch.int8)),
])
def test_anything_else_is_left_to_the_binding(calls, change):
    args = plain()
    args[change[0]] = change[1]
    assert calls.verify(*args, 1.0, 1.0, 0, 1.0, 0) is None
    if change[0] in (0, 3, 4):
        args = [StandIn((4, 100), torch.float32), plain()[3], 1.0, plain()[4], 0]
        args[{0: 0, 3: 1, 4: 3}[change[0]]] = StandIn((4, 4, 4), torch.float64)
        assert calls.sample(*args) is None


def test_numbers_that_are_not_numbers_are_left_to_the_binding(calls):
    assert calls.verify(*plain(), "1", 1.0, 0, 1.0, 0) is None
    assert calls.verify(*plain(), 1.0, 1.0, 0.5, 1.0, 0) is None
    assert calls.verify(*plain(), 1.0, 1.0, 0, None, 0) is None
    assert calls.verify(*plain(), 1.0, 1.0, 1 << 40, 1.0, 0) is None
    assert calls.verify(*plain()) is None


def test_a_tensor_that_is_not_on_a_gpu_is_named(calls):
    """Also on a machine without one: nothing asks for a stream before the tensors have been looked at."""
    f, i, u = torch.float32, torch.int32, torch.uint8
    host = [torch.zeros(2, 3, 8, dtype=f), torch.zeros(2, 2, 8, dtype=f), torch.zeros(2, 2, dtype=i), torch.zeros(2, 3, dtype=f)]
    with pytest.raises(ValueError, match="target_logits must be a CUDA tensor"):
        binding.spec_verify_sample(*host, 1.0, n_accepted=torch.zeros(2, dtype=i), next_token=torch.zeros(2, dtype=i), workspace=torch.zeros(64, dtype=u))
    with pytest.raises(ValueError, match="logits must be a CUDA tensor"):
        binding.spec_sample(host[0][0], torch.zeros(3, dtype=f), 1.0, tokens=torch.zeros(3, dtype=i))


@pytest.mark.parametrize("built", [True, False])
def test_without_the_module_the_binding_makes_the_calls(calls, monkeypatch, built):
    monkeypatch.setattr(binding, "_calls", calls if built else None)
    monkeypatch.setattr(binding, "_stream", lambda: 0)
    t = plain()
    with pytest.raises(binding.SpecError, match="null pointer"):
        binding.spec_verify_sample(*t[:4], 1.0, n_accepted=t[4], next_token=t[5], workspace=t[6])
    with pytest.raises(binding.SpecError):
        binding.spec_sample(StandIn((3, 0), torch.float32), t[3], 1.0, tokens=t[4])


def test_the_module_belongs_to_one_interpreter(calls):
    assert build.CALLS_PATH == binding._CALLS_PATH and build.CALLS_PATH.endswith("_calls" + sysconfig.get_config_var("EXT_SUFFIX"))


def test_a_machine_without_a_compiler_or_headers_does_without_the_module(tmp_path, monkeypatch, capsys):
    at = tmp_path / "_calls.so"
    monkeypatch.setattr(build, "CALLS_PATH", str(at))
    monkeypatch.setattr(build, "LIB_DIR", str(tmp_path))
    assert build.build_calls() == str(at) and build.build_calls() == str(at)
    with monkeypatch.context() as m:
        m.setattr(build.sysconfig, "get_paths", lambda: {"include": str(tmp_path)})
        assert build.build_calls() is None and not at.exists() and "calls.c is not built" in capsys.readouterr().err
    assert build.build_calls() == str(at)
    monkeypatch.setattr(build.shutil, "which", lambda name: None)
    assert build.build_calls() == str(at) and build.build_calls(force=True) is None and not at.exists()
