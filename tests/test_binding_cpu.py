"""The native marshalling of hgf.linear_forward (csrc/hgf_python.cpp), without a GPU: what it takes and refuses before any launch."""
import numpy as np
import pytest
import torch

from paper_2602_05269_b200 import build as hgf_build


@pytest.fixture(scope="module")
def call():
    hgf_build.build()
    from paper_2602_05269_b200 import hgf
    hgf.lib()
    return hgf._native_forward


class Stream:
    cuda_stream = 0


class Array:
    """Not a tensor, but with a tensor's methods, as the ctypes calls take it too."""
    def __init__(self, shape, address):
        self.shape, self.address = shape, address

    def data_ptr(self):
        return self.address

    def numel(self):
        n = 1
        for v in self.shape:
            n *= v
        return n


def arguments(**changed):
    x = torch.zeros(4, 64, dtype=torch.bfloat16)
    a = {"x": x, "packed": x, "gamma": 0.5, "d_in": 64, "d_out": 64, "At": None, "Bt": None, "gate": None, "y": x, "workspace": Array((16,), 4096),
         "flags": 0, "stream": Stream(), "ln_weight": None, "ln_bias": None, "eps": 1e-5, "gate_group": None}
    assert not set(changed) - set(a)
    return list({**a, **changed}.values())


# the status that hgf.h gives for each, found before the library touches a device
@pytest.mark.parametrize("changed,status", [
    ({"x": Array((4, 64), 0)}, 1), ({"packed": None}, 1), ({"y": None}, 1), ({"d_in": 0}, 1), ({"d_out": -1}, 1), ({"flags": 1 << 20}, 1),
    ({"d_in": 96}, 2), ({"x": Array((1 << 23, 64), 4096)}, 2), ({"At": Array((17, 64), 4096), "Bt": Array((64, 17), 4096), "gate": Array((64,), 4096)}, 2),
    ({"y": Array((4, 64), 4104)}, 3), ({"workspace": Array((16,), 4096)}, 4), ({"workspace": None}, None),
    ({"workspace": Array((1 << 24,), 4096), "ln_weight": Array((64,), 4096)}, 1), ({"workspace": Array((1 << 24,), 4096), "gate_group": 24}, 2),
    ({"workspace": Array((1 << 24,), 4096 + 128)}, 3),
])
def test_status_of_refused_calls(call, changed, status):
    if status is None:
        with pytest.raises(AttributeError):
            call(*arguments(**changed))
    else:
        assert call(*arguments(**changed)) == status


@pytest.mark.parametrize("changed", [{"d_in": 64.0}, {"gamma": "one"}, {"flags": None}, {"gate_group": 2.5}, {"x": 7}, {"stream": 7}])
def test_arguments_of_another_type_raise(call, changed):
    with pytest.raises((TypeError, AttributeError)):
        call(*arguments(**changed))


def test_wrong_number_of_arguments(call):
    with pytest.raises(TypeError):
        call(*arguments()[:-1])


# ---- the module is a way for the arguments only: without it, and for arguments that are not plain, the calls are what they are through ctypes -----------------
class Tensor(Array):
    """As much of a CUDA tensor as hgf.linear_forward looks at."""
    is_cuda, dtype, device = True, torch.bfloat16, "meta"

    def is_contiguous(self):
        return True


def outcome(hgf, **changed):
    a = {"x": Tensor((4, 64), 4096), "packed": Tensor((1,), 4096), "gamma": 0.5, "d_in": 64, "d_out": 64, "y": Tensor((4, 64), 4096), "workspace": Tensor((16,), 4096),
         "stream": Stream()}
    try:
        hgf.linear_forward(**{**a, **changed})
    except Exception as e:  # noqa: BLE001
        return type(e), getattr(e, "status", None)


class Index:
    def __index__(self):
        return 64


class Float:
    def __float__(self):
        return 0.5


# (all with a status or an exception: nothing gets as far as a device)
FORMS = [{}, {"x": Tensor((4, 64), 0)}, {"d_in": 96}, {"d_in": True}, {"d_in": np.int64(64)}, {"d_out": np.int32(64)}, {"d_in": 64.0}, {"d_in": Index()}, {"d_in": 2 ** 64 + 64},
         {"d_in": -64}, {"flags": np.uint32(0)}, {"flags": 2 ** 32}, {"flags": 1 << 20}, {"flags": True}, {"gamma": np.float32(0.5)}, {"gamma": 1}, {"gamma": Float()},
         {"gamma": "one"}, {"gamma": None}, {"gamma": torch.tensor(0.5)}, {"x": Tensor((np.int64(4), 64), 4096)}, {"x": Tensor((4, 64), np.int64(4096))},
         {"x": Tensor((4, 64), None)}, {"packed": Tensor((1,), 4096.0)}, {"workspace": Tensor((np.int64(16),), 4096)}, {"stream": type("S", (), {"cuda_stream": None})()},
         {"stream": type("S", (), {"cuda_stream": "0"})()}, {"stream": 7}, {"At": Tensor((16, 64), 4096)}, {"At": [1]}, {"gate_group": 24}, {"gate_group": "24"}, {"gate_group": "x"},
         {"gate_group": 2.5}, {"gate_group": 0}, {"ln_weight": Tensor((64,), 4096)}, {"ln_weight": Tensor((64,), 4096), "ln_bias": Tensor((64,), 4096), "eps": "1e-5"},
         {"ln_weight": Tensor((64,), 4096), "ln_bias": Tensor((64,), 4096), "eps": None}, {"eps": None}, {"ln_bias": 3}, {"ln_bias": Tensor((64,), 4096)}]


@pytest.mark.parametrize("changed", FORMS, ids=[str(i) for i in range(len(FORMS))])
def test_the_same_calls_are_taken_and_refused_as_through_ctypes(call, monkeypatch, changed):
    from paper_2602_05269_b200 import hgf
    got = outcome(hgf, **changed)
    monkeypatch.setattr(hgf, "_native_forward", None)
    assert got == outcome(hgf, **changed) and got is not None


def test_the_library_works_without_the_module(monkeypatch, tmp_path):
    from paper_2602_05269_b200 import hgf
    hgf_build.build()
    monkeypatch.setattr(hgf_build, "module_path", lambda: str(tmp_path / "missing.so"))
    monkeypatch.setattr(hgf, "_lib", None)
    monkeypatch.setattr(hgf, "_native_forward", None)
    with pytest.warns(RuntimeWarning, match="paper_2602_05269_b200.build"):
        hgf.lib()
    assert hgf.packed_bytes(64, 256) == 4 * 1024 and hgf.workspace_bytes(4, 64, 64, 0) > 0
    assert outcome(hgf) == (hgf.HgfError, 4)


def test_another_torch_or_python_has_a_module_of_its_own(monkeypatch):
    hgf_build.build()
    compiled = []

    class Done:
        returncode, stdout, stderr = 0, "", ""

    def run(cmd, **_):
        compiled.append(cmd)
        return Done()
    monkeypatch.setattr(hgf_build.subprocess, "run", run)
    monkeypatch.setattr(hgf_build.os, "replace", lambda a, b: None)
    hgf_build.build()
    assert not compiled
    monkeypatch.setattr(torch, "__version__", "1.2.3")
    hgf_build.build()
    assert [c[0] for c in compiled] == ["g++"] and "1.2.3" in compiled[0][compiled[0].index("-o") + 1]
    monkeypatch.undo()
    monkeypatch.setattr(hgf_build.subprocess, "run", run)
    monkeypatch.setattr(hgf_build.os, "replace", lambda a, b: None)
    tag = hgf_build.sysconfig.get_config_var("SOABI")
    monkeypatch.setattr(hgf_build.sysconfig, "get_config_var", lambda name: "cpython-399" if name == "SOABI" else tag)
    hgf_build.build()
    assert len(compiled) == 2 and "cpython-399" in compiled[1][compiled[1].index("-o") + 1]
    Done.returncode = 1
    with pytest.raises(RuntimeError, match=r"g\+\+ failed"):
        hgf_build.build()
