"""The argument checks of the hot calls, without a GPU: empty fake tensors claim to be on a CUDA device and reach every check;
the library refuses their null addresses before it launches anything."""
import ctypes
import subprocess
import sys

import pytest
import torch
from torch._subclasses.fake_tensor import FakeTensorMode

import paper_2607_28150_b200.binding as sg

SHAPE = sg.Shape(1, 1, 8, 2, 128, 4, 16, 16, 0x1000, 16 * 2 * 128, 2 * 128, 128)
NAMES = {"k": torch.bfloat16, "v": torch.bfloat16, "sel": torch.int32, "cu": torch.int32, "pk": torch.bfloat16, "pv": torch.bfloat16}


def fake(dtype, *size):
    with FakeTensorMode():
        return torch.empty(size, device="cuda", dtype=dtype)


def pack(**wrong):
    """sg_pack_kv with empty tensors (their addresses are null), some of them replaced."""
    a = {name: fake(dtype, 0) for name, dtype in NAMES.items()}
    a.update(wrong)
    return sg.sg_pack_kv(SHAPE, a["k"], a["v"], a["sel"], a["cu"], 4, a["pk"], a["pv"], None, 0)


def test_right_types_reach_the_library():
    with pytest.raises(sg.SmartGenError) as e:
        pack()
    assert e.value.status == sg.SG_ERR_INVALID


@pytest.mark.parametrize("name", list(NAMES))
def test_wrong_arguments_are_python_errors(name):
    with pytest.raises(TypeError, match="expected dtype"):
        pack(**{name: fake(torch.float64, 0)})
    with pytest.raises(TypeError, match="CUDA tensor"):
        pack(**{name: torch.empty(0, dtype=NAMES[name])})
    with pytest.raises(TypeError, match="CUDA tensor"):
        pack(**{name: [1, 2]})
    with pytest.raises(TypeError, match="required"):
        pack(**{name: None})
    with pytest.raises(ValueError, match="contiguous"):
        pack(**{name: fake(NAMES[name], 4, 4).t()})


def test_wrong_shape_stream_and_workspace_are_python_errors():
    e, f = fake(torch.bfloat16, 0), fake(torch.float32, 0)
    with pytest.raises(TypeError):
        sg.sg_score(None, e, e, f, None, None, 0)
    with pytest.raises((TypeError, AttributeError)):
        sg.sg_score(SHAPE, e, e, f, None, None, "stream")
    with pytest.raises(TypeError):
        sg.sg_score(SHAPE, e, e, f, 17, None, 0)


@pytest.mark.parametrize("layer", [-3, 2])
def test_layer_out_of_range_is_an_index_error(layer):
    q = fake(torch.bfloat16, 2, 1, 4, 8, 128)
    with pytest.raises(IndexError):
        sg.prefill_layer(SHAPE, layer, q, q, q, q, None, q, 4, q, q, q, None, 0)


def test_layers_have_to_be_contiguous_each():
    q = fake(torch.bfloat16, 2, 4, 8, 128).transpose(1, 2)
    with pytest.raises(ValueError, match="contiguous"):
        sg.prefill_layer(SHAPE, 0, q, q, q, q, None, q, 4, q, q, q, None, 0)


def test_exceptions_of_tensor_accessors_become_python_errors():
    """In a process of its own: an exception that leaves a C function ends the process."""
    calls = [
        "sg.sg_pack_kv(s, e, e, i, i, 4, e, e)",                                               # no driver to ask for the current stream
        "sg.sg_score(s, e, e, f, torch.sparse_coo_tensor(i[None, :0], f[:0], (4,)), None, 0)",     # tensors without storage
        "torch.vmap(lambda x: sg.sg_pack_kv(s, x, x, i, i, 4, x, x, None, 0))(b)",
        "torch.vmap(lambda x: sg.prefill_layer(s, 0, x, x, x, f, None, i, 4, i, x, x, None, 0))(b)",
        "torch.vmap(lambda x: sg.sg_push_blocks(s, 4, 0, i, x, x, x, x, None, 0))(b)",
    ]
    code = ("import os\nos.environ['CUDA_VISIBLE_DEVICES'] = ''\nimport torch\n"
            "from torch._subclasses.fake_tensor import FakeTensorMode\nimport paper_2607_28150_b200.binding as sg\n"
            "with FakeTensorMode():\n    e, b = (torch.empty(n, device='cuda', dtype=torch.bfloat16) for n in ((0,), (2, 4, 4)))\n"
            "    f, i = (torch.empty(0, device='cuda', dtype=t) for t in (torch.float32, torch.int32))\n"
            "    s = sg.Shape(1, 1, 8, 2, 128, 4, 16, 16, 0x1000, 16 * 2 * 128, 2 * 128, 128)\n"
            "    for call in %r:\n        try:\n            eval(call)\n        except RuntimeError:\n            print('RuntimeError')\n" % (calls,))
    res = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True)
    assert res.returncode == 0 and res.stdout.split() == ["RuntimeError"] * len(calls), res.stderr[-2000:]


@pytest.mark.parametrize("stream", [0, ctypes.c_void_p(0), ctypes.c_void_p(None), type("S", (), {"cuda_stream": 0})(), type("S", (), {"cuda_stream": None})()])
def test_forms_of_a_stream_handle(stream):
    e = fake(torch.bfloat16, 0)
    with pytest.raises(sg.SmartGenError):                 # the arguments are taken; the library refuses the null addresses
        sg.sg_score(SHAPE, e, e, fake(torch.float32, 0), None, None, stream)


@pytest.mark.parametrize("layer", [0, 1, -1])
def test_a_layer_out_of_a_sequence_of_tensors(layer):
    e, f, i = ([fake(t, 0), fake(t, 0)] for t in (torch.bfloat16, torch.float32, torch.int32))
    with pytest.raises(sg.SmartGenError):
        sg.prefill_layer(SHAPE, layer, e, tuple(e), {layer: e[0]}, f, None, i[0], 4, i, e, e, None, 0)
    with pytest.raises(IndexError):
        sg.prefill_layer(SHAPE, 2, e, e, e, f, None, i[0], 4, i, e, e, None, 0)
    with pytest.raises(TypeError, match="CUDA tensor"):
        sg.prefill_layer(SHAPE, layer, e, [1, 2], e, f, None, i[0], 4, i, e, e, None, 0)
    with pytest.raises(TypeError):
        sg.prefill_layer(SHAPE, layer, e, 17, e, f, None, i[0], 4, i, e, e, None, 0)


def test_module_built_against_another_torch_is_rebuilt_and_not_imported(monkeypatch):
    from paper_2607_28150_b200 import build
    assert sg._native.BUILT_FOR == build.native_stamp() and build.native_is_current()
    monkeypatch.setattr(torch, "__version__", "0.0.1")
    assert not build.native_is_current()
    code = ("import torch\ntorch.__version__ = '0.0.1'\ntry:\n    import paper_2607_28150_b200.binding\n"
            "except ImportError as e:\n    print(e)\n")
    res = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True)
    assert "does not fit this torch" in res.stdout and "torch 0.0.1" in res.stdout, res.stderr[-2000:]
