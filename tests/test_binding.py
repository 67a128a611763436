"""The C++ marshalling of the Python calls, without a GPU: fake tensors on a CUDA device and recorded calls in the library's place."""
import ctypes
import os
import shutil
import subprocess
import sys
import weakref

import pytest
import torch
from torch._subclasses.fake_tensor import FakeTensorMode

import paper_2506_22694_b200 as vt
from paper_2506_22694_b200 import build as vt_build

pytestmark = pytest.mark.filterwarnings("ignore:Accessing the data pointer of FakeTensor")
I32, F32, BF16 = torch.int32, torch.float32, torch.bfloat16


class Space:
    """A workspace as the binding looks at it."""
    ptr, nbytes = 4096, 1 << 20


@pytest.fixture
def calls():
    """The binding bound to functions that record their calls; the library's own again afterwards."""
    lib, made, keep = vt.lib(), [], []

    def recorder(name):
        types = getattr(lib, name).argtypes

        def record(*args):
            made.append((name, args))
            return 0
        keep.append(ctypes.CFUNCTYPE(ctypes.c_int, *types)(record))
        return ctypes.cast(keep[-1], ctypes.c_void_p).value

    vt._bind.use({name: recorder(name) for name in vt._BOUND}, lambda *a: Space(), lambda device: 77, lambda: 0)
    with FakeTensorMode():
        yield made
    vt._lib = None                                          # (the next call registers the library's functions)
    vt.lib()


def _t(shape, dtype, device="cuda"):
    return torch.empty(shape, dtype=dtype, device=device)


def _cases():
    """name -> (call, its tensor arguments by name)"""
    head = lambda: dict(h=_t((4, 64), BF16), W=_t((100, 64), BF16), map=_t(100, I32), temp=_t(4, F32), u=_t((4, 100), F32), ids=_t((4, 9), I32), lps=_t((4, 9), F32))
    pool = lambda: dict(token=_t(64, I32), parent=_t(64, I32), score=_t(64, F32))
    return {
        "head": (lambda a: vt.vt_draft_head(a["h"], a["W"], a["map"], a["temp"], 8, a["u"], ws=Space(), out=(a["ids"], a["lps"])), head),
        "expand": (lambda a: vt.vt_draft_head_expand(a["h"], a["W"], a["map"], a["temp"], 8, a["u"], a["frontier"], (a["token"], a["parent"], a["score"]),
                                                     0, 8, ws=Space(), out=(a["ids"], a["lps"])), lambda: dict(head(), **pool(), frontier=_t(4, I32))),
        "rerank": (lambda a: vt.vt_tree_rerank([a["token"], a["parent"], a["score"]], 64, 32), pool),
        "verify": (lambda a: vt.vt_verify_greedy(a["token"], a["parent"], a["target"], a["total"]),
                   lambda: dict(token=_t((2, 7), I32), parent=_t((2, 7), I32), target=_t((2, 8), I32), total=_t(1, torch.int64))),
        "build": (lambda a: vt.vt_build_vocab(a["ids"], 100, 50, ws=Space()), lambda: dict(ids=_t(1000, I32))),
        "trim": (lambda a: vt.vt_trim_head(a["full"], a["map"], a["trim"]), lambda: dict(full=_t((100, 64), BF16), map=_t(50, I32), trim=_t((50, 64), BF16))),
    }


NAMES = ["head", "expand", "rerank", "verify", "build", "trim"]


@pytest.mark.parametrize("name", NAMES)
def test_a_call_goes_through_once_on_the_current_stream(calls, name):
    call, args = _cases()[name]
    call(args())
    assert len(calls) == 1 and 77 in calls[0][1][-1:]


@pytest.mark.parametrize("name", NAMES)
def test_a_data_pointer_that_raises_is_an_exception(calls, name):
    """Not a crash: it used to be asked for where the interpreter's lock had been given up."""
    call, args = _cases()[name]
    for arg in args():
        a = args()
        torch._C._set_throw_on_mutable_data_ptr(a[arg])
        with pytest.raises(RuntimeError, match="data pointer"):
            call(a)
    assert not calls


@pytest.mark.parametrize("name", NAMES)
def test_wrong_types_devices_and_strides_are_refused(calls, name):
    call, args = _cases()[name]
    for arg, t in args().items():
        if arg in ("lps",) or (arg == "ids" and name != "build"):      # (the caller's outputs are taken as they are)
            continue
        wide = _t(t.shape[:-1] + (2 * t.shape[-1],), t.dtype)[..., ::2]
        for bad in (_t(t.shape, torch.float16), _t(t.shape, t.dtype, "cpu"), wide):
            a = args()
            a[arg] = bad
            if name == "build" and not bad.is_cuda:                    # (host ids: the call that streams them)
                continue
            if bad is wide and t.shape[-1] == 1:
                continue
            with pytest.raises(TypeError, match="must be a contiguous CUDA tensor of dtype"):
                call(a)
        a = args()
        a[arg] = [1, 2]
        with pytest.raises(AttributeError):
            call(a)
    assert not calls


@pytest.mark.parametrize("name,arg,shape", [
    ("head", "h", (4, 72)), ("head", "h", (4, 8, 8)), ("head", "map", 99), ("head", "temp", 5), ("head", "u", (4, 99)), ("head", "u", 400),
    ("expand", "frontier", 3), ("rerank", "score", 63), ("verify", "target", (2, 7)), ("verify", "parent", (1, 7)), ("verify", "token", 14),
    ("trim", "full", 6400),
])
def test_wrong_shapes_are_refused(calls, name, arg, shape):
    call, args = _cases()[name]
    a = args()
    a[arg] = _t(shape, a[arg].dtype)
    with pytest.raises(ValueError):
        call(a)
    assert not calls


@pytest.mark.parametrize("parts", [0, 1, 2, 4])
def test_a_pool_or_outputs_of_another_number_of_parts_are_refused(calls, parts):
    with pytest.raises(ValueError):
        vt.vt_tree_rerank([_t(64, I32)] * parts, 8, 8)
    a = _cases()["head"][1]()
    if parts != 2:
        with pytest.raises(ValueError):
            vt.vt_draft_head(a["h"], a["W"], None, a["temp"], 8, ws=Space(), out=[a["ids"]] * parts)
    assert not calls


def test_a_pool_given_as_a_list_is_kept_while_the_call_runs(calls):
    a = _cases()["expand"][1]()
    pool = [a.pop("token"), a.pop("parent"), a.pop("score")]
    refs, alive = [weakref.ref(t) for t in pool], []

    class Emptying(Space):
        @property
        def ptr(self):                                      # runs in the middle of the call, as another thread may
            pool.clear()
            alive.append([r() is not None for r in refs])
            return 4096

    vt.vt_draft_head_expand(a["h"], a["W"], a["map"], a["temp"], 8, a["u"], None, pool, 0, 8, ws=Emptying(), out=(a["ids"], a["lps"]))
    assert alive == [[True] * 3] and len(calls) == 1


def test_a_module_for_another_torch_is_built_anew(monkeypatch, tmp_path):
    copy = str(tmp_path / "_vt_bind.so")
    shutil.copyfile(vt_build.BIND, copy)
    monkeypatch.setattr(vt_build, "BIND", copy)
    asked = []
    monkeypatch.setattr(vt_build.subprocess, "check_call", lambda cmd: asked.append(cmd) or shutil.copyfile(copy, cmd[cmd.index("-o") + 1]))
    vt_build.build_bind()
    assert not asked
    monkeypatch.setattr(torch, "__version__", "0.0.1")
    vt_build.build_bind()
    assert len(asked) == 1 and any("torch 0.0.1" in a for a in asked[0])


def test_a_module_for_another_torch_is_not_loaded():
    code = "import torch; torch.__version__ = '0.0.1'; import paper_2506_22694_b200 as vt; vt.lib()"
    r = subprocess.run([sys.executable, "-c", code], cwd=os.path.dirname(os.path.dirname(os.path.abspath(__file__))), capture_output=True, text=True)
    assert r.returncode != 0 and "built for another Python or torch" in r.stderr and "this is" in r.stderr
