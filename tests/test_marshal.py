"""The extension module of the binding takes every call form that its Python twins take, with the same results and errors
(no GPU needed: calls that return before a launch)."""
import copy
import ctypes
import importlib.machinery
import importlib.util
import inspect
import os
import pickle
import shutil
import subprocess
import sys
import types
import weakref

import numpy as np
import pytest
import torch

import paper_2206_15014_b200 as nm

PACKAGE = os.path.dirname(os.path.abspath(nm.__file__))
SUFFIX = importlib.machinery.EXTENSION_SUFFIXES[0]

NAMES = ("nm_int_linear", "nm_int_linear_dsx", "nm_int_linear_q8", "nm_int_linear_bf16", "nm_absmax", "nm_quantize_act")


def _args(name):
    t = torch.zeros(64, dtype=torch.float32)
    w = nm.make_packed(128, 128, 2, 4, 8, t, t)
    return {"nm_int_linear": (t, 0, w, 0.5, t, t, t), "nm_int_linear_dsx": (t, 0, w, t, t, t, t),
            "nm_int_linear_q8": (t, 0, w, 0.5, t, t, 1.0, t), "nm_int_linear_bf16": (t, 0, w, 0.5, t, t, t),
            "nm_absmax": (t, 0, t), "nm_quantize_act": (None, 0, t, None)}[name]


def _outcome(fn, *args, **kw):
    try:
        return ("value", fn(*args, **kw))
    except Exception as e:
        return (type(e), getattr(e, "code", None), str(e))


@pytest.mark.parametrize("name", NAMES)
def test_same_outcome_as_the_twin(name):
    fast, twin = getattr(nm, name), inspect.unwrap(getattr(nm, name))
    assert fast is not twin and inspect.signature(fast) == inspect.signature(twin) and fast.__name__ == name
    args, names = _args(name), list(inspect.signature(twin).parameters)
    forms = [(args, {"stream": 0}), ((), dict(zip(names, args), stream=0)), (args[:2], dict(zip(names[2:], args[2:]), stream=0)),
             (args, {"stream": 0, "nope": 1}), (args + args[-1:], {names[0]: args[0], "stream": 0}), (args[:-1], {"stream": 0}),
             (args, {"stream": "x"})]
    for i in range(len(args)):  # every argument of every wrong kind, and of kinds that only the twin converts
        other = [1.5, "a", None, 2 ** 70, np.int64(0)]
        if names[i] not in ("tokens", "count", "absmax"):  # (nothing that would launch)
            other += [True, -1, torch.zeros(3)]
        forms += [(args[:i] + (v,) + args[i + 1:], {"stream": 0}) for v in other]
    for a, kw in forms:
        if name == "nm_quantize_act":
            kw = dict(kw, sx_out=args[2])  # the maximum's own buffer: refused before a launch
        assert _outcome(fast, *a, **kw) == _outcome(twin, *a, **kw), (a, kw)


def test_error_codes_and_descriptor_checks():
    t = torch.zeros(64)
    w = nm.make_packed(128, 100, 2, 4, 8, t, t)  # not whole k-blocks
    with pytest.raises(nm.NmError) as e:
        nm.nm_int_linear(t, 4, w, 0.5, t, None, t, stream=0)
    assert e.value.code == nm.NM_ERR_SHAPE and "nm_int_linear" in str(e.value)

    class Other(ctypes.Structure):
        _fields_ = nm.nm_packed_t._fields_

    with pytest.raises(ctypes.ArgumentError):
        nm.nm_int_linear(t, 0, Other(), 0.5, t, None, t, stream=0)


@pytest.mark.parametrize("name", NAMES)
def test_an_entry_does_what_a_function_does(name):
    fast, twin = getattr(nm, name), inspect.unwrap(getattr(nm, name))
    assert pickle.loads(pickle.dumps(fast)) is fast and copy.copy(fast) is fast
    held = types.SimpleNamespace(call=fast, other=[fast])
    again = copy.deepcopy(held)
    assert again.call is fast and again.other[0] is fast
    assert weakref.ref(fast)() is fast
    assert fast.__defaults__ == twin.__defaults__ and fast.__code__ is twin.__code__ and name in repr(fast)
    with pytest.raises(AttributeError):
        fast.no_such_attribute
    fast.note = 1
    try:
        assert fast.note == 1 and not hasattr(twin, "note")
    finally:
        del fast.note
    bound = type("Holder", (), {"call": fast})().call
    assert isinstance(bound, types.MethodType) and bound.__func__ is fast


def _imported_from(tmp_path, files):
    """The package with only the given files beside __init__.py, imported by another process: the type of an entry."""
    home = tmp_path / "paper_2206_15014_b200"
    home.mkdir()
    shutil.copy(os.path.join(PACKAGE, "__init__.py"), home)
    for name, source in files.items():
        if source is None:
            (home / name).write_bytes(b"not for this interpreter")
        else:
            shutil.copy(source, home / name)
    env = dict(os.environ, NMSPARSE_LIB=nm.LIB_PATH, PYTHONPATH=str(tmp_path))
    r = subprocess.run([sys.executable, "-c", "import paper_2206_15014_b200 as nm; assert nm.nm_version(); print(type(nm.nm_int_linear).__name__)"],
                       env=env, cwd=tmp_path, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr
    return r.stdout.split()[-1]


def test_the_package_is_complete_without_the_extension(tmp_path):
    assert _imported_from(tmp_path, {}) == "function"


def test_only_the_extension_of_this_interpreter_is_loaded(tmp_path):
    assert os.path.exists(os.path.join(PACKAGE, "_marshal" + SUFFIX)) and "." in SUFFIX[1:]
    assert _imported_from(tmp_path, {"_marshal.so": None, "_marshal.cpython-39-x86_64-linux-gnu.so": None}) == "function"


def test_the_library_is_built_where_the_extension_cannot_be(monkeypatch, tmp_path, capsys):
    spec = importlib.util.spec_from_file_location("nm_build", os.path.join(PACKAGE, "build.py"))
    build = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(build)
    built = []
    monkeypatch.setattr(build, "MARSHAL", str(tmp_path / "_marshal.so"))
    monkeypatch.setattr(build, "LIB", str(tmp_path / "lib.so"))
    monkeypatch.setattr(build, "CSRC", shutil.copytree(build.CSRC, tmp_path / "csrc"))
    monkeypatch.setenv("CC", str(tmp_path / "no_such_compiler"))
    monkeypatch.setenv("NVCC", shutil.which("true"))  # stands in for nvcc
    monkeypatch.setattr(build.os, "replace", lambda a, b: built.append(b))
    assert build.build() == build.LIB and built == [build.LIB]
    assert "not built" in capsys.readouterr().err
