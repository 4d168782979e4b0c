"""The module in front of the library (csrc/marshal.cpp) reads torch's objects by their layout: it is used only with the torch and the
Python that it was built for, built again when they change, and done without where it cannot be had.  CPU."""
import subprocess
import sys
import types

import pytest
import torch

import paper_2604_03260_b200 as package
from paper_2604_03260_b200 import binding as fb
from paper_2604_03260_b200 import build


@pytest.fixture
def put(monkeypatch):
    """put(m): the next load of the binding finds `m` in the place of the module (None: no module)"""
    fb.lib()                                    # (what is put back afterwards is the loaded state)
    def put(m):
        monkeypatch.setattr(fb, "_lib", None)
        monkeypatch.setattr(fb, "_marshal", None)
        monkeypatch.delattr(package, "_marshal", raising=False)
        monkeypatch.setitem(sys.modules, package.__name__ + "._marshal", m)
    return put


def module(built_for):
    """stands for a module built for `built_for`; records what it is given"""
    m = types.ModuleType(package.__name__ + "._marshal")
    m.__file__, m.given = "elsewhere", []
    m.init = lambda *args: m.given.append(args)
    if built_for is not None:
        m.built_for = built_for
    return m


def test_the_module_beside_the_library_is_the_one_in_use():
    fb.lib()
    assert fb._marshal.__file__ == build.MARSHAL and fb._marshal.built_for == build.marshal_abi()


@pytest.mark.parametrize("built_for", [None, "2.0.0 0123abcd cpython-310-x86_64-linux-gnu"])
def test_a_module_of_another_torch_is_given_nothing(put, built_for):
    m = module(built_for)
    put(m)
    with pytest.warns(RuntimeWarning, match="another torch or Python"):
        fb.lib()
    assert m.given == [] and fb._marshal is not m


def test_without_the_module_every_call_goes_through_ctypes(put):
    put(None)
    with pytest.warns(RuntimeWarning, match="through ctypes"):
        assert fb.focus_version() >= 100
    s = fb.make_shape(8, 4, 1000, 128, 4, 2, 16)
    assert fb.focus_tiles_workspace_bytes(s, 0) > 0
    x, m = torch.zeros((8, 1000, 128), dtype=torch.bfloat16), torch.zeros((8, 1000), dtype=torch.int32)
    with pytest.raises(AssertionError):                  # not on the GPU: refused by the binding, as ever
        fb.focus_assign(s, x, 8, x, m)
    with pytest.raises(AssertionError):
        fb.focus_assign_hidden(s, x[0], x, x, None, x, m, m)
    with pytest.raises(AssertionError):
        fb.focus_attn_fwd(s, x, x, x, m, m, m, 0, x, m)
    with pytest.raises(AssertionError):
        fb.focus_decode_step(s, x[:, 0], x, x, m, m, x[:, 0], m, m)


@pytest.mark.parametrize("cmd", [["false"], ["no-such-compiler"]])
def test_a_module_that_cannot_be_built_leaves_the_library(monkeypatch, tmp_path, cmd):
    old = tmp_path / "_marshal.so"
    old.write_text("of another torch")
    monkeypatch.setattr(build, "MARSHAL", str(old))
    monkeypatch.setattr(build, "_marshal_stamp", lambda: str(tmp_path / "stamp"))
    monkeypatch.setattr(build, "_marshal_cmd", lambda out: cmd)
    assert not build.build_marshal() and not old.exists()


@pytest.mark.parametrize("change", ["torch", "python", "flags"])
def test_the_module_is_built_again_after(monkeypatch, tmp_path, change):
    cmd = build._marshal_cmd
    monkeypatch.setattr(build, "_stale", lambda target, deps: False)            # the sources are as they were
    monkeypatch.setattr(build, "_marshal_stamp", lambda: str(tmp_path / "stamp"))
    assert build.marshal_stale()
    (tmp_path / "stamp").write_text("\n".join(cmd(build.MARSHAL)))
    assert not build.marshal_stale()
    if change == "torch":
        monkeypatch.setattr(torch, "__version__", "99.0")
    elif change == "python":
        monkeypatch.setattr(build.sysconfig, "get_config_var", lambda name: "another")
    else:
        monkeypatch.setattr(build, "_marshal_cmd", lambda out: cmd(out) + ["-DX"])
    assert build.marshal_stale()


def test_the_module_calls_the_library_that_the_binding_loaded():
    """not a copy that the loader finds for itself: none is linked, and the addresses come from the loaded one"""
    fb.lib()
    m = fb._marshal
    needed = subprocess.run(["readelf", "-d", m.__file__], check=True, capture_output=True, text=True).stdout
    assert "libtorch_python" in needed and "libfocus" not in needed
    for bad in ((), (fb.focus_shape,), (fb.focus_shape, 1, 2, 3, 4), (fb.focus_shape, 1, 2, 3, 4, 0), (fb.focus_shape, 1, 2, 3, 4, "x")):
        with pytest.raises((TypeError, ValueError)):
            m.init(*bad)
