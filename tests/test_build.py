"""When the extension module counts as built: it is compiled against the layout of torch's and Python's objects."""
import os

import pytest

from paper_2505_20776_b200 import api, build


def test_module_carries_what_it_was_built_for():
    assert api._binding().built_for == build.binding_tag()
    assert build.binding_fits()


def test_another_torch_makes_the_module_stale(monkeypatch, tmp_path):
    """A newer file is not enough: with another torch it is built again, and refused where nobody builds."""
    monkeypatch.setattr(build, "binding_tag", lambda: "specext binding for torch 0.0, cpython-0")
    assert not build.binding_fits()
    commands = []
    monkeypatch.setattr(build, "_run", lambda cmd, lib, verbose: commands.append(cmd) or lib)
    future = os.path.getmtime(build.BINDING_PATH) + 1000
    monkeypatch.setattr(build.os.path, "getmtime", lambda p: future if p == build.BINDING_PATH else 0.0)
    assert build.build_binding() == build.BINDING_PATH and len(commands) == 1
    monkeypatch.setattr(api, "_BINDING", None)
    with pytest.raises(RuntimeError, match="another torch or Python"):
        api._binding()


def test_the_library_does_not_wait_for_the_module(monkeypatch):
    """A failing host compiler leaves libspecext.so built: the C ABI does not depend on the module."""
    built = []
    monkeypatch.setattr(build, "_compile", lambda lib, sources, defines, verbose: built.append(lib) or lib)

    def broken(force=False, verbose=False):
        raise RuntimeError("g++ failed")

    monkeypatch.setattr(build, "build_binding", broken)
    with pytest.raises(RuntimeError, match="g\\+\\+ failed"):
        build.build(force=True)
    assert built == [build.LIB_PATH]
