"""When the native marshaller is built, what is left where it cannot be, and for whom it is used (no GPU needed)."""
import os
import re
import types

import pytest

from paper_2603_06738_b200 import binding, build


@pytest.mark.parametrize("compiler", ["false", "no-such-compiler"])
def test_the_library_is_built_without_a_compiler_for_the_marshaller(monkeypatch, tmp_path, compiler):
    """nvcc alone builds the library: a marshaller that does not compile leaves a warning, and none of an earlier build."""
    old = tmp_path / "_rib_marshal.so"
    old.write_bytes(b"of an earlier build")
    monkeypatch.setattr(build, "MARSHAL", old)
    monkeypatch.setattr(build, "LIB", tmp_path / "lib.so")
    monkeypatch.setattr(build, "sources", lambda: [])         # nothing to compile: what is asked is the order
    monkeypatch.setattr(build, "PKG", tmp_path)
    monkeypatch.setenv("NVCC", str(tmp_path / "nvcc"))
    nvcc = tmp_path / "nvcc"
    nvcc.write_text('#!/bin/sh\nfor a; do last=$a; done\necho linked > "$last"\n')
    nvcc.chmod(0o755)
    monkeypatch.setenv("CXX", compiler)
    with pytest.warns(RuntimeWarning, match="marshal"):
        lib = build.build(force=True)
    assert lib.read_text() == "linked\n"
    assert not old.exists()


def test_a_marshaller_for_another_torch_is_not_used():
    """It would import: nothing but its layout of a tensor is wrong."""
    for built_for in (None, build.marshal_identity().replace("torch ", "torch 1.")):
        module = types.SimpleNamespace(__name__="_rib_marshal", **({"built_for": built_for} if built_for else {}))
        with pytest.warns(RuntimeWarning, match="built for"):
            assert not binding._fits(module)
    assert binding._fits(types.SimpleNamespace(__name__="_rib_marshal", built_for=build.marshal_identity()))


def test_what_makes_a_marshaller_stale(monkeypatch, tmp_path):
    """Its source, the C header, the compiler flags, and the torch and the Python that it was compiled for."""
    files = {name: tmp_path / name for name in ("MARSHAL", "MARSHAL_SOURCE", "HEADER", "__file__")}
    for name, path in files.items():
        path.write_text(name)
        os.utime(path, (1000, 1000))
        monkeypatch.setattr(build, name, str(path) if name == "__file__" else path)
    monkeypatch.setattr(build, "PKG", tmp_path)
    (tmp_path / "_build").mkdir()
    assert build.marshal_stale()                        # nothing says what it was compiled for
    note = tmp_path / "_build" / "rib_marshal.built_for"
    note.write_text(build.marshal_identity())
    assert not build.marshal_stale()
    for name in ("MARSHAL_SOURCE", "HEADER", "__file__"):
        os.utime(files[name], (2000, 2000))
        assert build.marshal_stale(), name
        os.utime(files[name], (1000, 1000))
    note.write_text("torch 1.0, cpython-38")
    assert build.marshal_stale()


def test_the_marshaller_of_this_tree_says_what_it_was_built_for():
    build.build()
    from paper_2603_06738_b200 import _rib_marshal
    assert _rib_marshal.built_for == build.marshal_identity()


def test_the_backward_of_windows_of_16_does_not_spill():
    """Its arithmetic warps have 72 registers; 4 to 24 bytes of spills in them took 2 to 5 % of the kernel."""
    build.build()
    log = build.PKG / "_build" / "ptxas.log"
    if not log.exists():
        pytest.skip("the library was not compiled in this tree")
    spills = re.findall(r"Compiling entry function '[^']*rib_window16_bwd_kernel[^']*'.*?(\d+) bytes spill stores, (\d+) bytes spill loads", log.read_text(), re.S)
    assert spills == [("0", "0")] * 2              # ranks 16 and 32
