"""When the extension modules are built again: a change of the interpreter's or torch's binary interface
counts, not only the file times."""
import os

from paper_2002_10711_b200 import build


def test_a_module_for_another_torch_is_stale(tmp_path):
    source, target = tmp_path / "a.cpp", tmp_path / "a.so"
    source.write_text("")
    assert build._stale(str(target), "torch 1", str(source))           # not there yet
    tmp = tmp_path / "a.so.tmp"
    tmp.write_text("")
    build._install(str(tmp), str(target), "torch 1")
    assert not build._stale(str(target), "torch 1", str(source))
    assert build._stale(str(target), "torch 2", str(source))           # torch was upgraded
    os.utime(source, (os.path.getmtime(target) + 5,) * 2)
    assert build._stale(str(target), "torch 1", str(source))           # the source was edited
    os.utime(source, (os.path.getmtime(target) - 5,) * 2)
    os.remove(str(target) + ".abi")
    assert build._stale(str(target), "torch 1", str(source))           # built before there were notes


def test_the_built_modules_carry_their_interface():
    build.build()
    for module in (build.NATIVE, build.NATIVE_TORCH):
        with open(module + ".abi") as f:
            assert f.read()
