"""The library is rebuilt when any file it is made from is newer than it."""
import os

from paper_2511_08020_gb300 import build as b


def test_every_source_is_a_dependency():
    deps = {os.path.realpath(p) for p in b.dependencies()}
    made_from = {f for f in os.listdir(b.CSRC) if f.endswith((".cu", ".cpp", ".cuh", ".h"))} - {b.PROBE_SRC}
    assert {os.path.realpath(os.path.join(b.CSRC, f)) for f in made_from} <= deps
    assert os.path.realpath(b.__file__) in deps
    assert os.path.realpath(os.path.join(b.ROOT, "include", "dg.h")) in deps


def test_a_newer_element_source_is_compiled(tmp_path, monkeypatch):
    """dg_element.cu alone newer than the library: its objects are compiled and the library is linked anew."""
    lib = tmp_path / "libdg.so"
    lib.write_bytes(b"")
    files = [os.path.join(b.CSRC, f) for f in os.listdir(b.CSRC)] + [b.__file__, os.path.join(b.ROOT, "include", "dg.h")]
    newest = max(os.path.getmtime(p) for p in files)
    os.utime(lib, (newest + 10, newest + 10))
    compiled = []
    monkeypatch.setattr(b, "LIB", str(lib))
    monkeypatch.setattr(b, "LIBDIR", str(tmp_path))
    monkeypatch.setattr(b, "_compile", lambda src, obj, defines=(): compiled.append(src))

    class Linked:
        returncode = 0
    monkeypatch.setattr(b.subprocess, "run", lambda cmd, **kw: open(cmd[cmd.index("-o") + 1], "wb").close() or Linked)
    b.build()
    assert not compiled
    element = os.path.realpath(os.path.join(b.CSRC, b.ELEMENT_SRC))
    real = os.path.getmtime
    monkeypatch.setattr(b.os.path, "getmtime", lambda p: newest + 20 if os.path.realpath(p) == element else real(p))
    b.build()
    assert b.ELEMENT_SRC in compiled
