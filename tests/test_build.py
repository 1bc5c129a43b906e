"""The build brings a _caatpy.so up to date that was made for another torch or Python."""
import os

from paper_2506_19645_b200 import build


def test_extension_of_another_torch_is_stale(tmp_path, monkeypatch):
    so, note = tmp_path / "_caatpy.so", tmp_path / "caat_py.for"
    monkeypatch.setattr(build, "PYEXT", str(so))
    monkeypatch.setattr(build, "PYEXT_FOR", str(note))
    assert not build.pyext_current()                    # nothing built yet
    so.write_bytes(b"")
    assert not build.pyext_current()                    # built by something that did not say for what
    note.write_text(build._abi())
    assert build.pyext_current()
    monkeypatch.setattr(build.importlib.metadata, "version", lambda name: "0.0")
    assert not build.pyext_current()                    # another torch
    monkeypatch.undo()
    monkeypatch.setattr(build, "PYEXT", str(so))
    monkeypatch.setattr(build, "PYEXT_FOR", str(note))
    os.utime(so, (0, 0))
    assert not build.pyext_current()                    # older than its sources
