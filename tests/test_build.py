"""When the Python extension is built again: its source, the header, or the torch it is built against changed."""
import os

from paper_2603_14360_b200 import build


def test_extension_is_built_for_the_torch_that_loads_it(monkeypatch):
    build.build()
    assert build._native_is_current()
    monkeypatch.setattr(build.importlib.metadata, "version", lambda name: "0.0")
    assert not build._native_is_current()


def test_extension_follows_its_source(monkeypatch, tmp_path):
    build.build()
    copy = tmp_path / "_native.so"
    copy.write_bytes(b"")
    monkeypatch.setattr(build, "NATIVE", str(copy))
    assert build._native_is_current()
    os.utime(copy, (0, 0))
    assert not build._native_is_current()
