"""The library is rebuilt when any of its sources changes, kernel code in
headers (*.cuh) among them."""
import glob
import os

from paper_1802_08557_gb300 import build


def test_every_source_is_a_dependency():
    deps = {os.path.realpath(p) for p in build._deps()}
    sources = [p for pat in ("*.cu", "*.cuh", "*.h") for p in glob.glob(os.path.join(build.CSRC, pat))]
    assert any(p.endswith(".cuh") for p in sources)
    assert {os.path.realpath(p) for p in sources} <= deps


def test_a_changed_kernel_header_makes_the_library_stale(tmp_path, monkeypatch):
    lib = tmp_path / build.LIB_NAME
    src, cuh = tmp_path / "a.cu", tmp_path / "a.cuh"
    for p in (src, cuh, lib):
        p.write_text("")
    for p, t in ((src, 100), (cuh, 100), (lib, 200)):
        os.utime(p, (t, t))
    monkeypatch.setattr(build, "CSRC", str(tmp_path))
    monkeypatch.setattr(build, "INCLUDE", str(tmp_path))
    monkeypatch.setattr(build, "LIB_PATH", str(lib))
    monkeypatch.setattr(build, "__file__", str(src))
    assert build.up_to_date()
    os.utime(cuh, (300, 300))
    assert not build.up_to_date()
