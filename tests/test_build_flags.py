"""The library's device code is stored uncompressed, so that a process does not
wait for it to be unpacked at its first relaunch."""
import subprocess

from paper_2305_18575_gb300 import build


def test_every_source_compiles_without_compression(monkeypatch, tmp_path):
    seen = []

    def run(cmd, **kw):
        seen.append(cmd)
        return subprocess.CompletedProcess(cmd, 0, "", "")

    lib = tmp_path / "librei.so"
    (tmp_path / "librei.so.tmp").write_bytes(b"")
    monkeypatch.setattr(build, "LIB", str(lib))
    monkeypatch.setattr(build, "OBJDIR", str(tmp_path / "obj"))
    monkeypatch.setattr(build, "nvcc", lambda: "nvcc")
    monkeypatch.setattr(build, "build_peak", lambda cc=None: None)
    monkeypatch.setattr(build.subprocess, "run", run)
    build.build(force=True)
    compiles = [c for c in seen if "-c" in c]
    assert len(compiles) == len(build.SOURCES)
    assert all("--compress-mode=none" in c and "-lineinfo" in c for c in compiles)
