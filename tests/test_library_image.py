"""The library's device images are stored as they are: unpacking a compressed one
would cost the first context of every process about 11 ms."""
import types

from paper_2311_08872_gb300 import build as libbuild


def test_device_images_are_not_compressed(monkeypatch, tmp_path):
    """Every source file is compiled with the option that keeps nvcc from compressing
    large images (the commands are recorded, nothing is compiled)."""
    commands = []

    def popen(cmd, **kw):
        commands.append(cmd)
        return types.SimpleNamespace(communicate=lambda: (b"", None), returncode=0)

    lib = tmp_path / "lib.so"
    monkeypatch.setattr(libbuild, "LIB", str(lib))
    monkeypatch.setattr(libbuild, "BUILD_DIR", str(tmp_path))
    monkeypatch.setattr(libbuild, "nvcc", lambda: "nvcc")
    monkeypatch.setattr(libbuild, "subprocess", types.SimpleNamespace(
        Popen=popen, PIPE=None, STDOUT=None, run=lambda cmd, **kw: (tmp_path / "lib.so.tmp").write_bytes(b"")))
    assert libbuild.build(force=True) == str(lib)
    assert len(commands) == len(libbuild.SOURCES)
    assert all("--no-compress" in cmd for cmd in commands)
