"""What a build does where torch is missing, broken or another version than before (nothing is compiled here)."""
import pytest

from paper_2412_18106_b200 import build as B


@pytest.fixture
def steps(monkeypatch, tmp_path):
    done = []
    monkeypatch.setattr(B, "FASTCALL", str(tmp_path / "_fastcall.so"))
    monkeypatch.setattr(B, "FASTCALL_STAMP", str(tmp_path / "build" / "fastcall.torch"))
    monkeypatch.setattr(B, "_build_lib", lambda force, verbose: done.append("lib") or "lib.so")

    class Compiler:
        returncode = 0

        def communicate(self):
            done.append("fastcall")
            return (b"", None)

    def start():
        out = str(tmp_path / "out.so")
        open(out, "w").close()
        return Compiler(), out

    monkeypatch.setattr(B, "start_fastcall", start)
    return done


def test_the_library_is_built_without_torch(steps, monkeypatch):
    monkeypatch.setattr(B, "torch_version", lambda: None)
    assert B.build() == "lib.so" and steps == ["lib"]


def test_the_library_is_built_where_torch_does_not_import(steps, monkeypatch):
    def start():
        raise ImportError("libtorch.so: cannot open")
    monkeypatch.setattr(B, "start_fastcall", start)
    with pytest.raises(RuntimeError, match="fastcall"):
        B.build()
    assert steps == ["lib"]


def test_another_torch_version_makes_the_extension_stale(steps, monkeypatch):
    monkeypatch.setattr(B, "torch_version", lambda: "2.0")
    B.build()
    assert sorted(steps) == ["fastcall", "lib"]
    B.build()
    assert sorted(steps) == ["fastcall", "lib", "lib"]
    monkeypatch.setattr(B, "torch_version", lambda: "2.1")
    B.build()
    assert steps.count("fastcall") == 2
