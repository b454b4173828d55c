"""The native marshalling (csrc/binding.c) takes what the general path takes and
refuses what it refuses; without it the general path runs every call."""
import pytest

from paper_2311_04406_gb300 import abi, build


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    abi.load()


def test_calls_run_without_the_native_marshalling(monkeypatch, tmp_path):
    import torch
    monkeypatch.setattr(build, "BINDING", str(tmp_path / "_binding.so"))
    monkeypatch.setattr(abi, "_lib", None)
    monkeypatch.setattr(abi, "_nat", None)
    assert abi.load() is not None and abi._nat is None
    t = torch.zeros(8, dtype=torch.int64)
    with pytest.raises(ValueError, match="dst"):
        abi.mpc_transpose(32, 32, 2, 8, torch.zeros(16, dtype=torch.int64), t)
    with pytest.raises(ValueError, match=r"ins\[0\]"):
        abi.mpc_lincomb(32, 32, [1], [t[:4]], t)


def test_build_without_python_headers(monkeypatch, tmp_path):
    so = tmp_path / "_binding.so"
    so.write_bytes(b"of an older build")
    monkeypatch.setattr(build, "BINDING", str(so))
    monkeypatch.setattr(build.sysconfig, "get_paths", lambda: {"include": str(tmp_path)})
    assert build.binding_headers() is None
    build.build_binding(build.binding_headers())
    assert not so.exists()
    assert build.build() == build.LIB and not so.exists()
