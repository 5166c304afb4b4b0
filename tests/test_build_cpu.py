"""Building and loading with and without the binding's native call path, which needs
Python's headers: librlm.so alone has to serve every call (through ctypes)."""
import os
import subprocess

import pytest

rlm = pytest.importorskip("paper_2607_05583_gb300")
torch = pytest.importorskip("torch")

from paper_2607_05583_gb300 import build as cbuild


@pytest.fixture
def unloaded(monkeypatch):
    cbuild.build()
    monkeypatch.setattr(rlm, "_lib", None)
    monkeypatch.setattr(rlm, "_native", None)


def _refused_by_python():
    """A call that is not plain: the ctypes route's own check raises."""
    x = torch.zeros(1, 8)
    with pytest.raises(ValueError, match="contiguous CUDA"):
        rlm.rlm_mix_decode(x, None, x)


@pytest.mark.parametrize("broken", [False, True])
def test_the_library_alone_serves_every_call(monkeypatch, tmp_path, unloaded, broken):
    path = tmp_path / "_rlm_py.so"
    if broken:   # not this machine's
        path.write_bytes(b"no shared object")
    monkeypatch.setattr(cbuild, "PYLIB", str(path))
    if broken:
        with pytest.warns(UserWarning, match="ctypes"):
            rlm.load_library()
    else:
        rlm.load_library()
    assert rlm.rlm_version() == 100
    for name in ("mix_prefill", "mix_decode", "mix_backward", "mixer_prefill", "mixer_decode"):
        assert getattr(rlm._native, name)(1, 2, 3) is None
    _refused_by_python()


def test_build_if_missing_builds_the_call_path_too(monkeypatch, tmp_path, unloaded):
    built = []
    monkeypatch.setattr(cbuild, "PYLIB", str(tmp_path / "_rlm_py.so"))
    monkeypatch.setattr(cbuild, "build", lambda *a, **k: built.append(1))
    rlm.load_library(build_if_missing=True)
    assert built


def test_a_missing_library_names_the_build(monkeypatch, tmp_path, unloaded):
    monkeypatch.setattr(cbuild, "LIB", str(tmp_path / "librlm.so"))
    with pytest.raises(RuntimeError, match="not built"):
        rlm.load_library()


@pytest.mark.parametrize("headers", [True, False])
def test_build_without_python_headers_ends_at_the_library(monkeypatch, tmp_path, headers):
    ran = []

    def fake_run(cmd, **kw):   # the tools' part: every output file appears
        ran.append(cmd)
        open(cmd[cmd.index("-o") + 1], "w").close()
        return subprocess.CompletedProcess(cmd, 0, "", "")

    include = tmp_path / "include"
    include.mkdir()
    if headers:
        (include / "Python.h").write_text("")
    monkeypatch.setattr(cbuild, "BUILD", str(tmp_path))
    monkeypatch.setattr(cbuild, "LIB", str(tmp_path / "librlm.so"))
    monkeypatch.setattr(cbuild, "PYLIB", str(tmp_path / "_rlm_py.so"))
    monkeypatch.setattr(cbuild.sysconfig, "get_paths", lambda: {"include": str(include)})
    monkeypatch.setattr(cbuild.subprocess, "run", fake_run)
    assert cbuild.build() == str(tmp_path / "librlm.so")
    assert os.path.exists(cbuild.PYLIB) == headers
    n = len(ran)
    cbuild.build()   # nothing is stale
    assert len(ran) == n
