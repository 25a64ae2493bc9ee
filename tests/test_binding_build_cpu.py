"""The native call path of api.py is an addition to libbysdf.so: where it cannot
be built or loaded, the library builds, loads and works without it."""
import os
import subprocess
import sys

import pytest

from paper_2401_12724_gb300 import _native as N
from paper_2401_12724_gb300 import build as B


@pytest.fixture
def elsewhere(monkeypatch, tmp_path):
    """The build's products in tmp_path, made by a fake nvcc; a C++ compiler that fails."""
    calls = []
    real = subprocess.run

    def run(cmd, **kw):
        calls.append(cmd)
        if os.path.basename(cmd[0]) == "nvcc":
            with open(cmd[cmd.index("-o") + 1], "w"):
                pass
            return subprocess.CompletedProcess(cmd, 0, "", "")
        return real(cmd, **kw)

    monkeypatch.setattr(B, "LIB_PATH", str(tmp_path / "libbysdf.so"))
    monkeypatch.setattr(B, "BINDING_PATH", str(tmp_path / "_bysdf_torch.so"))
    monkeypatch.setattr(B, "BUILD_DIR", str(tmp_path / "_build"))
    monkeypatch.setattr(B.subprocess, "run", run)
    monkeypatch.setattr(B, "_nvcc", lambda: "/usr/local/cuda/bin/nvcc")
    return calls


@pytest.mark.parametrize("cxx", ["false", "no-such-compiler"])
def test_a_failed_binding_build_leaves_the_library(elsewhere, monkeypatch, cxx):
    monkeypatch.setenv("CXX", cxx)
    with pytest.warns(UserWarning, match="native call path"):
        assert B.build() == B.LIB_PATH
    assert os.path.exists(B.LIB_PATH) and not os.path.exists(B.BINDING_PATH)
    # and with the library up to date
    with pytest.warns(UserWarning, match="native call path"):
        assert B.build() == B.LIB_PATH


def test_a_failed_library_build_is_an_error(elsewhere, monkeypatch):
    monkeypatch.setattr(B.subprocess, "run",
                        lambda cmd, **kw: subprocess.CompletedProcess(cmd, 1, "", "no"))
    with pytest.raises(RuntimeError), pytest.warns(UserWarning):
        B.build()


def test_the_library_loads_beside_a_binding_that_does_not(monkeypatch, tmp_path):
    bad = tmp_path / "_bysdf_torch.so"
    bad.write_bytes(b"not a library")
    (tmp_path / "_bysdf_torch.so.abi").write_text(B._abi())
    N.load()
    monkeypatch.setattr(B, "BINDING_PATH", str(bad))
    monkeypatch.setattr(N, "_lib", None)
    monkeypatch.setattr(N, "calls", None)
    with pytest.warns(UserWarning, match="native call path"):
        lib = N.load(build_if_missing=False)
    assert N.calls is None and lib.bysdf_version().startswith(b"libbysdf")


def test_the_binding_is_built_and_loaded_here():
    r = subprocess.run([sys.executable, "-W", "error::UserWarning", "-c",
                        "import torch; from paper_2401_12724_gb300 import _native as N; "
                        "N.load(); assert N.calls is not None"],
                       cwd=B.ROOT, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr


def _fake_compiler(monkeypatch, made):
    def run(cmd, **kw):
        made.append(cmd)
        with open(cmd[cmd.index("-o") + 1], "w"):
            pass
        return subprocess.CompletedProcess(cmd, 0, "", "")
    monkeypatch.setattr(B.subprocess, "run", run)


def test_another_torch_builds_the_binding_again(elsewhere, monkeypatch):
    import torch

    made = []
    _fake_compiler(monkeypatch, made)
    B.build()
    n = len(made)
    B.build()
    assert len(made) == n  # up to date
    monkeypatch.setattr(torch, "__version__", "9.9.9+other")
    B.build()
    assert len(made) == n + 1 and made[-1][-1] == "-lc10_cuda"
    os.remove(B.BINDING_PATH + ".abi")
    B.build()
    assert len(made) == n + 2


def test_a_binding_for_another_torch_is_not_loaded(monkeypatch):
    import torch

    N.load()
    monkeypatch.setattr(torch, "__version__", "9.9.9+other")
    monkeypatch.setattr(N, "_lib", None)
    monkeypatch.setattr(N, "calls", None)
    with pytest.warns(UserWarning, match="another torch"):
        N.load(build_if_missing=False)
    assert N.calls is None
