"""The binding's native module is built again when the Python or torch that it was built for has been replaced (no compiler is run here)."""
import types

import pytest

from paper_2608_15211_b200 import build


@pytest.fixture
def compiled(tmp_path, monkeypatch):
    runs = []

    def run(cmd, **_):
        runs.append(cmd)
        (tmp_path / "_host.so").write_bytes(b"")
        return types.SimpleNamespace(returncode=0, stdout="", stderr="")

    monkeypatch.setattr(build, "HOST_PATH", str(tmp_path / "_host.so"))
    monkeypatch.setattr(build, "HOST_TAG_PATH", str(tmp_path / "_host.so.tag"), raising=False)
    monkeypatch.setattr(build.subprocess, "run", run)
    build.build_host()
    build.build_host()
    assert len(runs) == 1
    return runs


@pytest.mark.parametrize("module,name,value", [("importlib.metadata", "version", lambda _: "9.9.9"), ("sysconfig", "get_config_var", lambda _: "cpython-399")])
def test_another_python_or_torch(compiled, monkeypatch, module, name, value):
    monkeypatch.setattr(f"{module}.{name}", value)
    build.build_host()
    assert len(compiled) == 2
    build.build_host()
    assert len(compiled) == 2
