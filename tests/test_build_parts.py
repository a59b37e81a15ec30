"""The two libraries that build() makes do not depend on each other more than they have to."""
import os

import pytest

from paper_2501_12497_gb300 import build as B


@pytest.fixture
def fake(tmp_path, monkeypatch):
    """build() into an empty folder with compilers that only make their output; returns the commands run."""
    run = []

    def compiler(cmd, what, verbose=False):
        run.append(what)
        open(cmd[cmd.index("-o") + 1], "w").close()

    def nodes(obj, verbose):
        compiler(["-o", obj], "nodes")
        return "torch/lib"

    for name in ("LIB_PATH", "AUTOGRAD_PATH", "AUTOGRAD_FOR"):
        monkeypatch.setattr(B, name, str(tmp_path / os.path.basename(getattr(B, name, name))), raising=False)
    monkeypatch.setattr(B, "BUILD_DIR", str(tmp_path))
    monkeypatch.setattr(B, "_nvcc", lambda: "nvcc")
    monkeypatch.setattr(B, "_run", compiler)
    monkeypatch.setattr(B, "_compile_autograd", nodes)
    return run


def test_the_cuda_library_is_linked_when_the_nodes_fail(fake, monkeypatch):
    def no_torch(obj, verbose):
        raise RuntimeError("no torch headers")

    monkeypatch.setattr(B, "_compile_autograd", no_torch)
    with pytest.raises(RuntimeError, match="no torch headers"):
        B.build()
    assert os.path.exists(B.LIB_PATH) and not os.path.exists(B.AUTOGRAD_PATH)


def test_nodes_built_for_another_torch_are_built_again(fake, monkeypatch):
    B.build()
    assert "link of libmof.so" in fake and "link of _autograd.so" in fake
    del fake[:]
    B.build()
    assert not fake
    monkeypatch.setattr(B, "_torch_id", lambda: "another torch", raising=False)
    B.build()
    assert fake == ["nodes", "link of _autograd.so"]
    del fake[:]
    B.build()
    assert not fake
