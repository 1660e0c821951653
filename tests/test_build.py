"""The build: what the library needs, and when the binding's argument path is built again."""
import os
import sys

import pytest

import paper_2609_32704_b200.build as build


@pytest.fixture
def tiny(monkeypatch, tmp_path):
    """A build of one small source into tmp_path."""
    src = tmp_path / "csrc"
    src.mkdir()
    (src / "tiny.cu").write_text('extern "C" int tiny() { return 7; }\n')
    (src / "tiny.h").write_text("")
    for name, path in (("CSRC", src), ("OBJ_DIR", tmp_path / "build"), ("LIB_PATH", tmp_path / "libtiny.so"),
                       ("CALL_PATH", tmp_path / os.path.basename(build.CALL_PATH))):
        monkeypatch.setattr(build, name, str(path))
    return tmp_path


def test_the_library_needs_no_pytorch(tiny, monkeypatch, capfd):
    monkeypatch.setitem(sys.modules, "torch", None)  # import torch raises ImportError
    assert os.path.exists(build.build_library())
    assert not os.path.exists(build.CALL_PATH)
    assert "not built" in capfd.readouterr().err


def test_the_library_needs_no_host_compiler_for_extensions(tiny, monkeypatch, capfd):
    run = build.subprocess.run
    monkeypatch.setattr(build.subprocess, "run", lambda cmd, **kw: run(["no-such-" + cmd[0]] if cmd[0] == "g++" else cmd, **kw))
    assert os.path.exists(build.build_library())
    assert "not built" in capfd.readouterr().err
