"""The build: what the library needs, and when the binding's argument path is built again."""
import os
import sys
import sysconfig

import pytest

import paper_2609_32704_b200.binding as binding
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


def test_the_argument_path_is_built_again_for_another_pytorch(tiny, monkeypatch):
    torch = pytest.importorskip("torch")
    built = []

    def gxx(cmd, **kw):
        built.append(cmd)
        open(build.CALL_PATH, "w").close()
        return build.subprocess.CompletedProcess(cmd, 0, "", "")

    monkeypatch.setattr(build.subprocess, "run", gxx)
    os.makedirs(build.OBJ_DIR)
    for version, builds in (("9.9.0", 1), ("9.9.0", 1), ("9.9.1", 2), ("9.9.1", 2)):
        monkeypatch.setattr(torch, "__version__", version)
        build._build_call_module(False)
        assert len(built) == builds
        assert all(c[0] == "g++" for c in built)


def test_the_argument_path_carries_the_interpreters_tag():
    assert build.CALL_PATH.endswith(sysconfig.get_config_var("EXT_SUFFIX"))


def test_a_module_for_another_pytorch_is_refused_aloud(monkeypatch):
    torch = pytest.importorskip("torch")
    monkeypatch.setattr(binding, "_native", None)
    monkeypatch.setattr(torch, "__version__", "0.0.1")
    with pytest.warns(UserWarning, match="another torch.*Python path"):
        assert binding._call() is binding._PythonPath
