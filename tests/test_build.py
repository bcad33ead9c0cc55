"""The build script with stand-ins for the compilers (each writes the file named by -o): what it makes without PyTorch, and when."""
import os
import stat
import sys

import pytest

from paper_2609_28358_b200 import build


@pytest.fixture
def made(tmp_path, monkeypatch):
    """build.build() into tmp_path; returns what the stand-ins were asked to make since the last call, as file names."""
    log = tmp_path / "log"
    tool = tmp_path / "tool"
    tool.write_text(f"#!{sys.executable}\nimport sys\nout = sys.argv[sys.argv.index('-o') + 1]\nopen(out, 'w').close()\n"
                    f"open({str(log)!r}, 'a').write(out + '\\n')\n")
    tool.chmod(tool.stat().st_mode | stat.S_IXUSR)
    monkeypatch.setattr(build, "OBJ", str(tmp_path / "obj"))
    monkeypatch.setattr(build, "LIB", str(tmp_path / "libmq.so"))
    monkeypatch.setattr(build, "BINDING", str(tmp_path / "_mq_torch.so"))
    monkeypatch.setattr(build, "NVCC", str(tool))
    monkeypatch.setattr(build, "CXX", str(tool))

    def call():
        log.write_text("")
        assert build.build() == build.LIB
        return {os.path.basename(l).split(".tmp")[0] for l in log.read_text().split()}

    return call


def test_the_library_needs_no_pytorch(made, monkeypatch):
    monkeypatch.setitem(sys.modules, "torch", None)      # `import torch` raises ImportError
    names = made()
    assert "libmq.so" in names and "mq_api.o" in names and not names & {"mq_torch.o", "_mq_torch.so"}
    assert os.path.exists(build.LIB) and not os.path.exists(build.BINDING)
    monkeypatch.undo()


def test_the_binding_is_built_where_pytorch_is(made):
    assert {"libmq.so", "mq_torch.o", "_mq_torch.so"} <= made()
    assert made() == set()                               # up to date


def test_the_binding_follows_its_pytorch_and_python(made, monkeypatch):
    import torch

    made()
    monkeypatch.setattr(torch, "__version__", "0.0.0+other")
    assert made() == {"mq_torch.o", "_mq_torch.so"} and made() == set()
    monkeypatch.setattr(build.sysconfig, "get_config_var", lambda name: "cpython-other")
    assert made() == {"mq_torch.o", "_mq_torch.so"} and made() == set()
