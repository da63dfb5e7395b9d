"""What the build needs and leaves: the library wants nvcc alone, the PyTorch
binding comes on top where it can. With stand-ins for the compilers."""
import os
import stat
import sys
import warnings

import pytest

FAKE = """#!/bin/sh
echo "$0 $@" >> "{log}"
{fail}
while [ $# -gt 0 ]; do [ "$1" = -o ] && : > "$2"; shift; done
exit 0
"""


@pytest.fixture
def tools(tmp_path, monkeypatch):
    """build with its folders and compilers replaced; tools(gxx_fails) sets them up."""
    from paper_2106_03452_gb300 import build
    log, out = tmp_path / "log", tmp_path / "out"
    monkeypatch.setattr(build, "BUILD", str(out))
    monkeypatch.setattr(build, "LIB", str(out / "libdpsr.so"))
    monkeypatch.setattr(build, "_nvcc", lambda: str(tmp_path / "bin" / "nvcc"))
    monkeypatch.setenv("PATH", f"{tmp_path / 'bin'}:{os.environ['PATH']}")

    def setup(gxx_fails=False):
        (tmp_path / "bin").mkdir(exist_ok=True)
        for name in ("nvcc", "g++"):
            p = tmp_path / "bin" / name
            p.write_text(FAKE.format(log=log, fail="exit 1" if name == "g++" and gxx_fails else ""))
            p.chmod(p.stat().st_mode | stat.S_IXUSR)
        log.write_text("")

        def ran():
            lines = log.read_text().splitlines()
            log.write_text("")
            return sum("nvcc" in s.split()[0] for s in lines), sum("g++" in s.split()[0] for s in lines)
        return build, out, ran
    return setup


def test_the_library_builds_without_pytorch(tools, monkeypatch):
    build, out, ran = tools()
    monkeypatch.setitem(sys.modules, "torch", None)  # import torch raises
    assert build.build() == str(out / "libdpsr.so") and os.path.exists(build.LIB)
    assert ran() == (len(build.SOURCES) + 1, 0)
    build.build()
    assert ran() == (0, 0)


def test_a_failing_binding_leaves_the_library(tools, capsys):
    pytest.importorskip("torch")
    build, out, ran = tools(gxx_fails=True)
    assert os.path.exists(build.build()) and not (out / build.BIND_NAME).exists()
    assert "without its PyTorch binding" in capsys.readouterr().err
    ran()
    build, out, ran = tools()
    build.build()
    assert ran() == (0, 2) and (out / build.BIND_NAME).exists()  # the binding alone
    build.build()
    assert ran() == (0, 0)


def test_another_pytorch_rebuilds_the_binding_alone(tools, monkeypatch):
    torch = pytest.importorskip("torch")
    build, out, ran = tools()
    build.build()
    assert ran() == (len(build.SOURCES) + 1, 2)
    monkeypatch.setattr(torch, "__version__", "0.0.0")
    build.build()
    assert ran() == (0, 2)


@pytest.mark.parametrize("what", ["missing", "unstamped", "foreign", "broken"])
def test_python_answers_without_the_binding(what, tmp_path, monkeypatch):
    torch = pytest.importorskip("torch")
    from paper_2106_03452_gb300 import build, libdpsr as L
    build.build()
    path = tmp_path / "_dpsr_torch.so"
    if what != "missing":
        path.write_bytes(b"not a library")
    if what in ("foreign", "broken"):
        (tmp_path / "_dpsr_torch.so.stamp").write_text(
            (torch.__version__ if what == "broken" else "0.0.0") + "\nfingerprint")
    monkeypatch.setattr(L, "BIND_PATH", str(path))
    monkeypatch.setattr(L, "_bind", None)
    with pytest.warns(RuntimeWarning, match="no PyTorch binding"):
        b = L.binding()
    assert b.layer(1, 2, 3) is None and b.chamfer(1, 2) is None
    with warnings.catch_warnings():
        warnings.simplefilter("error")
        assert L.binding() is b  # one warning
