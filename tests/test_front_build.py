"""The _front module is compiled against one torch's headers and ABI: another torch, or a change of the build's
own file, has it built again, and a module that no longer fits does not stay."""
import os
import subprocess

import pytest

torch = pytest.importorskip("torch")


@pytest.fixture
def built(monkeypatch, tmp_path):
    """build.py with a module in a folder of its own, and a compiler that only writes its output file."""
    from paper_0907_3768_gb300 import build

    runs = []

    def compiler(cmd, **kw):
        runs.append(cmd)
        if not getattr(compiler, "fails", False):
            open(cmd[cmd.index("-o") + 1], "w").close()
        return subprocess.CompletedProcess(cmd, int(getattr(compiler, "fails", False)), "", "")

    monkeypatch.setattr(build, "FRONT", str(tmp_path / "_front.so"))
    monkeypatch.setattr(build, "FRONT_STAMP", str(tmp_path / "_front.so.built_against"), raising=False)
    monkeypatch.setattr(build.subprocess, "run", compiler)
    build.build_front()
    assert len(runs) == 1
    build.build_front()
    assert len(runs) == 1  # up to date
    return build, runs, compiler


def test_another_torch_builds_again(built, monkeypatch):
    build, runs, _ = built
    monkeypatch.setattr(torch, "__version__", "0.0.0")
    build.build_front()
    build.build_front()
    assert len(runs) == 2


def test_another_place_builds_again(built, monkeypatch, tmp_path):
    build, runs, _ = built
    monkeypatch.setattr(torch, "__file__", str(tmp_path / "torch" / "__init__.py"))
    build.build_front()
    assert len(runs) == 2


def test_a_newer_build_file_builds_again(built):
    build, runs, _ = built
    os.utime(build.FRONT, (1, 1))  # older than every source
    build.build_front()
    assert len(runs) == 2


def test_a_module_that_does_not_fit_does_not_stay(built, monkeypatch):
    build, runs, compiler = built
    monkeypatch.setattr(torch, "__version__", "0.0.0")
    compiler.fails = True
    with pytest.raises(RuntimeError):
        build.build_front()
    assert not os.path.exists(build.FRONT)
