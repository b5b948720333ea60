"""The front end's native half shortens a call's host side and computes nothing: without it the library
still builds and a context still solves, with a warning and the same results."""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")


@pytest.fixture
def no_front(monkeypatch, tmp_path):
    import __graft_entry__
    from paper_0907_3768_gb300 import _lib

    __graft_entry__.build()
    monkeypatch.setattr(_lib, "_front", None)
    monkeypatch.setattr(_lib, "FRONT_PATH", str(tmp_path / "_front.so"))


@pytest.mark.parametrize("error", [RuntimeError("g++ failed"), ImportError("no torch headers"), FileNotFoundError("g++")])
def test_library_builds_where_the_native_half_does_not(monkeypatch, error):
    from paper_0907_3768_gb300 import build

    def fail(force):
        raise error

    monkeypatch.setattr(build, "build_front", fail)
    with pytest.warns(RuntimeWarning, match="not built"):
        assert build.build() == build.LIB


def test_missing_native_half_is_a_warning(no_front):
    from paper_0907_3768_gb300 import api

    with pytest.warns(RuntimeWarning, match="in Python"):
        assert api._front_or_none() is None


def test_unloadable_native_half_is_a_warning(no_front):
    from paper_0907_3768_gb300 import _lib, api

    with open(_lib.FRONT_PATH, "w") as f:
        f.write("not a module")
    with pytest.warns(RuntimeWarning, match="in Python"):
        assert api._front_or_none() is None


@pytest.mark.gpu
@pytest.mark.parametrize("mass", [False, True])
def test_context_without_native_half_solves_the_same(no_front, monkeypatch, mass):
    from paper_0907_3768_gb300 import Context, _lib

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    wl = synth.make_workload(0, cells=np.arange(40))
    J, n = torch.from_numpy(wl.J).cuda(), torch.from_numpy(wl.n).cuda()
    out = []
    for native in (False, True):
        if native:
            monkeypatch.undo()
            ctx = Context.from_workload(wl)
        else:
            with pytest.warns(RuntimeWarning, match="in Python"):
                ctx = Context.from_workload(wl)
        assert (ctx._front is not None) == native and (_lib._front is not None) == native
        with ctx:
            ctx.set_grain_numbers(wl.n[0].astype(np.float64))
            out.append(ctx.solve_mass(J, n[:, 0].contiguous()) if mass else ctx.solve(J, n))
    assert list(out[0]) == list(out[1])
    for k in ("T", "L", "resid", "flags"):
        assert torch.equal(out[0][k], out[1][k]), k
