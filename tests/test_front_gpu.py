"""The front end's native call against its general Python path: the same outputs for every form of
J that it takes, and the same errors for what is refused."""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def solver():
    import __graft_entry__

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    __graft_entry__.build()
    from paper_0907_3768_gb300 import Context

    wl = synth.make_workload(0, cells=np.arange(40))
    with Context.from_workload(wl, precision="fp32") as ctx:
        ctx.set_grain_numbers(wl.n[0].astype(np.float64))
        yield ctx, torch.from_numpy(wl.J).cuda(), torch.from_numpy(wl.n).cuda()


@pytest.mark.gpu
@pytest.mark.parametrize("rows", ["dense", "padded", "odd stride", "every other", "one", "none"])
@pytest.mark.parametrize("mass", [False, True])
@pytest.mark.parametrize("wants", [(1, 1, 1), (0, 0, 0), (0, 1, 0), (1, 0, 1)])
def test_native_call_equals_general_path(solver, rows, mass, wants):
    ctx, J, n = solver
    if rows in ("padded", "odd stride"):
        J = torch.nn.functional.pad(J, (0, 4 if rows == "padded" else 3))[:, :ctx.K]
    cut = {"every other": slice(None, None, 2), "one": slice(0, 1), "none": slice(0, 0)}.get(rows, slice(None))
    J, n = J[cut], n[cut].contiguous()
    call, x = (ctx.solve_mass, n[:, 0].contiguous()) if mass else (ctx.solve, n)
    want = dict(zip(("want_L", "want_resid", "want_flags"), map(bool, wants)))
    new = call(J, x, **want)
    old = call(J, x, out=ctx.alloc_outputs(J.shape[0], J.stride(0), **want))
    assert list(new) == list(old)
    for k in old:
        assert (new[k] is None) == (old[k] is None)
        if old[k] is not None and k != "L_buf":  # its padding columns are not written
            assert new[k].shape == old[k].shape and new[k].stride() == old[k].stride() and new[k].dtype == old[k].dtype
            assert torch.equal(new[k], old[k])


@pytest.mark.gpu
@pytest.mark.parametrize("bad", ["cpu", "half", "columns", "transposed", "n rows", "n strided"])
def test_refused_as_before(solver, bad):
    ctx, J, n = solver
    J, n = {"cpu": (J.cpu(), n), "half": (J.half(), n), "columns": (J[:, 1:], n), "transposed": (J.t().contiguous().t(), n),
            "n rows": (J, n[1:]), "n strided": (J, n.t().contiguous().t())}[bad]
    with pytest.raises(ValueError):
        ctx.solve(J, n)


def test_native_call_declines_what_it_does_not_take():
    import __graft_entry__
    from paper_0907_3768_gb300 import _lib

    __graft_entry__.build()
    J, n = torch.zeros(3, 8), torch.zeros(3, 2)
    assert _lib.front().solve(0, 0, 2, 8, 0, J, n, False, True, True, True) is None  # host tensors: nothing is called
