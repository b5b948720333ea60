"""Small coupled calls: the absorption launched ahead clears the part counters of the split solve + emission,
pass after pass, and the tile's last part folds the residuals; bitwise against the two-kernel path."""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    __graft_entry__.build()


@pytest.mark.parametrize("precision", ["fp32", "bf16x3", "fp16x3"])
@pytest.mark.parametrize("where", ["1", "9", "parts", "ordered"])
@pytest.mark.parametrize("iters", [1, 2, 7])
def test_split_passes_equal_two_kernel_passes(where, precision, iters):
    from paper_0907_3768_gb300 import Context, padded_rows

    sms = torch.cuda.get_device_properties(0).multi_processor_count
    # "parts": several CTAs per tile of 8 cells; "ordered": enough terms that the first pass makes an order
    C = {"1": 1, "9": 9, "parts": 2 * sms, "ordered": 24 * sms}[where]
    wl = synth.make_workload(dict(synth.CONFIGS[0], K=202, n_sizes=48, n_cells=C, seed=29))
    rng = np.random.default_rng(3)
    kappa = wl.n.astype(np.float64) @ wl.C_abs
    E = (rng.uniform(0.3, 0.5, C)[:, None] / (4.0 * np.pi * kappa)).astype(np.float32)
    J, E = (padded_rows(torch.from_numpy(x).cuda()) for x in (wl.J, E))
    n = torch.from_numpy(wl.n).cuda()
    out = {}
    with Context.from_workload(wl, precision=precision) as ctx:
        for fused in (False, True, True):
            ctx.set_fused_emit(fused)
            out[fused] = ctx.solve_coupled(J, E, n, max_iters=iters, tol=0.0)
            assert ctx.check() == 0
    assert out[True][1:] == out[False][1:] and out[True][1] == iters
    for k in ("T", "L", "resid", "flags"):
        assert torch.equal(out[True][0][k], out[False][0][k]), k
