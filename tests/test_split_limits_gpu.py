"""Where a call with grain passes and more than 128 grains leaves the small-call kernel and comes back to it:
the same bits on both sides of each line as in two kernels, with few and with many wavelengths."""
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


@pytest.mark.parametrize("K,G", [(350, 180), (90, 400)])
@pytest.mark.parametrize("per_sm,over", [(28, 0), (28, 1), (32, 0), (32, 1), (44, 0), (44, 1), (52, 1)])
def test_both_sides_of_the_limits(per_sm, over, K, G):
    from paper_0907_3768_gb300 import Context, padded_rows

    cells = per_sm * torch.cuda.get_device_properties(0).multi_processor_count + over
    wl = synth.make_workload(dict(synth.CONFIGS[0], K=K, n_sizes=G, species=("silicate",), n_cells=211, seed=43))
    at = np.arange(cells) % 211
    J, n = padded_rows(torch.from_numpy(wl.J[at]).cuda()), torch.from_numpy(wl.n[at]).cuda()
    out = {}
    with Context.from_workload(wl, precision="bf16x3") as ctx:
        for fused in (False, True):
            ctx.set_fused_emit(fused)
            out[fused] = ctx.solve(J, n)
            assert ctx.check() == 0
    for k in ("T", "flags", "L", "resid"):
        assert torch.equal(out[True][k], out[False][k]), k
