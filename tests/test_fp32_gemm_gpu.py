"""The FP32 contraction's two ways to fill its stages (through registers, by cp.async): a cell's sums are taken
in ascending wavelength whatever the way, the rows' alignment, the tile and the batch, so T is bitwise equal."""
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


@pytest.mark.parametrize("K", [2, 15, 16, 17, 100, 203])
@pytest.mark.parametrize("G", [1, 17, 40, 64, 65, 96, 112, 128, 129, 250])  # one to eight columns per thread
def test_ways_and_alignments_agree(K, G):
    from paper_0907_3768_gb300 import Context

    sms = torch.cuda.get_device_properties(0).multi_processor_count
    cells = 128 * 4 * sms + 129  # more tiles than any limit of the choice; a ragged last one
    wl = synth.make_workload(dict(synth.CONFIGS[0], K=K, n_sizes=G, species=("silicate",), n_cells=313, seed=53,
                                  lam_um=(5.0, 200.0) if K == 2 else (0.09, 1000.0)))
    J = torch.from_numpy(wl.J).cuda()[torch.arange(cells, device="cuda") % 313]
    n = torch.from_numpy(wl.n).cuda()[torch.arange(cells, device="cuda") % 313].contiguous()
    ld = (K + 3) // 4 * 4
    # rows padded with NaN: nothing past K may enter a sum
    pad = lambda x, w: torch.cat([x, torch.full((len(x), w - K), float("nan"), device="cuda")], 1)[:, :K]  # noqa: E731
    with Context.from_workload(wl, precision="fp32") as ctx:
        run = lambda x, m: ctx.solve(x, m, want_L=False, want_resid=False)["T"]  # noqa: E731
        want = run(pad(J, ld + 4), n)  # aligned
        assert not torch.isnan(want).any()
        assert torch.equal(run(pad(J, ld + 1), n), want)  # odd rows
        assert torch.equal(run(pad(J, ld + 5)[1:], n[1:]), want[1:])  # and an odd start
        for a, b in ((0, 1), (5, 133), (1000, 1000 + 127 * sms)):
            assert torch.equal(run(pad(J[a:b], ld + 4), n[a:b]), want[a:b])
            assert torch.equal(run(pad(J[a:b], ld + 3), n[a:b]), want[a:b])
