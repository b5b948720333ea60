"""Temperatures alone of many cells: every SM solves a few grains of all cells, against the solve by cells.

A root is formed by the same operations whichever lane takes it (Eq. 7), so T and the flags of the
whole call must be bitwise equal to those of calls of few cells, which take one warp per cell: at
grain counts that fill, exceed by one or leave most of a group of 16, with cell counts just above
the line between the two and with remainders in both shares of the cells."""
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


@pytest.mark.parametrize("precision", ["bf16x3", "fp32"])
@pytest.mark.parametrize("flags", [True, False])
@pytest.mark.parametrize("over", [1, 3001])
@pytest.mark.parametrize("sizes", [1, 16, 17, 96, 240, 512])
def test_temperatures_equal_those_of_small_calls(sizes, over, flags, precision):
    from paper_0907_3768_gb300 import Context, padded_rows

    few = 128 * torch.cuda.get_device_properties(0).multi_processor_count  # the largest call solved by cells
    cfg = dict(synth.CONFIGS[0])
    cfg.update(K=24, n_sizes=sizes, species=("silicate",), n_cells=257, seed=7)
    wl = synth.make_workload(cfg)
    C = few + over
    scale = np.exp(np.random.default_rng(3).uniform(-12.0, 12.0, C)).astype(np.float32)
    Jh = wl.J[np.arange(C) % 257] * scale[:, None]
    Jh[5], Jh[C - 1, 3], Jh[C - 2] = 0.0, np.inf, np.nan  # below the table, above it, invalid
    J = padded_rows(torch.from_numpy(Jh.astype(np.float32)).cuda())
    n = torch.from_numpy(wl.n[np.arange(C) % 257]).cuda()
    with Context.from_workload(wl, precision=precision) as ctx:
        out = ctx.solve(J, n, want_L=False, want_resid=False, want_flags=flags)
        assert ctx.check() == 0
        for c0 in range(0, C, few):
            part = ctx.solve(J[c0:c0 + few], n[c0:c0 + few], want_L=False, want_resid=False, want_flags=flags)
            for k in ("T", "flags") if flags else ("T",):
                np.testing.assert_array_equal(out[k][c0:c0 + few].cpu().numpy(), part[k].cpu().numpy(), err_msg=k)
