"""The emission kernel's two forms (15 warps, or 23 that claim ahead) against the fused kernel.

A tile offers one item per 8 wavelengths; from 46 items on the 23-warp form runs.  Every item is
formed by the same operations in the same order (Eqs. 8-10), so T, the flags, L and the residual must
be bitwise equal on both sides of the line, for the smallest tiles, and in grain passes."""
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


@pytest.mark.parametrize("form", ["general", "mass"])
@pytest.mark.parametrize("cells", [1, 33, 20011])
@pytest.mark.parametrize("K,sizes", [(8, 24), (360, 24), (361, 24), (500, 240)])
def test_emission_kernel_equals_fused_kernel(K, sizes, cells, form):
    from paper_0907_3768_gb300 import Context, padded_rows

    cfg = dict(synth.CONFIGS[0])
    cfg.update(K=K, n_sizes=sizes, species=("silicate",), n_cells=min(cells, 257), seed=11)
    wl = synth.make_workload(cfg)
    at = np.arange(cells) % min(cells, 257)
    J = padded_rows(torch.from_numpy(wl.J[at]).cuda())
    n = torch.from_numpy(wl.n[at]).cuda()
    out = {}
    with Context.from_workload(wl, precision="bf16x3") as ctx:
        if form == "mass":
            ctx.set_grain_numbers(wl.n[0].astype(np.float64))
        for fused in (False, True):
            ctx.set_fused_emit(fused)
            o = ctx.solve_mass(J, n[:, 0].contiguous()) if form == "mass" else ctx.solve(J, n)
            assert ctx.check() == 0
            out[fused] = {k: o[k].cpu().numpy() for k in ("T", "flags", "L", "resid")}
    for k, v in out[False].items():
        np.testing.assert_array_equal(out[True][k], v, err_msg=k)
