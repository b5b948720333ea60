"""The fused kernel's splits of its 24 warps (12, 14 or 16 emit) and grains per lane, against the two-kernel path.

Which split runs follows from the shape; every value is formed by the same operations in the same order
(Eqs. 7-10), so T, the flags, L and the residual must be bitwise equal on both sides of each line."""
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


# (wavelengths, grains): 12, 14 and 16 emission warps at one to four grains per lane; the smallest and narrowest;
# then grain passes with a cell in one, two and more passes of the solver
SHAPES = [(9, 3), (16, 126), (100, 24), (300, 24), (400, 24), (190, 50), (205, 50), (220, 50), (150, 96), (170, 96), (187, 93), (200, 96),
          (100, 97), (150, 128), (184, 126), (220, 126), (61, 129), (400, 113), (500, 150), (500, 240), (200, 510)]


@pytest.mark.parametrize("form", ["general", "mass"])
@pytest.mark.parametrize("K,G", SHAPES)
def test_every_split_equals_two_kernel_path(K, G, form):
    from paper_0907_3768_gb300 import Context, padded_rows

    sms = torch.cuda.get_device_properties(0).multi_processor_count
    cells = 97 * sms + 17  # more than the small-call kernel takes; a ragged last tile
    wl = synth.make_workload(dict(synth.CONFIGS[0], K=K, n_sizes=G, species=("silicate",), n_cells=509, seed=41))
    at = np.arange(cells) % 509
    J, n = padded_rows(torch.from_numpy(wl.J[at]).cuda()), torch.from_numpy(wl.n[at]).cuda()
    out = {}
    with Context.from_workload(wl, precision="bf16x3") as ctx:
        if form == "mass":
            ctx.set_grain_numbers(wl.n[0].astype(np.float64))
        for fused in (False, True):
            ctx.set_fused_emit(fused)
            out[fused] = ctx.solve_mass(J, n[:, 0].contiguous()) if form == "mass" else ctx.solve(J, n)
            assert ctx.check() == 0
    for k in ("T", "flags", "L", "resid"):
        assert torch.equal(out[True][k], out[False][k]), k
