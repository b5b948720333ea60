"""Small calls: tiles of 8 or 16 cells with their k-groups split over CTAs, against the two-kernel path.

The split kernel forms every value by the same operations in the same order (Eqs. 7-10), so T, the
flags, L and the residual must be bitwise equal, on both sides of the cell counts where the lanes
per cell, the parts per tile and the kernel itself change."""
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


def _cells(where):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    return {"1": 1, "8": 8, "9": 9, "1 part": 8 * sms, "4 lanes": 16 * sms, "2 lanes": 16 * sms + 1,
            "two waves": 40 * sms - 3, "passes": 52 * sms, "few terms": 96 * sms, "fused": 96 * sms + 1}[where]


SHAPES = {"200x96": (200, 32, ("silicate", "graphite", "pah")), "37x5": (37, 5, ("silicate",)),
          "2x1": (2, 1, ("graphite",)), "61x240": (61, 120, ("silicate", "graphite")),
          "500x240": (500, 80, ("silicate", "graphite", "pah"))}  # several parts for the weights, ordered cells


@pytest.mark.parametrize("form", ["general", "mass", "resid only"])
@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("where", ["1", "8", "9", "1 part", "4 lanes", "2 lanes", "two waves", "passes", "few terms", "fused"])
def test_split_calls_equal_two_kernel_path(where, shape, form):
    from paper_0907_3768_gb300 import Context, padded_rows

    K, sizes, species = SHAPES[shape]
    cfg = dict(synth.CONFIGS[0])
    cfg.update(K=K, n_sizes=sizes, species=species, n_cells=_cells(where), seed=31,
               lam_um=(5.0, 200.0) if K == 2 else (0.09, 1000.0))
    wl = synth.make_workload(cfg)
    J = padded_rows(torch.from_numpy(wl.J).cuda())
    n = torch.from_numpy(wl.n).cuda()
    out = {}
    with Context.from_workload(wl, precision="bf16x3") as ctx:
        if form == "mass":
            ctx.set_grain_numbers(wl.n[0].astype(np.float64))
        for fused in (False, True):
            ctx.set_fused_emit(fused)
            o = (ctx.solve_mass(J, n[:, 0].contiguous()) if form == "mass"
                 else ctx.solve(J, n, want_L=form == "general"))
            assert ctx.check() == 0
            out[fused] = {k: o[k].cpu().numpy() for k in ("T", "flags", "L", "resid") if o[k] is not None}
    for k, v in out[False].items():
        np.testing.assert_array_equal(out[True][k], v, err_msg=k)
