"""The coupled iteration's buffers are made ready in the caller's stream: a first call on a side stream,
which nothing orders after the default one, does not depend on when the default stream's work ends."""
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


@pytest.mark.parametrize("cycles", [0, 100_000, 400_000, 1_000_000, 3_000_000])
def test_first_call_beside_a_busy_default_stream(cycles):
    from paper_0907_3768_gb300 import Context

    wl = synth.make_workload(dict(synth.CONFIGS[0], n_cells=2048, seed=23))
    rng = np.random.default_rng(2)
    kappa = wl.n.astype(np.float64) @ wl.C_abs
    E = (rng.uniform(0.0, 0.5, 2048)[:, None] / (4.0 * np.pi * kappa)).astype(np.float32)
    J, n, E = torch.from_numpy(wl.J).cuda(), torch.from_numpy(wl.n).cuda(), torch.from_numpy(E).cuda()
    side = torch.cuda.Stream()
    with Context.from_workload(wl, precision="fp32") as quiet, Context.from_workload(wl, precision="fp32") as busy:
        want, it, change = quiet.solve_coupled(J, E, n, tol=1e-6)
        torch.cuda.synchronize()
        torch.cuda._sleep(max(1, cycles))  # on the default stream
        with torch.cuda.stream(side):
            got, it_side, change_side = busy.solve_coupled(J, E, n, tol=1e-6)
        torch.cuda.synchronize()
        assert busy.check() == 0
    assert 2 < it < 50 and (it_side, change_side) == (it, change)
    for k in ("T", "L", "resid", "flags"):
        assert torch.equal(got[k], want[k]), k
