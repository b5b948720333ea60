"""The coupled iteration's kept emission order and its two forms of the J update: a cell's result
depends neither on the other cells of the call nor on the rows' alignment."""
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


@pytest.mark.parametrize("K", [64, 65, 301])
@pytest.mark.parametrize("iters", [1, 2, 5])
def test_coupled_cells_do_not_depend_on_batch_or_rows(K, iters):
    from paper_0907_3768_gb300 import Context

    sms = torch.cuda.get_device_properties(0).multi_processor_count
    C = 96 * sms + 40  # emitted in order
    cfg = dict(synth.CONFIGS[0])
    cfg.update(K=K, n_cells=C, seed=17)
    wl = synth.make_workload(cfg)
    rng = np.random.default_rng(2)
    kappa = wl.n.astype(np.float64) @ wl.C_abs
    E = (rng.uniform(0.0, 0.5, C)[:, None] / (4.0 * np.pi * kappa)).astype(np.float32)
    J, n, E = torch.from_numpy(wl.J).cuda(), torch.from_numpy(wl.n).cuda(), torch.from_numpy(E).cuda()
    pad = lambda x, ld: torch.nn.functional.pad(x, (0, ld - K))[:, :K]  # noqa: E731
    with Context.from_workload(wl, precision="fp32") as ctx:
        run = lambda a, b, ld: ctx.solve_coupled(pad(J[a:b], ld), pad(E[a:b], ld), n[a:b], max_iters=iters, tol=0.0)  # noqa: E731
        whole, it, change = run(0, C, (K + 3) // 4 * 4)
        assert it == iters and (change == float("inf")) == (iters == 1)
        odd, _, change_odd = run(0, C, K + 3 - K % 2)
        part, _, _ = run(1001, 1900, K)
    assert change_odd == change
    for k in ("T", "L", "resid", "flags"):
        assert torch.equal(odd[k], whole[k]), k
        assert torch.equal(part[k], whole[k][1001:1900]), k
