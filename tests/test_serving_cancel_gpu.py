"""A cancelled request that has work on the GPU is finished, and its memory the caller's again, only once that
work has retired: waiting for it ends then, and until then polling calls it active."""
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


@pytest.mark.parametrize("how", ["wait", "poll"])
def test_cancelled_request_ends_after_its_parts(how):
    from paper_0907_3768_gb300 import Context, DustError, Server

    wl = synth.make_workload(0, cells=np.arange(256))
    J, n = torch.from_numpy(wl.J).cuda(), torch.from_numpy(wl.n).cuda()
    side = torch.cuda.Stream()
    with Context.from_workload(wl) as ctx, Server(256 << 20, 4) as server:
        server.wait(ctx.submit(server, J, n)[0])  # the kernels are loaded
        server.reset_stats()
        torch.cuda.synchronize()
        with torch.cuda.stream(side):
            torch.cuda._sleep(200_000_000)  # about 0.1 s: the request's round waits for its inputs
            ticket, out = ctx.submit(server, J, n)
        while server.stats()["rounds"] == 0:
            pass  # until the round is queued
        server.cancel(ticket)
        if how == "poll":
            state = "active"
            while state == "active":
                state, _ = server.poll(ticket)
            assert state == "cancelled"
        else:
            with pytest.raises(DustError, match="cancelled"):
                server.wait(ticket)
        assert side.query()  # the inputs are there, so the round has run
        s = server.stats()
        assert (s["active"], s["hbm_in_use"], s["cancelled"]) == (0, 0, 1)
