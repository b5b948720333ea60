"""Rounds are queued without the server's lock: requests submitted, cancelled and polled by several threads
meanwhile give dust_solve's bits or are cancelled, and the server's counts add up."""
import threading

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


def test_submissions_and_cancellations_during_launches():
    from paper_0907_3768_gb300 import Context, DustError, Server

    threads, each = 4, 80
    wl = synth.make_workload(dict(synth.CONFIGS[0], n_cells=700, seed=47))
    J, n = torch.from_numpy(wl.J).cuda(), torch.from_numpy(wl.n).cuda()
    sizes = np.random.default_rng(5).integers(1, 701, (threads, each))
    counts, failed = [0, 0], []
    lock = threading.Lock()
    with Context.from_workload(wl, precision="fp32") as ctx, Server(256 << 20, 16) as server:
        want = ctx.solve(J, n)
        torch.cuda.synchronize()

        def work(t):
            try:
                stream = torch.cuda.Stream()
                with torch.cuda.stream(stream):
                    pending = []
                    for i, C in enumerate(sizes[t]):
                        pending.append((*ctx.submit(server, J[:C], n[:C]), C))
                        if i % 5 == 4:
                            server.cancel(pending[-1][0])
                        if i % 7 == 6:
                            server.stats()
                    for ticket, out, C in pending:
                        try:
                            server.wait(ticket)
                        except DustError as e:
                            assert "cancelled" in str(e)
                            with lock:
                                counts[1] += 1
                            continue
                        with lock:
                            counts[0] += 1
                        for k in ("T", "L", "resid", "flags"):
                            assert torch.equal(out[k], want[k][:C]), (k, C)
            except Exception as e:  # noqa: BLE001  (reported by the test's thread)
                failed.append(e)

        every = [threading.Thread(target=work, args=(t,)) for t in range(threads)]
        for th in every:
            th.start()
        for th in every:
            th.join()
        s = server.stats()
    assert not failed, failed
    assert sum(counts) == threads * each and (s["completed"], s["cancelled"], s["failed"]) == (counts[0], counts[1], 0)
