"""Calls of different sizes from several threads: a kernel's shared-memory limit belongs to the function, so
one call's smaller need must not undercut another's between its limit and its launch."""
import threading

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


# (wavelengths, sizes, cells) of two threads' calls that share a kernel: split solve + emission, fused
# solve + emission, two-kernel emission, grain-major GEMM of short and long tiles, cell-major GEMM
PAIRS = {"split": ((200, 16, 9, True), (200, 16, 1100, True)), "fused": ((100, 16, 16000, True), (200, 16, 16000, True)),
         "two kernels": ((100, 16, 64, False), (200, 16, 64, False)), "cell-major": ((64, 80, 64, True), (64, 100, 64, True))}


@pytest.mark.parametrize("pair", PAIRS)
def test_threads_with_calls_of_different_sizes(pair):
    from paper_0907_3768_gb300 import Context, padded_rows

    failed = []
    go = threading.Barrier(2)

    def work(K, sizes, C, fused_emit):
        try:
            wl = synth.make_workload(dict(synth.CONFIGS[0], K=K, n_sizes=sizes, n_cells=C, seed=37))
            J, n = padded_rows(torch.from_numpy(wl.J).cuda()), torch.from_numpy(wl.n).cuda()
            with torch.cuda.stream(torch.cuda.Stream()), Context.from_workload(wl, precision="bf16x3") as ctx:
                ctx.set_fused_emit(fused_emit)
                torch.cuda.synchronize()
                out = ctx.solve(J, n)
                want = {k: out[k].clone() for k in ("T", "L", "resid", "flags")}
                go.wait(60.0)
                for _ in range(10000):
                    ctx.solve(J, n, out=out)
                torch.cuda.current_stream().synchronize()
                assert ctx.check() == 0
                for k, v in want.items():
                    assert torch.equal(out[k], v), k
        except Exception as e:  # noqa: BLE001  (reported by the test's thread)
            failed.append(e)
            go.abort()

    threads = [threading.Thread(target=work, args=a) for a in PAIRS[pair]]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failed, failed
