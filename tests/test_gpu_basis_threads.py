"""Harmonic basis from several threads at once: calls whose blocks take different amounts of shared memory
share a kernel, and its limit."""
import threading

import pytest
import torch

hsma = pytest.importorskip("paper_1806_04801_gb300.hsma")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("calls", [((40, 100), (30, 100)), ((20, 200), (20, 30_000)), ((12, 100), (4, 100))])
def test_calls_of_several_sizes_at_once(calls, precision):
    g = torch.Generator(device="cuda")
    g.manual_seed(7)
    x = torch.rand((30_000, 3), generator=g, device="cuda", dtype=torch.float64) - 0.5
    want = {c: hsma.basis(x[:c[1]], c[0], 1.5, precision=precision) for c in calls}
    torch.cuda.synchronize()
    failed = []

    def work(c):
        p, n = c
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                for k in range(1000):
                    got = hsma.basis(x[:n], p, 1.5, precision=precision)
                    if k % 100 == 0 and not torch.equal(got, want[c]):
                        failed.append("values")
        except Exception as e:  # reported below, in the test's own thread
            failed.append(repr(e))

    threads = [threading.Thread(target=work, args=(c,)) for c in calls * 4]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failed, failed[:3]
