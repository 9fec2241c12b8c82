"""Instances of different widths created by several host threads at once: every creation succeeds, with its own tables."""
import threading

import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("top", [60000, 2**20])  # the bucket sort; the radix sort after it
def test_widths_do_not_disturb_each_other(top):
    from paper_1610_10061_gb300 import build
    build.build()
    from paper_1610_10061_gb300 import pm
    torch.cuda.set_device(0)
    rng = np.random.default_rng(1)
    data = [rng.integers(0, top, size=(16, m)).astype(np.int32) for m in (90, 2000, 14000, 19000)]
    dev = [torch.from_numpy(d).cuda() for d in data]
    failures, start = [], threading.Barrier(len(data))

    def create(k):
        torch.cuda.set_device(0)
        d, p = data[k], 5
        L = d.shape[1] - p + 1
        pi = torch.empty(16, L, dtype=torch.int16, device="cuda")
        delta = torch.empty(16, L, dtype=torch.int32, device="cuda")
        want = oracle.tables(d, p)
        start.wait()
        try:
            for i in range(300):
                inst = pm.Instance(dev[k], p)
                if i % 100 == 99:
                    pm.pm_instance_tables(inst.handle, pi, delta)
                    np.testing.assert_array_equal(pi.cpu().numpy().view(np.uint16), want[0])
                    np.testing.assert_array_equal(delta.cpu().numpy(), want[1])
                inst.close()
        except Exception as e:  # noqa: BLE001
            failures.append((k, i, e))

    threads = [threading.Thread(target=create, args=(k,)) for k in range(len(data))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failures, failures
