"""A launch by open facilities with two stages of copies whose waits run out: the error is reported, asynchronous calls
leave it for pm_eval_status, and the next launches are exact (accumulators and stages start clean)."""
import numpy as np
import pytest

import oracle
from paper_1610_10061_gb300.inputs import random_masks

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
PM_ERR_TIMEOUT = 7


@pytest.mark.parametrize("n,m,p,pop", [(3001, 400, 4, 3000), (900, 1300, 9, 4096)])  # many chunks a CTA; few
def test_two_stages(n, m, p, pop):
    from paper_1610_10061_gb300 import build
    build.build()
    from paper_1610_10061_gb300 import pm
    torch.cuda.set_device(0)
    d = np.random.default_rng(n).integers(0, 65536, size=(n, m)).astype(np.int32)
    masks = random_masks(pop, m, p, seed=1)
    want = oracle.eval_scan(*oracle.tables(d, p), masks)
    inst = pm.Instance(d, p)
    dev = torch.from_numpy(masks.view(np.int32)).cuda()
    costs = torch.empty(pop, dtype=torch.int64, device="cuda")
    for _ in range(2):
        before = pm.pm_debug_scan_launches()["direct"]
        pm.pm_debug_scan_timeout(1)
        pm.pm_eval_population(inst.handle, dev, pop, costs)
        assert pm.pm_debug_scan_launches()["direct"] == before + 1
        assert pm.pm_debug_scan_timeout(0) == 0
        assert pm.pm_eval_status(inst.handle) == PM_ERR_TIMEOUT
        for _ in range(2):
            pm.pm_eval_population(inst.handle, dev, pop, costs)
            np.testing.assert_array_equal(costs.cpu().numpy(), want)
        assert pm.pm_eval_status(inst.handle) == 0
    inst.close()
