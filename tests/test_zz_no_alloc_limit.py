"""Which populations the evaluation without allocation takes: those whose tiles of up to 128 individuals, tickets and sums fit
in its 8 MiB, whatever the way their evaluation takes; at the last size that fits and the first that does not, exact."""
import numpy as np
import pytest

import oracle
from paper_1610_10061_gb300.inputs import random_masks

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
PM_ERR_INVALID_ARG = 1


def _fits(m, p, pop):
    W = (m + 31) // 32
    G, least = 4, 16 if m + 1 < 32 * (p + 1) else 8
    while G > 1 and pop <= 32 * (G // 2) * least:
        G //= 2
    up = lambda x: -(-x // 256) * 256  # noqa: E731
    tiles = -(-pop // (32 * G))
    return 256 + up(tiles * 4) + up(tiles * W * 128 * G) + up(pop * 8) <= 8 << 20


# rank-split tiles of 32 and 64 individuals, which have more tickets; bit-sliced and by open facilities
@pytest.mark.parametrize("n,m,p", [(100, 3968, 5), (100, 3968, 400), (300, 3968, 90), (40, 70, 6), (2000, 500, 100),
                                   (2000, 500, 3)])
def test_last_size_that_fits(n, m, p):
    from paper_1610_10061_gb300 import build
    build.build()
    from paper_1610_10061_gb300 import pm
    torch.cuda.set_device(0)
    d = np.random.default_rng(n + m).integers(0, 60000, size=(n, m)).astype(np.int32)
    inst = pm.Instance(d, p)
    most = max(pop for pop in range(1, 1 << 20) if _fits(m, p, pop))
    masks = np.tile(random_masks(997, m, p, seed=1), (most // 997 + 2, 1))
    dev = torch.from_numpy(masks.view(np.int32)).cuda()
    want = oracle.eval_direct(d, masks[:997])
    for pop in (most, most - 127, most - 33):
        costs = torch.full((pop,), -1, dtype=torch.int64, device="cuda")
        pm.pm_eval_population_noalloc(inst.handle, dev, pop, costs)
        np.testing.assert_array_equal(costs.cpu().numpy(), np.resize(want, pop))
    with pytest.raises(pm.PMError) as e:
        pm.pm_eval_population_noalloc(inst.handle, dev, most + 1, torch.empty(most + 1, dtype=torch.int64, device="cuda"))
    assert e.value.status == PM_ERR_INVALID_ARG
    inst.close()
