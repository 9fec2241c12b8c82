"""The ways of scanning at the edges of their tiles, with the launch's own record of which one it took (sizes follow from
the number of SMs, so that a rule that moves fails here and does not reroute a test): the bit-sliced walk around its
32-rank blocks, its superblocks of 96 and 224 ranks and each tile width, and the lists of open facilities in an order
that suits the banks, with more ids of a class than a warp's holes."""
import numpy as np
import pytest

import oracle
from paper_1610_10061_gb300.inputs import random_masks

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pm():
    from paper_1610_10061_gb300 import build
    build.build()
    from paper_1610_10061_gb300 import pm as _pm
    torch.cuda.set_device(0)
    return _pm


def _population(n, per_sm, extra):
    """Individuals for `per_sm` units of 1024 pairs per SM on n clients, and `extra` more."""
    sm = torch.cuda.get_device_properties(0).multi_processor_count
    return 32 * -(-per_sm * sm // -(-n // 32)) + extra


def _eval(pm, kind, inst, masks):
    before = pm.pm_debug_scan_launches()
    got = inst.eval(masks)
    now = pm.pm_debug_scan_launches()
    assert {k for k in now if now[k] != before[k]} == {kind}, (kind, before, now)
    return got


def _distances(n, m, seed):
    d = np.random.default_rng(seed).integers(0, 50, size=(n, m)).astype(np.int32)
    d[0, 0] = 70000  # past 16 bits: never by open facilities
    return d


# n, m, p, individuals past whole words: L = m - p + 1 at and around 32, 96 and 224; tables of one, three and seven blocks
SLICED = [(97, 36, 5, 7), (64, 36, 4, 0), (65, 100, 5, 33), (33, 101, 5, 3), (129, 228, 5, 1), (257, 500, 6, 15),
          (2500, 61, 7, 1), (700, 9, 8, 31), (300, 1100, 9, 9), (310, 200, 60, 2)]


@pytest.mark.parametrize("cumulative", [False, True])
@pytest.mark.parametrize("n,m,p,extra", SLICED)
def test_sliced(pm, n, m, p, extra, cumulative):
    pop = _population(n, 24, extra)
    d = _distances(n, m, seed=n + m)
    inst = pm.Instance(d, p, cumulative=cumulative)
    masks = random_masks(pop, m, p, seed=extra)
    want = oracle.eval_scan(*oracle.tables(d, p), masks)
    np.testing.assert_array_equal(_eval(pm, "sliced", inst, masks), want)
    for groups in (1, 2, 4):
        inst.set_shape(pop, groups=groups, warps=8, splits=3)
        np.testing.assert_array_equal(_eval(pm, "sliced", inst, masks), want, err_msg=f"G={groups}")
    inst.close()


@pytest.mark.parametrize("m,p", [(100, 5), (230, 40), (260, 3)])
def test_sliced_sets_of_other_sizes(pm, m, p):
    n = 120
    pop = _population(n, 24, 11)
    d = _distances(n, m, seed=3)
    rng = np.random.default_rng(5)
    masks = random_masks(pop, m, p, seed=6)
    for t in range(0, pop, 7):
        k = int(rng.integers(0, p)) if t % 2 else min(m, p + int(rng.integers(1, 20)))
        masks[t] = random_masks(1, m, k, seed=t)[0] if k else 0
    pi, delta = oracle.tables(d, p)
    dist = delta.astype(np.int64).cumsum(axis=1)
    want = np.zeros(pop, dtype=np.int64)
    for t, row in enumerate(masks):  # a client without an open facility in its row adds nothing
        opened = np.unpackbits(row.view(np.uint8), bitorder="little")[pi]
        first = opened.argmax(axis=1)
        want[t] = np.where(opened.any(axis=1), np.take_along_axis(dist, first[:, None], axis=1)[:, 0], 0).sum()
    inst = pm.Instance(d, p)
    np.testing.assert_array_equal(_eval(pm, "sliced", inst, masks), want)
    inst.close()


def _pool(ids, m):
    return {"all": np.arange(m), "one class": np.arange(5, m, 8), "two classes": np.arange(m)[np.arange(m) % 8 < 2],
            "last words": np.arange(m - 70, m)}[ids]


@pytest.mark.parametrize("m,p,ids", [(1500, 16, "all"), (1500, 17, "all"), (4000, 33, "all"), (4001, 60, "all"),
                                     (4000, 33, "one class"), (4001, 60, "one class"), (4000, 45, "two classes"),
                                     (4000, 40, "last words"), (4001, 59, "last words")])
def test_ordered_lists(pm, m, p, ids):
    """A class of 60 ids has 52 more than places of its own: more than the 32 holes that a warp knows at once."""
    n = 700
    pop = _population(n, 12, 5)
    rng = np.random.default_rng(m + p)
    masks = np.zeros((pop, (m + 31) // 32), dtype=np.uint32)
    for t in range(pop):
        pick = rng.choice(_pool(ids if t % 3 else "all", m), size=p, replace=False)
        np.bitwise_or.at(masks[t], pick >> 5, np.uint32(1) << (pick & 31).astype(np.uint32))
    d = rng.integers(0, 65536, size=(n, m)).astype(np.int32)
    inst = pm.Instance(d, p)
    got = _eval(pm, "direct", inst, masks)
    np.testing.assert_array_equal(got, oracle.eval_scan(*oracle.tables(d, p), masks))
    inst.close()
