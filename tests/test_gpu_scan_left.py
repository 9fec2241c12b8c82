"""Bitsets of other sizes than p where the evaluation by open facilities is taken (csrc/scan_direct.cuh), bit-exact: a CTA
gathers them into tiles of 64 or 128 and scans, so none, one, a tile's worth and one more of them, scattered and all of
them, sets of more than p (whose cost is the p-median objective) and of fewer (bounded by the row), wide rows (64 a
tile), odd sizes, and a batch with both kinds of instances."""
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


def _distances(n, m, seed):
    return np.random.default_rng(seed).integers(0, 65536, size=(n, m)).astype(np.int32)


def _bounded(d, p, masks):
    """The scan ended at the row's end: a client without an open facility in its row adds nothing."""
    pi, delta = oracle.tables(d, p)
    dist = delta.astype(np.int64).cumsum(axis=1)
    out = np.zeros(len(masks), dtype=np.int64)
    for t, row in enumerate(masks):
        opened = np.unpackbits(row.view(np.uint8), bitorder="little")[pi]
        first = opened.argmax(axis=1)
        out[t] = np.where(opened.any(axis=1), np.take_along_axis(dist, first[:, None], axis=1)[:, 0], 0).sum()
    return out


def _resize(masks, which, m, sizes, seed):
    rng = np.random.default_rng(seed)
    for t in which:
        k = int(rng.choice(sizes))
        masks[t] = random_masks(1, m, k, seed=seed + int(t))[0] if k else 0
    return masks


SHAPES = [(301, 700, 4, 9000, False), (67, 2011, 9, 40003, True), (129, 12500, 3, 17000, False)]  # n, m, p, pop, cumulative


@pytest.mark.parametrize("count", [1, 129, 700, "all"])
@pytest.mark.parametrize("n,m,p,pop,cum", SHAPES)
def test_larger_sets_get_the_objective(pm, n, m, p, pop, cum, count):
    assert -(-n // 32) * -(-pop // 32) >= 12 * torch.cuda.get_device_properties(0).multi_processor_count
    d = _distances(n, m, seed=n)
    if count == "all":
        masks = random_masks(pop, m, 2 * p, seed=1)
    else:
        which = np.random.default_rng(count).choice(pop, size=count, replace=False)
        masks = _resize(random_masks(pop, m, p, seed=1), which, m, [p + 1, 3 * p, m // 3], seed=count)
    want = oracle.eval_scan(*oracle.tables(d, p), masks)  # the first open rank exists: the objective
    np.testing.assert_array_equal(want[::200], oracle.eval_direct(d, masks[::200]))
    inst = pm.Instance(d, p, cumulative=cum)
    dev = torch.from_numpy(masks.view(np.int32)).cuda()
    for _ in range(2):
        before = pm.pm_debug_scan_launches()["direct"]
        got = inst.eval(dev).cpu().numpy()
        assert pm.pm_debug_scan_launches()["direct"] == before + 1
        np.testing.assert_array_equal(got, want)
    inst.close()


def test_smaller_sets_are_bounded_by_the_row(pm):
    n, m, p, pop = 157, 500, 6, 13001
    d = _distances(n, m, seed=3)
    masks = _resize(random_masks(pop, m, p, seed=5), range(0, pop, 11), m, [0, 1, p - 1, p + 2, m], seed=9)
    masks[7, -1] |= np.uint32(1) << np.uint32(31)  # past m: ignored
    inst = pm.Instance(d, p)
    before = pm.pm_debug_scan_launches()["direct"]
    got = inst.eval(masks)
    assert pm.pm_debug_scan_launches()["direct"] == before + 1
    np.testing.assert_array_equal(got, _bounded(d, p, masks))
    inst.close()


def test_in_a_batch_beside_scanned_instances(pm):
    shapes, pops = [(900, 600, 4), (700, 310, 40), (203, 1999, 5)], [3000, 2000, 1037]
    data = [_distances(n, m, seed=k) for k, (n, m, _) in enumerate(shapes)]
    insts = [pm.Instance(d, s[2]) for d, s in zip(data, shapes)]
    batch = pm.Batch(insts)
    masks = [_resize(random_masks(P, s[1], s[2], seed=k), range(k, P, 3), s[1], [s[2] - 1, s[2] + 3], seed=k)
             for k, (s, P) in enumerate(zip(shapes, pops))]
    dev = torch.from_numpy(np.concatenate([mk.reshape(-1) for mk in masks]).view(np.int32)).cuda()
    before = pm.pm_debug_scan_launches()["mixed"]
    got = batch.eval(dev, pops).cpu().numpy()
    assert pm.pm_debug_scan_launches()["mixed"] == before + 1
    np.testing.assert_array_equal(got, np.concatenate([_bounded(d, s[2], mk) for d, s, mk in zip(data, shapes, masks)]))
    batch.close()
