"""The bit-sliced client walk (csrc/scan_tile.cuh) against the oracle's scan, bit-exact, where it can go wrong.

The walk is taken for launches of many (client, individual) pairs, so small instances get large populations.  Edges:
rows shorter than, equal to and just past a 32-rank block and past a superblock of 96 or 224 ranks; clients that do
not fill a unit of 32/G; populations that do not fill a word or a tile; bitsets with too few, too many and no open
facilities (unchecked calls, bounded by the row); distances near 2^31, whose sums leave 32 bits after one unit.
"""

import numpy as np
import pytest

import oracle
from paper_1610_10061_gb300.inputs import random_masks

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def pm():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1610_10061_gb300 import build

    build.build()
    from paper_1610_10061_gb300 import pm as _pm

    torch.cuda.set_device(0)
    return _pm


def _distances(n, m, top, seed):
    return np.random.default_rng(seed).integers(0, top, size=(n, m), endpoint=True).astype(np.int32)


def _bounded_scan(pi, delta, masks):
    """The scan of Section 4.2 ended at the row's end: a client without an open facility in its row adds nothing."""
    dist = delta.astype(np.int64).cumsum(axis=1)
    out = np.zeros(masks.shape[0], dtype=np.int64)
    for t, row in enumerate(masks):
        opened = np.unpackbits(row.view(np.uint8), bitorder="little")[pi]
        first = opened.argmax(axis=1)
        out[t] = np.where(opened.any(axis=1), np.take_along_axis(dist, first[:, None], axis=1)[:, 0], 0).sum()
    return out


# n, m, p, pop: L = m - p + 1 at and around block (32) and superblock (96, 224) edges
SHAPES = [(97, 36, 5, 32768 + 7), (64, 36, 4, 40000), (65, 100, 5, 32768 + 33), (33, 101, 5, 50003),
          (129, 228, 5, 16385), (257, 500, 6, 9999), (2500, 61, 7, 1025), (700, 9, 8, 4000), (300, 1100, 9, 9001)]


@pytest.mark.parametrize("cumulative", [False, True])
@pytest.mark.parametrize("n,m,p,pop", SHAPES)
def test_costs_equal_the_oracle(pm, n, m, p, pop, cumulative):
    d = _distances(n, m, 50, seed=n + m)
    inst = pm.Instance(d, p, cumulative=cumulative)
    masks = random_masks(pop, m, p, seed=pop)
    want = oracle.eval_scan(*oracle.tables(d, p), masks)
    np.testing.assert_array_equal(inst.eval(masks), want)
    for groups in (1, 2, 4):
        inst.set_shape(pop, groups=groups, warps=8, splits=3)
        np.testing.assert_array_equal(inst.eval(masks), want, err_msg=f"G={groups}")
    inst.close()


@pytest.mark.parametrize("m,p", [(100, 5), (230, 40), (70, 3)])
def test_bitsets_that_are_no_p_subsets_get_the_bounded_scan(pm, m, p):
    n, pop = 120, 20011
    d = _distances(n, m, 1000, seed=3)
    rng = np.random.default_rng(5)
    masks = random_masks(pop, m, p, seed=6)
    for t in range(0, pop, 3):
        k = int(rng.integers(0, p)) if t % 2 else min(m, p + int(rng.integers(1, 20)))
        masks[t] = random_masks(1, m, k, seed=t)[0] if k else 0
    inst = pm.Instance(d, p)
    np.testing.assert_array_equal(inst.eval(masks), _bounded_scan(*oracle.tables(d, p), masks))
    inst.close()


@pytest.mark.parametrize("top", [2**31 - 1, 2**29, 2**26])
def test_sums_past_32_bits(pm, top):
    n, m, p, pop = 4000, 90, 4, 1500
    d = np.random.default_rng(8).integers(top - top // 8, top, size=(n, m), endpoint=True).astype(np.int32)
    masks = random_masks(pop, m, p, seed=9)
    inst = pm.Instance(d, p)
    np.testing.assert_array_equal(inst.eval(masks), oracle.eval_scan(*oracle.tables(d, p), masks))
    inst.close()
