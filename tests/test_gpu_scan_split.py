"""The rank-split client walk (csrc/scan_split.cuh) against the oracle's scan, bit-exact, where it can go wrong.

Small launches take it.  Edges: rows shorter than, equal to and just past one and two 64-rank blocks; clients that do
not fill the warps or a warp's 4/G; populations that do not fill a word or a tile; bitsets with too few or too many
open facilities; distances whose 32-bit sums would overflow (the client walk takes those).
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


@pytest.mark.parametrize("cumulative", [False, True])
@pytest.mark.parametrize("n,m,p,pop", [(1, 66, 4, 5), (7, 67, 4, 33), (129, 68, 4, 64), (131, 131, 4, 65),
                                       (250, 132, 4, 128), (901, 133, 4, 129), (33, 12, 11, 300), (300, 700, 2, 255)])
def test_costs_equal_the_oracle(pm, n, m, p, pop, cumulative):
    d = np.random.default_rng(n + m).integers(0, 70000, size=(n, m), endpoint=True).astype(np.int32)
    masks = random_masks(pop, m, p, seed=pop)
    want = oracle.eval_scan(*oracle.tables(d, p), masks)
    inst = pm.Instance(d, p, cumulative=cumulative)
    np.testing.assert_array_equal(inst.eval(masks), want)
    for groups in (1, 2, 4):
        for warps, splits in ((32, 1), (3, 2)):
            inst.set_shape(pop, groups=groups, warps=warps, splits=splits)
            np.testing.assert_array_equal(inst.eval(masks), want, err_msg=f"G={groups} warps={warps} splits={splits}")
    inst.close()


def test_bitsets_that_are_no_p_subsets_get_the_bounded_scan(pm):
    n, m, p, pop = 77, 140, 9, 200
    d = np.random.default_rng(3).integers(0, 1000, size=(n, m)).astype(np.int32)
    masks = random_masks(pop, m, p, seed=6)
    for t in range(0, pop, 3):
        k = t % p if t % 2 else p + t % 20
        masks[t] = random_masks(1, m, k, seed=t)[0] if k else 0
    pi, delta = oracle.tables(d, p)
    dist = delta.astype(np.int64).cumsum(axis=1)
    want = np.zeros(pop, dtype=np.int64)
    for t, row in enumerate(masks):  # a client without an open facility in its row adds nothing
        opened = np.unpackbits(row.view(np.uint8), bitorder="little")[pi]
        first = opened.argmax(axis=1)
        want[t] = np.where(opened.any(axis=1), np.take_along_axis(dist, first[:, None], axis=1)[:, 0], 0).sum()
    inst = pm.Instance(d, p)
    np.testing.assert_array_equal(inst.eval(masks), want)
    inst.close()


@pytest.mark.parametrize("top", [2**31 - 1, 2**27])
def test_sums_at_the_edge_of_32_bits(pm, top):
    n, m, p, pop = 1000, 90, 4, 70
    d = np.random.default_rng(8).integers(top - 1000, top, size=(n, m), endpoint=True).astype(np.int32)
    masks = random_masks(pop, m, p, seed=9)
    want = oracle.eval_scan(*oracle.tables(d, p), masks)
    inst = pm.Instance(d, p)
    np.testing.assert_array_equal(inst.eval(masks), want)
    for warps, splits in ((1, 1), (32, 1), (32, 8)):
        inst.set_shape(pop, groups=2, warps=warps, splits=splits)
        np.testing.assert_array_equal(inst.eval(masks), want)
    inst.close()
