"""Rows that the bucket sort leaves to the radix sort: none, a few of them, more than it goes on for, and all, by distances
past 16 bits and by crowded ones, on instances that want 16-bit distances and on ones that do not, with more rows than
CTAs; negative distances among them."""
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


def _rows(kind, every, n, m):
    d = np.random.default_rng(n + m).integers(0, 60000, size=(n, m))
    which = np.arange(0, n, every) if every else np.array([], dtype=int)
    if kind == "past16":
        d[which, which % m] = 65536 + which
    else:
        d[which] = np.random.default_rng(2).integers(0, 20, size=(len(which), m))
        d[which, m // 3] = 65535
    return np.ascontiguousarray(d, dtype=np.int32)


@pytest.mark.parametrize("cumulative", [False, True])
@pytest.mark.parametrize("kind", ["past16", "crowded"])
@pytest.mark.parametrize("every", [0, 1, 5, 31, 33, 1000, 2999])
@pytest.mark.parametrize("n,m,p", [(3001, 300, 3), (3000, 301, 60)])
def test_tables_and_costs(pm, n, m, p, every, kind, cumulative):
    d = _rows(kind, every, n, m)
    pi, delta = oracle.tables(d, p)
    inst = pm.Instance(d, p, cumulative=cumulative)
    gpi, gde = inst.tables()
    np.testing.assert_array_equal(gpi, pi)
    np.testing.assert_array_equal(gde, delta)
    masks = random_masks(700, m, p, seed=1)
    np.testing.assert_array_equal(inst.eval(masks), oracle.eval_scan(pi, delta, masks))
    inst.close()


@pytest.mark.parametrize("p", [3, 60])
@pytest.mark.parametrize("row", [0, 1777, 2999])
def test_a_negative_distance_is_found_wherever_it_is(pm, row, p):
    for every in (0, 1):
        d = _rows("past16", every, 3000, 300)
        d[row, 299] = -1
        with pytest.raises(pm.PMError) as e:
            pm.Instance(d, p)
        assert e.value.status == 2
