"""The table build (csrc/tables.cu) against the oracle, bit-exact, where the bucket sort can go wrong.

Rows of equal distances (ties ordered by id through the buckets), a single distance in the matrix, distances crowded
in a small part of their range beside one far away (a bucket too full: those rows go to the radix sort), rows past
2^16 beside rows below it (radix sort of the former only), zero distances, row widths around the CTA sizes, and the
dense copies of either table alone, at odd row lengths, to device and host memory.
"""

import numpy as np
import pytest

import oracle

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


def _matrix(kind, n, m, rng):
    if kind == "uniform":
        return rng.integers(0, 60000, size=(n, m))
    if kind == "ties":
        return rng.integers(0, 4, size=(n, m))
    if kind == "equal":
        return np.full((n, m), 7)
    if kind == "zero":
        return np.zeros((n, m), dtype=np.int64)
    d = rng.integers(0, 30, size=(n, m)) if kind == "crowded" else rng.integers(0, 60000, size=(n, m))
    if kind == "crowded":
        d[:, m // 2] = 65535
    elif kind == "past16":  # every third row beyond 16 bits
        d[::3, 1] = 2**31 - 1
    return d


@pytest.mark.parametrize("cumulative", [False, True])
@pytest.mark.parametrize("kind", ["uniform", "ties", "equal", "zero", "crowded", "past16"])
@pytest.mark.parametrize("n,m,p", [(3, 2, 1), (5, 127, 4), (9, 257, 2), (7, 1024, 100), (6, 1025, 3), (4, 4099, 11),
                                   (3, 12000, 7), (2, 30000, 5)])
def test_tables_equal_the_oracle(pm, kind, n, m, p, cumulative):
    d = np.ascontiguousarray(_matrix(kind, n, m, np.random.default_rng(m)), dtype=np.int32)
    pi, delta = oracle.tables(d, p)
    inst = pm.Instance(d, p, cumulative=cumulative)
    gpi, gde = inst.tables()
    np.testing.assert_array_equal(gpi, pi)
    np.testing.assert_array_equal(gde, delta)
    L = m - p + 1
    dpi = torch.full((n * L + 1,), -1, dtype=torch.int16, device="cuda")
    dde = torch.full((n, L), -1, dtype=torch.int32, device="cuda")
    pm.pm_instance_tables(inst.handle, dpi[1:], None)  # starts at an odd place
    pm.pm_instance_tables(inst.handle, None, dde)
    np.testing.assert_array_equal(dpi[1:].cpu().numpy().view(np.uint16).reshape(n, L), pi)
    assert int(dpi[0]) == -1
    np.testing.assert_array_equal(dde.cpu().numpy(), delta)
    inst.close()
