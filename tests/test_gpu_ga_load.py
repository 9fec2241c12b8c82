"""A GA state whose deme bests are no p-subsets (the header of pm_ga_load does not refuse one): the scans' terms, which are
bounded by the rows and ignore bits from m on, whichever kernels the GA would take for its own states."""
import numpy as np
import pytest

from paper_1610_10061_gb300.inputs import euclid_instance

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pm():
    from paper_1610_10061_gb300 import build
    build.build()
    from paper_1610_10061_gb300 import pm as _pm
    torch.cuda.set_device(0)
    return _pm


def _edit(rows, how, m):
    if how == "bits from m on":
        rows[:, -1] |= np.uint32(0xFFFFFFFF) << np.uint32(m % 32)
    elif how == "fewer":
        for r in rows[::2]:
            w = int(np.flatnonzero(r)[0])
            r[w] &= r[w] - np.uint32(1)
    elif how == "none":
        rows[1] = 0
    elif how == "more":
        rows[:, 0] |= np.uint32(0x00F0F00F)


@pytest.mark.parametrize("migration", ["deme", "team"])
@pytest.mark.parametrize("how", ["as saved", "bits from m on", "fewer", "none", "more"])
def test_loaded_states_run_as_the_phases_run_them(pm, monkeypatch, how, migration):
    n, m, p, P, D = 90, 75, 6, 256, 32
    d = euclid_instance(100, seed=1)[:n, :m].copy()
    inst = pm.Instance(d, p)
    ga = pm.GA(inst, seed=3, pop=P, deme=D, migration=migration)
    ga.step(2)
    blob = bytearray(ga.save())
    ga.close()
    W, NB = (m + 31) // 32, P // D
    head = len(blob) - (NB * W * 4 + NB * 8 + W * 4 + P * W * 4 + P * 8)
    rows = np.frombuffer(blob, dtype=np.uint32, count=NB * W, offset=head).reshape(NB, W).copy()
    assert (np.unpackbits(rows.view(np.uint8), axis=1).sum(axis=1) == p).all()
    _edit(rows, how, m)
    blob[head:head + NB * W * 4] = rows.tobytes()
    out = []
    for deme in ("1", "0"):
        monkeypatch.setenv("PM_GA_DEME", deme)
        ga = pm.GA.load(inst, bytes(blob))
        assert (ga.info()["kernels_per_generation"] == 1) == (deme == "1" and how == "as saved")
        trace = ga.step(3)
        masks, costs = ga.population()
        out.append((trace, masks, costs, ga.result()))
        ga.close()
    for a, b in zip(out[0][:3], out[1][:3]):
        np.testing.assert_array_equal(a, b)
    assert out[0][3][:3] == out[1][3][:3]
    inst.close()
