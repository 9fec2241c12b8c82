"""A batch's launch divided into shares of equal estimated cost (csrc/batch.cu), bit-exact against the oracle, with the
launch's own record that it took them: tiles cut into the shares of several CTAs, CTAs with several tiles, scanned
instances beside ones evaluated by open facilities, sums past the packed reduction, individuals left out by a GA."""
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


def _distances(n, m, top, seed):
    return np.random.default_rng(seed).integers(0, top, size=(n, m), endpoint=True).astype(np.int32)


def _routes(pm, before=None):
    now = pm.pm_debug_scan_launches()
    return now if before is None else {k: now[k] - before[k] for k in now}


def _enough(shapes, pops):
    """Units of 1024 pairs above the line from which a batch is divided into shares (24 per SM)."""
    units = sum(-(-P // 32) * -(-n // 32) for (n, _, _, _), P in zip(shapes, pops))
    return units >= 24 * torch.cuda.get_device_properties(0).multi_processor_count


BATCHES = {  # (n, m, p, largest distance) and individuals of each instance; the kind of launch
    "both ways": ([(1500, 1500, 4, 60000), (600, 610, 60, 3000), (300, 299, 30, 90000), (900, 801, 5, 65535)],
                  [3000, 2500, 31, 2049], "mixed"),
    "several tiles a CTA": ([(60 + k % 50, 64 + k % 37, 3 + k % 9, 500) for k in range(200)], [300] * 200, "sliced"),
    "several CTAs a tile": ([(20003, 64, 6, 1000), (50, 40, 3, 1000)], [256, 33], "sliced"),
    "past 2^47": ([(70001, 40, 4, 2**31 - 1), (97, 90, 7, 2**31 - 1)], [64, 65], "sliced"),
}


@pytest.mark.parametrize("name", BATCHES)
def test_costs_equal_the_oracle(pm, name):
    shapes, pops, kind = BATCHES[name]
    assert _enough(shapes, pops)
    data = [_distances(n, m, top, seed=k) for k, (n, m, _, top) in enumerate(shapes)]
    insts = [pm.Instance(d, s[2], cumulative=k % 3 == 2) for k, (d, s) in enumerate(zip(data, shapes))]
    masks = [random_masks(P, s[1], s[2], seed=P + k) for k, (s, P) in enumerate(zip(shapes, pops))]
    want = np.concatenate([oracle.eval_scan(*oracle.tables(d, s[2]), mk) for d, s, mk in zip(data, shapes, masks)])
    dev = torch.from_numpy(np.concatenate([mk.reshape(-1) for mk in masks]).view(np.int32)).cuda()
    batch = pm.Batch(insts)
    for _ in range(2):  # the second launch finds the accumulators and tickets as the first one left them
        before = _routes(pm)
        got = batch.eval(dev, pops).cpu().numpy()
        taken = _routes(pm, before)
        assert taken[kind] == 1 and taken["shares"] == 1, taken
        np.testing.assert_array_equal(got, want)
    batch.close()
    for inst in insts:
        inst.close()


RULES = {  # shapes, individuals of each, the kind of launch, whether in shares
    "from 12 units per SM on": ([(900, 850, 85, 3000)] * 9, 256, "sliced", 1),
    "one deep walk among short ones": ([(700, 300, 30, 3000)] * 40 + [(290, 6000, 3, 3000)], 128, "split", 0),
    "few units": ([(1000, 1000, 8, 60000), (400, 300, 9, 3000)], 64, "split", 0),
    "populations of one word": ([(700, 200, 20, 500)] * 120, 32, "sliced", 1),
}


@pytest.mark.parametrize("name", RULES)
def test_rule_for_the_way(pm, name):
    shapes, pop, kind, shares = RULES[name]
    sm = torch.cuda.get_device_properties(0).multi_processor_count
    units = sum(-(-pop // 32) * -(-s[0] // 32) for s in shapes)
    assert units < 24 * sm and (units >= 12 * sm) == (name != "few units")
    data = {s: _distances(s[0], s[1], s[3], seed=k) for k, s in enumerate(dict.fromkeys(shapes))}
    insts = {s: pm.Instance(d, s[2]) for s, d in data.items()}
    batch = pm.Batch([insts[s] for s in shapes])
    masks = [random_masks(pop, s[1], s[2], seed=k) for k, s in enumerate(shapes)]
    dev = torch.from_numpy(np.concatenate([mk.reshape(-1) for mk in masks]).view(np.int32)).cuda()
    before = _routes(pm)
    got = batch.eval(dev, [pop] * len(shapes)).cpu().numpy().reshape(len(shapes), pop)
    taken = _routes(pm, before)
    assert taken[kind] == 1 and taken["shares"] == shares, taken
    for k in {0, 1, len(shapes) // 2, len(shapes) - 1}:
        np.testing.assert_array_equal(got[k], oracle.eval_direct(data[shapes[k]], masks[k]))
    batch.close()


@pytest.mark.parametrize("spec", ["0", "1"])
def test_ga_with_individuals_left_out(pm, monkeypatch, spec):
    """Children that are not evaluated (failed crossovers, mutation after an improvement) and instances that stop."""
    monkeypatch.setenv("PM_GA_SPEC", spec)
    shapes, P = [(2000, 500, 5, 60000), (1200, 400, 100, 5000), (650, 600, 6, 2**20)], 1024
    assert _enough(shapes, [P] * 3)
    data = [_distances(n, m, top, seed=7 + k) for k, (n, m, _, top) in enumerate(shapes)]
    insts = [pm.Instance(d, s[2]) for d, s in zip(data, shapes)]
    batch = pm.Batch(insts)
    before = _routes(pm)
    ga = batch.ga(seed=9, pop=P, deme=64, stream_id=2, saturation=1)
    ga.step(4)
    assert _routes(pm, before)["shares"] > 0
    for k, (inst, d) in enumerate(zip(insts, data)):
        alone = pm.GA(inst, seed=9, pop=P, deme=64, stream_id=2 + k, saturation=1)
        alone.step(4)
        m0, c0 = ga.population(k)
        m1, c1 = alone.population()
        np.testing.assert_array_equal(m0, m1)
        np.testing.assert_array_equal(c0, c1)
        np.testing.assert_array_equal(c0, oracle.eval_direct(d, m0))
        assert ga.result(k)[:3] == alone.result()[:3]
        alone.close()
    ga.close()
    batch.close()
