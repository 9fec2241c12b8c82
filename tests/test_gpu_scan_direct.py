"""The evaluation by open facilities (csrc/scan_direct.cuh) against the oracle, bit-exact, where it can go wrong.

It is taken where p is far below the expected first open rank (m + 1) / (p + 1), every distance is below 2^16 and the
launch has many (client, individual) pairs, so the instances here have few open facilities and large populations.
Edges: odd and even p, p = 1, odd m, clients that do not fill a chunk of eight, populations that do not fill a word
or pass one work item's range, distances at 2^16 - 1 and just past it (where the scan takes over), bitsets that are no
p-subsets, GAs and batches whose instances take different ways.
"""

import numpy as np
import pytest

import oracle
from paper_1610_10061_gb300.inputs import euclid_instance, graph_instance, random_masks

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
    yield _pm
    _pm.pm_debug_scan_timeout(0)


def _distances(n, m, top, seed):
    return np.random.default_rng(seed).integers(0, top, size=(n, m), endpoint=True).astype(np.int32)


SHAPES = [(70, 500, 3, 20000), (65, 501, 4, 20001), (33, 257, 1, 40000), (9, 400, 2, 131073), (2003, 300, 5, 1025),
          (640, 1999, 7, 4097), (64, 130, 3, 32)]


@pytest.mark.parametrize("cumulative", [False, True])
@pytest.mark.parametrize("n,m,p,pop", SHAPES)
def test_costs_equal_the_oracle(pm, n, m, p, pop, cumulative):
    d = _distances(n, m, 60000, seed=n + m)
    masks = random_masks(pop, m, p, seed=pop)
    inst = pm.Instance(d, p, cumulative=cumulative)
    want = oracle.eval_scan(*oracle.tables(d, p), masks)
    np.testing.assert_array_equal(inst.eval(masks), want)
    dm = torch.from_numpy(masks.view(np.int32)).cuda()
    costs = torch.empty(pop, dtype=torch.int64, device="cuda")
    G, words = pm.pm_columns_layout(inst.handle, pop)  # the facility-major form stays the scan's
    cols = torch.empty(words, dtype=torch.int32, device="cuda")
    pm.pm_population_columns(inst.handle, dm, pop, cols)
    pm.pm_eval_columns(inst.handle, cols, pop, costs)
    np.testing.assert_array_equal(costs.cpu().numpy(), want)
    inst.close()


@pytest.mark.parametrize("top", [65535, 65536, 2**31 - 1])
def test_distances_at_and_past_16_bits(pm, top):
    n, m, p, pop = 2500, 300, 3, 1500
    d = np.random.default_rng(1).integers(top - 40, top, size=(n, m), endpoint=True).astype(np.int32)
    masks = random_masks(pop, m, p, seed=2)
    inst = pm.Instance(d, p)
    np.testing.assert_array_equal(inst.eval(masks), oracle.eval_scan(*oracle.tables(d, p), masks))
    inst.close()


def test_bitsets_that_are_no_p_subsets_get_the_bounded_scan(pm):
    n, m, p, pop = 120, 301, 3, 20011
    d = _distances(n, m, 1000, seed=3)
    rng = np.random.default_rng(5)
    masks = random_masks(pop, m, p, seed=6)
    for t in range(0, pop, 37):
        k = int(rng.integers(0, p)) if t % 2 else p + int(rng.integers(1, 20))
        masks[t] = random_masks(1, m, k, seed=t)[0] if k else 0
    masks[5, -1] |= np.uint32(1) << np.uint32(31)  # a bit past m is ignored by the scan
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


def test_a_launch_that_gives_up_is_reported_and_the_next_one_is_exact(pm):
    n, m, p, pop = 2500, 300, 3, 1500
    d = euclid_instance(n, seed=2)[:, :m].copy()
    masks = random_masks(pop, m, p, seed=11)
    inst = pm.Instance(d, p)
    want = oracle.eval_scan(*oracle.tables(d, p), masks)
    pm.pm_debug_scan_timeout(1)
    with pytest.raises(pm.PMError) as e:
        inst.eval(masks)
    assert e.value.status == 7
    assert pm.pm_debug_scan_timeout(0) == 0
    for _ in range(2):
        np.testing.assert_array_equal(inst.eval(masks), want)
    inst.close()


def test_ga_generations_equal_the_oracle(pm):
    n, m, p, pop = 2000, 600, 12, 1024
    d = euclid_instance(n, seed=4)[:, :m].copy()
    pi, de = oracle.tables(d, p)
    st, trace, pops, costs = oracle.ga_run(pi, de, m, p, seed=3, P=pop, gens=2, record=True)
    inst = pm.Instance(d, p)
    ga = pm.GA(inst, seed=3, pop=pop)
    for g in range(2):
        np.testing.assert_array_equal(ga.step(1), trace[g:g + 1])
        gm, gc = ga.population()
        np.testing.assert_array_equal(gm, pops[g])
        np.testing.assert_array_equal(gc, costs[g])
    best, gens, evals, mask = ga.result()
    assert best == st.best_cost and evals == st.evals and gens == 2
    np.testing.assert_array_equal(mask, st.best)
    ga.close()
    inst.close()


@pytest.mark.parametrize("spec", [False, True])
def test_batches_of_both_ways(pm, monkeypatch, spec):
    """Instances evaluated by open facilities (few of them) beside scanned ones, in one launch."""
    if spec:
        monkeypatch.setenv("PM_GA_SPEC", "1")
    data = [(euclid_instance(700, seed=1), 3), (graph_instance(600, 2400, seed=2), 60),
            (euclid_instance(300, seed=3), 30), (euclid_instance(900, seed=5)[:, :801].copy(), 5)]
    insts = [pm.Instance(d, p, cumulative=k == 3) for k, (d, p) in enumerate(data)]
    batch = pm.Batch(insts)
    pops = [1500, 700, 31, 2049]
    masks = [random_masks(P, d.shape[1], p, seed=k) for k, ((d, p), P) in enumerate(zip(data, pops))]
    dev = torch.from_numpy(np.concatenate([mk.reshape(-1) for mk in masks]).view(np.int32)).cuda()
    got = batch.eval(dev, pops).cpu().numpy()
    off = 0
    for (d, p), mk, P in zip(data, masks, pops):
        np.testing.assert_array_equal(got[off:off + P], oracle.eval_scan(*oracle.tables(d, p), mk))
        off += P
    ga = batch.ga(seed=9, pop=1024, deme=64, stream_id=2)
    ga.step(2)
    for k, (inst, (d, _)) in enumerate(zip(insts, data)):
        alone = pm.GA(inst, seed=9, pop=1024, deme=64, stream_id=2 + k)
        alone.step(2)
        m0, c0 = ga.population(k)
        m1, c1 = alone.population()
        np.testing.assert_array_equal(m0, m1)
        np.testing.assert_array_equal(c0, c1)
        np.testing.assert_array_equal(c0[:64], oracle.eval_direct(d, m0[:64]))
        assert ga.result(k)[:3] == alone.result()[:3]
        alone.close()
    ga.close()
    batch.close()


@pytest.mark.parametrize("m,p,ids", [(1500, 16, None), (1500, 17, None), (4000, 33, None), (4001, 60, None),
                                     (4000, 33, "one class"), (4000, 45, "two classes"), (4000, 40, "last words")])
def test_lists_ordered_for_the_banks(pm, m, p, ids):
    """From 16 open facilities on the lists are ordered by the ids mod 8: random subsets, and subsets whose ids crowd a
    class (most of them then fill holes) or a few words."""
    n, pop = 700, 1100
    rng = np.random.default_rng(m + p)
    pool = {None: np.arange(m), "one class": np.arange(5, m, 8), "two classes": np.arange(m)[np.arange(m) % 8 < 2],
            "last words": np.arange(m - 64, m)}[ids]
    masks = np.zeros((pop, (m + 31) // 32), dtype=np.uint32)
    for t in range(pop):
        for j in rng.choice(pool if t % 3 else np.arange(m), size=p, replace=False):
            masks[t, j >> 5] |= np.uint32(1) << np.uint32(j & 31)
    d = _distances(n, m, 65535, seed=p)
    inst = pm.Instance(d, p)
    np.testing.assert_array_equal(inst.eval(masks), oracle.eval_direct(d, masks))
    inst.close()
