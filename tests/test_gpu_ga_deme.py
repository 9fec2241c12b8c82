"""The kernel over whole demes (a generation of a small instance): demes of a cluster, of one CTA and of less,
a last CTA that is not full, crossover rounds beyond lg D, more tries than a round has lanes, one open facility, both
migration variants -- against the per-phase kernels and the oracle, and with its bounded wait running out."""
import numpy as np
import pytest

import oracle
from paper_1610_10061_gb300.inputs import euclid_instance, graph_instance

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
PM_ERR_TIMEOUT = 7


@pytest.fixture(scope="module")
def pm():
    from paper_1610_10061_gb300 import build
    build.build()
    from paper_1610_10061_gb300 import pm as _pm
    yield _pm
    _pm.pm_debug_scan_timeout(0)


CASES = [  # n x m, p, GA parameters
    (100, 100, 5, dict(pop=64)),
    (100, 100, 5, dict(pop=512)),
    (33, 31, 1, dict(pop=48, deme=16)),
    (129, 64, 7, dict(pop=40, deme=8, xover_rounds=7)),
    (57, 120, 60, dict(pop=256, deme=128, mut_tries=40, migration="team")),
    (8, 200, 20, dict(pop=64, deme=32, xover_rounds=0, saturation=3)),
    (270, 270, 27, dict(pop=512, deme=256, mut_tries=0)),
    (100, 100, 8, dict(pop=1024, deme=512)),
    (264, 65, 2, dict(pop=6, deme=2)),
    (8, 4, 1, dict(pop=4096, deme=2)),
    (5, 7001, 3, dict(pop=64, deme=64)),
]


def _distances(n, m, seed):
    return np.random.default_rng(seed).integers(0, 65536, size=(n, m)).astype(np.int32)


@pytest.mark.parametrize("cumulative", [False, True])
@pytest.mark.parametrize("n,m,p,kw", CASES, ids=[f"{c[0]}x{c[1]}p{c[2]}" + str(c[3]["pop"]) for c in CASES])
def test_equals_the_phases(pm, monkeypatch, n, m, p, kw, cumulative):
    d = _distances(n, m, n + m)
    inst = pm.Instance(d, p, cumulative=cumulative)
    out = []
    for deme in ("1", "0"):
        monkeypatch.setenv("PM_GA_DEME", deme)
        ga = pm.GA(inst, seed=9, **kw)
        assert (ga.info()["kernels_per_generation"] == 1) == (deme == "1")
        traces = [ga.step(k) for k in (3, 1, 4)]
        masks, costs = ga.population()
        out.append((np.concatenate(traces), masks, costs, ga.result()))
        ga.close()
    (ta, ma, ca, ra), (tb, mb, cb, rb) = out
    np.testing.assert_array_equal(ta, tb)
    np.testing.assert_array_equal(ma, mb)
    np.testing.assert_array_equal(ca, cb)
    assert ra[:3] == rb[:3]
    np.testing.assert_array_equal(ra[3], rb[3])
    np.testing.assert_array_equal(ca, oracle.eval_direct(d, ma))
    inst.close()


def test_matches_the_oracle(pm):
    d, p = euclid_instance(150, seed=5), 12
    pi, de = oracle.tables(d, p)
    st, trace, pops, costs = oracle.ga_run(pi, de, 150, p, seed=21, P=128, D=64, gens=4, record=True, inst=0)
    ga = pm.GA(pm.Instance(d, p), seed=21, pop=128, deme=64)
    assert ga.info()["kernels_per_generation"] == 1
    np.testing.assert_array_equal(ga.step(4), trace)
    masks, got = ga.population()
    np.testing.assert_array_equal(masks, pops[-1])
    np.testing.assert_array_equal(got, costs[-1])
    assert ga.result()[2] == st.evals


def test_distances_of_17_bits_keep_the_phases(pm):
    d = _distances(60, 60, 1)
    d[3, 4] = 65536
    ga = pm.GA(pm.Instance(d, 5), seed=1, pop=64)
    assert ga.info()["kernels_per_generation"] > 1
    ga.step(3)
    masks, costs = ga.population()
    np.testing.assert_array_equal(costs, oracle.eval_direct(d, masks))


def test_a_wait_that_runs_out_is_reported(pm, monkeypatch):
    monkeypatch.setenv("PM_GA_GRAPH", "0")
    d = graph_instance(100, 200, seed=3)
    ga = pm.GA(pm.Instance(d, 5), seed=1, pop=256, deme=128)
    ga.step(2)
    pm.pm_debug_scan_timeout(1)
    with pytest.raises(pm.PMError) as e:
        ga.step(1)
    assert e.value.status == PM_ERR_TIMEOUT
    ga.step(3)
    masks, costs = ga.population()
    np.testing.assert_array_equal(costs, oracle.eval_direct(d, masks))
