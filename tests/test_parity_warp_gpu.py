"""Parity of the DP's launches over large populations with the oracle, through
the C ABI: two launches where replicas of more than 32 devices can occur (the
larger ones in the second, several devices per lane), one otherwise.

Full populations (and role search, where each replica runs in both roles) bit
for bit, and a large population of small-integer costs (many exact ties,
memory walls, a Min_TPS floor) on which every DP tie rule is exercised.
"""
import dataclasses

import numpy as np
import pytest

from oracle import oracle as O
from paper_2606_03770_gb300 import workloads as W

from test_parity_gpu import _edge_problem, assert_eval_equal, assert_genomes_equal, engine

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__ as ge
    ge.build()


def _launches(st, n):
    assert st["dp_launches"] == n and st["dp_runs_per_cta_small"] == (4 if n == 2 else 0), st
    assert (st["dp_runs_small"] > 0) == (n == 2) and st["device_errors"] == 0, st


@pytest.mark.parametrize("name,P,role_search", [("c3", 4096, 0), ("c3", 2048, 1), ("c5", 1024, 0)])
def test_two_launches_full_population(name, P, role_search):
    prob = dataclasses.replace(W.make_config(name, P=P), role_search=role_search)
    eng = engine(prob)
    g = W.random_genomes(prob.M, prob.K_max, P, seed=41)
    eng.eval(g)
    gpu = eng.results()
    ora = O.OracleProblem(prob).eval_population(g, prob.K_max, nthreads=O.num_threads())
    assert_eval_equal(gpu, ora)
    if role_search:
        assert np.array_equal(eng.get_population()["roles"], ora["roles"])
    st = eng.stats()
    _launches(st, 2)
    assert st["paper_candidates"] == ora["cand"]
    assert st["served"] == int((ora["bsel"] >= 0).sum())
    eng.close()


@pytest.mark.parametrize("min_tps", [0.0, 0.1])
def test_one_launch_ties_and_memory_walls(min_tps):
    """Small-integer costs on 24 devices and 12 blocks (exact ties between
    splits, masters and batches; devices that cannot hold a block), 8,192
    genomes of up to six replicas: the whole population, then a generation."""
    rng = np.random.default_rng(77)
    M, N, K, P = 24, 12, 6, 8192
    prob = _edge_problem(rng, M, N, P, K, integer=True, Q=64, min_tps=min_tps)
    g = W.random_genomes(M, K, P, seed=13)
    eng = engine(prob)
    eng.eval(g)
    gpu = eng.results()
    ora = O.OracleProblem(prob).eval_population(g, K, nthreads=O.num_threads())
    assert_eval_equal(gpu, ora)
    _launches(eng.stats(), 1)                               # no replica of more than 32 devices
    assert np.isfinite(ora["T"]).sum() > 1000
    ga = O.ga_of(prob)
    eidx = O.elites(ga, g, gpu["fitness"])
    eng.ga_step(5, 1)
    assert_genomes_equal(eng.get_population(), O.ga_step(ga, 5, 1, g, gpu["fitness"], eidx))
    eng.close()


def test_small_fleet_has_one_launch():
    """No replica of the 32-device workload has more than a device per lane."""
    eng = engine(W.make_config("c2"))
    eng.init_population(3)
    eng.eval()
    _launches(eng.stats(), 1)
    eng.close()
