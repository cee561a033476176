"""The order-statistic DP at the edges of its layouts, against the oracle.

One device per lane up to 32 devices, then 2, 3, 4 or 8: replicas just below,
at and above each boundary; replicas with as many devices as blocks (one
partition only) and with one device; costs its float estimate does not
describe (blocks of no cost, hosts faster than their devices, links that
dominate), where the walk falls back to the bisection over the keys; small
integers, so that thresholds, masters and batches tie, and fractions.
"""
import dataclasses

import numpy as np
import pytest

from oracle import oracle as O

from test_parity_gpu import _edge_problem, _genomes_from, assert_eval_equal, engine

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__ as ge
    ge.build()


# (blocks, replica sizes of each genome)
SIZES = [(3, [[1, 1, 1], [3], [2, 1]]),
         (32, [[32, 1], [31, 2], [33], [16, 17]]),              # as many devices as blocks; one too many
         (70, [[32, 33], [31, 34], [65], [1, 64]]),
         (100, [[63, 34], [96, 1], [97], [95, 2]]),
         (130, [[128, 1], [127, 2], [129], [64, 65]]),
         (160, [[140, 20], [129, 31], [100, 60]])]


def _check(prob, M, K, genomes, rng):
    g = _genomes_from(M, K, genomes, rng)
    eng = engine(prob)
    eng.eval(g)
    ora = O.OracleProblem(prob).eval_population(g, K, nthreads=O.num_threads())
    assert_eval_equal(eng.results(), ora)
    st = eng.stats()
    assert st["paper_candidates"] == ora["cand"] and st["device_errors"] == 0
    eng.close()
    return ora


@pytest.mark.parametrize("N,groups", SIZES)
@pytest.mark.parametrize("integer", [True, False])
def test_lane_layouts(N, groups, integer):
    rng = np.random.default_rng(300 + N)
    M, K = sum(groups[0]), max(len(x) for x in groups)
    genomes = groups * 3
    prob = _edge_problem(rng, M, N, len(genomes), K, integer=integer, Q=1, min_tps=0.001)
    prob.mem = np.maximum(prob.mem, np.uint64(4))               # every device holds a block and the head
    ora = _check(prob, M, K, genomes, rng)
    assert np.isfinite(ora["T"]).any()


@pytest.mark.parametrize("what", ["free blocks", "fast hosts", "slow links", "one slow device", "mixed scales"])
@pytest.mark.parametrize("role_search", [0, 1])
def test_costs_off_the_estimate(what, role_search):
    rng = np.random.default_rng(41)
    M, N, K = 40, 57, 4
    genomes = [[40], [33, 7], [20, 12, 8], [10, 10, 10, 10], [1, 39], [5, 3, 32]] * 3
    prob = _edge_problem(rng, M, N, len(genomes), K, integer=True, Q=1, min_tps=0.001, role_search=role_search)
    if what == "free blocks":
        prob.blk_flops = np.zeros_like(prob.blk_flops)
        prob.blk_bytes = np.array([0, 0, 3, 0], np.uint64)[:prob.V]
    elif what == "fast hosts":
        prob = dataclasses.replace(prob, mem=rng.integers(2, 6, M).astype(np.uint64),
                                   rate_cpu=rng.choice([0.25, 8.0, 64.0], M), bw_cpu=rng.choice([0.5, 16.0, 64.0], M),
                                   mem_cpu=rng.integers(0, 3 * N, M).astype(np.uint64))
    elif what == "slow links":
        prob.act_bytes = np.full_like(prob.act_bytes, 40)
    elif what == "one slow device":
        prob.rate[7] = 2.0 ** -30
    else:
        prob.rate = 2.0 ** rng.integers(-40, 40, M).astype(np.float64)
        prob.bw = 2.0 ** rng.integers(-40, 40, M).astype(np.float64)
    ora = _check(prob, M, K, genomes, rng)
    assert np.isfinite(ora["T"]).any()


@pytest.mark.parametrize("M,N", [(32, 120), (40, 90), (60, 100)])
def test_bisection_over_the_keys(M, N):
    """A head worth more than all blocks: the threshold is far from the estimate,
    more than the walk's steps, and the bisection takes over.  A walk reads an
    entry of the two rows at most twice, and four per lane before it; a bisection
    of 31 rounds reads more than that."""
    for seed in range(4):
        rng = np.random.default_rng(seed)
        prob = _edge_problem(rng, M, N, 1, 1, integer=True, Q=1, min_tps=0.0)
        prob.mem = np.full(M, 2**40, np.uint64)
        prob.head_flops = np.full_like(prob.head_flops, 3000)
        prob.rate = rng.uniform(0.1, 3, M)
        g = _genomes_from(M, 1, [[M]], rng)
        g["roles"][:] = 0
        eng = engine(prob)
        eng.eval(g)
        assert_eval_equal(eng.results(), O.OracleProblem(prob).eval_population(g, 1))
        st = eng.stats()
        walk = 2 * 2 * M * (N - M + 1) + 4 * 32 * -(-M // 32)
        assert st["dp_runs"] == 1 and st["dp_probes"] > walk, (st["dp_probes"], walk)
        eng.close()


@pytest.mark.parametrize("M,N", [(8, 700), (16, 1024)])
def test_long_models_on_small_fleets(M, N):
    """Up to 16 devices any number of blocks is accepted."""
    rng = np.random.default_rng(N)
    genomes = [[M], [1] * 4 + [M - 4], [M - 3, 3]] * 2
    prob = _edge_problem(rng, M, N, len(genomes), 5, integer=True, Q=1, min_tps=0.0)
    prob.mem = np.full(M, 2**20, np.uint64)
    ora = _check(prob, M, 5, genomes, rng)
    assert np.isfinite(ora["T"]).any()
