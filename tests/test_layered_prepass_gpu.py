"""The pre-pass's memory and latency tests on per-layer profiles: tight
memories (the longest run of blocks a device holds decides), latency limits in
the middle of what the replicas reach, costs that grow with the batch (searched)
and that do not (tested one by one), replicas on both sides of 32 devices.  Bit
for bit against the oracle, with variants rejected by either test."""
import dataclasses

import numpy as np
import pytest

from oracle import oracle as O
from paper_2606_03770_gb300 import workloads as W

from test_parity_gpu import _edge_problem, assert_eval_equal, engine

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__ as ge
    ge.build()


def _growing(prob):
    """Every decode variant's costs raised to those of the smaller batches."""
    def up(x):
        x = x.copy()
        x[1:] = np.maximum.accumulate(x[1:], axis=0)
        return x

    def sums(x):
        return np.concatenate([np.zeros((x.shape[0], 1), np.uint64),
                               np.cumsum(up(np.diff(x.astype(np.int64), axis=1)), axis=1).astype(np.uint64)], axis=1)

    rows = {k: up(getattr(prob, k)) for k in ("blk_flops", "blk_bytes", "blk_mem", "head_flops", "head_bytes",
                                              "head_mem", "act_bytes")}
    return dataclasses.replace(prob, PF=sums(prob.PF), PB=sums(prob.PB), PM=sums(prob.PM), **rows)


@pytest.mark.parametrize("M,N,K,spare", [(4, 3, 2, 1), (9, 12, 3, 2), (33, 40, 4, 1), (40, 64, 2, 3)])
@pytest.mark.parametrize("grows", [False, True])
@pytest.mark.parametrize("role_search", [0, 1])
def test_layered_prepass(M, N, K, spare, grows, role_search):
    from test_oracle_pins import _layered
    rng = np.random.default_rng(100 * M + N)
    P = 96
    prob = _layered(_edge_problem(rng, M, N, P, K, integer=True, Q=1, min_tps=1e-6, role_search=role_search), rng)
    if grows:
        prob = _growing(prob)
    # a few more units than the blocks need (1 or 2 each); in small fleets from nothing (no block)
    prob.mem = rng.integers(0 if M < 32 else 2, 3 + 2 * (spare + 1) * N // M, M).astype(np.uint64)
    g = W.random_genomes(M, K, P, seed=M)
    lam = O.OracleProblem(prob).eval_population(g, K, nthreads=O.num_threads())["L"]
    lam = lam[np.isfinite(lam)]
    assert lam.size
    # limits among the latencies reached (a bound from the least block's work decides few
    # variants there) and a hundredth of the least: below every bound, since the lightest
    # block's flops are a fifth of the heaviest's and devices differ by less than 20 times
    st = {"prechecked": 0, "tps_pruned": 0}
    for limit in (np.median(lam), np.quantile(lam, 0.1), 0.3 * lam.min(), 0.01 * lam.min()):
        prob.min_tps = float(1.0 / limit)
        eng = engine(prob)
        eng.eval(g)
        assert_eval_equal(eng.results(), O.OracleProblem(prob).eval_population(g, K, nthreads=O.num_threads()))
        for k in st:
            st[k] += eng.stats()[k]
        eng.close()
    assert min(st.values()) > 0, st
