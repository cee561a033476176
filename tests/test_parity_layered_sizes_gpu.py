"""The per-layer DP at the edges of its column and table sizes.

Replicas of one device, replicas with as many devices as blocks (columns of
one cell, no range-minimum levels), columns of 31 to 33 and 63 to 65 cells
(lane and thread edges), powers of two, and the largest model the per-layer
path takes; small-integer work, so that splits, masters and batches tie.  Bit
for bit against the oracle.
"""
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
SIZES = [(1, [[1]]), (2, [[2], [1, 1]]), (5, [[5], [4, 1], [3, 2]]),
         (34, [[2, 1], [3], [1, 2]]),                       # 33, 34 and 32 cells
         (33, [[3, 2, 1], [6], [1, 1, 4]]),                 # 31, 32, 33, 28, 30 cells
         (66, [[2, 3, 1], [4, 2]]),                         # 65, 64, 66, 63 cells
         (129, [[1, 2, 3], [5, 1]]),                        # 128 and 129 cells
         (40, [[40], [39, 1], [20, 20]]),                   # as many devices as blocks
         (180, [[1, 2], [3]])]                              # the largest model


@pytest.mark.parametrize("N,groups", SIZES)
@pytest.mark.parametrize("role_search", [0, 1])
def test_layered_sizes(N, groups, role_search):
    from test_oracle_pins import _layered
    rng = np.random.default_rng(1000 + N)
    M, K = sum(groups[0]), max(len(g) for g in groups)
    genomes = groups * 4
    prob = _layered(_edge_problem(rng, M, N, len(genomes), K, integer=True, Q=1, min_tps=0.01,
                                  role_search=role_search), rng, integer=True)
    g = _genomes_from(M, K, genomes, rng)
    eng = engine(prob)
    eng.eval(g)
    ora = O.OracleProblem(prob).eval_population(g, K, nthreads=O.num_threads())
    assert_eval_equal(eng.results(), ora)
    assert np.isfinite(ora["T"]).any() or N == 1            # (one block fits no device of that draw)
    eng.stats()                                             # raises on a device-side check
    eng.close()
