"""The initial population and the generation step at odd sizes, against the
oracle: orderings of 1 to 1,000 devices (lane edges, sizes that are no multiple
of the vector loads), one to 64 replicas, and every child mutated, by
regeneration of both chromosomes, by regrouping, or by each kind in turn (the
shuffle and the cut points are resolved by a warp, not step by step)."""
import numpy as np
import pytest

from oracle import oracle as O

from test_parity_gpu import _edge_problem, assert_genomes_equal, engine

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__ as ge
    ge.build()


@pytest.mark.parametrize("M", [1, 2, 3, 4, 31, 32, 33, 63, 64, 65, 66, 127, 200, 1000])
@pytest.mark.parametrize("kinds", [(0.0, 0.0, 0.0), (0.0, 1.0, 0.0), (0.25, 0.25, 0.25)])
def test_init_and_step(M, kinds):
    rng = np.random.default_rng(M)
    K, P = min(M, 64), 203
    prob = _edge_problem(rng, M, 3, P, K, integer=True, Q=5, min_tps=0.01)
    prob.p_mut, prob.p_kind, prob.tournament = 1.0, kinds + (1.0 - sum(kinds),), 1 + M % 40
    ga = O.ga_of(prob)
    eng = engine(prob)
    eng.init_population(M)
    pop = O.init_population(ga, M)
    for gen in (1, 2):
        assert_genomes_equal(eng.get_population(), pop)
        eng.eval(parts=False)
        fit = eng.results()["fitness"]
        eng.ga_step(M, gen)
        pop = O.ga_step(ga, M, gen, pop, fit, O.elites(ga, pop, fit))
    assert_genomes_equal(eng.get_population(), pop)
    eng.close()


@pytest.mark.parametrize("M,P,K", [(1, 1, 1), (2, 33, 2), (8, 64, 3), (8, 5000, 8), (9, 4095, 9), (9, 4096, 9), (16, 4097, 1),
                                   (17, 16384, 17), (24, 16390, 5), (25, 16384, 25), (32, 65536, 32), (33, 65536, 4)])
def test_init_on_both_sides_of_the_thread_per_genome(M, P, K):
    """Small fleets and large populations, where a thread takes a genome's draws, and the sizes next to them."""
    prob = _edge_problem(np.random.default_rng(M), M, 3, P, K, integer=True, Q=1, min_tps=0.01)
    eng = engine(prob)
    for seed in (1, 2**40 + 7):
        eng.init_population(seed)
        assert_genomes_equal(eng.get_population(), O.init_population(O.ga_of(prob), seed))
    eng.close()


@pytest.mark.parametrize("M", [2, 33, 63, 64])
@pytest.mark.parametrize("P", [8191, 8192])
def test_validation_on_both_sides_of_the_thread_per_genome(M, P):
    """Every kind of invalid genome, found and replaced, whether a warp or a thread takes a genome."""
    from paper_2606_03770_gb300 import e2ga
    prob = _edge_problem(np.random.default_rng(M), M, 3, P, 2, integer=True, Q=1, min_tps=0.01)
    eng = engine(prob)
    eng.init_population(3)
    pop = eng.get_population()
    eng.set_population(pop)                                  # all valid
    assert_genomes_equal(eng.get_population(), pop)
    bad = {k: v.copy() for k, v in pop.items()}
    two = np.flatnonzero(pop["nclus"] == 2)
    rng = np.random.default_rng(P)
    at = np.sort(rng.choice(two[two > 10], 9, replace=False))
    rng.shuffle(at)
    repeat, beyond, far, none, many, empty, total, extra, role = at
    bad["perm"][repeat, -1] = bad["perm"][repeat, 0]
    bad["perm"][beyond, 0] = M
    bad["perm"][far, M // 2] = 65535
    bad["nclus"][none] = 0
    bad["nclus"][many] = 3
    bad["sizes"][empty] = (M, 0)
    bad["sizes"][total, 1] += 1
    bad["nclus"][extra] = 1                                  # its second size is beyond
    bad["roles"][role] |= np.uint64(4)
    with pytest.raises(e2ga.E2Error, match=f"genome {at.min()} "):
        eng.set_population(bad)
    want = {k: v.copy() for k, v in pop.items()}
    want["perm"][at] = np.arange(M)
    want["sizes"][at] = (M, 0)
    want["nclus"][at] = 1
    want["roles"][at] = 0
    assert_genomes_equal(eng.get_population(), want)
    eng.close()
