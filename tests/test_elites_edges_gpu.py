"""The elite selection at the edges of its passes, against the oracle.

Many genomes tied at the threshold: the same w with different phases, the same
w and phase (the index decides), every genome at +inf, every genome distinct
by one low bit; populations around the sizes where the duplicate test and the
held keys change (1,024 keys per pass, 4,096 and 8,192 genomes), with
duplicates and with too few distinct genomes.  The fitness is set, not
evaluated, through the allocation-free call; and searches on populations of
copies through the generation step.
"""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2606_03770_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__ as ge
    ge.build()


def _fitness(what, P, rng):
    w, ph = rng.uniform(0, 5, P), rng.uniform(1, 6, P)
    if what == "plateau":                                   # most waits 0, the phase decides
        w[rng.random(P) < 0.7] = 0.0
    elif what == "ties":
        w, ph = rng.integers(0, 3, P).astype(float), rng.integers(1, 3, P).astype(float)
    elif what == "inf":
        w[:], ph[:] = np.inf, np.inf
    elif what == "few finite":
        keep = rng.random(P) < 0.01
        w[~keep], ph[~keep] = np.inf, np.inf
    elif what == "low bits":
        w = np.nextafter(1.0, 2.0) + np.arange(P) * 2.0 ** -52
        rng.shuffle(w)
    return np.stack([w, ph, 1 / ph, 1 / ph], axis=1)


@pytest.mark.parametrize("P", [1, 31, 1023, 1025, 4095, 4096, 8193])
@pytest.mark.parametrize("what", ["plateau", "ties", "inf", "few finite", "low bits"])
def test_selection(P, what):
    import torch
    from paper_2606_03770_gb300 import e2ga
    rng = np.random.default_rng(P)
    M, K = (15, 4) if P % 2 else (16, 3)                    # odd and even orderings, no chance repeats
    g = W.random_genomes(M, K, P, seed=P)
    fit = _fitness(what, P, rng)
    for d in rng.integers(0, P, P // 8):                    # copies, with their fitness
        s = int(rng.integers(0, P))
        for k in g:
            g[k][d] = g[k][s]
        fit[d] = fit[s]
    views = {np.dtype(np.uint16): np.int16, np.dtype(np.uint64): np.int64}
    dev = {k: torch.from_numpy(np.ascontiguousarray(v).view(views.get(v.dtype, v.dtype))).cuda() for k, v in g.items()}
    gs = e2ga.e2_genomes(*[dev[k].data_ptr() for k in ("perm", "sizes", "nclus", "roles")])
    fd = torch.from_numpy(fit).cuda()
    for Q in {1, max(1, P // 32), P - P // 4, P}:
        out = torch.full((Q,), -1, dtype=torch.int32, device="cuda")
        st = e2ga.e2_select_elites_noalloc(gs, fd.data_ptr(), P, M, K, Q, out.data_ptr(),
                                           torch.cuda.current_stream().cuda_stream)
        assert st == e2ga.E2_OK
        ga = O._ga_struct(P, M, K, Q, 4, 0.5, 0.3, (0.2, 0.5, 0.15, 0.15))
        assert np.array_equal(out.cpu().numpy(), O.elites(ga, g, fit)), Q


@pytest.mark.parametrize("P,distinct", [(1000, 20), (4095, 3), (4097, 64), (9000, 5)])
def test_generation_step_on_copies(P, distinct):
    """Populations of copies (far fewer distinct genomes than elites, and more)."""
    from paper_2606_03770_gb300.e2ga import Engine
    prob = W.make_config("c1_tiny", P=P)
    g = W.random_genomes(prob.M, prob.K_max, P, seed=2)
    src = np.random.default_rng(3).integers(0, distinct, P)
    g = {k: np.ascontiguousarray(v[src]) for k, v in g.items()}
    eng = Engine(prob)
    eng.eval(g)
    fit = eng.results()["fitness"]
    ga = O.ga_of(prob)
    eidx = O.elites(ga, g, fit)
    eng.ga_step(8, 3)
    assert np.array_equal(eng.elites()[0], eidx)
    nxt, ref = eng.get_population(), O.ga_step(ga, 8, 3, g, fit, eidx)
    for k in ref:
        assert np.array_equal(nxt[k], ref[k]), k
    eng.close()


@pytest.mark.parametrize("P", [2048, 2049])
@pytest.mark.parametrize("what", ["plateau", "ties", "inf"])
def test_selection_beside_the_small_populations(P, what):
    """The largest population ranked without a selection, and the smallest with one."""
    test_selection(P, what)
