"""Populations and results in the caller's device arrays, wherever they start:
arrays at 16-, 4- and 1-byte offsets of a larger buffer, single bytes to
several 16 KiB chunks, some of them in host memory, against the same arrays
copied one by one to host memory.  Nothing beside them is written."""
import numpy as np
import pytest

from paper_2606_03770_gb300 import e2ga
from test_parity_gpu import _edge_problem, assert_genomes_equal, engine

pytestmark = pytest.mark.gpu
GUARD = 64


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__ as ge
    ge.build()


class Carved:
    """Arrays of the given byte sizes, each `offset` bytes past 256 in a device buffer of its own."""

    def __init__(self, sizes, offset, host=()):
        import torch
        self.sizes, self.at = sizes, 256 + offset
        self.bufs = [torch.full((self.at + n + GUARD,), 0xA5, dtype=torch.uint8,
                                device="cpu" if i in host else "cuda") for i, n in enumerate(sizes)]

    def ptrs(self):
        return [b.data_ptr() + self.at for b in self.bufs]

    def take(self):
        out = []
        for b, n in zip(self.bufs, self.sizes):
            a = b.cpu().numpy()
            assert (a[:self.at] == 0xA5).all() and (a[self.at + n:] == 0xA5).all()
            out.append(a[self.at:self.at + n])
        return out


@pytest.mark.parametrize("P,M,K", [(1, 1, 1), (3, 5, 2), (64, 33, 7), (1031, 37, 11)])
@pytest.mark.parametrize("offset", [0, 4, 6, 1])
@pytest.mark.parametrize("host", [(), (0, 3)])
def test_device_arrays(P, M, K, offset, host):
    import torch
    rng = np.random.default_rng(P)
    prob = _edge_problem(rng, M, 3, P, K, integer=True, Q=1, min_tps=0.01)
    a, b = engine(prob), engine(prob)
    a.init_population(7)
    pop = a.get_population()                                   # host arrays: a copy each
    genomes = [pop[k].view(np.uint8).reshape(-1) for k in ("perm", "sizes", "nclus", "roles")]
    src = Carved([g.size for g in genomes], offset, host)
    for buf, g in zip(src.bufs, genomes):
        buf[src.at:src.at + g.size] = torch.from_numpy(g.copy()).to(buf.device)
    torch.cuda.synchronize()
    assert e2ga.e2_set_population(b.ctx, e2ga.e2_genomes(*src.ptrs())) == e2ga.E2_OK
    src.take()
    assert_genomes_equal(b.get_population(), pop)
    got = Carved([g.size for g in genomes], offset, host)
    assert e2ga.e2_get_population(b.ctx, e2ga.e2_genomes(*got.ptrs())) == e2ga.E2_OK
    torch.cuda.synchronize()
    for x, g in zip(got.take(), genomes):
        np.testing.assert_array_equal(x, g)

    b.eval(parts=False)
    sizes = [32 * P, 2 * P * M, 2 * P * K, 2 * P * K, 8 * P * K, 8 * P * K, 2 * P * M]
    want, res = [Carved(sizes, offset, h) for h in (range(7), host)]   # all in host memory: a copy each
    for c in (want, res):
        fit, *parts = c.ptrs()
        assert e2ga.e2_get_results(b.ctx, fit, e2ga.e2_partitions(*parts)) == e2ga.E2_OK
        torch.cuda.synchronize()
    for x, y in zip(res.take(), want.take()):
        np.testing.assert_array_equal(x, y)
    a.close(), b.close()


def test_first_bad_genome():
    """The error word set on the way of the copy names the first invalid genome, and none when all are valid."""
    import torch
    prob = _edge_problem(np.random.default_rng(1), 5, 3, 9, 2, integer=True, Q=1, min_tps=0.01)
    eng = engine(prob)
    eng.init_population(3)
    pop = {k: torch.from_numpy(v.view(np.dtype(f"i{v.itemsize}") if v.itemsize > 1 else v.dtype)).cuda()
           for k, v in eng.get_population().items()}
    eng.set_population(pop)
    pop["nclus"][4] = 0
    pop["nclus"][7] = 0
    with pytest.raises(e2ga.E2Error, match="genome 4 "):
        eng.set_population(pop)
    eng.close()


def test_outputs_that_share_memory():
    """Outputs of one call that share memory are written in the call's order: with
    one array for layers and gpu_layers, or one that starts inside the other, the
    later output stands where they meet."""
    import dataclasses
    import torch
    rng = np.random.default_rng(3)
    P, M, K, N = 4096, 24, 3, 30
    prob = _edge_problem(rng, M, N, P, K, integer=True, Q=1, min_tps=0.0)
    one = np.ones_like(prob.blk_mem)
    prob = dataclasses.replace(prob, blk_mem=one, mem=rng.integers(2, 5, M).astype(np.uint64), rate_cpu=np.ones(M),
                               bw_cpu=np.ones(M), mem_cpu=np.full(M, N, np.uint64))
    eng = engine(prob)
    eng.init_population(3)
    eng.eval()
    want = eng.results()
    layers, split = want["layers"].reshape(-1), want["gpu_layers"].reshape(-1)
    assert (layers != split).mean() > 0.1
    n = P * M
    for shift in (0, 8, n - 8):                                 # gpu_layers starts `shift` entries into layers
        buf = torch.full((2 * n,), -7, dtype=torch.int16, device="cuda")
        parts = e2ga.e2_partitions(buf.data_ptr(), None, None, None, None, buf.data_ptr() + 2 * shift)
        for _ in range(5):
            assert e2ga.e2_get_results(eng.ctx, None, parts) == e2ga.E2_OK
            torch.cuda.synchronize()
            got = buf.cpu().numpy()
            np.testing.assert_array_equal(got[shift:shift + n], split)
            np.testing.assert_array_equal(got[:shift], layers[:shift])
            assert (got[shift + n:] == -7).all()
    eng.close()
