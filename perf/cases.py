"""Timing cases of the deployment search, through the package's public calls.

A case is one thing that a user of the search has it do: a whole search on the
device (initial population, generations, elites), one generation with the host
in the loop, the evaluation of a given population, or the allocation-free elite
selection.  Fleets, links, models and populations are drawn from the seed over
the ranges of the repository's own workloads.
"""
import math

import numpy as np
import torch

from paper_2606_03770_gb300 import e2ga
from paper_2606_03770_gb300 import workloads as W

# Decoder blocks by model width (the three models of the repository's
# workloads) and the prompt lengths they are asked with.
MODELS = {
    "d4096": dict(d=4096, ffn=11008, kv_heads=None, vocab=32000, wbits=16, prompt=(512, 512)),
    "d8192": dict(d=8192, ffn=28672, kv_heads=8, vocab=128256, wbits=4, prompt=(256, 2048)),
    "d16384": dict(d=16384, ffn=53248, kv_heads=8, vocab=128256, wbits=4, prompt=(256, 4096)),
}
# Device TFLOP/s (log-uniform), memory GB and link Gbps of the fleet each model
# is served on (the widest one's links are log-uniform).
FLEETS = {
    "d4096": dict(tflops=(2, 30), mem_gb=(4, 16), link=("uniform", 0.1, 10)),
    "d8192": dict(tflops=(2, 30), mem_gb=(4, 32), link=("uniform", 0.1, 10)),
    "d16384": dict(tflops=(1, 60), mem_gb=(2, 64), link=("log", 0.05, 25)),
}
B_MAX = 8


def _case(kind, model, M, N, K, P, gens=1, roles=0, objective=0, offload=False, layered="", redraw=False,
          p_mut=0.3, name=None):
    c = dict(kind=kind, model=model, M=M, N=N, K=K, P=P, gens=gens, roles=roles, objective=objective,
             offload=offload, layered=layered, redraw=redraw, p_mut=p_mut)
    return dict(c, name=name) if name else c


def listed():
    return [
        # replanning a handful of devices: one short search, where launches and latency count
        _case("search", "d4096", 8, 32, 2, 64, gens=2, name="search-8dev"),
        # a search over a small cluster, start to finish on the device
        _case("search", "d8192", 32, 80, 8, 1024, gens=10, name="search-32dev"),
        # the same cluster driven from the host: population in, fitness and next population out
        _case("host", "d8192", 32, 80, 8, 1024, name="host-loop-32dev"),
        # odd sizes everywhere: what is left when some devices are away
        _case("search", "d8192", 37, 61, 11, 777, gens=3, name="search-37dev-odd"),
        # a larger fleet whose links change from generation to generation
        _case("search", "d8192", 128, 80, 16, 4096, gens=4, redraw=True, name="search-128dev-redraw"),
        # the brute-force role assignment on that fleet
        _case("search", "d8192", 128, 80, 16, 2048, gens=2, roles=1, name="roles-128dev"),
        # the long search: a low mutation rate, so that replicas converge
        _case("search", "d8192", 256, 80, 32, 8192, gens=10, p_mut=0.01, name="search-256dev"),
        # the largest fleet and model: one population scored, with its partitions
        _case("eval", "d16384", 512, 126, 64, 16384, name="eval-512dev"),
        # and one whole generation of it with the host in the loop
        _case("host", "d16384", 512, 126, 64, 16384, name="host-loop-512dev"),
        # a model that alternates sliding-window and full attention: blocks of two types
        _case("eval", "d8192", 32, 80, 8, 512, layered="alternate", name="eval-layered-32dev"),
        # the comparison planner (finishing time, strongest replicas prefill) on devices that
        # offload blocks to host memory
        _case("eval", "d8192", 32, 80, 8, 512, roles=2, objective=1, offload=True, name="eval-offload-32dev"),
        # elite selection for a caller that may not allocate
        _case("elites", "d16384", 512, 126, 64, 16384, name="elites-16384"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["search", "search", "host", "eval", "eval", "layered", "elites"])
    model = rng.choice(list(MODELS))
    if kind == "layered":                      # per-layer profiles: smaller fleets and populations
        M, N, P = _log_int(rng, 8, 64), rng.randint(24, 96), _log_int(rng, 32, 384)
        while P * M * N * N > 384 * 32 * 80 * 80:
            P = max(32, P // 2)
            if P == 32:
                M = max(8, M - 8)
                N = max(24, N - 8)
        return _case("eval", "d8192", M, N, rng.randint(2, min(12, M)), P, roles=rng.choice([0, 0, 1]),
                     layered=rng.choice(["alternate", "tail"]))
    M = _log_int(rng, 8, 512)
    N = rng.randint(24, 126)
    K = min(M, _log_int(rng, 2, 64))
    P = _log_int(rng, 64, 16384)
    if kind == "elites":
        return _case(kind, model, M, N, K, P)
    roles = rng.choice([0, 0, 0, 1, 2]) if K <= 16 else rng.choice([0, 0, 0, 2])
    if roles == 1:
        P = min(P, 2048)
    gens = rng.randint(1, 4) if kind == "search" else 1
    while gens > 1 and gens * P * M > 16384 * 512:
        gens -= 1
    return _case(kind, model, M, N, K, P, gens=gens, roles=roles, objective=rng.choice([0, 0, 1]) if K <= 12 else 0,
                 offload=rng.random() < 0.25, redraw=kind == "search" and rng.random() < 0.3,
                 p_mut=rng.choice([0.3, 0.3, 0.01]))


def _problem(case, seed):
    """Fleet, links and layer profile drawn from the seed."""
    rng = np.random.Generator(np.random.Philox(key=seed + 17))
    M, N, mdl, fl = case["M"], case["N"], dict(MODELS[case["model"]]), FLEETS[case["model"]]
    lo, hi = mdl.pop("prompt")

    def log_u(a, b, shape):
        return np.exp(rng.uniform(math.log(a), math.log(b), shape))

    rate = log_u(*fl["tflops"], M) * 1e12
    bw = log_u(50.0, 800.0, M) * 1e9
    mem = np.rint(rng.uniform(*fl["mem_gb"], M) * 1e9).astype(np.uint64)
    kind, llo, lhi = fl["link"]
    gbps = log_u(llo, lhi, (M, M)) if kind == "log" else rng.uniform(llo, lhi, (M, M))
    cong = rng.uniform(0.3, 1.0, (M, M))
    upper = np.triu(np.ones((M, M), bool), 1)
    link_bw = np.where(upper, gbps, gbps.T) * 1.25e8
    np.fill_diagonal(link_bw, np.inf)
    cong = np.where(upper, cong, cong.T)
    NP = int(round(float(np.mean(rng.integers(lo, hi + 1, 1000)))))
    host = {}
    if case["offload"]:
        host = dict(zip(("rate_cpu", "bw_cpu", "mem_cpu"), W.offload_fleet(M, seed)))
    if case["layered"]:
        prof = W.layered_profile(N=N, NP=NP, ND=NP, b_max=B_MAX, pattern=case["layered"], **mdl)
    else:
        prof = W.dense_profile(N=N, NP=NP, ND=NP, b_max=B_MAX, **mdl)
    return W.Problem(name="case", rate=rate, bw=bw, mem=mem, link_bw=link_bw, cong=cong, N=N, NP=NP, ND=NP,
                     P=case["P"], Q=max(1, math.ceil(case["P"] / 32)), K_max=case["K"], G=case["gens"],
                     p_mut=case["p_mut"], redraw=case["redraw"], role_search=case["roles"],
                     objective=case["objective"], seed=seed, **prof, **host)


def _population(case, seed):
    """Random orderings, groupings and roles, as device tensors in the ABI's layout."""
    P, M, K = case["P"], case["M"], case["K"]
    rng = np.random.Generator(np.random.Philox(key=seed + 7919))
    perm = torch.from_numpy(rng.random((P, M))).cuda().argsort(dim=1)
    R = torch.from_numpy(rng.integers(1, min(K, M) + 1, P)).cuda()
    cut = torch.from_numpy(rng.random((P, M))).cuda()
    cut[:, 0] = 2.0                                            # no cut before the first device
    rank = cut.argsort(dim=1).argsort(dim=1)                   # the R - 1 smallest keys are the cuts
    cluster = (rank < (R - 1)[:, None]).to(torch.int64).cumsum(dim=1)
    sizes = torch.zeros((P, K), dtype=torch.int64, device="cuda").scatter_add_(1, cluster, torch.ones_like(cluster))
    bits = torch.from_numpy(rng.integers(-(1 << 63), (1 << 63) - 1, P)).cuda()
    below = torch.where(R >= 64, torch.full_like(R, -1), (torch.ones_like(R) << R.clamp(max=63)) - 1)
    return dict(perm=perm.to(torch.int16), sizes=sizes.to(torch.int16), nclus=R.to(torch.uint8), roles=bits & below)


def _genome_outputs(P, M, K):
    return dict(perm=torch.empty((P, M), dtype=torch.int16, device="cuda"),
                sizes=torch.empty((P, K), dtype=torch.int16, device="cuda"),
                nclus=torch.empty(P, dtype=torch.uint8, device="cuda"),
                roles=torch.empty(P, dtype=torch.int64, device="cuda"))


def prepare(case, seed):
    P, M, K = case["P"], case["M"], case["K"]
    s = dict(case=case, seed=seed)
    if case["kind"] == "elites":
        # an evaluated population with some genomes copied, as elitism and tournaments leave it;
        # early in a search many genomes serve nothing (+inf), and short waits are often 0
        pop = _population(case, seed)
        rng = np.random.Generator(np.random.Philox(key=seed + 31))
        phase = np.exp(rng.uniform(-2.0, 4.0, P))
        phase[rng.random(P) < 0.2] = np.inf
        w = np.where(np.isinf(phase), np.inf, np.maximum(0.0, phase - 1.0) * 1.5)
        src, dst = rng.integers(0, P, P // 20), rng.permutation(P)[:P // 20]
        w[dst], phase[dst] = w[src], phase[src]
        for k in pop:
            pop[k][torch.from_numpy(dst).cuda()] = pop[k][torch.from_numpy(src).cuda()]
        fit = np.zeros((P, 4))
        fit[:, 0], fit[:, 1] = w, phase
        fit[:, 2] = fit[:, 3] = np.where(np.isinf(phase), 0.0, 1.0 / np.where(np.isinf(phase), 1.0, phase))
        s.update(pop=pop, fit=torch.from_numpy(fit).cuda(), Q=max(1, math.ceil(P / 32)))
        s["genomes"] = e2ga.e2_genomes(*[pop[k].data_ptr() for k in ("perm", "sizes", "nclus", "roles")])
        s["idx"] = torch.empty(s["Q"], dtype=torch.int32, device="cuda")
        return s
    s["eng"] = e2ga.Engine(_problem(case, seed))
    if case["kind"] == "search":
        s["next"] = _genome_outputs(P, M, K)
    else:
        pop = _population(case, seed)
        if case["kind"] == "host":
            pin = {k: v.cpu().pin_memory() for k, v in pop.items()}
            s.update(pop=pin, next={k: torch.empty_like(v).pin_memory() for k, v in pin.items()},
                     fit=torch.empty((P, 4), dtype=torch.float64).pin_memory())
        else:
            s["pop"] = pop
    return s


def _results(eng):
    """The evaluation's outputs, in the engine's device tensors."""
    out = dict(fitness=eng.fitness, layers=eng.layers, master=eng.master, bsel=eng.bsel, T=eng.T, L=eng.L,
               gpu_layers=eng.gpu_layers)
    return out


def run(s):
    case, seed = s["case"], s["seed"]
    if case["kind"] == "elites":
        st = e2ga.e2_select_elites_noalloc(s["genomes"], s["fit"].data_ptr(), case["P"], case["M"], case["K"],
                                           s["Q"], s["idx"].data_ptr(), torch.cuda.current_stream().cuda_stream)
        if st != e2ga.E2_OK:
            raise e2ga.E2Error(st, "e2_select_elites_noalloc")
        return dict(elites=s["idx"])
    eng = s["eng"]
    if case["kind"] == "eval":
        eng.eval(s["pop"])
        return _results(eng)
    if case["kind"] == "host":
        eng.run_generation_io(seed, 1, population=s["pop"], fitness=s["fit"], next_out=s["next"])
        return dict(fitness=s["fit"], **s["next"])
    eng.init_population(seed)
    for gen in range(1, case["gens"] + 1):
        if case["redraw"]:
            eng.redraw_congestion(seed, gen)
        eng.run_generation(seed, gen)
    parts = e2ga.e2_partitions(*[t.data_ptr() for t in (eng.layers, eng.master, eng.bsel, eng.T, eng.L,
                                                        eng.gpu_layers)])
    st = e2ga.e2_get_results(eng.ctx, eng.fitness.data_ptr(), parts)
    if st != e2ga.E2_OK:
        raise e2ga.E2Error(st, "e2_get_results", e2ga.e2_last_error(eng.ctx))
    eng.get_population(s["next"])
    idx, fit = eng.elites()                                    # what the search was run for
    return dict(_results(eng), elites=idx, elite_fitness=fit, **s["next"])


def work(case):
    """Each input read and each output written once.  Operations: what every
    partition needs, a stage time and a link time per device, a search over its
    block counts, and the latency's additions; with per-layer profiles, every
    cell of the recurrence once."""
    P, M, N, K = case["P"], case["M"], case["N"], case["K"]
    genomes = P * (2 * M + 2 * K + 1 + 8)
    fitness = 32 * P
    if case["kind"] == "elites":
        return dict(bytes=genomes + fitness + 4 * max(1, math.ceil(P / 32)), flops=4 * P)
    results = fitness + P * (4 * M + 4 * K + 16 * K)
    tables = 8 * 2 * M * M + 24 * M
    per_device = 6 + math.log2(N) if not case["layered"] else 2.0 * N
    flops = case["gens"] * P * M * per_device
    if case["kind"] == "search":
        return dict(bytes=tables + case["gens"] * 2 * genomes + results, flops=flops)
    if case["kind"] == "host":
        return dict(bytes=tables + 2 * genomes + fitness, flops=flops)
    return dict(bytes=tables + genomes + results, flops=flops)


def tolerance(case):
    # every result is fixed to the bit: one order of IEEE float64 operations, and whole numbers
    return "exact"


def exact(case, seed):
    """One population's evaluation in float64, straight from the recurrence: every
    split of every cell, every master, every batch.  None where that takes too
    long, and for searches (whole numbers of many generations)."""
    P, M, N, K = case["P"], case["M"], case["N"], case["K"]
    if case["kind"] != "eval" or case["roles"] == 1 or P * M * N * N > 512 * 32 * 80 * 80:
        return None
    p = _problem(case, seed)
    pop = {k: v.cpu().numpy() for k, v in _population(case, seed).items()}
    V, inf = B_MAX + 1, math.inf
    n = np.arange(N)
    with np.errstate(divide="ignore", invalid="ignore"):
        start, end = n[:, None], n[None, :]
        valid = end >= start
        count = np.where(valid, end - start + 1, 0).astype(np.uint64)

        def stage(v, d, head):                                 # [first block, last block]
            h = [int(x[v]) if head else 0 for x in (p.head_flops, p.head_bytes, p.head_mem)]
            if p.PF is not None:
                sums = [np.where(valid, x[v][1:][None, :] - x[v][:-1][:, None], 0).astype(np.float64)
                        for x in (p.PF, p.PB, p.PM)]
                f, y, b = sums[0] + h[0], sums[1] + h[1], sums[2] + h[2]
                t = np.maximum(f / p.rate[d], y / p.bw[d])
                return np.where(valid & (b <= float(p.mem[d])), t, inf)
            blk = [int(x[v]) for x in (p.blk_flops, p.blk_bytes, p.blk_mem)]
            room = int(p.mem[d]) - h[2]
            own = np.minimum(count, np.uint64(max(room, 0) // blk[2])).astype(np.float64)
            off = count.astype(np.float64) - own
            t = np.maximum((own * blk[0] + h[0]) / p.rate[d], (own * blk[1] + h[1]) / p.bw[d])
            ok = valid & (room >= 0)
            if p.mem_cpu is not None:
                ok &= off * blk[2] <= float(p.mem_cpu[d])
                t = t + np.where(off > 0, np.maximum(off * blk[0] / p.rate_cpu[d], off * blk[1] / p.bw_cpu[d]), 0.0)
            else:
                ok &= off == 0
            return np.where(ok, t, inf)

        cost = {v: torch.from_numpy(np.stack([np.stack([stage(v, d, h) for h in (0, 1)]) for d in range(M)])).cuda()
                for v in range(V)}
        beff = p.link_bw * p.cong
        tau = [float(p.act_bytes[v]) / beff for v in range(V)]

    def pipe(v, devs):
        """(T, Lambda) of the canonical partition, or None."""
        m = len(devs)
        if m > N:
            return None
        c = cost[v][torch.as_tensor(devs, device="cuda")]      # [m, 2, N, N]
        D = c[0, :1, 0, :].repeat(m, 1)                        # [master, last block]
        D[0] = c[0, 1, 0, :]
        cols = [D]
        for k in range(1, m):
            prev = torch.full((m, N), inf, dtype=torch.float64, device="cuda")
            prev[:, 1:] = cols[-1][:, :-1]
            ck = c[k, :1].expand(m, N, N)
            val = torch.maximum(prev[:, :, None], ck)
            val[k] = torch.maximum(prev[k][:, None], c[k, 1])
            cols.append(val.amin(dim=1).clamp_min(tau[v][devs[k - 1], devs[k]]))
        last = cols[-1][:, N - 1].cpu().numpy()
        mu = int(np.argmin(last))
        if last[mu] == inf:
            return None
        rows = torch.stack([x[mu] for x in cols]).cpu().numpy()
        cm = torch.stack([c[k, int(k == mu)] for k in range(m)]).cpu().numpy()
        i, times = N - 1, []
        for k in range(m - 1, 0, -1):
            link = tau[v][devs[k - 1], devs[k]]
            prev = np.concatenate([[inf], rows[k - 1][:-1]])
            j = int(np.argmin(np.maximum(np.maximum(prev, cm[k][:, i]), link)))
            times += [cm[k][j, i], link]
            i = j - 1
        times.append(cm[0][0, i])
        lam = 0.0
        for x in times[::-1]:
            lam = lam + float(x)
        return float(last[mu]), lam

    fit = np.zeros((P, 4))
    T, L = np.full((P, K), inf), np.full((P, K), inf)
    seen = {}
    for g in range(P):
        R, off, res = int(pop["nclus"][g]), 0, []
        for c in range(R):
            m = int(pop["sizes"][g, c])
            devs = tuple(int(x) for x in pop["perm"][g, off:off + m])
            off += m
            role = (int(pop["roles"][g]) >> c) & 1
            both = []
            for r in ((0, 1) if case["roles"] else (role,)):
                key = (devs, r)
                if key not in seen:
                    got = None
                    for v in (range(B_MAX, 0, -1) if r else (0,)):
                        x = pipe(v, devs)
                        if x is not None and (r == 0 or 1.0 / x[1] >= p.min_tps):
                            got = (v,) + x
                            break
                    seen[key] = got
                both.append(seen[key])
            res.append(both)
        if case["roles"]:                                      # the strongest replicas prefill
            strength = [p.NP / b[0][1] if b[0] else -1.0 for b in res]
            nP = R
            if R > 1:
                nP = min(max((2 * R * p.NP + p.NP + p.ND) // (2 * (p.NP + p.ND)), 1), R - 1)
            order = sorted(range(R), key=lambda c: (-strength[c], c))
            roles = [0 if order.index(c) < nP else 1 for c in range(R)]
            chosen = [(roles[c], res[c][roles[c]]) for c in range(R)]
        else:
            chosen = [((int(pop["roles"][g]) >> c) & 1, res[c][0]) for c in range(R)]
        S, A = [0.0, 0.0], [0.0, 0.0]
        for c, (r, x) in enumerate(chosen):
            if x is None:
                continue
            T[g, c], L[g, c] = x[1], x[2]
            rate = (x[0] if r else p.NP) / x[1]
            S[r] += rate
            A[r] += rate * x[2]
        w = phase = inf
        if S[0] and S[1]:
            tp, td = p.NP / S[0], p.ND / S[1]
            phase = max(tp, td)
            late = max(0.0, phase - p.t_a)
            w = (tp + late if late > 0 else 0.0) if not case["objective"] else A[0] / S[0] + p.ND * (A[1] / S[1])
        fit[g] = w, phase, S[0], S[1]
    return dict(fitness=fit, layers=None, master=None, bsel=None, T=T, L=L, gpu_layers=None)
