"""The workloads whose speed is tracked: parallel GOM for weighted Max-Cut through the library's public entry points.

A case is one of four things that a program does with the library:
  run       resume a population from a checkpoint, make some generations, read their counters and the new state
  batch     the same for many independent instances in one batched launch
  ims       advance the Interleaved Multi-start Scheme by some generations of its smallest population
  evaluate  the cut weights of a population that the caller holds (no handle, no allocation)
Every pass starts from the same checkpoint, so it can be repeated; the results are whole numbers, equal on every pass.
The start generation of a case (`start`) says where in a search it stands: a fresh random population (0), where most
donors differ at once, or a later one, where patterns repeat and most of a search's time is spent.

The learned trial filter and Forced Improvement are not listed: both are off by default, and neither shortens a search
on the workloads measured so far.
"""
import math

import numpy as np
import torch

from paper_2203_08680_gb300 import gom, instances

FOS_KINDS = {"neighbourhood": gom.GOM_FOS_NEIGHBOURHOOD, "singleton": gom.GOM_FOS_SINGLETON,
             "linkage_tree": gom.GOM_FOS_BFLT}


def listed():
    return [
        # the smallest parity configuration: a 10x10 torus, one short search; latency and launches are all of it
        dict(name="torus10_p16", kind="run", graph="torus2d", size=10, degree=4, wmin=1, wmax=100,
             fos="neighbourhood", bound=0, pop=16, start=0, gens=20),
        # the 100x100 torus configuration, the start of a search with a small population
        dict(name="torus100_p64", kind="run", graph="torus2d", size=100, degree=4, wmin=1, wmax=100,
             fos="neighbourhood", bound=0, pop=64, start=0, gens=50),
        # odd sizes throughout and signed weights beyond a byte, as in spin-glass instances
        dict(name="torus317_p100_signed", kind="run", graph="torus2d", size=317, degree=4, wmin=-1000, wmax=1000,
             fos="neighbourhood", bound=0, pop=100, start=20, gens=10),
        # the connectivity sweep: the 3D torus in the middle of a search
        dict(name="torus3d50_p128", kind="run", graph="torus3d", size=50, degree=6, wmin=1, wmax=100,
             fos="neighbourhood", bound=0, pop=128, start=40, gens=20),
        # the connectivity sweep: random 6-regular, the larger population
        dict(name="rreg200k_d6_p512", kind="run", graph="random_regular", size=200000, degree=6, wmin=1, wmax=100,
             fos="neighbourhood", bound=0, pop=512, start=20, gens=6),
        # the connectivity sweep: random 12-regular; hundreds of small colour groups of larger elements
        dict(name="rreg60k_d12_p512", kind="run", graph="random_regular", size=60000, degree=12, wmin=1, wmax=100,
             fos="neighbourhood", bound=0, pop=512, start=10, gens=4),
        # the headline workload, the 1000x1000 torus, well into a search
        dict(name="torus1000_p256", kind="run", graph="torus2d", size=1000, degree=4, wmin=1, wmax=100,
             fos="neighbourhood", bound=0, pop=256, start=60, gens=20),
        # the paper's linkage model at its smaller bound (10), a population that is no power of two
        dict(name="tree10_torus200_p300", kind="run", graph="torus2d", size=200, degree=4, wmin=1, wmax=100,
             fos="linkage_tree", bound=10, pop=300, start=10, gens=10),
        # the linkage model that reaches the optimum's neighbourhood: sets of up to 128 variables, the largest population
        dict(name="tree128_torus100_p1024", kind="run", graph="torus2d", size=100, degree=4, wmin=1, wmax=100,
             fos="linkage_tree", bound=128, pop=1024, start=6, gens=6),
        # many uneven instances in one launch (random regular graphs, populations of 32 to 256)
        dict(name="batch48", kind="batch", count=48, mix=1, nmin=1000, nmax=65536, dmin=3, dmax=8, gens=8),
        # the multi-start scheme over the linkage tree, one call's worth of generations
        dict(name="ims_tree128_torus100", kind="ims", graph="torus2d", size=100, degree=4, wmin=1, wmax=100,
             fos="linkage_tree", bound=128, base=128, c=2, max_pop=1024, steps=16),
        # the cut weights of a population held by the caller, no handle
        dict(name="evaluate_rreg200k_d6_p500", kind="evaluate", graph="random_regular", size=200000, degree=6, wmin=1,
             wmax=100, pop=500),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_graph(rng, most):
    """A graph of at most `most` vertices."""
    g = rng.choice(["torus2d", "torus2d", "torus3d", "random_regular", "random_regular"])
    if g == "torus2d":
        size, degree = _log_int(rng, 5, max(6, math.isqrt(most))), 4
    elif g == "torus3d":
        size, degree = _log_int(rng, 4, max(5, int(most ** (1 / 3)))), 6
    else:
        size, degree = _log_int(rng, 50, min(most, 200000)), rng.randint(3, 12)
        if degree > 8:
            size = min(size, 60000)
        size += size * degree % 2
    wmin, wmax = rng.choice([(1, 100), (1, 100), (1, 1), (1, 255), (-100, 100), (-1000, 1000)])
    return dict(graph=g, size=size, degree=degree, wmin=wmin, wmax=wmax)


def draw(rng):
    kind = rng.choice(["run"] * 7 + ["batch", "ims", "evaluate"])
    if kind == "batch":
        nmin = _log_int(rng, 200, 2000)
        return dict(kind="batch", count=rng.randint(2, 48), mix=rng.randint(2, 1000), nmin=nmin,
                    nmax=_log_int(rng, 2 * nmin, 40000), dmin=3, dmax=rng.randint(4, 8), gens=rng.randint(2, 8))
    if kind == "ims":
        c = rng.choice([2, 4])
        pops = rng.randint(2, 4 if c == 2 else 3)
        base = _log_int(rng, 4, 128)
        case = dict(kind="ims", **_draw_graph(rng, 10000), fos="linkage_tree", bound=_log_int(rng, 4, 128), base=base, c=c,
                    max_pop=base << (pops - 1), steps=c ** (pops - 1))
        if case["degree"] > 6 and case["graph"] == "random_regular":
            case.update(degree=6)
        return case
    if kind == "evaluate":
        graph = _draw_graph(rng, 200000)
        # the library's fixed scratch holds n words for each (power of two of) 32 individuals
        rows = 1 << (_noalloc_words() // _vertices(graph)).bit_length() - 1
        return dict(kind="evaluate", **graph, pop=min(_log_int(rng, 2, 1000), 32 * rows))
    fos = rng.choice(["neighbourhood"] * 5 + ["linkage_tree"] * 2 + ["singleton"])
    graph = _draw_graph(rng, 40000 if fos == "linkage_tree" else 500000)
    if fos == "linkage_tree" and graph["degree"] > 6:
        graph.update(degree=6)
    n = _vertices(graph)
    pop = min(_log_int(rng, 2, 1024), 200000000 // n)
    # a share of the largest listed case's trials times closure size
    most = 4e8 if fos == "neighbourhood" else 1e8
    unit = n * pop * (graph["degree"] ** 2 if fos == "neighbourhood" else 8 * graph["degree"])
    gens = max(1, min(20, int(most * 8 / max(unit, 1))))
    return dict(kind="run", **graph, fos=fos, bound=rng.choice([10, 10, 30, 64, 100]) if fos == "linkage_tree" else 0,
                pop=pop, start=rng.choice([0, 5, 20]), gens=gens)


def _noalloc_words():
    """GOM_NOALLOC_MAX_WORDS of include/gom.h."""
    return 4 * 1024 * 1024


def _vertices(case):
    return {"torus2d": case["size"] ** 2, "torus3d": case["size"] ** 3, "random_regular": case["size"]}[case["graph"]]


def _graph(case, seed):
    make = {"torus2d": instances.torus2d, "torus3d": instances.torus3d}
    weights = dict(seed=seed + 1, wmin=case["wmin"], wmax=case["wmax"])
    if case["graph"] == "random_regular":
        return instances.random_regular(case["size"], case["degree"], **weights)
    return make[case["graph"]](case["size"], **weights)


def _mix(case):
    """The sizes of a batch's instances (their graphs and weights come from prepare()'s seed)."""
    return instances.batch_mix(case["count"], seed=case["mix"], nmin=case["nmin"], nmax=case["nmax"], dmin=case["dmin"],
                               dmax=case["dmax"])


def _workspace(nbytes):
    t = torch.empty(nbytes + 256, dtype=torch.uint8, device="cuda")
    return t[(-t.data_ptr()) % 256:]


def _checkpoint(population):
    """The state that a checkpoint holds: population, elitist, its fitness, the generation counter."""
    pop, _, _ = population.population()
    elite, fe = population.elite()
    return pop, elite, fe, population.generation_counter()


def _counters(stats):
    return np.array([tuple(s.values()) for s in stats], dtype=np.int64)


def prepare(case, seed):
    if case["kind"] == "evaluate":
        g = _graph(case, seed)
        rng = torch.Generator(device="cuda").manual_seed(seed + 1)
        pop = torch.randint(0, 2, (case["pop"], g.n), dtype=torch.uint8, device="cuda", generator=rng)
        return dict(case=case, n=g.n, pop=pop,
                    csr=[torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (g.row_ptr, g.col, g.weight)])
    if case["kind"] == "batch":
        mix = _mix(case)
        pops = [gom.Population(instances.random_regular(n, d, seed=1000 * seed + s), p, seed=1000 * seed + s)
                for n, d, p, s in mix]
        workspace = _workspace(gom.gom_batch_workspace_bytes(len(pops)))
        batch = gom.gom_batch_create([q.ctx for q in pops], (4, 2, 0, 300), workspace)
        gom.gom_batch_generation(batch, 5)
        return dict(case=case, pops=pops, batch=batch, checkpoints=[_checkpoint(q) for q in pops],
                    cells=[q.p * q.n for q in pops], rows=[q.p for q in pops])
    g = _graph(case, seed)
    fos = gom.gom_build_fos(g, FOS_KINDS[case["fos"]], case["bound"])
    gom.gom_color_fos(g, fos)
    if case["kind"] == "ims":
        nbytes = gom.gom_ims_workspace_bytes(g, fos, case["base"], case["max_pop"])
        ims = gom.gom_ims_create(g, fos, case["base"], case["c"], case["max_pop"], seed + 1, _workspace(nbytes))
        views = [gom.gom_ims_population(ims, i) for i in range(gom.gom_ims_num_populations(ims))]
        checkpoints = []
        for i, v in enumerate(views):
            pop = torch.empty((case["base"] << i, g.n), dtype=torch.uint8, device="cuda")
            elite = torch.empty(g.n, dtype=torch.uint8, device="cuda")
            gom.gom_get_population(v, pop, None, False)
            checkpoints.append((pop, elite, gom.gom_get_elite(v, elite), 0))
        return dict(case=case, ims=ims, views=views, checkpoints=checkpoints)
    population = gom.Population(g, case["pop"], seed=seed + 1, fos=fos)
    if case["start"]:
        population.generation(case["start"], want_stats=False)
    return dict(case=case, population=population, checkpoint=_checkpoint(population))


def run(state):
    case = state["case"]
    if case["kind"] == "run":
        population = state["population"]
        population.set_population(*state["checkpoint"])
        stats, _ = population.generation(case["gens"])
        pop, fit, fe = population.population()
        elite, _ = population.elite()
        return dict(counters=_counters(stats), pop=pop, fitness=fit, elite=elite, elite_fitness=fe)
    if case["kind"] == "batch":
        # the exports go side by side into two buffers, one for the populations and one for their fitness
        pop = torch.empty(sum(state["cells"]), dtype=torch.uint8, device="cuda")
        fit = torch.empty(sum(state["rows"]), dtype=torch.int64, device="cuda")
        for q, saved in zip(state["pops"], state["checkpoints"]):
            q.set_population(*saved)
        runs = gom.gom_batch_generation(state["batch"], case["gens"])
        at, row = 0, 0
        for q, cells, rows in zip(state["pops"], state["cells"], state["rows"]):
            gom.gom_get_population(q.ctx, pop[at:at + cells], fit[row:row + rows], False)
            at, row = at + cells, row + rows
        return dict(generations=runs, pop=pop, fitness=fit)
    if case["kind"] == "ims":
        for view, saved in zip(state["views"], state["checkpoints"]):
            gom.gom_set_population(view, *saved)
        result = gom.gom_ims_run(state["ims"], case["steps"])
        out = dict(best=result["best_fitness"], reached=result["reached"])
        for i, (view, saved) in enumerate(zip(state["views"], state["checkpoints"])):
            pop = torch.empty_like(saved[0])
            fit = torch.empty(len(pop), dtype=torch.int64, device="cuda")
            out["elite_fitness%d" % i] = gom.gom_get_population(view, pop, fit)
            out["pop%d" % i], out["fitness%d" % i] = pop, fit
        return out
    fit = torch.empty(case["pop"], dtype=torch.int64, device="cuda")
    gom.gom_fitness_noalloc(*state["csr"], state["n"], state["pop"], case["pop"], fit)
    return fit


def _element_terms(case):
    """About (elements, variables and edges of one) of a case's linkage model, by its kind."""
    n, d = _vertices(case), case["degree"]
    if case["fos"] == "neighbourhood":
        return n, (d + 1) + d * d
    if case["fos"] == "singleton":
        return n, 1 + d
    return 2 * n, 4 + 3 * d  # a tree has about two sets a variable; most of them are small


def work(case):
    """Bytes: the checkpoint, the graph and the results, once each.  Operations: one per variable and edge of a trial."""
    if case["kind"] == "batch":
        mix = _mix(case)
        cells = sum(n * p for n, _, p, _ in mix)
        return {"bytes": 2 * cells + sum(8 * n * (d + 1) + 8 * p for n, d, p, _ in mix),
                "flops": case["gens"] * sum(n * p * ((d + 1) + d * d) for n, d, p, _ in mix)}
    n = _vertices(case)
    csr = 8 * n * (case["degree"] + 1)
    if case["kind"] == "evaluate":
        return {"bytes": n * case["pop"] + csr + 8 * case["pop"], "flops": n * case["degree"] // 2 * case["pop"]}
    m, terms = _element_terms(case)
    if case["kind"] == "ims":
        pops = [case["base"] << i for i in range(20) if case["base"] << i <= case["max_pop"]]
        trials = m * sum(p * (case["steps"] // case["c"] ** i) for i, p in enumerate(pops))
        return {"bytes": 2 * n * sum(pops) + csr + 8 * sum(pops), "flops": trials * terms}
    return {"bytes": 2 * n * (case["pop"] + 1) + csr + 8 * case["pop"], "flops": case["gens"] * m * case["pop"] * terms}


def exact(case, seed):
    """The cut weights in 64-bit integers; a search has no such value besides its own steps."""
    if case["kind"] != "evaluate":
        return None
    state = prepare(case, seed)
    row_ptr, col, weight = state["csr"]
    u = torch.repeat_interleave(torch.arange(state["n"], device="cuda"), row_ptr.diff())
    v, once = col.long(), u < col
    u, v, weight = u[once], v[once], weight[once].long()
    return torch.stack([(weight * (x[u] != x[v])).sum() for x in state["pop"]])
