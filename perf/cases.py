"""What a user of this framework has it do: population evaluation, control
loops, batched plans, HyperNEAT queries and substrates, recurrent networks,
speciation, one generation of variation, and serving, each through the public
entry points of ``paper_2404_01817_gb300.neat``.

``listed()`` holds one case per kind of use, from the smallest calls to the
largest; ``draw(rng)`` gives more of the same ranges.  ``prepare`` makes the
inputs and what a program keeps between calls, ``run`` is one pass,
``work`` what a pass cannot do without, ``exact`` the same results in 64 bits
from plain torch and numpy.
"""
import math

import numpy as np
import torch

from paper_2404_01817_gb300 import neat
from paper_2404_01817_gb300 import workloads as W

DEV = "cuda"


# ------------------------------------------------------------------ the cases

def listed():
    return [
        # The XOR population: 100 tiny genomes, transformed and evaluated on the
        # 4 input rows.  Two launches; latency is all there is.
        {"name": "xor_eval", "kind": "eval", "pop": 100, "inputs": 3, "outputs": 1, "max_nodes": 10,
         "max_conns": 20, "batch": 4, "mixed": False},
        # A supervised evaluation at odd sizes, every activation and aggregation:
        # a new generation transformed and run on a small data set.
        {"name": "ragged_eval", "kind": "eval", "pop": 1001, "inputs": 13, "outputs": 3, "max_nodes": 101,
         "max_conns": 403, "batch": 37, "mixed": True},
        # Large genomes with one input vector each, beyond the lane programs' limit
        # of 128 nodes: the serving range's largest populations at batch 1.
        {"name": "wide_eval", "kind": "eval", "pop": 4096, "inputs": 27, "outputs": 8, "max_nodes": 500,
         "max_conns": 2000, "batch": 1, "mixed": False},
        # The Ant control loop, the headline: a new population transformed and
        # compiled to lane programs, then 1000 steps as one graph.
        {"name": "ant_episode", "kind": "episode", "pop": 10000, "inputs": 27, "outputs": 8, "max_nodes": 50,
         "max_conns": 200, "steps": 1000},
        # Four populations of uneven sizes in one persistent launch per step.
        {"name": "uneven_plan", "kind": "plan", "pop": 2048, "inputs": 8, "outputs": 4,
         "sizes": "16 64 256 1024", "batch": 64},
        # CPPN genomes queried at every connection of a 16x16 three-layer substrate.
        {"name": "cppn_query", "kind": "cppn", "pop": 1000, "max_nodes": 32, "max_conns": 96, "resolution": 16,
         "layers": 3},
        # The substrates of such a query as controllers: one input vector each.
        {"name": "substrate_step", "kind": "substrate", "pop": 1000, "resolution": 16, "layers": 3, "batch": 1},
        # The same on a batch of 16 inputs (a data set or several environments).
        {"name": "substrate_batch", "kind": "substrate", "pop": 1000, "resolution": 16, "layers": 3, "batch": 16},
        # Recurrent Ant-shaped controllers: transform, compile, 10 control steps of
        # 8 iterations, a call per step.
        {"name": "recurrent_steps", "kind": "recurrent", "pop": 10000, "inputs": 27, "outputs": 8, "max_nodes": 50,
         "max_conns": 200, "batch": 1, "steps": 10, "iterations": 8},
        # Speciation of a generation: gene records, distances to 64
        # representatives, the nearest species.
        {"name": "speciate", "kind": "species", "pop": 10000, "reps": 64, "inputs": 27, "outputs": 8,
         "max_nodes": 50, "max_conns": 200},
        # One generation of variation: random words, crossover, mutation,
        # transform of the children and a first forward of them.
        {"name": "generation", "kind": "evolve", "pop": 10000, "inputs": 27, "outputs": 8, "max_nodes": 50,
         "max_conns": 200},
        # A burst of requests of mixed sizes to the server, waited for.
        {"name": "serve_burst", "kind": "serve", "burst": 1, "requests": 24, "steps": 20, "budget_mb": 256},
    ]


def _logu(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["eval", "eval", "eval", "episode", "plan", "cppn", "substrate", "recurrent", "species",
                       "evolve", "serve"])
    if kind == "eval":
        n = _logu(rng, 8, 512)
        c = {"pop": _logu(rng, 64, 4096), "inputs": min(27, n // 2), "outputs": min(8, max(1, n // 4)),
             "max_nodes": n, "max_conns": 4 * n + rng.randrange(4), "batch": _logu(rng, 1, 256),
             "mixed": rng.random() < 0.5}
        while c["pop"] * c["batch"] * n > 64e6:
            c["batch"] = (c["batch"] + 1) // 2
    elif kind == "episode":
        n = rng.randrange(12, 101)
        c = {"pop": _logu(rng, 100, 10000), "inputs": min(27, n // 2), "outputs": min(8, max(1, n // 4)),
             "max_nodes": n, "max_conns": 4 * n, "steps": _logu(rng, 10, 300)}
    elif kind == "plan":
        sizes = sorted(_logu(rng, 16, 1024) for _ in range(rng.randrange(2, 5)))
        c = {"pop": _logu(rng, 128, 2048), "inputs": 8, "outputs": 4, "sizes": " ".join(map(str, sizes)),
             "batch": _logu(rng, 1, 64)}
    elif kind == "cppn":
        c = {"pop": _logu(rng, 50, 1000), "max_nodes": rng.randrange(12, 33), "max_conns": 96,
             "resolution": rng.randrange(5, 17), "layers": rng.randrange(2, 4)}
    elif kind == "substrate":
        c = {"pop": _logu(rng, 50, 1000), "resolution": rng.randrange(5, 17), "layers": rng.randrange(2, 4),
             "batch": _logu(rng, 1, 16)}
    elif kind == "recurrent":
        n = rng.randrange(12, 81)
        c = {"pop": _logu(rng, 100, 10000), "inputs": min(27, n // 2), "outputs": min(8, max(1, n // 4)),
             "max_nodes": n, "max_conns": 4 * n, "batch": rng.choice([1, 1, _logu(rng, 2, 16)]), "steps": 4,
             "iterations": rng.randrange(2, 11)}
    elif kind == "species":
        n = rng.randrange(16, 101)
        c = {"pop": _logu(rng, 200, 10000), "reps": rng.randrange(3, 100), "inputs": n // 3, "outputs": 1 + n // 10,
             "max_nodes": n, "max_conns": 4 * n + rng.randrange(4)}
    elif kind == "evolve":
        n = rng.randrange(16, 101)
        c = {"pop": _logu(rng, 200, 10000), "inputs": n // 3, "outputs": 1 + n // 10, "max_nodes": n,
             "max_conns": 4 * n + rng.randrange(4)}
    else:
        c = {"burst": rng.randrange(1 << 20), "requests": rng.randrange(8, 25), "steps": rng.randrange(5, 21), "budget_mb": rng.choice([64, 256])}
    c["kind"] = kind
    return c


# --------------------------------------------------------------------- inputs

def _generator(seed, k=0):
    return torch.Generator(device=DEV).manual_seed(int(seed) * 1009 + k)


def _shuffled_rows(conns, gen):
    """The connection rows of each genome in random order, absent ones last
    (evolution appends connections in no topological order)."""
    key = torch.rand(conns.shape[:2], device=DEV, generator=gen)
    key[torch.isnan(conns[:, :, 0])] = 2.0
    at = key.argsort(dim=1)
    return torch.gather(conns, 1, at[:, :, None].expand_as(conns)).contiguous()


def _population(seed, pop, inputs, outputs, max_nodes, max_conns, mixed, factors=(2, 4)):
    """Feedforward genomes: tanh and sum, or every activation and aggregation."""
    p = W.random_dag_population_vec(seed, pop, inputs, outputs, max_nodes, max_conns,
                                    hidden_max=max(max_nodes - inputs - outputs, 0), edge_factors=factors)
    nodes, conns = torch.from_numpy(p.nodes).to(DEV), torch.from_numpy(p.conns).to(DEV)
    gen = _generator(seed, 1)
    if mixed:
        for col, ids in ((3, 4), (4, 7)):
            pick = torch.randint(0, ids, nodes.shape[:2], device=DEV, generator=gen).float()
            nodes[:, :, col] = torch.where(torch.isnan(nodes[:, :, 0]), nodes[:, :, col], pick)
    return nodes, _shuffled_rows(conns, gen)


def _cppns(case, seed):
    nodes, conns = _population(seed, case["pop"], 5, 1, case["max_nodes"], case["max_conns"], False, (1, 3))
    acts = torch.tensor([W.ACT_SIN, W.ACT_GAUSS, W.ACT_TANH, W.ACT_IDENTITY], device=DEV, dtype=torch.float32)
    pick = acts[torch.randint(0, 4, nodes.shape[:2], device=DEV, generator=_generator(seed, 2))]
    nodes[:, :, 4] = torch.where(torch.isnan(nodes[:, :, 0]), nodes[:, :, 4], pick)
    return nodes, conns


def _recurrent_population(case, seed):
    """Genomes whose connections join any node to any non-input one, cycles and
    self-loops among them, each pair once."""
    P, I, O, N, C = (case[k] for k in ("pop", "inputs", "outputs", "max_nodes", "max_conns"))
    gen = _generator(seed, 3)
    n = I + O + torch.randint(0, N - I - O + 1, (P, 1), device=DEV, generator=gen)
    row = torch.arange(N, device=DEV)[None, :]
    nodes = torch.zeros((P, N, 5), device=DEV)
    nodes[:, :, 0] = row
    nodes[:, :, 1] = torch.randn((P, N), device=DEV, generator=gen)
    nodes[:, :, 2] = 1.0
    nodes[:, :, 4] = float(W.ACT_TANH)
    nodes[(row >= n)] = math.nan
    m = n - I
    count = (2 * n + (torch.rand((P, 1), device=DEV, generator=gen) * 2 * n).long()).clamp(max=C)
    pair = (torch.rand((P, C), device=DEV, generator=gen) * (n * m)).long().sort(dim=1).values
    again = torch.zeros((P, C), dtype=torch.bool, device=DEV)
    again[:, 1:] = pair[:, 1:] == pair[:, :-1]
    conns = torch.empty((P, C, 4), device=DEV)
    conns[:, :, 0] = pair // m
    conns[:, :, 1] = I + pair % m
    conns[:, :, 2] = (torch.rand((P, C), device=DEV, generator=gen) >= 0.1).float()
    conns[:, :, 3] = torch.randn((P, C), device=DEV, generator=gen)
    conns[again] = math.nan
    conns = _shuffled_rows(conns, gen)
    conns[torch.arange(C, device=DEV)[None, :] >= count] = math.nan
    return nodes, conns.contiguous()


def _related(case, seed):
    """A population in mid-evolution: many perturbed copies of a hundred
    relatives of one ancestor, with dropped connections, so rows have holes."""
    I, O, N, C = (case[k] for k in ("inputs", "outputs", "max_nodes", "max_conns"))
    free = max(N - I - O, 2)
    base = W.related_population(seed, 100, I, O, N, C, ancestor_hidden=free // 2, ancestor_edges=int(0.6 * C),
                                new_nodes=free // 2, new_conns=int(0.15 * C), key_pool=20, acyclic=True)
    gen = _generator(seed, 4)
    of = torch.randint(0, 100, (case["pop"],), device=DEV, generator=gen)
    nodes, conns = torch.from_numpy(base.nodes).to(DEV)[of], torch.from_numpy(base.conns).to(DEV)[of]
    nodes[:, :, 1] += 0.5 * torch.randn(nodes.shape[:2], device=DEV, generator=gen)
    conns[:, :, 3] += 0.5 * torch.randn(conns.shape[:2], device=DEV, generator=gen)
    flip = torch.rand(conns.shape[:2], device=DEV, generator=gen) < 0.05
    conns[:, :, 2] = torch.where(flip, 1.0 - conns[:, :, 2], conns[:, :, 2])
    conns[torch.rand(conns.shape[:2], device=DEV, generator=gen) < 0.05] = math.nan
    return nodes.contiguous(), conns.contiguous()


def _requests(case, seed=0):
    """The requests of a burst: shapes from the serving ranges (64-4096 genomes,
    8-512 nodes, batch 1-256, log-uniform), genomes and observations by seed."""
    reqs = W.serving_requests(case["burst"], n_requests=case["requests"], steps=case["steps"])
    for i, r in enumerate(reqs):
        r["seed"] = int(seed) * 1009 + i
        while r["pop"] * r["batch"] * r["max_nodes"] > 32e6:
            r["batch"] = (r["batch"] + 1) // 2
    return reqs


def _observations(shape, seed):
    return torch.randn(shape, device=DEV, generator=_generator(seed, 5))


def _dims(case):
    return neat.dims(case["inputs"], case["outputs"], case["max_nodes"], case["max_conns"])


def _mutation():
    """The operator settings of a control task: structural rates 0.2 and 0.4,
    attribute perturbation 0.5 at rates 0.7 and 0.8, replacement 0.1."""
    return neat.mutation(node_add=0.2, conn_add=0.4, bias_init_std=1.0, bias_mutate_power=0.5, bias_mutate_rate=0.7,
                         bias_replace_rate=0.1, weight_init_std=1.0, weight_mutate_power=0.5, weight_mutate_rate=0.8,
                         weight_replace_rate=0.1)


def _plan_populations(case, seed):
    out = []
    for j, n in enumerate(int(s) for s in case["sizes"].split()):
        nodes, conns = _population(seed * 16 + j, case["pop"], case["inputs"], case["outputs"], n, 4 * n, True, (3, 4))
        x = _observations((case["pop"], case["batch"], case["inputs"]), seed * 16 + j)
        out.append((neat.dims(case["inputs"], case["outputs"], n, 4 * n), nodes, conns, x))
    return out


def _substrate_inputs(case, seed):
    R, gen = case["resolution"] ** 2, _generator(seed, 6)
    w = 0.25 * torch.randn((case["pop"], case["layers"] - 1, R, R), device=DEV, generator=gen)
    w[w.abs() < 0.2] = 0.0
    return w, torch.randn((case["pop"], case["batch"], R), device=DEV, generator=gen)


def prepare(case, seed):
    kind, pop = case["kind"], case.get("pop")
    s = {"case": case}
    if kind == "eval":
        d = s["d"] = _dims(case)
        s["nodes"], s["conns"] = _population(seed, pop, d.num_inputs, d.num_outputs, d.max_nodes, d.max_conns,
                                             case["mixed"])
        s["x"] = _observations((pop, case["batch"], d.num_inputs), seed)
        s["records"] = torch.zeros(neat.neat_transformed_bytes(pop, d), dtype=torch.uint8, device=DEV)
        s["status"] = torch.empty(pop, dtype=torch.int32, device=DEV)
        s["y"] = torch.empty((pop, case["batch"], d.num_outputs), device=DEV)
    elif kind == "episode":
        d = s["d"] = _dims(case)
        s["nodes"], s["conns"] = _population(seed, pop, d.num_inputs, d.num_outputs, d.max_nodes, d.max_conns, False)
        s["x"] = _observations((case["steps"], pop, d.num_inputs), seed)
        s["y"] = torch.empty((case["steps"], pop, d.num_outputs), device=DEV)
        # a control program tunes the staging once, on its first population, and
        # keeps its buffers and its graph
        s["records"], s["status"] = neat.neat_transform(s["nodes"], s["conns"], d)
        s["lanes"] = neat.neat_lanes_pack(s["records"], pop, d)
        s["stage"] = neat.neat_lanes_tune(s["lanes"], pop, d, s["x"], s["y"])
        s["cache"] = neat.LanesCache()
    elif kind == "plan":
        s["pops"] = []
        for d, nodes, conns, x in _plan_populations(case, seed):
            records, _ = neat.neat_transform(nodes, conns, d)
            y = torch.empty((pop, case["batch"], d.num_outputs), device=DEV)
            s["pops"].append({"transformed": records, "pop": pop, "dims": d, "inputs": x, "outputs": y})
        s["plan"] = neat.Plan(s["pops"], autotune=True)
    elif kind == "cppn":
        d = s["d"] = neat.dims(5, 1, case["max_nodes"], case["max_conns"])
        s["records"], _ = neat.neat_transform(*_cppns(case, seed), d)
        R = case["resolution"] ** 2
        s["w"] = torch.empty((pop, case["layers"] - 1, R, R), device=DEV)
    elif kind == "substrate":
        s["w"], s["x"] = _substrate_inputs(case, seed)
        s["y"] = torch.empty_like(s["x"])
    elif kind == "recurrent":
        d = s["d"] = _dims(case)
        s["nodes"], s["conns"] = _recurrent_population(case, seed)
        s["x"] = _observations((case["steps"], pop, case["batch"], d.num_inputs), seed)
        s["y"] = torch.empty((case["steps"], pop, case["batch"], d.num_outputs), device=DEV)
        s["records"], s["status"] = neat.neat_transform_recurrent(s["nodes"], s["conns"], d)
        if case["batch"] == 1:
            s["lanes"] = neat.neat_lanes_pack_recurrent(s["records"], pop, d)
            s["stage"] = neat.neat_lanes_query(s["lanes"]).max_warp_bytes
    elif kind == "species":
        d = s["d"] = _dims(case)
        s["nodes"], s["conns"] = _related(case, seed)
        at = torch.randperm(pop, device=DEV, generator=_generator(seed, 7))[:case["reps"]]
        s["rep_nodes"], s["rep_conns"] = s["nodes"][at].contiguous(), s["conns"][at].contiguous()
        stride = neat.neat_gene_stride(d)
        s["genes"] = torch.empty(pop * stride, dtype=torch.uint8, device=DEV)
        s["rep_genes"] = torch.empty(case["reps"] * stride, dtype=torch.uint8, device=DEV)
        s["distances"] = torch.empty((pop, case["reps"]), device=DEV)
    elif kind == "evolve":
        d = s["d"] = _dims(case)
        s["nodes"], s["conns"] = _related(case, seed)
        s["seed"] = int(seed)
        s["parents"] = torch.randint(0, pop, (pop, 2), device=DEV, generator=_generator(seed, 8), dtype=torch.int32)
        words, normals = neat.neat_mutation_sizes(d)
        s["cross_words"] = torch.empty((pop, d.max_nodes + d.max_conns), dtype=torch.int32, device=DEV)
        s["words"] = torch.empty((pop, words), dtype=torch.int32, device=DEV)
        s["normals"] = torch.empty((pop, normals), device=DEV)
        s["keys"] = torch.arange(100000, 100000 + pop, dtype=torch.int32, device=DEV)
        s["child_nodes"], s["child_conns"] = torch.empty_like(s["nodes"]), torch.empty_like(s["conns"])
        s["records"] = torch.zeros(neat.neat_transformed_bytes(pop, d), dtype=torch.uint8, device=DEV)
        s["status"] = torch.empty(pop, dtype=torch.int32, device=DEV)
        s["x"] = _observations((pop, 1, d.num_inputs), seed)
        s["mutation"] = _mutation()
    else:
        s["server"] = neat.Server(case["budget_mb"] << 20)
        s["requests"] = []
        for r in _requests(case, seed):
            p = W.request_population_fast(r)
            y = torch.empty((r["pop"], r["batch"], r["num_outputs"]), device=DEV)
            d = neat.dims(r["num_inputs"], r["num_outputs"], r["max_nodes"], r["max_conns"])
            s["requests"].append((p.nodes, p.conns, d, r["batch"], r["seed"], y))
    return s


# ------------------------------------------------------------------- one pass

def run(s):
    case = s["case"]
    kind, pop, d = case["kind"], case.get("pop"), s.get("d")
    if kind == "eval":
        neat.neat_transform(s["nodes"], s["conns"], d, s["records"], s["status"])
        y = neat.neat_forward(s["records"], pop, d, s["x"], s["y"])
        return y, s["records"], s["status"]
    if kind == "episode":
        neat.neat_transform(s["nodes"], s["conns"], d, s["records"], s["status"])
        neat.neat_lanes_pack(s["records"], pop, d, s["lanes"])
        return neat.neat_forward_lanes_steps(s["lanes"], pop, d, s["x"], s["y"], s["cache"], s["stage"]), s["status"]
    if kind == "plan":
        s["plan"].forward()
        return [p["outputs"] for p in s["pops"]]
    if kind == "cppn":
        return neat.neat_cppn_query(s["records"], pop, d, case["resolution"], case["layers"], weights=s["w"])
    if kind == "substrate":
        return neat.neat_substrate_forward(s["w"], s["x"], case["resolution"], case["layers"], outputs=s["y"])
    if kind == "recurrent":
        neat.neat_transform_recurrent(s["nodes"], s["conns"], d, s["records"], s["status"])
        if case["batch"] == 1:
            neat.neat_lanes_pack_recurrent(s["records"], pop, d, s["lanes"])
        for x, y in zip(s["x"], s["y"]):
            if case["batch"] == 1:
                neat.neat_forward_lanes_recurrent(s["lanes"], pop, d, x, case["iterations"], y, s["stage"], pdl=True)
            else:
                neat.neat_forward_recurrent(s["records"], pop, d, x, case["iterations"], y)
        return s["y"], s["status"]
    if kind == "species":
        neat.neat_distance_prepare(s["nodes"], s["conns"], d, s["genes"])
        neat.neat_distance_prepare(s["rep_nodes"], s["rep_conns"], d, s["rep_genes"])
        dist = neat.neat_distance(s["genes"], pop, s["rep_genes"], case["reps"], d, 1.0, 0.5, s["distances"])
        return dist, neat.neat_speciate(dist, 3.5)
    if kind == "evolve":
        neat.neat_fill_words(s["seed"], 0, s["cross_words"])
        neat.neat_fill_words(s["seed"], 1, s["words"])
        neat.neat_fill_normal(s["seed"], 0, s["normals"])
        neat.neat_crossover(s["nodes"], s["conns"], d, s["parents"], s["cross_words"], s["child_nodes"],
                            s["child_conns"])
        neat.neat_mutate(s["child_nodes"], s["child_conns"], d, s["mutation"], s["words"], s["normals"], s["keys"])
        neat.neat_transform(s["child_nodes"], s["child_conns"], d, s["records"], s["status"])
        y = neat.neat_forward(s["records"], pop, d, s["x"])
        return s["child_nodes"], s["child_conns"], s["records"], s["status"], y
    tickets = [s["server"].submit(nodes, conns, rd, batch, case["steps"], seed, y, borrow=True)
               for nodes, conns, rd, batch, seed, y in s["requests"]]
    for t in tickets:
        code, result = s["server"].wait(t)
        if code != neat.NEAT_OK or result.status != neat.NEAT_OK:
            raise RuntimeError("request %d: %d" % (t, code))
    return [r[-1] for r in s["requests"]]


# ----------------------------------------------------------------------- work

def _genome_bytes(case):
    return 20 * case["max_nodes"] + 16 * case["max_conns"]


def _edges(inputs, outputs, max_nodes, max_conns, lo, hi):
    """About how many enabled connections a drawn genome has."""
    n = (inputs + outputs + max_nodes) / 2
    m = n - inputs
    return 0.9 * min(0.5 * (lo + hi) * n, max_conns, inputs * m + m * m / 2)


def work(case):
    kind, pop = case["kind"], case.get("pop")
    if kind in ("eval", "episode", "recurrent"):
        I, O, N, C = (case[k] for k in ("inputs", "outputs", "max_nodes", "max_conns"))
        vectors = pop * case.get("batch", 1) * case.get("steps", 1)
        edges = _edges(I, O, N, C, 2, 4)
        return {"bytes": pop * _genome_bytes(case) + 4 * vectors * (I + O),
                "flops": 2.0 * vectors * edges * case.get("iterations", 1)}
    if kind == "plan":
        b = f = 0.0
        for n in (int(s) for s in case["sizes"].split()):
            edges, nodes = _edges(case["inputs"], case["outputs"], n, 4 * n, 3, 4), (12 + n) / 2
            vectors = pop * case["batch"]
            b += pop * (16 * nodes + 6 * edges) + 4 * vectors * (case["inputs"] + case["outputs"])
            f += 2.0 * vectors * edges
        return {"bytes": b, "flops": f}
    if kind == "cppn":
        # distinct queries: the layers share one grid, so each (source, target)
        # pair has one value, written to layers - 1 blocks
        R = case["resolution"] ** 2
        edges = _edges(5, 1, case["max_nodes"], case["max_conns"], 1, 3)
        return {"bytes": 4.0 * pop * (case["layers"] - 1) * R * R, "flops": 2.0 * pop * R * R * edges}
    if kind == "substrate":
        R = case["resolution"] ** 2
        cells = pop * (case["layers"] - 1) * R * R
        return {"bytes": 4.0 * cells + 8.0 * pop * case["batch"] * R, "flops": 2.0 * cells * case["batch"]}
    if kind == "species":
        genes = 0.8 * (case["max_nodes"] + case["max_conns"])
        return {"bytes": (pop + case["reps"]) * _genome_bytes(case) + pop * (4.0 * case["reps"] + 4),
                "flops": 4.0 * pop * case["reps"] * genes}
    if kind == "evolve":
        # both parents read, the child written; the random numbers are made on the way
        return {"bytes": 3.0 * pop * _genome_bytes(case) + 4.0 * pop * (case["inputs"] + case["outputs"]),
                "flops": 10.0 * pop * (case["max_nodes"] + case["max_conns"])}
    b = f = 0.0
    for r in _requests(case):
        I, O, N, C = r["num_inputs"], r["num_outputs"], r["max_nodes"], r["max_conns"]
        vectors = r["pop"] * r["batch"] * r["steps"]
        b += r["pop"] * (20 * N + 16 * C) + 4.0 * vectors * O
        f += 2.0 * vectors * _edges(I, O, N, C, 2, 4)
    return {"bytes": b, "flops": f}


# ------------------------------------------------------------ 64-bit results

def _act(z, act):
    return [lambda: z, lambda: torch.tanh(z), lambda: torch.sigmoid(z), lambda: torch.relu(z), lambda: torch.sin(z),
            lambda: torch.exp(-z * z), lambda: z.abs()][act]()


class _Networks:
    """The networks of a population in 64 bits, for genomes whose node keys are
    their rows: values are [pop * max_nodes][columns]."""

    def __init__(self, nodes, conns, inputs, outputs):
        self.P, self.N = nodes.shape[:2]
        self.I, self.O = inputs, outputs
        flat = nodes.reshape(-1, 5)
        self.bias, self.response = flat[:, 1].double(), flat[:, 2].double()
        present = ~torch.isnan(flat[:, 0])
        at = torch.arange(self.P * self.N, device=DEV)
        used = present & (at % self.N >= inputs)
        self.agg = torch.where(used, flat[:, 3], -1.0).long()
        self.act = torch.where(used, flat[:, 4], -1.0).long()
        c = conns.reshape(-1, 4)
        g = torch.arange(self.P, device=DEV).repeat_interleave(conns.shape[1])
        on = ~torch.isnan(c[:, 0]) & (c[:, 2] != 0)
        c, g = c[on], g[on]
        src, dst = g * self.N + c[:, 0].long(), g * self.N + c[:, 1].long()
        by = dst.argsort(stable=True)
        self.src, self.dst, self.w = src[by], dst[by], c[by, 3].double()
        self.degree = torch.bincount(self.dst, minlength=self.P * self.N)
        self.first = self.degree.cumsum(0) - self.degree
        self.used = used

    def groups(self, where):
        """The used nodes among `where`, by aggregation, largest degree first."""
        out = []
        for agg in range(4):
            ids = torch.nonzero(where & self.used & (self.agg == agg)).flatten()
            if ids.numel():
                ids = ids[self.degree[ids].argsort(descending=True)]
                deg = self.degree[ids]
                counts = [int(k) for k in (deg[None, :] > torch.arange(int(deg[0]), device=DEV)[:, None]).sum(1)]
                out.append((agg, ids, counts))
        return out

    def evaluate(self, groups, v):
        """New values of the groups' nodes from the values v."""
        for agg, ids, counts in groups:
            acc = torch.zeros((ids.numel(), v.shape[1]), dtype=torch.float64, device=DEV)
            for k, m in enumerate(counts):
                e = self.first[ids[:m]] + k
                t = self.w[e][:, None] * v[self.src[e]]
                if k == 0:
                    acc[:m] = t
                elif agg == 1:
                    acc[:m] *= t
                elif agg == 2:
                    acc[:m] = torch.fmax(acc[:m], t)
                else:
                    acc[:m] += t
            if agg == 3:
                acc /= self.degree[ids].clamp(min=1)[:, None]
            z = self.bias[ids][:, None] + self.response[ids][:, None] * acc
            del acc
            act = self.act[ids]
            kinds = act.unique().tolist()
            if len(kinds) == 1:
                z = _act(z, kinds[0])
            else:
                for a in kinds:
                    m = act == a
                    z[m] = _act(z[m], a)
            yield ids, z

    def start(self, x):
        """Values with the inputs x [P][B][I] in place, 0 elsewhere."""
        v = torch.zeros((self.P, self.N, x.shape[1]), dtype=torch.float64, device=DEV)
        v[:, :self.I] = x.double().transpose(1, 2)
        return v.view(self.P * self.N, -1)

    def outputs(self, v):
        return v.view(self.P, self.N, -1)[:, self.I:self.I + self.O].transpose(1, 2)

    def levels(self):
        depth = torch.zeros(self.P * self.N, dtype=torch.int64, device=DEV)
        while True:
            new = torch.zeros_like(depth).scatter_reduce_(0, self.dst, depth[self.src] + 1, "amax")
            if torch.equal(new, depth):
                return [self.groups(depth == k) for k in range(int(depth.max()) + 1)]
            depth = new

    def forward(self, x, levels=None):
        v = self.start(x)
        for groups in levels or self.levels():
            for ids, z in list(self.evaluate(groups, v)):
                v[ids] = z
        return self.outputs(v)

    def iterate(self, x, iterations):
        v = self.start(x)
        groups = self.groups(self.used)
        for _ in range(iterations):
            new = v.clone()
            for ids, z in self.evaluate(groups, v):
                new[ids] = z
            v = new
        return self.outputs(v)


def _as_float32_range(y):
    """Values beyond float32's range as the infinities that they become there."""
    return torch.where(y.abs() > 3.4028235e38, y.sign() * math.inf, y)


def _philox_normals(seed, step, count):
    """neat_fill_normal's values from its definition: Philox-4x32-10 (Salmon et
    al., SC 2011) on counter (block, step, 0x4f4253), Box-Muller on word pairs."""
    blk = np.arange((count + 3) // 4, dtype=np.uint64)
    low = np.uint64(0xFFFFFFFF)
    c = [blk & low, blk >> np.uint64(32), np.full_like(blk, step), np.full_like(blk, 0x4F4253)]
    k0, k1 = seed & 0xFFFFFFFF, seed >> 32
    for _ in range(10):
        p0, p1 = np.uint64(0xD2511F53) * c[0], np.uint64(0xCD9E8D57) * c[2]
        c = [(p1 >> np.uint64(32)) ^ c[1] ^ np.uint64(k0), p1 & low, (p0 >> np.uint64(32)) ^ c[3] ^ np.uint64(k1),
             p0 & low]
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    u = [((x >> np.uint64(8)).astype(np.float64) + 0.5) / 16777216.0 for x in c]
    r0, r1 = np.sqrt(-2 * np.log(u[0])), np.sqrt(-2 * np.log(u[2]))
    t0, t1 = 2 * np.pi * u[1], 2 * np.pi * u[3]
    return np.stack([r0 * np.cos(t0), r0 * np.sin(t0), r1 * np.cos(t1), r1 * np.sin(t1)], 1).reshape(-1)[:count]


def _exact_distances(nodes, conns, reps_n, reps_c):
    """The genome distance with coefficients 1 and 0.5, by dense tables over the
    distinct node keys and connection pairs."""
    def table(rows, code, values):
        on = ~torch.isnan(code)
        ids, of = torch.unique(code[on].long(), return_inverse=True)
        g = torch.nonzero(on)[:, 0]
        has = torch.zeros((rows, ids.numel()), dtype=torch.float64, device=DEV)
        has[g, of] = 1.0
        cols = []
        for v in values:
            t = torch.zeros_like(has)
            t[g, of] = v[on].double()
            cols.append(t)
        return has, cols

    P = nodes.shape[0]
    n, c = torch.cat([nodes, reps_n]), torch.cat([conns, reps_c])
    out = torch.zeros((P, reps_n.shape[0]), dtype=torch.float64, device=DEV)
    pair = c[:, :, 0].double() * 2.0 ** 24 + c[:, :, 1].double()
    for code, values, whole in ((n[:, :, 0].double(), [n[:, :, k] for k in (1, 2, 3, 4)], (2, 3)),
                                (pair, [c[:, :, 3], (c[:, :, 2] != 0).float()], (1,))):
        has, cols = table(n.shape[0], code, values)
        count = has.sum(1)
        for j in range(reps_n.shape[0]):
            both = has[:P] * has[P + j]
            off = sum(((t[:P] - t[P + j]) != 0).double() if k in whole else (t[:P] - t[P + j]).abs()
                      for k, t in enumerate(cols))
            disjoint = count[:P] + count[P + j] - 2 * both.sum(1)
            most = torch.maximum(count[:P], count[P + j]).clamp(min=1)
            out[:, j] += (disjoint + 0.5 * (off * both).sum(1)) / most
    return out


def exact(case, seed):
    kind, pop = case["kind"], case.get("pop")
    if kind in ("eval", "episode"):
        nodes, conns = _population(seed, pop, case["inputs"], case["outputs"], case["max_nodes"], case["max_conns"],
                                   case.get("mixed", False))
        net = _Networks(nodes, conns, case["inputs"], case["outputs"])
        levels = net.levels()
        if kind == "eval":
            x = _observations((pop, case["batch"], case["inputs"]), seed)
            return _as_float32_range(net.forward(x, levels)), None, None
        x = _observations((case["steps"], pop, case["inputs"]), seed).transpose(0, 1)
        return torch.cat([net.forward(part, levels).transpose(0, 1) for part in x.split(250, dim=1)]), None
    if kind == "plan":
        return [_as_float32_range(_Networks(nodes, conns, case["inputs"], case["outputs"]).forward(x))
                for _, nodes, conns, x in _plan_populations(case, seed)]
    if kind == "cppn":
        nodes, conns = _cppns(case, seed)
        res = case["resolution"]
        grid = (-1 + 2 * torch.arange(res, device=DEV, dtype=torch.float64) / (res - 1)).float()
        xy = torch.stack([grid.repeat(res), grid.repeat_interleave(res)], 1)
        R = res * res
        q = torch.cat([xy.repeat_interleave(R, 0), xy.repeat(R, 1), torch.ones(R * R, 1, device=DEV)], 1)
        parts = []
        for g in range(0, pop, 50):
            net = _Networks(nodes[g:g + 50], conns[g:g + 50], 5, 1)
            w = net.forward(q[None].expand(net.P, -1, -1)).reshape(net.P, 1, R, R)
            w = torch.where(w.float().abs() < np.float32(0.2), 0.0, w)
            parts.append(w.expand(-1, case["layers"] - 1, -1, -1))
        return torch.cat(parts)
    if kind == "substrate":
        w, v = _substrate_inputs(case, seed)
        v = v.double()
        for k in range(case["layers"] - 1):
            v = torch.tanh(torch.bmm(v, w[:, k].double()))
        return v
    if kind == "recurrent":
        net = _Networks(*_recurrent_population(case, seed), case["inputs"], case["outputs"])
        x = _observations((case["steps"], pop, case["batch"], case["inputs"]), seed)
        return torch.stack([net.iterate(step, case["iterations"]) for step in x]), None
    if kind == "species":
        nodes, conns = _related(case, seed)
        at = torch.randperm(pop, device=DEV, generator=_generator(seed, 7))[:case["reps"]]
        return _exact_distances(nodes, conns, nodes[at], conns[at]), None
    if kind == "serve":
        out = []
        for r in _requests(case, seed):
            p = W.request_population_fast(r)
            net = _Networks(torch.from_numpy(p.nodes).to(DEV), torch.from_numpy(p.conns).to(DEV), r["num_inputs"],
                            r["num_outputs"])
            x = _philox_normals(r["seed"], r["steps"] - 1, r["pop"] * r["batch"] * r["num_inputs"])
            x = torch.from_numpy(x).to(DEV).reshape(r["pop"], r["batch"], r["num_inputs"])
            out.append(net.forward(x))
        return out
    # a generation's numbers are copies of genes and single rounded updates of
    # them, chosen by random words: there is no more exact value to give
    return None
