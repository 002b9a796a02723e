"""Mutation and crossover at the edges of their two forms (a warp per genome
up to 128 node rows and 512 connection rows, a block beyond) against the
oracle: every structural step, rows with holes, a lone genome and partial
blocks.  Structure exactly; mutated values within one float rounding of a
multiply-add (the tolerance of the other evolve tests); crossover bit for bit.
"""
import numpy as np
import pytest

import oracle
from paper_2404_01817_gb300 import workloads as W
from tests.test_gpu_evolve import BUSY, _compare, _configs, _dev, _gpu_mutate, _random_inputs, neat  # noqa: F401

pytestmark = pytest.mark.gpu

SIZES = [(5, 0), (6, 1), (32, 33), (33, 64), (64, 257), (65, 31), (128, 512), (128, 513), (129, 512)]


def _population(N, C, pop, seed):
    p = W.random_dag_population_vec(seed, pop, 3, 2, N, max(C, 1), hidden_max=N - 5, edge_factors=(1, 3))
    nodes, conns = p.nodes, p.conns[:, :C].copy()
    rng = np.random.default_rng(seed)
    keys = np.concatenate([np.arange(5), 5 + rng.choice((1 << 24) - 6, N - 5, replace=False)]).astype(np.float32)
    if N > 5:
        keys[-1] = (1 << 24) - 1
    rows = ~np.isnan(nodes[:, :, 0])
    nodes[:, :, 0][rows] = np.broadcast_to(keys, nodes.shape[:2])[rows]
    c = ~np.isnan(conns[:, :, 0])
    conns[c, :2] = keys[conns[c, :2].astype(int)]
    for g in range(pop):
        nodes[g] = nodes[g][rng.permutation(N)]
        conns[g] = conns[g][rng.permutation(C)]
    return W.Population(np.ascontiguousarray(nodes), np.ascontiguousarray(conns), 3, 2)


@pytest.mark.parametrize("N,C", SIZES)
@pytest.mark.parametrize("feedforward", [1, 0])
def test_mutation_forms(neat, N, C, feedforward):  # noqa: F811
    g_cfg, o_cfg = _configs(neat, **dict(BUSY, feedforward=feedforward))
    for count in (1, 5, 700 if N <= 65 else 90):
        p = _population(N, C, count, 7 * N + C + count)
        u, z = _random_inputs(N + count, count, N, C)
        keys = 7_000_000 + np.arange(count)
        gn, gc = _gpu_mutate(neat, p, g_cfg, u, z, keys)
        on, oc = oracle.mutate(p.nodes, p.conns, 3, 2, o_cfg, u, z, keys)
        _compare(gn, gc, on, oc, f"{N}/{C} x {count}")


@pytest.mark.parametrize("N,C", SIZES)
def test_crossover_forms(neat, N, C):  # noqa: F811
    import torch
    d = neat.dims(3, 2, N, C)
    for count in (1, 5, 700 if N <= 65 else 90):
        p = _population(N, C, count, 5 * N + C + count)
        rng = np.random.default_rng(N + count)
        if C > 2:                                  # the same pair twice in a parent: its lowest row counts
            p.conns[0, -1, :3] = p.conns[0, 0, :3]
        parents = rng.integers(0, count, size=(count, 2)).astype(np.int32)
        parents[-1] = (0, 0)
        words = rng.integers(0, 2**32, size=(count, N + C), dtype=np.uint64).astype(np.uint32)
        cn, cc = neat.neat_crossover(_dev(p.nodes), _dev(p.conns), d, _dev(parents), _dev(words.view(np.int32)))
        torch.cuda.synchronize()
        on, oc = oracle.crossover(p.nodes, p.conns, parents, words)
        np.testing.assert_array_equal(cn.cpu().numpy(), on)
        np.testing.assert_array_equal(cc.cpu().numpy(), oc)
