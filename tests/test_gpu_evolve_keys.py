"""The cycle check of connection addition on malformed genomes, whose keys reach
beyond 2^24: a key is a node's own only when all of it agrees, in the warp form
and in the block form alike (which of them runs depends on the population's
size), against the oracle.
"""
import numpy as np
import pytest

import oracle
from paper_2404_01817_gb300 import workloads as W
from tests.test_gpu_evolve import _compare, _configs, _gpu_mutate, _random_inputs, neat  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,C,count", [(12, 30, 900), (73, 289, 1499), (73, 289, 1501)])
def test_keys_beyond_24_bits(neat, N, C, count):  # noqa: F811
    big = np.float32(1 << 24)
    g_cfg, o_cfg = _configs(neat, conn_add=1.0, weight_init_std=1.0)
    p = W.random_dag_population_vec(N, count, 3, 2, N, C, hidden_max=N - 5, edge_factors=(1, 3))
    rng = np.random.default_rng(N + count)
    even = np.nan_to_num(p.conns[:, :, :2]) % 2 == 0           # 2^24 + an even key is a float
    # connections from and to keys that no node has but whose low 24 bits a node has
    p.conns[:, :, :2][even & (rng.random(even.shape) < 0.3)] += big
    # and some hidden nodes whose low bits are another node's, with connections of their own
    for g in range(0, count, 2):
        for key in (6, 8, 10):
            if (p.nodes[g, :, 0] == key).any():
                row = int(np.flatnonzero(p.nodes[g, :, 0] == key)[0])
                p.nodes[g, row, 0] = 2 * (key % 3) + big
    u, z = _random_inputs(N, count, N, C)
    u[:, 4] = 0
    keys = 7_000_000 + np.arange(count)
    gn, gc = _gpu_mutate(neat, p, g_cfg, u, z, keys)
    on, oc = oracle.mutate(p.nodes, p.conns, 3, 2, o_cfg, u, z, keys)
    _compare(gn, gc, on, oc, f"{N}/{C} x {count}")
