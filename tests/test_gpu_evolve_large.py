"""Mutation and crossover of populations large enough for a warp per genome
above 288 and 208 connection rows, and one short of it (a block per genome),
against the oracle: crossover bit for bit, mutation as in the other tests."""
import numpy as np
import pytest

import oracle
from tests.test_gpu_evolve import BUSY, _compare, _configs, _dev, _gpu_mutate, _random_inputs, neat  # noqa: F401
from tests.test_gpu_evolve_forms import _population

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,C", [(73, 289), (128, 512)])
@pytest.mark.parametrize("count", [1499, 1501])
def test_mutation_of_large_populations(neat, N, C, count):  # noqa: F811
    g_cfg, o_cfg = _configs(neat, **BUSY)
    p = _population(N, C, count, N + count)
    u, z = _random_inputs(N + count, count, N, C)
    keys = 7_000_000 + np.arange(count)
    gn, gc = _gpu_mutate(neat, p, g_cfg, u, z, keys)
    on, oc = oracle.mutate(p.nodes, p.conns, 3, 2, o_cfg, u, z, keys)
    _compare(gn, gc, on, oc, f"{N}/{C} x {count}")


@pytest.mark.parametrize("N,C", [(53, 209), (64, 257), (100, 400)])
@pytest.mark.parametrize("more", [-1, 1])
def test_crossover_of_large_populations(neat, N, C, more):  # noqa: F811
    count = 12 * C + more
    p = _population(N, C, count, N + C + more)
    rng = np.random.default_rng(count)
    parents = rng.integers(0, count, size=(count, 2)).astype(np.int32)
    words = rng.integers(0, 2**32, size=(count, N + C), dtype=np.uint64).astype(np.uint32)
    cn, cc = neat.neat_crossover(_dev(p.nodes), _dev(p.conns), neat.dims(3, 2, N, C), _dev(parents),
                                 _dev(words.view(np.int32)))
    on, oc = oracle.crossover(p.nodes, p.conns, parents, words)
    np.testing.assert_array_equal(cn.cpu().numpy(), on)
    np.testing.assert_array_equal(cc.cpu().numpy(), oc)
