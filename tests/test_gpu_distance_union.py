"""Distances from the union tables (one table over a tile's genes) against
those from one hash table per record, which the same records take with room
for more genes: bit for bit.  Every tile width, genomes with none to all 255
genes in common (the counts are bytes), lone and odd a-genomes, the largest
keys (present in some genomes only, so that they are looked up in tables that
lack them), infinite, NaN and signed-zero attributes.
"""
import numpy as np
import pytest

import oracle
from tests.parity import assert_outputs_close
from tests.test_gpu_distance import _pad, _prepare, neat  # noqa: F401

pytestmark = pytest.mark.gpu

TOP = (1 << 24) - 1


def _population(N, C, pop, seed, special):
    """Genomes that share most of a pool of keys; the pool holds TOP and the
    pair (TOP, TOP)."""
    rng = np.random.default_rng(seed)
    pool_n = np.append(rng.choice(TOP, N + N // 4, replace=False), TOP)
    ends = np.append(rng.choice(TOP, 40, replace=False), TOP)
    pairs = np.array([(a, b) for a in ends for b in ends], dtype=np.float32)
    pool_c = np.concatenate([rng.permutation(pairs[:-1])[:C + C // 4], pairs[-1:]])
    nodes = np.full((pop, N, 5), np.nan, np.float32)
    conns = np.full((pop, C, 4), np.nan, np.float32)
    for g in range(pop):
        n = N if g % 3 == 0 else int(rng.integers(0, N + 1))
        m = C if g % 4 == 0 else int(rng.integers(0, C + 1))
        nodes[g, :n, 0] = rng.choice(pool_n, n, replace=False)
        nodes[g, :n, 1:3] = rng.standard_normal((n, 2))
        nodes[g, :n, 3:] = rng.integers(0, 3, (n, 2))
        conns[g, :m, :2] = pool_c[rng.choice(len(pool_c), m, replace=False)]
        conns[g, :m, 2] = rng.integers(0, 2, m)
        conns[g, :m, 3] = rng.standard_normal(m)
    if special:
        for a in (nodes[:, :, 1], conns[:, :, 3]):
            rows = np.argwhere(~np.isnan(a))
            for r, v in zip(rows[rng.choice(len(rows), min(9, len(rows)), replace=False)],
                            (np.inf, -np.inf, np.nan, -0.0, 0.0, 3e38, -3e38, 1e-45, -np.inf)):
                a[tuple(r)] = v
    return nodes, conns


@pytest.mark.parametrize("N,C,pop,reps", [(5, 0, 3, 5), (7, 1, 1, 8), (16, 255, 33, 1), (16, 255, 65, 2),
                                          (16, 255, 18, 4), (50, 200, 131, 21), (24, 60, 700, 9)])
@pytest.mark.parametrize("special", [False, True])
def test_union_tables_agree_with_hash_tables(neat, N, C, pop, reps, special):  # noqa: F811
    nodes, conns = _population(N, C, max(pop, reps), 100 * N + C, special)
    if not special:
        nodes[1:3], conns[1:3] = nodes[0], conns[0]           # all genes in common
    d, genes, st = _prepare(neat, nodes, conns)
    big, big_genes, st_big = _prepare(neat, _pad(nodes, max(N, 256)), _pad(conns, max(C, 256)))
    np.testing.assert_array_equal(st, st_big)
    assert (st == 0).all()
    out = neat.neat_distance(genes, pop, genes, reps, d, 1.0, 0.5).cpu().numpy()
    want = neat.neat_distance(big_genes, pop, big_genes, reps, big, 1.0, 0.5).cpu().numpy()
    np.testing.assert_array_equal(out, want)
    if not special:
        ref, _, _ = oracle.distance(nodes[:pop], conns[:pop], nodes[:reps], conns[:reps], 1.0, 0.5)
        assert_outputs_close(out, ref, what="union tables")
