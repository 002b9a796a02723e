"""The substrate query on records of neat_transform_recurrent, which hold no
order: evaluated in node row order, so a genome whose nodes come after what
they read has the weights of neat_transform's record bit for bit, and one in
which a node that the output depends on reads a later row (or itself) has NaN.
"""
import numpy as np
import pytest

from paper_2404_01817_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _edges(p, g):
    c = p.conns[g]
    return c[~np.isnan(c[:, 0]) & (c[:, 2] != 0.0), :2].astype(int)


def _topological_rows(p, g):
    """Rows of genome g, every node after the nodes that its enabled connections read."""
    key = {int(k): r for r, k in enumerate(p.nodes[g, :, 0]) if not np.isnan(k)}
    reads = {k: set() for k in key}
    for a, b in _edges(p, g):
        if a in key and b in key:
            reads[b].add(a)
    done, rows = set(), []
    while len(done) < len(key):
        ready = [k for k in key if k not in done and reads[k] <= done]
        rows += [key[k] for k in ready]
        done |= set(ready)
    return rows + [r for r in range(p.max_nodes) if r not in rows]


def _in_row_order(p, g):
    """Whether every node that the output (key 5) depends on reads earlier rows or inputs only."""
    key = {int(k): r for r, k in enumerate(p.nodes[g, :, 0]) if not np.isnan(k)}
    edges = [(a, b) for a, b in _edges(p, g) if a in key and b in key and b >= 5]
    need, grown = {5}, True
    while grown:
        more = {a for a, b in edges if b in need} - need
        need |= more
        grown = bool(more)
    return all(a < 5 or key[a] < key[b] for a, b in edges if b in need)


@pytest.mark.parametrize("nmax,cmax", [(6, 8), (33, 96), (64, 200), (150, 600)])
@pytest.mark.parametrize("res,layers", [(3, 2), (7, 3)])
def test_cppn_query_of_recurrent_records(nmax, cmax, res, layers):
    import torch
    from paper_2404_01817_gb300 import neat
    P = 24
    p = W.random_dag_population(31 + nmax, P, 5, 1, nmax, cmax, hidden=lambda r: int(r.integers(0, nmax - 5)),
                                edges=lambda r, n: min(cmax - 1, int(r.integers(n, 4 * n))), acts=W.ALL_ACTS,
                                aggs=W.ALL_AGGS)
    rng = np.random.default_rng(nmax)
    for g in range(P):
        if g % 3 == 0:
            p.nodes[g] = p.nodes[g][_topological_rows(p, g)]
        elif g % 3 == 1:                                   # inputs anywhere; the rest as drawn, or mixed
            p.nodes[g] = p.nodes[g][rng.permutation(nmax)]
    p.conns[2, -1] = (5, 5, 1, 0.5)                        # the output reads itself
    p.nodes[3, 0, 3] = 9.0                                 # an error
    d = neat.dims(5, 1, nmax, cmax)
    nodes, conns = torch.from_numpy(p.nodes).cuda(), torch.from_numpy(p.conns).cuda()
    ordered, _ = neat.neat_transform(nodes, conns, d)
    rows, status = neat.neat_transform_recurrent(nodes, conns, d)
    expect = neat.neat_cppn_query(ordered, P, d, res, layers, 0.1).cpu().numpy()
    got = neat.neat_cppn_query(rows, P, d, res, layers, 0.1).cpu().numpy()
    follows = [_in_row_order(p, g) and not int(status[g]) & neat.G_ERROR_MASK for g in range(P)]
    assert sum(follows) >= P // 3 - 1 and not follows[2] and not follows[3]
    for g in range(P):
        np.testing.assert_array_equal(got[g], expect[g] if follows[g] else np.full_like(got[g], np.nan), err_msg=str(g))
    assert neat.neat_device_error() == 0
