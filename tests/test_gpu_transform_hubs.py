"""Nodes of many incoming connections in the block form of the transform, whose
rows are sorted before they are searched: in-degrees around the line, several
such nodes in a genome, connection rows in any order with holes, against the
oracle.
"""
import numpy as np
import pytest

import oracle
from paper_2404_01817_gb300 import workloads as W
from tests.parity import assert_outputs_close, assert_topology_equal

pytestmark = pytest.mark.gpu


def _population(N, C, I, degrees, pop):
    """Output j reads degrees[j] of the inputs (one less in odd genomes); hidden nodes follow in a chain."""
    O = len(degrees)
    p = W.empty_population(pop, N, C, I, O)
    rng = np.random.default_rng(N + C)
    for g in range(pop):
        p.nodes[g, :, 0] = np.arange(N)
        p.nodes[g, :, 1] = rng.standard_normal(N)
        p.nodes[g, :, 2], p.nodes[g, :, 3], p.nodes[g, :, 4] = 1.0, W.AGG_SUM, W.ACT_TANH
        rows = [(a, I + j) for j, m in enumerate(degrees) for a in rng.permutation(I)[:m - g % 2]]
        rows += [(I, I + O)] + [(k - 1, k) for k in range(I + O + 1, N)]
        at = np.sort(rng.permutation(C)[:len(rows)]) if g % 3 else rng.permutation(C)[:len(rows)]
        p.conns[g, at, :2] = rows
        p.conns[g, at, 2] = 1.0
        p.conns[g, at, 3] = rng.standard_normal(len(rows)) / 32
        p.nodes[g] = p.nodes[g][rng.permutation(N)]
    return p


@pytest.mark.parametrize("N,C,I,degrees", [(140, 513, 132, (128, 129, 130)), (200, 8192, 150, (150, 127, 129)),
                                           (513, 2100, 500, (500, 500, 128, 500, 129)),
                                           (1024, 8192, 1000, (1000,) * 4 + (128, 129, 256, 1000))])
def test_many_incoming_connections(N, C, I, degrees):
    import torch
    from paper_2404_01817_gb300 import neat
    pop, O = 12, len(degrees)
    p = _population(N, C, I, degrees, pop)
    d = neat.dims(I, O, N, C)
    nodes, conns = torch.from_numpy(p.nodes).cuda(), torch.from_numpy(p.conns).cuda()
    rec, st = neat.neat_transform(nodes, conns, d)
    ref = oracle.transform(p.nodes, p.conns, I, O)
    assert_topology_equal(neat.decode_records(rec.cpu().numpy(), pop, d), ref, pop, f"{N}/{C}")
    np.testing.assert_array_equal(st.cpu().numpy().astype(np.uint32), ref["status"])
    rec, st = neat.neat_transform_recurrent(nodes, conns, d)
    x = W.normal_inputs(N, (pop, 2, I))
    y = neat.neat_forward_recurrent(rec, pop, d, torch.from_numpy(x).cuda(), 2).cpu().numpy()
    expect, status = oracle.forward_recurrent(p.nodes, p.conns, I, O, x, 2)
    np.testing.assert_array_equal(st.cpu().numpy().astype(np.uint32), status)
    assert_outputs_close(y, expect, what=f"recurrent {N}/{C}")
