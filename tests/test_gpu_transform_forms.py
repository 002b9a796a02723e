"""The transform's two forms (a warp per genome up to 128 node rows and 512
connection rows, a block beyond) at the edges of their ranges: records and
status words against the oracle, on well-formed and malformed genomes with
keys far apart, permuted rows and holes.
"""
import numpy as np
import pytest

import oracle
from paper_2404_01817_gb300 import workloads as W
from tests.parity import assert_outputs_close, assert_topology_equal

pytestmark = pytest.mark.gpu

I, O = 3, 2
# (max_nodes, max_conns): around 32-row words, the forms' limits, no connection rows
SIZES = [(5, 0), (7, 1), (31, 33), (32, 128), (33, 31), (64, 257), (65, 129), (127, 511), (128, 512), (128, 513),
         (129, 512), (129, 40), (257, 2049), (500, 2000), (1000, 3)]


@pytest.fixture(scope="module")
def neat():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2404_01817_gb300 import neat as N
    return N


def _population(N, C, pop, seed):
    base = W.random_dag_population_vec(seed, pop, I, O, N, max(C, 1), hidden_max=N - I - O, edge_factors=(1, 4))
    nodes, conns = base.nodes, base.conns[:, :C].copy()
    rng = np.random.default_rng(seed)
    for g in range(pop):
        nv = np.nonzero(~np.isnan(nodes[g, :, 0]))[0]
        nodes[g, nv, 3] = rng.integers(0, 4, nv.size)
        nodes[g, nv, 4] = rng.integers(0, 7, nv.size)
        # hidden keys spread over the whole key range, its largest among them
        keys = np.arange(N, dtype=np.float32)
        hidden = rng.choice((1 << 24) - I - O - 1, N - I - O, replace=False) + I + O
        keys[I + O:] = hidden
        if N > I + O:
            keys[-1] = (1 << 24) - 1
        nodes[g, nv, 0] = keys[nv]
        cv = np.nonzero(~np.isnan(conns[g, :, 0]))[0]
        conns[g, cv, :2] = keys[conns[g, cv, :2].astype(int)]
        free = np.nonzero(np.isnan(conns[g, :, 0]))[0]
        kind = g % 16
        if kind == 1 and cv.size and free.size:                          # a cycle
            conns[g, free[0]] = (conns[g, cv[0], 1], conns[g, cv[0], 0], 1, 0.5)
        elif kind == 2 and nv.size > 1:                                  # duplicate key
            nodes[g, nv[-1], 0] = nodes[g, nv[-2], 0]
        elif kind == 3:                                                  # fractional key
            nodes[g, nv[-1], 0] += 0.5
        elif kind == 4:
            nodes[g, nv[-1], 4] = 7
        elif kind == 5 and cv.size and free.size:                        # duplicate connection
            conns[g, free[-1]] = conns[g, cv[0]]
        elif kind == 6 and cv.size:
            conns[g, cv[-1], 2:] = (1, np.nan)
        elif kind == 7:                                                  # missing output
            nodes[g, I] = np.nan
        elif kind == 8 and free.size:                                    # dangling, once
            conns[g, free[0]] = (1, 999, 1, 1.0)
        elif kind == 9 and free.size > 1:                                # dangling, twice the same
            conns[g, free[0]] = (1, 999, 1, 1.0)
            conns[g, free[-1]] = (1, 999, 0, 2.0)
        elif kind == 10 and free.size > 1:                               # dangling, different
            conns[g, free[0]] = (998, 999, 0, 1.0)
            conns[g, free[-1]] = (999, 998, 1, 2.0)
        elif kind == 11 and free.size:
            conns[g, free[0]] = (I, 0, 1, 1.0)                           # into an input
        elif kind == 12:                                                 # nothing but the inputs and outputs
            nodes[g, I + O:] = np.nan
            conns[g] = np.nan
        elif kind == 13 and cv.size:                                     # a connection key that is none
            conns[g, cv[0], 0] = -1.0
        if kind != 0:
            nodes[g] = nodes[g][rng.permutation(N)]
            conns[g] = conns[g][rng.permutation(C)]
    return W.Population(nodes, np.ascontiguousarray(conns), I, O)


@pytest.mark.parametrize("N,C", SIZES)
def test_transform_forms_match_the_oracle(neat, N, C):
    import torch
    for count in (1, 5, 640):                   # a lone genome, a partial block, several genomes per block
        if count == 640 and N * max(C, 1) > 130 * 600:
            count = 96
        pop = _population(N, C, count, 11 * N + C)
        d = neat.dims(I, O, N, C)
        rec, st = neat.neat_transform(torch.from_numpy(pop.nodes).cuda(), torch.from_numpy(pop.conns).cuda(), d)
        ref = oracle.transform(pop.nodes, pop.conns, I, O)
        assert_topology_equal(neat.decode_records(rec.cpu().numpy(), count, d), ref, count, f"{N}/{C} x {count}")
        np.testing.assert_array_equal(st.cpu().numpy().astype(np.uint32), ref["status"])


@pytest.mark.parametrize("N,C", [(31, 33), (64, 257), (128, 512), (129, 512)])
def test_recurrent_transform_forms(neat, N, C):
    """Positions follow node rows, edges ascend by connection row: after two
    iterations the outputs are the oracle's, with the cycles of the population
    allowed."""
    import torch
    pop = _population(N, C, 48, 5 * N + C)
    rows = ~np.isnan(pop.nodes[:, :, 3])
    pop.nodes[rows, 3], pop.nodes[rows, 4] = W.AGG_SUM, W.ACT_TANH     # bounded values: rounding stays small
    d = neat.dims(I, O, N, C)
    rec, st = neat.neat_transform_recurrent(torch.from_numpy(pop.nodes).cuda(), torch.from_numpy(pop.conns).cuda(), d)
    x = W.normal_inputs(N, (48, 3, I))
    y = neat.neat_forward_recurrent(rec, 48, d, torch.from_numpy(x).cuda(), 2).cpu().numpy()
    ref, status = oracle.forward_recurrent(pop.nodes, pop.conns, I, O, x, 2)
    np.testing.assert_array_equal(st.cpu().numpy().astype(np.uint32), status)
    assert_outputs_close(y, ref, what=f"recurrent {N}/{C}")
