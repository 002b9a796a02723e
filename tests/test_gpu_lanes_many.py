"""Recurrent lane programs of more genomes than five blocks per SM, where one
warp, two or four share a program by the blocks an SM has room for: the bits of
the recurrent forward on the same records, overlapping launches or not.
"""
import numpy as np
import pytest

from paper_2404_01817_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [16, 32, 44, 64])
@pytest.mark.parametrize("pop", [12160, 12161, 17000])
def test_many_recurrent_programs(N, pop):
    import torch
    from paper_2404_01817_gb300 import neat
    I, O, C = 5, 3, 3 * N
    p = W.random_dag_population_vec(N + pop, pop, I, O, N, C, hidden_max=N - I - O, edge_factors=(1, 3))
    d = neat.dims(I, O, N, C)
    rec, _ = neat.neat_transform_recurrent(torch.from_numpy(p.nodes).cuda(), torch.from_numpy(p.conns).cuda(), d)
    lanes = neat.neat_lanes_pack_recurrent(rec, pop, d)
    stage = neat.neat_lanes_query(lanes).max_warp_bytes
    x = torch.from_numpy(W.normal_inputs(N, (pop, 1, I))).cuda()
    ref = neat.neat_forward_recurrent(rec, pop, d, x, 3).cpu().numpy()
    for pdl in (False, True):
        outs = [neat.neat_forward_lanes_recurrent(lanes, pop, d, x, 3, stage_bytes=stage, pdl=pdl) for _ in range(2)]
        for y in outs:
            np.testing.assert_array_equal(y.cpu().numpy(), ref)
    assert neat.neat_device_error() == 0
