"""One input vector per genome, records above 8 KB and more genomes than a few
waves of staged ones: the default forward reads the records in place.  The same bits as staged evaluation (an explicit
launch shape), with every activation and aggregation, genomes with errors,
node rows at both ends of the range and partial blocks.
"""
import numpy as np
import pytest

from paper_2404_01817_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,C,pop", [(150, 700, 10001), (257, 1000, 6002), (64, 8192, 1201), (1024, 4096, 1603),
                                     (1024, 4096, 7)])
def test_in_place_forward_equals_staged(N, C, pop):
    import torch
    from paper_2404_01817_gb300 import neat
    I, O = 9, 4
    p = W.random_dag_population_vec(N + pop, pop, I, O, N, C, hidden_max=N - I - O, edge_factors=(2, 4))
    rng = np.random.default_rng(N)
    rows = ~np.isnan(p.nodes[:, :, 0])
    p.nodes[:, :, 3][rows] = rng.integers(0, 4, rows.sum())
    p.nodes[:, :, 4][rows] = rng.integers(0, 7, rows.sum())
    p.nodes[0, :, 3:][rows[0]] = (W.AGG_SUM, W.ACT_TANH)
    if pop > 3:
        p.nodes[2, I, 0] = np.nan                                      # a missing output: NaN results
    d = neat.dims(I, O, N, C)
    assert neat.neat_record_stride(d) > 8192
    rec, _ = neat.neat_transform(torch.from_numpy(p.nodes).cuda(), torch.from_numpy(p.conns).cuda(), d)
    x = torch.from_numpy(W.normal_inputs(N, (pop, 1, I))).cuda()
    y = neat.neat_forward(rec, pop, d, x).cpu().numpy()
    shape = neat.neat_default_launch(pop, d, 1)
    np.testing.assert_array_equal(y, neat.neat_forward(rec, pop, d, x, launch=shape).cpu().numpy())
    if pop > 3:
        assert np.isnan(y[2]).all()
