"""Two columns per thread in tiles of 64, which the default forward takes for
33 to 64 vectors of large populations of large genomes: the same bits as tiles of 32 columns with one per thread (an
explicit launch shape), with every activation and aggregation, tanh and sum
alone, nodes of more edges than the straight-line sums hold, errors, and
batches that leave the last pair and the last tile ragged.
"""
import numpy as np
import pytest

from paper_2404_01817_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batch", [33, 37, 64, 65, 129])
@pytest.mark.parametrize("N,C,factors", [(9, 20, (1, 2)), (40, 400, (6, 10)), (101, 403, (2, 4)), (150, 600, (2, 4))])
def test_pairs_equal_single_columns(N, C, factors, batch):
    _compare(N, C, factors, batch, 131)


@pytest.mark.parametrize("batch", [33, 37, 63, 64, 65])
@pytest.mark.parametrize("N,C,factors", [(95, 380, (2, 4)), (96, 960, (6, 10)), (101, 403, (2, 4)), (128, 512, (2, 4))])
@pytest.mark.parametrize("pop", [999, 1000, 1003])
def test_pairs_at_the_limits_of_their_range(N, C, factors, batch, pop):
    _compare(N, C, factors, batch, pop)


def _compare(N, C, factors, batch, pop):
    import torch
    from paper_2404_01817_gb300 import neat
    I, O = 5, 3
    p = W.random_dag_population_vec(N + batch, pop, I, O, N, C, hidden_max=N - I - O, edge_factors=factors)
    rng = np.random.default_rng(N)
    rows = ~np.isnan(p.nodes[:, :, 0])
    p.nodes[:, :, 3][rows] = rng.integers(0, 4, rows.sum())
    p.nodes[:, :, 4][rows] = rng.integers(0, 7, rows.sum())
    half = np.where(np.isnan(p.nodes[:60, :, 0]), np.nan, 1.0)
    p.nodes[:60, :, 3], p.nodes[:60, :, 4] = half * W.AGG_SUM, half * W.ACT_TANH
    p.nodes[7, I, 0] = np.nan                                          # a missing output: NaN results
    d = neat.dims(I, O, N, C)
    rec, _ = neat.neat_transform(torch.from_numpy(p.nodes).cuda(), torch.from_numpy(p.conns).cuda(), d)
    x = torch.from_numpy(W.normal_inputs(N, (pop, batch, I))).cuda()
    y = neat.neat_forward(rec, pop, d, x).cpu().numpy()
    shape = neat.neat_default_launch(pop, d, batch)
    assert shape.tile == 32
    np.testing.assert_array_equal(y, neat.neat_forward(rec, pop, d, x, launch=shape).cpu().numpy())
    assert np.isnan(y[7]).all()
