"""Two columns per thread where the default forward takes it: 33 to 64 vectors of
genomes of 64 to 255 node rows, enough of them to fill the device (up to 127
rows: few enough to fit it at once, or many more).  The form that ran is read from the
profiler's kernel names; outputs equal tiles of 32 columns (an explicit launch
shape) bit for bit, with every activation and aggregation, tanh and sum alone,
nodes of more edges than the straight-line sums hold, and errors.
"""
import numpy as np
import pytest

from paper_2404_01817_gb300 import workloads as W

pytestmark = pytest.mark.gpu

PAIRS = "forward_kernel<false, false, true>"


def _kernels(call):
    import torch
    from torch.profiler import ProfilerActivity, profile
    for _ in range(3):                                 # a process's first session may come back empty
        with profile(activities=[ProfilerActivity.CUDA]) as prof:
            out = call()
            torch.cuda.synchronize()
        names = [e.name for e in prof.events() if "forward" in e.name]
        if names:
            break
    return out, names


# (rows, connection rows, genomes, edge factors, pairs): the lines of 64, 128 and
# 256 rows, too few genomes, too many for one wave, groups too large for three on an SM
CASES = [(63, 252, 900, (2, 4), False), (64, 640, 900, (6, 10), True), (101, 403, 1001, (2, 4), True),
         (127, 508, 760, (2, 4), True), (127, 508, 800, (2, 4), False), (101, 403, 600, (2, 4), False),
         (101, 403, 1500, (2, 4), False), (101, 403, 2400, (2, 4), True),
         (128, 512, 500, (2, 4), True), (128, 1280, 3001, (6, 10), True), (128, 512, 300, (2, 4), False),
         (200, 800, 501, (2, 4), True), (255, 600, 700, (1, 2), True), (256, 700, 700, (1, 2), False),
         (200, 4000, 600, (2, 4), False)]


@pytest.mark.parametrize("batch", [33, 37, 63, 64])
@pytest.mark.parametrize("N,C,pop,factors,pairs", CASES)
def test_pairs_taken_and_equal(N, C, pop, factors, pairs, batch):
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
    y, names = _kernels(lambda: neat.neat_forward(rec, pop, d, x))
    assert len(names) == 1 and (PAIRS in names[0]) == pairs, names
    shape = neat.neat_default_launch(pop, d, batch)
    assert shape.tile == 32
    np.testing.assert_array_equal(y.cpu().numpy(), neat.neat_forward(rec, pop, d, x, launch=shape).cpu().numpy())
    assert np.isnan(y[7].cpu().numpy()).all()
