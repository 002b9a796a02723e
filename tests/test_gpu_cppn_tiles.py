"""The query kernel's value tiles (512, 256 and 128 columns) and edge forms
(widened, or as in the record where those do not fit), chosen from the dims:
weights equal neat_forward's outputs on the same coordinates bit for bit, at
resolutions whose pair counts leave a thread's four columns ragged.
"""
import numpy as np
import pytest

from paper_2404_01817_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nmax,cmax", [(6, 0), (6, 8), (90, 300), (150, 3000), (100, 7000)])
@pytest.mark.parametrize("res,layers", [(2, 4), (3, 2), (7, 3)])
def test_cppn_tiles_equal_forward(nmax, cmax, res, layers):
    import torch
    from paper_2404_01817_gb300 import neat
    P = 9
    pop = W.random_dag_population(17 + nmax, P, 5, 1, nmax, cmax, hidden=lambda r: int(r.integers(0, nmax - 5)),
                                  edges=lambda r, n: min(cmax, int(r.integers(n, 5 * n))), acts=W.ALL_ACTS,
                                  aggs=W.ALL_AGGS)
    pop.nodes[0, :, 3] = np.where(np.isnan(pop.nodes[0, :, 0]), np.nan, W.AGG_SUM)      # sums only
    d = neat.dims(5, 1, nmax, cmax)
    rec, _ = neat.neat_transform(torch.from_numpy(pop.nodes).cuda(), torch.from_numpy(pop.conns).cuda(), d)
    w = neat.neat_cppn_query(rec, P, d, res, layers, 0.0).cpu().numpy()
    coord = (-1.0 + 2.0 * np.arange(res) / (res - 1)).astype(np.float32)
    node = np.arange(res * res)
    s, t = (i.ravel() for i in np.meshgrid(node, node, indexing="ij"))
    x = np.stack([coord[s % res], coord[s // res], coord[t % res], coord[t // res], np.ones(s.size, np.float32)], 1)
    xb = torch.from_numpy(np.ascontiguousarray(np.broadcast_to(x, (P,) + x.shape))).cuda()
    y = neat.neat_forward(rec, P, d, xb).cpu().numpy()[:, :, 0]
    for block in range(layers - 1):
        np.testing.assert_array_equal(w[:, block].reshape(P, -1), y)
