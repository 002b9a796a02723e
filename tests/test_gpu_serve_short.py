"""Requests of a few steps, on both sides of the line where the server copies
their records to compact ones: outputs equal the direct evaluation bit for bit.
"""
import numpy as np
import pytest

from tests.test_gpu_serve import _direct, _request, neat  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("pop,nmax,batch", [(50, 12, 1), (300, 64, 16), (900, 100, 33), (200, 300, 64)])
@pytest.mark.parametrize("steps", [1, 2, 4, 5, 30])
def test_short_requests_equal_direct(neat, pop, nmax, batch, steps):  # noqa: F811
    import torch
    req, p = _request(7, pop, nmax, batch)
    d = neat.dims(p.num_inputs, p.num_outputs, p.max_nodes, p.max_conns)
    y = torch.full((steps, pop, batch, p.num_outputs), float("inf"), device="cuda")
    srv = neat.Server(256 << 20, max_active=4)
    t = srv.submit(p.nodes, p.conns, d, batch, steps, req["seed"], y, out_step_stride=pop * batch * p.num_outputs)
    code, res = srv.wait(t, 60000)
    assert code == neat.NEAT_OK and res.genome_forwards == pop * batch * steps
    direct, _ = _direct(neat, p, batch, steps, req["seed"])
    np.testing.assert_array_equal(y.cpu().numpy(), direct)
    srv.close()
