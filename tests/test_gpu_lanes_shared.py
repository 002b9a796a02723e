"""Recurrent lane programs whose beats one, two or four warps share (chosen
by the number of blocks an SM gets and holds): outputs bit-identical to
neat_forward_recurrent over the sizes where each is taken, fewer beats than
warps, the program staged and read from device memory, and overlapping
launches that follow one another with other inputs."""
import numpy as np
import pytest

from paper_2404_01817_gb300 import workloads as W
from tests.test_gpu_lanes_recurrent import _dev, _prepare, neat  # noqa: F401

pytestmark = pytest.mark.gpu


def _cyclic(seed, pop, N, C):
    I, O = max(1, N // 3), max(1, N // 8)
    p = W.random_dag_population_vec(seed, pop, I, O, N, C, hidden_max=N - I - O, edge_factors=(1, 4))
    rng = np.random.default_rng(seed)
    flip = (p.conns[:, :, 0] >= I) & (p.conns[:, :, 1] >= I) & (rng.random(p.conns.shape[:2]) < 0.5)
    p.conns[flip, :2] = p.conns[flip, 1::-1]
    return p


@pytest.mark.parametrize("N,C,pop", [(3, 4, 17), (5, 8, 5000), (12, 48, 10000), (32, 128, 9729), (32, 128, 6081),
                                     (44, 176, 6080), (50, 200, 10000), (60, 240, 9800), (128, 512, 3000)])
def test_shared_beats_bit_equal(neat, N, C, pop):  # noqa: F811
    p = _cyclic(N + pop, pop, N, C)
    d, rec, st, lanes = _prepare(neat, p)
    assert (st.cpu().numpy() & 0xFF == 0).all()
    xs = [_dev(W.normal_inputs(s, (pop, p.num_inputs))) for s in (1, 2, 3)]
    for K in (1, 2, 7):
        want = [neat.neat_forward_recurrent(rec, pop, d, x.view(pop, 1, -1), K).view(pop, -1).cpu().numpy()
                for x in xs]
        for kw in ({}, {"pdl": True}, {"stage_bytes": 16}):
            got = [neat.neat_forward_lanes_recurrent(lanes, pop, d, x, K, **kw) for x in xs]
            for g, w in zip(got, want):
                np.testing.assert_array_equal(g.cpu().numpy(), w, err_msg=f"K={K} {kw}")
