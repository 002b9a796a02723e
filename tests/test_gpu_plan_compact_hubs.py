"""Compact copies of records whose nodes have more edges than one lane goes through
(around 32, and hundreds): a plan that makes copies equals neat_forward on the
full records bit for bit.
"""
import numpy as np
import pytest

from paper_2404_01817_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("degrees", [(31, 32, 33, 34), (200, 200, 64, 1), (129, 0, 200, 128)])
def test_compact_copies_of_many_edges(degrees):
    import torch
    from torch.profiler import ProfilerActivity, profile
    from paper_2404_01817_gb300 import neat
    pop, I, O, hidden, batch = 1200, 200, len(degrees), 160, 32
    N, C = I + O + hidden, 1400
    p = W.empty_population(pop, N, C, I, O)
    rng = np.random.default_rng(sum(degrees))
    p.nodes[:, :, 0] = np.arange(N)
    p.nodes[:, :, 1] = rng.standard_normal((pop, N))
    p.nodes[:, :, 2], p.nodes[:, :, 3], p.nodes[:, :, 4] = 1.0, W.AGG_SUM, W.ACT_TANH
    rows = [(a, I + j) for j, m in enumerate(degrees) for a in rng.permutation(I)[:m]]
    rows += [(a, I + O + k) for k in range(hidden) for a in rng.permutation(I)[:3]]     # nothing reads these but the first
    rows.append((I + O, I))
    rows = np.array(rows)[rng.permutation(len(rows))]
    p.conns[:, :len(rows), :2] = rows
    p.conns[:, :len(rows), 2] = 1.0
    p.conns[:, :len(rows), 3] = rng.standard_normal((pop, len(rows))) / 8
    d = neat.dims(I, O, N, C)
    rec, _ = neat.neat_transform(torch.from_numpy(p.nodes).cuda(), torch.from_numpy(p.conns).cuda(), d)
    x = torch.from_numpy(W.normal_inputs(1, (pop, batch, I))).cuda()
    y = torch.full((pop, batch, O), 7.0, device="cuda")
    plan = neat.Plan([{"transformed": rec, "pop": pop, "dims": d, "inputs": x, "outputs": y}])
    names = []
    for _ in range(3):                                 # a process's first session may come back empty
        with profile(activities=[ProfilerActivity.CUDA]) as prof:
            plan.forward(0)
            torch.cuda.synchronize()
        names = [e.name for e in prof.events()]
        if names:
            break
    assert any("compact_kernel" in n for n in names), names
    np.testing.assert_array_equal(y.cpu().numpy(), neat.neat_forward(rec, pop, d, x).cpu().numpy())
    assert neat.neat_device_error() == 0
    plan.close()
