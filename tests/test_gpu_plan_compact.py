"""A plan's compact records (only the nodes that the outputs depend on): its
outputs equal neat_forward's on the full records bit for bit, at node counts
around the 32-bit words of the node sets, with genomes of no needed nodes, of
nothing but needed ones and with errors; and when the records change under the
plan into ones that outgrow the shapes it chose.
"""
import numpy as np
import pytest

from paper_2404_01817_gb300 import workloads as W

pytestmark = pytest.mark.gpu

I, O = 5, 3


def _genomes(kind, N, C, pop, seed):
    p = W.random_dag_population_vec(seed, pop, I, O, N, C, hidden_max=N - I - O, edge_factors=(1, 3))
    rng = np.random.default_rng(seed)
    rows = ~np.isnan(p.nodes[:, :, 0])
    p.nodes[:, :, 3][rows] = rng.integers(0, 4, rows.sum())
    p.nodes[:, :, 4][rows] = rng.integers(0, 7, rows.sum())
    if kind == "mixed":
        p.conns[0] = np.nan                                    # outputs without connections
        p.nodes[1, I, 0] = np.nan                              # a missing output: an error
        p.conns[2, :, 2] = np.where(np.isnan(p.conns[2, :, 2]), np.nan, 0.0)   # every connection disabled
    else:                                                      # every hidden node feeds an output, all rows used
        p.nodes[:, :, 0] = np.arange(N)
        p.nodes[:, :, 1] = rng.standard_normal((pop, N))
        p.nodes[:, :, 2], p.nodes[:, :, 3], p.nodes[:, :, 4] = 1.0, 0.0, 1.0
        p.conns[:] = np.nan
        for g in range(pop):
            hidden = np.arange(I + O, N)
            k = 0
            for h in hidden[:(C - 1) // 2]:
                p.conns[g, k] = (rng.integers(0, I) if h == I + O else h - 1, h, 1, rng.standard_normal())
                p.conns[g, k + 1] = (h, I + rng.integers(0, O), 1, rng.standard_normal())
                k += 2
    return p


@pytest.mark.parametrize("sizes,batch", [((33, 512), 64), ((31, 32, 64, 1024), 37), ((300,), 130), ((700, 40), 1)])
def test_compact_plan_equals_forward_also_when_the_records_change(sizes, batch):
    import torch
    from paper_2404_01817_gb300 import neat
    pop = 600
    pops, first = [], []
    for j, N in enumerate(sizes):
        d = neat.dims(I, O, N, 4 * N)
        p = _genomes("mixed", N, 4 * N, pop, 10 * N + j)
        rec, _ = neat.neat_transform(torch.from_numpy(p.nodes).cuda(), torch.from_numpy(p.conns).cuda(), d)
        x = torch.from_numpy(W.normal_inputs(N, (2, pop, batch, I))).cuda()
        y = torch.full((2, pop, batch, O), 7.0, device="cuda")
        pops.append({"transformed": rec, "pop": pop, "dims": d, "inputs": x, "outputs": y})
    plan = neat.Plan(pops, autotune=False)

    def check(what):
        for steps in (False, True):
            for p in pops:
                p["outputs"].fill_(7.0)
            if steps:
                plan.forward_steps(0, 2)
            else:
                plan.forward(0)
                plan.forward(1)
            for p in pops:
                for s in range(2):
                    ref = neat.neat_forward(p["transformed"], pop, p["dims"], p["inputs"][s])
                    np.testing.assert_array_equal(p["outputs"][s].cpu().numpy(), ref.cpu().numpy(),
                                                  err_msg=f"{what} {p['dims'].max_nodes} step {s} graph {steps}")
        assert neat.neat_device_error() == 0

    check("as created")
    for p in pops:                                             # other genomes in the same buffers
        d = p["dims"]
        q = _genomes("needed", d.max_nodes, d.max_conns, pop, 3)
        neat.neat_transform(torch.from_numpy(q.nodes).cuda(), torch.from_numpy(q.conns).cuda(), d, p["transformed"])
    check("records changed")
    plan.close()
