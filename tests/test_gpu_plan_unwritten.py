"""A plan created before its records are written: whatever the buffer holds then
is not followed, and once neat_transform has written them the plan's outputs
equal neat_forward's bit for bit.
"""
import numpy as np
import pytest

from paper_2404_01817_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("word", [0, 0x00010100, 0x00020100, 0x00002000, -1])
@pytest.mark.parametrize("sizes,batch", [((24, 200), 64), ((90,), 1)])
def test_plan_created_before_the_transform(word, sizes, batch):
    import torch
    from paper_2404_01817_gb300 import neat
    pop, I, O = 500, 5, 3
    pops, genomes = [], []
    for N in sizes:
        d = neat.dims(I, O, N, 4 * N)
        p = W.random_dag_population_vec(N, pop, I, O, N, 4 * N, hidden_max=N - I - O, edge_factors=(1, 3))
        rec = torch.full((neat.neat_transformed_bytes(pop, d) // 4,), word, dtype=torch.int32, device="cuda")
        x = torch.from_numpy(W.normal_inputs(N, (pop, batch, I))).cuda()
        pops.append({"transformed": rec, "pop": pop, "dims": d, "inputs": x,
                     "outputs": torch.full((pop, batch, O), 7.0, device="cuda")})
        genomes.append(p)
    plan = neat.Plan(pops)
    for p, q in zip(genomes, pops):
        neat.neat_transform(torch.from_numpy(p.nodes).cuda(), torch.from_numpy(p.conns).cuda(), q["dims"],
                            q["transformed"])
    plan.forward(0)
    for q in pops:
        ref = neat.neat_forward(q["transformed"], pop, q["dims"], q["inputs"])
        np.testing.assert_array_equal(q["outputs"].cpu().numpy(), ref.cpu().numpy())
    assert neat.neat_device_error() == 0
    plan.close()
