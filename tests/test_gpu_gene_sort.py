"""Gene records at the edges of the warp form's sort (one to eight registers
of 32 connection keys, one or two of node keys; 32-bit and 64-bit keys) and
of its loads (batches of 128 rows), against the block form's, which the same
genomes take with one more row than a warp handles: byte for byte, and the
keys against numpy's sort."""
import numpy as np
import pytest

from tests.test_gpu_distance import _pad, _records, _written, neat  # noqa: F401

pytestmark = pytest.mark.gpu

def _repeats(keys):
    keys = keys[~np.isnan(keys)]
    return len(np.unique(keys)) != len(keys)


COUNTS = [0, 1, 2, 31, 32, 33, 64, 65, 96, 97, 127, 128, 129, 160, 161, 192, 193, 224, 225, 255, 256]


@pytest.mark.parametrize("top", [1 << 12, (1 << 12) + 1, 1 << 24])
@pytest.mark.parametrize("N,C", [(64, 256), (33, 129), (5, 1)])
def test_gene_sort_edges(neat, top, N, C):  # noqa: F811
    rng = np.random.default_rng(top + N)
    counts = [m for m in COUNTS if m <= C]
    pop = 2 * len(counts) + 1
    nodes = np.full((pop, N, 5), np.nan, np.float32)
    conns = np.full((pop, C, 4), np.nan, np.float32)
    for g in range(pop):
        m = counts[g % len(counts)]
        n = (g * 7) % (N + 1) if g % 5 else N
        keys = rng.choice(top, n, replace=False)
        if n:
            keys[0] = top - 1
        nodes[g, rng.permutation(N)[:n]] = np.column_stack([keys, rng.standard_normal((n, 2)), rng.integers(0, 3, (n, 2))])
        ends = rng.choice(top, 40, replace=False)
        ends[0] = top - 1
        pick = rng.permutation(1600)[:m]
        conns[g, rng.permutation(C)[:m]] = np.column_stack([ends[pick // 40], ends[pick % 40],
                                                            rng.integers(0, 2, m), rng.standard_normal(m)])
    last = pop - 1                                           # a pair twice, far apart in the rows
    conns[last, 0] = conns[last, C - 1] = (top - 1, 0, 1, 0.5)
    warp, st_w = _records(neat, nodes, conns, 3, 2)
    block, st_b = _records(neat, _pad(nodes, 65), _pad(conns, 257), 3, 2)
    np.testing.assert_array_equal(st_w, st_b)
    twice = np.array([_repeats(nodes[g, :, 0]) or _repeats(conns[g, :, 0].astype(np.float64) * 2.0 ** 24 + conns[g, :, 1])
                      for g in range(pop)])
    np.testing.assert_array_equal(st_w != 0, twice)
    assert twice[last] == (C > 1) and not twice[:last].all()
    for g in range(pop):
        np.testing.assert_array_equal(_written(warp[g]), _written(block[g]), err_msg=f"genome {g}")
    for g in np.flatnonzero(~twice):
        n, m = (int(x) for x in warp[g, :8].view(np.uint32))
        present = nodes[g, ~np.isnan(nodes[g, :, 0]), 0].astype(np.uint32)
        np.testing.assert_array_equal(warp[g, 16:16 + 4 * n].view(np.uint32), np.sort(present))
        off = 16 + (4 * n + 15) // 16 * 16 + 16 * n
        ends = conns[g, ~np.isnan(conns[g, :, 0]), :2].astype(np.uint64)
        np.testing.assert_array_equal(warp[g, off:off + 8 * m].view(np.uint64),
                                      np.sort(ends[:, 0] << np.uint64(24) | ends[:, 1]))
