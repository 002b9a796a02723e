"""Random fills into slices of any alignment and length: the values of an aligned
fill, and nothing written beside the slice.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 2, 3, 4, 5, 7, 8, 1023, 4097])
@pytest.mark.parametrize("offset", [0, 1, 2, 3, 4])
def test_fills_of_slices(n, offset):
    import torch
    from paper_2404_01817_gb300 import neat
    for dtype, fill in ((torch.int32, neat.neat_fill_words), (torch.float32, neat.neat_fill_normal)):
        whole = fill(5, 6, torch.empty(8192, dtype=dtype, device="cuda")).cpu().numpy()
        guarded = torch.full((n + 12,), 77, dtype=dtype, device="cuda")
        fill(5, 6, guarded[offset:offset + n])
        got = guarded.cpu().numpy()
        np.testing.assert_array_equal(got[offset:offset + n], whole[:n])
        assert (got[:offset] == 77).all() and (got[offset + n:] == 77).all()
