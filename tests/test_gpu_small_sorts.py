"""Sorts up to 16384 pairs count their digits inside the scatter: both sides of that line, of the tile
of 2048, of one and several 8-bit passes, and all digits equal, against a stable NumPy sort."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [2, 31, 2048, 4095, 16383, 16384, 16385])
@pytest.mark.parametrize("nbits,spread", [(3, 8), (8, 1), (8, 256), (20, 1 << 20), (63, 1 << 62)])
def test_small_sort_pairs_stable(n, nbits, spread):
    import torch
    import paper_2412_18629_gb300 as rs
    ctx = rs.Context(box=10.0, link_len=0.2, softening=0.01, particle_mass=1.0)
    keys = np.random.default_rng(n * 64 + nbits).integers(0, spread, n).astype(np.int64)
    vals = np.arange(n, dtype=np.int32)
    k, v = rs.rs_sort_pairs(ctx, torch.from_numpy(keys).cuda(), torch.from_numpy(vals).cuda(), nbits=nbits)
    order = np.argsort(keys, kind="stable")
    assert np.array_equal(v.cpu().numpy(), vals[order])
    assert np.array_equal(k.cpu().numpy(), keys[order])
