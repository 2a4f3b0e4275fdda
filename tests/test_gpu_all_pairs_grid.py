"""The all-pairs 6D kernels on a node with more work items (128 members against 1024 targets each) than
their grid has blocks: a block takes several, and the hierarchy and the split parameters equal those of the
batched form's searches bit for bit."""
import numpy as np
import pytest

from helpers import assert_hier_equal

pytestmark = pytest.mark.gpu

MAX_BLOCKS = 1 << 16  # of the all-pairs kernels
SIZES = (100001, 40000, 12)


def test_more_items_than_blocks():
    import torch
    import paper_2412_18629_gb300 as rs
    assert sum(-(-g // 128) * -(-g // 1024) for g in SIZES) > MAX_BLOCKS
    rng = np.random.default_rng(31)
    n = sum(SIZES)
    pos = (50.0 + rng.normal(0.0, 1.0, (n, 3)) * rng.uniform(0.0, 1.0, (n, 1)) ** 2).astype(np.float32)
    vel = (rng.normal(0.0, 200.0, (n, 3)) + 2000.0 * rng.integers(0, 3, (n, 1))).astype(np.float32)
    off = np.concatenate([[0], np.cumsum(SIZES)])
    labels = np.repeat(off[:-1], SIZES)
    dev = [torch.from_numpy(a).cuda() for a in (pos, vel, np.arange(n), labels)]
    got = {}
    for mode in ("plain", "batched"):
        ctx = rs.Context(box=100.0, link_len=0.3, softening=0.01, particle_mass=1e10, mode=mode)
        rs.rs_fof6d(ctx, *dev)
        got[mode] = ({k: v.cpu().numpy() for k, v in rs.rs_fof6d_copy(ctx).items()},
                     rs.rs_fof6d_node_params(ctx).cpu().numpy().view(np.uint32))
        ctx.close()
    assert_hier_equal(got["plain"][0], got["batched"][0])
    assert np.array_equal(got["plain"][1], got["batched"][1])
    assert got["plain"][0]["level"].max() > 0
