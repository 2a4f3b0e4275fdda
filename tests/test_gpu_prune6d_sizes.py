"""The batched form's 6D searches on nodes at the edges of their tiles (32-member buckets, 1024-member
superbuckets, 32 superboxes a step, the sampled bounds from 4096 members): the whole hierarchy must
equal the plain form's all-pairs searches bit for bit, for ordinary and for degenerate nodes."""
import numpy as np
import pytest

from helpers import assert_hier_equal

pytestmark = pytest.mark.gpu

SIZES = (10, 31, 32, 33, 64, 65, 1023, 1024, 1025, 1056, 2048, 2049, 4095, 4096, 4097, 5000, 32768, 32800, 34000)
BOX = 100.0


def _node(rng, g, kind):
    """Positions and velocities of one group of g members."""
    centre = rng.uniform(20.0, 80.0, 3)
    r = rng.uniform(0.0, 1.0, g) ** 2.5
    d = rng.normal(size=(g, 3))
    pos = centre + d / np.linalg.norm(d, axis=1, keepdims=True) * r[:, None]
    vel = rng.normal(0.0, 200.0, (g, 3))
    if kind == "lattice":  # many equal distances, repeated points
        pos = centre + rng.integers(0, 6, (g, 3)) * 0.25
        vel = rng.integers(-2, 3, (g, 3)) * 64.0
    elif kind == "cold":  # no velocity dispersion: that term drops out of the metric
        vel[:] = 100.0
    elif kind == "streams":  # separate in velocity only
        vel += 3000.0 * rng.integers(0, 3, (g, 1))
    elif kind == "outliers":
        far = rng.random(g) < 0.02
        pos[far] += rng.normal(0.0, 8.0, (int(far.sum()), 3))
    return pos.astype(np.float32) % np.float32(BOX), vel.astype(np.float32)


@pytest.mark.parametrize("kind", ("cusp", "lattice", "cold", "streams", "outliers"))
def test_searches_equal_all_pairs_at_tile_edges(kind):
    import torch
    import paper_2412_18629_gb300 as rs
    rng = np.random.default_rng(17)
    parts = [_node(rng, g, kind) for g in SIZES]
    pos, vel = np.concatenate([p[0] for p in parts]), np.concatenate([p[1] for p in parts])
    n = len(pos)
    ids = rng.permutation(n).astype(np.int64)
    group = np.repeat(np.arange(len(SIZES)), SIZES)
    least = np.array([ids[group == k].min() for k in range(len(SIZES))])
    order = rng.permutation(n)
    dev = [torch.from_numpy(np.ascontiguousarray(a[order])).cuda() for a in (pos, vel, ids, least[group])]
    got = {}
    for mode in ("plain", "batched"):
        ctx = rs.Context(box=BOX, link_len=0.3, softening=0.01, particle_mass=1e10, mode=mode)
        rs.rs_fof6d(ctx, *dev)
        hier = {k: v.cpu().numpy() for k, v in rs.rs_fof6d_copy(ctx).items()}
        got[mode] = hier, rs.rs_fof6d_node_params(ctx).cpu().numpy().view(np.uint32)
        ctx.close()
    assert_hier_equal(got["batched"][0], got["plain"][0])
    assert np.array_equal(got["batched"][1], got["plain"][1])
    assert sorted(got["plain"][0]["size"][:len(SIZES)]) == sorted(SIZES)
