"""The certified tree walks on nodes at the edges of their tiles (32-member leaves, cells of 256, the
35-entry levels of the stack, short lists), with a normal, a subnormal and a zero squared softening:
the flags equal the plain form's direct sums and every recorded interval holds the float64 sum."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SIZES = (10, 31, 32, 33, 63, 65, 255, 256, 257, 1000, 2047, 2049, 9000)
BOX, MASS, G = 100.0, 1.0e10, 4.30091e-9


@pytest.mark.parametrize("softening", (0.01, 1.0e-22, 0.0))
@pytest.mark.parametrize("theta", (0.0, 0.9))
def test_walks_at_tile_edges(softening, theta):
    import torch
    import paper_2412_18629_gb300 as rs
    rng = np.random.default_rng(23)
    pos, vel = [], []
    for g in SIZES:
        d = rng.normal(size=(g, 3))
        r = rng.uniform(0.01, 1.0, g) ** 2
        pos.append(rng.uniform(20.0, 80.0, 3) + d / np.linalg.norm(d, axis=1, keepdims=True) * r[:, None])
        vel.append(rng.normal(0.0, np.sqrt(G * MASS * g), (g, 3)))  # members on both sides of E = 0
    pos, vel = np.concatenate(pos).astype(np.float32), np.concatenate(vel).astype(np.float32)
    n = len(pos)
    ids = np.arange(n)
    off = np.concatenate([[0], np.cumsum(SIZES)])
    labels = np.repeat(off[:-1], SIZES)
    dev = [torch.from_numpy(a).cuda() for a in (pos, vel, ids, labels)]
    got = {}
    for mode in ("plain", "batched"):
        ctx = rs.Context(box=BOX, link_len=0.3, softening=softening, particle_mass=MASS, mode=mode, tree_min=10,
                         tree_theta=theta)
        rs.rs_fof6d(ctx, *dev)
        if mode == "batched":
            rs.rs_tree_record(ctx, True)
        _, bound, _ = rs.rs_unbind(ctx, dev[0], dev[1], want_potential=mode == "plain")
        got[mode] = bound.cpu().numpy()
        if mode == "batched":
            lo, hi = (t.cpu().numpy() for t in rs.rs_tree_bounds(ctx))
            stats = rs.rs_tree_stats(ctx)
            members = rs.rs_fof6d_copy(ctx)["member_idx"].cpu().numpy()
        ctx.close()
    assert np.array_equal(got["plain"], got["batched"])
    assert 0 < got["plain"].sum() < len(got["plain"])
    assert np.isfinite(lo).all() and stats["tree_members"] == len(lo)
    for a, b in zip(off[:-1], off[1:]):  # level 0: the groups in order of their smallest id
        p = members[a:b]
        u = (pos[p] - pos[p[0]]).astype(np.float64)
        r2 = ((u[:, None, :] - u[None, :, :]) ** 2).sum(2) + float(np.float32(softening)) ** 2
        np.fill_diagonal(r2, np.inf)
        s = (1.0 / np.sqrt(r2)).sum(1)
        assert (lo[a:b] <= s).all() and (s <= hi[a:b]).all()
