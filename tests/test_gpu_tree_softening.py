"""The certified tree walks at softenings far below the members' spacing, whose square is still a normal
float32: a member's own term 1 / eps is then up to 1e18 times a neighbour's, and must not touch its sum.
Every recorded interval holds the float64 sum and the flags equal the plain form's direct sums, in nodes
of one leaf, of several and of several levels."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SIZES = (20, 33, 300, 2049, 9000)
BOX, MASS, G = 100.0, 1.0e10, 4.30091e-9


@pytest.mark.parametrize("softening", (1.0e-4, 1.0e-6, 1.0e-8, 1.0e-10, 1.0e-12, 1.0e-18))
def test_intervals_hold_at_small_softening(softening):
    import torch
    import paper_2412_18629_gb300 as rs
    rng = np.random.default_rng(29)
    pos, vel = [], []
    for g in SIZES:
        d = rng.normal(size=(g, 3))
        r = rng.uniform(0.01, 1.0, g) ** 2
        pos.append(rng.uniform(20.0, 80.0, 3) + d / np.linalg.norm(d, axis=1, keepdims=True) * r[:, None])
        vel.append(rng.normal(0.0, np.sqrt(G * MASS * g), (g, 3)))  # members on both sides of E = 0
    pos, vel = np.concatenate(pos).astype(np.float32), np.concatenate(vel).astype(np.float32)
    ids = np.arange(len(pos))
    off = np.concatenate([[0], np.cumsum(SIZES)])
    dev = [torch.from_numpy(a).cuda() for a in (pos, vel, ids, np.repeat(off[:-1], SIZES))]
    got = {}
    for mode in ("plain", "batched"):
        ctx = rs.Context(box=BOX, link_len=0.3, softening=softening, particle_mass=MASS, mode=mode, tree_min=10)
        rs.rs_fof6d(ctx, *dev)
        rs.rs_tree_record(ctx, mode == "batched")
        _, bound, _ = rs.rs_unbind(ctx, dev[0], dev[1], want_potential=mode == "plain")
        got[mode] = bound.cpu().numpy()
        if mode == "batched":
            lo, hi = (t.cpu().numpy() for t in rs.rs_tree_bounds(ctx))
            members = rs.rs_fof6d_copy(ctx)["member_idx"].cpu().numpy()
        ctx.close()
    assert np.isfinite(lo).all() and np.isfinite(hi).all()
    outside = 0
    for a, b in zip(off[:-1], off[1:]):  # level 0: the groups in order of their smallest id
        p = members[a:b]
        u = (pos[p] - pos[p[0]]).astype(np.float64)
        r2 = ((u[:, None, :] - u[None, :, :]) ** 2).sum(2) + float(np.float32(softening)) ** 2
        np.fill_diagonal(r2, np.inf)
        s = (1.0 / np.sqrt(r2)).sum(1)
        outside += int(((s < lo[a:b]) | (hi[a:b] < s)).sum())
    assert outside == 0
    assert np.array_equal(got["plain"], got["batched"])
    assert 0 < got["plain"].sum() < len(got["plain"])
