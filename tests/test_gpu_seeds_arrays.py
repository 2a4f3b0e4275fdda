"""rs_assign_seeds works on the contents of the arrays it is given: the same result for later positions
and velocities in new arrays and in the arrays of rs_fof6d, equal to the oracle's, and the hierarchy's own
data (that the properties are made from) stays as it was."""
import numpy as np
import pytest

import oracle
from helpers import gpu_ctx, small_snapshot, to_dev

pytestmark = pytest.mark.gpu


def test_seeds_of_changed_positions():
    import torch
    import paper_2412_18629_gb300 as rs
    s = small_snapshot(1 << 15, 32.0, 75, n_max=5000)
    rng = np.random.default_rng(5)
    L = np.float32(s["box"])
    pos2 = np.mod(s["pos"] + rng.normal(0.0, 0.05, s["pos"].shape).astype(np.float32), L)
    pos2[pos2 >= L] = 0.0
    vel2 = (s["vel"] + rng.normal(0.0, 100.0, s["vel"].shape)).astype(np.float32)
    new = [torch.from_numpy(a).cuda() for a in (pos2, vel2)]
    got = {}
    for where in ("new arrays", "in place"):
        ctx = gpu_ctx(s, mode="batched")
        pos, vel, ids = to_dev(s)
        lab, _ = rs.rs_fof3d(ctx, pos, ids)
        rs.rs_fof6d(ctx, pos, vel, ids, lab)
        hier = {k: v.cpu().numpy() for k, v in rs.rs_fof6d_copy(ctx).items()}
        hier["params"] = rs.rs_fof6d_node_params(ctx).cpu().numpy()[:, :3]
        rs.rs_unbind(ctx, pos, vel)
        props = rs.rs_halo_props(ctx).cpu().numpy()
        if where == "in place":
            pos.copy_(new[0])
            vel.copy_(new[1])
        a = (pos, vel) if where == "in place" else new
        got[where] = [t.cpu().numpy() for t in rs.rs_assign_seeds(ctx, *a)[:3]]
        assert np.array_equal(rs.rs_halo_props(ctx).cpu().numpy(), props), where
        ctx.close()
    want = oracle.assign_seeds(hier, pos2, vel2, s["box"])
    for where, g in got.items():
        for a, w in zip(g, want):
            assert np.array_equal(a, w), where
    assert not np.array_equal(want[0], oracle.assign_seeds(hier, s["pos"], s["vel"], s["box"])[0])
