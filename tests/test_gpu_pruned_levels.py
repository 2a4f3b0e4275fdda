"""The batched form's pruned 6D searches on every level of small snapshots (levels of few pairs take the
all-pairs kernels unless a smallest node of the bounded searches is set): the hierarchy and the split
parameters equal the oracle's, and the tallies show that the searches ran."""
import numpy as np
import pytest

import oracle
from helpers import assert_hier_equal, gpu_ctx, small_snapshot, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("min_members", (2, 64))
@pytest.mark.parametrize("n,box,seed,n_max,sub", [(1 << 14, 25.0, 24, 3000, 1), (1 << 16, 40.0, 25, 5000, 2),
                                                  (1 << 17, 50.0, 26, 20000, 2)])
def test_pruned_searches_on_every_level(n, box, seed, n_max, sub, min_members):
    import paper_2412_18629_gb300 as rs
    s = small_snapshot(n, box, seed, n_max=n_max, sub_levels=sub)
    ctx = gpu_ctx(s, mode="batched")
    ctx.nn_bounds(1.0, min_members)
    pos, vel, ids = to_dev(s)
    lab, _ = rs.rs_fof3d(ctx, pos, ids)
    ctx.profile(True)
    ctx.count_work(True)
    rs.rs_fof6d(ctx, pos, vel, ids, lab)
    work, ran = ctx.count_work(False), ctx.profile_totals()
    got = {k: v.cpu().numpy() for k, v in rs.rs_fof6d_copy(ctx).items()}
    params = rs.rs_fof6d_node_params(ctx).cpu().numpy()[:, :3]
    ctx.close()
    want = oracle.hierarchy(s["pos"], s["vel"], s["ids"], lab.cpu().numpy(), s["box"])
    assert_hier_equal(got, want)
    assert np.array_equal(params, want["params"])
    assert work["nn_d6"] > 0 and work["link_d6"] > 0 and work["bounded_nodes"] > 0
    levels = int(want["level"].max()) + 1
    deep = sum(int((want["size"][want["level"] == k].max() >= min_members)) for k in range(levels))
    # near and far searches of neighbours and links a level
    assert ran["k_nn6d_pruned"][1] >= 2 * deep and ran["k_link6d_pruned"][1] == 2 * deep
    assert ("k_nn6d" in ran) == (deep < levels)
