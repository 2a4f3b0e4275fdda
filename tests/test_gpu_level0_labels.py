"""Level 0 of the hierarchy from labels of a dense and of a sparse range: group sizes, members in
ascending id and the particles of no kept group, at the edges of the counting and key blocks (2048
particles each), with one label for most particles and with more labels than a block's table holds."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
MIN = 10


@pytest.mark.parametrize("sparse", [False, True])
@pytest.mark.parametrize("n,n_labels,skew", [(1, 1, 0.0), (2047, 3, 0.9), (2048, 2048, 0.0), (2049, 100, 0.5),
                                             (70001, 6000, 0.05), (70001, 20, 0.0)])
def test_level0_of_labels(n, n_labels, skew, sparse):
    import torch
    import paper_2412_18629_gb300 as rs
    rng = np.random.default_rng(n + n_labels)
    lab = rng.integers(0, n_labels, n)
    lab[rng.random(n) < skew] = n_labels // 2
    lab = lab.astype(np.int64) * ((1 << 40) if sparse else 1)
    ids = rng.permutation(n).astype(np.int64)
    pos = (rng.random((n, 3)) * 10.0).astype(np.float32)
    vel = rng.normal(size=(n, 3)).astype(np.float32)
    ctx = rs.Context(box=10.0, link_len=0.2, softening=0.01, particle_mass=1.0)
    rs.rs_fof6d(ctx, *(torch.from_numpy(a).cuda() for a in (pos, vel, ids, lab)))
    got = {k: v.cpu().numpy() for k, v in rs.rs_fof6d_copy(ctx).items()}
    values, counts = np.unique(lab, return_counts=True)
    kept = values[counts >= MIN]
    top = got["level"] == 0
    assert np.array_equal(got["size"][top], counts[counts >= MIN])
    order = np.argsort(ids)  # particles by ascending id
    off = got["member_off"]
    for q, v in enumerate(kept):
        want = order[lab[order] == v]
        assert np.array_equal(got["member_idx"][off[q]:off[q + 1]], want)
        assert got["min_id"][q] == ids[want[0]]
    assert np.array_equal(got["deepest"] >= 0, np.isin(lab, kept))
    ctx.close()
