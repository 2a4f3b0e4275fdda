"""Matching of particles between snapshots by a table (ids of a dense range) and by a sort (any other),
on both sides of the line between them and for node counts around whole digits of the sort."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


def _ids(kind, n, rng):
    ids = rng.permutation(n).astype(np.int64)
    top = {"dense": n - 1, "table": 2 * n + 4095, "sort": 2 * n + 4096, "wide": (1 << 62) + 5}[kind]
    ids[ids == n - 1] = top  # the largest id decides
    return ids


@pytest.mark.parametrize("kind", ["dense", "table", "sort", "wide"])
@pytest.mark.parametrize("n,nodes1,nodes2", [(1, 1, 1), (300, 255, 256), (5000, 257, 16), (40000, 3, 70000)])
def test_track_by_table_and_by_sort(kind, n, nodes1, nodes2):
    import torch
    import paper_2412_18629_gb300 as rs
    rng = np.random.default_rng(n + nodes1)
    ids1 = _ids(kind, n, rng)
    seed1 = rng.integers(-1, nodes1, n).astype(np.int64)
    keep = rng.permutation(n)[: max(1, n - n // 4)]  # some particles are gone, some ids are new
    ids2 = np.concatenate([ids1[keep], np.arange(n // 8, dtype=np.int64) + (1 << 61)])
    seed2 = rng.integers(-1, nodes2, len(ids2)).astype(np.int64)
    ctx = rs.Context(box=10.0, link_len=0.2, softening=0.01, particle_mass=1.0)
    dev = [torch.from_numpy(a).cuda() for a in (ids1, seed1, ids2, seed2)]
    got = rs.rs_track(ctx, dev[0], dev[1], nodes1, dev[2], dev[3], nodes2)
    want = oracle.track(ids1, seed1, nodes1, ids2, seed2, nodes2)
    for g, w in zip(got, want):
        assert np.array_equal(g.cpu().numpy(), np.asarray(w))
