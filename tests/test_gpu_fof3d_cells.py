"""3D FoF on dense sub-cells: pairs of cells whose particles are linked by none, one or all of millions
of pairs (sampled, listed in chunks of 1024 particles and tested by a block), across the periodic
boundary, in boxes of a few cells (every pair of cells) and of many, against the oracle's labels."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


def _clumps(rng, ll, sizes, gaps, start, L):
    """Tight clumps along x, the facing sides of neighbours `gaps` link lengths apart."""
    x, parts = start, []
    for g, gap in zip(sizes, [*gaps, 0.0]):
        p = rng.uniform(0.0, 0.2 * ll, (g, 3))
        p[:, 0] += x
        p[:, 1:] += 0.4 * L
        parts.append(p)
        x = p[:, 0].max() + gap * ll
    return np.concatenate(parts)


@pytest.mark.parametrize("cells", (3, 5, 6, 7, 8, 9, 40))
@pytest.mark.parametrize("sizes", ((1, 1, 1), (8, 8, 8), (9, 8, 3), (1500, 40, 1025), (3000, 2500, 7)))
@pytest.mark.parametrize("gaps", ((0.9, 0.9), (1.001, 0.9), (0.97, 1.02), (1.0005, 1.0005)))
def test_clumps_match_the_oracle(cells, sizes, gaps):
    import torch
    import paper_2412_18629_gb300 as rs
    rng = np.random.default_rng(cells * 1000 + sum(sizes))
    ll = 0.3
    L = cells * 0.99 * ll / np.sqrt(3.0)
    pos = _clumps(rng, ll, sizes, gaps, 0.6 * L, L)  # runs through the boundary in small boxes
    pos = np.concatenate([pos, rng.uniform(0.0, L, (3 * cells, 3))])
    pos = np.mod(pos, L).astype(np.float32)
    pos[pos >= np.float32(L)] = 0.0
    ids = rng.permutation(len(pos)).astype(np.int64)
    ctx = rs.Context(box=L, link_len=ll, softening=0.01, particle_mass=1.0)
    lab, ng = rs.rs_fof3d(ctx, torch.from_numpy(pos).cuda(), torch.from_numpy(ids).cuda())
    lab = lab.cpu().numpy()
    ctx.close()
    want = oracle.fof3d(pos, ids, np.float32(L), np.float32(ll))
    assert np.array_equal(lab, want)
    assert ng == len(np.unique(want))
