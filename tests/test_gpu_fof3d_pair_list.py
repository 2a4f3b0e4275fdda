"""3D FoF with more pairs of dense cells than the pair list holds: clumps of nine particles two sub-cells
apart (81 pairs of particles a pair of cells), so that each has 26 clumps within the stencil. The labels
are right, and a pair of cells of thousands of particles among them is not left to one thread."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

LL = 0.3
CELL = 0.99 * LL / np.sqrt(3.0)


def _lattice(k):
    """Cell centres of every second cell of a box of 2 k cells an axis."""
    return (2.0 * np.stack(np.meshgrid(*[np.arange(k)] * 3, indexing="ij"), -1).reshape(-1, 3) + 0.5) * CELL


def _run(pos, L, ids, repeat=1):
    import torch
    import paper_2412_18629_gb300 as rs
    ctx = rs.Context(box=L, link_len=LL, softening=0.01, particle_mass=1.0)
    dev = [torch.from_numpy(a).cuda() for a in (pos, ids)]
    for _ in range(repeat):
        e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
        e[0].record()
        lab, ng = rs.rs_fof3d(ctx, *dev)
        e[1].record()
        torch.cuda.synchronize()
    ctx.close()
    return lab.cpu().numpy(), ng, e[0].elapsed_time(e[1])


@pytest.mark.parametrize("jitter", (0.0, 0.2))
def test_list_overflow_matches_the_oracle(jitter):
    rng = np.random.default_rng(37)
    k = 12
    centre = _lattice(k) + rng.uniform(-jitter, jitter, (k ** 3, 3)) * CELL
    size = np.full(k ** 3, 9)
    size[rng.choice(k ** 3, 6, replace=False)] = (1025, 1500, 40, 1024, 2100, 12)
    L = 2 * k * CELL * 0.9999
    pos = np.repeat(centre, size, axis=0) + rng.uniform(-0.05, 0.05, (size.sum(), 3)) * CELL
    pos = np.mod(pos, L).astype(np.float32)
    ids = rng.permutation(len(pos)).astype(np.int64)
    lab, ng, _ = _run(pos, L, ids)
    want = oracle.fof3d(pos, ids, np.float32(L), np.float32(LL))
    assert np.array_equal(lab, want) and ng == len(np.unique(want))


def test_large_cells_beside_a_full_list():
    rng = np.random.default_rng(38)
    k = 30
    centre = _lattice(k)
    size = np.full(k ** 3, 9)
    size[-2:] = 10000  # neighbours along z, the last rows of the stencil: the list is full by then
    L = 2 * k * CELL * 0.9999
    owner = np.repeat(np.arange(k ** 3), size)
    pos = (centre[owner] + rng.uniform(-0.02, 0.02, (len(owner), 3)) * CELL).astype(np.float32)
    ids = rng.permutation(len(pos)).astype(np.int64)
    least = np.full(k ** 3, len(pos))
    np.minimum.at(least, owner, ids)
    lab, ng, ms = _run(pos, L, ids, repeat=2)
    assert np.array_equal(lab, least[owner]) and ng == k ** 3
    assert ms < 250.0  # one thread over the 1e8 pairs of the two large cells takes seconds
