"""The warp form of the pairwise tree over chunk totals (rs_cro_sum) at the edges of its groups of 32,
32^2 and 32^3 chunks: bit for bit the oracle's level-by-level tree."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("chunks", (2, 3, 31, 32, 33, 63, 64, 65, 1023, 1024, 1025, 1056, 1057, 32768, 32801))
def test_groups_of_chunks(chunks):
    import torch
    import paper_2412_18629_gb300 as rs
    rng = np.random.default_rng(chunks)
    a = rng.normal(0, 1, 1024 * chunks - 5)
    a[:2048] *= np.exp(rng.uniform(-30, 30, len(a[:2048])))
    ctx = rs.Context(box=10.0, link_len=0.2, softening=0.01, particle_mass=1.0)
    got = rs.rs_cro_sum(ctx, torch.from_numpy(a).cuda()).item()
    ctx.close()
    assert got == oracle.cro_sum(a)
