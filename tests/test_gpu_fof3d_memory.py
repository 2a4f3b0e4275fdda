"""Scratch memory of rs_fof3d: what it takes a particle decides how large a snapshot one GPU can hold."""
import pytest

pytestmark = pytest.mark.gpu


def test_memory_of_the_call():
    import torch
    import paper_2412_18629_gb300 as rs
    n, L = 1 << 24, 256.0
    g = torch.Generator(device="cuda").manual_seed(3)
    pos = torch.rand((n, 3), generator=g, device="cuda") * (L * 0.999)
    ids, lab = torch.arange(n, device="cuda"), torch.empty(n, dtype=torch.int64, device="cuda")
    ctx = rs.Context(box=L, link_len=0.28, softening=0.01, particle_mass=1.0)
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    rs.rs_fof3d(ctx, pos, ids, lab)
    used = free - torch.cuda.mem_get_info()[0]
    ctx.close()
    rows = (int(L / (0.99 * 0.28 / 3.0 ** 0.5)) + 1) ** 2
    # buffers are kept an eighth larger than asked for; 64 MB for modules and 2 MB pages
    assert used <= (56 * n + 4 * rows) * 9 // 8 + (64 << 20), used / n
