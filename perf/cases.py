"""The workloads this library is timed on: what a halo-finding program asks of it, through its
Python entry points, from the smallest snapshot of the tests to the largest of the benchmark.

Snapshots follow the recipe of paper_2412_18629_gb300/synth.py (40% of the particles in NFW halos
drawn from dN/dn ~ n^-1.9, subhalos in halos above 1000 particles, uniform background, shuffled
order, permuted ids), drawn with torch on the GPU so that preparing a 2^27-particle snapshot takes
seconds instead of minutes.

Node and member counts differ from snapshot to snapshot, so a program keeps its results in buffers
of a fixed capacity (zero beyond the counts), as the states here do.

Kinds of case:
    pipeline   the four calls on one snapshot (3D FoF, 6D hierarchy, unbinding, properties)
    stream     rs_run_batched over independent snapshots on concurrent lanes
    fof3d      3D FoF labels alone
    unbind     unbinding with the potential as an output, and properties, of a kept hierarchy
    seeds      seed assignment of two snapshots of the same particles, and their tracking
    mlp        surrogate inference, or one batch's gradient
"""
import math

import numpy as np
import torch

import paper_2412_18629_gb300 as rs
from paper_2412_18629_gb300 import synth

DEV = "cuda:0"
MASS = 1.0e10
LINK_B = 0.28
SOFTENING = 0.01  # of the mean interparticle spacing


def listed():
    return [
        # The smallest snapshot of the tests and of the smoke run, in the plain form with the
        # potential as an output: every launch and every read-back counts.
        {"name": "pipeline-2^14-plain", "kind": "pipeline", "n": 1 << 14, "box": 25.0, "n_max": 2.0e3,
         "sub": 1, "mode": "plain", "potential": True, "gate": 0},
        # A small box of a test run or of one zoom region (L = 64 Mpc/h).
        {"name": "pipeline-2^18-batched", "kind": "pipeline", "n": 1 << 18, "box": 64.0, "n_max": 3.0e4,
         "sub": 0, "mode": "batched", "potential": False, "gate": 0},
        # An odd-sized snapshot of ordinary size with large halos in it.
        {"name": "pipeline-ragged-batched", "kind": "pipeline", "n": 1777777, "box": 121.1, "n_max": 2.0e5,
         "sub": 1, "mode": "batched", "potential": False, "gate": 0},
        # The batched + surrogate form on 2^25 particles in L = 320 Mpc/h, halos up to 5e5.
        {"name": "pipeline-2^25-surrogate", "kind": "pipeline", "n": 1 << 25, "box": 320.0, "n_max": 5.0e5,
         "sub": 1, "mode": "surrogate", "potential": False, "gate": 0},
        # The largest single-GPU snapshot: 2^27 particles in L = 512 Mpc/h, halos up to 2e6 with
        # three levels of subhalos.
        {"name": "pipeline-2^27-batched", "kind": "pipeline", "n": 1 << 27, "box": 512.0, "n_max": 2.0e6,
         "sub": 3, "mode": "batched", "potential": False, "gate": 0},
        # Many independent snapshots of 2^18 .. 2^22 particles on four lanes: a set of mocks.
        {"name": "stream-10x-4lanes", "kind": "stream", "snaps": 10, "log2_min": 18, "log2_max": 22,
         "n_max": 2.0e5, "sub": 1, "lanes": 4},
        # 3D FoF alone on 2^24 particles in L = 256 Mpc/h: group catalogues without substructure.
        {"name": "fof3d-2^24", "kind": "fof3d", "n": 1 << 24, "box": 256.0, "n_max": 3.0e4, "sub": 1,
         "sparse_ids": False, "check_ids": False},
        # Binding energies as a product: the direct float32 potential of every member.
        {"name": "unbind-potential-2^19", "kind": "unbind", "n": 1 << 19, "box": 80.6, "n_max": 2.0e5,
         "sub": 1, "mode": "batched", "passes": 1},
        # Seed halos of two outputs of a simulation, and their progenitors and descendants.
        {"name": "seeds-track-2^21", "kind": "seeds", "n": 1 << 21, "box": 128.0, "n_max": 3.0e4, "sub": 1},
        # Surrogate inference over the members of large halos.
        {"name": "mlp-forward-10^6", "kind": "mlp", "n": 1000000, "grad": False},
        # One batch of the surrogate's training: its gradient and squared error.
        {"name": "mlp-gradient-4096", "kind": "mlp", "n": 4096, "grad": True},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _box_of(n):
    """A box of about one particle per (Mpc/h)^3, as the benchmarked snapshots have."""
    return round(float(np.cbrt(float(n))), 3)


def draw(rng):
    kind = rng.choice(["pipeline", "pipeline", "pipeline", "stream", "fof3d", "fof3d", "unbind", "unbind",
                       "seeds", "mlp"])
    n_max = float(_log_int(rng, 2.0e3, 5.0e5))
    sub = rng.randrange(0, 4)
    if kind == "pipeline":
        mode = rng.choice(["plain", "batched", "batched", "surrogate"])
        n = _log_int(rng, 1 << 14, (1 << 19) if mode == "plain" else (1 << 25))
        return {"kind": kind, "n": n, "box": _box_of(n), "n_max": min(n_max, 5.0e4) if mode == "plain" else n_max,
                "sub": sub, "mode": mode, "potential": mode == "plain", "gate": rng.randrange(0, 2)}
    if kind == "stream":
        lo = rng.randrange(14, 20)
        return {"kind": kind, "snaps": rng.randrange(3, 13), "log2_min": lo, "log2_max": lo + rng.randrange(1, 4),
                "n_max": min(n_max, 2.0e5), "sub": sub, "lanes": rng.randrange(1, 7)}
    if kind == "fof3d":
        n = _log_int(rng, 1 << 12, 1 << 25)
        return {"kind": kind, "n": n, "box": _box_of(n), "n_max": n_max, "sub": sub,
                "sparse_ids": rng.random() < 0.3, "check_ids": rng.random() < 0.3}
    if kind == "unbind":
        n = _log_int(rng, 1 << 15, 1 << 21)
        return {"kind": kind, "n": n, "box": _box_of(n), "n_max": min(n_max, 2.0e5), "sub": sub,
                "mode": rng.choice(["plain", "batched"]), "passes": rng.choice([1, 1, 3])}
    if kind == "seeds":
        n = _log_int(rng, 1 << 15, 1 << 23)
        return {"kind": kind, "n": n, "box": _box_of(n), "n_max": min(n_max, 2.0e5), "sub": sub}
    grad = rng.random() < 0.5
    return {"kind": "mlp", "n": _log_int(rng, 256, 1 << 17) if grad else _log_int(rng, 1024, 1 << 24), "grad": grad}


# ---------------------------------------------------------------------------------------------
# Snapshots

def _plan(np_rng, n, box, n_max, sub_levels):
    """NFW halos and their subhalos: own particle counts, concentrations, virial radii, centres,
    bulk velocities, dispersions, and the top-level halo each belongs to."""
    rho_bar = n * MASS / box ** 3
    budget = int(0.4 * n)
    slope, n_min = 1.9, 20
    a = 1.0 - slope
    lo, hi = n_min ** a, n_max ** a
    sizes = np.zeros(0, np.int64)
    while sizes.sum() < budget:
        u = np_rng.random(max(64, budget // 200))
        s = np.clip(((lo + u * (hi - lo)) ** (1.0 / a)).astype(np.int64), n_min, int(n_max))
        sizes = np.concatenate([sizes, s])
    keep = int(np.searchsorted(np.cumsum(sizes), budget))
    sizes = sizes[:keep + 1]
    sizes[-1] -= int(sizes.sum()) - budget
    if sizes[-1] < n_min:
        sizes = sizes[:-1]
    rows = []

    def sub_of(count, centre, bulk, levels, top):
        r_vir = (3.0 * count * MASS / (4.0 * math.pi * 200.0 * rho_bar)) ** (1.0 / 3.0)
        sigma = math.sqrt(synth.G_NEWTON * count * MASS / r_vir) / math.sqrt(2.0)
        own = count
        if levels > 0 and count > 1000:
            for _ in range(int(np_rng.integers(0, 11))):
                s = int(count * np_rng.uniform(0.01, 0.10))
                if s < 20 or own - s < count // 2:
                    continue
                own -= s
                d = np_rng.normal(size=3)
                d *= np_rng.uniform(0.0, 0.8 * r_vir) / np.linalg.norm(d)
                sub_of(s, centre + d, bulk + np_rng.normal(0.0, sigma, 3), levels - 1, top)
        rows.append((own, count, r_vir, sigma, *centre, *bulk, top))

    centres = np_rng.uniform(0.0, box, (len(sizes), 3))
    small = sizes <= 1000 if sub_levels > 0 else np.ones(len(sizes), bool)
    for h in np.flatnonzero(~small):
        sub_of(int(sizes[h]), centres[h], np.zeros(3), sub_levels, int(h))
    big = np.array(rows, dtype=np.float64).reshape(-1, 11)
    c = sizes[small].astype(np.float64)
    r_vir = (3.0 * c * MASS / (4.0 * math.pi * 200.0 * rho_bar)) ** (1.0 / 3.0)
    sigma = np.sqrt(synth.G_NEWTON * c * MASS / r_vir) / math.sqrt(2.0)
    flat = np.column_stack([c, c, r_vir, sigma, centres[small], np.zeros((len(c), 3)), np.flatnonzero(small)])
    return np.concatenate([big, flat]), len(sizes)


def _snapshot(n, box, n_max, sub_levels, seed, sparse_ids=False):
    """pos, vel, ids on the GPU, the halo of each particle (-1: background), link length, softening."""
    np_rng = np.random.default_rng(seed)
    gen = torch.Generator(device=DEV)
    gen.manual_seed(int(seed))
    plan, _ = _plan(np_rng, n, box, min(n_max, 0.2 * n), sub_levels)
    own = torch.from_numpy(plan[:, 0].astype(np.int64)).to(DEV)
    P = torch.from_numpy(plan).to(DEV)
    row = torch.repeat_interleave(torch.arange(len(plan), device=DEV), own)
    m = row.numel()
    # radii: mu(x) = ln(1 + x) - x / (1 + x) inverted by interpolation on a logarithmic grid
    grid = np.logspace(-4.0, 2.0, 16384)
    mu = np.log1p(grid) - grid / (1.0 + grid)
    conc = 10.0 * (P[:, 1] / 1.0e4) ** -0.1
    mu_c = (torch.log1p(conc) - conc / (1.0 + conc))[row]
    gx, gm = torch.from_numpy(grid).to(DEV).log(), torch.from_numpy(mu).to(DEV)
    target = torch.rand(m, generator=gen, device=DEV, dtype=torch.float64).mul_(mu_c).clamp_(float(mu[0]), float(mu[-1]))
    k = torch.searchsorted(gm, target).clamp_(1, len(grid) - 1)
    t = (target - gm[k - 1]) / (gm[k] - gm[k - 1])
    r = torch.exp(gx[k - 1] + t * (gx[k] - gx[k - 1])) / conc[row] * P[:, 2][row]
    d = torch.randn((m, 3), generator=gen, device=DEV)
    d /= d.norm(dim=1, keepdim=True).clamp_min_(1e-12)
    pos64 = torch.empty((n, 3), dtype=torch.float64, device=DEV)
    pos64[:m] = P[:, 4:7][row] + d * r[:, None]
    vel = torch.empty((n, 3), device=DEV)
    vel[:m] = (P[:, 7:10][row] + torch.randn((m, 3), generator=gen, device=DEV) * P[:, 3][row][:, None]).float()
    pos64[m:] = torch.rand((n - m, 3), generator=gen, device=DEV, dtype=torch.float64) * box
    vel[m:] = 50.0 * torch.randn((n - m, 3), generator=gen, device=DEV)
    halo = torch.full((n,), -1, dtype=torch.int64, device=DEV)
    halo[:m] = P[:, 10].long()[row]
    del row, r, d, t, k, target, mu_c
    pos = torch.remainder(pos64, box).float()
    del pos64
    pos[pos >= float(np.float32(box))] = 0.0
    order = torch.randperm(n, generator=gen, device=DEV)
    ids = torch.randperm(n, generator=gen, device=DEV)
    if sparse_ids:  # unique ids spread over 2^40 instead of 0 .. n - 1
        ids = ids * ((1 << 40) // n) + 7
    spacing = box / float(np.cbrt(float(n)))
    return {"pos": pos[order].contiguous(), "vel": vel[order].contiguous(), "ids": ids, "halo": halo[order],
            "box": box, "link_length": float(np.float32(LINK_B * spacing)),
            "softening": float(np.float32(SOFTENING * spacing))}


def _context(s, **kw):
    return rs.Context(box=s["box"], link_len=s["link_length"], softening=s["softening"], particle_mass=MASS, **kw)


def _halo_labels(s):
    """Groups as a halo catalogue gives them: every top-level halo's smallest id, own id outside."""
    halo, ids = s["halo"], s["ids"]
    nh = int(halo.max().item()) + 1
    least = torch.full((nh,), torch.iinfo(torch.int64).max, dtype=torch.int64, device=DEV)
    inside = halo >= 0
    least.scatter_reduce_(0, halo[inside], ids[inside], "amin")
    return torch.where(inside, least[halo.clamp_min(0)], ids)


def _buffers(n):
    """Result buffers of one snapshot of n particles: room for n // 20 nodes and 2 n members."""
    nodes, members = max(256, n // 20), 2 * n

    def zeros(*shape, dtype=torch.int64):
        return torch.zeros(shape, dtype=dtype, device=DEV)

    return {"parent": zeros(nodes), "level": zeros(nodes, dtype=torch.int32), "min_id": zeros(nodes),
            "size": zeros(nodes), "member_off": zeros(nodes + 1), "member_idx": zeros(members),
            "bound": zeros(members, dtype=torch.uint8), "props": zeros(nodes, 160, dtype=torch.uint8)}


def _keep(buffers, results):
    for k, v in results.items():
        buffers[k][:v.shape[0]].copy_(v)


def _train(ctx, seed):
    """A surrogate trained on the exact potentials of a 2^19-particle snapshot."""
    s = _snapshot(1 << 19, 80.6, 3.0e4, 1, 1000003 + seed)
    ex = _context(s, mode="batched")
    labels, _ = rs.rs_fof3d(ex, s["pos"], s["ids"])
    rs.rs_fof6d(ex, s["pos"], s["vel"], s["ids"], labels)
    rs.rs_unbind(ex, s["pos"], s["vel"], want_potential=True)
    feat, psi = rs.rs_surrogate_features(ex)
    keep = torch.arange(0, feat.shape[0], max(1, feat.shape[0] // 50000), device=DEV)
    rs.rs_mlp_train(ctx, feat[keep].contiguous(), psi[keep].contiguous(), epochs=20, batch=2048, seed=seed)
    torch.cuda.synchronize()
    ex.close()


# ---------------------------------------------------------------------------------------------
# Surrogate network (8 -> 64 -> 64 -> 1): parameters and samples of the features' ranges

def _mlp_data(case, seed):
    np_rng = np.random.default_rng(seed)
    w = np.zeros(rs.MLP_PARAMS, np.float32)
    w[:512] = np_rng.uniform(-1, 1, 512) * math.sqrt(6.0 / 8.0)
    w[512:576] = np_rng.normal(0, 0.05, 64)
    w[576:4672] = np_rng.uniform(-1, 1, 4096) * math.sqrt(6.0 / 64.0)
    w[4672:4736] = np_rng.normal(0, 0.05, 64)
    w[4736:4800] = np_rng.uniform(-1, 1, 64) * math.sqrt(6.0 / 64.0)
    w[4800] = -1.0
    gen = torch.Generator(device=DEV)
    gen.manual_seed(int(seed))
    n = case["n"]
    frac = torch.sort(torch.rand((n, 4), generator=gen, device=DEV), dim=1).values
    x = torch.empty((n, 8), device=DEV)
    x[:, 0] = 1.5 * torch.rand(n, generator=gen, device=DEV) ** 2
    x[:, 1:5] = frac
    x[:, 5] = torch.randn((n, 3), generator=gen, device=DEV).norm(dim=1)
    x[:, 6] = 3.0 + 3.0 * torch.rand(n, generator=gen, device=DEV)
    x[:, 7] = -0.5 - 3.0 * torch.rand(n, generator=gen, device=DEV)
    t = x[:, 7] + 0.1 * torch.randn(n, generator=gen, device=DEV)
    return w, x, t


# ---------------------------------------------------------------------------------------------

def prepare(case, seed):
    kind = case["kind"]
    if kind == "pipeline":
        s = _snapshot(case["n"], case["box"], case["n_max"], case["sub"], seed)
        ctx = _context(s, mode=case["mode"], surrogate_gate=case["gate"])
        if case["mode"] == "surrogate":
            _train(ctx, seed)
        buffers = _buffers(case["n"])
        if case["potential"]:
            buffers["phi"] = torch.zeros(2 * case["n"], device=DEV)
        return {"case": case, "s": s, "ctx": ctx, "buffers": buffers}
    if kind == "stream":
        span = case["log2_max"] - case["log2_min"] + 1
        snaps = []
        for k in range(case["snaps"]):
            n = 1 << (case["log2_min"] + k % span)
            snaps.append(_snapshot(n, float(np.cbrt(float(n))), case["n_max"], case["sub"], 1000 * seed + k))
        ctx = _context(snaps[0], mode="batched")
        sizes = [s["ids"].numel() for s in snaps]
        out = rs.BatchOutputs(sizes, [max(256, n // 20) for n in sizes], 0)
        for t in out.parent + out.props:
            t.zero_()
        return {"case": case, "snaps": snaps, "ctx": ctx, "out": out}
    if kind == "fof3d":
        s = _snapshot(case["n"], case["box"], case["n_max"], case["sub"], seed, case["sparse_ids"])
        return {"case": case, "s": s, "ctx": _context(s, mode="batched", check_ids=case["check_ids"])}
    if kind == "unbind":
        s = _snapshot(case["n"], case["box"], case["n_max"], case["sub"], seed)
        ctx = _context(s, mode=case["mode"], unbind_passes=case["passes"])
        rs.rs_fof6d(ctx, s["pos"], s["vel"], s["ids"], _halo_labels(s))
        b = _buffers(case["n"])
        return {"case": case, "s": s, "ctx": ctx, "phi": torch.zeros(2 * case["n"], device=DEV),
                "bound": b["bound"], "props": b["props"]}
    if kind == "seeds":
        s = _snapshot(case["n"], case["box"], case["n_max"], case["sub"], seed)
        gen = torch.Generator(device=DEV)
        gen.manual_seed(int(seed) + 1)
        order = torch.randperm(case["n"], generator=gen, device=DEV)
        drift = (s["pos"].double() + s["vel"].double() * (synth.MPC_PER_GYR_PER_KMS * 1.0e-5)) % s["box"]
        pos = drift.float()
        pos[pos >= float(np.float32(s["box"]))] = 0.0
        kick = 5.0 * torch.randn(s["vel"].shape, generator=gen, device=DEV)
        later = dict(s, pos=pos[order].contiguous(), vel=(s["vel"] + kick)[order].contiguous(), ids=s["ids"][order])
        both = []
        for snap in (s, later):
            ctx = _context(snap, mode="batched")
            labels, _ = rs.rs_fof3d(ctx, snap["pos"], snap["ids"])
            rs.rs_fof6d(ctx, snap["pos"], snap["vel"], snap["ids"], labels)
            both.append((ctx, snap))
        tables = [torch.zeros(max(256, case["n"] // 20), dtype=torch.int64, device=DEV) for _ in range(8)]
        return {"case": case, "both": both, "tables": tables}
    w, x, t = _mlp_data(case, seed)
    ctx = rs.Context(box=64.0, link_len=0.28, softening=0.01, particle_mass=MASS, mode="batched")
    rs.rs_mlp_set_params(ctx, w)
    return {"case": case, "ctx": ctx, "x": x, "t": t}


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "pipeline":
        s, ctx = state["s"], state["ctx"]
        buf = state["buffers"]
        labels, n_groups = rs.rs_fof3d(ctx, s["pos"], s["ids"])
        rs.rs_fof6d(ctx, s["pos"], s["vel"], s["ids"], labels)
        phi, _, _ = rs.rs_unbind(ctx, s["pos"], s["vel"], want_potential=case["potential"], bound_out=buf["bound"])
        rs.rs_halo_props(ctx, props_out=buf["props"])
        hierarchy = rs.rs_fof6d_copy(ctx)
        deepest = hierarchy.pop("deepest")
        _keep(buf, hierarchy)
        if phi is not None:
            _keep(buf, {"phi": phi})
        return dict(buf, labels=labels, n_groups=n_groups, deepest=deepest, n_nodes=ctx.n_nodes,
                    n_members=ctx.n_members)
    if kind == "stream":
        out = state["out"]
        counts = rs.rs_run_batched(state["ctx"], state["snaps"], out, lanes=case["lanes"])
        return {"counts": counts, "labels": out.labels, "deepest": out.deepest, "parent": out.parent,
                "props": out.props}
    if kind == "fof3d":
        labels, n_groups = rs.rs_fof3d(state["ctx"], state["s"]["pos"], state["s"]["ids"])
        return {"labels": labels, "n_groups": n_groups}
    if kind == "unbind":
        s, ctx = state["s"], state["ctx"]
        phi, _, _ = rs.rs_unbind(ctx, s["pos"], s["vel"], want_potential=True, bound_out=state["bound"])
        rs.rs_halo_props(ctx, props_out=state["props"])
        _keep(state, {"phi": phi})
        return {"phi": state["phi"], "bound": state["bound"], "props": state["props"]}
    if kind == "seeds":
        found = [rs.rs_assign_seeds(ctx, s["pos"], s["vel"]) for ctx, s in state["both"]]
        (c1, s1), (c2, s2) = state["both"]
        track = rs.rs_track(c2, s1["ids"], found[0][0], c1.n_nodes, s2["ids"], found[1][0], c2.n_nodes)
        for table, t in zip(state["tables"], [*found[0][1:3], *found[1][1:3], *track]):
            table[:t.shape[0]].copy_(t)
        return {"seed": [f[0] for f in found], "n_seeds": [f[3] for f in found], "tables": state["tables"]}
    if case["grad"]:
        grad, sse = rs.rs_mlp_gradient(state["ctx"], state["x"], state["t"])
        return {"grad": grad, "sse": sse}
    return rs.rs_mlp_forward(state["ctx"], state["x"])


# ---------------------------------------------------------------------------------------------

def _pairs(n, n_max):
    """Expected sum of g^2 over the halos: 40% of the particles, dN/dn ~ n^-1.9 on [20, n_max]."""
    hi = min(n_max, 0.2 * n)
    return 0.4 * n * ((hi ** 1.1 - 20 ** 1.1) / 1.1) / ((hi ** 0.1 - 20 ** 0.1) / 0.1)


def work(case):
    """Bytes: inputs once and outputs once (about 0.9 hierarchy members and 0.005 nodes per particle
    in these snapshots). Flops: the direct potential (11 per ordered pair) where it is an output,
    the network's multiply-adds, otherwise the 6D distances of each member's neighbours (about 20
    operations to about 30 members that no search can leave out) and of its far field."""
    kind = case["kind"]
    if kind == "mlp":
        per = 2 * (8 * 64 + 64 * 64 + 64)
        if case["grad"]:
            return {"bytes": case["n"] * 36 + 2 * 4 * rs.MLP_PARAMS, "flops": 3 * per * case["n"]}
        return {"bytes": case["n"] * 36 + 4 * rs.MLP_PARAMS, "flops": per * case["n"]}
    if kind == "stream":
        span = case["log2_max"] - case["log2_min"] + 1
        n = sum(1 << (case["log2_min"] + k % span) for k in range(case["snaps"]))
        return {"bytes": int(n * (32 + 16 + 0.005 * 168)), "flops": 0.9 * n * 1200}
    n = case["n"]
    if kind == "fof3d":
        return {"bytes": n * 28, "flops": n * 80}
    if kind == "seeds":
        return {"bytes": 2 * n * (24 + 8 + 8 + 8), "flops": 2 * n * 20}
    if kind == "unbind":
        return {"bytes": int(0.5 * n * (24 + 5) + 0.005 * n * 160), "flops": 11 * _pairs(n, case["n_max"])}
    members = 0.9 * n
    flops = members * 1200 + (11 * _pairs(n, case["n_max"]) if case["potential"] else 0)
    return {"bytes": int(n * (32 + 16) + members * 9 + 0.005 * n * 200), "flops": flops}


# ---------------------------------------------------------------------------------------------
# 64-bit values

def _exact_mlp(case, seed):
    w, x, t = _mlp_data(case, seed)

    def bf(a):
        return a.to(torch.bfloat16).double()

    W = torch.from_numpy(w).to(DEV)
    W1, b1 = bf(W[:512].reshape(8, 64)), W[512:576].double()
    W2, b2 = bf(W[576:4672].reshape(64, 64)), W[4672:4736].double()
    W3, b3 = bf(W[4736:4800]), W[4800].double()
    ys, grad, sse = [], None, 0.0
    for lo in range(0, case["n"], 1 << 20):
        xb = bf(x[lo:lo + (1 << 20)])
        h1 = bf((xb @ W1 + b1).float().relu())
        h2 = bf((h1 @ W2 + b2).float().relu())
        y = h2 @ W3 + b3
        ys.append(y)
        if case["grad"]:
            e = y - t[lo:lo + (1 << 20)].double()
            dy = 2.0 * e / case["n"]
            d2 = bf(torch.where(h2 > 0, dy[:, None] * W3, torch.zeros_like(h2)).float())
            d1 = bf(torch.where(h1 > 0, d2 @ W2.T, torch.zeros_like(h1)).float())
            part = torch.cat([(xb.T @ d1).reshape(-1), d1.sum(0), (h1.T @ d2).reshape(-1), d2.sum(0),
                              (dy[:, None] * h2).sum(0), dy.sum().reshape(1)])
            grad = part if grad is None else grad + part
            sse += float((e * e).sum())
    return {"grad": grad, "sse": sse} if case["grad"] else torch.cat(ys)


def _components(g, a, b):
    """Smallest member index of every member's component under the links a - b."""
    lab = torch.arange(g, device=DEV)
    while True:
        low = torch.minimum(lab[a], lab[b])
        new = lab.scatter_reduce(0, a, low, "amin").scatter_reduce(0, b, low, "amin")
        new = new[new]
        if torch.equal(new, lab):
            return lab
        lab = new


def _split(u, v):
    """The children of one node as member index tensors, by the definition of the 6D links."""
    g = u.shape[0]
    inv = []
    for c in (u, v):
        c = c.double()
        mean = c.sum(0) / g
        var = ((c * c).sum(0) / g - mean * mean).sum()
        inv.append((1.0 / var).float() if float(var) > 0 else torch.zeros((), device=DEV))
    step = max(1, (1 << 27) // g)
    idx = torch.arange(g, device=DEV)

    def d6(lo, hi):
        out = []
        for c, s in ((u, inv[0]), (v, inv[1])):
            d = [c[None, :, k] - c[lo:hi, None, k] for k in range(3)]
            out.append(((d[0] * d[0] + d[1] * d[1]) + d[2] * d[2]) * s)
        return out[0] + out[1]

    nn2 = torch.empty(g, device=DEV)
    for lo in range(0, g, step):
        hi = min(g, lo + step)
        d = d6(lo, hi)
        d[idx[: hi - lo], idx[lo:hi]] = math.inf
        nn2[lo:hi] = d.min(1).values
    l2 = torch.sort(nn2).values[(7 * g + 9) // 10 - 1]
    a, b = [], []
    for lo in range(0, g, step):
        hi = min(g, lo + step)
        i, j = torch.nonzero(d6(lo, hi) <= l2, as_tuple=True)
        keep = j > i + lo
        a.append(i[keep] + lo)
        b.append(j[keep])
    lab = _components(g, torch.cat(a), torch.cat(b))
    count = torch.bincount(lab, minlength=g)
    roots = torch.nonzero((count >= 10) & (count < g)).flatten()
    return [torch.nonzero(lab == r).flatten() for r in roots.tolist()]


def _exact_unbind(case, seed):
    """Potentials of every (node, member) in 64 bits: the hierarchy by all pairs of every node."""
    s = _snapshot(case["n"], case["box"], case["n_max"], case["sub"], seed)
    pos, vel, ids, labels = s["pos"], s["vel"], s["ids"], _halo_labels(s)
    L = float(np.float32(case["box"]))
    eps2 = float(np.float32(s["softening"])) ** 2
    kept = torch.nonzero(s["halo"] >= 0).flatten()
    kept = kept[torch.argsort(ids[kept])]
    kept = kept[torch.argsort(labels[kept], stable=True)]
    _, sizes = torch.unique_consecutive(labels[kept], return_counts=True)
    level = [m for m in torch.split(kept, sizes.tolist()) if m.numel() >= 10]
    phi = []
    while level:
        below = []
        for mem in level:
            p = pos[mem]
            u = p - p[0]
            u = torch.where(u > 0.5 * L, u - L, torch.where(u < -0.5 * L, u + L, u))
            g = u.shape[0]
            ud = u.double()
            S = torch.empty(g, dtype=torch.float64, device=DEV)
            step = max(1, (1 << 26) // g)
            for lo in range(0, g, step):
                hi = min(g, lo + step)
                r2 = torch.full((hi - lo, g), eps2, dtype=torch.float64, device=DEV)
                for k in range(3):
                    d = ud[None, :, k] - ud[lo:hi, None, k]
                    r2 += d * d
                w = r2.rsqrt_()
                w[torch.arange(hi - lo, device=DEV), torch.arange(lo, hi, device=DEV)] = 0.0
                S[lo:hi] = w.sum(1)
            phi.append(-(synth.G_NEWTON * MASS) * S)
            below += [mem[c] for c in _split(u, vel[mem])]
        level = below
    phi = torch.cat(phi)
    kept = torch.zeros(2 * case["n"], dtype=torch.float64, device=DEV)
    kept[:phi.shape[0]] = phi
    return {"phi": kept, "bound": None, "props": None}


def exact(case, seed):
    if case["kind"] == "mlp":
        return _exact_mlp(case, seed)
    if case["kind"] == "unbind" and case["passes"] == 1 and case["n"] <= 1 << 19:
        return _exact_unbind(case, seed)
    return None  # whole numbers and bytes, or potentials of a hierarchy that takes minutes by all pairs
