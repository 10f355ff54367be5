"""The docking library's work as its users have it done, for measurement.

Each case is one call (or one call and its backward) of the public Python
binding on inputs that lie on the GPU: docking searches from a handful of
ligands to a screening batch, with the options that change the work (record
format, FP64 re-score, bucketed layout, several sites, exhaustive search),
scoring, differentiation and refinement of given poses, and the packer.

Inputs are drawn on the GPU from the seed: random molecular trees (1.5 A
bonds at 109.5 degrees, non-bonded atoms at least 1.2 A apart where four
tries allow it, rotatable bonds among the edges whose two ends have another
neighbour), a pocket grid (Gaussian wells of pseudo-atoms on a 7-11 A shell,
+5 within 2.5 A of one), poses about the pocket's centre. The size recipes are
those of the repository's named workloads.
"""
import math

import torch

import paper_2303_06150_gb300 as lg

# Ligand size recipes.
#   small: 12-24 atoms, 1-3 rotatable bonds
#   screen: round(N(38, 14)) atoms in [8, 100], Poisson(6) bonds in [0, 24]
#   bimodal: 70% 15-35 atoms with 0-8 bonds, 30% 60-120 atoms with 8-30 bonds
#   rigidish: 8-20 atoms, 0-3 bonds (what an exhaustive search can take)
RECIPES = ("small", "screen", "bimodal", "rigidish")
# Expected atoms, rotatable bonds and moving atoms of a bond, per ligand (for work()).
MEANS = {"small": (18.0, 2.0, 3.5), "screen": (38.0, 6.0, 7.0), "bimodal": (44.5, 8.5, 9.0), "rigidish": (14.0, 1.5, 3.0)}

# Grids of the named workloads: points per axis, channels, spacing (A), pseudo-atoms.
GRIDS = {"g40": (40, 4, 0.5, 150), "g96": (96, 8, 0.375, 600)}

# The production search and the quick one of the named workloads.
SCREEN = dict(restarts=256, step=10, passes=3, top_k=30)
QUICK = dict(restarts=8, step=30, passes=2, top_k=4)


def _dock(name, recipe, ligands, grid="g96", fmt="f32", batching="plain", rescore=False, mode="greedy", sites=1,
          search=SCREEN):
    return dict(name=name, call="dock", recipe=recipe, ligands=ligands, grid=grid, fmt=fmt, batching=batching,
                rescore=rescore, mode=mode, sites=sites, **search)


def listed():
    return [
        # a service's smallest request: a few dozen small ligands, quick search; launches and host time count
        _dock("dock_quick", "small", 32, grid="g40", search=QUICK),
        # a chemist re-docks a handful of analogues with the production search: too few ligands to fill the chip
        _dock("dock_series", "screen", 5),
        # the screening batch: the main use
        _dock("dock_screen", "screen", 20000),
        # a screening batch on 16-bit records whose kept poses are re-scored and re-ranked in FP64
        _dock("dock_rescore_f16", "screen", 6000, fmt="f16", rescore=True),
        # a mixed library of small and large ligands in the bucketed layout
        _dock("dock_bimodal_buckets", "bimodal", 5000, fmt="f16", batching="buckets_static"),
        # a small library against the twelve sites of one target
        _dock("dock_sites", "screen", 301, sites=12),
        # exhaustive search of small ligands (the reference answer for the greedy search)
        _dock("dock_exhaustive", "rigidish", 97, grid="g40", mode="exhaustive", search=QUICK),
        # a refinement loop or re-scoring service: many poses of one library on inputs prepared once
        dict(name="score_prepared", call="score_prepared", recipe="screen", ligands=20000, grid="g96", poses=30),
        # a docked library's few best poses scored against another grid, once
        dict(name="score_few", call="score", recipe="screen", ligands=5001, grid="g96", poses=3),
        # a differentiable objective: scores and their backward
        dict(name="score_backward", call="grad", recipe="screen", ligands=1500, grid="g96", poses=16),
        # gradient refinement of a docked batch's best poses
        dict(name="refine", call="refine", recipe="screen", ligands=4000, grid="g96", poses=16, steps=50),
        # a library classified and packed (bucket planning, inspection)
        dict(name="pack", call="pack", recipe="bimodal", ligands=50000, grid="g96"),
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    call = rng.choice(["dock", "dock", "dock", "sites", "exhaustive", "score_prepared", "score", "grad", "refine",
                       "pack"])
    grid = "g96"
    if call == "dock":
        kind = rng.choice(["screen", "screen", "bimodal", "small"])
        if kind == "small":
            s = dict(restarts=rng.randint(1, 40), step=rng.choice([15, 20, 30, 45]), passes=rng.randint(1, 3))
            s["top_k"] = rng.randint(1, s["restarts"])
            return _named_off(_dock("", "small", _log_int(rng, 1, 3000), grid="g40", fmt=rng.choice(["f32", "f16"]),
                                    search=s))
        s = dict(restarts=rng.choice([64, 100, 128, 256]), step=rng.choice([10, 10, 12, 15]), passes=rng.randint(1, 3),
                 top_k=rng.randint(1, 30))
        return _named_off(_dock("", kind, _log_int(rng, 1, 9000 if kind == "screen" else 4000), grid=grid,
                                fmt=rng.choice(["f32", "f32", "f16", "bf16"]),
                                batching=rng.choice(["plain", "plain", "buckets", "buckets_static", "queue"]),
                                rescore=rng.random() < 0.3, search=s))
    if call == "sites":
        s = dict(SCREEN, restarts=rng.choice([64, 256]))
        return _named_off(_dock("", "screen", _log_int(rng, 1, 500), grid=grid, fmt=rng.choice(["f32", "f16"]),
                                sites=rng.randint(2, 12), search=s))
    if call == "exhaustive":
        s = dict(restarts=rng.randint(1, 16), step=rng.choice([30, 40, 45, 60]), passes=1)
        s["top_k"] = rng.randint(1, s["restarts"])
        return _named_off(_dock("", "rigidish", _log_int(rng, 1, 120), grid="g40", mode="exhaustive", search=s))
    recipe = rng.choice(["screen", "bimodal"])
    c = dict(call=call, recipe=recipe, ligands=_log_int(rng, 1, 12000 if recipe == "screen" else 6000), grid=grid)
    if call == "pack":
        c["ligands"] = _log_int(rng, 1, 60000)
    elif call == "refine":
        c.update(ligands=_log_int(rng, 1, 4000 if recipe == "screen" else 1200), poses=rng.randint(1, 16),
                 steps=rng.randint(5, 50))
    else:
        c["poses"] = rng.randint(1, 40 if call != "grad" else 20)
    return c


def _named_off(case):
    case.pop("name")
    return case


# ------------------------------------------------------------------ inputs --

def _uniform(g, shape, lo=0.0, hi=1.0):
    return torch.rand(shape, generator=g, device="cuda") * (hi - lo) + lo


def _sizes(g, recipe, L):
    def ints(lo, hi):
        return torch.randint(lo, hi + 1, (L,), generator=g, device="cuda")

    if recipe == "small":
        return ints(12, 24), ints(1, 3)
    if recipe == "rigidish":
        return ints(8, 20), ints(0, 3)
    if recipe == "screen":
        atoms = torch.randn((L,), generator=g, device="cuda") * 14 + 38
        rot = torch.poisson(torch.full((L,), 6.0, device="cuda"), generator=g)
        return atoms.round().clamp(8, 100).long(), rot.clamp(0, 24).long()
    small = _uniform(g, (L,)) < 0.7
    return torch.where(small, ints(15, 35), ints(60, 120)), torch.where(small, ints(0, 8), ints(8, 30))


def _unit(v):
    return v / v.norm(dim=-1, keepdim=True)


def _topology(g, atoms):
    """Parents [L, nmax] and degrees of one random tree per ligand: atom i joins an earlier atom of fewer than four bonds."""
    L, nmax = len(atoms), int(atoms.max())
    rows = torch.arange(L, device="cuda")
    parent = torch.zeros((L, nmax), dtype=torch.long, device="cuda")
    deg = torch.zeros((L, nmax), dtype=torch.long, device="cuda")
    for i in range(1, nmax):
        free = (deg[:, :i] < 4).cumsum(1).float()
        p = torch.searchsorted(free, _uniform(g, (L, 1)) * free[:, -1:], right=True).clamp(max=i - 1)[:, 0]
        grows = (atoms > i).long()
        parent[:, i] = p
        deg[rows, p] += grows
        deg[:, i] = grows
    return parent, deg


def _positions(g, parent, tries=6):
    """Positions [L, nmax, 3]: each atom at the first of `tries` azimuths that keeps 1.2 A, or at the roomiest."""
    L, nmax = parent.shape
    rows = torch.arange(L, device="cuda")
    pos = torch.zeros((L, nmax, 3), device="cuda")
    ca, sa = math.cos(math.radians(109.5)), math.sin(math.radians(109.5))
    for i in range(1, nmax):
        p = parent[:, i]
        phi = _uniform(g, (L, tries, 1), 0.0, 2 * math.pi)
        at = pos[rows, p]
        if i == 1:
            d = _unit(torch.randn((L, tries, 3), generator=g, device="cuda"))
        else:
            e = _unit(pos[rows, torch.where(p != 0, parent[rows, p], torch.ones_like(p))] - at)
            z = torch.zeros_like(e)
            steep = e[:, 2].abs() > math.cos(math.radians(8.0))
            z[:, 0], z[:, 2] = steep.float(), (~steep).float()
            n1 = _unit(z - (z * e).sum(-1, keepdim=True) * e)
            n2 = torch.linalg.cross(e, n1)
            d = ca * e[:, None] + sa * (phi.cos() * n1[:, None] + phi.sin() * n2[:, None])
        new = at[:, None] + 1.5 * d
        near = ((pos[:, None, :i] - new[:, :, None]) ** 2).sum(-1)
        near.scatter_(2, p[:, None, None].expand(L, tries, 1), float("inf"))
        near = near.amin(2)
        good = near >= 1.44
        pos[:, i] = new[rows, torch.where(good.any(1), good.float().argmax(1), near.argmax(1))]
    return pos


def _library(g, recipe, L, nc):
    """A ligand library, and what exact() needs of it as padded tensors. Sizes and topologies belong to
    the case; conformations, types and which bonds turn come from the seed."""
    shape = torch.Generator(device="cuda")
    shape.manual_seed(1000003 * (1 + RECIPES.index(recipe)) + L)
    atoms, rot = _sizes(shape, recipe, L)
    parent, deg = _topology(shape, atoms)
    pos = _positions(g, parent)
    nmax = pos.shape[1]
    types = torch.randint(0, nc, (L, nmax), generator=g, device="cuda")
    child = torch.arange(1, nmax, device="cuda").expand(L, nmax - 1)
    edge = child < atoms[:, None]
    may = edge & (deg.gather(1, parent[:, 1:]) >= 2) & (deg[:, 1:] >= 2)
    key = torch.where(may, _uniform(g, (L, nmax - 1)), torch.full((), 2.0, device="cuda"))
    turns = may & (key.argsort(1).argsort(1) < rot[:, None])
    have = torch.arange(nmax, device="cuda")[None] < atoms[:, None]

    def offsets(n):
        return torch.cat([torch.zeros(1, dtype=torch.long, device="cuda"), n.cumsum(0)]).int()

    lib = lg.Ligands(offsets(atoms), pos[have].contiguous(), types[have].to(torch.uint8),
                     torch.stack([parent[:, 1:], child], -1)[edge].int().contiguous(), offsets(turns.sum(1)),
                     (child - 1)[turns].int().contiguous())
    return lib, dict(atoms=atoms, pos=pos, parent=parent, types=types, turns=turns, have=have)


def _grid(g, name, site=0):
    G, nc, h, points = GRIDS[name]
    origin = torch.tensor([30.0 * site, -7.0 * site, 11.0 * site], device="cuda")
    r = _uniform(g, (points,), 7.0 ** 3, 11.0 ** 3) ** (1.0 / 3.0)
    where = h * (G - 1) / 2 + r[:, None] * _unit(torch.randn((points, 3), generator=g, device="cuda"))
    w = torch.randn((points, nc), generator=g, device="cuda") * 0.3 - 1.0
    axis = h * torch.arange(G, device="cuda")
    d2 = (axis[None, :, None] - where[:, None, :]) ** 2          # [points, G, 3]
    e = torch.exp(-d2 / (2 * 1.2 ** 2))
    b = (e[:, :, 0, None] * w[:, None, :]).reshape(points, G * nc)
    v = torch.empty((G, G, G, nc), device="cuda")
    for z in range(G):
        v[z] = ((e[:, z, 2, None] * e[:, :, 1]).T @ b).reshape(G, G, nc)
        plane = d2[:, z, 2, None] + d2[:, :, 1]                  # [points, y]
        close = torch.zeros((G, G), dtype=torch.bool, device="cuda")
        for k in range(0, points, 150):
            close |= ((plane[k:k + 150, :, None] + d2[k:k + 150, None, :, 0]) < 2.5 ** 2).any(0)
        v[z][close] = 5.0
    return lg.PocketGrid(v, origin.tolist(), h)


def _poses(g, lib, grid, P):
    """P poses per ligand, packed: within 1 A of the pocket's centre, any rotation, torsions on whole degrees."""
    L, n = lib.n_ligands, torch.from_numpy(lib.n_rot).cuda().long()
    c = grid.spacing * (grid.values.shape[0] - 1) / 2
    t = _uniform(g, (L, P, 3), -1.0, 1.0) + c + torch.tensor(grid.origin, device="cuda")
    q = _unit(torch.randn((L, P, 4), generator=g, device="cuda"))
    q = torch.where(q[..., :1] < 0, -q, q)
    most = int(n.max())
    th = torch.randint(-180, 180, (L, P, most), generator=g, device="cuda").float() * (math.pi / 180)
    full = torch.cat([t, q, th], -1)
    return full[(torch.arange(7 + most, device="cuda") < 7 + n[:, None])[:, None].expand(L, P, 7 + most)].contiguous()


def _inputs(case, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    nc = GRIDS[case["grid"]][1]
    lib, about = _library(g, case["recipe"], case["ligands"], nc)
    grids = [_grid(g, case["grid"], s) for s in range(case.get("sites", 1))]
    poses = _poses(g, lib, grids[0], case["poses"]) if "poses" in case else None
    return lib, about, grids, poses


def prepare(case, seed):
    lib, _, grids, poses = _inputs(case, seed)
    state = dict(case=case, lib=lib, grids=grids, poses=poses, seed=seed, channels=GRIDS[case["grid"]][1])
    if case["call"] == "score_prepared":
        state["prep"] = lg.prepare_scoring(lib, grids[0])
    if case["call"] == "grad":
        # the caller's objective weights each pose's score
        g = torch.Generator(device="cuda")
        g.manual_seed(seed + 1)
        state["weight"] = _uniform(g, (lib.n_ligands, case["poses"]), 0.5, 1.5)
    return state


def run(state):
    c, lib, grids, poses = state["case"], state["lib"], state["grids"], state["poses"]
    if c["call"] == "dock":
        args = dict(restarts=c["restarts"], torsion_step_deg=c["step"], passes=c["passes"], top_k=c["top_k"],
                    seed=state["seed"], batching=c["batching"], grid_format=c["fmt"], rescore_fp64=c["rescore"],
                    mode=c["mode"])
        r = lg.dock_sites(lib, grids, **args) if c["sites"] > 1 else lg.dock_batch(lib, grids[0], **args)
        return dict(scores=r.scores, poses=r.poses, status=r.status, scores_f64=r.scores_f64)
    if c["call"] == "score_prepared":
        return state["prep"].score(poses, c["poses"])
    if c["call"] == "score":
        return lg.score_poses(lib, grids[0], poses, c["poses"])
    if c["call"] == "grad":
        x = poses.detach().requires_grad_(True)
        s = lg.pose_score(x, lib, grids[0], c["poses"])
        s.backward(state["weight"])
        return dict(scores=s.detach(), grad=x.grad)
    if c["call"] == "refine":
        x, s, _ = lg.refine_poses(lib, grids[0], poses, c["poses"], steps=c["steps"])
        return dict(poses=x, scores=s)
    bits, axis, bucket, status = lg.pack_ligands(lib, state["channels"])
    return dict(bits=bits, axis=axis, bucket=bucket, status=status)


# -------------------------------------------------------------------- work --

SAMPLE = 29  # FP32 operations of one atom sample: position, box test, cell, polynomial


def work(case):
    N, n, m = MEANS[case["recipe"]]
    G, nc, _, _ = GRIDS[case["grid"]]
    L, sites = case["ligands"], case.get("sites", 1)
    ligands = L * (N * 13 + (N - 1) * 8 + n * 4 + 8)
    grid = 4 * G ** 3 * nc * sites
    if case["call"] == "pack":
        return dict(bytes=ligands + L * (n * 40 + 8), flops=L * N * 6)
    if case["call"] == "dock":
        out = L * case["top_k"] * (4 + 4 * (7 + n) + (8 if case["rescore"] else 0)) * sites
        nt = 360 // case["step"]
        if case["mode"] == "exhaustive":
            # every combination's sum over the atoms; rot is uniform on 0..3
            flops = L * case["restarts"] * 24 * sum(nt ** k for k in range(4)) / 4 * N
        else:
            # the rigid stage, the first pass's sweeps, and half of the later ones (bonds already at their optimum)
            sweeps = 1 + 0.5 * max(0, case["passes"] - 1)
            flops = L * sites * case["restarts"] * (24 * N + sweeps * n * (nt - 1) * m) * SAMPLE
        return dict(bytes=ligands + grid + out, flops=flops)
    poses = L * case["poses"]
    io = poses * 4 * (7 + n)
    evals = 1 if case["call"].startswith("score") else 3 if case["call"] == "grad" else 2 * (case["steps"] + 1)
    rw = 2 if case["call"] in ("grad", "refine") else 1
    return dict(bytes=ligands + grid + rw * io + 4 * poses, flops=evals * poses * (N * SAMPLE + n * 90))


# ------------------------------------------------------------------- exact --

def _score64(about, grid, full, P, lo, hi):
    """FP64 scores [hi - lo, P] of the padded poses `full` [hi - lo, P, 7 + n] of ligands lo .. hi - 1."""
    atoms, parent, turns = about["atoms"][lo:hi], about["parent"][lo:hi], about["turns"][lo:hi]
    have, types = about["have"][lo:hi], about["types"][lo:hi]
    B, nmax = have.shape
    rows = torch.arange(B, device="cuda")
    x0 = about["pos"][lo:hi].double() * have[..., None]
    y = (x0 - (x0.sum(1) / atoms[:, None])[:, None])[:, None].expand(B, P, nmax, 3)
    most = full.shape[-1] - 7
    # a bond's side below it (away from atom 0), by walking parents (a parent's index is below its child's)
    slot = (turns.cumsum(1) - 1).masked_fill(~turns, most)
    below = torch.zeros((B, nmax, most + 1), dtype=torch.bool, device="cuda")
    for i in range(1, nmax):
        below[:, i] = below[rows, parent[:, i]]
        below[rows, i, slot[:, i - 1]] = True
    count = turns.sum(1)
    for b in range(most):
        real = b < count
        e = (slot == b).float().argmax(1)                       # the edge of bond b
        child, up = e + 1, parent[rows, e + 1]
        side = below[:, :, b] & have
        small = 2 * side.sum(1) <= atoms                        # the smaller side moves; on a tie the one without atom 0
        moves = torch.where(small[:, None], side, ~side & have) & real[:, None]
        v, u = torch.where(small, child, up), torch.where(small, up, child)
        pv, pu = y[rows, :, v], y[rows, :, u]                   # [B, P, 3]
        k = torch.where(real[:, None, None], pv - pu, torch.ones_like(pv))
        k = _unit(k)[:, :, None]
        d = y - pv[:, :, None]
        th = full[:, :, 7 + b].double()[..., None, None]
        kk = torch.linalg.cross(k.expand_as(d), d)
        turned = pv[:, :, None] + d * th.cos() + kk * th.sin() + k * (k * d).sum(-1, keepdim=True) * (1 - th.cos())
        y = torch.where(moves[:, None, :, None], turned, y)
    q = _unit(full[:, :, 3:7].double())[:, :, None]
    w, r = q[..., :1], q[..., 1:].expand_as(y)
    c = torch.linalg.cross(r, y)
    x = y + 2 * (w * c + torch.linalg.cross(r, c)) + full[:, :, None, :3].double()
    val = grid.values
    n = torch.tensor([val.shape[2], val.shape[1], val.shape[0]], device="cuda")
    h = float(torch.tensor(grid.spacing, dtype=torch.float32))
    o = torch.tensor(grid.origin, dtype=torch.float32, device="cuda").double()
    ug = (x - o) / h
    inside = ((ug >= 0) & (ug <= n - 1)).all(-1)
    i = torch.minimum(ug.detach().floor().clamp(min=0).long(), n - 2)
    f = ug - i
    ty = types[:, None].expand(B, P, nmax)
    E = 0
    for corner in range(8):
        d = [(corner >> k) & 1 for k in range(3)]
        wt = 1
        for k in range(3):
            wt = wt * (f[..., k] if d[k] else 1 - f[..., k])
        E = E + wt * val[i[..., 2] + d[2], i[..., 1] + d[1], i[..., 0] + d[0], ty].double()
    E = torch.where(inside, E, torch.full((), 5.0, dtype=torch.float64, device="cuda"))
    return -(E * have[:, None]).sum(-1)


def exact(case, seed):
    # Docking and refinement take decisions by comparing FP32 scores: at a near-tie either choice is
    # valid and what follows is another pose, so their outputs have no value in 64 bits. The packer
    # returns whole numbers.
    if case["call"] not in ("score", "score_prepared", "grad"):
        return None
    lib, about, grids, poses = _inputs(case, seed)
    L, P = lib.n_ligands, case["poses"]
    n = about["turns"].sum(1)
    most = int(n.max())
    real = (torch.arange(7 + most, device="cuda") < 7 + n[:, None])[:, None].expand(L, P, 7 + most)
    full = torch.zeros((L, P, 7 + most), dtype=torch.float64, device="cuda")
    full[real] = poses.double()
    grad = case["call"] == "grad"
    step = max(1, (400_000 if grad else 4_000_000) // (P * about["have"].shape[1]))
    scores, grads = [], []
    if grad:
        weight = prepare(case, seed)["weight"].double()
    for lo in range(0, L, step):
        hi = min(L, lo + step)
        x = full[lo:hi].clone().requires_grad_(grad)
        s = _score64(about, grids[0], x, P, lo, hi)
        if grad:
            (s * weight[lo:hi]).sum().backward()
            grads.append(x.grad)
        scores.append(s.detach())
    scores = torch.cat(scores)
    return dict(scores=scores, grad=torch.cat(grads)[real]) if grad else scores
