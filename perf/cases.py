"""The workloads this library is timed on, each through its public calls.

A case is a dict of plain values; `prepare` makes what a program has in hand before the
call (device or pinned host buffers, a planned batch, an embedding that is kept), `run`
is one call as such a program makes it, `exact` the same numbers from plain torch in 64
bits (the integer decisions as well, so that the list of links is the same one).

A case fixes the shape of its body; the seed sets the body into the cube in one of the 48
ways that map the grid onto itself, numbers its vertices and triangles from another start,
and draws populations and weights.  So every input is another one, while the counts of
blocks and links, which the shape decides, stay those of the case.

Kinds of case
    embed       embed(): a mesh into a fresh forest, all levels, and the cut-link table
    embed_host  the same from pinned host vertices, with the table and the finest mask
                written to pinned host buffers
    batch       the captured replay of a planned batch of meshes of uneven size
    moving      new vertex positions for one planned mesh, then the replay (with headroom)
    reembed     a local deformation, re-embedded incrementally
    fwd_bwd     force and its gradient with respect to the vertices
    lbm         one lattice-Boltzmann step that consumes the table, and the force
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2512_01251_gb300 as P
from paper_2512_01251_gb300 import autograd as PA

GRID = float(1 << 20)  # vertices are multiples of 2^-20


# --------------------------------------------------------------------------- #
# the cases
# --------------------------------------------------------------------------- #
def listed():
    return [
        # the smallest call: 312 triangles, 584 blocks; launches and host time are all of it
        dict(name="embed_312", kind="embed", tris=312, R=2, levels=2, lattice=19, lmax=0, scale=1.0),
        # an odd root (coordinates are not a power of two wide: the wide integer paths), a
        # coarse flattened body, more triangles per cell in one axis than in the others
        dict(name="embed_4k_odd_root", kind="embed", tris=4048, R=3, levels=3, lattice=27, lmax=12, scale=0.5),
        # few large triangles on a fine grid: each crosses many cells
        dict(name="embed_1k_fine", kind="embed", tris=1103, R=12, levels=3, lattice=19, lmax=6, scale=0.8),
        # the ordinary case: a scanned body of about 112K triangles, D3Q19
        dict(name="embed_112k", kind="embed", tris=111392, R=16, levels=3, lattice=19, lmax=8, scale=1.0),
        # a million triangles end to end from pinned host memory into pinned host memory
        dict(name="embed_1m_host", kind="embed_host", tris=1000003, R=32, levels=3, lattice=19, lmax=16, scale=0.7),
        # the largest: 7.2M triangles, 65M cells, D3Q27
        dict(name="embed_7m", kind="embed", tris=7197216, R=32, levels=4, lattice=27, lmax=32, scale=0.5),
        # many bodies at once, 1K to 500K triangles each, roots 8 to 24, 2 to 4 levels
        dict(name="batch_10", kind="batch", meshes=10, sizes=5, lattice=19),
        # a body that moves every time step, its counts changing with it
        dict(name="moving_112k", kind="moving", tris=111392, R=16, levels=3, lattice=19, lmax=8, scale=1.0, headroom=30),
        # a local deformation of a large body
        dict(name="reembed_1m", kind="reembed", tris=999698, R=32, levels=4, lattice=27, lmax=32, scale=0.5, cone=0.995),
        # training step on the ordinary body: force, dF/dq, dq/dvertices
        dict(name="fwd_bwd_112k", kind="fwd_bwd", tris=111392, R=16, levels=3, lattice=19, lmax=8, scale=1.0),
        # the same on a coarse design mesh: thousands of links per vertex
        dict(name="fwd_bwd_coarse", kind="fwd_bwd", tris=999, R=8, levels=3, lattice=27, lmax=4, scale=0.9),
        # the solver's time step with the force on the body (6M finest cells)
        dict(name="lbm_112k", kind="lbm", tris=111392, R=16, levels=3, lattice=19, lmax=8, scale=1.0),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["embed", "embed", "embed", "embed_host", "batch", "moving", "reembed", "fwd_bwd", "lbm"])
    lattice = rng.choice([19, 27])
    if kind == "batch":
        return dict(kind=kind, meshes=rng.randint(2, 8), sizes=rng.randint(1000, 9999), lattice=lattice)
    # finest cells per axis: 4 R 2^levels, up to 2048 for a plain embedding
    R, levels = rng.randint(2, 32), rng.randint(2, 4)
    most = 2048 if kind in ("embed", "reembed") else (1024 if kind == "embed_host" else 512)
    while 4 * R << levels > most:
        R, levels = rng.randint(2, 32), rng.randint(2, 4)
    hi = {"embed": 5e6, "embed_host": 2e6, "moving": 5e5, "reembed": 2e6, "fwd_bwd": 5e5, "lbm": 5e5}[kind]
    c = dict(kind=kind, tris=_log(rng, 300, hi), R=R, levels=levels, lattice=lattice, lmax=rng.randint(0, 24),
             scale=round(rng.uniform(0.4, 1.0), 3))
    if kind == "moving":
        c["headroom"] = rng.choice([30, 50])
    if kind == "reembed":
        c["R"] = max(R, 12)  # the window has to be smaller than the domain
        while 4 * c["R"] << c["levels"] > most:
            c["levels"] -= 1
        c["cone"] = 0.99
    return c


# --------------------------------------------------------------------------- #
# inputs
# --------------------------------------------------------------------------- #
def _device():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _legendre(lmax, theta):
    """Orthonormal associated Legendre values [l, m] at cos(theta)."""
    x, s = np.cos(theta), np.sin(theta)
    p = np.zeros((lmax + 1, lmax + 1, theta.size))
    p[0, 0] = math.sqrt(0.25 / math.pi)
    for m in range(1, lmax + 1):
        p[m, m] = -math.sqrt((2 * m + 1) / (2.0 * m)) * s * p[m - 1, m - 1]
    for m in range(lmax + 1):
        for l in range(m + 1, lmax + 1):
            a = math.sqrt((4.0 * l * l - 1.0) / (l * l - m * m))
            b = math.sqrt(((l - 1.0) ** 2 - m * m) / (4.0 * (l - 1.0) ** 2 - 1.0)) if l > m + 1 else 0.0
            p[l, m] = a * (x * p[l - 1, m] - b * p[l - 2, m] if l > m + 1 else x * p[l - 1, m])
    return p


def _snap(x):
    return torch.round(x * GRID) / GRID


def _star(tris, seed, lmax, scale, radius=0.3, device=None):
    """A closed star-shaped surface on a latitude-longitude grid with about `tris`
    triangles, counter-clockwise outward: float32 vertices (multiples of 2^-20 inside the
    unit cube) and int32 triangles.  Degree-l coefficients have deviation 0.08 / l^1.5;
    axes are scaled by (1, 0.5 + scale / 2, scale) and turned at random."""
    device = device or _device()
    n_phi = max(5, int(round(math.sqrt(tris / 2.0))))
    n_theta = max(3, int(round(tris / (2.0 * n_phi))) + 1)
    theta = np.arange(n_theta + 1) * (math.pi / n_theta)
    phi = np.arange(n_phi) * (2.0 * math.pi / n_phi)
    rng = np.random.default_rng(seed)
    for _ in range(100):
        g, tr = [np.ones(theta.size)], [np.ones(phi.size)]
        leg = _legendre(lmax, theta)
        for m in range(-lmax, lmax + 1):
            a = np.array([rng.normal(0.0, 0.08 / l ** 1.5) for l in range(max(abs(m), 1), lmax + 1)])
            if a.size:
                f = math.sqrt(2.0) if m else 1.0
                g.append(f * (a[:, None] * leg[max(abs(m), 1):, abs(m)]).sum(axis=0))
                tr.append(np.cos(m * phi) if m >= 0 else np.sin(-m * phi))
        q = rng.normal(size=4)
        w, x, y, z = q / np.linalg.norm(q)
        turn = np.array([[1 - 2 * (y * y + z * z), 2 * (x * y - z * w), 2 * (x * z + y * w)],
                         [2 * (x * y + z * w), 1 - 2 * (x * x + z * z), 2 * (y * z - x * w)],
                         [2 * (x * z - y * w), 2 * (y * z + x * w), 1 - 2 * (x * x + y * y)]])
        centre = 0.5 + rng.uniform(-0.01, 0.01, size=3)
        dev = dict(dtype=torch.float64, device=device)
        rad = radius * (torch.tensor(np.stack(g, 1), **dev) @ torch.tensor(np.stack(tr, 0), **dev))
        th, ph = torch.tensor(theta, **dev)[:, None], torch.tensor(phi, **dev)[None, :]
        pts = torch.stack([rad * th.sin() * ph.cos(), rad * th.sin() * ph.sin(), rad * th.cos().expand_as(rad)], -1)
        pts = torch.cat([pts[0, :1], pts[1:-1].reshape(-1, 3), pts[-1, :1]])
        pts = pts * torch.tensor([1.0, 0.5 + 0.5 * scale, scale], **dev) @ torch.tensor(turn.T.copy(), **dev)
        pts = _snap(pts + torch.tensor(centre, **dev))
        if float(rad.min()) > 0.0 and float(pts.min()) > 0.01 and float(pts.max()) < 0.99:
            break
        radius *= 0.95
    nr = n_theta - 1
    j = torch.arange(n_phi, device=device)
    jn = (j + 1) % n_phi
    ring = 1 + n_phi * torch.arange(nr, device=device)[:, None]
    a, b, c, d = ring[:-1] + j, ring[:-1] + jn, ring[1:] + j, ring[1:] + jn
    zero = torch.zeros_like(j)
    mid = torch.stack([torch.stack([a, c, b], -1), torch.stack([b, c, d], -1)], 1).reshape(-1, 3)
    t = torch.cat([torch.stack([zero, 1 + j, 1 + jn], -1), mid,
                   torch.stack([zero + 1 + nr * n_phi, ring[-1] + jn, ring[-1] + j], -1)])
    return pts.to(torch.float32).contiguous(), t.to(torch.int32).contiguous()


def _placed(vs, t, seed):
    """The vertex arrays `vs` (one body at several times) and its triangles, turned or
    reflected by a symmetry of the cube and renumbered from another first vertex and
    triangle; a reflection reverses the triangles so that they stay outward."""
    rng = np.random.default_rng(seed)
    axes, flip = rng.permutation(3), rng.integers(0, 2, size=3)
    sv, stt = int(rng.integers(vs[0].shape[0])), int(rng.integers(t.shape[0]))
    odd = (int(axes[0] > axes[1]) + int(axes[0] > axes[2]) + int(axes[1] > axes[2]) + int(flip.sum())) % 2
    sign = torch.tensor(1.0 - 2.0 * flip, dtype=torch.float32, device=t.device)
    off = torch.tensor(1.0 * flip, dtype=torch.float32, device=t.device)
    out = [(v[:, torch.tensor(axes, device=t.device)] * sign + off).roll(sv, 0).contiguous() for v in vs]
    t = ((t + sv) % vs[0].shape[0]).roll(stt, 0)
    return out, (t[:, [0, 2, 1]] if odd else t).to(torch.int32).contiguous()


def _shape(case):
    return _star(case["tris"], 7 * case["tris"] + case["R"], case["lmax"], case["scale"])


def _mesh(case, seed):
    """Vertices, triangles, and the vertices one step later (None for a body at rest)."""
    v, t = _shape(case)
    later = [_moved(v)] if case["kind"] == "moving" else [_deformed(case, v)] if case["kind"] == "reembed" else []
    vs, t = _placed([v] + later, t, seed)
    return vs[0], t, (vs[1] if later else None)


def _batch_specs(case):
    """Sizes of a batch: triangles log-uniform 1K..500K, root 8..24, levels 2..4."""
    rng = np.random.default_rng(case["sizes"])
    return [dict(tris=int(round(math.exp(rng.uniform(math.log(1e3), math.log(5e5))))), R=int(rng.integers(8, 25)),
                 levels=int(rng.integers(2, 5)), radius=float(rng.uniform(0.15, 0.35))) for _ in range(case["meshes"])]


def _batch_mesh(spec, seed, j):
    v, t = _star(spec["tris"], spec["tris"], 8, 1.0, spec["radius"])
    (v,), t = _placed([v], t, 1000 * seed + j)
    return v, t


_DIRS = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1),
         (1, 1, 0), (-1, -1, 0), (1, -1, 0), (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1), (-1, 0, 1),
         (0, 1, 1), (0, -1, -1), (0, 1, -1), (0, -1, 1),
         (1, 1, 1), (-1, -1, -1), (1, 1, -1), (-1, -1, 1), (1, -1, 1), (-1, 1, -1), (-1, 1, 1), (1, -1, -1)]


def _weights(lattice):
    by = {19: (1 / 3, 1 / 18, 1 / 36, 0.0), 27: (8 / 27, 2 / 27, 1 / 54, 1 / 216)}[lattice]
    return [by[sum(abs(x) for x in c)] for c in _DIRS[:lattice]]


def _populations(lattice, ncell, seed):
    """Post-collision populations of a uniform flow (0.05, 0, 0) with 1 % noise, float32."""
    gen = torch.Generator(device=_device()).manual_seed(seed + 17)
    out = torch.randn((lattice, ncell), generator=gen, device=_device())
    for i, w in enumerate(_weights(lattice)):
        cu = 0.05 * _DIRS[i][0]
        out[i].mul_(0.01).add_(1.0).mul_(w * (1.0 + 3.0 * cu + 4.5 * cu * cu - 1.5 * 0.0025))
    return out


def _link_weights(n, seed):
    gen = torch.Generator(device=_device()).manual_seed(seed + 29)
    return torch.randn(n, generator=gen, device=_device())


def _deformed(case, v):
    """The vertices inside a cone about one of them pushed outwards by about 300 grid steps."""
    x = v.to(torch.float64)
    d = x - x.mean(dim=0)
    u = d / d.norm(dim=1, keepdim=True)
    sel = (u @ u[v.shape[0] * 2 // 5]) >= case["cone"]
    return _snap(torch.where(sel[:, None], x + torch.round(u * 300.0) / GRID, x)).to(torch.float32)


def _extent(case, v, new, t):
    """The extent of the moved triangles in root blocks (y_lo, y_hi, z_lo, z_hi)."""
    hit = (v != new).any(dim=1)[t.long()].any(dim=1)
    pts = torch.cat([v[t[hit].long()].reshape(-1, 3), new[t[hit].long()].reshape(-1, 3)])
    lo = torch.floor(pts.amin(dim=0) * case["R"]).int().tolist()
    hi = (torch.floor(pts.amax(dim=0) * case["R"]).int() + 1).tolist()
    return lo[1], hi[1], lo[2], hi[2]


def _moved(v):
    """The body a time step later: a little larger and displaced by a fraction of a cell."""
    x = v.to(torch.float64)
    off = torch.tensor([0.003, -0.002, 0.001], dtype=torch.float64, device=v.device)
    return _snap((x - 0.5) * 1.01 + 0.5 + off).to(torch.float32)


def prepare(case, seed):
    kind, lat = case["kind"], case["lattice"]
    st = dict(case=case)
    if kind == "batch":
        specs = _batch_specs(case)
        st["meshes"] = [P.emb_mesh_create(*_batch_mesh(s, seed, j), s["R"]) for j, s in enumerate(specs)]
        st["batch"] = P.emb_batch_create(st["meshes"], [s["levels"] for s in specs], [2] * len(specs),
                                         [lat] * len(specs))
    else:
        v, t, later = _mesh(case, seed)
        st.update(v=v, t=t)
    R, levels = case.get("R"), case.get("levels")
    if kind == "moving":
        st["meshes"] = [P.emb_mesh_create(v, t, R)]
        st["batch"] = P.emb_batch_create(st["meshes"], [levels], [2], [lat], headroom=case["headroom"])
        st["v"] = later
    if kind in ("batch", "moving"):
        s = torch.cuda.Stream()
        P.emb_batch_autotune(st["batch"], s)
        P.emb_batch_capture(st["batch"], s)
        s.synchronize()
    if kind == "embed_host":
        E = P.embed(v, t, R, levels, 2, lat)
        cap = E.links["q"].numel() * 65 // 64 + 1024
        pin = dict(pin_memory=True)
        st["links_out"] = dict(cell=torch.empty(cap, dtype=torch.int32, **pin), dir=torch.empty(cap, dtype=torch.uint8, **pin),
                               q=torch.empty(cap, dtype=torch.float32, **pin), tri=torch.empty(cap, dtype=torch.int32, **pin),
                               count=torch.zeros(1, dtype=torch.int64, **pin))
        st["mask_out"] = torch.empty(E.masks[-1].numel(), dtype=torch.int64, **pin)
        st["v"], st["t"] = v.cpu().pin_memory(), t.cpu().pin_memory()
    if kind in ("reembed", "fwd_bwd", "lbm"):
        st["E"] = E = P.embed(v, t, R, levels, 2, lat)
        if kind == "reembed":
            st["v"], st["extent"] = later, _extent(case, v, later, t)
        else:
            st["pop"] = _populations(lat, 64 * P.emb_forest_num_blocks(E.forest, levels), seed)
        if kind == "fwd_bwd":
            st["w"] = _link_weights(E.links["q"].numel(), seed)
        if kind == "lbm":
            st["out"], st["pre"] = torch.empty_like(st["pop"]), torch.empty_like(st["pop"])
    return st


# --------------------------------------------------------------------------- #
# one pass
# --------------------------------------------------------------------------- #
def _embedding(E, links, blocks=True):
    out = dict(masks=E.masks, flags=E.flags, cell=links["cell"], dir=links["dir"], tri=links["tri"], q=links["q"])
    if blocks:
        out["blocks"] = E.fetch_blocks()
    return out


def run(state):
    case = state["case"]
    kind, lat = case["kind"], case["lattice"]
    if kind == "embed":
        E = P.embed(state["v"], state["t"], case["R"], case["levels"], 2, lat)
        return _embedding(E, E.links)
    if kind == "embed_host":
        v, t = state["v"].to("cuda", non_blocking=True), state["t"].to("cuda", non_blocking=True)
        E = P.embed(v, t, case["R"], case["levels"], 2, lat, links_out=state["links_out"],
                    finest_mask_out=state["mask_out"])
        return _embedding(E, E.links)
    if kind == "batch":
        P.emb_batch_launch(state["batch"])
        got = [P.emb_batch_results(state["batch"], j) for j in range(len(state["meshes"]))]
        return [dict(r["links"], mask=r["masks"][-1], blocks=r["blocks"][-1]) for r in got]
    if kind == "moving":
        P.emb_mesh_update(state["meshes"][0], state["v"])
        P.emb_batch_launch(state["batch"])
        return P.emb_batch_results(state["batch"], 0)
    E = state["E"]
    if kind == "reembed":
        P.reembed_window(E, state["v"], state["extent"])
        return _embedding(E, E.links)
    if kind == "fwd_bwd":
        v = state["v"].detach().requires_grad_()
        q = PA.CutLinkQ.apply(v, E)
        force = PA.mex_force(q, E, state["pop"])
        gq, grad = torch.autograd.grad(force[0] + (state["w"] * q).sum(), (q, v))
        return dict(force=force.detach(), q=q.detach(), grad_q=gq, grad=grad)
    force = P.emb_mex_force(E.forest, lat, E.links["cell"], E.links["dir"], E.links["q"], state["pop"])
    pop = P.emb_lbm_step(E.forest, lat, E.links, 1.2, state["pop"], out=state["out"], pre=state["pre"])
    return dict(force=force, pop=pop)


# --------------------------------------------------------------------------- #
# what a pass cannot do without
# --------------------------------------------------------------------------- #
def _sizes(tris, R, levels, lattice, scale, radius=0.3):
    """Estimated (blocks over all levels, finest cells, links): the surface of an ellipsoid
    counted in finest cells.  About 5 finest blocks per block-sized patch of surface; a
    direction pair +-c is crossed |c| / 2 times per cell-sized patch on average."""
    a, b, c, p = radius, radius * (0.5 + 0.5 * scale), radius * scale, 1.6
    area = 4.0 * math.pi * (((a * b) ** p + (a * c) ** p + (b * c) ** p) / 3.0) ** (1.0 / p)
    per = 1.5 + 6 * math.sqrt(2.0) / 2 + (2 * math.sqrt(3.0) if lattice == 27 else 0.0)
    blocks, finest = float(R) ** 3, 0.0
    for L in range(1, levels + 1):
        finest = min(5.0 * area * float(R << L) ** 2, float(R << L) ** 3)
        blocks += finest
    return blocks, 64.0 * finest, per * area * float(4 * R << levels) ** 2


def work(case):
    kind, lat = case["kind"], case["lattice"]
    if kind == "batch":
        ws = [work(dict(kind="embed", tris=s["tris"], R=s["R"], levels=s["levels"], lattice=lat, scale=1.0))
              for s in _batch_specs(case)]
        return {k: sum(w[k] for w in ws) for k in ("bytes", "flops")}
    tris = case["tris"]
    blocks, cells, links = _sizes(tris, case["R"], case["levels"], lat, case["scale"])
    if kind in ("embed", "embed_host", "moving"):
        # 12 B a triangle and 12 B a vertex in (half as many vertices); a mask word and the
        # coordinates of a block, and 13 B a link out.  One exact line and segment test a
        # link, about 50 operations, and a box test a triangle and level.
        return dict(bytes=18.0 * tris + 20.0 * blocks + 13.0 * links,
                    flops=50.0 * links + 100.0 * tris * (case["levels"] + 1))
    if kind == "reembed":
        # the moved vertices are all read; the table and the masks are rewritten
        return dict(bytes=6.0 * tris + 16.0 * blocks + 26.0 * links, flops=0.1 * 50.0 * links)
    if kind == "fwd_bwd":
        # cell, dir, q, tri, w and up to three populations a link; the three vertices of its
        # triangle come from the caches; a gradient a vertex
        return dict(bytes=(17.0 + 12.0) * links + 18.0 * tris, flops=150.0 * links)
    return dict(bytes=8.0 * lat * cells + (9.0 + 12.0) * links, flops=10.0 * lat * cells + 30.0 * links)


# --------------------------------------------------------------------------- #
# the same numbers in 64 bits, by plain torch
# --------------------------------------------------------------------------- #
def _sign_dot(n, v):
    """Exact n . v for int64 |n| < 2^53, |v| < 2^27: its sign, and its value in float64."""
    lo = (n & 0x3FFFFF) * v
    hi = ((n >> 22) * v).sum(-1) + (lo.sum(-1) >> 22)
    lo = lo.sum(-1) & 0x3FFFFF
    return torch.where(hi != 0, hi.sign(), lo.sign()), hi.to(torch.float64) * 4194304.0 + lo.to(torch.float64)


def _cross(a, b):
    return torch.stack([a[..., 1] * b[..., 2] - a[..., 2] * b[..., 1], a[..., 2] * b[..., 0] - a[..., 0] * b[..., 2],
                        a[..., 0] * b[..., 1] - a[..., 1] * b[..., 0]], -1)


def _first_sign(w):
    """Sign of the first component that is not zero (0 if none)."""
    s = w.sign()
    return torch.where(s[..., 0] != 0, s[..., 0], torch.where(s[..., 1] != 0, s[..., 1], s[..., 2]))


def _spread(counts):
    """Item -> owner and item's rank in its owner, for owners with these counts."""
    own = torch.repeat_interleave(torch.arange(counts.numel(), device=counts.device), counts)
    first = torch.cumsum(counts, 0) - counts
    return own, torch.arange(own.numel(), device=counts.device) - first[own]


def _crossings(X, h, c):
    """Every crossing of a lattice line along c (through the cell centres) with a triangle:
    triangle, index of the last centre before it, distance to that centre in steps of h c.
    Centres are pushed by (e, e^2, e^3), e -> 0+, so none lies on a plane or an edge."""
    dev, half = X.device, h // 2
    cv = torch.tensor(c, device=dev)
    a = next(i for i in range(3) if c[i])
    rows = []
    for b in ((a + 1) % 3, (a + 2) % 3):
        r = [0, 0, 0]
        r[b] = 1
        r[a] -= c[b] * c[a]
        rows.append((b, torch.tensor(r, device=dev)))
    step = 400000
    for t0 in range(0, X.shape[0], step):
        T = X[t0:t0 + step]
        n = _cross(T[:, 1] - T[:, 0], T[:, 2] - T[:, 0])
        nc = (n * cv).sum(-1)
        lo, cnt = [], []
        for _, r in rows:
            u = (T * r).sum(-1) - half * int(r.sum())
            first = -torch.div(-u.amin(1), h, rounding_mode="floor")
            lo.append(first)
            cnt.append((torch.div(u.amax(1), h, rounding_mode="floor") - first + 1).clamp(min=0))
        own, k = _spread(torch.where(nc != 0, cnt[0] * cnt[1], torch.zeros_like(nc)))
        if own.numel() == 0:
            continue
        i0 = torch.zeros((own.numel(), 3), dtype=torch.int64, device=dev)  # the line's cell with index 0 on axis a
        i0[:, rows[0][0]] = lo[0][own] + k % cnt[0][own]
        i0[:, rows[1][0]] = lo[1][own] + torch.div(k, cnt[0][own], rounding_mode="floor")
        sn = nc.sign()[own]
        keep = torch.ones_like(own, dtype=torch.bool)
        rel = T[own] - ((2 * i0 + 1) * half)[:, None, :]
        for j in range(3):
            u, v = rel[:, j], rel[:, (j + 1) % 3]
            s = (_cross(u, v) * cv).sum(-1)
            keep &= torch.where(s != 0, s.sign(), _first_sign(_cross(cv.expand_as(u), v - u))) == sn
        own, i0, sn = own[keep], i0[keep], sn[keep]
        n, m, A = n[own], nc[own].abs().to(torch.float64), T[own][:, 0]
        at = lambda q: A - (2 * (i0 + q[:, None] * cv) + 1) * half  # noqa: E731
        est = torch.floor(_sign_dot(n, at(torch.zeros_like(own)))[1] * sn / (m * h)).long()
        ahead = torch.zeros_like(est)
        for d in (-1, 0, 1, 2):
            s = _sign_dot(n, at(est + d))[0]
            ahead += (torch.where(s != 0, s, -_first_sign(n)) == sn).long()
        k = est - 2 + ahead
        yield own + t0, i0 + k[:, None] * cv, _sign_dot(n, at(k))[1] * sn / (m * h)


def _box_hits(T, lo, hi):
    """Exact overlap of triangles T (n, 3, 3) with closed boxes (separating axes)."""
    ok = ((T.amin(1) <= hi) & (T.amax(1) >= lo)).all(-1)
    f = torch.stack([T[:, 1] - T[:, 0], T[:, 2] - T[:, 1], T[:, 0] - T[:, 2]], 1)
    n = _cross(f[:, 0], f[:, 1])
    ok &= _sign_dot(n, torch.where(n > 0, lo, hi) - T[:, 0])[0] <= 0
    ok &= _sign_dot(n, torch.where(n > 0, hi, lo) - T[:, 0])[0] >= 0
    V, E = T - lo[:, None], hi - lo
    for d in range(3):
        e = torch.zeros(3, dtype=torch.int64, device=T.device)
        e[d] = 1
        for j in range(3):
            ax = _cross(e.expand_as(f[:, j]), f[:, j])
            p, t = (V * ax[:, None]).sum(-1), ax * E
            ok &= (p.amax(1) >= t.clamp(max=0).sum(-1)) & (p.amin(1) <= t.clamp(min=0).sum(-1))
    return ok


def _reference(v, t, R, levels, lattice, band=2):
    """Finest blocks, solid cells, their block-id grid, and the link table with q in 64 bits."""
    dev = v.device
    k = (R & -R).bit_length() - 1
    X = (v.to(torch.float64) * GRID).round().long() * (R >> k)
    X = X[t.long()]
    lin = torch.arange(R ** 3, device=dev)
    blocks = torch.stack([lin % R, lin // R % R, lin // (R * R)], -1)
    rho = [float(band)]
    for _ in range(levels - 1):
        rho.append(max(band, rho[-1] / 2 + 2.5))
    grid = lin.int().view(R, R, R)
    for L in range(levels):
        h = 1 << (18 - k - L)
        W, dil, nb = 4 * h, int((rho[levels - 1 - L] - 0.5) * h), R << L
        flag = torch.zeros(blocks.shape[0], dtype=torch.bool, device=dev)
        for t0 in range(0, X.shape[0], 200000):
            T = X[t0:t0 + 200000]
            b0 = (-torch.div(-(T.amin(1) - dil - W), W, rounding_mode="floor")).clamp(min=0)
            n = (torch.div(T.amax(1) + dil, W, rounding_mode="floor").clamp(max=nb - 1) - b0 + 1).clamp(min=0)
            own, r = _spread(n.prod(-1))
            b = b0[own] + torch.stack([r % n[own, 0], torch.div(r, n[own, 0], rounding_mode="floor") % n[own, 1],
                                       torch.div(r, n[own, 0] * n[own, 1], rounding_mode="floor")], -1)
            ids = grid[b[:, 2], b[:, 1], b[:, 0]].long()
            sel = ids >= 0
            sel &= ~flag[ids.clamp(min=0)]
            own, b, ids = own[sel], b[sel], ids[sel]
            flag[ids[_box_hits(T[own], b * W - dil, b * W + W + dil)]] = True
        child = torch.stack([torch.tensor([i & 1, i >> 1 & 1, i >> 2], device=dev) for i in range(8)])
        blocks = (2 * blocks[flag][:, None] + child).reshape(-1, 3)
        nb *= 2
        key = (blocks[:, 2] * nb + blocks[:, 1]) * nb + blocks[:, 0]
        blocks = blocks[key.argsort()]
        grid = torch.full((nb, nb, nb), -1, dtype=torch.int32, device=dev)
        grid[blocks[:, 2], blocks[:, 1], blocks[:, 0]] = torch.arange(blocks.shape[0], dtype=torch.int32, device=dev)
    n, h = 4 * R << levels, 1 << (18 - k - levels)
    # solid: an odd number of crossings of the +x line lie beyond the centre
    keys = [torch.zeros(0, dtype=torch.int64, device=dev)]
    for _, i, _ in _crossings(X, h, (1, 0, 0)):
        keys.append((i[:, 2] * n + i[:, 1]) * (n + 2) + (i[:, 0] + 1).clamp(0, n + 1))
    keys = torch.cat(keys).sort()[0]
    local = torch.arange(64, device=dev)
    local = torch.stack([local & 3, local >> 2 & 3, local >> 4], -1)
    solid = torch.empty((blocks.shape[0], 64), dtype=torch.bool, device=dev)
    for b0 in range(0, blocks.shape[0], 1 << 17):
        i = 4 * blocks[b0:b0 + (1 << 17), None] + local
        line = (i[..., 2] * n + i[..., 1]) * (n + 2)
        solid[b0:b0 + (1 << 17)] = ((torch.searchsorted(keys, line + n + 2) - torch.searchsorted(keys, line + i[..., 0] + 1)) % 2) > 0
    ref = dict(X=X, blocks=blocks, grid=grid, solid=solid, n=n, h=h)
    # links: fluid cells with a solid neighbour, in (cell, dir) order
    keys = []
    for d in range(1, lattice):
        for b0 in range(0, blocks.shape[0], 1 << 17):
            cell, s = _at(ref, 4 * blocks[b0:b0 + (1 << 17), None] + local + torch.tensor(_DIRS[d], device=dev))
            i = ((cell >= 0) & s & ~solid[b0:b0 + (1 << 17)]).reshape(-1).nonzero()[:, 0]
            keys.append((i + 64 * b0) * 32 + d)
    link = torch.cat(keys).sort()[0]
    ref["cell"], ref["dir"] = link >> 5, link & 31
    q = torch.full((link.numel(),), float("inf"), dtype=torch.float64, device=dev)
    hits = []
    for d in range(1, lattice, 2):
        for tri, i, s in _crossings(X, h, _DIRS[d]):
            (ca, sa), (cb, sb) = _at(ref, i), _at(ref, i + torch.tensor(_DIRS[d], device=dev))
            both = (ca >= 0) & (cb >= 0) & (sa != sb)
            key = torch.where(sa, cb * 32 + d + 1, ca * 32 + d)[both]
            at = torch.searchsorted(link, key)
            val = torch.where(sa, 1.0 - s, s)[both]
            hits.append((at, val, tri[both]))
            q.scatter_reduce_(0, at, val, "amin")
    ref["q"], ref["tri"] = q, torch.full_like(link, X.shape[0])
    for at, val, tri in hits:
        near = val == q[at]
        ref["tri"].scatter_reduce_(0, at[near], tri[near], "amin")
    return ref


def _at(ref, i):
    """Cell id (-1 where its block is missing or outside) and whether it is solid."""
    n = ref["n"]
    inside = ((i >= 0) & (i < n)).all(-1)
    j = i.clamp(0, n - 1)
    b = ref["grid"][j[..., 2] >> 2, j[..., 1] >> 2, j[..., 0] >> 2].long()
    t = (j[..., 0] & 3) + 4 * (j[..., 1] & 3) + 16 * (j[..., 2] & 3)
    ok = inside & (b >= 0)
    return torch.where(ok, b * 64 + t, -torch.ones_like(b)), ok & ref["solid"][b.clamp(min=0), t]


def _cell_index(ref, cell):
    t = cell & 63
    return 4 * ref["blocks"][cell >> 6] + torch.stack([t & 3, t >> 2 & 3, t >> 4], -1)


def _bouzidi(ref, pop):
    """Per link: c, f_i, the population returned against it, and its derivative in q."""
    c = torch.tensor(_DIRS, device=pop.device)[ref["dir"]]
    cell, d, q = ref["cell"], ref["dir"], ref["q"]
    opp = torch.where(d % 2 == 1, d + 1, d - 1)
    fi, fo = pop[d, cell].double(), pop[opp, cell].double()
    back, bs = _at(ref, _cell_index(ref, cell) - c)
    has = (back >= 0) & ~bs
    fp = pop[d, back.clamp(min=0)].double()
    near = torch.where(has, 2 * q * fi + (1 - 2 * q) * fp, fi)
    g = torch.where(q < 0.5, near, fi / (2 * q) + (2 * q - 1) / (2 * q) * fo)
    dg = torch.where(q < 0.5, torch.where(has, 2 * (fi - fp), torch.zeros_like(fi)), (fo - fi) / (2 * q * q))
    return c.double(), opp, fi, g, dg


def _exact_links(v, t, R, levels, lattice):
    return _reference(v, t, R, levels, lattice)["q"]


def exact(case, seed):
    if _device() != "cuda":
        return None  # minutes on a CPU for the larger cases
    kind, lat = case["kind"], case["lattice"]
    if kind == "batch":
        out = []
        for j, s in enumerate(_batch_specs(case)):
            q = _exact_links(*_batch_mesh(s, seed, j), s["R"], s["levels"], lat)
            out.append(dict(cell=None, dir=None, q=q, tri=None, mask=None, blocks=None))
        return out
    v, t, later = _mesh(case, seed)
    v = v if later is None else later
    none = [None] * (case["levels"] + 1)
    if kind == "moving":
        q = _exact_links(v, t, case["R"], case["levels"], lat)
        return dict(blocks=none, masks=none, links=dict(cell=None, dir=None, q=q, tri=None))
    if kind in ("embed", "embed_host", "reembed"):
        q = _exact_links(v, t, case["R"], case["levels"], lat)
        return dict(masks=none, flags=none[1:] if kind != "reembed" else [], cell=None, dir=None, tri=None, q=q, blocks=none)
    ref = _reference(v, t, case["R"], case["levels"], lat)
    pop = _populations(lat, ref["solid"].numel(), seed)
    c, opp, fi, g, dg = _bouzidi(ref, pop)
    force = (c * (fi + g)[:, None]).sum(0)
    if kind == "fwd_bwd":
        w = _link_weights(ref["q"].numel(), seed).double() + c[:, 0] * dg
        T = ref["X"][ref["tri"]].double()
        e1, e2 = T[:, 1] - T[:, 0], T[:, 2] - T[:, 0]
        n = torch.linalg.cross(e1, e2)
        hit = (2 * _cell_index(ref, ref["cell"]) + 1).double() * (ref["h"] / 2) + (ref["q"] * ref["h"])[:, None] * c - T[:, 0]
        nn = (n * n).sum(-1)
        l1 = (n * torch.linalg.cross(hit, e2)).sum(-1) / nn
        l2 = (n * torch.linalg.cross(e1, hit)).sum(-1) / nn
        per = n * (w * GRID * (case["R"] // (case["R"] & -case["R"])) / (ref["h"] * (n * c).sum(-1)))[:, None]
        grad = torch.zeros((v.shape[0], 3), dtype=torch.float64, device=v.device)
        for j, lam in enumerate((1 - l1 - l2, l1, l2)):
            grad.index_add_(0, t[:, j].long()[ref["tri"]], per * lam[:, None])
        return dict(force=force, q=ref["q"], grad_q=w, grad=grad)
    # pull streaming, the returned populations at the links, BGK collision
    fluid = ~ref["solid"].reshape(-1)
    cells = _cell_index(ref, torch.arange(fluid.numel(), device=pop.device))
    f = torch.empty(pop.shape, dtype=torch.float64, device=pop.device)
    for i in range(lat):
        src, s = _at(ref, cells - torch.tensor(_DIRS[i], device=pop.device))
        f[i] = torch.where(src >= 0, pop[i, src.clamp(min=0)], pop[i]).double() * (~s)
    f[opp, ref["cell"]] = g
    cc, wt = torch.tensor(_DIRS[:lat], device=pop.device).double(), torch.tensor(_weights(lat), device=pop.device).double()
    rho = f.sum(0)
    u = (cc.T @ f) / rho
    out = torch.empty_like(f)
    for i in range(lat):
        cu = (cc[i][:, None] * u).sum(0)
        out[i] = f[i] - 1.2 * (f[i] - wt[i] * rho * (1 + 3 * cu + 4.5 * cu * cu - 1.5 * (u * u).sum(0)))
    return dict(force=force, pop=torch.where(fluid, out, torch.zeros_like(out)))
