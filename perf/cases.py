"""Timed cases: what a user of this library has it do, through its public entry points.

Each case is one step of a program: a frame update, a collision query, a metric, an
optimisation step, a render.  listed() holds the sizes of the repository's own workloads
(the single frame, the 200k-face physics frame, the varying-topology sequence, the
64-scene batch, the template fit, the 10K-point metrics); draw() spreads the same paths
over their whole ranges.  Meshes are seeded tori and spheres with smooth displacements,
deformed by four-bone skinning, generated on the device.

exact() restates each path in float64 torch, without the library.
"""
from __future__ import annotations

import math

import torch

from paper_2606_00444_gb300 import MeshBatch, MeshBVH, Workspace, chamfer, emd, gs_render, gs_render_capacity, morton_order
from paper_2606_00444_gb300.autograd import Chamfer, Interpolate, PointMeshDistance, chamfer_state

DEV = "cuda"


def listed() -> list[dict]:
    return [
        # The smallest call: one frame at the paper's mesh sizes (a 5k-face reconstruction
        # is indexed, a 1.2k-face template and some particles are projected onto it, the
        # template's tree and Gaussians follow).  Latency and launches.
        dict(name="frame_5k", path="frame", template=1152, faces=5000, queries=4099),
        # The fixed-topology frame update: new vertices, boxes and 3 Gaussians per face.
        dict(name="update_200k", path="update", faces=200_000, per_face=3, offsets=False),
        # The varying-topology frame's rebuild of the collision tree.
        dict(name="rebuild_200k", path="rebuild", faces=200_000),
        # Two physics steps at the paper's mesh sizes: refit, then warm-started contacts.
        dict(name="contact_20k", path="contact", faces=20_000, particles=20_011, cutoff=0.05),
        # Two physics steps of the million-particle scene.
        dict(name="contact_1m", path="contact", faces=200_000, particles=1 << 20, cutoff=0.05),
        # The Chamfer metric: 10K samples per side, per-sample results kept.
        dict(name="chamfer_10k", path="chamfer", faces=200_000, samples=10_000),
        # A step of the differentiable template fit, forward and backward.
        dict(name="fit_1m", path="fit", faces=81_608, target=45_000, samples=1 << 20),
        # 64 scenes rebuilt, queried (unbounded) and rebound in single launches.
        dict(name="batch_64", path="batch", scenes=64, faces_min=1_000, faces_max=200_000),
        # The Gaussian render of the physics frame.
        dict(name="render_600k", path="render", faces=200_000, per_face=3, width=1280, height=720, capacity=False),
        # The Earth Mover's Distance metric on 10K samples.
        dict(name="emd_10k", path="emd", points=10_000, eps=1e-4),
        # Signed contact (penetration depth) of a million particles.
        dict(name="signed_1m", path="signed", faces=200_000, particles=1 << 20, cutoff=0.05),
        # A tracked frame of a varying-topology sequence: rebuild, k-NN projection.
        dict(name="track_40k", path="track", faces=40_000, points=13_700, k=4, anchor=0.2),
    ]


def draw(rng) -> dict:
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    path = rng.choice(["frame", "update", "rebuild", "contact", "chamfer", "fit", "batch", "render", "emd", "signed",
                       "track"])
    if path == "frame":
        return dict(path=path, template=log(300, 20_000), faces=log(1_000, 50_000), queries=log(100, 50_000))
    if path == "update":
        faces = log(1_000, 2_400_000)
        return dict(path=path, faces=faces, per_face=rng.randint(1, 4) if faces < 800_000 else 1,
                    offsets=rng.random() < 0.5)
    if path == "rebuild":
        return dict(path=path, faces=log(1_000, 2_400_000))
    if path == "contact":
        return dict(path=path, faces=log(2_000, 400_000), particles=log(1_000, 2_000_000),
                    cutoff=rng.choice([0.02, 0.05, 0.1]))
    if path == "chamfer":
        return dict(path=path, faces=log(2_000, 400_000), samples=log(1_000, 100_000))
    if path == "fit":
        return dict(path=path, faces=log(2_000, 82_000), target=log(5_000, 50_000), samples=log(10_000, 1 << 20))
    if path == "batch":
        lo = log(500, 4_000)
        return dict(path=path, scenes=rng.randint(2, 64), faces_min=lo, faces_max=log(2 * lo, 150_000))
    if path == "render":
        w, h = rng.choice([(512, 512), (640, 360), (801, 599), (1280, 720)])
        return dict(path=path, faces=log(5_000, 200_000), per_face=rng.randint(1, 3), width=w, height=h,
                    capacity=rng.random() < 0.5)
    if path == "emd":
        return dict(path=path, points=log(2_000, 10_000), eps=rng.choice([1e-3, 3e-4, 1e-4]))
    if path == "signed":
        return dict(path=path, faces=log(2_000, 400_000), particles=log(1_000, 1 << 20),
                    cutoff=rng.choice([0.05, 0.2]))
    return dict(path=path, faces=log(2_000, 60_000), points=log(500, 40_000), k=rng.randint(1, 8),
                anchor=rng.choice([0.0, 0.2]))


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------
def _gen(seed: int) -> torch.Generator:
    g = torch.Generator(device=DEV)
    g.manual_seed(1_000_003 * seed + 17)
    return g


def _uniform(g, lo: float, hi: float, *shape) -> torch.Tensor:
    return lo + (hi - lo) * torch.rand(*shape, generator=g, device=DEV, dtype=torch.float64)


def _torus(faces: int, g, amp: float = 0.0):
    """A grid torus (radii 1, 0.35) of about `faces` faces, its tube displaced smoothly by
    up to `amp` of its radius: (V float64, F int32)."""
    nv = max(3, round(math.sqrt(faces / 3.2)))
    nu = max(3, round(faces / (2 * nv)))
    u = 2 * math.pi * torch.arange(nu, device=DEV, dtype=torch.float64)[:, None] / nu
    v = 2 * math.pi * torch.arange(nv, device=DEV, dtype=torch.float64)[None, :] / nv
    ph = _uniform(g, 0.0, 2 * math.pi, 2)
    r = 0.35 * (1 + amp * torch.sin(3 * u + ph[0]) * torch.cos(2 * v + ph[1]))
    ring = 1 + r * torch.cos(v)
    V = torch.stack([ring * torch.cos(u), ring * torch.sin(u), r * torch.sin(v)], -1).reshape(-1, 3)
    i = torch.arange(nu, device=DEV)[:, None].expand(nu, nv)
    j = torch.arange(nv, device=DEV)[None, :].expand(nu, nv)
    i1, j1 = (i + 1) % nu, (j + 1) % nv
    q00, q10, q11, q01 = ((a * nv + b).reshape(-1) for a, b in ((i, j), (i1, j), (i1, j1), (i, j1)))
    F = torch.cat([torch.stack([q00, q10, q11], 1), torch.stack([q00, q11, q01], 1)])
    return V, F.int()


def _sphere(faces: int, g, amp: float = 0.0, radius: float = 1.0):
    """A subdivided octahedron of about `faces` faces on a sphere whose radius is displaced
    smoothly by up to `amp`: (V float64, F int32), counter-clockwise from outside."""
    n = max(1, round(math.sqrt(faces / 8)))
    a, b = torch.meshgrid(torch.arange(n, device=DEV), torch.arange(n, device=DEV), indexing="ij")
    up = a + b < n
    a0, b0 = a[up], b[up]
    down = a + b < n - 1
    a1, b1 = a[down], b[down]
    pts = torch.cat([torch.stack([torch.stack([a0, b0]), torch.stack([a0 + 1, b0]), torch.stack([a0, b0 + 1])]),
                     torch.stack([torch.stack([a1 + 1, b1]), torch.stack([a1 + 1, b1 + 1]),
                                  torch.stack([a1, b1 + 1])])], 2)          # [corner, (a, b), face]
    lat = torch.stack([pts[:, 0], pts[:, 1], n - pts[:, 0] - pts[:, 1]], -1)   # [corner, face, xyz], sums to n
    tri = []
    for s in range(8):
        sg = torch.tensor([1 - 2 * (s & 1), 1 - (s & 2), 1 - (s >> 1 & 2)], device=DEV)
        t = lat * sg
        tri.append(t if int(sg.prod()) > 0 else t.flip(0))
    P = torch.cat(tri, 1).transpose(0, 1).reshape(-1, 3)                  # three corners per face
    m = 2 * n + 1
    key = ((P[:, 0] + n) * m + P[:, 1] + n) * m + P[:, 2] + n
    uniq, inv = torch.unique(key, return_inverse=True)
    L = torch.stack([uniq // (m * m) - n, uniq // m % m - n, uniq % m - n], 1).double()
    V = L / L.norm(dim=1, keepdim=True)
    ph = _uniform(g, 0.0, 2 * math.pi, 2)
    theta, phi = torch.atan2(V[:, 1], V[:, 0]), torch.acos(V[:, 2].clamp(-1, 1))
    r = 1 + amp * torch.sin(phi) * torch.sin(3 * theta + ph[0]) * torch.cos(2 * phi + ph[1])
    return V * (radius * r)[:, None], inv.reshape(-1, 3).int()


def _scan_order(V, F):
    """The faces in the order of a grid scan, as an extracted isosurface stores them."""
    c = ((V[F.long()].mean(1) + 2) * 32).long()
    return F[torch.argsort((c[:, 0] * 256 + c[:, 1]) * 256 + c[:, 2], stable=True)].contiguous()


def _poses(V, g, count: int, step: float = 2 * math.pi / 125):
    """`count` consecutive frames of a four-bone linear-blend skinning of a ring-shaped mesh
    (float32): bones at ring angles 0, 90, 180, 270 degrees, rotations up to 30 degrees."""
    ang = torch.arange(4, device=DEV, dtype=torch.float64) * (math.pi / 2)
    pivot = torch.stack([ang.cos(), ang.sin(), torch.zeros_like(ang)], 1)
    axis = torch.nn.functional.normalize(_uniform(g, -1.0, 1.0, 4, 3), dim=1)
    phase = _uniform(g, 0.0, 2 * math.pi, 4)
    d = torch.atan2(V[:, 1], V[:, 0])[:, None] - ang
    d = torch.remainder(d + math.pi, 2 * math.pi) - math.pi
    w = torch.softmax(-4.0 * d * d, 1)
    out = []
    for t in range(count):
        a = (math.pi / 6) * torch.sin(step * t + phase)
        X = torch.zeros_like(V)
        for b in range(4):
            p = V - pivot[b]
            k = axis[b].expand_as(p)
            R = p * a[b].cos() + torch.cross(k, p, dim=1) * a[b].sin() + k * (p @ axis[b])[:, None] * (1 - a[b].cos())
            X += w[:, b:b + 1] * (R + pivot[b])
        out.append(X.float().contiguous())
    return out


def _samples(V, F, n: int, g):
    """n area-uniform surface samples: (face int32, weights float32 [n, 3])."""
    t = V.double()[F.long()]
    area = torch.cross(t[:, 1] - t[:, 0], t[:, 2] - t[:, 0], dim=1).norm(dim=1)
    cdf = area.cumsum(0)
    face = torch.searchsorted(cdf, _uniform(g, 0.0, 1.0, n) * cdf[-1], right=True).clamp(max=len(F) - 1)
    r = _uniform(g, 0.0, 1.0, n, 2)
    s = r[:, 0].sqrt()
    return face.int(), torch.stack([1 - s, s * (1 - r[:, 1]), s * r[:, 1]], 1).float()


def _points(V, F, face, bary) -> torch.Tensor:
    return (V.double()[F.long()[face.long()]] * bary.double()[:, :, None]).sum(1).float()


def _grid_order(P) -> torch.Tensor:
    """Permutation of the points along a Z curve over their box."""
    lo = P.amin(0)
    cell = ((P - lo) / (P.amax(0) - lo).amax().clamp_min(1e-30) * 1023).long()
    key = torch.zeros(len(P), dtype=torch.int64, device=DEV)
    for bit in range(10):
        for axis in range(3):
            key |= (cell[:, axis] >> bit & 1) << (3 * bit + 2 - axis)
    return torch.argsort(key)


def _particles(V, n: int, g, grow: float = 0.2) -> torch.Tensor:
    """n points uniform in the mesh box grown by `grow`, stored along a Z curve."""
    lo, hi = V.amin(0).double() - grow, V.amax(0).double() + grow
    P = lo + (hi - lo) * _uniform(g, 0.0, 1.0, n, 3)
    return P[_grid_order(P)].float().contiguous()


def _inputs(case: dict, seed: int) -> dict:
    """The arrays of a case, from its seed alone (shared by prepare and exact)."""
    g, p = _gen(seed), case["path"]
    if p == "frame":
        VT, FT = _sphere(case["template"], g)
        VG, FG = _sphere(case["faces"], g, 0.1)
        VT, VG = VT.float(), VG.float()
        Q = torch.cat([VT, _uniform(g, -1.5, 1.5, case["queries"], 3).float()])
        return dict(VT=VT, FT=FT, VG=VG, FG=FG, Q=Q)
    if p == "update":
        V, F = _torus(case["faces"], g)
        m = case["per_face"]
        cnt = (torch.arange(len(F), device=DEV) % (2 * m + 1))[torch.randperm(len(F), generator=g, device=DEV)]
        gstart = torch.nn.functional.pad(cnt.cumsum(0), (1, 0)).int()
        gface = torch.repeat_interleave(torch.arange(len(F), device=DEV), cnt)
        bary = _uniform(g, 0.05, 1.0, len(gface), 3)
        goff = _uniform(g, -0.01, 0.01, len(gface)).float() if case["offsets"] else None
        return dict(V0=V.float(), F=F, V=_poses(V, g, 1)[0], gstart=gstart, gface=gface.int(),
                    gbary=(bary / bary.sum(1, keepdim=True)).float(), goff=goff)
    if p == "rebuild":
        V0, F0 = _torus(case["faces"], g, 0.2)
        V1, F1 = _torus(case["faces"], g, 0.2)
        return dict(V0=V0.float(), F0=_scan_order(V0, F0), V=V1.float(), F=_scan_order(V1, F1))
    if p in ("contact", "signed"):
        V, F = _torus(case["faces"], g)
        return dict(V0=V.float(), F=F, frames=_poses(V, g, 3), P=_particles(V, case["particles"], g))
    if p == "chamfer":
        V, F = _torus(case["faces"], g)
        VA, VB = _poses(V, g, 1)[0], V.float()
        n = case["samples"]
        return dict(VA=VA, VB=VB, F=F, SA=_points(VA, F, *_samples(VA, F, n, g)), SB=_points(VB, F, *_samples(VB, F, n, g)))
    if p == "fit":
        VT, FT = _sphere(case["faces"], g, 0.02, 0.9)
        VG, FG = _sphere(case["target"], g, 0.15, 0.9)
        VT, VG, n = VT.float(), VG.float(), case["samples"]
        face, bary = _samples(VT, FT, n, g)
        return dict(VT=VT, FT=FT, VG=VG, FG=_scan_order(VG, FG), face=face, bary=bary,
                    SG=_points(VG, FG, *_samples(VG, FG, n, g)))
    if p == "batch":
        fmin, fmax = case["faces_min"], case["faces_max"]
        meshes, queries = [], []
        for s in range(case["scenes"]):                  # log-uniform sizes, in no order
            faces = round(fmin * (fmax / fmin) ** math.modf((s + 0.5) * 0.6180339887498949)[0])
            V, F = _torus(faces, g, 0.1) if s % 2 == 0 else _sphere(faces, g, 0.1)
            V = V.float()
            ext = (V.amax(0) - V.amin(0)).double()
            lo = V.amin(0).double() - 0.1 * ext
            meshes.append((V, F))
            queries.append((lo + 1.2 * ext * _uniform(g, 0.0, 1.0, 4 * len(V), 3)).float())
        return dict(meshes=meshes, queries=queries)
    if p == "render":
        V, F = _torus(case["faces"], g)
        n = case["per_face"] * len(F)
        gface = torch.arange(len(F), device=DEV).repeat_interleave(case["per_face"])
        bary = _uniform(g, 0.05, 1.0, n, 3)
        gauss = _bind64(_poses(V, g, 1)[0], F, gface, bary / bary.sum(1, keepdim=True))
        eye = torch.tensor([0.4, -2.6, 1.5], dtype=torch.float64)
        zc = -eye / eye.norm()
        xc = torch.linalg.cross(zc, torch.tensor([0.0, 0.0, 1.0], dtype=torch.float64))
        xc = xc / xc.norm()
        R = torch.stack([xc, torch.linalg.cross(zc, xc), zc])
        f, w, h = 1100.0 * case["width"] / 1280, case["width"], case["height"]
        return dict(gauss=tuple(y.float().contiguous() for y in gauss), opacity=_uniform(g, 0.4, 0.9, n).float(),
                    color=_uniform(g, 0.0, 1.0, n, 3).float(),
                    camera=(R, -R @ eye, f, f, 0.5 * w, 0.5 * h, w, h))
    if p == "emd":
        VA, FA = _sphere(20_000, g, 0.1, 0.9)
        VB, FB = _sphere(20_000, g, 0.1)
        n = case["points"]
        return dict(A=_points(VA, FA, *_samples(VA, FA, n, g)), B=_points(VB, FB, *_samples(VB, FB, n, g)))
    V0, F0 = _torus(case["faces"], g, 0.2)
    V1, F1 = _torus(case["faces"], g, 0.2)
    Vt, Ft = _torus(2 * case["points"], g, 0.2)
    return dict(V0=V0.float(), F0=_scan_order(V0, F0), V=V1.float(), F=_scan_order(V1, F1),
                Q=Vt.float()[:case["points"]].contiguous())


def _query_out(n: int, dist: str = "dist2", face=None) -> dict:
    e = lambda *s: torch.empty(*s, device=DEV)  # noqa: E731
    return {"face": torch.full((n,), -1, dtype=torch.int32, device=DEV) if face is None else face,
            "bary": e(n, 3), "point": e(n, 3), dist: e(n)}


def prepare(case: dict, seed: int) -> dict:
    """The inputs and what a program keeps from call to call: meshes whose topology is fixed
    with the tree built from their rest pose, queries stored in Morton order, workspaces,
    output arrays."""
    x, p = _inputs(case, seed), case["path"]
    s = dict(case=dict(case), **x)
    if p == "frame":
        s["target"] = MeshBVH(len(x["VG"]), len(x["FG"]), DEV)
        s["template"] = MeshBVH.from_mesh(x["VT"], x["FT"])
        s["gface"] = torch.arange(len(x["FT"]), dtype=torch.int32, device=DEV)
        s["gbary"] = torch.full((len(x["FT"]), 3), 1 / 3, device=DEV)
        s["out"] = _query_out(len(x["Q"]))
    elif p == "update":
        s["mesh"] = MeshBVH.from_mesh(x["V0"], x["F"], method="ploc")
        s["arrays"] = s["mesh"].arrays()
        n = len(x["gbary"])
        s["out"] = tuple(torch.empty(n, c, device=DEV) for c in (3, 4, 3))
    elif p == "rebuild":
        s["mesh"] = MeshBVH.from_mesh(x["V0"], x["F0"])
        s["arrays"] = s["mesh"].arrays()
    elif p in ("contact", "signed"):
        P = x["P"]
        s["mesh"] = MeshBVH.from_mesh(x["V0"], x["F"], method="ploc")
        if p == "signed":
            s["out"] = _query_out(len(P), "sdist")
        else:
            s["ws"], s["out"] = Workspace(torch.device(DEV)), [_query_out(len(P))]
            s["out"].append(_query_out(len(P), face=s["out"][0]["face"]))
        s["mesh"].refit(x["frames"][0])
        if p == "contact":                               # the step before the timed ones
            s["mesh"].contact(P, case["cutoff"], s["out"][0], ws=s["ws"])
        else:                                            # (its first call derives the adjacency)
            s["mesh"].signed_distance(P[:1].contiguous(), case["cutoff"])
    elif p == "chamfer":
        s["A"] = MeshBVH.from_mesh(x["VB"], x["F"], method="ploc")
        s["B"] = MeshBVH.from_mesh(x["VB"], x["F"], method="ploc")
        s["ws"] = Workspace(torch.device(DEV))
    elif p == "fit":
        s["tmpl"] = MeshBVH.from_mesh(x["VT"], x["FT"], method="ploc")
        s["targ"] = MeshBVH.from_mesh(x["VG"], x["FG"], method="ploc")
        o = morton_order(_points(x["VT"], x["FT"], x["face"], x["bary"])).long()
        s["face"], s["bary"] = x["face"][o].contiguous(), x["bary"][o].contiguous()
        s["SG"] = x["SG"][morton_order(x["SG"]).long()].contiguous()
        s["V"] = x["VT"].clone().requires_grad_(True)
        s["state"] = chamfer_state(case["samples"], case["samples"], DEV)
    elif p == "batch":
        s["V"], s["vo"], s["F"], s["fo"] = MeshBatch.concat(x["meshes"], DEV)
        s["Q"] = torch.cat([q[morton_order(q).long()] for q in x["queries"]])
        off = torch.tensor([0] + [len(q) for q in x["queries"]], device=DEV)
        s["qo"] = off.cumsum(0).int()
        s["gface"] = torch.cat([torch.arange(len(f), dtype=torch.int32, device=DEV) for _, f in x["meshes"]])
        s["gbary"] = torch.full((len(s["gface"]), 3), 1 / 3, device=DEV)
        s["batch"] = MeshBatch(case["scenes"], len(s["V"]), len(s["F"]), DEV)
        s["out"] = _query_out(len(s["Q"]))
        s["gout"] = tuple(torch.empty(len(s["F"]), c, device=DEV) for c in (3, 4, 3))
    elif p == "render":
        s["ws"] = Workspace(torch.device(DEV))
        w, h = case["width"], case["height"]
        s["out"] = (torch.empty(h, w, 3, device=DEV), torch.empty(h, w, device=DEV))
        s["counts"] = torch.zeros(2, dtype=torch.int32, device=DEV)
    elif p == "emd":
        s["ws"] = Workspace(torch.device(DEV))
    else:
        s["mesh"] = MeshBVH.from_mesh(x["V0"], x["F0"])
        s["out"] = torch.empty_like(x["Q"])
    return s


def run(s: dict):
    case = s["case"]
    p = case["path"]
    if p == "frame":
        s["target"].build(s["VG"], s["FG"])
        out = s["target"].closest_point(s["Q"], out=s["out"])
        s["template"].refit(out["point"][:len(s["VT"])])
        mu, quat, scale = s["template"].bind_gaussians(s["gface"], s["gbary"])
        return dict(out, mu=mu, quat=quat, scale=scale)
    if p == "update":
        mu, quat, scale = s["mesh"].refit_bind(s["V"], s["gstart"], s["gbary"], s["goff"], out=s["out"])
        a = s["arrays"]
        return dict(mu=mu, quat=quat, scale=scale, verts=a["verts"], root=a["root"], boxes=a["nodes"][:, :, :3])
    if p == "rebuild":
        s["mesh"].build(s["V"], s["F"])
        a = s["arrays"]
        return dict(keys=a["keys"], perm=a["perm"], root=a["root"], boxes=a["nodes"][:, :, :3],
                    links=a["nodes_i"][:, :, 3])
    if p == "contact":
        for V, out in zip(s["frames"][1:], s["out"]):
            s["mesh"].refit(V)
            s["mesh"].contact(s["P"], case["cutoff"], out, ws=s["ws"])
        return s["out"]
    if p == "signed":
        s["mesh"].refit(s["frames"][1])
        return s["mesh"].signed_distance(s["P"], case["cutoff"], out=s["out"])
    if p == "chamfer":
        s["A"].refit(s["VA"])
        return chamfer(s["A"], s["SA"], s["B"], s["SB"], per_sample=True, ws=s["ws"])
    if p == "fit":
        V = s["V"]
        V.grad = None
        S = Interpolate.apply(V, s["tmpl"], s["face"], s["bary"])
        cd = Chamfer.apply(S, V, s["tmpl"], s["SG"], s["VG"], s["targ"], s["state"])
        d2, face = PointMeshDistance.apply(V, s["VG"], s["targ"])
        (cd[0] + cd[1] + d2.mean()).backward()
        return dict(chamfer=cd.detach(), dist2=d2.detach(), face=face, grad=V.grad)
    if p == "batch":
        b = s["batch"]
        b.build(s["V"], s["vo"], s["F"], s["fo"])
        out = b.closest_point(s["Q"], s["qo"], out=s["out"])
        mu, quat, scale = b.bind_gaussians(s["gface"], s["fo"], s["gbary"], out=s["gout"])
        return dict(out, mu=mu, quat=quat, scale=scale)
    if p == "render":
        if case["capacity"]:
            return gs_render_capacity(*s["gauss"], s["opacity"], s["color"], *s["camera"],
                                      max_instances=4 * len(s["opacity"]) + 400_000, ws=s["ws"], out=s["out"], counts=s["counts"])
        return gs_render(*s["gauss"], s["opacity"], s["color"], *s["camera"], ws=s["ws"], out=s["out"])
    if p == "emd":
        mean, sigma, _ = emd(s["A"], s["B"], case["eps"], ws=s["ws"], want_assignment=True)
        return mean, sigma
    s["mesh"].build(s["V"], s["F"])
    w = case["anchor"]
    return s["mesh"].knn_project(s["Q"], case["k"], anchor=s["Q"] if w else None, anchor_weight=w, out=s["out"],
                                 want_faces=True)


# ---------------------------------------------------------------------------
# Work
# ---------------------------------------------------------------------------
def work(case: dict) -> dict:
    """Inputs read once and outputs written once; per query one face test (60 operations)
    and a descent of two box tests (30) per level of a balanced tree."""
    p, F = case["path"], case.get("faces", 0)
    mesh = 12 * F + 6 * F                                # indices; a vertex (12 B) per two faces
    tree = 64 * F + 48 * F                               # node records and packed triangles written

    def search(n, f):
        return n * (60 + 30 * math.log2(max(f, 2)))

    if p == "frame":
        n, t = case["template"] // 2 + 2 + case["queries"], case["template"]
        return dict(bytes=mesh + tree + 44 * n + 112 * t + 12 * t + 52 * t, flops=search(n, F) + 100 * F + 200 * t)
    if p == "update":
        n = F * case["per_face"]
        return dict(bytes=mesh + tree + 8 * F + 4 * F + (52 + 4 * case["offsets"]) * n, flops=200 * F + 12 * n)
    if p == "rebuild":
        return dict(bytes=mesh + tree + 8 * F, flops=100 * F)
    if p == "contact":
        n = case["particles"]
        return dict(bytes=2 * (mesh + tree + 48 * n), flops=2 * (search(n, F) + 30 * F))
    if p == "signed":
        n = case["particles"]
        return dict(bytes=mesh + tree + 44 * n, flops=search(n, F) + 60 * F)
    if p == "chamfer":
        n = 2 * case["samples"]
        return dict(bytes=mesh + 2 * tree + 32 * n, flops=search(n, F) + 30 * F)
    if p == "fit":
        n, t = case["samples"], case["target"]
        return dict(bytes=12 * 2 * n + 16 * n + 2 * 16 * n + 112 * (F + t) + 18 * (F + t) + 12 * F,
                    flops=search(n, F) + search(n + F // 2, t) + 30 * (2 * n + F // 2))
    if p == "batch":
        lo, hi, b = case["faces_min"], case["faces_max"], case["scenes"]
        f = b * (hi - lo) / math.log(hi / lo)            # the mean of a log-uniform size
        return dict(bytes=130 * f + 44 * 2 * f + 56 * f, flops=search(2 * f, f / b) + 300 * f)
    if p == "render":
        n, px = F * case["per_face"], case["width"] * case["height"]
        return dict(bytes=56 * n + 16 * px, flops=300 * n + 30 * 4 * px)
    if p == "emd":
        n = case["points"]
        return dict(bytes=28 * n, flops=8 * n * n)
    n = case["points"]
    return dict(bytes=mesh + tree + (24 + 8 * case["k"]) * n, flops=search(n, F) + 60 * case["k"] * n + 100 * F)


# ---------------------------------------------------------------------------
# The same in float64
# ---------------------------------------------------------------------------
def _dot(a, b):
    return (a * b).sum(-1)


def _segment(q, a, b):
    """Parameter of the closest point of segment ab and the squared distance."""
    ab = b - a
    t = (_dot(q - a, ab) / _dot(ab, ab).clamp_min(1e-300)).clamp(0, 1)
    r = q - a - t[..., None] * ab
    return t, _dot(r, r)


def _triangle(q, tri):
    """Weights [..., 3] and squared distance of the closest point of each triangle to q."""
    a, b, c = tri[..., 0, :], tri[..., 1, :], tri[..., 2, :]
    e, f, p = b - a, c - a, q - a
    ee, ef, ff, pe, pf = _dot(e, e), _dot(e, f), _dot(f, f), _dot(p, e), _dot(p, f)
    det = (ee * ff - ef * ef).clamp_min(1e-300)
    v, w = (ff * pe - ef * pf) / det, (ee * pf - ef * pe) / det
    inside = (v > 0) & (w > 0) & (v + w < 1)
    r = p - v[..., None] * e - w[..., None] * f
    d = torch.where(inside, _dot(r, r), torch.full_like(v, math.inf))
    W = torch.stack([1 - v - w, v, w], -1)
    for i, j in ((0, 1), (1, 2), (2, 0)):
        t, s = _segment(q, tri[..., i, :], tri[..., j, :])
        E = torch.zeros_like(W)
        E[..., i], E[..., j] = 1 - t, t
        better = s < d
        d = torch.where(better, s, d)
        W = torch.where(better[..., None], E, W)
    return W, d


def _distance2(q, tri):
    """Squared distance alone, for [queries, faces] blocks."""
    a, b, c = tri[:, 0], tri[:, 1], tri[:, 2]
    e, f, g = b - a, c - a, c - b
    ee, ef, ff, gg = _dot(e, e), _dot(e, f), _dot(f, f), _dot(g, g).clamp_min(1e-300)
    p = q[:, None, :] - a
    pp, pe, pf = _dot(p, p), _dot(p, e), _dot(p, f)
    det = (ee * ff - ef * ef).clamp_min(1e-300)
    v, w = (ff * pe - ef * pf) / det, (ee * pf - ef * pe) / det
    inside = (v > 0) & (w > 0) & (v + w < 1)
    n = torch.cross(e, f, dim=1)
    h = _dot(p, n)
    d = torch.where(inside, h * h / _dot(n, n).clamp_min(1e-300), math.inf)
    t = (pe / ee.clamp_min(1e-300)).clamp(0, 1)
    d = torch.minimum(d, pp - 2 * t * pe + t * t * ee)
    t = (pf / ff.clamp_min(1e-300)).clamp(0, 1)
    d = torch.minimum(d, pp - 2 * t * pf + t * t * ff)
    pg, bb = pf - pe - _dot(g, e), pp - 2 * pe + ee          # (q - b) . g and |q - b|^2
    t = (pg / gg).clamp(0, 1)
    return torch.minimum(d, bb - 2 * t * pg + t * t * gg).clamp_min(0)


def _nearest(Q, V, F, cutoff: float = math.inf, k: int = 1):
    """The k nearest faces of every query (lowest id among faces within 1e-6 of the nearest
    for k = 1, -1 beyond the cutoff) with weights, points and squared distances, in float64.
    Queries are taken in spatially close groups; a group's candidates are the faces whose
    box comes within the group's bound on the k-th nearest distance."""
    Q, T = Q.double(), V.double()[F.long()]
    lo, hi = T.amin(1), T.amax(1)
    diag = float((hi.amax(0) - lo.amin(0)).norm())
    n = len(Q)
    order = _grid_order(Q)
    face = torch.full((n, k), -1, dtype=torch.int64, device=DEV)
    for i0 in range(0, n, 1024):
        idx = order[i0:i0 + 1024]
        q = Q[idx]
        c = 0.5 * (q.amin(0) + q.amax(0))
        r = float((q - c).norm(dim=1).max())
        reach = float(torch.topk((T[:, 0] - c).norm(dim=1), min(k, len(T)), largest=False).values[-1])
        bound = min(2 * r + reach, r + cutoff) * (1 + 1e-5) + 1e-9 * diag
        cand = ((torch.maximum(lo - c, c - hi).clamp_min(0)).norm(dim=1) <= bound).nonzero()[:, 0]
        if len(cand) == 0:
            continue
        step = max(1, (1 << 23) // len(cand))
        for j0 in range(0, len(q), step):
            d = _distance2(q[j0:j0 + step], T[cand])
            if k == 1:
                m = d.amin(1)
                win = (m.sqrt() * (1 + 1e-6) + 1e-12 * diag) ** 2
                f = torch.where(d <= win[:, None], cand[None, :], len(T)).amin(1)[:, None]
                f = torch.where(m[:, None] > cutoff * cutoff, -1, f)
            else:
                f = cand[torch.topk(d, min(k, len(cand)), dim=1, largest=False).indices]
            face[idx[j0:j0 + step], :f.shape[1]] = f
    hit = face >= 0
    W, d = _triangle(Q[:, None, :].expand(n, k, 3), T[face.clamp_min(0)])
    P = (W[..., None] * T[face.clamp_min(0)]).sum(2)
    zero = torch.zeros((), dtype=torch.float64, device=DEV)
    return (face, torch.where(hit[..., None], W, zero), torch.where(hit[..., None], P, zero),
            torch.where(hit, d, math.inf))


def _query64(Q, V, F, cutoff: float = math.inf) -> dict:
    _, W, P, d = _nearest(Q, V, F, cutoff)
    return dict(face=None, bary=W[:, 0], point=P[:, 0], dist2=d[:, 0])


def _bind64(V, F, gface, gbary, goff=None):
    """Centre, rotation (w >= 0) and scale of face-bound Gaussians."""
    a, b, c = V.double()[F.long()[gface.long()]].unbind(1)
    e, f = b - a, c - a
    nu = torch.cross(e, f, dim=1)
    l, an = e.norm(dim=1), nu.norm(dim=1)
    e1, n = e / l[:, None], nu / an[:, None]
    e2 = torch.cross(n, e1, dim=1)
    w = gbary.double()
    mu = w[:, :1] * a + w[:, 1:2] * b + w[:, 2:] * c + (0 if goff is None else goff.double()[:, None] * n)
    R = torch.stack([e1, e2, n], 2)
    d = R.diagonal(dim1=1, dim2=2)
    S = torch.stack([1 + d.sum(1), 1 + d[:, 0] - d[:, 1] - d[:, 2], 1 - d[:, 0] + d[:, 1] - d[:, 2],
                     1 - d[:, 0] - d[:, 1] + d[:, 2]], 1)          # 4 q_k^2
    off = torch.stack([R[:, 2, 1] - R[:, 1, 2], R[:, 0, 2] - R[:, 2, 0], R[:, 1, 0] - R[:, 0, 1],
                       R[:, 0, 1] + R[:, 1, 0], R[:, 0, 2] + R[:, 2, 0], R[:, 1, 2] + R[:, 2, 1]], 1)
    pair = torch.tensor([[-1, 0, 1, 2], [0, -1, 3, 4], [1, 3, -1, 5], [2, 4, 5, -1]], device=DEV)
    br = S.argmax(1)
    p = 0.5 * S.gather(1, br[:, None]).sqrt()
    q = off.gather(1, pair[br].clamp_min(0)) / (4 * p)
    q.scatter_(1, br[:, None], p)
    q = torch.where(q[:, :1] < 0, -q, q)
    h = an / l
    return mu, q, torch.stack([l / 3, h / 3, 0.01 * (l + h) / 6], 1)


def _signed64(Q, V, F, cutoff: float) -> dict:
    """The signed distance by the pseudo-normal of the face, edge or vertex the nearest
    point lies on."""
    face, W, P, d = (x[:, 0] for x in _nearest(Q, V, F, cutoff))
    T, Fl = V.double()[F.long()], F.long()
    N = torch.nn.functional.normalize(torch.cross(T[:, 1] - T[:, 0], T[:, 2] - T[:, 0], dim=1), dim=1)
    VN = torch.zeros(len(V), 3, dtype=torch.float64, device=DEV)
    for k in range(3):
        x, y = T[:, (k + 1) % 3] - T[:, k], T[:, (k + 2) % 3] - T[:, k]
        ang = torch.acos((_dot(x, y) / (x.norm(dim=1) * y.norm(dim=1))).clamp(-1, 1))
        VN.index_add_(0, Fl[:, k], ang[:, None] * N)
    ends = torch.stack([Fl[:, [1, 2, 0]], Fl[:, [2, 0, 1]]], 2)          # the edge opposite corner k
    ekey = ends.amin(2) * len(V) + ends.amax(2)
    _, eid = torch.unique(ekey, return_inverse=True)
    EN = torch.zeros(int(eid.max()) + 1, 3, dtype=torch.float64, device=DEV)
    for k in range(3):
        EN.index_add_(0, eid[:, k], N)
    f, zero = face.clamp_min(0), W == 0
    cnt = zero.sum(1)
    M = torch.where((cnt == 0)[:, None], N[f], EN[eid[f].gather(1, zero.long().argmax(1)[:, None])[:, 0]])
    M = torch.where((cnt >= 2)[:, None], VN[Fl[f].gather(1, W.argmax(1)[:, None])[:, 0]], M)
    sign = torch.where(_dot(Q.double() - P, M) >= 0, 1.0, -1.0)
    return dict(face=None, bary=W, point=P, sdist=torch.where(face >= 0, sign * d.sqrt(), math.inf))


def _render64(x: dict, case: dict):
    """The forward equations of Gaussian splatting, tile by tile and front to back."""
    mu, quat, scale = (y.double() for y in x["gauss"])
    Rc, t, fx, fy, cx, cy, W, H = x["camera"]
    Rc, t = Rc.float().double().to(DEV), t.float().double().to(DEV)
    X = mu @ Rc.T + t
    keep = X[:, 2] > 0.01
    w, i, j, k = torch.nn.functional.normalize(quat, dim=1).unbind(1)
    R = torch.stack([1 - 2 * (j * j + k * k), 2 * (i * j - w * k), 2 * (i * k + w * j), 2 * (i * j + w * k),
                     1 - 2 * (i * i + k * k), 2 * (j * k - w * i), 2 * (i * k - w * j), 2 * (j * k + w * i),
                     1 - 2 * (i * i + j * j)], 1).reshape(-1, 3, 3)
    M = Rc @ (R * scale[:, None, :])
    z = X[:, 2]
    J = torch.zeros(len(z), 2, 3, dtype=torch.float64, device=DEV)
    J[:, 0, 0], J[:, 0, 2], J[:, 1, 1], J[:, 1, 2] = fx / z, -fx * X[:, 0] / z ** 2, fy / z, -fy * X[:, 1] / z ** 2
    S = J @ M
    S = S @ S.transpose(1, 2)
    a, b, c = S[:, 0, 0] + 0.3, S[:, 0, 1], S[:, 1, 1] + 0.3
    det = a * c - b * b
    mid = 0.5 * (a + c)
    rad = (3 * (mid + (mid * mid - det).clamp_min(0.1).sqrt()).sqrt()).ceil()
    u, v = fx * X[:, 0] / z + cx, fy * X[:, 1] / z + cy
    gx, gy = -(-W // 16), -(-H // 16)
    x0, x1 = (((u - rad) / 16).trunc().clamp(0, gx)).long(), (((u + rad + 15) / 16).trunc().clamp(0, gx)).long()
    y0, y1 = (((v - rad) / 16).trunc().clamp(0, gy)).long(), (((v + rad + 15) / 16).trunc().clamp(0, gy)).long()
    cnt = torch.where(keep & (det > 0), (x1 - x0) * (y1 - y0), 0).clamp_min(0)
    order = torch.argsort(z.float(), stable=True)
    order = order[cnt[order] > 0]
    g = torch.repeat_interleave(order, cnt[order])
    start = cnt[order].cumsum(0) - cnt[order]
    r = torch.arange(len(g), device=DEV) - torch.repeat_interleave(start, cnt[order])
    wid = (x1 - x0)[g]
    tile = (y0[g] + r // wid) * gx + x0[g] + r % wid
    tile, perm = torch.sort(tile, stable=True)
    g = g[perm]
    first = torch.searchsorted(tile, torch.arange(gx * gy + 1, device=DEV))
    length = first[1:] - first[:-1]
    con = torch.stack([u, v, c / det, -b / det, a / det, x["opacity"].double()], 1)
    col = x["color"].double()
    tiles = torch.argsort(length, descending=True)
    tiles = tiles[length[tiles] > 0]
    pix = torch.arange(256, device=DEV)
    T = torch.ones(gx * gy, 256, dtype=torch.float64, device=DEV)
    C = torch.zeros(gx * gy, 256, 3, dtype=torch.float64, device=DEV)
    done = torch.zeros(gx * gy, 256, dtype=torch.bool, device=DEV)
    rank = 0
    while len(tiles):
        px, py = (tiles % gx * 16)[:, None] + pix % 16, (tiles // gx * 16)[:, None] + pix // 16
        Tt, Ct, Dt = T[tiles], C[tiles], done[tiles]
        ends = length[tiles]
        for rank in range(rank, rank + 64):
            live = ends > rank
            gi = g[(first[tiles] + rank).clamp(max=len(g) - 1)]
            U, Vv, ca, cb, cc, op = con[gi][:, :, None].unbind(1)
            dx, dy = U - px, Vv - py
            e = -0.5 * (ca * dx * dx + cc * dy * dy) - cb * dx * dy
            alpha = (op * torch.exp(e)).clamp(max=0.99)
            use = live[:, None] & ~Dt & (e <= 0) & (alpha >= 1 / 255)
            Tn = Tt * (1 - alpha)
            stop = use & (Tn < 1e-4)
            Dt |= stop
            use &= ~stop
            Ct += torch.where(use, alpha * Tt, 0.0)[:, :, None] * col[gi][:, None, :]
            Tt = torch.where(use, Tn, Tt)
        rank += 1
        T[tiles], C[tiles], done[tiles] = Tt, Ct, Dt
        tiles = tiles[(ends > rank) & ~Dt.all(1)]

    def image(y):
        return y.reshape(gy, gx, 16, 16, -1).permute(0, 2, 1, 3, 4).reshape(gy * 16, gx * 16, -1)[:H, :W].contiguous()

    return image(C), image(T)[:, :, 0]


def exact(case: dict, seed: int):
    p = case["path"]
    if p in ("rebuild", "batch", "emd"):
        return None          # integers and copies; 1e12 pairs; an assignment problem of n^3 steps
    x = _inputs(case, seed)
    if p == "frame":
        out = _query64(x["Q"], x["VG"], x["FG"])
        gface = torch.arange(len(x["FT"]), device=DEV)
        mu, quat, scale = _bind64(out["point"][:len(x["VT"])], x["FT"], gface,
                                  torch.full((len(gface), 3), 1 / 3, device=DEV))
        return dict(out, mu=mu, quat=quat, scale=scale)
    if p == "update":
        mu, quat, scale = _bind64(x["V"], x["F"], x["gface"], x["gbary"], x["goff"])
        return dict(mu=mu, quat=quat, scale=scale, verts=torch.nn.functional.pad(x["V"].double(), (0, 1)),
                    root=torch.stack([x["V"].amin(0), x["V"].amax(0)]).double(), boxes=None)
    if p in ("contact", "signed"):
        if p == "signed":
            return _signed64(x["P"], x["frames"][1], x["F"], case["cutoff"])
        return [_query64(x["P"], V, x["F"], case["cutoff"]) for V in x["frames"][1:]]
    if p == "chamfer":
        a, b = _query64(x["SA"], x["VB"], x["F"]), _query64(x["SB"], x["VA"], x["F"])
        return (torch.stack([a["dist2"].mean(), b["dist2"].mean()]),
                dict(faceA=None, baryA=a["bary"], dist2A=a["dist2"], faceB=None, baryB=b["bary"], dist2B=b["dist2"]))
    if p == "fit":
        VT, FT, VG, FG = x["VT"].double(), x["FT"].long(), x["VG"].double(), x["FG"].long()
        S = (VT[FT[x["face"].long()]] * x["bary"].double()[:, :, None]).sum(1)
        _, _, PA, dA = (y[:, 0] for y in _nearest(S, VG, FG))
        fB, WB, PB, dB = (y[:, 0] for y in _nearest(x["SG"], VT, FT))
        _, _, PV, dV = (y[:, 0] for y in _nearest(VT, VG, FG))
        grad = 2 * (VT - PV) / len(VT)
        gS = 2 * (S - PA) / len(S)
        grad.index_put_((FT[x["face"].long()],), x["bary"].double()[:, :, None] * gS[:, None, :], accumulate=True)
        gB = -2 * (x["SG"].double() - PB) / len(x["SG"])
        grad.index_put_((FT[fB],), WB[:, :, None] * gB[:, None, :], accumulate=True)
        return dict(chamfer=torch.stack([dA.mean(), dB.mean()]), dist2=dV, face=None, grad=grad)
    if p == "render":
        out = _render64(x, case)
        return (*out, None) if case["capacity"] else out
    face, W, P, d = _nearest(x["Q"], x["V"], x["F"], k=case["k"])
    diag = (x["V"].amax(0) - x["V"].amin(0)).double().norm()
    wt = torch.where(face >= 0, 1 / torch.maximum(d.sqrt(), 1e-6 * diag), 0.0)
    q = (wt[:, :, None] * P).sum(1) / wt.sum(1, keepdim=True)
    a = case["anchor"]
    return (1 - a) * q + a * x["Q"].double(), None, d
