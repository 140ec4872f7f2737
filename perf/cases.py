"""The work whose speed this library is judged by, as a user's program calls it.

``listed()`` names twelve cases over the library's range: collision queries
from the smallest launch to a million points in every precision and network
family, a multi-body scene, the two fitting steps, the collision-penalty
gradient, the mesh distance that gives fitting targets, the voxel baseline and
the cloth step.  ``draw()`` gives more of the same ranges.  ``prepare()`` makes
what a program holds before the call (seeded inputs on the GPU, loaded
contexts, output buffers), ``run()`` is one pass through the public entry
points, ``work()`` what that pass cannot do without and ``exact()`` its results
in 64 bits from plain torch.
"""

import functools
import math

import numpy as np
import torch

import paper_2110_01614_gb300 as nsdf
from paper_2110_01614_gb300.autograd import sdf_query
from paper_2110_01614_gb300.fit import penalty_gradient

EPS = 0.002          # collision threshold of the workloads, in body units
BETA = 100.0         # softplus sharpness

# name: (width, hidden layers, skip layer, Fourier frequencies).  "tiny" is the
# multi-body / unit network, "deep" its deepest tensor-core form, "body" the
# body-scale network, "dragon" and "bunny" the paper's Fourier-feature ReLU ones.
NETS = {
    "tiny": (64, 3, -1, 0),
    "deep": (64, 7, -1, 0),
    "body": (512, 8, 4, 0),
    "dragon": (256, 8, -1, 128),
    "bunny": (256, 4, -1, 128),
}
PRECISION = {"fp32": nsdf.NSDF_FP32, "bf16": nsdf.NSDF_BF16, "fp16": nsdf.NSDF_FP16}


def listed():
    return [
        # one small body against a few thousand cloth vertices, every frame: latency
        {"name": "collide_tiny_bf16", "kind": "collide", "net": "tiny", "precision": "bf16",
         "n": 4096, "pose": False},
        # a garment patch against the paper's smaller network placed by a pose
        {"name": "collide_bunny_fp16_ragged", "kind": "collide", "net": "bunny",
         "precision": "fp16", "n": 40013, "pose": True},
        # the headline query: a million vertices against the body-scale network
        {"name": "collide_body_bf16_1m", "kind": "collide", "net": "body", "precision": "bf16",
         "n": 1 << 20, "pose": False},
        # the same million against the paper's larger network
        {"name": "collide_dragon_bf16_1m", "kind": "collide", "net": "dragon",
         "precision": "bf16", "n": 1 << 20, "pose": False},
        # distances and normals in full precision: checks, contact refinement
        {"name": "query_body_fp32", "kind": "query", "net": "body", "precision": "fp32",
         "n": 131077},
        # a scene of 16 posed bodies of uneven size in one launch
        {"name": "grouped_posed_bf16", "kind": "grouped", "net": "tiny", "precision": "bf16",
         "bodies": 16, "lo": 2000, "hi": 400000, "pose": True},
        # one gradient step of fitting the body-scale network (L1, tensor cores)
        {"name": "fit_body_bf16", "kind": "fit_l1", "net": "body", "precision": "bf16",
         "n": 250000},
        # one gradient step of fitting a small network (L1 + eikonal, FP32)
        {"name": "fit_tiny_fp32_eikonal", "kind": "fit_eikonal", "net": "tiny", "n": 250000},
        # the force of a collision penalty on a million vertices
        {"name": "penalty_tiny_1m", "kind": "penalty", "net": "tiny", "n": 1 << 20},
        # exact distances of a fitting batch to a mesh of 20,480 triangles
        {"name": "mesh_targets_250k", "kind": "mesh", "level": 5, "n": 250000, "near": 0.8},
        # the voxel baseline: a million lookups in a 256^3 grid
        {"name": "voxel_collide_1m", "kind": "voxel", "nodes": 256, "n": 1 << 20},
        # one Verlet step of a 1024 x 1024 cloth
        {"name": "cloth_step_1024", "kind": "cloth", "nx": 1024, "ny": 1024},
    ]


def _log_int(rng, lo, hi):
    """An integer, log-uniform in [lo, hi]; two in three are odd."""
    v = int(math.exp(rng.uniform(math.log(lo), math.log(hi))))
    if rng.random() < 0.66:
        v |= 1
    return max(lo, min(hi, v))


def draw(rng):
    kind = rng.choice(["collide", "collide", "collide", "query", "grouped", "fit_l1",
                       "fit_eikonal", "penalty", "mesh", "voxel", "cloth"])
    if kind in ("collide", "query"):
        net = rng.choice(["tiny", "deep", "body", "dragon", "bunny"])
        prec = rng.choice(["bf16", "fp16", "fp32"])
        top = 1 << 20
        if prec == "fp32":               # CUDA cores: the same seconds, fewer points
            top = {"body": 131077, "dragon": 300000, "bunny": 600000}.get(net, top)
        case = {"kind": kind, "net": net, "precision": prec, "n": _log_int(rng, 1000, top)}
        if kind == "collide":
            case["pose"] = rng.random() < 0.5
        return case
    if kind == "grouped":
        hi = _log_int(rng, 4000, 400000)
        return {"kind": kind, "net": "tiny", "precision": rng.choice(["bf16", "fp16", "fp32"]),
                "bodies": rng.randint(2, 24), "lo": _log_int(rng, 500, 3000), "hi": hi,
                "pose": rng.random() < 0.5}
    if kind == "fit_l1":
        return {"kind": kind, "net": rng.choice(["body", "dragon", "bunny"]),
                "precision": rng.choice(["bf16", "fp16"]), "n": _log_int(rng, 20000, 250000)}
    if kind == "fit_eikonal":
        return {"kind": kind, "net": "tiny", "n": _log_int(rng, 20000, 250000)}
    if kind == "penalty":
        return {"kind": kind, "net": rng.choice(["tiny", "deep"]),
                "n": _log_int(rng, 10000, 1 << 20)}
    if kind == "mesh":
        level = rng.randint(3, 6)        # 1,280 to 81,920 triangles
        return {"kind": kind, "level": level,
                "n": _log_int(rng, 2000, 250000 if level < 6 else 60000),
                "near": rng.choice([0.0, 0.5, 0.8])}
    if kind == "voxel":
        return {"kind": kind, "nodes": rng.randint(48, 256), "n": _log_int(rng, 10000, 1 << 20)}
    return {"kind": "cloth", "nx": _log_int(rng, 64, 1100), "ny": _log_int(rng, 64, 900)}


# ---------------------------------------------------------------- inputs

def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(1_000_003 * int(seed) + 17)
    return g


def _rand(g, *shape):
    return torch.rand(*shape, generator=g, device="cuda")


def _randn(g, *shape):
    return torch.randn(*shape, generator=g, device="cuda")


def _pad4(xyz):
    out = torch.zeros(xyz.shape[0], 4, device="cuda")
    out[:, :3] = xyz
    return out


def _body_points(g, n):
    """90% in a thin shell about an ellipsoid (a garment on a body), 10% anywhere."""
    near = (9 * n) // 10
    u = _randn(g, near, 3)
    u = u / u.norm(dim=1, keepdim=True)
    axes = torch.tensor([0.3, 0.5, 0.2], device="cuda")
    xyz = torch.cat([u * axes + 0.01 * _randn(g, near, 3), 2.0 * _rand(g, n - near, 3) - 1.0])
    return _pad4(xyz[torch.randperm(n, generator=g, device="cuda")])


def _layers(net):
    """[(out, in)] of every layer, the output unit last."""
    width, layers, skip, ff = NETS[net]
    shapes = [(width - 3 if l == skip - 1 else width, width if l or ff else 3)
              for l in range(layers)]
    return shapes + [(1, width)]


def _blob(net, g):
    """Packed weights: a geometric initialisation (softplus) or He's (Fourier, ReLU)."""
    ff = NETS[net][3]
    parts = [2.0 * _randn(g, 3 * ff)] if ff else []
    shapes = _layers(net)
    for out, fan_in in shapes[:-1]:
        parts += [_randn(g, out * fan_in) * math.sqrt(2.0 / (fan_in if ff else out)),
                  torch.zeros(out, device="cuda")]
    width = shapes[-1][1]
    if ff:
        parts += [_randn(g, width) / math.sqrt(width), torch.zeros(1, device="cuda")]
    else:
        parts += [math.sqrt(math.pi / width) + 1e-4 * _randn(g, width),
                  torch.full((1,), -0.5, device="cuda")]
    return torch.cat(parts)


def _poses(g, n):
    """Rigid transforms: uniform rotations, shifts of up to 0.3."""
    q = _randn(g, n, 4)
    w, x, y, z = (q / q.norm(dim=1, keepdim=True)).unbind(1)
    T = torch.zeros(n, 4, 4, device="cuda")
    T[:, 0, 0], T[:, 0, 1], T[:, 0, 2] = 1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y)
    T[:, 1, 0], T[:, 1, 1], T[:, 1, 2] = 2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x)
    T[:, 2, 0], T[:, 2, 1], T[:, 2, 2] = 2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)
    T[:, :3, 3] = 0.6 * _rand(g, n, 3) - 0.3
    T[:, 3, 3] = 1.0
    return T


def _capsule(p):
    """Exact signed distance to a capsule: fitting targets that need no mesh."""
    a = torch.tensor([-0.2, -0.3, 0.1], device=p.device, dtype=p.dtype)
    b = torch.tensor([0.25, 0.35, -0.05], device=p.device, dtype=p.dtype)
    t = (((p - a) @ (b - a)) / ((b - a) @ (b - a))).clamp(0.0, 1.0)
    return (p - a - t[:, None] * (b - a)).norm(dim=1) - 0.22


@functools.lru_cache(maxsize=None)
def _icosphere(level):
    """Unit icosphere: vertices [V, 3] and outward faces [F, 3]."""
    t = (1.0 + math.sqrt(5.0)) / 2.0
    V = np.array([[-1, t, 0], [1, t, 0], [-1, -t, 0], [1, -t, 0], [0, -1, t], [0, 1, t],
                  [0, -1, -t], [0, 1, -t], [t, 0, -1], [t, 0, 1], [-t, 0, -1], [-t, 0, 1]])
    V /= np.linalg.norm(V, axis=1, keepdims=True)
    near = np.linalg.norm(V[:, None] - V[None], axis=2) < 1.1      # edges of the icosahedron
    F = np.array([(i, j, k) for i in range(12) for j in range(i) for k in range(j)
                  if near[i, j] and near[j, k] and near[i, k]])
    for _ in range(level):
        edges = np.sort(np.concatenate([F[:, [0, 1]], F[:, [1, 2]], F[:, [2, 0]]]), axis=1)
        pairs, of = np.unique(edges, axis=0, return_inverse=True)
        m = V[pairs].sum(axis=1)
        ab, bc, ca = len(V) + of.reshape(3, -1)
        V = np.concatenate([V, m / np.linalg.norm(m, axis=1, keepdims=True)])
        a, b, c = F.T
        F = np.concatenate([np.stack(x, 1) for x in
                            ((a, ab, ca), (b, bc, ab), (c, ca, bc), (ab, bc, ca))])
    n = np.cross(V[F[:, 1]] - V[F[:, 0]], V[F[:, 2]] - V[F[:, 0]])
    inward = (n * V[F[:, 0]]).sum(axis=1) < 0
    F[inward] = F[inward][:, ::-1]
    return V, F.astype(np.int32)


def _mesh(g, level):
    """A closed bumpy body of 20 * 4**level triangles."""
    V, F = _icosphere(level)
    u = torch.from_numpy(V).float().cuda()
    k = 3.0 * _randn(g, 6, 3)
    r = 0.5 + 0.05 * torch.sin(u @ k.T + 6.28 * _rand(g, 6)).mean(dim=1)
    return (u * r[:, None]).contiguous(), torch.from_numpy(F).cuda()


def _mesh_points(g, V, F, n, near):
    """Fitting samples: a share near the surface (sigma 0.01), the rest anywhere."""
    k = int(near * n)
    t = V[F.long()[torch.randint(F.shape[0], (k,), generator=g, device="cuda")]]
    u, v = _rand(g, k, 1).sqrt(), _rand(g, k, 1)
    p = (1 - u) * t[:, 0] + u * (1 - v) * t[:, 1] + u * v * t[:, 2]
    return _pad4(torch.cat([p + 0.01 * _randn(g, k, 3), 2.0 * _rand(g, n - k, 3) - 1.0]))


def _grouped_total(case):
    """Points of a scene: the mean of its bodies' log-uniform sizes, times their number."""
    lo, hi = case["lo"], max(case["lo"], case["hi"])
    mean = (hi - lo) / math.log(hi / lo) if hi > lo else lo
    return int(mean * case["bodies"])


def _inputs(case, seed):
    """Everything the pass reads, as tensors made from the seed alone."""
    g = _generator(seed)
    kind = case["kind"]
    if kind in ("collide", "query"):
        blob = _blob(case["net"], g)
        pts = (_pad4(2.0 * _rand(g, case["n"], 3) - 1.0) if case["net"] in ("tiny", "deep")
               else _body_points(g, case["n"]))
        return {"blob": blob, "pts": pts, "T": _poses(g, 1)[0] if case.get("pose") else None}
    if kind == "grouped":
        k = case["bodies"]
        u = _rand(g, k).double().cpu()
        lo, hi = math.log(case["lo"]), math.log(max(case["lo"], case["hi"]))
        counts = torch.exp(lo + (hi - lo) * u)
        # uneven sizes by the seed, the same number of points in every such scene
        total = _grouped_total(case)
        counts = (counts * (total / counts.sum())).long().clamp(min=1)
        counts[counts.argmax()] += total - counts.sum()
        offsets = torch.cumsum(counts, 0) - counts
        return {"blobs": [_blob(case["net"], g) for _ in range(k)],
                "pts": _body_points(g, int(counts.sum())), "counts": counts.cuda(),
                "offsets": offsets.cuda(), "T": _poses(g, k) if case["pose"] else None}
    if kind in ("fit_l1", "fit_eikonal"):
        blob = _blob(case["net"], g)
        pts = _body_points(g, case["n"])
        return {"blob": blob, "pts": pts, "d": _capsule(pts[:, :3].double()).float()}
    if kind == "penalty":
        return {"blob": _blob(case["net"], g), "pts": _body_points(g, case["n"])}
    if kind == "mesh":
        V, F = _mesh(g, case["level"])
        return {"V": V, "F": F, "pts": _mesh_points(g, V, F, case["n"], case["near"])}
    if kind == "voxel":
        m = case["nodes"]
        c = torch.linspace(-1.0, 1.0, m, device="cuda")
        z, y, x = torch.meshgrid(c, c, c, indexing="ij")
        k = _randn(g, 3)
        grid = _capsule(torch.stack([x, y, z], -1).reshape(-1, 3))
        grid = grid + 0.01 * torch.sin(4.0 * (x * k[0] + y * k[1] + z * k[2])).reshape(-1)
        return {"grid": grid.contiguous(), "pts": _body_points(g, case["n"])}
    nx, ny = case["nx"], case["ny"]
    h = 2.0 / (max(nx, ny) - 1)
    i, j = torch.meshgrid(torch.arange(ny, device="cuda"), torch.arange(nx, device="cuda"),
                          indexing="ij")
    a = _rand(g, 4)
    x, z = -1.0 + h * j, -1.0 + h * i
    y = 0.6 + 0.05 * torch.sin(5.0 * x + 6.28 * a[0]) * torch.cos(4.0 * z + 6.28 * a[1])
    X = _pad4(torch.stack([x, y, z], -1).reshape(-1, 3) + 0.05 * h * _randn(g, nx * ny, 3))
    prev = X.clone()
    prev[:, 1] += 1e-3
    return {"x": X, "prev": prev, "h": h}


# ---------------------------------------------------------------- the passes

def _context(case, blobs):
    width, layers, skip, ff = NETS[case["net"]]
    arch = nsdf.make_arch(width, layers, skip, BETA, activation="relu" if ff else "softplus",
                          ff_freqs=ff)
    net = nsdf.NeuralSDF(arch, PRECISION[case.get("precision", "fp32")], n_nets=len(blobs))
    for k, b in enumerate(blobs):
        net.load(b, net=k)
    return net


def prepare(case, seed):
    kind = case["kind"]
    s = _inputs(case, seed)
    s["kind"] = kind
    if kind in ("collide", "query", "penalty", "fit_eikonal", "fit_l1"):
        s["net"] = _context(case, [s["blob"]])
    if kind in ("collide", "query", "grouped", "voxel"):
        s["out_pts"] = torch.empty_like(s["pts"])
        s["out_ns"] = torch.empty_like(s["pts"])
    if kind in ("collide", "voxel"):
        # the hit byte is an optional output; programs of the FP32 form read f instead
        s["hit"] = (None if case.get("precision") == "fp32" else
                    torch.empty(s["pts"].shape[0], dtype=torch.uint8, device="cuda"))
    if kind == "collide":
        s["T"] = None if s["T"] is None else s["T"].cpu().numpy()
    elif kind == "grouped":
        s["net"] = _context(case, s["blobs"])
        s["total"] = s["pts"].shape[0]
    elif kind == "fit_l1":
        s["grad"] = torch.empty_like(s["blob"])
        s["loss"] = torch.zeros(1, device="cuda")
    elif kind == "fit_eikonal":
        s["blob"].requires_grad_(True)
    elif kind == "mesh":
        s["out"] = torch.empty(s["pts"].shape[0], device="cuda")
    elif kind == "voxel":
        s["nodes"] = case["nodes"]
    elif kind == "cloth":
        s["nx"], s["ny"] = case["nx"], case["ny"]
    return s


def run(s):
    kind = s["kind"]
    if kind == "collide":
        s["net"].collide(s["pts"], EPS, T=s["T"], out_pts=s["out_pts"], out_n_sdf=s["out_ns"],
                         out_hit=s["hit"])
        return {"pts": s["out_pts"], "n_sdf": s["out_ns"], "hit": s["hit"]}
    if kind == "query":
        return {"n_sdf": s["net"].query(s["pts"], out=s["out_ns"])}
    if kind == "grouped":
        if s["T"] is None:
            nsdf.nsdf_query_grouped(s["net"].ctx, s["pts"], s["offsets"], s["counts"], s["total"],
                                    EPS, s["out_pts"], s["out_ns"])
        else:
            nsdf.nsdf_query_grouped_T(s["net"].ctx, s["pts"], s["offsets"], s["counts"],
                                      s["total"], EPS, s["T"], s["out_pts"], s["out_ns"])
        return {"pts": s["out_pts"], "n_sdf": s["out_ns"]}
    if kind == "fit_l1":
        s["net"].load(s["blob"])              # the step's weights, then their gradient
        nsdf.nsdf_l1_grad(s["net"].ctx, s["pts"], s["d"], s["grad"], s["loss"])
        return {"grad": s["grad"], "loss": s["loss"]}
    if kind == "fit_eikonal":
        f, g = sdf_query(s["pts"], s["blob"], s["net"])
        loss = (f - s["d"]).abs().mean() + 0.1 * ((g.norm(dim=1) - 1.0) ** 2).mean()
        grad, = torch.autograd.grad(loss, s["blob"])
        return {"loss": loss.detach(), "f": f.detach(), "g": g.detach(), "grad": grad}
    if kind == "penalty":
        return {"force": penalty_gradient(s["net"], s["blob"], s["pts"], EPS)}
    if kind == "mesh":
        nsdf.nsdf_mesh_sdf(s["V"], s["F"], s["pts"], s["out"])
        return {"sdf": s["out"]}
    if kind == "voxel":
        nsdf.nsdf_voxel_collide(s["grid"], s["nodes"], (-1.0,) * 3, (1.0,) * 3, s["pts"], EPS,
                                s["out_pts"], s["out_ns"], s["hit"])
        return {"pts": s["out_pts"], "n_sdf": s["out_ns"], "hit": s["hit"]}
    nsdf.nsdf_cloth_step(s["x"], s["prev"], s["nx"], s["ny"], s["h"], s["h"], 1e5, 9.81, 1e-3)
    return {"x_new": s["prev"]}


def work(case):
    kind = case["kind"]
    if kind == "cloth":
        n = case["nx"] * case["ny"]
        return {"bytes": 48.0 * n, "flops": 130.0 * n}
    n = case.get("n", 0)
    if kind == "voxel":
        return {"bytes": 49.0 * n + 4.0 * min(case["nodes"] ** 3, 8 * n), "flops": 80.0 * n}
    if kind == "mesh":
        # one distance (about 60) and one solid angle (about 100) a level of a hierarchy
        faces = 20 * 4 ** case["level"]
        return {"bytes": 20.0 * n + 18.0 * faces, "flops": 160.0 * n * math.log2(faces)}
    shapes = _layers(case["net"])
    ff = NETS[case["net"]][3]
    mac = sum(o * i for o, i in shapes)                  # forward, and the transposed chain
    params = 4.0 * (mac + sum(o for o, _ in shapes) + 3 * ff)
    query = 2.0 * (2 * mac + 6 * ff)
    if kind == "grouped":
        n = _grouped_total(case)
        return {"bytes": 48.0 * n + case["bodies"] * params, "flops": query * n}
    if kind == "collide":
        return {"bytes": (49.0 if case["precision"] != "fp32" else 48.0) * n + params,
                "flops": query * n}
    if kind == "query":
        return {"bytes": 32.0 * n + params, "flops": query * n}
    if kind == "penalty":
        return {"bytes": 32.0 * n + params, "flops": query * n}
    if kind == "fit_l1":                                 # query chain + weight gradients
        return {"bytes": 20.0 * n + 2 * params, "flops": (query + 2.0 * mac) * n}
    # f and grad f, then reverse mode over the primal and the tangent stream
    return {"bytes": 36.0 * n + 2 * params, "flops": (query + 2.0 * 6 * mac) * n}


# ---------------------------------------------------------------- 64 bits

def _unpack(net, blob):
    ff = NETS[net][3]
    B, at, layers = None, 0, []
    if ff:
        B, at = blob[:3 * ff].reshape(ff, 3), 3 * ff
    for o, i in _layers(net):
        layers.append((blob[at:at + o * i].reshape(o, i), blob[at + o * i:at + o * i + o]))
        at += o * i + o
    return B, layers


def _field(net, blob, p, chunk=65536):
    """f and grad f at p [n, 3] by the chain rule, in the type of p."""
    skip = NETS[net][2]
    B, layers = _unpack(net, blob)
    r = 1.0 / math.sqrt(2.0)
    fs, gs = [], []
    for q in p.split(chunk):
        x = q
        if B is not None:
            ph = 2.0 * math.pi * (q @ B.T)
            x = torch.cat([ph.sin(), ph.cos()], 1)
        slopes = []
        for l, (W, b) in enumerate(layers[:-1]):
            if l == skip:
                x = torch.cat([x, q], 1) * r
            z = x @ W.T + b
            if B is not None:
                x, s = z.clamp(min=0.0), (z > 0).to(z.dtype)
            else:
                u = torch.exp(-BETA * z.abs())
                x = z.clamp(min=0.0) + torch.log1p(u) / BETA
                s = torch.where(z >= 0, 1.0 / (1.0 + u), u / (1.0 + u))
            slopes.append(s)
        W, b = layers[-1]
        fs.append((x @ W.T + b)[:, 0])
        g, direct = W.expand(q.shape[0], -1), torch.zeros_like(q)
        for l in reversed(range(len(layers) - 1)):
            g = (g * slopes[l]) @ layers[l][0]
            if l == skip:
                g = g * r
                direct, g = direct + g[:, -3:], g[:, :-3]
        if B is not None:
            m = B.shape[0]
            g = 2.0 * math.pi * ((g[:, :m] * ph.cos() - g[:, m:] * ph.sin()) @ B)
        gs.append(g + direct)
    return torch.cat(fs), torch.cat(gs)


def _solve(f, g, pts, T=None):
    """Normals, distances and contact points from f and grad f."""
    N = g / g.norm(dim=1, keepdim=True)
    if T is not None:
        N = N @ T[:3, :3].T
    x = pts.double().clone()
    x[:, :3] += (EPS - f).clamp(min=0.0)[:, None] * N
    return {"pts": x, "n_sdf": torch.cat([N, f[:, None]], 1)}


def _collide64(net, blob, pts, T=None):
    p = pts[:, :3].double()
    if T is not None:
        T = T.double()
        inv = torch.linalg.inv(T)
        p = p @ inv[:3, :3].T + inv[:3, 3]
    return _solve(*_field(net, blob.double(), p), pts, T)


def _mesh64(V, F, P):
    """Distance to the closest triangle, negative where the winding number exceeds 1/2."""
    tri = V.double()[F.long()]                                         # [F, 3, 3]
    a, b, c = (tri[None, :, k] for k in range(3))
    out, step = [], max(1, (1 << 24) // F.shape[0])

    def dot(u, v):
        return u[..., 0] * v[..., 0] + u[..., 1] * v[..., 1] + u[..., 2] * v[..., 2]

    ab, bc, ca = b - a, c - b, a - c
    nrm = torch.linalg.cross(ab, -ca)
    nn = dot(nrm, nrm)
    lens = [dot(e, e) for e in (ab, bc, ca)]
    sides = [torch.linalg.cross(nrm, e) for e in (ab, bc, ca)]       # inward edge normals
    for q in P[:, :3].double().split(step):
        A, B, C = (q[:, None] - v for v in (a, b, c))
        best, inside = None, None
        for X, e, ee, side in zip((A, B, C), (ab, bc, ca), lens, sides):
            d = X - (dot(X, e) / ee).clamp(0.0, 1.0)[..., None] * e
            d2 = dot(d, d)
            best = d2 if best is None else torch.minimum(best, d2)
            ok = dot(X, side) >= 0
            inside = ok if inside is None else inside & ok
        best = torch.where(inside, torch.minimum(best, dot(A, nrm) ** 2 / nn), best)
        la, lb, lc = (dot(X, X).sqrt() for X in (A, B, C))
        num = -dot(A, torch.linalg.cross(B, C))
        den = la * lb * lc + dot(A, B) * lc + dot(A, C) * lb + dot(B, C) * la
        w = torch.atan2(num, den).sum(dim=1) / (2.0 * math.pi)
        d = best.min(dim=1).values.sqrt()
        out.append(torch.where(w > 0.5, -d, d))
    return torch.cat(out)


def _voxel64(grid, m, pts):
    p = pts[:, :3].double()
    h = 2.0 / (m - 1)
    q = p.clamp(-1.0, 1.0)
    u = (q + 1.0) / h
    c = u.floor().clamp(0, m - 2).long()
    t = u - c
    G = grid.double()
    v = {(i, j, k): G[(c[:, 0] + i) + m * ((c[:, 1] + j) + m * (c[:, 2] + k))]
         for i in (0, 1) for j in (0, 1) for k in (0, 1)}
    f = torch.zeros_like(t[:, 0])
    g = torch.zeros_like(p)
    for at, val in v.items():
        w = [t[:, a] if at[a] else 1.0 - t[:, a] for a in range(3)]
        f = f + w[0] * w[1] * w[2] * val
        for a in range(3):
            o = [w[x] for x in range(3) if x != a]
            g[:, a] += (1.0 if at[a] else -1.0) * o[0] * o[1] * val / h
    out = p - q
    g = torch.where(out != 0, torch.zeros_like(g), g)
    d = out.norm(dim=1)
    far = d > 0
    g = g + torch.where(far[:, None], out / d.clamp(min=1e-300)[:, None], torch.zeros_like(g))
    return _solve(f + d, g, pts)


def _cloth64(s, nx, ny):
    x, prev = s["x"].double().reshape(ny, nx, 4), s["prev"].double().reshape(ny, nx, 4)
    h = float(np.float32(s["h"]))
    dt2 = float(np.float32(1e-3)) ** 2
    acc = torch.zeros(ny, nx, 3, device="cuda", dtype=torch.float64)
    acc[..., 1] = -float(np.float32(9.81))
    for di in (-1, 0, 1):
        for dj in (-1, 0, 1):
            if di == 0 and dj == 0:
                continue
            r = h if di == 0 or dj == 0 else math.sqrt(2.0) * h
            i0, i1, j0, j1 = max(0, -di), ny - max(0, di), max(0, -dj), nx - max(0, dj)
            d = x[i0 + di:i1 + di, j0 + dj:j1 + dj, :3] - x[i0:i1, j0:j1, :3]
            n = d.norm(dim=-1, keepdim=True)
            acc[i0:i1, j0:j1] += torch.where(n > 0, 1e5 * (n - r) / n, torch.zeros_like(n)) * d
    out = x.clone()
    out[..., :3] = 2.0 * x[..., :3] - prev[..., :3] + dt2 * acc
    return out.reshape(-1, 4)


def exact(case, seed):
    kind = case["kind"]
    s = _inputs(case, seed)
    # a 16-bit ReLU network takes its slopes from 16-bit pre-activations, so its normals
    # (and weight gradients) are another function of the inputs than the 64-bit ones
    own_slopes = case.get("net") in ("dragon", "bunny") and case["precision"] != "fp32"
    if kind in ("collide", "query"):
        r = _collide64(case["net"], s["blob"], s["pts"], s["T"])
        n_sdf = None if own_slopes else r["n_sdf"]
        return {"n_sdf": n_sdf} if kind == "query" else {"pts": r["pts"], "n_sdf": n_sdf, "hit": None}
    if kind == "grouped":
        parts = []
        for k, (o, c) in enumerate(zip(s["offsets"].tolist(), s["counts"].tolist())):
            T = None if s["T"] is None else s["T"][k]
            parts.append(_collide64(case["net"], s["blobs"][k], s["pts"][o:o + c], T))
        return {key: torch.cat([r[key] for r in parts]) for key in ("pts", "n_sdf")}
    if kind in ("fit_l1", "fit_eikonal"):
        blob = s["blob"].double().requires_grad_(True)
        n, total = case["n"], 0.0
        fs, gs = [], []
        for p, d in zip(s["pts"][:, :3].double().split(32768), s["d"].double().split(32768)):
            if kind == "fit_l1":
                f, _ = _forward_only(case["net"], blob, p)
                loss = (f - d).abs().sum() / n
            else:
                f, g = _field(case["net"], blob, p)
                loss = ((f - d).abs().sum() + 0.1 * ((g.norm(dim=1) - 1.0) ** 2).sum()) / n
                fs.append(f.detach())
                gs.append(g.detach())
            loss.backward()
            total = total + loss.detach()
        if kind == "fit_l1":
            grad = blob.grad.clone()
            grad[:3 * NETS[case["net"]][3]] = 0.0     # the frequencies are not trained
            return {"grad": None if own_slopes else grad, "loss": total.reshape(1)}
        return {"loss": total, "f": torch.cat(fs), "g": torch.cat(gs), "grad": blob.grad}
    if kind == "penalty":
        f, g = _field(case["net"], s["blob"].double(), s["pts"][:, :3].double())
        force = torch.zeros(case["n"], 4, device="cuda", dtype=torch.float64)
        force[:, :3] = -2.0 * (EPS - f).clamp(min=0.0)[:, None] * g
        return {"force": force}
    if kind == "mesh":
        return {"sdf": _mesh64(s["V"], s["F"], s["pts"])}
    if kind == "voxel":
        return {**_voxel64(s["grid"], case["nodes"], s["pts"]), "hit": None}
    return {"x_new": _cloth64(s, case["nx"], case["ny"])}


def _forward_only(net, blob, p):
    """f at p with a graph to the blob (first-order losses)."""
    skip = NETS[net][2]
    B, layers = _unpack(net, blob)
    x = p
    if B is not None:
        ph = 2.0 * math.pi * (p @ B.detach().T)
        x = torch.cat([ph.sin(), ph.cos()], 1)
    for l, (W, b) in enumerate(layers[:-1]):
        if l == skip:
            x = torch.cat([x, p], 1) / math.sqrt(2.0)
        z = x @ W.T + b
        x = z.clamp(min=0.0)
        if B is None:
            x = x + torch.log1p(torch.exp(-BETA * z.abs())) / BETA
    W, b = layers[-1]
    return (x @ W.T + b)[:, 0], None
