"""What a user of this package has it do, as cases that can be timed and compared.

A case is a dict of plain values.  ``prepare`` makes what a program has in hand before the call (SDB objects, calibrated
where the precision asks for it, point sets, output buffers of a batch), ``run`` makes one pass through the public entry
points, ``work`` says what that pass cannot do without and ``exact`` gives its values in 64 bits from plain torch.

Kinds:

* ``mesh``     one SDB polygonized into an indexed mesh (``gh.polygonize(..., indexed=True)``), optionally with the vertex
               normals that a viewer computes from it;
* ``batch``    several SDBs, analytic and neural, polygonized together (``gh.Batch``);
* ``query``    f at a list of points (``gh.eval_points``);
* ``adjoint``  the parameter gradient of a loss on surface points (``gh.backward``);
* ``train``    a differentiable polygonization, a loss on its mesh and the gradient (``autograd.polygonize_*``).

A mesh goes into buffers that the program keeps (``gh.Buffers``), larger than the mesh and zero beyond it.  Its triangles
come in no particular order (the vertices do): ``mesh`` and ``batch`` return the vertices and the counts of triangles,
surface cells and vertices; the triangles themselves go into the normals and into the area term of the training losses.
"""
import math

import numpy as np
import torch

from paper_2111_05778_gb300 import autograd, gh, synth

LO, HI = -1.0, 1.0
FORM_RADIAL = {"r0": synth.MLP_R0, "alpha": synth.MLP_ALPHA, "beta": synth.MLP_BETA, "radial": True, "lam": 1.0}
FORM_PLAIN = {"r0": 0.0, "alpha": 1.0, "beta": 1.0, "radial": False, "lam": synth.PAPER_LAMBDA}


def listed():
    return [
        # the smallest mesh: one sphere at preview resolution, where launches and latency count
        {"name": "mesh_sphere_64", "kind": "mesh", "sdb": "sphere", "N": 64, "lo": LO, "hi": HI, "precision": "fp32",
         "normals": False},
        # one of each primitive on an odd grid and an offset domain, shaded by a viewer
        {"name": "mesh_prims_201", "kind": "mesh", "sdb": "prims", "N": 201, "lo": -1.0, "hi": 1.1, "precision": "fp32",
         "normals": True},
        # the analytic workload of the benchmark: 36 primitives at N = 512
        {"name": "mesh_csg_512", "kind": "mesh", "sdb": "csg", "N": 512, "lo": LO, "hi": HI, "precision": "fp32",
         "normals": False},
        # a neural SDB with the default precision
        {"name": "mesh_mlp256_fp32_192", "kind": "mesh", "sdb": "mlp", "width": 256, "N": 192, "lo": LO, "hi": HI,
         "precision": "fp32", "normals": False},
        # tensor-core hopping with FP32 refinement, a narrower network on an odd grid
        {"name": "mesh_mlp128_bf16_385", "kind": "mesh", "sdb": "mlp", "width": 128, "N": 385, "lo": LO, "hi": HI,
         "precision": "bf16", "normals": False},
        # the headline workload of the benchmark: width 256 at N = 1024, split-BF16 refinement
        {"name": "mesh_mlp256_bf16x6_1024", "kind": "mesh", "sdb": "mlp", "width": 256, "N": 1024, "lo": LO, "hi": HI,
         "precision": "bf16x6", "normals": False},
        # a service that polygonizes mixed requests together (as the benchmark's batch, smaller)
        {"name": "batch_mixed_8", "kind": "batch", "items": 8, "max_N": 512, "precision": "bf16x6"},
        # a few distance queries to a network of the paper's form: collision checks, picking
        {"name": "query_paper64_777", "kind": "query", "sdb": "mlp", "width": 64, "mid": synth.PAPER_NMID,
         "form": "plain", "n": 777, "precision": "fp32"},
        # distance values for a large point set
        {"name": "query_mlp256_1m", "kind": "query", "sdb": "mlp", "width": 256, "mid": synth.MLP_NMID,
         "form": "radial", "n": (1 << 20) + 77, "precision": "fp32"},
        # the gradient of a vertex loss at the benchmark's size (the vertices of an N = 256 mesh)
        {"name": "adjoint_mlp256_111k", "kind": "adjoint", "width": 256, "mid": synth.MLP_NMID, "form": "radial",
         "V": 111146},
        # fitting an analytic scene: mesh, loss, gradient of centres and sizes
        {"name": "train_csg_128", "kind": "train", "sdb": "csg", "N": 128},
        # fitting a network: new weights, mesh, loss, gradient of the weights
        {"name": "train_mlp128_96", "kind": "train", "sdb": "mlp", "width": 128, "N": 96},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


# the largest grid a drawn neural mesh takes, by precision and width: none costs more than the headline case
_MAX_N = {("fp32", 64): 420, ("fp32", 128): 300, ("fp32", 256): 192, ("bf16", 64): 640, ("bf16", 128): 512,
          ("bf16", 256): 512, ("bf16x6", 64): 1000, ("bf16x6", 128): 900, ("bf16x6", 256): 800}


def draw(rng):
    kind = rng.choice(["mesh", "mesh", "mesh", "mesh", "batch", "query", "query", "adjoint", "train"])
    width = rng.choice([64, 128, 256])
    if kind == "mesh":
        lo = round(rng.uniform(-1.15, -1.0), 3)
        hi = round(rng.uniform(1.0, 1.15), 3)
        c = {"kind": "mesh", "lo": lo, "hi": hi, "normals": rng.random() < 0.25}
        if rng.random() < 0.5:
            c.update(sdb=rng.choice(["sphere", "prims", "csg", "csg"]), precision="fp32", N=_log(rng, 40, 600))
        else:
            prec = rng.choice(["fp32", "bf16", "bf16x6"])
            c.update(sdb="mlp", width=width, precision=prec, N=_log(rng, 40, _MAX_N[prec, width]))
        return c
    if kind == "batch":
        return {"kind": "batch", "items": rng.randint(2, 8), "max_N": _log(rng, 96, 512),
                "precision": rng.choice(["bf16", "bf16x6"])}
    if kind == "query":
        if rng.random() < 0.25:
            return {"kind": "query", "sdb": "csg", "n": _log(rng, 1, 1 << 22), "precision": "fp32"}
        form = rng.choice(["radial", "plain"])
        return {"kind": "query", "sdb": "mlp", "width": width, "mid": rng.randint(3, 7), "form": form,
                "n": _log(rng, 1, 1 << 20), "precision": rng.choice(["fp32", "fp32", "bf16", "bf16x6"])}
    if kind == "adjoint":
        return {"kind": "adjoint", "width": width, "mid": rng.randint(3, 7), "form": rng.choice(["radial", "plain"]),
                "V": _log(rng, 200, 200000)}
    if rng.random() < 0.5:
        return {"kind": "train", "sdb": "csg", "N": _log(rng, 48, 256)}
    return {"kind": "train", "sdb": "mlp", "width": width, "N": _log(rng, 40, 128)}


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _prims(case, seed):
    if case["sdb"] == "sphere":
        rng = np.random.default_rng(seed)
        return synth.sphere_prims(rng.uniform(0.45, 0.55), rng.uniform(-0.05, 0.05, 3))
    return synth.primitive_scene(seed) if case["sdb"] == "prims" else synth.csg_prims(seed)


def _params(case, seed):
    return synth.mlp_params(seed, case["width"], case.get("mid", synth.MLP_NMID))


def _form(case):
    return FORM_PLAIN if case.get("form") == "plain" else FORM_RADIAL


def _layers64(case, params):
    return [(torch.from_numpy(W).cuda().double(), torch.from_numpy(b).cuda().double())
            for W, b in synth.unpack_layers(params, case["width"], case.get("mid", synth.MLP_NMID))]


def _net(layers, p):
    a = p
    for W, b in layers[:-1]:
        a = torch.relu(torch.addmm(b, a, W.t()))
    W, b = layers[-1]
    return (a @ W.t() + b)[:, 0]


def _f_mlp(layers, form, p):
    r = p.square().sum(1).sqrt() if form["radial"] else 0.0
    return (form["alpha"] * _net(layers, p) + r - form["r0"]) / form["beta"] / form["lam"]


def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _surface_points(case, seed):
    """Points next to the zero set (radial form: |p| = 0.6 - 0.1 g(p), a contraction), and a loss gradient there."""
    g = _generator(seed)
    u = torch.randn(case["V"], 3, device="cuda", generator=g)
    u = u / u.norm(dim=1, keepdim=True)
    r = torch.full((case["V"], 1), synth.MLP_R0, device="cuda")
    if _form(case)["radial"]:
        layers = [(W.float(), b.float()) for W, b in _layers64(case, _params(case, seed))]
        for _ in range(4):
            r = synth.MLP_R0 - synth.MLP_ALPHA * _net(layers, u * r)[:, None]
    v = (u * r).contiguous()
    d = v - torch.tensor([0.02, -0.03, 0.01], device="cuda")
    n = d.norm(dim=1, keepdim=True)
    return v, (2.0 / case["V"] * (n - 0.55) * d / n).contiguous()


# room for triangles per N^2 (twice what a typical seed has)
_ROOM = {"sphere": 5, "prims": 5, "mlp": 7, "csg": 14}


def _buffers(sdb, N):
    cap = _ROOM[sdb] * N * N + 4096
    bufs = gh.Buffers(cap, cap_verts=cap // 2)
    bufs.verts.zero_()
    return bufs


def _batch_spec(case, seed):
    """(kind, seed, N, width) of each item: analytic and neural in turn, N spread over [max_N / 8, max_N]."""
    rng = np.random.default_rng(case["items"] + case["max_N"])
    spec = []
    for b in range(case["items"]):
        N = max(32, int(case["max_N"] * 2.0 ** (-3.0 * rng.random())))
        spec.append(("csg" if b % 2 == 0 else "mlp", 100 * seed + b, N if b else case["max_N"],
                     int(rng.choice(synth.BATCH_WIDTHS))))
    return spec


def prepare(case, seed):
    seed = int(seed) % 100000
    kind = case["kind"]
    if kind == "mesh":
        if case["sdb"] != "mlp":
            sdb = gh.CsgSdb(_prims(case, seed))
        else:
            sdb = gh.MlpSdb(_params(case, seed), case["width"])
            if case["precision"] != "fp32":
                sdb.calibrate(case["N"], case["lo"], case["hi"])
        return {"case": case, "sdb": sdb, "bufs": _buffers(case["sdb"], case["N"])}
    if kind == "batch":
        sdbs, Ns = [], []
        for k, s, N, width in _batch_spec(case, seed):
            if k == "csg":
                sdbs.append(gh.CsgSdb(synth.csg_prims(s)))
            else:
                sdbs.append(gh.MlpSdb(synth.mlp_params(s, width), width))
                sdbs[-1].calibrate(N)
            Ns.append(N)
        batch = gh.Batch(sdbs, Ns, [14 * n * n + 4096 for n in Ns], precision=case["precision"], indexed=True)
        for b in batch.bufs:
            b.verts.zero_()
        return {"case": case, "batch": batch}
    if kind == "query":
        if case["sdb"] == "csg":
            sdb = gh.CsgSdb(_prims(case, seed))
        else:
            sdb = gh.MlpSdb(_params(case, seed), case["width"], case["mid"], **_form(case))
        return {"case": case, "sdb": sdb, "points": _query_points(case, seed)}
    if kind == "adjoint":
        v, dl = _surface_points(case, seed)
        return {"case": case, "sdb": gh.MlpSdb(_params(case, seed), case["width"], case["mid"], **_form(case)),
                "v": v, "dl": dl}
    if case["sdb"] == "csg":
        p = torch.from_numpy(synth.csg_prims(seed)).cuda()
    else:
        p = torch.from_numpy(_params(case, seed)).cuda()
    return {"case": case, "params": p.requires_grad_(True)}


def _query_points(case, seed):
    return torch.rand(case["n"], 3, device="cuda", generator=_generator(seed)) * 2.0 - 1.0


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def _normals(verts, faces):
    """Area-weighted vertex normals, as a viewer computes them."""
    f = faces.long()
    a, b, c = verts[f[:, 0]], verts[f[:, 1]], verts[f[:, 2]]
    n = torch.cross(b - a, c - a, dim=1)
    out = torch.zeros_like(verts)
    return out.index_add_(0, f.reshape(-1), n.repeat_interleave(3, 0))


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "mesh":
        b = state["bufs"]
        gh.polygonize_into(state["sdb"], case["N"], b, case["lo"], case["hi"], case["precision"])
        out = {"verts": b.verts, "counts": b.counts}
        if case["normals"]:
            out["normals"] = _normals(b.verts, b.faces[:int(b.counts[0])])
        return out
    if kind == "batch":
        state["batch"].run()
        return [{"verts": b.verts, "counts": b.counts} for b in state["batch"].bufs]
    if kind == "query":
        return gh.eval_points(state["sdb"], state["points"], case["precision"])
    if kind == "adjoint":
        return gh.backward(state["sdb"], state["v"], state["dl"])
    p = state["params"]
    if case["sdb"] == "csg":
        v, f = autograd.polygonize_csg(p, case["N"])
    else:
        v, f = autograd.polygonize_mlp(p, case["width"], N=case["N"])
    # pull the vertices towards a sphere and keep the area small
    a, b, c = v[f[:, 0]], v[f[:, 1]], v[f[:, 2]]
    area = torch.cross(b - a, c - a, dim=1).norm(dim=1).sum()
    loss = (v.norm(dim=1) - 0.55).square().mean() + 0.01 * area
    (grad,) = torch.autograd.grad(loss, p)
    return {"loss": loss.detach(), "grad": grad}


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
# evaluations of the rays per N^2 log2 N, crossing edges' end points per N^2, triangles per N^2 (one sphere of radius
# 0.5-0.6 in the cube; the CSG scene has about 1.7 times its area, the seven primitives about half)
_SHAPE = {"sphere": (1.5, 1.8, 2.4), "mlp": (1.9, 2.0, 3.4), "csg": (2.7, 3.5, 5.7), "prims": (1.9, 1.4, 1.7)}
_FLOP_PRIMS = {"sphere": 9, "prims": 150, "csg": 650}


def _flop_mlp(width, mid):
    return 2 * (3 * width + mid * width * width + width)


def _mesh_work(sdb, N, flop, param_bytes):
    hops, ends, tris = _SHAPE[sdb]
    evals = hops * N * N * math.log2(N) + ends * N * N
    t = tris * N * N
    # the soup with its edge keys, the faces, the vertices (half as many as triangles)
    return {"bytes": t * (36 + 24 + 12 + 6) + param_bytes, "flops": evals * flop}


def work(case):
    kind = case["kind"]
    if kind == "mesh" or kind == "train":
        if case["sdb"] == "mlp":
            n = synth.mlp_param_count(case["width"])
            w = _mesh_work("mlp", case["N"], _flop_mlp(case["width"], synth.MLP_NMID), 4 * n)
        else:
            w = _mesh_work(case["sdb"], case["N"], _FLOP_PRIMS[case["sdb"]], 80 * 36)
        if kind == "train":
            verts = 0.5 * _SHAPE[case["sdb"]][2] * case["N"] ** 2
            w["flops"] += verts * (3 * _flop_mlp(case["width"], synth.MLP_NMID) if case["sdb"] == "mlp" else 650)
            w["bytes"] += 12 * verts
        return w
    if kind == "batch":
        total = {"bytes": 0.0, "flops": 0.0}
        for k, _, N, width in _batch_spec(case, 0):
            w = _mesh_work(k, N, _flop_mlp(width, synth.MLP_NMID) if k == "mlp" else 650, 0)
            total = {q: total[q] + w[q] for q in total}
        return total
    if kind == "query":
        if case["sdb"] == "csg":
            return {"bytes": 16.0 * case["n"] + 80 * 36, "flops": 650.0 * case["n"]}
        return {"bytes": 16.0 * case["n"] + 4 * synth.mlp_param_count(case["width"], case["mid"]),
                "flops": float(case["n"]) * _flop_mlp(case["width"], case["mid"])}
    return {"bytes": 24.0 * case["V"] + 8 * synth.mlp_param_count(case["width"], case["mid"]),
            "flops": 3.0 * case["V"] * _flop_mlp(case["width"], case["mid"])}


# ---------------------------------------------------------------------------
# the same values in 64 bits
# ---------------------------------------------------------------------------
def _prim64(row, p):
    """Exact distances of the seven primitives (rows as in synth), float64."""
    kind, par = int(row[0]), [float(x) for x in row[5:8]]
    q = (p - torch.tensor(row[2:5], device=p.device)) @ torch.tensor(row[8:17].reshape(3, 3), device=p.device).t()
    x, y, z = q[:, 0], q[:, 1], q[:, 2]
    if kind == synth.SPHERE:
        return q.square().sum(1).sqrt() - par[0]
    rho = (x * x + z * z).sqrt()
    if kind == synth.TORUS:
        return ((rho - par[0]).square() + y * y).sqrt() - par[1]
    if kind == synth.BOX:
        e = q.abs() - torch.tensor(par, device=p.device, dtype=p.dtype)
        return e.clamp(min=0).square().sum(1).sqrt() + e.max(1).values.clamp(max=0)
    if kind == synth.CAPSULE:
        return (x * x + (y - y.clamp(-par[0], par[0])).square() + z * z).sqrt() - par[1]
    if kind == synth.CONE:
        R, H = par[0], par[1]
        db = ((rho - rho.clamp(max=R)).square() + (y + H).square()).sqrt()
        t = (((rho - R) * -R + (y + H) * 2 * H) / (R * R + 4 * H * H)).clamp(0, 1)
        ds = ((rho - (R - t * R)).square() + (y - (2 * H * t - H)).square()).sqrt()
        inside = (y > -H) & (y < H) & (rho * 2 * H < R * (H - y))
        d = torch.minimum(db, ds)
        return torch.where(inside, -d, d)
    if kind == synth.CYLINDER:
        e0 = rho - par[0]
    else:  # hexagonal prism: fold into one wedge
        x, z, a = x.abs(), z.abs(), par[0]
        s3 = math.sqrt(3.0)
        d = (-0.5 * x + 0.5 * s3 * z).clamp(min=0)
        x, z = x + d, z - s3 * d
        n = ((x - a).square() + (z - z.clamp(-a / s3, a / s3)).square()).sqrt()
        e0 = torch.where(x < a, -n, n)
    e1 = y.abs() - par[1]
    return (e0.clamp(min=0).square() + e1.clamp(min=0).square()).sqrt() + torch.maximum(e0, e1).clamp(max=0)


def _f_prims(rows, p):
    f = _prim64(rows[0], p)
    for row in rows[1:]:
        d = _prim64(row, p)
        f = torch.minimum(f, d) if row[1] == synth.UNION else torch.maximum(f, -d if row[1] == synth.SUBTRACT else d)
    return f


def _in_chunks(f, p, chunk=1 << 20):
    return torch.cat([f(p[i:i + chunk]) for i in range(0, p.shape[0], chunk)])


def _verts64(f, N, lo, hi, near=None):
    """The zero crossings of f on the lattice edges, by lower end point (a, b, c), then axis; `near`: where f has to be
    evaluated at all, from |p| (elsewhere its sign is that of |p| - 0.6 and no edge crosses)."""
    lo, hi = float(np.float32(lo)), float(np.float32(hi))
    h = float(np.float32((hi - lo) / N))
    t = lo + h * torch.arange(N + 1, device="cuda", dtype=torch.float64)
    val = torch.empty(N + 1, N + 1, N + 1, device="cuda", dtype=torch.float64)
    step = max(1, (1 << 22) // (N + 1) ** 2)
    for a in range(0, N + 1, step):
        p = torch.stack(torch.meshgrid(t[a:a + step], t, t, indexing="ij"), -1).reshape(-1, 3)
        if near is None:
            v = _in_chunks(f, p)
        else:
            r = p.square().sum(1).sqrt()
            v = r - synth.MLP_R0
            at = ((r > near[0]) & (r < near[1])).nonzero()[:, 0]
            if at.numel():
                v[at] = _in_chunks(f, p[at])
        val[a:a + step] = v.reshape(-1, N + 1, N + 1)
    found = []
    for ax in range(3):
        m = N  # edges along ax: lower ends 0 .. N - 1
        A, B = val.narrow(ax, 0, m), val.narrow(ax, 1, m)
        at = ((A < 0) != (B < 0)).nonzero()
        fa, fb = A[at[:, 0], at[:, 1], at[:, 2]], B[at[:, 0], at[:, 1], at[:, 2]]
        pos = lo + h * at.double()
        pos[:, ax] += h * fa / (fa - fb)
        key = ((at[:, 0] * (N + 1) + at[:, 1]) * (N + 1) + at[:, 2]) * 3 + ax
        found.append((key, pos))
    key, pos = torch.cat([k for k, _ in found]), torch.cat([q for _, q in found])
    return pos[key.argsort()]


def _padded(v, rows):
    return torch.cat([v, torch.zeros(rows - v.shape[0], 3, device=v.device, dtype=v.dtype)])


def _verts_of(sdb, case, seed, N, lo, hi):
    if sdb == "mlp":
        layers = _layers64(case, _params(case, seed))
        g0 = float(_net(layers, torch.zeros(1, 3, device="cuda", dtype=torch.float64)).abs())
        # |g(p)| <= |p| + |g(0)| (a 1-Lipschitz network): the zeros of |p| - r0 + alpha g lie in this shell
        s = synth.MLP_ALPHA
        near = ((synth.MLP_R0 - s * g0) / (1 + s) - 0.01, (synth.MLP_R0 + s * g0) / (1 - s) + 0.01)
        h = (hi - lo) / N
        near = (near[0] - 2 * h, near[1] + 2 * h)
        return _verts64(lambda p: _f_mlp(layers, FORM_RADIAL, p), N, lo, hi, near)
    rows = _prims(case, seed) if sdb != "csg" else synth.csg_prims(seed)
    return _verts64(lambda p: _f_prims(rows, p), N, lo, hi)


def exact(case, seed):
    seed = int(seed) % 100000
    kind = case["kind"]
    if kind == "mesh":
        if case["N"] > 520:
            return None
        v = _verts_of(case["sdb"], case, seed, case["N"], case["lo"], case["hi"])
        out = {"verts": _padded(v, (_ROOM[case["sdb"]] * case["N"] ** 2 + 4096) // 2), "counts": None}
        return dict(out, normals=None) if case["normals"] else out
    if kind == "batch":
        out = []
        for k, s, N, width in _batch_spec(case, seed):
            v = None
            if N <= 320:
                v = _padded(_verts_of(k, {"width": width}, s, N, LO, HI), (14 * N * N + 4096) // 2 + 4096)
            out.append({"verts": v, "counts": None})
        return out
    if kind == "query":
        p = _query_points(case, seed).double()
        if case["sdb"] == "csg":
            rows = synth.csg_prims(seed)
            return _in_chunks(lambda q: _f_prims(rows, q), p)
        layers, form = _layers64(case, _params(case, seed)), _form(case)
        return _in_chunks(lambda q: _f_mlp(layers, form, q), p, 1 << 17)
    if kind == "adjoint":
        return _adjoint64(case, seed)
    return None


def _adjoint64(case, seed):
    v, dl = (x.double() for x in _surface_points(case, seed))
    layers, form = _layers64(case, _params(case, seed)), _form(case)
    flat = [t.requires_grad_(True) for layer in layers for t in layer]
    total = [torch.zeros_like(t) for t in flat]
    for i in range(0, case["V"], 1 << 15):
        p = v[i:i + (1 << 15)].requires_grad_(True)
        f = _f_mlp(layers, form, p)
        (gx,) = torch.autograd.grad(f.sum(), p, retain_graph=True)
        s = -(dl[i:i + (1 << 15)] * gx).sum(1) / gx.square().sum(1)
        for t, g in zip(total, torch.autograd.grad((s.detach() * f).sum(), flat)):
            t += g
    return torch.cat([t.reshape(-1) for t in total])
