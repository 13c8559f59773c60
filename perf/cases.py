"""Performance cases of the skeletal-animation library.

Every case is work that a program using the library has it do, through the
public entry points of `paper_2505_06703_gb300.anim`: the fused frame (plain,
layered, skinned, from and to host memory), the forward from local poses, the
raster of the crowd, the adjoint (as a loss and through autograd) and the IK
step, from a handful of characters to the benchmark's crowds.  Skeletons,
clips, poses and meshes are synthetic, drawn from the seed alone: trees of
the shapes this repository's benchmark uses, rest rotations within 30 degrees
of identity, translations scaled to unit extent, keys at 30 Hz.

A case's "schedule" is the five values of Context.get_schedule that a program
has kept from an earlier autotuning run on this GPU and re-applies with
set_schedule ("" for a program that never tuned and runs on the defaults).

exact() restates each operation in plain torch float64, level by level down
the tree, without the library.
"""
import math

import numpy as np
import torch

import paper_2505_06703_gb300 as anim

RATE_HZ = 30.0
MIX_SIZES = ((32, 8), (128, 16), (512, 70), (1024, 256), (2048, 2048))
MIX_FRACTIONS = (0.40, 0.30, 0.15, 0.10, 0.05)
IK_EFFECTORS = 8
ADAM = {"lr": 1e-2, "betas": (0.9, 0.999), "eps": 1e-8}


# ------------------------------------------------------------------- cases
def listed():
    return [
        # the smallest batch of the benchmark: one party of characters whose local poses come from
        # elsewhere (physics, a network), skin matrices out; launch latency is most of it
        {"name": "forward_party", "kind": "forward", "skeleton": "tree", "chars": 64, "joints": 64, "depth": 12,
         "schedule": ""},
        # a squad on screen of a game that never tunes: few characters, an odd joint count, one frame
        {"name": "frame_squad", "kind": "frame", "skeleton": "tree", "chars": 37, "joints": 67, "depth": 14,
         "keys": 45, "clips": 2, "schedule": ""},
        # the headline frame: 4,096 bipeds with cloth and tail chains and one 1,024-joint dragon
        {"name": "frame_crowd", "kind": "frame", "skeleton": "biped", "chars": 4096, "dragons": 1, "keys": 30,
         "clips": 2, "schedule": "16 1 4096 2 0"},
        # a crowd of five skeleton types from 32 to 2,048 joints in one frame
        {"name": "frame_mixed", "kind": "frame", "skeleton": "mixed", "chars": 10000, "keys": 30, "clips": 2,
         "schedule": "32 2 4096 2 0"},
        # the headline crowd with four clips blended by per-character weights and an additive layer
        {"name": "frame_layers", "kind": "layers", "skeleton": "biped", "chars": 4096, "dragons": 1, "keys": 30,
         "clips": 4, "schedule": "16 3 4096 1 0"},
        # the headline crowd skinned for rendering: vertices out, the skin matrices stay on the chip
        {"name": "frame_skinned", "kind": "skinned", "skeleton": "biped", "chars": 4096, "dragons": 1, "keys": 30,
         "clips": 2, "verts": 1500, "schedule": "16 2 4096 1 0"},
        # the picture of that crowd at full HD: object ids (picking) and shaded colours
        {"name": "crowd_picture", "kind": "raster", "chars": 4097, "verts": 1500, "width": 1920, "height": 1080,
         "cols": 64, "scale": 11.0},
        # the paper's experiment: 10,000 characters of a 300-joint tree from given local poses
        {"name": "forward_crowd", "kind": "forward", "skeleton": "tree", "chars": 10000, "joints": 300, "depth": 60,
         "schedule": "32 3 4096 1 0"},
        # pose fitting by gradients: loss and its gradients for 1,024 characters of a 256-joint tree
        {"name": "loss_fit", "kind": "loss", "skeleton": "tree", "chars": 1024, "joints": 256, "depth": 96,
         "schedule": "16 3 2048 0 7"},
        # a network's layer: joint positions of ragged skeletons and their gradients through autograd, never tuned
        {"name": "autograd_ragged", "kind": "autograd", "skeleton": "ragged", "chars": 2001, "joints": 341,
         "depth": 57, "schedule": ""},
        # inverse kinematics in progress, the program keeping Adam's moments: 128- and 1,024-joint characters
        {"name": "ik_fit", "kind": "ik", "skeleton": "ik", "chars": 8192, "steps": 2, "schedule": "16 3 2048 1 0"},
        # the headline frame for a program whose inputs and outputs live in host memory
        {"name": "frame_host", "kind": "host", "skeleton": "biped", "chars": 4096, "dragons": 1, "keys": 30,
         "clips": 2, "schedule": "16 1 4096 2 0"},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["frame", "frame", "layers", "skinned", "raster", "forward", "forward", "loss", "autograd", "ik",
                       "host"])
    if kind == "raster":
        w, h = rng.choice([(640, 360), (1280, 720), (1920, 1080), (997, 641)])
        cols = rng.randint(5, 64)
        return {"kind": kind, "chars": _log_int(rng, 24, 4000), "verts": rng.randint(300, 1500), "width": w, "height": h,
                "cols": cols, "scale": round(w / (2.7 * cols), 2)}
    c = {"kind": kind}
    most = {"frame": 2_000_000, "layers": 2_000_000, "skinned": 1_500_000, "forward": 2_500_000, "loss": 2_000_000,
            "autograd": 900_000, "ik": 3_000_000, "host": 1_500_000}[kind]
    total = _log_int(rng, 3000, most)
    skeletons = {"frame": ["tree", "tree", "biped", "mixed", "ragged"], "layers": ["tree", "biped", "ragged"],
                 "skinned": ["tree", "biped"], "forward": ["tree", "tree", "biped", "mixed"], "loss": ["tree", "ragged"],
                 "autograd": ["tree", "ragged"], "ik": ["ik"], "host": ["biped", "mixed"]}[kind]
    s = c["skeleton"] = rng.choice(skeletons)
    if s in ("tree", "ragged"):
        c["joints"] = _log_int(rng, 21, 700)
        c["depth"] = min(rng.randint(8, 120), c["joints"] - 4)
    mean = {"tree": c.get("joints", 0), "ragged": 0.6 * c.get("joints", 0), "biped": 512, "mixed": 333, "ik": 576}[s]
    c["chars"] = max(5, min(20000, int(total / mean)))
    if s == "biped":
        c["dragons"] = rng.randint(0, 2)
    if kind in ("frame", "layers", "skinned", "host"):
        c["keys"] = rng.choice([2, 17, 30, 30, 47, 90])
        c["clips"] = rng.randint(2, 4) if kind == "layers" else rng.choice([1, 2, 2])
    if kind == "skinned":
        c["verts"] = rng.randint(200, 1500)
    if kind == "ik":
        c["steps"] = rng.randint(1, 3)
    tuned = {"frame": "16 2 2048 2 0", "layers": "16 3 4096 1 0", "skinned": "16 2 4096 1 0", "forward": "32 3 4096 1 0",
             "loss": "16 3 2048 0 7", "autograd": "16 3 2048 0 7", "ik": "16 3 2048 1 0", "host": "16 2 2048 2 0"}
    c["schedule"] = tuned[kind] if rng.random() < 0.5 else ""
    return c


# --------------------------------------------------------------- skeletons
def _random_tree(n, depth, rng):
    """Joints 0..depth-1 form a spine, every other joint picks a parent among the earlier joints above the
    depth limit; renumbered in depth-first order with the children shuffled, as exporters number them."""
    par = [-1] * n
    dep = [1] * n
    cand = [0] if depth > 1 else []
    for i in range(1, n):
        p = i - 1 if i < depth else cand[int(rng.integers(len(cand)))]
        par[i] = p
        dep[i] = dep[p] + 1
        if dep[i] < depth:
            cand.append(i)
    return _relabel(par, rng)


def _relabel(par, rng):
    n = len(par)
    kids = [[] for _ in range(n)]
    for i in range(1, n):
        kids[par[i]].append(i)
    order, stack = [], [0]
    while stack:
        u = stack.pop()
        order.append(u)
        ch = kids[u]
        stack.extend(ch[int(k)] for k in rng.permutation(len(ch)))
    new = {o: k for k, o in enumerate(order)}
    return np.array([-1 if par[o] < 0 else new[par[o]] for o in order], np.int32)


def _biped(rng):
    """A 40-joint body of depth 11 with 8 cloth and tail chains of 59 joints, one at the deepest body joint."""
    par = [-1] + [i - 1 if i < 11 else -2 for i in range(1, 40)]
    dep = list(range(1, 12)) + [0] * 29
    for i in range(11, 40):
        p = int(rng.choice([j for j in range(i) if dep[j] < 11]))
        par[i], dep[i] = p, dep[p] + 1
    for a in [10] + [int(x) for x in rng.choice([j for j in range(40) if j != 10], 7, replace=False)]:
        par.append(a)
        for _ in range(58):
            par.append(len(par) - 1)
    return _relabel(par, rng)


def _parents(case, rng):
    """(parent arrays of the case's types, type of each character)"""
    s, n_chars = case["skeleton"], case["chars"]
    if s == "tree":
        return [_random_tree(case["joints"], case["depth"], rng)], np.zeros(n_chars, np.int32)
    if s == "ragged":
        n, d = case["joints"], case["depth"]
        sizes = [(n, d), (n * 5 // 8 + 1, max(2, d * 5 // 8)), (n // 4 + 3, max(2, d // 4))]
        return [_random_tree(k, min(e, k), rng) for k, e in sizes], rng.permutation(np.arange(n_chars, dtype=np.int32) % 3)
    if s == "biped":
        dragons = case.get("dragons", 0)
        types = [_biped(rng)] + ([np.arange(-1, 1023, dtype=np.int32)] if dragons else [])
        return types, np.array([0] * n_chars + [1] * dragons, np.int32)
    if s == "mixed":
        types = [np.arange(-1, n - 1, dtype=np.int32) if n == d else _biped(rng) if n == 512 else _random_tree(n, d, rng)
                 for n, d in MIX_SIZES]
        ct = np.repeat(np.arange(5, dtype=np.int32), [int(round(f * n_chars)) for f in MIX_FRACTIONS])[:n_chars]
        ct = np.concatenate([ct, np.zeros(n_chars - len(ct), np.int32)])
        return types, rng.permutation(ct)
    types = [_random_tree(128, 16, rng), _random_tree(1024, 256, rng)]  # the IK mix
    return types, (np.arange(n_chars) % 2).astype(np.int32)


def _quats(rng, shape, degrees):
    axis = rng.normal(size=(*shape, 3))
    axis /= np.linalg.norm(axis, axis=-1, keepdims=True)
    half = np.deg2rad(rng.uniform(0.0, degrees, size=shape))[..., None] / 2
    return np.concatenate([axis * np.sin(half), np.cos(half)], axis=-1)


def _type(par, case, rng):
    """Rest pose and, where the case samples clips, the clips (and an additive layer), of unit extent: the
    longest root-to-joint path is at most 1 in every key."""
    n = len(par)
    rest_q, rest_t = _quats(rng, (n,), 30.0), rng.uniform(-0.1, 0.1, size=(n, 3))
    length = np.linalg.norm(rest_t, axis=1)
    keys = add = None
    if "keys" in case:
        shape = (case["clips"], case["keys"], n)
        keys = np.zeros((*shape, 8))
        keys[..., :4] = _quats(rng, shape, 30.0)
        keys[..., 4:7] = rest_t + rng.uniform(-0.01, 0.01, size=(*shape, 3))
        length = np.maximum(length, np.linalg.norm(keys[..., 4:7], axis=-1).max(axis=(0, 1)))
        if case["kind"] == "layers":
            add = np.zeros((*shape[1:], 8))
            add[..., :4] = _quats(rng, shape[1:], 15.0)
            add[..., 4:7] = rng.uniform(-0.005, 0.005, size=(*shape[1:], 3))
    far = np.zeros(n)
    for i, p in enumerate(par):
        far[i] = length[i] + (far[p] if p >= 0 else 0.0)
    scale = 1.0 / far.max()
    t = {"parents": par, "rest_q": rest_q.astype(np.float32), "rest_t": (rest_t * scale).astype(np.float32),
         "scale": scale}
    for name, k in (("keys", keys), ("add", add)):
        if k is not None:
            k[..., 4:7] *= scale
            t[name] = k.astype(np.float32)
    if "verts" in case:
        t["mesh"] = _mesh(par, case["verts"], rng)
    return t


def _mesh(par, nv, rng):
    """Vertices grouped by a home joint in joint order, weighted to it and up to three relatives; a strip of faces."""
    n = len(par)
    child = np.full(n, -1)
    for j in range(n - 1, 0, -1):
        child[par[j]] = j
    home = np.arange(nv) * n // nv
    pos = rng.uniform(-0.5, 0.5, size=(n, 3))[home] + rng.uniform(-0.03, 0.03, size=(nv, 3))
    nrm = rng.normal(size=(nv, 3))
    nrm /= np.linalg.norm(nrm, axis=1, keepdims=True)
    p1 = par[home]
    p2 = np.where(p1 >= 0, par[np.maximum(p1, 0)], -1)
    bones = np.stack([home, p1, p2, child[home]], axis=1)
    w = -np.sort(-rng.uniform(0.05, 1.0, size=(nv, 4)), axis=1)
    few = rng.uniform(size=nv) < 0.25  # a quarter of the vertices use fewer influences
    w[few & (rng.uniform(size=nv) < 0.5), 2] = 0.0
    w[few, 3] = 0.0
    w[bones < 0] = 0.0
    w /= w.sum(axis=1, keepdims=True)
    return {"pos": pos.astype(np.float32), "nrm": nrm.astype(np.float32), "bones": np.maximum(bones, 0).astype(np.int32),
            "weights": w.astype(np.float32), "faces": _strip(nv)}


def _strip(nv):
    return np.array([(v, v + 1, v + 2) if v % 2 == 0 else (v, v + 2, v + 1) for v in range(nv - 2)], np.int32)


# ------------------------------------------------------------------ inputs
def _gpu_quats(gen, rows, degrees):
    axis = torch.nn.functional.normalize(torch.randn(rows, 3, generator=gen, device="cuda"), dim=1)
    half = torch.rand(rows, 1, generator=gen, device="cuda") * (math.radians(degrees) / 2)
    return torch.cat([axis * torch.sin(half), torch.cos(half)], dim=1)


def _uniform(gen, lo, hi, *shape):
    return torch.rand(*shape, generator=gen, device="cuda") * (hi - lo) + lo


def _inputs(case, seed):
    """Everything drawn for a case: types, the characters' types, and the per-character and per-joint inputs."""
    rng = np.random.default_rng(seed)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    kind = case["kind"]
    if kind == "raster":
        n, nv = case["chars"], case["verts"]
        x = {"types": [{"parents": np.array([-1], np.int32), "rest_q": np.array([[0, 0, 0, 1]], np.float32),
                        "rest_t": np.zeros((1, 3), np.float32), "mesh": _mesh(np.array([-1]), nv, rng)}],
             "char_type": np.zeros(n, np.int32)}
        # what the skinning leaves: patches of three vertices around points of a body of unit extent
        body = _uniform(gen, -0.5, 0.5, n, nv // 3 + 1, 3).repeat_interleave(3, dim=1)[:, :nv]
        pos = body + _uniform(gen, -0.03, 0.03, n, nv, 3)
        nrm = torch.nn.functional.normalize(torch.randn(n, nv, 3, generator=gen, device="cuda"), dim=2)
        x["vertices"] = torch.cat([pos, nrm], dim=2).reshape(n * nv, 6).contiguous()
        return x
    parents, char_type = _parents(case, rng)
    types = [_type(p, case, rng) for p in parents]
    n = len(char_type)
    rows = int(sum(len(parents[t]) for t in char_type))
    x = {"types": types, "char_type": char_type}
    if "keys" in case:
        x["time"] = _uniform(gen, 0.0, 1.0 if case["keys"] <= 30 else case["keys"] / RATE_HZ, n)
        if kind == "layers":
            w = _uniform(gen, 0.0, 1.0, n, 4)
            off = _uniform(gen, 0.0, 1.0, n, 4) < 1.0 / 3.0  # a third of the layers are off, never the first
            off[:, 0] = False
            x["weights"] = torch.where(off, torch.zeros_like(w), w)
            x["add_w"] = _uniform(gen, 0.0, 1.0, n)
        else:
            x["blend"] = _uniform(gen, 0.0, 1.0, n)
        if kind == "host":
            x["time"], x["blend"] = x["time"].cpu().pin_memory(), x["blend"].cpu().pin_memory()
        return x
    scale = torch.tensor([t["scale"] for t in types], device="cuda", dtype=torch.float32)
    per_char = torch.as_tensor(np.array([len(p) for p in parents])[char_type], device="cuda")
    row_scale = scale[torch.as_tensor(char_type, device="cuda").long()].repeat_interleave(per_char)[:, None]
    if kind == "ik":
        x["q"] = _gpu_quats(gen, rows, 30.0)
        x["t"] = torch.cat([torch.as_tensor(types[t]["rest_t"]) for t in char_type]).cuda()
        # a fit in progress: moments of the size the effectors' gradients have
        x["m"] = 0.05 * torch.randn(rows, 4, generator=gen, device="cuda")
        x["v"] = _uniform(gen, 0.05, 0.4, rows, 4) ** 2
        x["targets"] = _uniform(gen, -0.3, 0.3, n, IK_EFFECTORS, 3)
        x["effectors"] = np.stack([_deep_leaves(p) for p in parents])
        return x
    x["q"] = _gpu_quats(gen, rows, 30.0) * _uniform(gen, 0.8, 1.2, rows, 1)  # not normalized by the caller
    x["t"] = _uniform(gen, -0.1, 0.1, rows, 3) * row_scale
    if kind == "loss":
        x["target"] = _uniform(gen, -0.5, 0.5, rows, 3)
    elif kind == "autograd":
        x["grad"] = torch.randn(rows, 3, generator=gen, device="cuda")
    return x


def _deep_leaves(par):
    dep = _depths(par)
    leaf = np.ones(len(par), bool)
    leaf[par[par >= 0]] = False
    ids = np.nonzero(leaf)[0]
    return np.sort(ids[np.argsort(-dep[ids], kind="stable")][:IK_EFFECTORS]).astype(np.int32)


def _depths(par):
    d = np.zeros(len(par), np.int64)
    for i, p in enumerate(par):
        d[i] = 0 if p < 0 else d[p] + 1
    return d


# ----------------------------------------------------------- prepare, run
def prepare(case, seed):
    x = _inputs(case, seed)
    kind = case["kind"]
    types = x["types"]
    ctx = anim.Context(0)
    ids = ctx.create_skeletons([t["parents"] for t in types], rest_q=[t["rest_q"] for t in types],
                               rest_t=[t["rest_t"] for t in types])
    for i, t in zip(ids, types):
        if "keys" in t:
            ctx.upload_clips(i, t["keys"], RATE_HZ)
        if "add" in t:
            ctx.upload_additive(i, t["add"], RATE_HZ)
        if "mesh" in t:
            ctx.upload_mesh(i, t["mesh"])
            if kind == "raster":
                ctx.upload_faces(i, t["mesh"]["faces"])
    plan = ctx.plan(np.asarray(ids, np.int32)[x["char_type"]])
    if case.get("schedule"):
        ctx.set_schedule(plan, [int(v) for v in case["schedule"].split()])
    s = {"case": case, "ctx": ctx, "plan": plan}
    s.update((k, v) for k, v in x.items() if isinstance(v, torch.Tensor))
    new = lambda *shape: torch.empty(shape, dtype=torch.float32, device="cuda")  # noqa: E731
    if kind in ("frame", "layers"):
        s["out"] = new(plan.total, 12)
    elif kind == "host":
        s["out"] = torch.empty((plan.total, 12), dtype=torch.float32, pin_memory=True)
    elif kind == "skinned":
        s["out"] = new(int(ctx.vertex_offsets(plan)[-1]), 6)
    elif kind == "raster":
        h, w = case["height"], case["width"]
        s["vis"] = torch.empty((h, w), dtype=torch.int64, device="cuda")
        s["ids"] = torch.empty((h, w), dtype=torch.int32, device="cuda")
        s["rgba"] = torch.empty((h, w), dtype=torch.int32, device="cuda")
    elif kind == "loss":
        s["grad_q"], s["grad_t"], s["loss"] = new(plan.total, 4), new(plan.total, 3), new(plan.n_chars)
    elif kind == "autograd":
        s["fn"] = anim.hierarchy_fn()
        s["q"].requires_grad_(True)
        s["t"].requires_grad_(True)
    elif kind == "ik":
        s["ik"] = ctx.ik(plan, x["effectors"])
        s["ik"].reset()
        s["loss"] = new(plan.n_chars)
    return s


def run(s):
    case, ctx, plan = s["case"], s["ctx"], s["plan"]
    kind = case["kind"]
    if kind == "frame":
        return ctx.evaluate_frame(plan, s["time"], s["blend"], out=s["out"])
    if kind == "layers":
        return ctx.evaluate_frame_layers(plan, s["time"], s["weights"], s["add_w"], out=s["out"])
    if kind == "skinned":
        return ctx.evaluate_frame_skinned(plan, s["time"], s["blend"], verts=s["out"])
    if kind == "host":
        return ctx.evaluate_frame_host(plan, s["time"], s["blend"], out=s["out"])
    if kind == "raster":
        return ctx.raster(plan, s["vertices"], case["width"], case["height"], case["cols"], 2.6, 15.0, 15.0,
                          case["scale"], ids=s["ids"], rgba=s["rgba"], vis=s["vis"])
    if kind == "forward":
        return ctx.forward_local(plan, s["q"], s["t"])[0]
    if kind == "loss":
        return ctx.loss_backward(plan, s["q"], s["t"], s["target"], s["grad_q"], s["grad_t"], s["loss"])
    if kind == "autograd":
        p = s["fn"].apply(s["q"], s["t"], ctx, plan)
        return (p, *torch.autograd.grad(p, (s["q"], s["t"]), s["grad"]))
    for _ in range(case["steps"]):
        s["ik"].step(s["q"], s["m"], s["v"], s["t"], s["targets"], loss=s["loss"], **ADAM)
    return s["q"], s["m"], s["v"], s["loss"]


# -------------------------------------------------------------------- work
def work(case):
    kind = case["kind"]
    if kind == "raster":
        n, nv, px = case["chars"], case["verts"], case["width"] * case["height"]
        # every vertex once, both images; per vertex the projection, per face the three edge functions
        return {"bytes": n * nv * 24 + 8 * px, "flops": n * nv * (8 + 40)}
    parents, char_type = _parents(case, np.random.default_rng(0))
    sizes = np.array([len(p) for p in parents])
    n, rows, table = len(char_type), int(sizes[char_type].sum()), int(sizes.sum())
    if "keys" in case:
        clips = case["clips"] + (1 if kind == "layers" else 0)
        keys = clips * case["keys"] * table * 32
        per_char = 24 if kind == "layers" else 8
        out = n * case["verts"] * 24 if kind == "skinned" else rows * 48
        mesh = len(sizes) * case["verts"] * 48 if kind == "skinned" else 0
        # a slerp and a lerp per clip and a slerp per blend (about 45 each), the composition and the bind product
        flops = rows * (45 * (2 * clips - 1) + 66 + 66) + (n * case["verts"] * 4 * 36 if kind == "skinned" else 0)
        return {"bytes": keys + table * 52 + n * per_char + out + mesh, "flops": flops}
    if kind == "forward":
        return {"bytes": rows * (28 + 48) + table * 52, "flops": rows * (40 + 66 + 66)}
    if kind == "loss":
        return {"bytes": rows * (28 + 12 + 28) + n * 4, "flops": rows * 250}
    if kind == "autograd":
        # positions out, then poses and position gradients in, gradients out
        return {"bytes": rows * (28 + 12 + 28 + 12 + 28), "flops": rows * 350}
    active = np.zeros(len(parents))
    for k, p in enumerate(parents):
        on = np.zeros(len(p), bool)
        for j in _deep_leaves(p):
            while j >= 0:
                on[j] = True
                j = p[j]
        active[k] = on.sum()
    rows = float(active[char_type].sum())  # the effectors' ancestors: q, t, m, v in; q, m, v out
    return {"bytes": case["steps"] * (rows * (16 + 12 + 6 * 16 - 16) + n * (IK_EFFECTORS * 12 + 4)),
            "flops": case["steps"] * rows * 330}


# ------------------------------------------------------------------- exact
def _mul(a, b):
    ax, ay, az, aw = a.unbind(-1)
    bx, by, bz, bw = b.unbind(-1)
    return torch.stack([aw * bx + ax * bw + ay * bz - az * by, aw * by - ax * bz + ay * bw + az * bx,
                        aw * bz + ax * by - ay * bx + az * bw, aw * bw - ax * bx - ay * by - az * bz], -1)


def _unit(q):
    return q / q.norm(dim=-1, keepdim=True)


def _rot(q):
    x, y, z, w = _unit(q).unbind(-1)
    return torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y),
                        2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x),
                        2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)], -1).reshape(*q.shape[:-1], 3, 3)


def _slerp(a, b, w):
    """On the shorter arc; w broadcasts over the leading dimensions."""
    a, b = _unit(a), _unit(b)
    b = torch.where((a * b).sum(-1, keepdim=True) < 0, -b, b)
    th = 2 * torch.atan2((a - b).norm(dim=-1), (a + b).norm(dim=-1))[..., None]
    w = w.expand(th.shape[:-1])[..., None]
    sn = torch.sin(th)
    small = th < 1e-9
    sn = torch.where(small, torch.ones_like(sn), sn)
    wa = torch.where(small, 1 - w, torch.sin((1 - w) * th) / sn)
    wb = torch.where(small, w, torch.sin(w * th) / sn)
    return _unit(wa * a + wb * b)


def _levels(par):
    d = _depths(par)
    order = np.argsort(d, kind="stable")
    cuts = np.searchsorted(d[order], np.arange(d.max() + 2))
    return [torch.as_tensor(order[cuts[k]:cuts[k + 1]], device="cuda") for k in range(d.max() + 1)]


def _compose(par, R, t):
    """Model rotations and translations of [characters, joints, ...] local ones, level by level."""
    R, t = R.clone(), t.clone()
    up = torch.as_tensor(np.asarray(par, np.int64), device="cuda")
    for lv in _levels(par)[1:]:
        p = up[lv]
        Rp = R[:, p]
        t[:, lv] = t[:, p] + (Rp @ t[:, lv, :, None])[..., 0]
        R[:, lv] = Rp @ R[:, lv]
    return R, t


def _sample(keys, time, clip):
    """(q, t) of one clip [keys, joints, 8] at each character's time; the key index is decided in float32."""
    u = time.float() * np.float32(RATE_HZ)
    k = torch.floor(u)
    al = (u - k).double()[:, None]
    k = k.long() % keys.shape[1]
    a, b = keys[clip][k], keys[clip][(k + 1) % keys.shape[1]]
    return _slerp(a[..., :4], b[..., :4], al), a[..., 4:7] + al[..., None] * (b[..., 4:7] - a[..., 4:7])


def _local(case, ty, x, rows):
    """Local rotations and translations the Simulation stage gives the characters `rows` of type ty."""
    keys = torch.as_tensor(ty["keys"], device="cuda").double()
    time = x["time"].cuda()[rows]
    q, t = _sample(keys, time, 0)
    if case["kind"] != "layers":
        if case["clips"] > 1:
            w = x["blend"].cuda()[rows].double()[:, None]
            qb, tb = _sample(keys, time, 1)
            q, t = _slerp(q, qb, w), t + w[..., None] * (tb - t)
        return _rot(q), t
    wts = x["weights"][rows].double()
    W = wts[:, 0].clone()
    acc = W[:, None, None] * t
    for i in range(1, case["clips"]):
        w = wts[:, i]
        W = W + w
        qi, ti = _sample(keys, time, i)
        f = torch.where(W > 0, w / torch.where(W > 0, W, torch.ones_like(W)), torch.zeros_like(W))
        q = torch.where((W > 0)[:, None, None], _slerp(q, qi, f[:, None]), q)
        acc = acc + w[:, None, None] * ti
    t = torch.where((W > 0)[:, None, None], acc / torch.where(W > 0, W, torch.ones_like(W))[:, None, None], t)
    a = x["add_w"][rows].double()
    qa, ta = _sample(torch.as_tensor(ty["add"], device="cuda").double()[None], time, 0)
    one = torch.zeros_like(qa)
    one[..., 3] = 1
    return _rot(_mul(q, _slerp(one, qa, a[:, None]))), t + a[:, None, None] * ta


def _groups(x):
    """For each type: (type, its characters, their joints' rows [characters, joints])."""
    ct = x["char_type"]
    sizes = np.array([len(t["parents"]) for t in x["types"]])
    off = np.concatenate([[0], np.cumsum(sizes[ct])])
    for k, ty in enumerate(x["types"]):
        chars = np.nonzero(ct == k)[0]
        if len(chars):
            rows = torch.as_tensor(off[chars][:, None] + np.arange(sizes[k])[None], device="cuda")
            yield k, ty, torch.as_tensor(chars, device="cuda"), rows


def _total(x):
    sizes = np.array([len(t["parents"]) for t in x["types"]])
    return int(sizes[x["char_type"]].sum())


def _skin(ty, R, t):
    """Skin matrices [characters, joints, 3, 4]: model pose times inverse of the rest pose's model pose."""
    Rr, tr = _compose(ty["parents"], _rot(torch.as_tensor(ty["rest_q"], device="cuda").double())[None],
                      torch.as_tensor(ty["rest_t"], device="cuda").double()[None])
    Rb = Rr.transpose(-1, -2)
    tb = -(Rb @ tr[..., None])
    return torch.cat([R @ Rb, R @ tb + t[..., None]], dim=-1)


def _lbs(mesh, S):
    pos, nrm, wts = (torch.as_tensor(mesh[k], device="cuda").double() for k in ("pos", "nrm", "weights"))
    bones = torch.as_tensor(mesh["bones"], device="cuda").long()
    B = 0
    for k in range(4):
        B = B + wts[:, k, None, None] * S[:, bones[:, k]]
    v = (B[..., :3] @ pos[..., None])[..., 0] + B[..., 3]
    return torch.cat([v, torch.nn.functional.normalize((B[..., :3] @ nrm[..., None])[..., 0], dim=-1)], dim=-1)


def _adjoint(par, q, t, g, Rm, p):
    """Gradients of a loss with dLoss/dp = g with respect to the unnormalized q and t, from the subtree sums of
    forces and moments."""
    F, T = g.clone(), torch.linalg.cross(p, g)
    up = torch.as_tensor(np.asarray(par, np.int64), device="cuda")
    for lv in reversed(_levels(par)[1:]):
        F.index_add_(1, up[lv], F[:, lv])
        T.index_add_(1, up[lv], T[:, lv])
    tau = T - torch.linalg.cross(p, F)
    has = (up >= 0)[None, :, None]
    Rt = Rm[:, up.clamp(min=0)].transpose(-1, -2)
    tau = torch.where(has, (Rt @ tau[..., None])[..., 0], tau)
    dt = torch.where(has, (Rt @ F[..., None])[..., 0], F)
    n = q.norm(dim=-1, keepdim=True)
    return 2 / n * _mul(torch.cat([tau, torch.zeros_like(n)], -1), q / n), dt


def exact(case, seed):
    x = _inputs(case, seed)
    kind = case["kind"]
    if kind == "raster":
        return None  # whole numbers
    f64 = {"dtype": torch.float64, "device": "cuda"}
    total, n = _total(x), len(x["char_type"])
    if kind == "skinned":
        out = torch.empty(n, case["verts"], 6, **f64)
    elif kind in ("frame", "layers", "host", "forward"):
        out = torch.empty(total, 12, **f64)
    elif kind == "ik":
        q, m, v = x["q"].double(), x["m"].double(), x["v"].double()
        loss = torch.empty(n, **f64)
    else:
        pos, gq, gt, loss = (torch.empty(*s, **f64) for s in ((total, 3), (total, 4), (total, 3), (n,)))
    for k, ty, chars, rows in _groups(x):
        par = ty["parents"]
        for at in range(0, len(chars), 2048):  # bounds the temporaries
            c, r = chars[at:at + 2048], rows[at:at + 2048]
            if "keys" in case:
                S = _skin(ty, *_compose(par, *_local(case, ty, x, c)))
                if kind == "skinned":
                    out[c] = _lbs(ty["mesh"], S)
                else:
                    out[r.reshape(-1)] = S.reshape(-1, 12)
                continue
            t = x["t"][r].double()
            if kind == "ik":
                _exact_ik(case, x, k, par, c, r, t, q, m, v, loss)
                continue
            ql = x["q"][r].double()
            R, p = _compose(par, _rot(ql), t)
            if kind == "forward":
                out[r.reshape(-1)] = _skin(ty, R, p).reshape(-1, 12)
                continue
            if kind == "loss":
                d = p - x["target"][r].double()
                loss[c] = d.square().sum(dim=(1, 2))
                g = 2 * d
            else:
                g = x["grad"][r].double()
            dq, dt = _adjoint(par, ql, t, g, R, p)
            pos[r.reshape(-1)], gq[r.reshape(-1)], gt[r.reshape(-1)] = (z.reshape(r.numel(), -1) for z in (p, dq, dt))
    if kind == "ik":
        return q, m, v, loss
    if kind == "loss":
        return gq, gt, loss
    if kind == "autograd":
        return pos, gq, gt
    return out.reshape(-1, 6) if kind == "skinned" else out.cpu() if kind == "host" else out


def _exact_ik(case, x, k, par, c, r, t, q, m, v, loss):
    """The case's Adam steps on the ancestors of the effectors of the characters c (rows r) of type k."""
    eff = x["effectors"][k]
    on = np.zeros(len(par), bool)
    for j in eff:
        while j >= 0:
            on[j] = True
            j = par[j]
    act = torch.as_tensor(np.nonzero(on)[0], device="cuda")
    e = torch.as_tensor(eff, device="cuda").long()
    (b1, b2), lr, eps = ADAM["betas"], ADAM["lr"], ADAM["eps"]
    ra = r[:, act].reshape(-1)
    for step in range(1, case["steps"] + 1):
        ql = q[r]
        R, p = _compose(par, _rot(ql), t)
        d = p[:, e] - x["targets"][c].double()
        loss[c] = d.square().sum(dim=(1, 2))
        g = torch.zeros_like(p)
        g[:, e] = 2 * d
        dq = _adjoint(par, ql, t, g, R, p)[0][:, act].reshape(-1, 4)
        m[ra] = b1 * m[ra] + (1 - b1) * dq
        v[ra] = b2 * v[ra] + (1 - b2) * dq.square()
        den = (v[ra] / (1 - b2 ** step)).sqrt() + eps
        q[ra] = q[ra] - lr / (1 - b1 ** step) * m[ra] / den
