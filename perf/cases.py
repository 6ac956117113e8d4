"""The workloads this geometry stage is timed on, through its public entry points.

A case is a dict of plain values; ``prepare`` builds what a user's program holds before the call (device buffers,
uniforms, a context with its stream, a partition, a frame, a server with registered meshes), ``run`` makes one pass
and returns its whole output, ``exact`` gives the same output in 64 bits from plain tensor code, and ``work`` the
bytes and operations a pass cannot do without.  Kinds:

* ``draw``  -- one ``gp_submit_drawcall`` (every method, batching mode, shader; with a partition kept from load time,
  or partitioned at submit because the topology is new);
* ``frame`` -- one ``gp_frame_submit`` of many skinned draws configured by a saved autotune table;
* ``serve`` -- a burst of requests to ``gp_server_submit`` and the wait for them;
* ``walk``  -- ``gp_random_walk`` steps of agents on a toroidal activity field;
* ``loop``  -- one ``gp_loop_subdivide`` step.

Meshes are closed tori in a locality order (triangles sorted by the Morton code of their centroid, 5% of the
256-triangle blocks permuted, vertex ids permuted), the recipe of the repository's scanned-model stand-in, or open
grids in scanline order, as in its correctness and frame workloads.  Everything is made on the GPU from the seed.
"""
import math
import random

import numpy as np
import torch

import paper_1805_08893_gb300 as gp

SHADERS = {"mvp": gp.GP_SHADER_MVP, "skin": gp.GP_SHADER_SKIN, "envelope": gp.GP_SHADER_ENVELOPE,
           "load": gp.GP_SHADER_LOAD}
# operations to shade one vertex (a multiply-add counts two)
SHADER_FLOPS = {"mvp": 39, "skin": 4 * 51 + 39, "envelope": 2 * (16 * 36 + 8), "load": 42}
TUNED = {"max_unique": 320, "max_tris": 426, "hash_slots": 2048}  # the limits the benchmark draws hash/phash with
LIMITS = {"default": {}, "tuned": TUNED, "small": {"max_unique": 64, "max_tris": 64},
          "s255": {"batch_indices": 255}, "s96": {"batch_indices": 96}}


def listed():
    return [
        # one small mesh (the 64 x 64-vertex grid) at the context's defaults: what a call costs when launches count
        {"name": "draw_small", "kind": "draw", "variant": "hash", "mode": 1, "shader": "mvp", "mesh": "grid",
         "tris": 7938, "limits": "default", "threads": 0, "kept": True, "steps": 0},
        # the benchmark's scanned model: 7.2M triangles, hash over dynamic batches at the tuned limits
        {"name": "draw_large", "kind": "draw", "variant": "hash", "mode": 1, "shader": "mvp", "mesh": "torus",
         "tris": 7_200_000, "limits": "tuned", "threads": 0, "kept": True, "steps": 0},
        # simplification envelopes, the heavy shader: parallel hashing, 32-byte output corners, a ragged count
        {"name": "draw_envelope", "kind": "draw", "variant": "phash", "mode": 1, "shader": "envelope",
         "mesh": "torus", "tris": 1_997_119, "limits": "tuned", "threads": 0, "kept": True, "steps": 0},
        # sort-based reuse on a buddha-sized model at the paper's limits
        {"name": "draw_sort", "kind": "draw", "variant": "sort", "mode": 1, "shader": "mvp", "mesh": "torus",
         "tris": 1_085_780, "limits": "default", "threads": 0, "kept": True, "steps": 0},
        # an animated character crowd in one buffer: the default context (hash, static batches) with skinning
        {"name": "draw_skin", "kind": "draw", "variant": "hash", "mode": 0, "shader": "skin", "mesh": "torus",
         "tris": 499_979, "limits": "default", "threads": 0, "kept": True, "steps": 0},
        # warp voting on a streamed mesh without preprocessing
        {"name": "draw_warp", "kind": "draw", "variant": "warp", "mode": 0, "shader": "mvp", "mesh": "torus",
         "tris": 1_085_780, "limits": "default", "threads": 0, "kept": True, "steps": 0},
        # no reuse, the method of choice for a simple shader; ragged against blocks and 16-byte words
        {"name": "draw_naive", "kind": "draw", "variant": "naive", "mode": 0, "shader": "mvp", "mesh": "torus",
         "tris": 3_000_001, "limits": "default", "threads": 0, "kept": True, "steps": 0},
        # topology that changes every call (cut or streamed geometry): the dynamic partition is part of the call
        {"name": "draw_new_topology", "kind": "draw", "variant": "hash", "mode": 1, "shader": "mvp",
         "mesh": "torus", "tris": 500_003, "limits": "default", "threads": 0, "kept": False, "steps": 0},
        # a game frame: 240 skinned draws of 100 to 50,000 triangles in one graph launch, configured by size
        {"name": "frame_skin", "kind": "frame", "draws": 240, "tmin": 100, "tmax": 50_000, "sizes": 3},
        # a server's burst: 64 requests over 32 resident meshes, half of them skinned
        {"name": "serve_burst", "kind": "serve", "meshes": 32, "requests": 64, "tmin": 500, "tmax": 100_000,
         "sizes": 5},
        # ten steps of the random walk: 300,000 agents on a 256 x 256 field
        {"name": "walk", "kind": "walk", "variant": "hash", "agents": 300_000, "width": 256, "height": 256,
         "steps": 10, "batch": 512, "threads": 512},
        # one Loop subdivision step of a closed model at the paper's batch limits
        {"name": "loop", "kind": "loop", "variant": "hash", "mesh": "torus", "tris": 500_000, "mode": 1},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["draw"] * 8 + ["frame", "serve", "walk", "loop"])
    if kind == "frame":
        tmin = _log(rng, 50, 1000)
        return {"kind": "frame", "draws": _log(rng, 8, 240), "tmin": tmin, "tmax": tmin * _log(rng, 4, 50),
                "sizes": rng.randrange(1 << 20)}
    if kind == "serve":
        tmin = _log(rng, 50, 2000)
        return {"kind": "serve", "meshes": rng.randint(4, 32), "requests": rng.randint(4, 64), "tmin": tmin,
                "tmax": tmin * _log(rng, 4, 50), "sizes": rng.randrange(1 << 20)}
    if kind == "walk":
        variant = rng.choice(["naive", "warp", "sort", "hash", "phash"])
        return {"kind": "walk", "variant": variant, "agents": _log(rng, 1000, 300_000),
                "width": rng.randint(40, 512), "height": rng.randint(40, 512), "steps": rng.randint(1, 10),
                "batch": 32 * rng.randint(4, 18), "threads": rng.choice([128, 256, 512])}
    if kind == "loop":
        variant = rng.choice(["naive", "warp", "sort", "hash", "phash"])
        return {"kind": "loop", "variant": variant, "mesh": rng.choice(["torus", "grid"]),
                "tris": _log(rng, 2000, 500_000),
                "mode": rng.randint(0, 1) if variant in ("sort", "hash", "phash") else 0}
    variant = rng.choice(["naive", "warp", "sort", "hash", "hash", "phash", "multi"])
    mode = rng.randint(0, 1) if variant in ("sort", "hash", "phash") else 0
    limits = "default"
    if mode == 1:
        limits = rng.choice(["default", "tuned", "small"])
    elif variant not in ("naive", "multi"):
        limits = rng.choice(["default", "s255", "s96"])
    shader = rng.choice(["mvp", "skin", "envelope", "load"])
    return {"kind": "draw", "variant": variant, "mode": mode, "shader": shader,
            "mesh": rng.choice(["torus", "torus", "grid"]), "tris": _log(rng, 1000, 4_000_000), "limits": limits,
            "threads": rng.choice([0, 128, 256]), "kept": not (mode == 1 and rng.random() < 0.3),
            "steps": rng.choice([64, 256]) if shader == "load" else 0}


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _gen(seed, salt=0):
    return torch.Generator(device="cuda").manual_seed((int(seed) * 1_000_003 + salt) % (1 << 62))


def _rand(n, g):
    return torch.rand(n, generator=g, device="cuda", dtype=torch.float64)


def _spread21(x):
    x = (x | (x << 32)) & 0x1F00000000FFFF
    x = (x | (x << 16)) & 0x1F0000FF0000FF
    x = (x | (x << 8)) & 0x100F00F00F00F00F
    x = (x | (x << 4)) & 0x10C30C30C30C30C3
    return (x | (x << 2)) & 0x1249249249249249


def _torus(tris, g):
    """(vertices f32 [V, 8], triangles int64 [T, 3]): the first ``tris`` triangles of a closed torus grid with 2%
    radial noise, in locality order, vertex ids permuted."""
    nu = max(4, int(round(math.sqrt(tris / 2.0))))
    nv = max(4, -(-tris // (2 * nu)))
    V = nu * nv
    i = torch.arange(nu, device="cuda").repeat_interleave(nv)
    j = torch.arange(nv, device="cuda").repeat(nu)
    a, b = 2 * math.pi * i.double() / nu, 2 * math.pi * j.double() / nv
    ca, sa, cb, sb = a.cos(), a.sin(), b.cos(), b.sin()
    nrm = torch.stack([ca * cb, sa * cb, sb], 1)
    centre = torch.stack([ca, sa, torch.zeros_like(ca)], 1)
    smooth = centre + 0.4 * nrm
    pos = centre + 0.4 * (1 + 0.02 * (2 * _rand(V, g) - 1))[:, None] * nrm
    i1, j1 = (i + 1) % nu, (j + 1) % nv
    p, q, r, s = i * nv + j, i1 * nv + j, i1 * nv + j1, i * nv + j1
    t = torch.stack([p, q, r, p, r, s], 1).view(-1, 3)
    cent = smooth[t].mean(1)
    cell = ((cent - cent.amin(0)) / (cent.amax(0) - cent.amin(0)).clamp_min(1e-30) * (2**21 - 1)).long()
    code = _spread21(cell[:, 0]) | (_spread21(cell[:, 1]) << 1) | (_spread21(cell[:, 2]) << 2)
    t = t[torch.sort(code, stable=True)[1]][:tris]
    nb = t.shape[0] // 256
    m = int(round(0.05 * nb))
    if m >= 2:
        chosen = torch.randperm(nb, generator=g, device="cuda")[:m].sort()[0]
        blocks = torch.arange(nb, device="cuda")
        blocks[chosen] = chosen[torch.randperm(m, generator=g, device="cuda")]
        t = torch.cat([t[:nb * 256].view(nb, 256, 3)[blocks].view(-1, 3), t[nb * 256:]])
    verts = torch.empty(V, 8, dtype=torch.float32, device="cuda")
    perm = torch.randperm(V, generator=g, device="cuda")
    verts[perm] = torch.cat([pos, nrm, (a / (2 * math.pi))[:, None], (b / (2 * math.pi))[:, None]], 1).float()
    return verts, perm[t]


def _grid(tris, g):
    """An open grid of ``w`` x ``h`` quads in scanline order (as many as ``tris`` triangles need), ids in order."""
    w = max(1, int(round(math.sqrt(tris / 2.0))))
    h = max(1, -(-tris // (2 * w)))
    y, x = torch.meshgrid(torch.linspace(-1, 1, h + 1, dtype=torch.float64, device="cuda"),
                          torch.linspace(-1, 1, w + 1, dtype=torch.float64, device="cuda"), indexing="ij")
    fa, fb = (0.5 + 1.5 * _rand(2, g)) * math.pi
    z = 0.1 * (fa * x).sin() * (fb * y).cos()
    nrm = torch.stack([-0.1 * fa * (fa * x).cos() * (fb * y).cos(), 0.1 * fb * (fa * x).sin() * (fb * y).sin(),
                       torch.ones_like(z)], -1)
    nrm = nrm / nrm.norm(dim=-1, keepdim=True)
    verts = torch.cat([torch.stack([x, y, z], -1), nrm, torch.stack([(x + 1) / 2, (y + 1) / 2], -1)], -1)
    jj, ii = torch.meshgrid(torch.arange(h, device="cuda"), torch.arange(w, device="cuda"), indexing="ij")
    p = (jj * (w + 1) + ii).view(-1)
    t = torch.stack([p, p + 1, p + w + 2, p, p + w + 2, p + w + 1], 1).view(-1, 3)
    return verts.view(-1, 8).float().contiguous(), t[:tris]


def _mesh(kind, tris, g):
    return _torus(tris, g) if kind == "torus" else _grid(tris, g)


def _skinned(verts, g):
    """64-byte rows: each vertex bound to the 4 nearest of 64 bone centres, random weights."""
    V = verts.shape[0]
    centres = verts[torch.randint(0, V, (64,), generator=g, device="cuda"), :3]
    ids = torch.cdist(verts[:, :3], centres).topk(4, dim=1, largest=False)[1].int()
    w = 1 - _rand((V, 4), g)
    rows = torch.zeros(V, 16, dtype=torch.float32, device="cuda")
    rows[:, :8] = verts
    rows.view(torch.int32)[:, 8] = ids[:, 0] | (ids[:, 1] << 8) | (ids[:, 2] << 16) | (ids[:, 3] << 24)
    rows[:, 9:13] = (w / w.sum(1, keepdim=True)).float()
    return rows


def _camera(r):
    """(M [4, 4], N [3, 3]) of a seeded look-at camera, built in float64, rounded once."""
    eye = r.normal(size=3)
    eye *= 3.0 / np.linalg.norm(eye)
    f = -eye / np.linalg.norm(eye)
    s = np.cross(f, (0.0, 0.0, 1.0) if abs(f[2]) < 0.99 else (1.0, 0.0, 0.0))
    s /= np.linalg.norm(s)
    R = np.stack([s, np.cross(s, f), -f])
    view = np.eye(4)
    view[:3, :3], view[:3, 3] = R, -R @ eye
    t = 1.0 / math.tan(math.radians(30.0))
    proj = np.array([[t * 9 / 16, 0, 0, 0], [0, t, 0, 0], [0, 0, -100.1 / 99.9, -20.0 / 99.9], [0, 0, -1, 0]])
    return (proj @ view).astype(np.float32), R.astype(np.float32)


def _palette(r):
    """64 bones, each a 3x4 [R | t] with a small rotation and offset."""
    ax = r.normal(size=(64, 3))
    ax /= np.linalg.norm(ax, axis=1, keepdims=True)
    ang = r.uniform(-0.2, 0.2, size=(64, 1, 1))
    K = np.zeros((64, 3, 3))
    K[:, 0, 1], K[:, 0, 2], K[:, 1, 0] = -ax[:, 2], ax[:, 1], ax[:, 2]
    K[:, 1, 2], K[:, 2, 0], K[:, 2, 1] = -ax[:, 0], -ax[:, 1], ax[:, 0]
    pal = np.empty((64, 3, 4))
    pal[:, :, :3] = np.eye(3) + np.sin(ang) * K + (1 - np.cos(ang)) * (K @ K)
    pal[:, :, 3] = r.uniform(-0.05, 0.05, size=(64, 3))
    return pal.astype(np.float32)


def _directions():
    k = np.arange(16) + 0.5
    z = 1 - k / 8
    r, ang = np.sqrt(1 - z * z), math.pi * (3 - math.sqrt(5)) * k
    return np.stack([r * np.cos(ang), r * np.sin(ang), z], 1).astype(np.float32)


def _item(mesh, shader, tris, seed, salt, steps=0):
    """One draw's inputs: vertex rows, triangles, the uniform values and their blob."""
    g, r = _gen(seed, salt), np.random.default_rng([int(seed), salt])
    verts, t = _mesh(mesh, tris, g)
    v = {"M": None}
    v["M"], v["N"] = _camera(r)
    if shader == "skin":
        verts, v["palette"] = _skinned(verts, g), _palette(r)
        blob = gp.uniforms_skin(v["M"], v["N"], v["palette"])
    elif shader == "envelope":
        v["d"] = np.float32(0.02 * float((verts[:, :3].amax(0) - verts[:, :3].amin(0)).norm()))
        v["dirs"] = _directions()
        blob = gp.uniforms_envelope(v["d"], v["dirs"])
    elif shader == "load":
        v["steps"] = steps
        blob = gp.uniforms_load(v["M"], v["N"], steps)
    else:
        blob = gp.uniforms_mvp(v["M"], v["N"])
    return {"verts": verts, "tris": t, "idx": t.reshape(-1).int(), "values": v, "blob": blob, "shader": shader}


def _sizes(case, count):
    """Triangle counts, log-uniform in [tmin, tmax]."""
    r = random.Random(case["sizes"])
    return [_log(r, case["tmin"], case["tmax"]) for _ in range(count)]


def _spans(items):
    """Where each item's triangles lie in one output buffer (16-byte aligned), and the buffer's length."""
    at, o = [], 0
    for it in items:
        n = it["tris"].shape[0] * 3 * (8 if it["shader"] == "envelope" else 7)
        at.append((o, n))
        o += (n + 3) // 4 * 4
    return at, o


def _frame_items(case, seed):
    return [_item("torus" if k % 2 else "grid", "skin", n, seed, 1 + k)
            for k, n in enumerate(_sizes(case, case["draws"]))]


def _serve_items(case, seed):
    """The meshes, and the mesh of each request."""
    items = [_item("torus" if k % 2 else "grid", "skin" if k % 4 < 2 else "mvp", n, seed, 1 + k)
             for k, n in enumerate(_sizes(case, case["meshes"]))]
    r = random.Random(case["sizes"] + 1)
    return items, [r.randrange(case["meshes"]) for _ in range(case["requests"])]


def _activity(case, seed):
    """A floor and 8 Gaussians on the torus, quantised to integers."""
    g, w, h = _gen(seed, 7), case["width"], case["height"]
    cx, cy, sig, amp = _rand(8, g) * w, _rand(8, g) * h, 8 + 32 * _rand(8, g), 0.5 + _rand(8, g)
    x = (torch.arange(w, device="cuda").double()[None, :] - cx[:, None]).abs()
    y = (torch.arange(h, device="cuda").double()[None, :] - cy[:, None]).abs()
    x, y = torch.minimum(x, w - x), torch.minimum(y, h - y)
    field = 0.05 + (amp[:, None, None] * torch.exp(-(x[:, None, :] ** 2 + y[:, :, None] ** 2)
                                                   / (2 * sig[:, None, None] ** 2))).sum(0)
    return (field * 4096).round().int().contiguous()


class _Held:
    """A library handle that is given back with the state that holds it."""

    def __init__(self, handle, give_back, *before):
        self.handle, self.give_back, self.before = handle, give_back, before

    def __del__(self):
        try:
            self.give_back(self.handle)
        except Exception:
            pass


def _limits(case):
    return dict(LIMITS[case["limits"]], threads_per_group=case["threads"])


def prepare(case, seed):
    stream = torch.cuda.current_stream()
    kind = case["kind"]
    if kind == "draw":
        it = _item(case["mesh"], case["shader"], case["tris"], seed, 0, case["steps"])
        K = gp.gp_out_floats(SHADERS[case["shader"]])
        ctx = _Held(gp.gp_create(case["variant"], mode=case["mode"], stream=stream, **_limits(case)), gp.gp_destroy)
        part = gp.gp_partition(ctx.handle, it["idx"])[0] if case["mode"] == 1 and case["kept"] else 0
        out = torch.zeros(case["tris"] * 3 * K, dtype=torch.float32, device="cuda")
        return {"kind": kind, "ctx": ctx, "part": part, "it": it, "sid": SHADERS[case["shader"]], "out": out}
    if kind == "frame":
        items = _frame_items(case, seed)
        at, n = _spans(items)
        out = torch.zeros(n, dtype=torch.float32, device="cuda")
        ctx = _Held(gp.gp_create("hash", stream=stream), gp.gp_destroy)
        # a table as the autotuner saves it: voting for small draws, hashing in half and whole blocks above
        row = {"variant": gp.GP_WARP, "mode": 0, "batch_indices": 96, "max_unique": 0, "max_tris": 0,
               "threads_per_group": 0, "batches": 0}
        half = dict(row, variant=gp.GP_HASH, mode=1, batch_indices=0, max_unique=128, threads_per_group=128)
        whole = dict(half, max_unique=256, threads_per_group=256)
        gp.gp_autotune_set_table(ctx.handle, [
            {"shader_id": gp.GP_SHADER_SKIN, "tris_lo": lo, "tris_hi": hi, "config": c}
            for lo, hi, c in ((0, 1024, row), (1024, 8192, half), (8192, 1 << 31, whole))])
        descs = [gp.draw_desc(it["idx"], it["verts"], gp.GP_SHADER_SKIN, it["blob"], out[o:o + m])
                 for it, (o, m) in zip(items, at)]
        frame = _Held(gp.gp_frame_create(ctx.handle, descs), gp.gp_frame_destroy, ctx)
        return {"kind": kind, "ctx": ctx, "frame": frame, "items": items, "out": out}
    if kind == "serve":
        items, reqs = _serve_items(case, seed)
        at, n = _spans([items[k] for k in reqs])
        out = torch.zeros(n, dtype=torch.float32, device="cuda")
        ctx = _Held(gp.gp_create("hash", stream=stream), gp.gp_destroy)
        server = _Held(gp.gp_server_create(ctx.handle), gp.gp_server_destroy, ctx)
        ids = [gp.gp_server_add_mesh(server.handle, it["idx"].cpu().numpy().view(np.uint32), it["verts"].cpu().numpy())
               for it in items]
        todo = [(ids[k], SHADERS[items[k]["shader"]], items[k]["blob"], out[o:o + m]) for k, (o, m) in zip(reqs, at)]
        torch.cuda.synchronize()  # the server draws on its own streams
        return {"kind": kind, "ctx": ctx, "server": server, "todo": todo, "out": out}
    if kind == "walk":
        g, n = _gen(seed, 9), case["agents"]
        start = (torch.randint(0, case["width"], (n,), generator=g, device="cuda") << 16
                 | torch.randint(0, case["height"], (n,), generator=g, device="cuda")).int()
        return {"kind": kind, "case": dict(case), "seed": int(seed), "act": _activity(case, seed), "start": start,
                "pos": torch.empty_like(start), "scratch": torch.empty_like(start), "stream": stream,
                "count": torch.zeros(3, dtype=torch.int64, device="cuda")}
    it = _loop_mesh(case, seed)
    idx, T = it["idx"], it["tris"].shape[0]
    adj = gp.gp_loop_adjacency(idx.cpu().numpy().view(np.uint32), it["verts"].shape[0])
    s = {"kind": kind, "it": it, "adj": [torch.from_numpy(x.view(np.int32)).cuda() for x in adj],
         "out": torch.zeros(36 * T, dtype=torch.float32, device="cuda"), "variant": case["variant"], "more": {},
         "count": torch.zeros(3, dtype=torch.int64, device="cuda"), "stream": stream}
    if case["mode"] == 1:  # dynamic batches of at most 64 triangles and 64 unique vertices, 64 threads
        ctx = gp.gp_create(case["variant"], mode=1, stream=stream, max_unique=64, max_tris=64)
        part, nb = gp.gp_partition(ctx, idx)
        starts = torch.zeros(nb + 1, dtype=torch.int32, device="cuda")
        gp.gp_partition_starts(ctx, part, starts)
        gp.gp_destroy(ctx)
        s["more"] = {"starts": starts, "num_batches": torch.tensor([nb], dtype=torch.int32, device="cuda"),
                     "max_batches": nb, "max_batch_indices": 192, "max_unique": 64, "threads": 64}
    return s


def _loop_mesh(case, seed):
    # whole meshes only: a square torus or grid of about case["tris"] triangles
    w = max(4, int(round(math.sqrt(case["tris"] / 2.0))))
    return _item(case["mesh"], "mvp", 2 * w * w, seed, 0)


def run(s):
    kind = s["kind"]
    if kind == "draw":
        it = s["it"]
        gp.gp_submit_drawcall(s["ctx"].handle, it["idx"], it["verts"], s["sid"], it["blob"], s["out"],
                              partition=s["part"])
        return s["out"]
    if kind == "frame":
        gp.gp_frame_submit(s["frame"].handle, s["ctx"].handle)
        return s["out"]
    if kind == "serve":
        h = s["server"].handle
        for mesh, sid, blob, out in s["todo"]:
            gp.gp_server_submit(h, mesh, sid, blob, out)
        gp.gp_server_wait(h)
        return s["out"]
    if kind == "walk":
        c = s["case"]
        s["pos"].copy_(s["start"])
        s["count"].zero_()
        gp.gp_random_walk(s["act"], s["pos"], s["scratch"], s["count"], c["steps"], s["seed"], variant=c["variant"],
                          batch_agents=c["batch"], threads=c["threads"], stream=s["stream"])
        return {"pos": s["pos"], "count": s["count"]}
    s["count"].zero_()
    gp.gp_loop_subdivide(s["it"]["idx"], s["it"]["verts"], s["adj"], s["out"], s["count"], variant=s["variant"],
                         stream=s["stream"], **s["more"])
    return {"out": s["out"], "count": s["count"]}


# ---------------------------------------------------------------------------
# the same results in 64 bits
# ---------------------------------------------------------------------------

def _shaded(it):
    """Every vertex of an item shaded in float64: [V, 7] or [V, 8]."""
    rows, u = it["verts"], it["values"]
    p, n = rows[:, 0:3].double(), rows[:, 3:6].double()
    if it["shader"] == "envelope":
        h = torch.zeros_like(p[:, 0])
        for a in torch.from_numpy(u["dirs"]).double().cuda():
            x, acc = 0.5 * (p @ a), torch.zeros_like(h)
            for k in range(31, -1, -1):
                acc = acc * x + 1.0 / math.factorial(k)
            h += acc
        off = (float(u["d"]) * h / len(u["dirs"]))[:, None] * n
        one = torch.ones_like(h)[:, None]
        return torch.cat([p - off, one, p + off, one], 1)
    if it["shader"] == "skin":
        ids, w = rows.view(torch.int32)[:, 8], rows[:, 9:13].double()
        pal = torch.from_numpy(u["palette"]).double().cuda()
        q, m = torch.zeros_like(p), torch.zeros_like(n)
        for k in range(4):
            B = pal[((ids >> (8 * k)) & 255).long()]
            q += w[:, k:k + 1] * ((B[:, :, :3] @ p[:, :, None])[:, :, 0] + B[:, :, 3])
            m += w[:, k:k + 1] * (B[:, :, :3] @ n[:, :, None])[:, :, 0]
        p, n = q, m
    M, N = torch.from_numpy(u["M"]).double().cuda(), torch.from_numpy(u["N"]).double().cuda()
    clip, nn = p @ M[:, :3].T + M[:, 3], n @ N.T
    if it["shader"] == "load":
        c, sig = 1e-3 * p[:, 0] + 0.5, torch.ones_like(p[:, 0])
        for _ in range(u["steps"]):
            sig = 0.5 * sig + c
        nn = nn * sig[:, None]
    return torch.cat([clip, nn], 1)


def _drawn(it):
    return _shaded(it)[it["tris"].reshape(-1)].reshape(-1)


def _flat(items):
    at, n = _spans(items)
    out = torch.zeros(n, dtype=torch.float64, device="cuda")
    for it, (o, m) in zip(items, at):
        out[o:o + m] = _drawn(it)
    return out


def _subdivided(it):
    """One Loop step in float64 from the directed edges of an oriented manifold."""
    p, t = it["verts"][:, :3].double(), it["tris"]
    V, T = p.shape[0], t.shape[0]
    a, b, c = t.reshape(-1), t[:, [1, 2, 0]].reshape(-1), t[:, [2, 0, 1]].reshape(-1)  # edge k: (a, b), c opposite
    key, order = torch.sort(a * V + b)
    at = torch.searchsorted(key, b * V + a).clamp_max(3 * T - 1)
    inner = key[at] == b * V + a
    d = c[order[at]]  # the other triangle's third vertex, where there is one
    m = 0.5 * (p[a] + p[b])
    m[inner] = (0.375 * (p[a] + p[b]) + 0.125 * (p[c] + p[d]))[inner]
    total, count = torch.zeros_like(p), torch.zeros(V, dtype=torch.float64, device="cuda")
    total.index_add_(0, a, p[b])
    count.index_add_(0, a, torch.ones_like(p[a, 0]))
    k = count.clamp_min(1)[:, None]
    beta = (0.625 - (0.375 + 0.25 * torch.cos(2 * math.pi / k)) ** 2) / k
    even = (1 - k * beta) * p + beta * total
    rim, ra, rb = torch.zeros_like(p), a[~inner], b[~inner]
    rim.index_add_(0, ra, p[rb])
    rim.index_add_(0, rb, p[ra])
    on = torch.zeros(V, dtype=torch.bool, device="cuda")
    on[ra] = True
    on[rb] = True
    even[on] = (0.75 * p + 0.125 * rim)[on]
    E, M = even[t], m.view(T, 3, 3)
    corners = [E[:, 0], M[:, 0], M[:, 2], E[:, 1], M[:, 1], M[:, 0], E[:, 2], M[:, 2], M[:, 1], M[:, 0], M[:, 1],
               M[:, 2]]
    return torch.stack(corners, 1).reshape(-1)


def exact(case, seed):
    kind = case["kind"]
    if kind == "draw":
        return _drawn(_item(case["mesh"], case["shader"], case["tris"], seed, 0, case["steps"]))
    if kind == "frame":
        return _flat(_frame_items(case, seed))
    if kind == "serve":
        items, reqs = _serve_items(case, seed)
        return _flat([items[k] for k in reqs])
    if kind == "walk":  # whole numbers only
        return None
    return {"out": _subdivided(_loop_mesh(case, seed)), "count": None}


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------

def _mesh_work(tris, shader, steps=0):
    """One draw: every index and referenced vertex read once and shaded once, every output corner written."""
    V = tris / 2
    return (12 * tris + (64 if shader == "skin" else 32) * V + 12 * tris * (8 if shader == "envelope" else 7),
            V * (SHADER_FLOPS[shader] + 2 * steps))


def work(case):
    kind = case["kind"]
    if kind == "draw":
        b, f = _mesh_work(case["tris"], case["shader"], case["steps"])
        return {"bytes": b, "flops": f}
    if kind in ("frame", "serve"):
        if kind == "frame":
            each = [_mesh_work(n, "skin") for n in _sizes(case, case["draws"])]
        else:
            sizes, r = _sizes(case, case["meshes"]), random.Random(case["sizes"] + 1)
            picks = [r.randrange(case["meshes"]) for _ in range(case["requests"])]
            each = [_mesh_work(sizes[k], "skin" if k % 4 < 2 else "mvp") for k in picks]
        return {"bytes": sum(x[0] for x in each), "flops": sum(x[1] for x in each)}
    if kind == "walk":
        # the field once, positions in and out; per agent and step the 8 kept moves' likelihoods and their draw
        return {"bytes": 4 * case["width"] * case["height"] + 8 * case["agents"],
                "flops": 16 * case["agents"] * case["steps"]}
    # per triangle 3 indices, 3 opposite ids and 144 bytes out; per vertex its row, ring (6 ids), offset and flag
    T = case["tris"]
    return {"bytes": T * (24 + 144) + T / 2 * (32 + 24 + 8), "flops": T / 2 * 40 + T * 3 * 15}
