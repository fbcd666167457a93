"""What the framework is timed on: whole calls of the LB-IB step through its
Python entry points (``Sim``, ``lbib_step``, ``lbib_batch_step`` and the
read-outs), over the range of boxes, object loads, storage types and options
its users run.

Every case is a channel of the repository's own configurations, its
benchmark or its tests (the 40x20x20 sphere channel, the 256x128x128 and
512x256x256 red-cell channels, the batch of 64 mixed channels, the serving
requests, the obstacle channel) or a ragged box between them.  Meshes,
placements, starting shapes and body forces come from the seed.

A pass of a single channel starts the run again from given node positions
(``lbib_fluid_init``, ``object_set_nodes``, ``object_set_velocities``), steps
it and reads the result back: a run of a parameter study on one handle.
Starting again also keeps a pass the same however often it is repeated; the
coupled channel itself becomes unstable after 10^4 steps (10^3 for the finest
meshes).  A pass of a batch is one chunk of a scheduler that advances resident
channels: it goes on from where they are, and starts them again once they have
run LIFE steps.
"""
import numpy as np
import torch

from paper_1312_3426_gb300 import lbib

MODULI = dict(ks=0.1, kb=0.03, kal=0.1, kag=0.4, kv=1.0)
FRICTION = 0.05
SCALE_LOG2 = {"f32": 0, "f16s": 12, "bf16s": 12}
BYTES = {"f32": 4, "f16s": 2, "bf16s": 2}
LIFE = 960
REPULSION = ((5e-5, 2.0, 0.3), (1e-6, 1.2, 0.1))


# ------------------------------------------------------------------ the cases

def _channel(nx, ny, nz, objects, storage, steps, level=3, radius=8.0, posts=False, read="nodes"):
    return dict(kind="channel", nx=nx, ny=ny, nz=nz, objects=objects, level=level, radius=radius, posts=posts,
                storage=storage, steps=steps, read=read)


def _batch(sims, box, objects, storage, steps, mix, level=0):
    """level 0: bodies of level 2, 3 or 4 scaled to the box, else `level` and radius 8."""
    return dict(kind="batch", sims=sims, bx=box[0], by=box[1], bz=box[2], objects=objects, storage=storage,
                steps=steps, mix=mix, level=level)


def listed():
    return [
        # the smallest run: one sphere in the 40x20x20 channel, where launches and latencies count
        dict(_channel(40, 20, 20, 1, "f32", 500, level=2, radius=4.0), name="sphere_40x20x20_f32"),
        # fluid alone in an odd, ragged box (start-up flow against the analytic profile), with the fluid read-outs
        dict(_channel(101, 37, 53, 0, "f32", 800, read="fluid"), name="free_101x37x53_f32"),
        # one small serving request, run to completion alone
        dict(_channel(64, 48, 48, 3, "f16s", 400), name="rbc3_64x48x48_f16s"),
        # one middle-sized serving request in a ragged box
        dict(_channel(117, 70, 66, 20, "f32", 300), name="rbc20_117x70x66_f32"),
        # the blood-cell example: posts in the channel, an inflow plane, soft-sphere repulsion, odd width
        dict(_channel(199, 50, 30, 10, "f16s", 300, level=2, radius=5.0, posts=True), name="posts_199x50x30_f16s"),
        # the headline channel in FP32 and in 16-bit storage
        dict(_channel(256, 128, 128, 200, "f32", 384), name="rbc200_256x128x128_f32"),
        dict(_channel(256, 128, 128, 200, "f16s", 384), name="rbc200_256x128x128_f16s"),
        # the largest channel
        dict(_channel(512, 256, 256, 2000, "f32", 128), name="rbc2000_512x256x256_f32"),
        dict(_channel(512, 256, 256, 2000, "bf16s", 128), name="rbc2000_512x256x256_bf16s"),
        # many independent channels of mixed size and load in one batched call
        dict(_batch(64, (128, 64, 64), 40, "f32", 96, 3), name="batch64_f32"),
        # the resident set of the serving loop: one chunk of requests up to 192x96x96
        dict(_batch(24, (192, 96, 96), 100, "f16s", 128, 4, level=3), name="serving24_f16s"),
        # a control loop: every step new forces go in and every object's analysis comes back
        dict(_channel(256, 128, 128, 200, "f32", 128, read="loop"), name="control_256x128x128_f32"),
    ]


def _log_int(rng, lo, hi):
    return int(round(float(np.exp(rng.uniform(np.log(lo), np.log(hi))))))


def draw(rng):
    storage = rng.choice(["f32", "f16s", "bf16s"])
    kind = rng.choice(["channel", "channel", "channel", "free", "posts", "batch", "loop"])
    if kind == "batch":
        wide = rng.random() < 0.5
        return _batch(_log_int(rng, 4, 64 if not wide else 24), (192, 96, 96) if wide else (128, 64, 64),
                      rng.randint(1, 100 if wide else 40), storage, rng.randint(64, 96), rng.randint(10, 10 ** 6), level=3 if wide else 0)
    level = rng.choice([2, 3, 3, 3, 4])
    radius = {2: 4.0, 3: 8.0, 4: 8.0}[level]
    lo = int(2 * radius) + 8
    nx = _log_int(rng, max(40, lo), 512)
    ny, nz = _log_int(rng, max(20, lo), 256), _log_int(rng, max(20, lo), 256)
    if kind == "free":
        nx, ny, nz = _log_int(rng, 24, 512), _log_int(rng, 16, 256), _log_int(rng, 16, 256)
    if kind == "posts":
        nx, ny, nz, level, radius = _log_int(rng, 100, 300), _log_int(rng, 30, 64), _log_int(rng, 30, 64), 2, 5.0
    steps = int(min(500, max(64, 1.6e9 / (nx * ny * nz))))
    sites = _sites(nx, ny, nz, radius)[1]
    share = np.exp(rng.uniform(np.log(0.02), np.log(0.35)))
    objects = 0 if kind == "free" else max(1, min(int(sites * share), 16 if kind == "posts" else 2000))
    read = {"free": "fluid", "loop": "loop"}.get(kind, "nodes")
    return _channel(nx, ny, nz, objects, storage, min(steps, 128) if kind == "loop" else steps, level=level,
                    radius=radius, posts=kind == "posts", read=read)


# ------------------------------------------------------------------ inputs

_MESHES = {}


def _mesh(level, biconcave):
    """Unit icosphere of `level` midpoint subdivisions, or the biconcave
    red-cell profile of Evans and Fung (1972) on it; triangles inward."""
    key = (level, biconcave)
    if key in _MESHES:
        return _MESHES[key]
    t = (1.0 + 5.0 ** 0.5) / 2.0
    v = np.array([[-1, t, 0], [1, t, 0], [-1, -t, 0], [1, -t, 0], [0, -1, t], [0, 1, t], [0, -1, -t], [0, 1, -t],
                  [t, 0, -1], [t, 0, 1], [-t, 0, -1], [-t, 0, 1]], dtype=np.float64)
    # faces: triples of mutually adjacent vertices (edge length 2)
    d2 = np.einsum("ijk,ijk->ij", v[:, None] - v[None], v[:, None] - v[None])
    adj = np.abs(d2 - 4.0) < 1e-9
    f = np.array([(a, b, c) for a in range(12) for b in range(a + 1, 12) for c in range(b + 1, 12)
                  if adj[a, b] and adj[b, c] and adj[a, c]])
    v /= np.linalg.norm(v, axis=1, keepdims=True)
    for _ in range(level):
        e = np.sort(np.concatenate([f[:, [0, 1]], f[:, [1, 2]], f[:, [2, 0]]]), axis=1)
        u, inv = np.unique(e, axis=0, return_inverse=True)
        m = 0.5 * (v[u[:, 0]] + v[u[:, 1]])
        m /= np.linalg.norm(m, axis=1, keepdims=True)
        ab, bc, ca = (inv.reshape(-1) + len(v)).reshape(3, -1)
        v = np.concatenate([v, m])
        f = np.concatenate([np.stack(s, 1) for s in ((f[:, 0], ab, ca), (f[:, 1], bc, ab), (f[:, 2], ca, bc),
                                                     (ab, bc, ca))])
    n = np.cross(v[f[:, 1]] - v[f[:, 0]], v[f[:, 2]] - v[f[:, 0]])
    out = np.einsum("ij,ij->i", n, v[f].mean(1)) > 0
    f[out] = f[out][:, [0, 2, 1]]
    if biconcave:
        r2 = np.clip(v[:, 0] ** 2 + v[:, 1] ** 2, 0.0, 1.0)
        v[:, 2] *= 0.5 * (0.2072 + 2.0026 * r2 - 1.1228 * r2 * r2)
    _MESHES[key] = (v, f.astype(np.int32))
    return _MESHES[key]


def _sites(nx, ny, nz, radius):
    """Sites of a grid on which spheres of this radius stay 2 apart and 2
    from the walls: counts per axis, and all."""
    s = 2.0 * radius + 2.0
    n = (int(nx // s), max(0, int((ny - 2.0 - s - 2.0) // s) + 1), int(nz // s))
    return n, n[0] * n[1] * n[2]


def _rotations(rng, n):
    q = rng.standard_normal((n, 4))
    w, x, y, z = (q / np.linalg.norm(q, axis=1, keepdims=True)).T
    return np.array([[1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y)],
                     [2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x)],
                     [2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)]]).transpose(2, 0, 1)


def _scene(nx, ny, nz, objects, level, radius, posts, rng):
    """Box, template and node positions of one channel: `objects` bodies on
    random grid sites with a jitter, turned at random and slightly stretched
    at constant volume, so that every membrane force is at work."""
    s = dict(nx=nx, ny=ny, nz=nz, force=(float(rng.uniform(0.5e-5, 1.5e-5)), 0.0, 0.0), solid=None, inlet=None)
    if posts:
        solid = np.zeros((nz, ny, nx), dtype=bool)
        for p in range(3):
            x0, z0 = int((p + 0.5) * nx / 3) + int(rng.integers(-2, 3)), int(rng.uniform(0.1, 0.5) * nz)
            solid[z0:z0 + max(3, nz // 5), 1:ny - 1, x0 - 2:x0 + 2] = True
        s["solid"], s["inlet"] = solid, ((0, 1, 1, ny - 1, 0, nz), (float(rng.uniform(0.005, 0.01)), 0.0, 0.0))
    n, total = _sites(nx, ny, nz, radius)
    count = min(objects, total)
    s["tpl"] = s["X"] = None
    if count:
        pick = rng.permutation(total)
        i = np.stack([pick % n[0], pick // n[0] % n[1], pick // (n[0] * n[1])], 1).astype(np.float64)
        pitch = np.array([nx / n[0], (ny - 4.0) / n[1], nz / n[2]])
        slack = 0.5 * (pitch - 2.0 * radius - 2.0)
        c = (i + 0.5) * pitch + np.array([0.0, 2.0, 0.0]) + rng.uniform(-1.0, 1.0, (total, 3)) * slack
        if posts:  # bodies start clear of the posts
            post = np.argwhere(solid[:, ny // 2])[:, ::-1] + 0.5
            d = c[:, None, [0, 2]] - post[None]
            d -= np.array([nx, nz]) * np.round(d / np.array([nx, nz]))
            c = c[np.sqrt((d * d).sum(-1)).min(1) > radius + 1.5]
        c = c[:count]
        count = len(c)
        x, tris = _mesh(level, level > 2 or radius > 4.0)
        a = 1.0 + rng.uniform(-0.02, 0.02, (count, 3))
        a[:, 2] = 1.0 / (a[:, 0] * a[:, 1])
        X = np.einsum("oij,oj,nj->oni", _rotations(rng, count), a * radius, x) + c[:, None]
        s["tpl"], s["X"] = (x, tris, radius), np.ascontiguousarray(X)
    return s


def _batch_shapes(case):
    """Box and load of every channel of a batch (the same for every seed):
    box log-uniform from 32 up, 0 to `objects` bodies of level 2 to 4."""
    rng = np.random.default_rng(case["mix"])
    out = []
    for _ in range(case["sims"]):
        nx, ny, nz = (int(round(np.exp(rng.uniform(np.log(32), np.log(case[b]))))) for b in ("bx", "by", "bz"))
        level, count = int(rng.integers(2, 5)), int(rng.integers(0, case["objects"] + 1))
        radius, inner = 8.0, min(nx, ny - 2, nz)
        if case["level"]:
            level = case["level"]
        else:  # mean edge 0.55 or more: finer meshes make the explicit membrane update unstable
            radius = min(8.0, max(3.0, 0.2 * inner))
            while level > 2 and 2.0 * max(radius, 0.55 * 2 ** level / 1.05) + 6.0 > inner:
                level -= 1
            radius = max(radius, 0.55 * 2 ** level / 1.05)
        out.append((nx, ny, nz, count, level, radius))
    return out


def _scenes(case, seed):
    rng = np.random.default_rng([int(seed), 1312])
    if case["kind"] == "batch":
        return [_scene(*shape, False, rng) for shape in _batch_shapes(case)]
    return [_scene(case["nx"], case["ny"], case["nz"], case["objects"], case["level"], case["radius"], case["posts"],
                   rng)]


def _loop_forces(case, seed, n_obj):
    return np.random.default_rng([int(seed), 3426]).uniform(-2e-5, 2e-5, (case["steps"], n_obj, 3))


def _sim(s, storage):
    g = lbib.Sim(s["nx"], s["ny"], s["nz"], body_force=s["force"], friction=FRICTION, precision=storage,
                 pop_scale_log2=SCALE_LOG2[storage])
    if s["X"] is not None:
        x, tris, radius = s["tpl"]
        g.template_create(x, tris, (radius,) * 3, **MODULI)
        for o in range(len(s["X"])):
            g.object_add(0, s["X"][o].mean(0))
            g.object_set_nodes(o, s["X"][o])
    if s["solid"] is not None:
        lbib.lbib_set_solid(g.h, s["solid"])
        lbib.lbib_set_inlet(g.h, *s["inlet"])
        lbib.lbib_set_repulsion(g.h, *REPULSION)
    g.fluid_init()
    return g


def prepare(case, seed):
    scenes = _scenes(case, seed)
    st = dict(case=case, scenes=scenes, sims=[_sim(s, case["storage"]) for s in scenes])
    st["handles"] = [g.h for g in st["sims"]]
    st["run"] = 0
    if case.get("read") == "loop":
        st["forces"] = _loop_forces(case, seed, len(scenes[0]["X"]))
    return st


def _start_again(g, s):
    g.fluid_init()
    if s["X"] is not None:
        at_rest = np.zeros(s["X"].shape[1:])
        for o in range(len(s["X"])):
            g.object_set_nodes(o, s["X"][o])
            g.object_set_velocities(o, at_rest)


# ------------------------------------------------------------------ one pass

def run(st):
    case = st["case"]
    if case["kind"] == "batch":
        if st["run"] + case["steps"] > LIFE:
            for g, s in zip(st["sims"], st["scenes"]):
                _start_again(g, s)
            st["run"] = 0
        st["run"] += case["steps"]
        lbib.lbib_batch_step(st["handles"], case["steps"])
        read = [g.read_nodes() for g in st["sims"] if g.obj_tid]
        return {"nodes": np.concatenate([r[0] for r in read]) if read else np.zeros((0, 3)),
                "node_velocities": np.concatenate([r[1] for r in read]) if read else np.zeros((0, 3)),
                "velocity": np.concatenate([g.velocity().reshape(-1) for g in st["sims"]])}
    g, s = st["sims"][0], st["scenes"][0]
    _start_again(g, s)
    out = {}
    if case["read"] == "loop":
        # step k's analysis is read while step k + 1 runs
        n, rec = len(s["X"]), np.empty((case["steps"], len(s["X"]), 14))
        for k in range(case["steps"]):
            g.objects_set_force(st["forces"][k])
            g.step(1)
            lbib.lbib_objects_analyze_async(g.h, k & 1)
            if k:
                lbib.lbib_objects_analyze_wait(g.h, (k - 1) & 1, n, rec[k - 1])
        lbib.lbib_objects_analyze_wait(g.h, (case["steps"] - 1) & 1, n, rec[case["steps"] - 1])
        out["analysis"] = rec
    else:
        g.step(case["steps"])
    if s["X"] is not None:
        out["nodes"], out["node_velocities"] = g.read_nodes()
    out["velocity"] = g.velocity()
    if case["read"] == "fluid":
        out["density"], out["mass"] = g.density(), g.mass()
    return out


def work(case):
    """Per step: every stored population read once and written once, and per
    node its position and velocity in and out (48 bytes each way).  About 250
    operations per cell, 150 per node, 150 per edge and 100 per triangle."""
    if case["kind"] == "batch":
        shapes = _batch_shapes(case)
    else:
        shapes = [(case["nx"], case["ny"], case["nz"], case["objects"], case["level"], case["radius"])]
    cells = nodes = 0
    for nx, ny, nz, objects, level, radius in shapes:
        cells += nx * (ny - 2) * nz
        nodes += min(objects, _sites(nx, ny, nz, radius)[1]) * (10 * 4 ** level + 2)
    return {"bytes": case["steps"] * (cells * 38 * BYTES[case["storage"]] + nodes * 96),
            "flops": case["steps"] * (cells * 250 + nodes * (150 + 3 * 150 + 2 * 100))}


# ------------------------------------------------------------------ 64 bits

def exact(case, seed):
    """The same run in 64 bits with plain torch: pull streaming, BGK with
    Guo's force, the five membrane forces, trilinear coupling."""
    scenes = _scenes(case, seed)
    forces = _loop_forces(case, seed, len(scenes[0]["X"])) if case.get("read") == "loop" else None
    got = [_Run64(s).go(case["steps"], forces) for s in scenes]
    if case["kind"] == "batch":
        return {"nodes": np.concatenate([r.X for r in got if len(r.X)]) if any(len(r.X) for r in got) else
                np.zeros((0, 3)),
                "node_velocities": np.concatenate([r.V for r in got if len(r.X)]) if any(len(r.X) for r in got) else
                np.zeros((0, 3)),
                "velocity": np.concatenate([r.u.reshape(-1) for r in got])}
    r = got[0]
    out = {"velocity": r.u}
    if len(r.X):
        out["nodes"], out["node_velocities"] = r.X, r.V
    if forces is not None:
        out["analysis"] = r.records
    if case["read"] == "fluid":
        out["density"], out["mass"] = r.rho, r.mass
    return out


class _Run64:
    def __init__(self, s):
        self.s = s
        self.dev = "cuda" if torch.cuda.is_available() else "cpu"
        self.e = [(x, y, z) for x in (-1, 0, 1) for y in (-1, 0, 1) for z in (-1, 0, 1) if x * x + y * y + z * z < 3]
        self.E = self.t(np.array(self.e, dtype=np.float64))
        self.w = self.t(np.array([(1 / 3, 1 / 18, 1 / 36)[x * x + y * y + z * z] for x, y, z in self.e])[:, None])
        self.shape = (s["nz"], s["ny"] - 2, s["nx"])
        self.solid = self.t(s["solid"][:, 1:-1]).reshape(-1) if s["solid"] is not None else None
        self.source = self.sources()

    def t(self, a):
        return torch.as_tensor(np.ascontiguousarray(a), device=self.dev)

    def go(self, steps, forces):
        s, zyx = self.s, self.shape
        n = zyx[0] * zyx[1] * zyx[2]
        h = torch.zeros((19, n), dtype=torch.float64, device=self.dev)
        u = torch.zeros((3, n), dtype=torch.float64, device=self.dev)
        bodies = s["X"] is not None
        if bodies:
            X = self.t(s["X"])
            V = torch.zeros_like(X)
            self.template()
        records = []
        for k in range(steps):
            G = self.t(np.float32(s["force"]).astype(np.float64))[:, None]
            if bodies:
                F = self.membrane(X) + (self.repulsion(X) if s["solid"] is not None else 0.0)
                drag, spread = self.couple(X.reshape(-1, 3), V.reshape(-1, 3), u)
                G = G + spread
                V = V + F + drag.reshape(X.shape)
                if forces is not None:
                    V = V + self.t(forces[k]).float().double()[:, None]
                X = X + V
            h, u, rho = self.fluid(h, G)
            if forces is not None:
                records.append(self.analyse(X, V))
        pad = lambda a, v: np.pad(a.reshape(a.shape[:-1] + zyx).cpu().numpy(),  # noqa: E731
                                  ((0, 0),) * a.dim() + ((1, 1), (0, 0)), constant_values=v)
        cells = n - (int(self.solid.sum()) if self.solid is not None else 0)
        self.u, self.rho, self.mass = pad(u, 0.0), pad(rho, 1.0), float(cells + h.sum())
        self.X, self.V = (a.reshape(-1, 3).cpu().numpy() if bodies else np.zeros((0, 3)) for a in
                          ((X, V) if bodies else (None, None)))
        self.records = torch.stack(records).cpu().numpy() if records else None
        return self

    # ---- fluid
    def sources(self):
        """Where population q of each cell comes from, in the flat [19][cells]
        array: cell - e_q, or the cell's own opposite one at a wall or post."""
        nz, nyf, nx = self.shape
        n = nz * nyf * nx
        cell = torch.arange(n, device=self.dev)
        x, y, z = cell % nx, cell // nx % nyf, cell // (nx * nyf)
        out = torch.empty((19, n), dtype=torch.int64, device=self.dev)
        for q, (ex, ey, ez) in enumerate(self.e):
            from_y = y - ey
            c = ((z - ez) % nz * nyf + from_y.clamp(0, nyf - 1)) * nx + (x - ex) % nx
            back = (from_y < 0) | (from_y >= nyf)
            if self.solid is not None:
                back |= self.solid[c]
            out[q] = torch.where(back, self.e.index((-ex, -ey, -ez)) * n + cell, q * n + c)
        return out.reshape(-1)

    def along(self, v):
        """e_q . v for every direction."""
        out = self.E[:, 0, None] * v[0]
        return out.addcmul_(self.E[:, 1, None], v[1]).addcmul_(self.E[:, 2, None], v[2])

    def fluid(self, h, F):
        g = h.reshape(-1)[self.source].reshape(h.shape)
        if self.s["inlet"] is not None:
            (x0, x1, y0, y1, z0, z1), v = self.s["inlet"]
            v = self.t(np.float32(v).astype(np.float64))
            at = g.reshape((19,) + self.shape)[:, z0:z1, y0 - 1:y1 - 1, x0:x1]
            drho, eu = at.sum(0), (self.E @ v)[:, None, None, None]
            at.copy_(self.w[..., None, None] * (drho + (1 + drho) * (3 * eu + 4.5 * eu * eu - 1.5 * (v @ v))))
        drho = g.sum(0)
        rho = 1.0 + drho
        u = (torch.stack([(self.E[:, k, None] * g).sum(0) for k in range(3)]) + 0.5 * F) / rho
        eu, eF = self.along(u), self.along(F)
        # tau = 1: the equilibrium plus Guo's force term at half weight
        g = self.w * (drho + rho * (3 * eu + 4.5 * eu * eu - 1.5 * (u * u).sum(0)) +
                      0.5 * (3 * (eF - (u * F).sum(0)) + 9 * eu * eF))
        if self.solid is not None:
            g[:, self.solid] = 0.0
            u[:, self.solid] = 0.0
            rho = torch.where(self.solid, torch.zeros_like(rho), rho)
        return g, u, rho

    # ---- coupling
    def couple(self, X, V, u):
        """Drag on every node, and the force spread onto the cells."""
        nz, nyf, nx = self.shape
        d = self.t(np.array([(k & 1, k >> 1 & 1, k >> 2 & 1) for k in range(8)]))[:, None]
        i0 = torch.floor(X - 0.5)
        f = X - 0.5 - i0
        w = torch.where(d == 1, f, 1 - f).prod(-1)
        i = i0.long() + d
        y = i[..., 1] - 1
        c = (i[..., 2] % nz * nyf + y.clamp(0, nyf - 1)) * nx + i[..., 0] % nx
        w = w * ((y >= 0) & (y < nyf))
        if self.solid is not None:
            w = w * ~self.solid[c]
        v = (w * u[:, c]).sum(1).T
        drag = float(np.float32(FRICTION)) * (v - V)
        spread = torch.zeros_like(u)
        spread.index_add_(1, c.reshape(-1), -(w[..., None] * drag).reshape(-1, 3).T)
        return drag, spread

    # ---- membranes
    def template(self):
        x, tris, radius = self.s["tpl"]
        x = self.t(x * radius)[None]
        self.tri = t = self.t(tris.astype(np.int64))
        owner = {}
        for a, b, c in tris.tolist():
            for i, j, k in ((a, b, c), (b, c, a), (c, a, b)):
                owner[(i, j)] = k  # triangle (k, i, j)
        quads = [(owner[(b, c)], b, c, owner[(c, b)]) for b, c in owner if b < c]
        self.quad = self.t(np.array(quads, dtype=np.int64))
        self.L0 = (x[:, self.quad[:, 1]] - x[:, self.quad[:, 2]]).norm(dim=-1)
        self.theta0 = self.angle(x)[0]
        self.S0 = self.normals(x, t).norm(dim=-1) / 2
        self.Sg0, self.V0 = self.S0.sum(), self.volume(x)

    @staticmethod
    def normals(x, t):
        a = x[:, t[:, 0]]
        return torch.linalg.cross(x[:, t[:, 1]] - a, x[:, t[:, 2]] - a)

    def volume(self, x):
        r = x - x[:, :1]
        return -(r[:, self.tri[:, 0]] * self.normals(r, self.tri)).sum((-1, -2)) / 6

    def angle(self, x):
        a, b, c, d = (x[:, self.quad[:, k]] for k in range(4))
        n1, n2 = torch.linalg.cross(b - a, c - a), torch.linalg.cross(c - d, b - d)
        n1, n2 = n1 / n1.norm(dim=-1, keepdim=True), n2 / n2.norm(dim=-1, keepdim=True)
        alpha = torch.atan2(torch.linalg.cross(n1, n2).norm(dim=-1), (n1 * n2).sum(-1))
        return torch.where(((d - b) * n1).sum(-1) > 0, np.pi - alpha, np.pi + alpha), n1, n2

    def membrane(self, x):
        m = {k: float(np.float32(v)) for k, v in MODULI.items()}
        F = torch.zeros_like(x)
        q, t = self.quad, self.tri
        c = x[:, q[:, 2]] - x[:, q[:, 1]]
        L = c.norm(dim=-1)
        lam = L / self.L0
        kap = (lam ** 0.5 + lam ** -2.5) / (lam + lam ** -3)
        f = (m["ks"] * kap * (L - self.L0) / self.L0 / L)[..., None] * c
        theta, n1, n2 = self.angle(x)
        s = (m["kb"] * (theta / self.theta0 - 1))[..., None]
        F.index_add_(1, q[:, 0], s * n1)
        F.index_add_(1, q[:, 3], s * n2)
        F.index_add_(1, q[:, 1], f - 0.5 * s * (n1 + n2))
        F.index_add_(1, q[:, 2], -f - 0.5 * s * (n1 + n2))
        N = self.normals(x, t)
        S = N.norm(dim=-1) / 2
        Sg = S.sum(-1, keepdim=True)
        w = -m["kal"] * (S - self.S0) / S - m["kag"] * (Sg - self.Sg0) / Sg
        dV = (self.volume(x) / self.V0 - 1)[:, None]
        fv = (m["kv"] * dV / 6)[..., None] * N
        centre = (x[:, t[:, 0]] + x[:, t[:, 1]] + x[:, t[:, 2]]) / 3
        for k in range(3):
            r = x[:, t[:, k]] - centre
            F.index_add_(1, t[:, k], w[..., None] * r / r.norm(dim=-1, keepdim=True) + fv)
        return F

    def repulsion(self, X):
        """Soft spheres between nodes of different bodies, and at the walls."""
        (a, n, rc), (wa, wn, wrc) = (tuple(float(np.float32(v)) for v in p) for p in REPULSION)
        x = X.reshape(-1, 3)
        body = torch.arange(len(X), device=self.dev).repeat_interleave(X.shape[1])
        F = torch.zeros_like(x)
        L = torch.tensor([self.s["nx"], 1e30, self.s["nz"]], dtype=torch.float64, device=self.dev)
        for lo in range(0, len(x), 2048):
            d = x[lo:lo + 2048, None] - x[None]
            d = d - L * torch.round(d / L)
            r = d.norm(dim=-1)
            near = (r < rc) & (r > 0) & (body[lo:lo + 2048, None] != body[None])
            i, j = near.nonzero(as_tuple=True)
            F.index_add_(0, i + lo, (a * n * r[i, j] ** -(n + 2))[:, None] * d[i, j])
        low, high = x[:, 1] - 1.0, self.s["ny"] - 1.0 - x[:, 1]
        push = lambda d: torch.where(d < wrc, wa * wn * d.clamp(min=1e-3) ** -(wn + 1), torch.zeros_like(d))  # noqa: E731
        F[:, 1] += push(low) - push(high)
        return F.reshape(X.shape)

    def analyse(self, X, V):
        lo, hi = X.amin(1), X.amax(1)
        area = self.normals(X, self.tri).norm(dim=-1).sum(-1, keepdim=True) / 2
        return torch.cat([X.mean(1), torch.stack([lo, hi], -1).reshape(len(X), 6), self.volume(X)[:, None], area,
                          V.mean(1)], 1)
