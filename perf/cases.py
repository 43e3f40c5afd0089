"""The workloads whose speed is followed: contact steps over the range of sizes,
types and options that programs use, each through the library's public calls.

    listed()             the cases, dicts of plain values with a name
    draw(rng)            one more case of the same ranges
    prepare(case, seed)  inputs on the GPU (or in host memory) and the context a program keeps
    run(state)           one pass through the public entry points, and its outputs
    work(case)           bytes and operations one pass cannot do without
    exact(case, seed)    what run() returns, in 64 bits, from plain torch

Scenes are made from the seed: jittered lattices (node spacing h/2, the
paper's grid of twice the element size) cut to boxes and ellipsoids, turned at
random, in pairs that approach along x and touch, with rigid motions plus a
few per cent of vibration, area-like unit normals on surface nodes and 0
inside.
"""
import math

import numpy as np
import torch

from paper_2108_02259_gb300 import apic

DEV = "cuda" if torch.cuda.is_available() else "cpu"

_STEP = dict(kind="step", nodes=200_000, bodies=4, h=1 / 256, n_iter=8, dtype="float32", friction="scalar",
             normals="given", deterministic=False, memory="device")


def _step(name, **kw):
    return {"name": name, **_STEP, **kw}


def listed():
    return [
        # two 8^3-node cubes: the smallest scene in use (one launch-bound step of an interactive program)
        _step("two_cubes_1k", nodes=1024, bodies=2, h=1 / 32, n_iter=10),
        # a small impact with the single augury term (N = 1) the paper runs, a mesh size that is no power of two
        _step("impact_17k_n1", nodes=17_003, bodies=2, h=0.011, n_iter=1),
        # the ordinary scene: two boxes and two balls
        _step("four_bodies_200k", nodes=200_000),
        # normals from the grid mass, for a caller that has neither normals nor a mesh; odd sizes, three bodies
        _step("mass_normals_600k", nodes=600_011, bodies=3, h=1 / 512, n_iter=4, normals="mass"),
        # the largest scene one call steps in the benchmark, friction per pair of bodies
        _step("eight_bodies_4m", nodes=4_000_000, bodies=8, h=1 / 512, friction="pair"),
        # the bitwise reproducible mode
        _step("deterministic_200k", nodes=199_999, deterministic=True),
        # double precision, for validation and stiff problems
        _step("fp64_50k", nodes=50_021, dtype="float64"),
        # a host program whose arrays are page-locked numpy arrays
        _step("host_arrays_200k", nodes=200_000, memory="host"),
        # many independent scenes in one call, as a parameter study or the serving loop steps them
        dict(name="batch_64_scenes", kind="batch", scenes=64, min_nodes=1_000, max_nodes=200_000, n_iter=8),
        # a few small ones: an early, uneven batch of the serving loop
        dict(name="batch_9_small", kind="batch", scenes=9, min_nodes=1_000, max_nodes=9_000, n_iter=8),
        # the contact step inside the explicit time integrator: elastic blocks on springs, normals from their meshes
        dict(name="augury_128k", kind="augury", side=40, n_iter=4, steps=4, dtype="float32"),
        # normals of the surface mesh of a large block, as each step of a moving mesh needs them
        dict(name="node_normals_1m", kind="normals", nx=100, ny=100, nz=100, dtype="float32"),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    pick = rng.random()
    if pick < 0.60:
        c = dict(_STEP)
        c["nodes"] = _log_uniform(rng, 1_000, 4_000_000) | 1
        c["bodies"] = rng.randint(2, 8)
        c["h"] = rng.choice([1 / 64, 1 / 128, 1 / 256, 1 / 512, 0.004, 0.0123])
        c["n_iter"] = rng.choice([1, 2, 4, 8, 8, 10])
        c["friction"] = rng.choice(["scalar", "scalar", "pair"])
        option = rng.random()
        if option < 0.15:
            c["normals"] = "mass"
        elif option < 0.30:
            c["deterministic"] = True
        elif option < 0.45:
            c["dtype"], c["nodes"] = "float64", _log_uniform(rng, 1_000, 300_000) | 1
        elif option < 0.55:
            c["memory"], c["nodes"] = "host", _log_uniform(rng, 1_000, 1_000_000) | 1
        return c
    if pick < 0.80:
        lo = _log_uniform(rng, 1_000, 10_000)
        return dict(kind="batch", scenes=rng.randint(2, 64), min_nodes=lo, max_nodes=_log_uniform(rng, lo, 150_000),
                    n_iter=rng.choice([2, 4, 8]))
    if pick < 0.90:
        return dict(kind="augury", side=rng.randint(8, 48), n_iter=rng.choice([1, 2, 4]), steps=rng.randint(2, 4),
                    dtype=rng.choice(["float32", "float32", "float64"]))
    return dict(kind="normals", nx=rng.randint(10, 110), ny=rng.randint(10, 110), nz=rng.randint(10, 110),
                dtype=rng.choice(["float32", "float64"]))


# ------------------------------------------------------------------ inputs


def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) * 7919 + 12345)
    return g


def _rotation(host):
    q, r = np.linalg.qr(host.standard_normal((3, 3)))
    q = q * np.sign(np.diag(r))
    if np.linalg.det(q) < 0:
        q[:, 0] = -q[:, 0]
    return torch.as_tensor(q, dtype=torch.float64, device=DEV)


def _direction(host):
    d = host.standard_normal(3)
    return d / np.linalg.norm(d)


def _body(host, gen, count, spacing, shape):
    """`count` lattice points innermost in a box or an ellipsoid, jittered, and their outward normals."""
    axes = host.uniform(0.6, 1.0, 3)
    vol = (4.0 / 3.0 * math.pi if shape == "ellipsoid" else 8.0) * float(np.prod(axes))
    radius = (count * spacing**3 / vol) ** (1.0 / 3.0) * 1.15
    ext = [int(math.ceil(radius * a / spacing)) + 2 for a in axes]
    grids = [torch.arange(-e, e + 1, device=DEV) for e in ext]
    lat = torch.stack([t.reshape(-1) for t in torch.meshgrid(*grids, indexing="ij")], 1)
    ax = torch.as_tensor(axes, device=DEV) * radius
    q = lat.to(torch.float64) * spacing / ax
    level = q.square().sum(1).sqrt() if shape == "ellipsoid" else q.abs().amax(1)
    keep = torch.argsort(level, stable=True)[:count]
    if shape != "ellipsoid":
        keep = keep.sort().values  # a box keeps its lattice numbering, a ball is numbered from its centre out
    lat, q = lat[keep], q[keep]
    occ = torch.zeros([2 * e + 3 for e in ext], dtype=torch.bool, device=DEV)
    li = lat + torch.as_tensor(ext, device=DEV) + 1
    occ[li[:, 0], li[:, 1], li[:, 2]] = True
    surface = torch.zeros(count, dtype=torch.bool, device=DEV)
    for k in range(3):
        for s in (-1, 1):
            nb = li.clone()
            nb[:, k] += s
            surface |= ~occ[nb[:, 0], nb[:, 1], nb[:, 2]]
    if shape == "ellipsoid":
        g = q / ax
    else:
        g = torch.where(q.abs() >= q.abs().amax(1, keepdim=True) - 1e-12, torch.sign(q), torch.zeros_like(q))
    g = g / g.norm(dim=1, keepdim=True).clamp_min(1e-300)
    normal = torch.where(surface[:, None], g, torch.zeros_like(g))
    jitter = (torch.rand(count, 3, generator=gen, device=DEV, dtype=torch.float64) * 2 - 1) * (0.2 * spacing)
    return lat.to(torch.float64) * spacing + jitter, normal


def _scene(seed, nodes, bodies, h, dtype, pair_friction=False):
    """x, v, C, m, normals, body ids of one scene, its scalar friction and (or None) its friction table."""
    host, gen = np.random.default_rng([2108, int(seed)]), _gen(seed)
    per = [nodes // bodies + (1 if b < nodes % bodies else 0) for b in range(bodies)]
    made = []
    for b in range(bodies):
        pts, nrm = _body(host, gen, per[b], h / 2, "ellipsoid" if b % 2 else "box")
        R = _rotation(host)
        made.append((pts @ R.T, nrm @ R.T))
    pitch = 1.1 * max(float((p.amax(0) - p.amin(0)).max()) for p, _ in made) + 6 * h
    cols = max(1, math.isqrt((bodies + 1) // 2))
    xs, vs, Cs, ms, ns, ids = [], [], [], [], [], []
    for b, (pts, nrm) in enumerate(made):
        side = 1.0 if b % 2 == 0 else -1.0
        if b % 2 == 0:
            gap = host.uniform(-1.0, 1.0) * h
        edge = float(pts[:, 0].amax() if side > 0 else pts[:, 0].amin())
        pair = b // 2
        c = torch.as_tensor([0.5 - edge - side * gap / 2, 0.4 + pitch * (pair % cols), 0.4 + pitch * (pair // cols)],
                            dtype=torch.float64, device=DEV)
        v0 = _direction(host) * host.uniform(0, 2)
        v0[0] = side * abs(v0[0])
        w = _direction(host) * host.uniform(0, 5)
        skew = torch.as_tensor([[0, -w[2], w[1]], [w[2], 0, -w[0]], [-w[1], w[0], 0]], dtype=torch.float64, device=DEV)
        n = pts.shape[0]
        v = torch.as_tensor(v0, device=DEV) + pts @ skew.T
        v = v + 0.02 * torch.randn(n, 3, generator=gen, device=DEV, dtype=torch.float64)
        C = skew + 0.2 * torch.randn(n, 3, 3, generator=gen, device=DEV, dtype=torch.float64)
        m = torch.exp(0.3 * torch.randn(n, generator=gen, device=DEV, dtype=torch.float64))
        xs.append(pts + c)
        vs.append(v)
        Cs.append(C)
        ms.append(m / m.sum())
        ns.append(nrm)
        ids.append(torch.full((n,), b, dtype=torch.int32, device=DEV))
    x, body = torch.cat(xs).contiguous(), torch.cat(ids)
    v, C, m, nrm = (torch.cat(t).to(dtype).contiguous() for t in (vs, Cs, ms, ns))
    table = None
    if pair_friction:
        table = host.uniform(0.1, 0.5, (bodies, bodies))
        table = np.triu(table) + np.triu(table, 1).T
    return dict(x=x, v=v, C=C, m=m, nrm=nrm, body=body, h=h, mu=0.3, mu_pair=table, bodies=bodies)


def _step_scene(case, seed):
    return _scene(seed, case["nodes"], case["bodies"], case["h"], getattr(torch, case["dtype"]),
                  case["friction"] == "pair")


def _batch_scenes(case, seed):
    host = np.random.default_rng([4, int(seed)])
    out = []
    for i in range(case["scenes"]):
        # the sizes are the case's own: every seed steps the same mix
        u = (i + 0.5) / case["scenes"]
        nodes = int(math.exp(math.log(case["min_nodes"]) + u * math.log(case["max_nodes"] / case["min_nodes"])))
        h = [1 / 64, 1 / 128, 1 / 256][i % 3]
        out.append(_scene(int(host.integers(1 << 30)), nodes, 2 + i % 5, h, torch.float32))
    return out


def _lattice_mesh(nx, ny, nz):
    """Node ids of a lattice (x fastest) and the triangles of its boundary, wound outwards."""
    idx = torch.arange(nx * ny * nz, dtype=torch.int32, device=DEV).reshape(nz, ny, nx)
    tri = []
    for d in range(3):
        for end in (0, 1):
            f = idx.select(2 - d, idx.shape[2 - d] - 1 if end else 0)
            a, b, c, e = f[:-1, :-1], f[:-1, 1:], f[1:, 1:], f[1:, :-1]
            # with axes (slow, fast) of the face, a -> b runs along the fast one
            flip = (d == 1) != (end == 0)
            for t in ((a, b, c), (a, c, e)):
                t = t if not flip else (t[0], t[2], t[1])
                tri.append(torch.stack([s.reshape(-1) for s in t], 1))
    return idx, torch.cat(tri).contiguous()


def _elastic(case, seed):
    """Two elastic lattice blocks on springs that meet: arrays of the time integrator."""
    n, dtype = case["side"], getattr(torch, case["dtype"])
    spacing, speed = 1 / 256, 12.0
    h = 2 * spacing
    gen = _gen(seed)
    idx, tri = _lattice_mesh(n, n, n)
    lat = torch.stack([t.reshape(-1) for t in torch.meshgrid(*[torch.arange(n, device=DEV)] * 3, indexing="ij")], 1)
    lat = (lat.flip(1).to(torch.float64) - (n - 1) / 2) * spacing
    half = (n - 1) * spacing / 2 + 0.25 * h
    nb = n**3
    x = torch.cat([lat + torch.tensor([0.5 - half, 0.5, 0.5], device=DEV, dtype=torch.float64),
                   lat + torch.tensor([0.5 + half, 0.5, 0.5], device=DEV, dtype=torch.float64)])
    x = x + (torch.rand(x.shape, generator=gen, device=DEV, dtype=torch.float64) - 0.5) * (0.02 * spacing)
    k_axis = (1.0 / nb) / spacing**3 * speed**2 * spacing
    pairs, rest, k = [], [], []

    def add(a, b, length, stiffness):
        p = torch.stack([a.reshape(-1), b.reshape(-1)], 1)
        pairs.append(p)
        rest.append(torch.full((p.shape[0],), length, dtype=torch.float64, device=DEV))
        k.append(torch.full((p.shape[0],), stiffness, dtype=torch.float64, device=DEV))

    d = spacing * math.sqrt(2.0)
    add(idx[:, :, :-1], idx[:, :, 1:], spacing, k_axis)
    add(idx[:, :-1, :], idx[:, 1:, :], spacing, k_axis)
    add(idx[:-1], idx[1:], spacing, k_axis)
    for a, b in ((idx[:, :-1, :-1], idx[:, 1:, 1:]), (idx[:, :-1, 1:], idx[:, 1:, :-1]),
                 (idx[:-1, :, :-1], idx[1:, :, 1:]), (idx[:-1, :, 1:], idx[1:, :, :-1]),
                 (idx[:-1, :-1], idx[1:, 1:]), (idx[:-1, 1:], idx[1:, :-1])):
        add(a, b, d, 0.5 * k_axis)
    springs, rest, k = torch.cat(pairs), torch.cat(rest), torch.cat(k)
    v = torch.zeros_like(x)
    v[:nb, 0], v[nb:, 0] = 1.0, -1.0
    v = v + 0.02 * torch.randn(v.shape, generator=gen, device=DEV, dtype=torch.float64)
    dt = 0.1 * spacing / speed
    return dict(x=x.contiguous(), v=v.to(dtype), C=torch.zeros(2 * nb, 9, dtype=dtype, device=DEV),
                av=torch.zeros(2 * nb, 3, dtype=dtype, device=DEV), aC=torch.zeros(2 * nb, 9, dtype=dtype, device=DEV),
                m=torch.full((2 * nb,), 1.0 / nb, dtype=dtype, device=DEV),
                body=torch.arange(2, dtype=torch.int32, device=DEV).repeat_interleave(nb),
                springs=torch.cat([springs, springs + nb]).contiguous(), rest=torch.cat([rest, rest]),
                k=torch.cat([k, k]), tri=torch.cat([tri, tri + nb]).contiguous(), h=h, mu=0.3, dt=dt, tau=dt)


def _mesh(case, seed):
    idx, tri = _lattice_mesh(case["nx"], case["ny"], case["nz"])
    n = idx.numel()
    z, y, x = torch.meshgrid(*[torch.arange(case[k], device=DEV) for k in ("nz", "ny", "nx")], indexing="ij")
    pts = torch.stack([x.reshape(-1), y.reshape(-1), z.reshape(-1)], 1).to(torch.float64) / 512
    pts = pts + (torch.rand(n, 3, generator=_gen(seed), device=DEV, dtype=torch.float64) - 0.5) * (0.4 / 512)
    return pts.contiguous(), tri


# ------------------------------------------------------------ what programs do


def prepare(case, seed):
    ctx = apic.Context(0)
    if case["kind"] == "step":
        s = _step_scene(case, seed)
        if case["memory"] == "host":
            keep = {k: s[k].cpu().pin_memory() for k in ("x", "v", "C", "m", "nrm", "body")}
            out = [torch.empty_like(keep[k]).pin_memory() for k in ("v", "C")]
            s.update({k: t.numpy() for k, t in keep.items()})
            return dict(case=case, ctx=ctx, s=s, out=[t.numpy() for t in out], keep=(keep, out))
        if case["normals"] == "mass":
            s["nrm"] = None
        return dict(case=case, ctx=ctx, s=s, out=(None, None))
    if case["kind"] == "batch":
        scenes = _batch_scenes(case, seed)
        total = sum(s["x"].shape[0] for s in scenes)
        v = torch.empty(total, 3, device=DEV)
        C = torch.empty(total, 3, 3, device=DEV)
        batch, at = [], 0
        for s in scenes:
            n = s["x"].shape[0]
            batch.append(apic.BatchScene(s["x"], s["v"], s["C"], s["m"], s["nrm"], s["body"], s["h"], s["mu"],
                                         n_bodies=s["bodies"], v_out=v[at:at + n], C_out=C[at:at + n]))
            at += n
        return dict(case=case, ctx=ctx, batch=batch, out=(v, C))
    if case["kind"] == "augury":
        e = _elastic(case, seed)
        live = {k: e[k].clone() for k in ("x", "v", "C", "av", "aC")}
        return dict(case=case, ctx=ctx, e=e, live=live)
    x, tri = _mesh(case, seed)
    return dict(case=case, ctx=ctx, x=x, tri=tri)


def run(state):
    case = state["case"]
    if case["kind"] == "step":
        s = state["s"]
        r = apic.contact_step(state["ctx"], s["x"], s["v"], s["C"], s["m"], s["nrm"], s["body"], s["h"], s["mu"],
                              case["n_iter"], n_bodies=s["bodies"], mu_pair=s["mu_pair"],
                              flags=apic.APIC_DETERMINISTIC if case["deterministic"] else 0, v_out=state["out"][0],
                              C_out=state["out"][1])
        return r.v, r.C
    if case["kind"] == "batch":
        apic.contact_step_batched(state["ctx"], state["batch"], case["n_iter"])
        return state["out"]
    if case["kind"] == "augury":
        e, live = state["e"], state["live"]
        for k, t in live.items():  # every pass starts from the same state
            t.copy_(e[k])
        apic.augury_steps(state["ctx"], live["x"], live["v"], live["C"], live["av"], live["aC"], e["m"], e["body"],
                          e["springs"], e["rest"], e["k"], e["tri"], e["h"], e["mu"], case["n_iter"], e["dt"], e["tau"],
                          case["steps"], n_bodies=2, init=True)
        return [live[k] for k in ("x", "v", "C", "av", "aC")]
    return apic.node_normals(state["ctx"], state["x"], state["tri"], fp64=case["dtype"] == "float64")


def work(case):
    if case["kind"] == "normals":
        nx, ny, nz = case["nx"], case["ny"], case["nz"]
        tri = 4 * ((nx - 1) * (ny - 1) + (ny - 1) * (nz - 1) + (nx - 1) * (nz - 1))
        n, surface = nx * ny * nz, nx * ny * nz - max(nx - 2, 0) * max(ny - 2, 0) * max(nz - 2, 0)
        # positions of the surface nodes, the triangles, every normal written
        return {"bytes": 24 * surface + 12 * tri + 3 * n * (8 if case["dtype"] == "float64" else 4), "flops": 40 * tri}
    if case["kind"] == "batch":
        total = 0
        for i in range(case["scenes"]):
            u = (i + 0.5) / case["scenes"]
            total += int(math.exp(math.log(case["min_nodes"]) + u * math.log(case["max_nodes"] / case["min_nodes"])))
        return {"bytes": 140 * total, "flops": 2400.0 * total * (case["n_iter"] + 1)}
    # per particle and step: x, body and (v, C, m, normal) read, (v, C) written; about 2,400 operations a transfer pair
    size = 8 if case["dtype"] == "float64" else 4
    if case["kind"] == "augury":
        n, steps = 2 * case["side"] ** 3, case["steps"] + 1
        springs = 2 * (3 * (case["side"] - 1) * case["side"] ** 2 + 6 * case["side"] * (case["side"] - 1) ** 2)
        return {"bytes": steps * (n * (2 * 24 + 4 + 49 * size) + 24 * springs),
                "flops": steps * (2400.0 * n * (case["n_iter"] + 1) + 30.0 * springs)}
    per = 24 + 4 + (3 + 9 + 1 + (3 if case["normals"] == "given" else 0) + 12) * size
    return {"bytes": case["nodes"] * per, "flops": 2400.0 * case["nodes"] * (case["n_iter"] + 1)}


# ------------------------------------------- the method in 64 bits, plain torch


def _basis(t):
    """Quadratic B-spline weights of the nodes i-1 .. i+2 at the offset t in a cell, and their derivatives."""
    s = 1 - t
    w = torch.stack([s * s, 2 - t * t, 1 + 2 * t - t * t, t * t], -1) / 4
    g = torch.stack([-s, -t, s, t], -1) / 2
    return w, g


class _Grid:
    """One dense background grid around the particles, and the transfers between them."""

    def __init__(self, x, h):
        q = x / h
        cell = torch.floor(q)
        t = q - cell
        cell = cell.to(torch.int64)
        lo = cell.amin(0) - 1
        self.dims = (cell.amax(0) + 3 - lo).tolist()
        self.size = self.dims[0] * self.dims[1] * self.dims[2]
        self.h = h
        c = cell - 1 - lo
        self.first = (c[:, 2] * self.dims[1] + c[:, 1]) * self.dims[0] + c[:, 0]
        self.w, self.g = _basis(t)
        self.d = (torch.arange(4, device=x.device) - 1).to(torch.float64) - t[..., None]

    def rows(self):
        """(nodes [n, 4], weights [n, 4], gradients [n, 3, 4], offsets [n, 3, 4]) of each x-row of the 4^3 stencil."""
        w, g, d = self.w, self.g, self.d
        run = torch.arange(4, device=w.device)
        for kz in range(4):
            for ky in range(4):
                node = (self.first + (kz * self.dims[1] + ky) * self.dims[0])[:, None] + run
                wyz = (w[:, 1, ky] * w[:, 2, kz])[:, None]
                yield node, w[:, 0] * wyz, (ky, kz), (d[:, 0], d[:, 1, ky, None], d[:, 2, kz, None])

    def scatter_mass(self, m):
        out = torch.zeros(self.size, dtype=torch.float64, device=m.device)
        for node, w, _, _ in self.rows():
            out.index_add_(0, node.reshape(-1), (w * m[:, None]).reshape(-1))
        return out

    def scatter(self, m, v, C):
        out = torch.zeros(self.size, 3, dtype=torch.float64, device=m.device)
        for node, w, _, d in self.rows():
            u = v[:, None, :] + self.h * (d[0][..., None] * C[:, None, :, 0] + d[1][..., None] * C[:, None, :, 1]
                                          + d[2][..., None] * C[:, None, :, 2])
            out.index_add_(0, node.reshape(-1), ((w * m[:, None])[..., None] * u).reshape(-1, 3))
        return out

    def gather(self, f):
        v = torch.zeros(self.first.shape[0], 3, dtype=torch.float64, device=f.device)
        C = torch.zeros(self.first.shape[0], 3, 3, dtype=torch.float64, device=f.device)
        for node, w, _, d in self.rows():
            a = w[..., None] * f[node]
            v += a.sum(1)
            for k in range(3):
                C[:, :, k] += (d[k][..., None] * a).sum(1)
        return v, C * (2 / self.h)

    def gather_mass(self, m):
        """Interpolated mass and its gradient (cell units)."""
        rho = torch.zeros(self.first.shape[0], dtype=torch.float64, device=m.device)
        grad = torch.zeros(self.first.shape[0], 3, dtype=torch.float64, device=m.device)
        w, g = self.w, self.g
        for node, wr, (ky, kz), _ in self.rows():
            f = m[node]
            rho += (wr * f).sum(1)
            grad[:, 0] += (g[:, 0] * f).sum(1) * w[:, 1, ky] * w[:, 2, kz]
            row = (w[:, 0] * f).sum(1)
            grad[:, 1] += row * g[:, 1, ky] * w[:, 2, kz]
            grad[:, 2] += row * w[:, 1, ky] * g[:, 2, kz]
        return rho, grad


def _contact(x, v, C, m, nrm, body, h, mu, n_iter, mu_pair=None, bodies=1):
    """V_hat, C_hat of one contact step: the series with the Coulomb cone rule."""
    grid = _Grid(x, h)
    body = body.to(torch.int64)
    per_body = None
    if nrm is None or mu_pair is not None:
        per_body = [grid.scatter_mass(torch.where(body == b, m, torch.zeros_like(m))) for b in range(bodies)]
    if nrm is None:
        nrm = torch.zeros_like(x)
        for b in range(bodies):
            rho, grad = grid.gather_mass(per_body[b])
            length = grad.norm(dim=1)
            on = (body == b) & (rho > 0) & (length > 0.5 * rho)
            nrm = torch.where(on[:, None], -grad / length.clamp_min(1e-300)[:, None], nrm)
    if mu_pair is not None:
        table = torch.as_tensor(mu_pair, dtype=torch.float64, device=x.device)
        num, den = torch.zeros_like(m), torch.zeros_like(m)
        for b in range(bodies):
            near = torch.where(body == b, torch.zeros_like(m), grid.gather_mass(per_body[b])[0])
            num += table[body, b] * near
            den += near
        mu = torch.where(den > 0, num / den.clamp_min(1e-300), table[body, body])
    mass = grid.scatter_mass(m)
    inv = torch.where(mass > 0, 1 / mass.clamp_min(1e-300), torch.zeros_like(mass))[:, None]

    def undesirable(dv):
        dn = (dv * nrm).sum(1, keepdim=True)
        vt = dv - dn * nrm
        size = vt.norm(dim=1, keepdim=True)
        m_ = mu[:, None] if torch.is_tensor(mu) else mu
        keep = torch.where(size > 0, torch.minimum(size, -m_ * dn) / size.clamp_min(1e-300), torch.zeros_like(size))
        return torch.where(dn <= 0, vt * (1 - keep), dv)

    hv, hC = grid.gather(grid.scatter(m, v, C) * inv)
    dv, dC = hv - v, hC - C
    for _ in range(n_iter):
        wv, wC = undesirable(dv), dC
        hv, hC = grid.gather(grid.scatter(m, wv, wC) * inv)
        dv, dC = dv + hv - wv, dC + hC - wC
    return v + dv, C + dC


def _mesh_normals(x, tri):
    t = tri.to(torch.int64)
    a, b, c = x[t[:, 0]], x[t[:, 1]], x[t[:, 2]]
    area = 0.5 * torch.linalg.cross(b - a, c - a)
    s = torch.zeros_like(x)
    for k in range(3):
        s.index_add_(0, t[:, k], area)
    length = s.norm(dim=1, keepdim=True)
    return torch.where(length > 0, s / length.clamp_min(1e-300), torch.zeros_like(s))


def _integrate(e, n_iter, steps):
    """Explicit time steps of the elastic blocks with the contact step as the preferred velocity."""
    x, v, C, m = (e[k].to(torch.float64).clone() for k in ("x", "v", "C", "m"))
    i, j = e["springs"][:, 0].to(torch.int64), e["springs"][:, 1].to(torch.int64)
    dt, tau = e["dt"], e["tau"]

    def accelerate(c_bar):
        d = x[j] - x[i]
        length = d.norm(dim=1, keepdim=True)
        pull = e["k"][:, None] * (length - e["rest"][:, None]) / length * d
        f = torch.zeros_like(x).index_add_(0, i, pull).index_add_(0, j, -pull)
        a = f / m[:, None]
        vbar = v + c_bar * a
        nrm = _mesh_normals(x, e["tri"])
        vh, Ch = _contact(x, vbar, C.reshape(-1, 3, 3), m, nrm, e["body"], e["h"], e["mu"], n_iter)
        return a + (vh - vbar) / tau, (Ch.reshape(-1, 9) - C) / tau

    av, aC = accelerate(tau)
    for _ in range(steps):
        v, C = v + 0.5 * dt * av, C + 0.5 * dt * aC
        x = x + dt * v
        av, aC = accelerate(0.5 * dt + tau)
        v, C = v + 0.5 * dt * av, C + 0.5 * dt * aC
    return [x, v, C, av, aC]


def _double(s, *names):
    return [None if s[k] is None else s[k].to(torch.float64) for k in names]


def exact(case, seed):
    if case["kind"] == "step":
        s = _step_scene(case, seed)
        if case["normals"] == "mass":
            s["nrm"] = None
        v, C = _contact(*_double(s, "x", "v", "C", "m", "nrm"), s["body"], s["h"], s["mu"], case["n_iter"],
                        s["mu_pair"], s["bodies"])
        return (v.cpu().numpy(), C.cpu().numpy()) if case["memory"] == "host" else (v, C)
    if case["kind"] == "batch":
        got = [_contact(*_double(s, "x", "v", "C", "m", "nrm"), s["body"], s["h"], s["mu"], case["n_iter"])
               for s in _batch_scenes(case, seed)]
        return torch.cat([g[0] for g in got]), torch.cat([g[1] for g in got])
    if case["kind"] == "augury":
        return _integrate(_elastic(case, seed), case["n_iter"], case["steps"])
    return _mesh_normals(*_mesh(case, seed))
