"""What a user of this library has it do, as cases that can be timed and whose outputs can be compared.

Every case is one pass through the public entry points on seeded synthetic shapes of the kinds that the
repository's own configurations use: solid tori with spheres along the core, CAD-like slabs with through
holes and organic unions of ellipsoids, both with near-medial spheres.  The generators here are written for
the device (a mesh of two million tets takes a fraction of a second) and stand on their own: a jittered
lattice split into Kuhn tets, cut to the shape, cleaned to a manifold.

How many elements a diagram has depends on the shape, so a case names its geometry (`geom`), and a seed places
that shape anew: a shift on the integer grid, a rotation of the axes, and another numbering of the spheres.
Every input and output value then differs from seed to seed while the tables keep their sizes.
"""
import math

import numpy as np
import torch

from paper_2403_18761_gb300 import rpd

MAX_COORD = (1 << 21) - 1                     # integer coordinate bound of the library's grid
KUHN = ((0, 1, 3, 7), (0, 1, 5, 7), (0, 2, 3, 7), (0, 2, 6, 7), (0, 4, 5, 7), (0, 4, 6, 7))
FACE = ((1, 2, 3), (0, 2, 3), (0, 1, 3), (0, 1, 2))   # face f lies opposite corner f
EDGE = ((0, 1), (0, 2), (0, 3), (1, 2), (1, 3), (2, 3))
HALF = (2.0, 1.0, 0.5)                        # the slab is a 4 x 2 x 1 box
HOLE = 0.2                                    # half side of its square through holes


def listed():
    return [
        # one small CAD part or one shape of a data set of thousands: launches and round trips count
        dict(name="build_torus_1k", what="build", geom=1, shape="torus", tets=1000, spheres=32, k=16, precision="fp32"),
        # the smallest named workload, in its own precision
        dict(name="build_torus_5k_fp64", what="build", geom=2, shape="torus", tets=5051, spheres=64, k=16, precision="fp64"),
        # an organic shape of the middle of the range, in the FP64 mode that the FP32 filter is compared with
        dict(name="build_blob_60k_fp64", what="build", geom=12, shape="blob", tets=60000, spheres=3000, parts=40, thin=1.0, k=32,
             precision="fp64"),
        # the CAD-like workload: a genus-3 block
        dict(name="build_slab_205k", what="build", geom=4, shape="slab", tets=205000, spheres=2000, parts=3, k=32,
             precision="fp32"),
        # the largest workload, on which the throughput is quoted
        dict(name="build_blob_2m", what="build", geom=3, shape="blob", tets=2000000, spheres=20000, parts=200, thin=1.5, k=32,
             precision="fp32"),
        # the medial mesh of a shape: a build that measures the restricted power edges, and the thinning
        dict(name="medial_slab_205k", what="medial", geom=6, shape="slab", tets=205000, spheres=2000, parts=3, k=32,
             precision="fp32", sigma=0.3),
        # a data set of shapes of uneven size, from host arrays, in one call
        dict(name="batch_32", what="batch", geom=7, shapes=32, tets_low=1000, tets_high=100000, k=16, precision="fp32"),
        # topology repair from a coarse start: pins, shrinking, partial updates until nothing fails
        dict(name="repair_slab_125k", what="repair", geom=8, shape="slab", tets=125000, spheres=256, parts=4, k=32,
             precision="fp32", rounds=8),
        # a sphere from every boundary triangle: the training pairs of the learned proposer
        dict(name="shrink_slab_125k", what="shrink", geom=9, shape="slab", tets=125000, spheres=256, parts=3),
        # a round's handful of pins against the same boundary
        dict(name="shrink_24_pins", what="shrink", geom=10, shape="slab", tets=125000, spheres=256, parts=2, pins=24),
        # every surface sample against the medial mesh's envelope: the geometric check of a refinement round
        dict(name="envelope_blob_300k", what="envelope", geom=11, shape="blob", tets=300000, spheres=3000, parts=60),
        # training the proposer network: forward, backward and Adam on batches of pairs
        dict(name="train_proposer", what="train", rows=65536, batch=8192, steps=100),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    what = rng.choice(("build", "build", "build", "build", "medial", "batch", "repair", "shrink", "envelope", "train"))
    precision = rng.choice(("fp32", "fp32", "fp64"))
    k = rng.choice((16, 24, 32))
    geom = rng.randrange(1 << 30)
    if what == "batch":
        return dict(what=what, geom=geom, shapes=rng.randint(5, 40), tets_low=1000, tets_high=_log_int(rng, 8000, 80000), k=k,
                    precision=precision)
    if what == "train":
        return dict(what=what, rows=_log_int(rng, 3000, 65000), batch=rng.choice((1024, 2048, 3001, 8192)),
                    steps=rng.randint(20, 100))
    if what == "repair":
        return dict(what=what, geom=geom, shape="slab", tets=_log_int(rng, 20000, 125000), spheres=rng.randint(64, 256),
                    parts=rng.randint(0, 5), k=32, precision="fp32", rounds=8)
    if what == "shrink":
        c = dict(what=what, geom=geom, shape="slab", tets=_log_int(rng, 8000, 125000), spheres=256, parts=rng.randint(0, 5))
        return dict(c, pins=rng.randint(1, 300)) if rng.random() < 0.4 else c
    shape = rng.choice(("torus", "slab", "blob"))
    tets = _log_int(rng, 1000, 1000000 if what == "build" else 300000)
    c = dict(what=what, geom=geom, shape=shape, tets=tets, spheres=max(32, int(tets / math.exp(rng.uniform(math.log(80), math.log(500))))))
    if shape != "torus":
        c["parts"] = rng.randint(0, 5) if shape == "slab" else rng.randint(12, 150)
    if what == "envelope":
        return c
    c.update(k=k, precision=precision)
    return dict(c, sigma=rng.choice((0.1, 0.3))) if what == "medial" else c


# ------------------------------------------------------------------ shapes
def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


class _Shape:
    """A solid: its box, a signed distance (negative inside) and sphere sampling."""

    def __init__(self, kind, parts, gen, dev):
        self.kind, self.gen, self.dev = kind, gen, dev
        f = dict(dtype=torch.float64, device=dev)
        if kind == "torus":
            self.R, self.r = 1.0, 0.4
            self.lo, self.hi = torch.tensor([-1.4, -1.4, -0.4], **f), torch.tensor([1.4, 1.4, 0.4], **f)
        elif kind == "slab":
            self.hi = torch.tensor(HALF, **f)
            self.lo = -self.hi
            self.holes = [] if parts == 0 else [0.0] if parts == 1 else np.linspace(-1.3, 1.3, parts).tolist()
        else:   # ellipsoids of axes U(0.1, 0.5), centres on a random walk, so that the union is connected
            self.axes = 0.1 + 0.4 * self.rand(parts, 3)
            q = torch.linalg.qr(self.randn(parts, 3, 3))[0]
            self.rot = q
            step = self.randn(parts, 3)
            step = 0.25 * step / step.norm(dim=1, keepdim=True)
            u = self.rand(parts).tolist()
            c = [torch.zeros(3, **f)]
            for n in range(1, parts):
                c.append(c[int(u[n] * n)] + step[n])
            c = torch.stack(c)
            self.centers = c - c.mean(dim=0)
            reach = self.axes.max(dim=1).values[:, None]
            self.lo, self.hi = (self.centers - reach).min(dim=0).values, (self.centers + reach).max(dim=0).values

    def rand(self, *n):
        return torch.rand(*n, dtype=torch.float64, device=self.dev, generator=self.gen)

    def randn(self, *n):
        return torch.randn(*n, dtype=torch.float64, device=self.dev, generator=self.gen)

    def volume(self):
        if self.kind == "torus":
            return 2 * math.pi ** 2 * self.R * self.r ** 2
        if self.kind == "slab":
            return 8.0 - len(self.holes) * (2 * HOLE) ** 2
        p = self.lo + (self.hi - self.lo) * self.rand(100000, 3)
        return float((self.sdf(p) < 0).double().mean() * (self.hi - self.lo).prod())

    def prims(self, x):
        """Distances from interior points of the slab to its planes and holes."""
        d = [self.hi[a] - x[:, a] for a in range(3)] + [self.hi[a] + x[:, a] for a in range(3)]
        for c in self.holes:
            d.append(torch.hypot((x[:, 0] - c).abs().sub(HOLE).clamp(min=0), x[:, 1].abs().sub(HOLE).clamp(min=0)))
        return torch.stack(d, dim=1)

    def sdf(self, x):
        if self.kind == "torus":
            return torch.hypot(torch.hypot(x[:, 0], x[:, 1]) - self.R, x[:, 2]) - self.r
        out = []
        amin = self.axes.min(dim=1).values
        m = torch.einsum("eij,ej->eij", self.rot, 1.0 / self.axes)
        off = torch.einsum("ei,eij->ej", self.centers, m)
        for p in x.split(1 << 17):
            y = torch.einsum("ni,eij->enj", p, m) - off[:, None, :]
            out.append(((y.norm(dim=2) - 1.0) * amin[:, None]).min(dim=0).values)
        return torch.cat(out)

    def spheres(self, n, h, thin):
        """n spheres (fewer where the shape is too small for them): on the core circle of a torus, else
        near the medial axis, at most one in a cell of `thin` lattice
        spacings (a tet takes at most 32 candidate spheres)."""
        if self.kind == "torus":
            n = min(n, int(8 * math.pi * self.R / h))
            th = 2 * math.pi * torch.arange(n, dtype=torch.float64, device=self.dev) / n + 0.1234
            c = torch.stack([self.R * th.cos(), self.R * th.sin(), torch.zeros_like(th)], dim=1)
            return c + 0.02 * self.randn(n, 3), self.r * (0.75 + 0.25 * self.rand(n))
        cs, rs = [], []
        for _ in range(24):
            if self.kind == "slab":
                p = self.lo + (self.hi - self.lo) * self.rand(1 << 17, 3)
                d = self.prims(p).sort(dim=1).values
                ok = (d[:, 0] > 0) & (d[:, 1] - d[:, 0] < 0.02)
                for c in self.holes:
                    ok &= ~(((p[:, 0] - c).abs() < HOLE) & (p[:, 1].abs() < HOLE))
                p, d = p[ok], d[ok, 0]
            else:   # points of a random ellipsoid where the depth has a ridge
                e = torch.multinomial(self.axes.prod(dim=1), 1 << 15, replacement=True, generator=self.gen)
                y = self.randn(len(e), 3)
                y = y / y.norm(dim=1, keepdim=True) * self.rand(len(e), 1) ** (1 / 3)
                p = self.centers[e] + torch.einsum("nij,nj->ni", self.rot[e], y * self.axes[e])
                d = -self.sdf(p)
                step = 0.01 * torch.eye(3, dtype=torch.float64, device=self.dev)
                g = torch.stack([(self.sdf(p + s) - self.sdf(p - s)) / 0.02 for s in step], dim=1)
                ok = (d > 0.02) & (g.norm(dim=1) < 0.6)
                p, d = p[ok], d[ok]
            cs.append(p)
            rs.append(d)
            if sum(len(r) for r in rs) > 2 * n:
                break
        c, r = torch.cat(cs), torch.cat(rs)
        cell = ((c - self.lo) / (thin * h)).floor().long()
        key = (cell[:, 0] * (1 << 20) + cell[:, 1]) * (1 << 20) + cell[:, 2]
        _, inv = torch.unique(key, return_inverse=True)
        first = torch.full((int(inv.max()) + 1,), len(c), dtype=torch.long, device=self.dev)
        first.scatter_reduce_(0, inv, torch.arange(len(c), device=self.dev), "amin")
        keep = first.sort().values[:n]
        return c[keep], r[keep]


def _matched_faces(t, nv):
    """Pairs (a, b) of face indices (4 tet + face) that are the same triangle; the sorted face keys."""
    f = t[:, torch.tensor(FACE, device=t.device)].sort(dim=2).values
    key, order = ((f[..., 0] * nv + f[..., 1]) * nv + f[..., 2]).reshape(-1).sort()
    same = key[1:] == key[:-1]
    return order[:-1][same], order[1:][same], key


def _manifold(t, nv):
    """Drops the tets at vertices whose star is not one face-connected cluster with a disk or sphere as link."""
    dev = t.device
    face = torch.tensor(FACE, device=dev)
    for _ in range(24):
        a, b, key = _matched_faces(t, nv)
        loc = t[:, face].argsort(dim=2)
        corner = (torch.arange(len(t), device=dev)[:, None, None] * 4 + face[None].expand(len(t), 4, 3).gather(2, loc)).reshape(-1, 3)
        ca, cb = corner[a].reshape(-1), corner[b].reshape(-1)
        lab = torch.arange(4 * len(t), device=dev)
        for _ in range(16):
            new = lab.scatter_reduce(0, ca, lab[cb], "amin").scatter_reduce(0, cb, lab[ca], "amin")
            new = new[new]
            if torch.equal(new, lab):
                break
            lab = new
        v = t.reshape(-1)
        clusters = torch.bincount(v[lab == torch.arange(len(lab), device=dev)], minlength=nv)
        e = t[:, torch.tensor(EDGE, device=dev)].sort(dim=2).values
        ek = torch.unique(e[..., 0] * nv + e[..., 1])
        fk = torch.unique_consecutive(key)
        n = lambda x: torch.bincount(x, minlength=nv)   # noqa: E731
        link = n(ek // nv) + n(ek % nv) - n(fk // (nv * nv)) - n(fk // nv % nv) - n(fk % nv) + n(v)
        bad = (n(v) > 0) & ((clusters != 1) | ((link != 1) & (link != 2)))
        if not bool(bad.any()):
            break
        t = t[~bad[t].any(dim=1)]
    return t


def _mesh(shape, tets, dev, bits=None):
    """(vertices, tets, lattice spacing, grid bits): a jittered Kuhn lattice cut to the shape, on the grid."""
    h = (6.0 * shape.volume() / tets) ** (1.0 / 3.0)
    if shape.kind == "slab":   # the spacing divides every side: the planes are lattice planes
        m = max(2, round(1.0 / h))
        h, lo = 1.0 / m, shape.lo
        n = (torch.round(2 * shape.hi * m)).long().tolist()
    else:
        lo = shape.lo - h
        n = [int(v) for v in torch.ceil((shape.hi + h - lo) / h).long().tolist()]
    ext = float(torch.maximum(shape.lo.abs(), shape.hi.abs()).max()) + 2 * h
    if bits is None:   # the finest grid that takes the shape with room for its shift
        bits = int(math.log2((MAX_COORD - 16384) / (ext * 1.05 + 0.1)))
    ax = [torch.arange(k + 1, device=dev) for k in n]
    idx = torch.stack(torch.meshgrid(*ax, indexing="ij"), dim=-1).reshape(-1, 3)
    jit = (2 * shape.rand(len(idx), 3) - 1) * 0.1 * h
    cube = torch.stack(torch.meshgrid(*[torch.arange(k, device=dev) for k in n], indexing="ij"), dim=-1).reshape(-1, 3)
    stride = torch.tensor([(n[1] + 1) * (n[2] + 1), n[2] + 1, 1], device=dev)
    if shape.kind == "slab":
        # vertices keep the planes they lie on: box faces and, as lattice planes, the walls of the square holes
        flat = (idx == 0) | (idx == torch.tensor(n, device=dev))
        keep = torch.ones(len(cube), dtype=torch.bool, device=dev)
        w = max(1, round(HOLE * m))
        for c in shape.holes:
            i0, j0 = round((c + HALF[0]) * m), round(HALF[1] * m)
            keep &= ~((cube[:, 0] >= i0 - w) & (cube[:, 0] < i0 + w) & (cube[:, 1] >= j0 - w) & (cube[:, 1] < j0 + w))
            in_x, in_y = (idx[:, 0] - i0).abs() <= w, (idx[:, 1] - j0).abs() <= w
            flat[:, 0] |= in_x & in_y & ((idx[:, 0] - i0).abs() == w)
            flat[:, 1] |= in_x & in_y & ((idx[:, 1] - j0).abs() == w)
        jit[flat] = 0.0
        cube = cube[keep]
    p = torch.round((lo + h * idx + jit) * (1 << bits)) / (1 << bits)
    base = (cube * stride).sum(dim=1)
    if shape.kind != "slab":
        s = shape.sdf(p)
        off = torch.tensor([sum(((c >> a) & 1) * int(stride[a]) for a in range(3)) for c in range(8)], device=dev)
        base = base[(s[base[:, None] + off] < 0).any(dim=1)]
    off = torch.tensor([sum(((c >> a) & 1) * int(stride[a]) for a in range(3)) for c in range(8)], device=dev)
    t = (base[:, None] + off)[:, torch.tensor(KUHN, device=dev)].reshape(-1, 4)
    if shape.kind != "slab":
        t = t[s[t].mean(dim=1) < 0]
    e = p[t[:, 1:]] - p[t[:, :1]]
    det = (e[:, 0] * torch.linalg.cross(e[:, 1], e[:, 2])).sum(dim=1)
    t = torch.where((det < 0)[:, None], t[:, [0, 1, 3, 2]], t)
    if shape.kind != "slab":
        t = _manifold(t, len(p))
    used = torch.zeros(len(p), dtype=torch.long, device=dev)
    used[t.reshape(-1)] = 1
    at = used.cumsum(0) - 1
    return p[used > 0].contiguous(), at[t].int().contiguous(), h, bits


def _inputs(case, seed):
    """(vertices, tets, centres, radii, grid bits): the case's shape as the seed places it."""
    dev = _device()
    gen = torch.Generator(device=dev)
    gen.manual_seed(int(case["geom"]) * 7919 + 17)
    shape = _Shape(case["shape"], case.get("parts", 0), gen, dev)
    v, t, h, bits = _mesh(shape, case["tets"], dev, case.get("bits"))
    c, r = shape.spheres(case["spheres"], h, case.get("thin", 2.0))
    s = float(1 << bits)
    rng = np.random.default_rng([int(seed), int(case["geom"])])
    shift = torch.tensor(rng.integers(-16384, 16385, 3) / s, device=dev)
    axes = torch.tensor(np.roll(np.arange(3), int(rng.integers(3))), device=dev)
    v, c, r = v[:, axes] + shift, torch.round(c[:, axes] * s) / s + shift, torch.round(r * s) / s
    if case.get("what") != "repair":   # the repair picks its pins by sphere number
        p = torch.tensor(rng.permutation(len(c)), device=dev)
        c, r = c[p], r[p]
    return v.contiguous(), t, c.contiguous(), r.contiguous(), bits


def _batch_cases(case):
    rng = np.random.default_rng(case["geom"])
    out = []
    for n in range(case["shapes"]):
        t = math.exp(rng.uniform(math.log(case["tets_low"]), math.log(case["tets_high"])))
        s = min(math.exp(rng.uniform(math.log(32), math.log(4000))), max(32, t / 30))
        kind = ("torus", "slab", "blob")[n % 3]
        parts = int(rng.integers(6, 24)) if kind == "blob" else (n // 3) % 6 if t > 20000 else 0
        out.append(dict(geom=case["geom"] * 64 + n, shape=kind, tets=int(t), spheres=int(s), parts=parts, bits=19))
    return out


# ------------------------------------------------------------------- cases
def prepare(case, seed):
    what = case["what"]
    if what == "train":
        dev = _device()
        gen = torch.Generator(device=dev)
        gen.manual_seed(int(seed) * 7919 + 17)
        x = torch.rand(case["rows"], rpd.RPD_PIN_FEATURES, device=dev, generator=gen) * 2 - 1
        t = torch.sin(2 * x[:, 0]) + 0.5 * x[:, 1] * x[:, 2] - 2
        return dict(case=case, seed=seed, x=x, t=t)
    if what == "batch":   # the call takes host arrays
        shapes = [tuple(a.cpu().numpy() for a in _inputs(c, seed)[:4]) for c in _batch_cases(case)]
        return dict(case=case, shapes=shapes, bits=19)
    v, t, c, r, bits = _inputs(case, seed)
    s = dict(case=case, args=(v, t, c, r), bits=bits)
    if what in ("shrink", "envelope"):   # the diagram is at hand, the query is what is measured
        ctx = rpd.rpd_build(v, t, c, r, k=32, grid_bits=bits)
        pts, normals, faces = ctx.rpd_surface_samples()
        if case.get("pins"):
            gen = torch.Generator(device=pts.device)
            gen.manual_seed(int(seed))
            pick = torch.randperm(len(pts), device=pts.device, generator=gen)[: case["pins"]]
            pts, normals, faces = pts[pick].contiguous(), normals[pick].contiguous(), faces[pick].contiguous()
        s.update(ctx=ctx, pts=pts, normals=normals, faces=faces)
    return s


def _tables(ctx, kinds=(1, 2, 3, 4)):
    out = {}
    for kind in kinds:
        keys, chi = ctx.rpd_euler(kind)
        _, beta = ctx.rpd_components(kind)
        _, flag = ctx.rpd_contractible(kind)
        out["kind%d" % kind] = [keys, chi, beta, flag]
    return out


def run(state):
    case = state["case"]
    what = case["what"]
    if what == "train":
        net = rpd.Mlp(seed=state["seed"])
        loss = net.train(state["x"], state["t"], case["steps"], batch=case["batch"])
        return dict(loss=torch.tensor(loss, dtype=torch.float32), params=net.params())
    if what == "batch":
        ctx = rpd.rpd_build_batch(state["shapes"], precision=case["precision"], k=case["k"], grid_bits=state["bits"])
        out = _tables(ctx)
        out["pieces"] = list(ctx.rpd_pieces())
        out["rows"] = [ctx.shape_offsets(kind) for kind in range(5)]
        return out
    if what == "shrink":
        return list(state["ctx"].rpd_shrink(state["pts"], state["normals"], state["faces"]))
    if what == "envelope":
        return list(state["ctx"].rpd_envelope_distance(state["pts"]))
    ctx = rpd.rpd_build(*state["args"], precision=case["precision"], k=case["k"], grid_bits=state["bits"],
                        edge_lengths=what == "medial")
    out = {}
    if what == "medial":
        info, edges, faces = ctx.rpd_medial(case["sigma"])
        out.update(info=info, edges=edges, faces=faces, lengths=list(ctx.rpd_edge_lengths()))
    if what == "repair":
        out["rounds"] = list(ctx.rpd_repair(case["rounds"]))
        out["spheres"] = list(ctx.rpd_spheres())
    out.update(_tables(ctx))
    out["pieces"] = list(ctx.rpd_pieces())
    return out


def work(case):
    what = case["what"]
    if what == "train":   # three hidden layers forward, their weight gradients, two input gradients
        b = min(case["batch"], case["rows"])
        mac = 32 * 128 * 2 + 128 * 128 * 6 + 128 * 3
        return {"bytes": 4.0 * min(case["rows"], b * case["steps"]) * 31 + 4 * 37377, "flops": 2.0 * mac * b * case["steps"]}
    if what == "batch":
        mean = (case["tets_high"] - case["tets_low"]) / math.log(case["tets_high"] / case["tets_low"])
        tets, spheres = mean * case["shapes"], mean * case["shapes"] / 150
    else:
        tets, spheres = case["tets"], case["spheres"]
    if what in ("shrink", "envelope"):
        # surface of the lattice cut: two triangles per boundary square of side h
        area = 28.0 if case["shape"] == "slab" else 16.0 if case["shape"] == "torus" else 1.2 * case.get("parts", 1)
        vol = 8.0 if case["shape"] == "slab" else 3.2 if case["shape"] == "torus" else 0.06 * case.get("parts", 1)
        tri = 2 * area / (6 * vol / tets) ** (2 / 3)
        if what == "shrink":
            pins = case.get("pins") or tri
            return {"bytes": 72.0 * tri + pins * 88, "flops": 10.0 * 150 * pins}
        return {"bytes": 32.0 * tri + 96 * spheres, "flops": 20.0 * 40 * tri}
    # inputs once; element tables and pieces once (about two pieces a tet, 7 faces, 12 edges and 6 vertices a sphere)
    pieces = 2.0 * tets
    nbytes = 24 * tets / 5.7 + 16 * tets + 32 * spheres + 40 * pieces + spheres * (13 + 7 * 17 + 12 * 21 + 6 * 25)
    return {"bytes": nbytes, "flops": 400.0 * pieces}


# ------------------------------------------------------- 64-bit references
def _exact_pieces(v, t, c, r):
    """(tet, sphere, volume, first moment) of every piece: each (tet, sphere) pair clipped against all the
    other spheres that may own a part of the tet, as a growing set of simplices in barycentric coordinates."""
    x = v[t.long()]
    d = ((x[:, :, None, :] - c) ** 2).sum(dim=3) - r ** 2                      # tets x 4 x spheres
    alive = torch.ones(len(t), len(c), dtype=torch.bool, device=v.device)
    for j in range(len(c)):
        alive &= ~(d[:, :, j:j + 1] < d).all(dim=1)
    pt, ps = alive.nonzero(as_tuple=True)
    order = torch.where(alive, torch.arange(len(c), device=v.device), len(c)).sort(dim=1).values
    bary = torch.eye(4, dtype=torch.float64, device=v.device).expand(len(pt), 4, 4)
    of = torch.arange(len(pt), device=v.device)
    for s in range(int(alive.sum(dim=1).max())):
        j = order[pt[of], s]
        cut = (j < len(c)) & (j != ps[of])
        f = d[pt[of], :, ps[of]] - d[pt[of], :, j.clamp(max=len(c) - 1)]
        f = torch.where(cut[:, None], torch.einsum("nkc,nc->nk", bary, f), -1.0)
        f, o = f.sort(dim=1)                                                   # the kept corners first
        b = bary.gather(1, o[:, :, None].expand(-1, -1, 4))
        n = (f < 0).sum(dim=1)
        at = lambda m, a, k: b[m, a] + (b[m, k] - b[m, a]) * (f[m, a] / (f[m, a] - f[m, k]))[:, None]   # noqa: E731
        parts, owner = [b[n == 4]], [of[n == 4]]
        m = n == 1
        parts.append(torch.stack([b[m, 0], at(m, 0, 1), at(m, 0, 2), at(m, 0, 3)], dim=1))
        owner.append(of[m])
        for m, top, low in ((n == 2, (lambda m: b[m, 0], lambda m: at(m, 0, 2), lambda m: at(m, 0, 3)),
                             (lambda m: b[m, 1], lambda m: at(m, 1, 2), lambda m: at(m, 1, 3))),
                            (n == 3, (lambda m: b[m, 0], lambda m: b[m, 1], lambda m: b[m, 2]),
                             (lambda m: at(m, 0, 3), lambda m: at(m, 1, 3), lambda m: at(m, 2, 3)))):
            p, q = [g(m) for g in top], [g(m) for g in low]                    # a prism in three simplices
            for w in ((p[0], p[1], p[2], q[0]), (p[1], p[2], q[0], q[1]), (p[2], q[0], q[1], q[2])):
                parts.append(torch.stack(w, dim=1))
                owner.append(of[m])
        bary, of = torch.cat(parts), torch.cat(owner)
    e = x[pt[of]][:, 1:] - x[pt[of]][:, :1]
    whole = (e[:, 0] * torch.linalg.cross(e[:, 1], e[:, 2])).sum(dim=1) / 6
    b = bary[:, 1:, 1:] - bary[:, :1, 1:]
    vol = whole * (b[:, 0] * torch.linalg.cross(b[:, 1], b[:, 2])).sum(dim=1).abs()
    mid = torch.einsum("nc,ncx->nx", bary.mean(dim=1), x[pt[of]])
    pv = torch.zeros(len(pt), dtype=torch.float64, device=v.device).index_add(0, of, vol)
    pm = torch.zeros(len(pt), 3, dtype=torch.float64, device=v.device).index_add(0, of, vol[:, None] * mid)
    keep = pv > 0
    return pv[keep], pm[keep]


def _nearest(tri, x):
    """For centres x [m, 3]: the nearest point on any of the triangles, per row of a [m] choice that the mask
    in `tri` leaves; tri = (A, B, C, allowed [m, n])."""
    A, B, C, allowed = tri

    def on_segment(P, Q):
        e = Q - P
        u = (((x[:, None] - P) * e).sum(dim=2) / (e * e).sum(dim=1)).clamp(0, 1)
        return P + u[..., None] * e

    e1, e2 = B - A, C - A
    a11, a12, a22 = (e1 * e1).sum(dim=1), (e1 * e2).sum(dim=1), (e2 * e2).sum(dim=1)
    g = x[:, None] - A
    b1, b2 = (g * e1).sum(dim=2), (g * e2).sum(dim=2)
    det = a11 * a22 - a12 * a12
    s, u = (b1 * a22 - b2 * a12) / det, (b2 * a11 - b1 * a12) / det
    best, dist = None, None
    for q, ok in ((A + s[..., None] * e1 + u[..., None] * e2, (s >= 0) & (u >= 0) & (s + u <= 1)),
                  (on_segment(A, B), None), (on_segment(B, C), None), (on_segment(C, A), None)):
        w = ((q - x[:, None]) ** 2).sum(dim=2)
        w = w if ok is None else torch.where(ok, w, math.inf)
        if best is None:
            best, dist = q, w
        else:
            m = w < dist
            best, dist = torch.where(m[..., None], q, best), torch.where(m, w, dist)
    dist = torch.where(allowed, dist, math.inf)
    near = dist.argmin(dim=1)
    row = torch.arange(len(x), device=x.device)
    return best[row, near], dist[row, near].sqrt()


def _exact_shrink(case, seed):
    v, t, _, _, bits = _inputs(case, seed)
    t = t.long()
    a, b, _ = _matched_faces(t, len(v))
    open_ = torch.ones(4 * len(t), dtype=torch.bool, device=v.device)
    open_[a] = False
    open_[b] = False
    face = open_.nonzero()[:, 0]
    ids = t[face // 4].gather(1, torch.tensor(FACE, device=v.device)[face % 4])
    A, B, C = (v[ids[:, k]] for k in range(3))
    pin = (A + B + C) / 3
    n = torch.linalg.cross(B - A, C - A)
    inward = v[t[face // 4].gather(1, (face % 4)[:, None])[:, 0]] - pin
    n = n / n.norm(dim=1, keepdim=True)
    n = torch.where(((n * inward).sum(dim=1) < 0)[:, None], -n, n)
    who = torch.arange(len(pin), device=v.device)
    if case.get("pins"):
        gen = torch.Generator(device=v.device)
        gen.manual_seed(int(seed))
        who = torch.randperm(len(pin), device=v.device, generator=gen)[: case["pins"]]
    cs, rs = [], []
    every = torch.arange(len(pin), device=v.device)
    for w in who.split(max(1, (1 << 23) // len(pin))):
        p, m = pin[w], n[w]
        r = torch.full((len(w),), 2.0 ** (23 - bits), dtype=torch.float64, device=v.device)
        live = torch.ones(len(w), dtype=torch.bool, device=v.device)
        for _ in range(100):
            c = p + r[:, None] * m
            q, dist = _nearest((A, B, C, every != w[:, None]), c)
            pq = q - p
            dn = (pq * m).sum(dim=1)
            rn = (pq * pq).sum(dim=1) / (2 * dn)
            live = live & ~(dist >= r * (1 - 1e-12)) & (dn > 0) & (rn < r)
            if not bool(live.any()):
                break
            r = torch.where(live, rn, r)
        cs.append(p + r[:, None] * m)
        rs.append(r)
    return [torch.cat(cs), torch.cat(rs), None]


def exact(case, seed):
    if case["what"] == "shrink" and case["tets"] <= 200000:
        return _exact_shrink(case, seed)
    if case["what"] == "build" and case["tets"] * case["spheres"] <= 4000000:
        v, t, c, r, _ = _inputs(case, seed)
        none = {"kind%d" % k: [None] * 4 for k in (1, 2, 3, 4)}
        return dict(none, pieces=[None, None, *_exact_pieces(v, t, c, r)])
    return None
