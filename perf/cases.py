"""Performance cases of the MBOIT puzzle-piece renderer: what a program that renders with the library asks of it.

Each case is one call (or one fixed sequence of calls) of the package's public interface on a seeded synthetic
volume.  Inputs have the statistics of the benchmark's own workloads (Gaussian blobs plus value noise, a
six-point transfer function, Morton-order pieces) and are made on the GPU, so that they can be remade often.

  listed()            the named cases
  draw(rng)           one more case of the same ranges
  prepare(case, seed) the volume, its buffers and its views, as a program holds them
  run(state)          one pass through the public entry points; returns moments and images whole
  work(case)          bytes and floating-point operations one pass cannot do without
  exact(case, seed)   the same outputs in 64-bit arithmetic (plain torch), without the library's code
"""
import functools
import math
from types import SimpleNamespace

import numpy as np
import torch

import paper_2501_12581_gb300 as mb

STEP = 0.5
ABSORBANCE_MAX = 10.0
OVERESTIMATION = 0.3
POWER = {"power4": 2, "power6": 3, "power8": 4}
TRIG = {"trig6": 3, "trig8": 4}
VIEW_DIR = (0.57, 0.49, 0.66)


# ---------------------------------------------------------------------------
# the cases

def _case(kind, call="frame", width=512, height=512, views=1, pieces=8, tuned=False, moments="power4", storage="f32",
          bias=5e-5, opacity=27.0, **more):
    return dict(kind=kind, call=call, width=width, height=height, views=views, pieces=pieces, tuned=tuned,
                moments=moments, storage=storage, bias=bias, opacity=opacity, **more)


def _grid(nx, ny, nz, brick_log2=4, ortho=False, **more):
    return _case("grid", nx=nx, ny=ny, nz=nz, brick_log2=brick_log2, ortho=ortho, **more)


def _octree(base, max_level=2, adaptive=False, **more):
    return _case("octree", base=base, max_level=max_level, adaptive=adaptive, **more)


def listed():
    return [
        # a small preview volume in an interactive viewer: one launch of little work, latency counts
        dict(_grid(64, 64, 64, 3, ortho=True, width=256, height=256, pieces=4, opacity=8.3), name="grid64"),
        # a crop of a simulation box: odd sizes in every axis, a ragged image, no tuning call
        dict(_grid(301, 227, 181, width=1000, height=723, pieces=7, opacity=15.0), name="grid_ragged"),
        # the 512^3 benchmark frame of a program that tunes once and renders many frames
        dict(_grid(512, 512, 512, width=2048, height=2048, pieces=64, tuned=True), name="grid512"),
        # an ensemble of small grids shown side by side, one frame for all of them
        dict(_grid(64, 64, 64, 3, call="multi", volumes=8, width=256, height=256, pieces=4, opacity=8.3),
             name="grid_volumes"),
        # half of the pieces switched off, the two passes called one by one
        dict(_grid(256, 256, 256, call="subset", width=1024, height=768, pieces=16), name="grid_subset"),
        # the distributed form of the method: per-piece moment images, their sum, per-piece colours, their sum
        dict(_grid(256, 256, 256, call="pieces", width=1024, height=1024, pieces=16), name="grid_pieces"),
        # a coarse octree in two small views
        dict(_octree(8, width=512, height=512, views=2, pieces=8, opacity=18.0), name="octree8"),
        # the 72-piece octree benchmark frame
        dict(_octree(26, width=2560, height=2560, pieces=72, tuned=True), name="octree26"),
        # the same octree sampled at each leaf's own resolution, for interaction
        dict(_octree(26, width=1024, height=1024, pieces=72, adaptive=True), name="octree26_adaptive"),
        # more moments for thicker media: 16-bit trigonometric and float32 power moments
        dict(_octree(13, width=1024, height=1024, pieces=24, moments="trig8", storage="f16", bias=2e-3),
             name="octree13_trig8"),
        dict(_octree(13, width=1024, height=1024, pieces=24, moments="power8"), name="octree13_power8"),
        # an unstructured mesh, as the solver that the method was published for has them
        dict(_case("mesh", cells=64, width=1024, height=1024, pieces=24, tuned=True, opacity=8.3), name="mesh64"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """A case of the listed ranges: every kind of volume and call, odd sizes, other moment sets and storages."""
    kind = rng.choice(["grid", "grid", "grid", "octree", "octree", "mesh"])
    size = dict(width=_log(rng, 96, 1400), height=_log(rng, 96, 1400))
    moments = rng.choice(["power4", "power4", "power4", "power6", "power8", "trig6", "trig8"])
    storage = rng.choice(["f16", "bf16"]) if moments in TRIG else "f32"
    bias = {"f32": 5e-5, "f16": 2e-3, "bf16": 2e-2}[storage]
    fmt = dict(moments=moments, storage=storage, bias=bias)
    if kind == "grid":
        call = rng.choice(["frame", "frame", "subset", "pieces", "multi"])
        if call == "multi":
            n = _log(rng, 33, 128)
            return _grid(n, n + rng.randrange(9), n, 3, call="multi", volumes=rng.randrange(2, 9), pieces=4,
                         width=_log(rng, 64, 512), height=_log(rng, 64, 512), opacity=8.3)
        if call == "pieces":
            size = dict(width=_log(rng, 96, 900), height=_log(rng, 96, 900))
        return _grid(_log(rng, 48, 400), _log(rng, 48, 400), _log(rng, 48, 400), rng.choice([3, 4]), call=call,
                     ortho=rng.random() < 0.3, pieces=rng.randrange(2, 17), views=rng.choice([1, 1, 2]),
                     tuned=call == "frame" and rng.random() < 0.3, opacity=15.0, **size, **fmt)
    if kind == "octree":
        level = rng.choice([1, 2, 2])
        return _octree(_log(rng, 4, 24), level, rng.random() < 0.3, pieces=rng.randrange(2, 33),
                       tuned=rng.random() < 0.3, opacity=20.0, **size, **fmt)
    return _case("mesh", cells=_log(rng, 10, 64), pieces=rng.randrange(2, 17), opacity=8.3, **size)


# ---------------------------------------------------------------------------
# inputs

def _axis(n, lo, hi):
    return torch.linspace(lo, hi, n, dtype=torch.float64, device="cuda")


class _Field:
    """64 Gaussian blobs (8 on small volumes) plus three octaves of value noise in the unit cube."""

    def __init__(self, gen, blobs, noise):
        u = torch.rand(blobs, 5, generator=gen, dtype=torch.float64)
        self.c = u[:, :3].cuda()
        self.s = (1 / 16 + u[:, 3] / 8).cuda()
        self.a = (0.3 + 0.7 * u[:, 4]).cuda()
        self.noise = [(0.15 * 0.5 ** o, torch.rand(*[8 * 2 ** o + 1] * 3, generator=gen, dtype=torch.float64).cuda())
                      for o in range(3)] if noise else []

    @staticmethod
    def _weights(x, n):
        """[len(x)][n] weights of linear interpolation between n lattice values at x in [0, 1]."""
        j = torch.arange(n, device=x.device, dtype=x.dtype)
        return (1 - ((x * (n - 1))[:, None] - j).abs()).clamp(min=0)

    def tensor_grid(self, x, y, z):
        """Values [z][y][x] on the tensor grid of three coordinate lists."""
        g = [torch.exp(-(q[None] - self.c[:, c:c + 1]) ** 2 / (2 * self.s[:, None] ** 2)) for c, q in
             enumerate((x, y, z))]
        out = torch.empty(len(z), len(y), len(x), dtype=torch.float32, device="cuda")
        xa = g[0] * self.a[:, None]
        w = [[self._weights(q, v.shape[0]) for q in (z, y, x)] for _, v in self.noise]
        for z0 in range(0, len(z), 64):
            zy = g[2][:, z0:z0 + 64, None] * g[1][:, None, :]
            v = (zy.reshape(zy.shape[0], -1).T @ xa).reshape(-1, len(y), len(x))
            for (amp, lat), (wz, wy, wx) in zip(self.noise, w):
                v += amp * (wy @ torch.einsum("za,abx->zbx", wz[z0:z0 + 64], lat @ wx.T))
            out[z0:z0 + 64] = v.float()
        return out

    def points(self, p):
        """Values at points p [m][3] (x, y, z) in the unit cube."""
        v = torch.zeros(len(p), dtype=torch.float64, device="cuda")
        for b in range(len(self.a)):
            v += self.a[b] * torch.exp(-((p - self.c[b]) ** 2).sum(1) / (2 * self.s[b] ** 2))
        return v

    def leaves(self, origin, size):
        """Values [m][9][9][9] on the vertex lattices of cubes (origin [m][3], one size) of the unit cube."""
        out = torch.empty(len(origin), 9, 9, 9, dtype=torch.float32, device="cuda")
        h = torch.arange(9, device="cuda", dtype=torch.float64) * (size / 8)
        for b in range(0, len(origin), 8192):
            q = origin[b:b + 8192, :, None] + h                                  # [m][3][9]
            g = torch.exp(-(q[:, :, None] - self.c.T[None, :, :, None]) ** 2 / (2 * self.s[None, None, :, None] ** 2))
            g = g.float()
            zy = (g[:, 2, :, :, None] * (g[:, 1] * self.a.float()[None, :, None])[:, :, None, :]).flatten(2)
            v = torch.bmm(zy.transpose(1, 2), g[:, 0]).reshape(-1, 9, 9, 9)
            for amp, lat in self.noise:
                n = lat.shape[0]
                i = (q * (n - 1)).floor().clamp(0, n - 2)
                f = (q * (n - 1) - i).float()
                i = i.long()
                flat = lat.float().flatten()
                r = 0.0
                for dz in (0, 1):
                    for dy in (0, 1):
                        for dx in (0, 1):
                            k = ((i[:, 2, :, None, None] + dz) * n + i[:, 1, None, :, None] + dy) * n + i[:, 0, None, None] + dx
                            wx = f[:, 0] if dx else 1 - f[:, 0]
                            wy = f[:, 1] if dy else 1 - f[:, 1]
                            wz = f[:, 2] if dz else 1 - f[:, 2]
                            r = r + flat[k] * wx[:, None, None] * wy[:, None, :, None] * wz[:, :, None, None]
                v = v + amp * r
            out[b:b + 8192] = v
        return out


def _morton(p, bits):
    p = p.astype(np.int64)
    code = np.zeros(len(p), np.int64)
    for b in range(bits):
        for c in range(3):
            code |= ((p[:, c] >> b) & 1) << (3 * b + c)
    return code


def _pieces(order, n_pieces, rng):
    """Contiguous ranges of uneven size (ratio up to 8) of the ordered units: piece id per unit."""
    n = len(order)
    n_pieces = min(n_pieces, n)
    cum = np.concatenate([[0.0], np.cumsum(8.0 ** rng.random(n_pieces))])
    cut = np.maximum((cum / cum[-1] * n).round().astype(np.int64), np.arange(n_pieces + 1))
    cut = np.minimum(cut, n - np.arange(n_pieces, -1, -1))
    piece = np.empty(n, np.int32)
    for i in range(n_pieces):
        piece[order[cut[i]:cut[i + 1]]] = i
    return piece, n_pieces


def _transfer_function(rng, alpha_max):
    pos = np.concatenate([[0.0], np.sort(rng.random(4)), [1.0]])
    x = np.arange(256) / 255.0
    alpha = alpha_max * (0.05 + 0.95 * rng.random(6))
    return np.stack([np.interp(x, pos, rng.random(6)) for _ in range(3)] + [np.interp(x, pos, alpha)], 1).astype(np.float32)


def _view(case, ext, turn):
    """A camera outside the box [0, ext], turned by `turn` about z."""
    f = lambda a: np.asarray(a, dtype=np.float32)  # noqa: E731
    ext = np.asarray(ext, np.float64)
    diag = float(np.linalg.norm(ext))
    c, s = math.cos(turn), math.sin(turn)
    w = np.array([c * VIEW_DIR[0] - s * VIEW_DIR[1], s * VIEW_DIR[0] + c * VIEW_DIR[1], VIEW_DIR[2]])
    w /= np.linalg.norm(w)
    u = np.cross(w, [0.0, 0.0, 1.0])
    u /= np.linalg.norm(u)
    v = np.cross(u, w)
    W, H = case["width"], case["height"]
    if case.get("ortho"):
        dist, su, sv = 1.5 * diag, 1.02 * diag * W / max(W, H), 1.02 * diag * H / max(W, H)
    else:
        th = math.tan(math.radians(15.0))
        dist, su, sv = 1.8 * diag, th * W / H, th
    return SimpleNamespace(eye=f(ext / 2 - dist * w), u=f(u), v=f(v), w=f(w), width=W, height=H,
                           projection=mb.MBOIT_ORTHO if case.get("ortho") else mb.MBOIT_PERSPECTIVE,
                           scale_u=np.float32(su), scale_v=np.float32(sv), near=np.float32(dist - diag / 2),
                           far=np.float32(dist + diag / 2))


@functools.lru_cache(maxsize=4)
def _hex_tets(n):
    """The five-tet split of an n^3 grid of cubes (mirrored in every other cube) and its face neighbours."""
    even = np.array([[0, 1, 2, 4], [3, 2, 1, 7], [5, 4, 7, 1], [6, 7, 4, 2], [1, 2, 4, 7]])
    corner = lambda e: np.stack([e & 1, e >> 1 & 1, e >> 2 & 1], -1)  # noqa: E731
    z, y, x = np.meshgrid(*[np.arange(n)] * 3, indexing="ij")
    cell = np.stack([x.ravel(), y.ravel(), z.ravel()], 1)
    odd = (cell.sum(1) % 2).astype(bool)
    tets = np.empty((n ** 3, 5, 4), np.int32)
    for t in range(5):
        for k in range(4):
            e = corner(even[t, k])
            p = cell + np.where(odd[:, None], [1 - e[0], e[1], e[2]], e)
            tets[:, t, k] = (p[:, 2] * (n + 1) + p[:, 1]) * (n + 1) + p[:, 0]
    tets = tets.reshape(-1, 4)
    P = np.stack([tets % (n + 1), tets // (n + 1) % (n + 1), tets // (n + 1) ** 2], -1).astype(np.int64)
    e = P[:, 1:] - P[:, :1]
    flip = np.einsum("ij,ij->i", np.cross(e[:, 0], e[:, 1]), e[:, 2]) < 0
    tets[flip, 2], tets[flip, 3] = tets[flip, 3].copy(), tets[flip, 2].copy()
    face = np.sort(np.stack([np.delete(tets, i, 1) for i in range(4)], 1).reshape(-1, 3), 1).astype(np.int64)
    key = (face[:, 0] << 42) | (face[:, 1] << 21) | face[:, 2]
    order = np.argsort(key, kind="stable")
    same = np.nonzero(key[order][1:] == key[order][:-1])[0]
    nb = np.full(len(key), -1, np.int32)
    nb[order[same]], nb[order[same + 1]] = order[same + 1] // 4, order[same] // 4
    return cell, tets, nb.reshape(-1, 4)


def _tet_volume(q, tets):
    """Six signed volumes of the tets from integer corner positions q [nv][3] (exact)."""
    a = q[tets[:, 0].long()]
    e = [q[tets[:, i].long()] - a for i in (1, 2, 3)]
    return (torch.linalg.cross(e[0], e[1], dim=1) * e[2]).sum(1)


def _scene(case, seed, which=0):
    """The arrays of one volume, from the seed alone."""
    gen = torch.Generator().manual_seed((int(seed) * 1000003 + 7919 * which) & 0x7fffffff)
    rng = np.random.default_rng([int(seed) & 0x7fffffff, which])
    tf_rng = np.random.default_rng([int(seed) & 0x7fffffff, 99])          # volumes of one frame share the table
    kind = case["kind"]
    s = SimpleNamespace(step=STEP, moment_bias=case["bias"], overestimation=OVERESTIMATION,
                        absorbance_max=ABSORBANCE_MAX, moment_set=case["moments"], storage=case["storage"])
    if kind == "grid":
        nx, ny, nz = case["nx"], case["ny"], case["nz"]
        small = max(nx, ny, nz) <= 128
        n = max(nx, ny, nz) - 1
        field = _Field(gen, 8 if small else 64, not small)
        s.field = field.tensor_grid(_axis(nx, 0, (nx - 1) / n), _axis(ny, 0, (ny - 1) / n), _axis(nz, 0, (nz - 1) / n))
        s.brick_log2 = case["brick_log2"]
        B = 1 << s.brick_log2
        s.bricks = tuple((m - 2 + B) // B for m in (nx, ny, nz))
        bz, by, bx = np.meshgrid(*[np.arange(m) for m in s.bricks[::-1]], indexing="ij")
        order = np.argsort(_morton(np.stack([bx.ravel(), by.ravel(), bz.ravel()], 1), 10), kind="stable")
        s.piece_of_brick, s.n_pieces = _pieces(order, case["pieces"], rng)
        ext, values, cells = (nx - 1, ny - 1, nz - 1), s.field, n
    elif kind == "octree":
        levels = case["max_level"]
        D = case["base"] * 8 << levels
        field = _Field(gen, 64, True)
        o = torch.arange(case["base"], device="cuda") * (8 << levels)
        cur = torch.stack(torch.meshgrid(o, o, o, indexing="ij"), -1).reshape(-1, 3).flip(1)
        table, vals = [], []
        for level in range(levels + 1):
            size = 8 << (levels - level)
            v = field.leaves(cur.double() / D, size / D)
            keep = torch.ones(len(cur), dtype=torch.bool, device="cuda")
            if level < levels:
                grad = torch.stack([v.diff(dim=c).abs().flatten(1).amax(1) for c in (1, 2, 3)]).amax(0)
                keep[grad.argsort(descending=True, stable=True)[:int(round(0.2 * len(cur)))]] = False
            table.append(torch.cat([cur[keep], torch.full((int(keep.sum()), 1), level, device="cuda")], 1))
            vals.append(v[keep])
            half = torch.tensor([[x, y, z] for z in (0, 1) for y in (0, 1) for x in (0, 1)], device="cuda") * (size // 2)
            cur = (cur[~keep][None] + half[:, None]).reshape(-1, 3)
        table = torch.cat(table).cpu().numpy().astype(np.int32)
        order = np.argsort(_morton(table[:, :3], 14), kind="stable")
        s.leaves = np.ascontiguousarray(table[order])
        s.values = torch.cat(vals)[torch.from_numpy(order).cuda()].contiguous()
        s.max_level, s.dims, s.brick_log2, s.adaptive_step = levels, (D + 1,) * 3, 3, case["adaptive"]
        s.piece_of_leaf, s.n_pieces = _pieces(np.arange(len(table)), case["pieces"], rng)
        ext, values, cells = (D,) * 3, s.values, D
    else:
        n = case["cells"]
        cell, tets, nbrs = _hex_tets(n)
        g = torch.arange(n + 1, dtype=torch.float64)
        P0 = torch.stack(torch.meshgrid(g, g, g, indexing="ij"), -1).reshape(-1, 3).flip(1)
        J = torch.rand(P0.shape, generator=gen, dtype=torch.float64) * 0.6 - 0.3
        J[(P0 == 0) | (P0 == n)] = 0.0                                     # the mesh fills its box
        P0, J, T = P0.cuda(), J.cuda(), torch.from_numpy(tets).cuda()
        v0 = _tet_volume((P0 * 16384).long(), T)
        while True:                                                        # no tet below 5 % of its volume
            q = ((P0 + J) * 16384).round().long()
            bad = _tet_volume(q, T).double() < 0.05 * v0.double()
            if not bad.any():
                break
            J[T[bad].long().unique()] *= 0.5
        P = q.double() / 16384
        values = _Field(gen, 8, False).points(P / n).float()
        s.verts = torch.cat([P.float(), values[:, None]], 1).cpu().numpy()
        s.tets, s.neighbors, s.box, s.quantum_log2 = tets, nbrs, (float(n),) * 3, 14
        piece, s.n_pieces = _pieces(np.argsort(_morton(cell, 7), kind="stable"), case["pieces"], rng)
        s.piece_of_tet = np.repeat(piece, 5)
        ext, cells = (n,) * 3, n
    lo, hi = (float(x) for x in (values.min(), values.max()))
    s.tf_range = (np.float32(lo), np.float32(hi)) if case["call"] != "multi" else (np.float32(0.0), np.float32(2.5))
    s.tf = _transfer_function(tf_rng, min(0.4, case["opacity"] / cells))
    s.ext = ext
    s.views = [_view(case, ext, 2 * math.pi * (i + which / 16) / max(case["views"], 1)) for i in range(case["views"])]
    return s


def _subset(n_pieces):
    """Every other piece."""
    return list(range(0, n_pieces, 2))


# ---------------------------------------------------------------------------
# one pass

def prepare(case, seed):
    s = SimpleNamespace(call=case["call"], moments=case["moments"])
    scenes = [_scene(case, seed, i) for i in range(case.get("volumes", 1))]
    s.vols = []
    for sc in scenes:
        flat = sc.field if case["kind"] == "grid" else sc.values if case["kind"] == "octree" else None
        s.vols.append(mb.Volume(sc, field=flat))
    s.vol = s.vols[0]
    s.views = [v for sc in scenes for v in sc.views]
    s.owner = [i for i, sc in enumerate(scenes) for _ in sc.views]
    s.mom = s.vol.moments_for(s.views)
    s.rgba = mb.Volume.color_buffer(s.views)
    s.storage = case["storage"]
    n = scenes[0].n_pieces
    if s.call == "pieces":
        s.n = n
        s.piece_mom = s.vol.moments_for(s.views, n)
        s.piece_rgba = mb.Volume.color_buffer(s.views, n)
    if s.call == "subset":
        s.pieces = _subset(n)
    if case["tuned"]:
        s.vol.autotune(s.views, s.mom, s.rgba)
    return s


def _plane(v):
    return (v.width * v.height + 3) // 4 * 4


def _outputs(s):
    """The moment slabs (16-bit planes by their own type) and the images, view by view."""
    moments, images, m, c = [], [], 0, 0
    words = 1 + (TRIG[s.moments] if s.moments in TRIG else 2 * POWER[s.moments])
    for v in s.views:
        slab = s.mom[m:m + words * _plane(v)]
        m += words * _plane(v)
        if s.moments in TRIG:
            t = slab[_plane(v):].view(torch.float16 if s.storage == "f16" else torch.bfloat16)
            moments.append([slab[:_plane(v)], t])
        else:
            moments.append([slab])
        images.append(s.rgba[c:c + 4 * v.width * v.height].view(v.height, v.width, 4))
        c += 4 * v.width * v.height
    return {"moments": moments, "rgba": images}


def run(s):
    if s.call == "frame":
        s.vol.render_frame(s.views, s.mom, s.rgba)
    elif s.call == "multi":
        mb.Volume.render_frame_multi(s.vols, s.views, s.owner, s.mom, s.rgba)
    elif s.call == "subset":
        s.vol.render_moments(s.views, s.mom, pieces=s.pieces)
        s.vol.reconstruct_blend(s.views, s.mom, s.rgba, pieces=s.pieces)
    else:
        v = s.views[0]
        s.vol.render_moments(s.views, s.piece_mom, mode=mb.MBOIT_MOMENTS_PER_PIECE)
        s.vol.composite(mb.MBOIT_OP_MOMENTS_SUM, v.width, v.height, len(s.views), s.n, s.piece_mom, s.mom)
        s.vol.reconstruct_blend(s.views, s.mom, s.piece_rgba, mode=mb.MBOIT_COLOR_PER_PIECE)
        s.vol.composite(mb.MBOIT_OP_COLOR_SUM_RESOLVE, v.width, v.height, len(s.views), s.n, s.piece_rgba, s.rgba,
                        global_moments=s.mom)
        out = _outputs(s)
        if s.moments in TRIG:   # the 16-bit planes interleave with float32 ones: per-piece slabs stay as they are
            return {**out, "piece_rgba": s.piece_rgba}
        return {**out, "piece_moments": s.piece_mom, "piece_rgba": s.piece_rgba}
    return _outputs(s)


# ---------------------------------------------------------------------------
# the work a pass cannot do without

def _extent(case):
    if case["kind"] == "grid":
        return (case["nx"] - 1, case["ny"] - 1, case["nz"] - 1)
    return (case["base"] * 8 << case["max_level"],) * 3 if case["kind"] == "octree" else (case["cells"],) * 3


def _rays(v, px, py):
    """Rays of pixels (float32, every operation rounded, in the order the interface defines)."""
    f = np.float32
    fx, fy = px.astype(f) + f(0.5), py.astype(f) + f(0.5)
    if v.projection == mb.MBOIT_ORTHO:
        sx, sy = (fx / f(v.width) - f(0.5)) * v.scale_u, (fy / f(v.height) - f(0.5)) * v.scale_v
        o = np.stack([(v.eye[c] + sx * v.u[c]) + sy * v.v[c] for c in range(3)], 1)
        return o, np.broadcast_to(v.w, o.shape).copy()
    sx, sy = (f(2) * fx / f(v.width) - f(1)) * v.scale_u, (f(2) * fy / f(v.height) - f(1)) * v.scale_v
    d = np.stack([(v.w[c] + sx * v.u[c]) + sy * v.v[c] for c in range(3)], 1)
    d /= np.sqrt((d[:, 0] * d[:, 0] + d[:, 1] * d[:, 1]) + d[:, 2] * d[:, 2])[:, None]
    return np.broadcast_to(v.eye, d.shape).copy(), d


def _span(o, d, ext):
    """Ray parameters of the box [0, ext] (entry, exit), float64."""
    with np.errstate(divide="ignore", invalid="ignore"):
        a, b = -o.astype(np.float64) / d, (np.asarray(ext, np.float64) - o) / d
    return np.nanmax(np.minimum(a, b), 1).clip(0), np.nanmin(np.maximum(a, b), 1)


def _samples(case):
    """Lattice points inside the box over all views, from a coarse set of rays."""
    total = 0.0
    for i in range(case.get("volumes", 1)):
        for j in range(case["views"]):
            v = _view(case, _extent(case), 2 * math.pi * (j + i / 16) / max(case["views"], 1))
            y, x = np.meshgrid(np.linspace(0, v.height - 1, 64).round(), np.linspace(0, v.width - 1, 64).round(),
                               indexing="ij")
            t0, t1 = _span(*_rays(v, x.ravel(), y.ravel()), _extent(case))
            total += float(np.maximum(t1 - t0, 0).mean()) / STEP * v.width * v.height
    return total


def work(case):
    n = _samples(case)
    px = case["width"] * case["height"] * case["views"] * case.get("volumes", 1)
    moments = case["moments"]
    # floating-point operations of a sample (fma = 2): position, interpolation, table, depth and moments of pass 1;
    # table, opacity, moment bound and colour of pass 2
    p1 = {"grid": 49, "octree": 55, "mesh": 90}[case["kind"]] + {"power4": 0, "power6": 4, "power8": 8, "trig6": 12,
                                                                 "trig8": 20}[moments]
    p2 = 33 + {"power4": 35, "power6": 120, "power8": 220, "trig6": 250, "trig8": 400}[moments]
    if case["call"] in ("subset", "pieces"):
        p2 += 30                                     # pass 2 samples the volume again
    if case["call"] == "subset":
        n *= 0.5
    if case["kind"] == "octree" and case["adaptive"]:
        n *= 0.35                                    # coarse leaves are sampled on a coarser lattice
    slab = 4 + 4 * (TRIG[moments] if moments in TRIG else 2 * POWER[moments])
    volume = {"grid": lambda: 4 * case["nx"] * case["ny"] * case["nz"] * case.get("volumes", 1),
              "octree": lambda: _leaf_count(case) * 729 * 4,
              "mesh": lambda: (case["cells"] + 1) ** 3 * 16 + case["cells"] ** 3 * 5 * 32}[case["kind"]]()
    image = px * (slab + 16)
    if case["call"] == "pieces":
        image += px * case["pieces"] * 2 * (slab + 16)   # written by the passes, read by the sums
        volume *= 2
    elif case["call"] == "subset":
        image += px * slab
    return {"bytes": float(volume + image), "flops": float(n * (p1 + p2))}


def _leaf_count(case):
    cur, total = case["base"] ** 3, 0
    for level in range(case["max_level"] + 1):
        r = int(round(0.2 * cur)) if level < case["max_level"] else 0
        total += cur - r
        cur = 8 * r
    return total


# ---------------------------------------------------------------------------
# the same in 64 bits

def _sampler(case, s):
    """p [m][3] (float32 positions inside the box) -> (value, piece, level shift), 64 bits."""
    kind = case["kind"]
    if kind == "grid":
        field = s.field.double().flatten()
        nx, ny = case["nx"], case["ny"]
        pob = torch.from_numpy(s.piece_of_brick).cuda()

        def sample(p):
            i = p.floor()
            f = p - i
            i = i.long()
            c = (i[:, 2] * ny + i[:, 1]) * nx + i[:, 0]
            b = i >> s.brick_log2
            piece = pob[(b[:, 2] * s.bricks[1] + b[:, 1]) * s.bricks[0] + b[:, 0]]
            return _trilinear(field, c, nx, nx * ny, f), piece, None
        return sample
    if kind == "octree":
        D, levels = s.dims[0] - 1, s.max_level
        nb = D // 8
        leaves = torch.from_numpy(s.leaves).cuda().long()
        fmap = torch.full((nb, nb, nb), -1, dtype=torch.long, device="cuda")
        ids = torch.arange(len(leaves), device="cuda")
        for level in range(levels + 1):
            at = leaves[:, 3] == level
            k = 1 << (levels - level)
            o = leaves[at][:, :3] // 8
            for dz in range(k):
                for dy in range(k):
                    for dx in range(k):
                        fmap[o[:, 2] + dz, o[:, 1] + dy, o[:, 0] + dx] = ids[at]
        fmap = fmap.flatten()
        values = s.values.flatten()
        pol = torch.from_numpy(s.piece_of_leaf).cuda()

        def sample(p):
            b = p.floor().long() // 8
            leaf = fmap[(b[:, 2] * nb + b[:, 1]) * nb + b[:, 0]]
            L = leaves[leaf]
            shift = levels - L[:, 3]
            q = (p - L[:, :3]) * torch.pow(0.5, shift.double())[:, None]
            i = q.floor().clamp(max=7)
            f = q - i
            i = i.long()
            return (_trilinear(values, leaf * 729 + (i[:, 2] * 9 + i[:, 1]) * 9 + i[:, 0], 9, 81, f), pol[leaf],
                    shift if s.adaptive_step else None)
        return sample
    n = case["cells"]
    verts = torch.from_numpy(s.verts).cuda().double()
    T = torch.from_numpy(s.tets).cuda().long()
    P = verts[T][:, :, :3]
    A = torch.cat([P, torch.ones_like(P[:, :, :1])], 2).transpose(1, 2)      # columns (x, y, z, 1) of the corners
    inv = torch.linalg.inv(A)
    lin = (verts[T][:, None, :, 3] @ inv)[:, 0]                              # the value as an affine function
    pot = torch.from_numpy(s.piece_of_tet).cuda()

    def sample(p):
        p = _snap(p)
        home = p.floor().long().clamp(max=n - 1)
        best = torch.full((len(p),), -math.inf, dtype=torch.float64, device="cuda")
        tet = torch.zeros(len(p), dtype=torch.long, device="cuda")
        ring = [(0, 0, 0)] + [(x, y, z) for z in (-1, 0, 1) for y in (-1, 0, 1) for x in (-1, 0, 1) if x or y or z]
        live = torch.arange(len(p), device="cuda")
        for dx, dy, dz in ring:
            c = home[live] + torch.tensor([dx, dy, dz], device="cuda")
            ok = ((c >= 0) & (c < n)).all(1)
            c = c.clamp(0, n - 1)
            base = ((c[:, 2] * n + c[:, 1]) * n + c[:, 0]) * 5
            ph = torch.cat([p[live], torch.ones_like(p[live][:, :1])], 1)
            for k in range(5):
                low = (inv[base + k] * ph[:, None]).sum(2).amin(1)
                low = torch.where(ok, low, -math.inf)
                better = low > best[live]
                best[live] = torch.where(better, low, best[live])
                tet[live] = torch.where(better, base + k, tet[live])
            live = live[best[live] < 0]
            if not len(live):
                break
        return (lin[tet] * torch.cat([p, torch.ones_like(p[:, :1])], 1)).sum(1), pot[tet], None
    return sample


def _snap(p):
    """Positions on the lattice that the mesh's point location works on (2^-14)."""
    return torch.round(p * 16384) / 16384


def _trilinear(v, c, sy, sz, f):
    x, y, z = f.unbind(1)
    at = lambda k: v[c + k].double()  # noqa: E731
    lerp = lambda a, b, t: a + t * (b - a)  # noqa: E731
    lo = lerp(lerp(at(0), at(1), x), lerp(at(sy), at(sy + 1), x), y)
    hi = lerp(lerp(at(sz), at(sz + 1), x), lerp(at(sz + sy), at(sz + sy + 1), x), y)
    return lerp(lo, hi, z)


def _power_fraction(m, z, N, beta):
    """Fraction of the optical depth in front of z [p][k] from moments m [p][2N + 1]: the canonical representation
    through z, its other support points from the kernel polynomial, its weights from the kernel's diagonal."""
    law = [1.0, 0.0, 0.375 if N == 2 else 0.5, 0.0, 0.375, 0.0, 0.3125, 0.0, 0.2734375]
    b = [(1 - beta) * m[:, j] / m[:, 0] + beta * law[j] for j in range(2 * N + 1)]
    mu = b[1]
    sd = (b[2] - mu * mu).sqrt()
    h = [sum(math.comb(j, i) * b[i] * (-mu) ** (j - i) for i in range(j + 1)) / sd ** j for j in range(2 * N + 1)]
    H = torch.stack([torch.stack([h[i + j] for j in range(N + 1)], 1) for i in range(N + 1)], 1)
    Li = torch.linalg.inv(torch.linalg.cholesky_ex(H)[0])
    x0 = (z - mu[:, None]) / sd[:, None]

    def kernel(x):
        y = [sum(Li[:, i, j, None] * x ** j for j in range(i + 1)) for i in range(N + 1)]
        return y, sum(t * t for t in y)
    y, K = kernel(x0)
    q = [sum(Li[:, i, j, None] * y[i] for i in range(j, N + 1)) for j in range(N + 1)]
    r = list(q)                                       # K(x0 + 1 / s, x0) s^N, highest power of s first
    for k in range(N):
        for i in range(N - 1, k - 1, -1):
            r[i] = r[i] + x0 * r[i + 1]
    A = OVERESTIMATION / K
    for root in _roots([c / r[0] for c in r[1:]]):
        safe = torch.where(root < -1e-9, root, torch.full_like(root, -1.0))
        A = A + torch.where(root < -1e-9, 1 / kernel(x0 + 1 / safe)[1], 0.0)
    return A.clamp(0, 1)


def _roots(c):
    """Roots of the monic polynomial s^n + c[0] s^(n-1) + ... whose roots are all real (n = 2, 3, 4)."""
    n = len(c)
    if n == 2:
        d = (c[0] * c[0] / 4 - c[1]).clamp(min=0).sqrt()
        big = -c[0] / 2 - torch.where(c[0] >= 0, d, -d)
        return [big, torch.where(big != 0, c[1] / big, 0.0)]
    if n == 3:
        r = _cubic(*c)
    else:
        a, b, cc, d = c
        p = b - 0.375 * a * a
        q = cc - 0.5 * a * b + 0.125 * a ** 3
        w = d - 0.25 * a * cc + a * a * b / 16 - 3 * a ** 4 / 256
        m = _cubic(p, 0.25 * p * p - w, -0.125 * q * q)[0].clamp(min=1e-280)
        e = (2 * m).sqrt()
        g = q / (2 * e)
        d1 = (e * e - 4 * (0.5 * p + m + g)).clamp(min=0).sqrt()
        d2 = (e * e - 4 * (0.5 * p + m - g)).clamp(min=0).sqrt()
        r = [0.5 * (e + d1) - a / 4, 0.5 * (e - d1) - a / 4, 0.5 * (d2 - e) - a / 4, 0.5 * (-d2 - e) - a / 4]
    out = []
    for s in r:
        for _ in range(3):
            f, df = torch.ones_like(s), torch.zeros_like(s)
            for k in c:
                df = df * s + f
                f = f * s + k
            step = torch.where(df != 0, f / torch.where(df != 0, df, 1.0), 0.0)
            s = s - torch.where(step.abs() < 1e-3 * (1 + s.abs()), step, 0.0)
        out.append(s)
    return out


def _cubic(a, b, c):
    """Roots of s^3 + a s^2 + b s + c, all real, the largest first."""
    p = (b - a * a / 3).clamp(max=-1e-300)
    q = 2 * a ** 3 / 27 - a * b / 3 + c
    m = 2 * (-p / 3).sqrt()
    th = torch.acos((3 * q / (p * m)).clamp(-1, 1)) / 3
    return [m * torch.cos(th - 2 * math.pi * k / 3) - a / 3 for k in (0, 1, 2)]


def _trig_fraction(tau, z, n, beta):
    """The same from n complex trigonometric moments tau [p][n] (already divided by b0), depth angle 0.9 pi z."""
    t = [torch.ones_like(tau[:, 0])] + [(1 - beta) * tau[:, j] for j in range(n)]
    G = torch.stack([torch.stack([t[k - l].conj() if k >= l else t[l - k] for l in range(n + 1)], 1)
                     for k in range(n + 1)], 1)
    Li = torch.linalg.inv(torch.linalg.cholesky_ex(G)[0])
    phi = 0.9 * math.pi * z
    u0 = torch.polar(torch.ones_like(phi), phi)

    def kernel(u):
        y = [sum(Li[:, i, j, None] * u.conj() ** j for j in range(i + 1)) for i in range(n + 1)]
        return y, sum((v.conj() * v).real for v in y)
    y, K = kernel(u0)
    g = [sum(Li[:, i, j, None].conj() * y[i] for i in range(j, n + 1)) * u0 ** j for j in range(n + 1)]
    coef = [torch.zeros_like(phi) for _ in range(n + 1)]
    for k in range(n + 1):                            # (s + i)^k (s - i)^(n - k)
        p = np.poly1d([1.0])
        for _ in range(k):
            p = p * np.poly1d([1.0, 1j])
        for _ in range(n - k):
            p = p * np.poly1d([1.0, -1j])
        for m, v in enumerate(np.concatenate([np.zeros(n - p.order), p.c])):
            coef[m] = coef[m] + (g[k] * complex(v)).real
    A = OVERESTIMATION / K
    edge = torch.tan(phi / 2)
    for s in _roots([c / K for c in coef[1:]]):
        e = torch.complex(s * s - 1, 2 * s) / (s * s + 1)
        A = A + torch.where(s < edge, 1 / kernel(u0 * e)[1], 0.0)
    return A


def _exact_view(case, s, v, sample, selected):
    """Moments and colour sums of one view: per piece or (selected pieces) of all of them, and the image."""
    moments, npx = case["moments"], v.width * v.height
    n_out = len(selected) if case["call"] == "pieces" else 1
    nm = TRIG[moments] if moments in TRIG else 2 * POWER[moments]
    dtype = torch.complex128 if moments in TRIG else torch.float64
    mom = torch.zeros(n_out, npx, nm, dtype=dtype, device="cuda")
    b0 = torch.zeros(n_out, npx, dtype=torch.float64, device="cuda")
    col = torch.zeros(n_out, npx, 4, dtype=torch.float64, device="cuda")
    tf = torch.from_numpy(s.tf.astype(np.float64)).cuda()
    table = torch.cat([tf[:, :3], -torch.log1p(-tf[:, 3:]) * STEP], 1)
    lo, hi = float(s.tf_range[0]), float(s.tf_range[1])
    ext = torch.tensor(np.asarray(s.ext, np.float64), device="cuda")
    near, far = math.log(float(v.near)), math.log(float(v.far))
    sel = torch.zeros(s.n_pieces, dtype=torch.bool, device="cuda")
    sel[selected] = True
    everything = len(selected) == s.n_pieces and n_out == 1
    o, d = _rays(v, np.arange(npx) % v.width, np.arange(npx) // v.width)
    t0, t1 = _span(o, d, s.ext)
    k0 = np.floor(t0 / STEP - 0.5).astype(np.int64).clip(0) - 2
    count = np.where(t1 >= t0, np.floor(t1 / STEP - 0.5).astype(np.int64) + 3 - k0, 0)
    first = 0
    while first < npx:
        # as many pixels as make some 8 M lattice points
        longest = np.maximum.accumulate(count[first:first + (1 << 20)]) * np.arange(1, min(1 << 20, npx - first) + 1)
        last = first + max(1, int(np.searchsorted(longest, 8 << 20)))
        c = np.arange(first, min(last, npx))
        first = last
        kmax = int(count[c].max())
        if kmax <= 0:
            continue
        k = torch.from_numpy(k0[c].clip(0)).cuda()[:, None] + torch.arange(kmax, device="cuda")
        t = (k.double() + 0.5) * STEP
        O, D = torch.from_numpy(o[c]).cuda().double(), torch.from_numpy(d[c]).cuda().double()
        p = (t[..., None] * D[:, None] + O[:, None]).float().double()
        inside = ((p >= 0) & (p < ext)).all(2)
        if case["kind"] == "mesh":                    # no tet owns a point that snaps onto the far faces
            inside &= (_snap(p) < ext).all(2)
        r, kk = inside.nonzero(as_tuple=True)
        value, piece, shift = sample(p[r, kk])
        x = ((value - lo) * (255.0 / (hi - lo))).clamp(0, 255)
        i = x.floor().long().clamp(max=254)
        f = (x - i)[:, None]
        e = table[i] + f * (table[i + 1] - table[i])
        a1 = e[:, 3]
        if shift is not None:
            a1 = torch.where(k[r, kk] % (1 << shift) == 0, a1 * (1 << shift), 0.0)
        a1 = a1.clamp(max=ABSORBANCE_MAX)
        if not everything:
            a1 = torch.where(sel[piece.long()], a1, 0.0)
        a = torch.zeros_like(t)
        a[r, kk] = a1
        rgb = torch.zeros(*t.shape, 3, dtype=torch.float64, device="cuda")
        rgb[r, kk] = e[:, :3]
        z = (2 * (torch.log(t) - near) / (far - near) - 1).clamp(-1, 1)
        idx = torch.from_numpy(c).cuda()
        if n_out > 1:
            owner = torch.full_like(k, -1)
            owner[r, kk] = piece.long()
        basis = [torch.polar(torch.ones_like(z), (j + 1) * 0.9 * math.pi * z) for j in range(nm)] if moments in TRIG else \
            [z ** (j + 1) for j in range(nm)]
        for j in range(n_out):
            w = a if n_out == 1 else torch.where(owner == selected[j], a, 0.0)
            b0[j, idx] = w.sum(1)
            for q in range(nm):
                mom[j, idx, q] = (w * basis[q]).sum(1)
        m0, m = b0[:, idx].sum(0), mom[:, idx].sum(0)
        hit = m0 > 0
        if not hit.any():
            continue
        if moments in TRIG:
            A = _trig_fraction(_stored(m / m0[:, None], case["storage"])[hit], z[hit], nm, case["bias"])
        else:
            A = _power_fraction(torch.cat([m0[:, None], m], 1)[hit], z[hit], nm // 2, case["bias"])
        wgt = torch.exp(-m0[hit, None] * A) * -torch.expm1(-a[hit])
        for j in range(n_out):
            w = wgt if n_out == 1 else torch.where(owner[hit] == selected[j], wgt, 0.0)
            col[j, idx[hit], :3] = (w[..., None] * rgb[hit]).sum(1)
            col[j, idx[hit], 3] = w.sum(1)
    C, m0 = col.sum(0), b0.sum(0)
    A = -torch.expm1(-m0)
    image = torch.cat([C[:, :3] * torch.where(C[:, 3] > 0, A / C[:, 3].clamp(min=1e-300), 0.0)[:, None], A[:, None]], 1)
    return b0, mom, col, image.view(v.height, v.width, 4)


def _stored(tau, storage):
    """Rounded to the 16-bit storage format, as the interface defines it."""
    kind = torch.float16 if storage == "f16" else torch.bfloat16
    return torch.complex(tau.real.to(kind).double(), tau.imag.to(kind).double())


def _slabs(case, v, b0, mom):
    """[j] slabs of float words in the interface's layout (power moments)."""
    P, n, npx = _plane(v), mom.shape[2], mom.shape[1]
    out = torch.zeros(mom.shape[0], (1 + n) * P, dtype=torch.float64, device="cuda")
    out[:, :npx] = b0
    out[:, P:5 * P].view(-1, P, 4)[:, :npx] = mom[:, :, :4]
    if n > 4:
        out[:, 5 * P:].view(-1, P, n - 4)[:, :npx] = mom[:, :, 4:]
    return out


def exact(case, seed):
    res = {"moments": [], "rgba": []}
    piece_moments, piece_rgba = [], []
    for i in range(case.get("volumes", 1)):
        s = _scene(case, seed, i)
        sample = _sampler(case, s)
        selected = _subset(s.n_pieces) if case["call"] == "subset" else list(range(s.n_pieces))
        for v in s.views:
            b0, mom, col, image = _exact_view(case, s, v, sample, selected)
            if case["moments"] in TRIG:
                P, n = _plane(v), mom.shape[2]
                plane = torch.zeros(P, dtype=torch.float64, device="cuda")
                plane[:len(b0[0])] = b0.sum(0)
                tau = torch.zeros(n, P, 2, dtype=torch.float64, device="cuda")
                m0 = b0.sum(0)
                t = torch.where(m0[:, None] > 0, mom.sum(0) / m0.clamp(min=1e-300)[:, None], 0.0)
                tau[:, :len(m0)] = torch.view_as_real(t).transpose(0, 1)
                res["moments"].append([plane, tau.flatten()])
            else:
                res["moments"].append([_slabs(case, v, b0.sum(0, keepdim=True), mom.sum(0, keepdim=True))[0]])
                piece_moments.append(_slabs(case, v, b0, mom).flatten())
            res["rgba"].append(image)
            piece_rgba.append(col.flatten())
    if case["call"] == "pieces":
        res["piece_rgba"] = torch.cat(piece_rgba)
        if case["moments"] not in TRIG:
            res["piece_moments"] = torch.cat(piece_moments)
    return res
