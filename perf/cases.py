"""The calls whose speed is tracked: the DPSR layer (forward and backward)
from the smallest to the largest grid, its batched training step and its
host-buffer form, and the kernels that losses around it run on (grid lookup,
mesh points, mesh sampling, Chamfer distance), each through the entry point
that a program calls.

Grids and clouds are those of the paper's schedule, of synth.py's workloads
and of the tests: r = 32 .. 512, 1 000 .. 200 000 points on closed surfaces
with unit normals and position noise, sigma 2 .. 3.
"""
from __future__ import annotations

import math
import random

import torch

from paper_2106_03452_gb300 import libdpsr as L
from paper_2106_03452_gb300.dpsr import Batch, Plan, dpsr
from paper_2106_03452_gb300.loop import GridSample
from paper_2106_03452_gb300.mesh import MeshPoints, sample
from paper_2106_03452_gb300.optimize import chamfer

DEV = "cuda"
JITTER = 0.003  # position noise of the clouds (synth.py)


def listed():
    return [
        # first level of the coarse-to-fine optimisation: one small solve, where launches count
        dict(name="layer_r32", op="layer", r=32, n=3000, sigma=2.0),
        # an anisotropic domain with an odd number of points
        dict(name="layer_r64_box", op="layer", r=64, n=8191, sigma=2.0, bx=1.0, by=0.75, bz=1.5),
        # the layer at the grid size that the paper trains with
        dict(name="layer_r128", op="layer", r=128, n=20000, sigma=2.0),
        # the last level of the optimisation: 256^3, the noisy cloud of the r = 256 loop
        dict(name="layer_r256", op="layer", r=256, n=100000, sigma=3.0),
        # the largest grid
        dict(name="layer_r512", op="layer", r=512, n=200000, sigma=3.0),
        # reconstruction without gradients, as most served requests are
        dict(name="forward_r256", op="forward", r=256, n=150001, sigma=2.0),
        # a training step of the learning setting: clouds of uneven size and both grid sizes
        dict(name="train_batch", op="train", count=12, mix=3, n_lo=1000, n_hi=50000, sigma=2.0),
        # one whole solve from pinned host buffers and back
        dict(name="host_r128", op="host", r=128, n=20000, sigma=2.0),
        # a loss on chi at target points: lookup and its adjoint
        dict(name="lookup_r256", op="lookup", r=256, m=200000),
        # Chamfer distance of the optimisation: 20 000 mesh samples against the input cloud
        dict(name="chamfer_20k", op="chamfer", na=20000, nb=20000, noise=0.005),
        # mesh points of the indicator and the gradient through them (Eq. 6)
        dict(name="mesh_r128", op="mesh", r=128),
        # 20 000 points drawn by area on the triangles that a 128^3 mesh has
        dict(name="sample_20k", op="sample", t=150001, m=20000),
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    op = rng.choice(["layer", "layer", "layer", "forward", "train", "host", "lookup", "chamfer", "mesh", "sample"])
    sigma = rng.choice([2.0, 3.0, 2.5, 5.0])
    if op in ("layer", "forward"):
        r = rng.choice([32, 64, 128, 256, 512])
        c = dict(op=op, r=r, n=_log_int(rng, 1000, 199999), sigma=sigma)
        if op == "layer" and rng.random() < 0.25:
            c.update(bx=1.0, by=round(rng.uniform(0.6, 1.0), 3), bz=round(rng.uniform(1.0, 1.6), 3))
        return c
    if op == "train":
        return dict(op=op, count=rng.randint(3, 12), mix=rng.randrange(1 << 16), n_lo=1000, n_hi=50000, sigma=sigma)
    if op == "host":
        return dict(op=op, r=rng.choice([64, 128]), n=_log_int(rng, 1000, 50000), sigma=sigma)
    if op == "lookup":
        return dict(op=op, r=rng.choice([64, 128, 256]), m=_log_int(rng, 2000, 200000))
    if op == "chamfer":
        return dict(op=op, na=_log_int(rng, 1000, 30000), nb=_log_int(rng, 1000, 30000),
                    noise=rng.choice([0.0005, 0.005, 0.05]))
    if op == "mesh":
        return dict(op=op, r=rng.choice([32, 64, 128, 256]))
    return dict(op=op, t=_log_int(rng, 4000, 800000), m=_log_int(rng, 4000, 50000))


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------
def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    return g


def _shape(g, k):
    """k ellipsoids: centres U[0.3, 0.7]^3, semi-axes U[0.08, 0.25], random rotations."""
    c = 0.3 + 0.4 * torch.rand((k, 3), generator=g, device=DEV)
    a = 0.08 + 0.17 * torch.rand((k, 3), generator=g, device=DEV)
    q = torch.nn.functional.normalize(torch.randn((k, 4), generator=g, device=DEV), dim=1)
    w, x, y, z = q.unbind(1)
    rot = torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - z * w), 2 * (x * z + y * w),
                       2 * (x * y + z * w), 1 - 2 * (x * x + z * z), 2 * (y * z - x * w),
                       2 * (x * z - y * w), 2 * (y * z + x * w), 1 - 2 * (x * x + y * y)], 1).reshape(k, 3, 3)
    return c, a, rot


def _cloud(g, shape, n, jitter=JITTER):
    """n points on the boundary of the union, with outward unit normals and noise."""
    c, a, rot = shape
    k = c.shape[0]
    m = 4 * n + 256
    which = torch.randint(0, k, (m,), generator=g, device=DEV)
    d = torch.nn.functional.normalize(torch.randn((m, 3), generator=g, device=DEV), dim=1)
    p = c[which] + torch.einsum("mij,mj->mi", rot[which], a[which] * d)
    nr = torch.nn.functional.normalize(torch.einsum("mij,mj->mi", rot[which], d / a[which]), dim=1)
    keep = torch.ones(m, dtype=torch.bool, device=DEV)
    for j in range(k):
        inside = ((((p - c[j]) @ rot[j]) / a[j]) ** 2).sum(1) < 1.0
        keep &= ~inside | (which == j)
    i = keep.nonzero().reshape(-1)
    i = i[torch.arange(n, device=DEV) % i.numel()]
    p = p[i] + jitter * torch.randn((n, 3), generator=g, device=DEV)
    return p.contiguous(), nr[i].contiguous()


def _indicator(shape, r):
    """A smooth indicator of the union on the r^3 grid: -0.5 inside, 0.5 outside."""
    c, a, rot = shape
    t = torch.arange(r, device=DEV, dtype=torch.float32) / r
    x = torch.stack(torch.meshgrid(t, t, t, indexing="ij"), -1).reshape(-1, 3)
    f = None
    for j in range(c.shape[0]):
        e = ((((x - c[j]) @ rot[j]) / a[j]).norm(dim=1) - 1.0) * a[j].min()
        f = e if f is None else torch.minimum(f, e)
    return (0.5 * torch.tanh(f * (r / 4.0))).reshape(r, r, r).contiguous()


def _box(case):
    return (case["bx"], case["by"], case["bz"]) if "bx" in case else None


def _train_sizes(case):
    rng = random.Random(case["mix"])
    rs = [rng.choice([64, 128]) for _ in range(case["count"])]
    return rs, [_log_int(rng, case["n_lo"], case["n_hi"]) for _ in rs]


def _soup(g, t):
    """t triangles of the size that extraction gives: small, on the boundary of an ellipsoid."""
    shape = _shape(g, 1)
    p, nr = _cloud(g, shape, t, 0.0)
    e = 0.6 / math.sqrt(t)
    tris = p[:, None, :] + e * torch.randn((t, 3, 3), generator=g, device=DEV)
    return tris.contiguous(), nr


def _inputs(case, seed):
    """The arrays of a case, made from the seed alone."""
    g = _gen(seed)
    op = case["op"]
    if op in ("layer", "forward", "host"):
        p, n = _cloud(g, _shape(g, 4), case["n"])
        b = _box(case)
        if b is not None:
            p = p * torch.tensor(b, device=DEV)
        r = case["r"]
        d = torch.randn((r, r, r), generator=g, device=DEV) if op != "forward" else None
        return dict(p=p, n=n, dchi=d)
    if op == "train":
        rs, ns = _train_sizes(case)
        out = []
        for r, n in zip(rs, ns):
            shape = _shape(g, 3)
            p, nr = _cloud(g, shape, n, 0.005)
            out.append(dict(r=r, p=p, n=nr, target=_indicator(shape, r)))
        return out
    if op == "lookup":
        shape = _shape(g, 3)
        q, _ = _cloud(g, shape, case["m"], 0.0)
        return dict(chi=_indicator(shape, case["r"]), q=q, w=torch.randn(case["m"], generator=g, device=DEV))
    if op == "chamfer":  # mesh samples and the cloud they are fitted to
        shape = _shape(g, 3)
        b, _ = _cloud(g, shape, case["nb"])
        a, _ = _cloud(g, shape, case["na"], case["noise"])
        return dict(a=a, b=b)
    if op == "mesh":
        return dict(chi=_indicator(_shape(g, 3), case["r"]), centre=torch.tensor([0.5, 0.5, 0.5], device=DEV))
    tris, nr = _soup(g, case["t"])
    return dict(tris=tris, nrm=nr, seed=seed)


def prepare(case, seed):
    op = case["op"]
    x = _inputs(case, seed)
    s = dict(op=op, case=dict(case), x=x)
    if op in ("layer", "forward", "host"):
        s["plan"] = Plan(case["r"], case["sigma"], n_max=case["n"], box=_box(case))
    if op == "layer":
        x["p"].requires_grad_(True)
        x["n"].requires_grad_(True)
    elif op == "host":
        pin = lambda t: t.cpu().pin_memory()  # noqa: E731
        r, n = case["r"], case["n"]
        s["x"] = dict(p=pin(x["p"]), n=pin(x["n"]), dchi=pin(x["dchi"]))
        s["chi"] = torch.empty((r, r, r), pin_memory=True)
        s["dp"], s["dn"] = torch.empty((n, 3), pin_memory=True), torch.empty((n, 3), pin_memory=True)
    elif op == "train":
        rs = [i["r"] for i in x]
        b = Batch(rs, [case["sigma"]] * len(rs), [i["p"].shape[0] for i in x])
        s["batch"], s["out"] = b, []
        for k, i in enumerate(x):
            r, e = i["r"], torch.empty_like
            chi, dchi = torch.empty((r, r, r), device=DEV), torch.empty((r, r, r), device=DEV)
            o = (chi, dchi, e(i["p"]), e(i["n"]))
            b.bind(k, i["p"], i["n"], *o)
            b.bind_target(k, i["target"])
            s["out"].append(o)
    elif op in ("lookup", "mesh"):
        x["chi"].requires_grad_(True)
    elif op == "chamfer":
        x["a"].requires_grad_(True)
    return s


# ---------------------------------------------------------------------------
# One pass
# ---------------------------------------------------------------------------
def run(s):
    op, x = s["op"], s["x"]
    if op == "layer":
        chi = dpsr(x["p"], x["n"], s["plan"])
        dp, dn = torch.autograd.grad(chi, (x["p"], x["n"]), x["dchi"])
        return dict(chi=chi, dpoints=dp, dnormals=dn)
    if op == "forward":
        return dict(chi=s["plan"].forward(x["p"], x["n"]))
    if op == "train":
        s["batch"].train_step()
        return [dict(chi=o[0], dchi=o[1], dpoints=o[2], dnormals=o[3]) for o in s["out"]]
    if op == "host":
        L.dpsr_solve_host(s["plan"].handle, x["p"].data_ptr(), x["n"].data_ptr(), x["p"].shape[0],
                          x["dchi"].data_ptr(), s["chi"].data_ptr(), s["dp"].data_ptr(), s["dn"].data_ptr())
        return dict(chi=s["chi"], dpoints=s["dp"], dnormals=s["dn"])
    if op == "lookup":
        v = GridSample.apply(x["chi"], x["q"])
        (g,) = torch.autograd.grad(v, x["chi"], x["w"])
        return dict(values=v, dchi=g)
    if op == "chamfer":
        loss = chamfer(x["a"], x["b"])
        (g,) = torch.autograd.grad(loss, x["a"])
        return dict(loss=loss, da=g)
    if op == "mesh":
        # the loss sum |p - centre|^2 / 2 over the mesh points; the points themselves
        # come in an order of their own at each call, their gradient on the grid does not
        p, _ = MeshPoints.apply(x["chi"])
        (g,) = torch.autograd.grad(p, x["chi"], p.detach() - x["centre"])
        return dict(points=p.shape[0], dchi=g)
    p, n = sample(x["tris"], x["nrm"], s["case"]["m"], x["seed"])
    return dict(points=p, normals=n)


# ---------------------------------------------------------------------------
# What a pass cannot do without
# ---------------------------------------------------------------------------
def _fft_flops(r, transforms):
    return transforms * 2.5 * r ** 3 * math.log2(float(r) ** 3)  # real transforms of r^3 values


def work(case):
    op = case["op"]
    if op in ("layer", "host"):  # points, normals and their gradients; chi and dchi
        return dict(bytes=48 * case["n"] + 8 * case["r"] ** 3, flops=_fft_flops(case["r"], 8))
    if op == "forward":
        return dict(bytes=24 * case["n"] + 4 * case["r"] ** 3, flops=_fft_flops(case["r"], 4))
    if op == "train":
        rs, ns = _train_sizes(case)
        return dict(bytes=sum(48 * n + 12 * r ** 3 for r, n in zip(rs, ns)), flops=sum(_fft_flops(r, 8) for r in rs))
    if op == "lookup":  # at most the whole grid is read; it is written once
        return dict(bytes=4 * case["r"] ** 3 + min(4 * case["r"] ** 3, 32 * case["m"]) + 20 * case["m"],
                    flops=60 * case["m"])
    if op == "chamfer":  # one distance per point at least
        return dict(bytes=24 * case["na"] + 12 * case["nb"], flops=20 * (case["na"] + case["nb"]))
    if op == "mesh":
        return dict(bytes=8 * case["r"] ** 3, flops=8 * case["r"] ** 3)
    return dict(bytes=36 * case["t"] + 24 * case["m"], flops=20 * case["t"] + 40 * case["m"])


# ---------------------------------------------------------------------------
# The same in 64 bits
# ---------------------------------------------------------------------------
def _corners(c, r, box=None):
    """Trilinear stencil of points c (64 bits): [(flat index, weight)] of the 8 corners."""
    x = c * r if box is None else c * (r / torch.tensor(box, device=c.device, dtype=c.dtype))
    f = torch.floor(x.detach())
    t, i = x - f, f.long()
    out = []
    for k in range(8):
        d = [(k >> 2) & 1, (k >> 1) & 1, k & 1]
        w = 1.0
        for a in range(3):
            w = w * (t[:, a] if d[a] else 1.0 - t[:, a])
        j = [(i[:, a] + d[a]) % r for a in range(3)]
        out.append(((j[0] * r + j[1]) * r + j[2], w))
    return out


def _solve64(p, n, r, sigma, box=None):
    st = _corners(p, r, box)
    f = torch.fft.fftfreq(r, 1.0 / r, device=DEV, dtype=torch.float64)
    lens = (1.0, 1.0, 1.0) if box is None else box
    fx, fy, fz = f[:, None, None], f[None, :, None], f[None, None, : r // 2 + 1].abs()
    u2 = (fx / lens[0]) ** 2 + (fy / lens[1]) ** 2 + (fz / lens[2]) ** 2
    u2[0, 0, 0] = 1.0
    h = torch.exp(-2.0 * sigma ** 2 * (fx ** 2 + fy ** 2 + fz ** 2) / r ** 2) / (-2.0 * math.pi * u2)
    h[0, 0, 0] = 0.0
    del u2
    acc = None
    for a, fa in enumerate((fx, fy, fz)):
        v = torch.zeros(r ** 3, device=DEV, dtype=torch.float64)
        for j, w in st:
            v = v.index_add(0, j, w * n[:, a])
        u = torch.where(fa.abs() == r // 2, torch.zeros_like(fa), fa) / lens[a]
        term = torch.fft.rfftn(v.reshape(r, r, r)) * (u * h)
        acc = term if acc is None else acc + term
    y = torch.fft.irfftn(1j * acc, s=(r, r, r))
    flat = y.reshape(-1)
    mu = sum((w * flat[j]).sum() for j, w in st) / p.shape[0]
    return 0.5 / (flat[0] - mu).abs() * (y - mu)


def _layer64(p, n, r, sigma, dchi, box=None):
    p, n = p.double().requires_grad_(True), n.double().requires_grad_(True)
    chi = _solve64(p, n, r, sigma, box)
    d = dchi(chi.detach()) if callable(dchi) else dchi.double()
    dp, dn = torch.autograd.grad(chi, (p, n), d)
    return chi.detach(), d, dp, dn


_KUHN = ((1, 3), (1, 5), (2, 3), (2, 6), (4, 5), (4, 6))  # with corners 0 and 7: the cube's six tetrahedra


def _mesh64(chi):
    """(corners T x 3 x 3, unit normals) of the level set 0 of the linear interpolant in each tetrahedron."""
    r = chi.shape[0]
    f = torch.stack([torch.roll(chi, (-(c & 1), -((c >> 1) & 1), -((c >> 2) & 1)), (0, 1, 2)).reshape(-1)
                     for c in range(8)], 1)
    neg = f < 0
    cell = (neg.any(1) & ~neg.all(1)).nonzero().reshape(-1)
    f, neg = f[cell], neg[cell]
    base = torch.stack([cell // (r * r), (cell // r) % r, cell % r], 1).double()
    off = torch.tensor([[c & 1, (c >> 1) & 1, (c >> 2) & 1] for c in range(8)], device=chi.device).double()
    tri, up = [], []
    for mid in _KUHN:
        q = (0,) + mid + (7,)
        for m in range(1, 15):
            ins = [a for a in range(4) if (m >> a) & 1]
            outs = [a for a in range(4) if not (m >> a) & 1]
            sel = torch.ones(cell.numel(), dtype=torch.bool, device=chi.device)
            for a in range(4):
                sel &= neg[:, q[a]] == bool((m >> a) & 1)
            fs, bs = f[sel], base[sel]

            def cut(a, b):
                a, b = min(a, b), max(a, b)
                t = (fs[:, q[a]] / (fs[:, q[a]] - fs[:, q[b]]))[:, None]
                return (bs + off[q[a]] + t * (off[q[b]] - off[q[a]])) / r

            d = off[[q[a] for a in outs]].mean(0) - off[[q[a] for a in ins]].mean(0)
            if len(ins) == 2:
                v = [cut(ins[0], outs[0]), cut(ins[0], outs[1]), cut(ins[1], outs[1]), cut(ins[1], outs[0])]
                parts = [(v[0], v[1], v[2]), (v[0], v[2], v[3])]
            else:
                o, rest = (ins[0], outs) if len(ins) == 1 else (outs[0], ins)
                parts = [tuple(cut(o, b) for b in rest)]
            for t in parts:
                tri.append(torch.stack(t, 1))
                up.append(d.expand(tri[-1].shape[0], 3))
    tri, up = torch.cat(tri), torch.cat(up)
    n = torch.linalg.cross(tri[:, 1] - tri[:, 0], tri[:, 2] - tri[:, 0])
    n = torch.where((n * up).sum(1, keepdim=True) < 0, -n, n)
    ln = n.norm(dim=1, keepdim=True)
    return tri, torch.where(ln > 0, n / ln.clamp_min(1e-300), torch.zeros_like(n))


def _splat64(q, v, r):
    g = torch.zeros(r ** 3, device=DEV, dtype=torch.float64)
    for j, w in _corners(q.double(), r):
        g.index_add_(0, j, w * v)
    return g.reshape(r, r, r)


def _nearest64(a, b):
    return torch.cat([((x[:, None, :] - b[None]) ** 2).sum(-1).argmin(1) for x in a.split(512)])


def _u01_64(seed, i):
    """SplitMix64's finaliser of a counter, as 53-bit uniforms (int64 arithmetic wraps)."""
    wrap = lambda v: v - (1 << 64) if v >= 1 << 63 else v  # noqa: E731
    shr = lambda z, k: (z >> k) & ((1 << (64 - k)) - 1)  # noqa: E731
    z = wrap(seed & (2 ** 64 - 1)) + wrap(0x9E3779B97F4A7C15) * (i + 1)
    z = (z ^ shr(z, 30)) * wrap(0xBF58476D1CE4E5B9)
    z = (z ^ shr(z, 27)) * wrap(0x94D049BB133111EB)
    return shr(z ^ shr(z, 31), 11).double() / 2.0 ** 53


def exact(case, seed):
    op = case["op"]
    x = _inputs(case, seed)
    if op in ("layer", "host"):
        chi, _, dp, dn = _layer64(x["p"], x["n"], case["r"], case["sigma"], x["dchi"], _box(case))
        return dict(chi=chi, dpoints=dp, dnormals=dn)
    if op == "forward":
        with torch.no_grad():
            return dict(chi=_solve64(x["p"].double(), x["n"].double(), case["r"], case["sigma"]))
    if op == "train":
        out = []
        for i in x:
            grad = lambda c, t=i["target"]: 2.0 / c.numel() * (c - t.double())  # noqa: E731
            chi, d, dp, dn = _layer64(i["p"], i["n"], i["r"], case["sigma"], grad)
            out.append(dict(chi=chi, dchi=d, dpoints=dp, dnormals=dn))
        return out
    if op == "lookup":
        flat = x["chi"].double().reshape(-1)
        v = sum(w * flat[j] for j, w in _corners(x["q"].double(), case["r"]))
        return dict(values=v, dchi=_splat64(x["q"], x["w"].double(), case["r"]))
    if op == "chamfer":
        a, b = x["a"].double(), x["b"].double()
        i, j = _nearest64(a, b), _nearest64(b, a)
        loss = ((a - b[i]) ** 2).sum(1).mean() + ((b - a[j]) ** 2).sum(1).mean()
        g = 2.0 / a.shape[0] * (a - b[i])
        g.index_add_(0, j, 2.0 / b.shape[0] * (a[j] - b))
        return dict(loss=loss, da=g)
    if op == "mesh":
        tri, n = _mesh64(x["chi"].double())
        p = tri.mean(1)
        return dict(points=p.shape[0], dchi=_splat64(p, -((p - x["centre"].double()) * n).sum(1), case["r"]))
    t, m = x["tris"].double(), case["m"]
    area = 0.5 * torch.linalg.cross(t[:, 1] - t[:, 0], t[:, 2] - t[:, 0]).norm(dim=1)
    cum = torch.cumsum(area, 0)
    i = torch.arange(m, device=DEV)
    k = torch.searchsorted(cum, _u01_64(seed, 3 * i) * cum[-1], right=True).clamp_max(t.shape[0] - 1)
    u, v = _u01_64(seed, 3 * i + 1), _u01_64(seed, 3 * i + 2)
    flip = u + v > 1.0
    u, v = torch.where(flip, 1.0 - u, u)[:, None], torch.where(flip, 1.0 - v, v)[:, None]
    c = t[k]
    return dict(points=c[:, 0] + u * (c[:, 1] - c[:, 0]) + v * (c[:, 2] - c[:, 0]), normals=x["nrm"].double()[k])
