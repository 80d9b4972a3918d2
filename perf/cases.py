"""What the speed of this framework is measured on: the calls that a program makes with it, over the sizes, block sides,
precisions and mesh kinds that its configurations, tests and benchmark use.

A case is a dict of plain values.  ``prepare`` makes what a program has in hand before the call (a context, a block set
on its mesh, source tensors on the GPU), ``run`` is one pass through the public entry points, ``exact`` the same values
in 64 bits in plain torch, ``work`` the bytes and operations that a pass cannot do without.

Kinds
-----
``solve``      new sources into a block set, solve, potentials out: the step of a time-stepping program
               (mesh "box": an unrefined lattice of blocks; "torus", "tori": refined around one or two Gaussian rings;
               "batch": several independent random sparse problems in one block set)
``vector``     the same for the three components of a field on one refined mesh
``gradient``   forward solve and adjoint solve through torch.autograd: potentials and gradients
``host``       sources from pinned host memory and potentials back into host memory
``static``     the exact convolution of a few blocks without device allocation
``refine``     one refinement step of a level on the GPU
``laplacian``  the 7-point consistency check of a field
"""
import functools
import math

import numpy as np
import torch

from paper_1911_10228_gb300 import autograd as A
from paper_1911_10228_gb300 import flgf as F
from paper_1911_10228_gb300 import inputs as I

DEV = torch.device("cuda" if torch.cuda.is_available() else "cpu")


def listed():
    return [
        # the smallest solve of the test configurations (4^3 blocks of 8^3 cells, one octree level): launches and latency
        dict(name="box_4x4x4_n8_fp32", kind="solve", mesh="box", b0=4, b1=4, b2=4, N=8, ni=6, prec="fp32", graph=True),
        # a latency-critical caller with its own memory pool: a handful of blocks, no allocation
        dict(name="static_27_n16_fp32", kind="static", b0=3, b1=3, b2=3, N=16, ni=6, prec="fp32"),
        # the ordinary large lattice of the benchmark: 256^3 cells
        dict(name="box_16x16x16_n16_fp32", kind="solve", mesh="box", b0=16, b1=16, b2=16, N=16, ni=6, prec="fp32",
             graph=True),
        # double precision on a ragged lattice of odd extents
        dict(name="box_11x9x13_n16_fp64", kind="solve", mesh="box", b0=11, b1=9, b2=13, N=16, ni=6, prec="fp64",
             graph=True),
        # the refined mesh of the benchmark: three levels around a ring, FP32 with compensated coarse levels
        dict(name="torus_l3_n16_fp32", kind="solve", mesh="torus", nbase=8, levels=3, N=16, ni=6, prec="fp32",
             graph=True),
        # the same ring in double precision with small blocks
        dict(name="torus_l3_n8_fp64", kind="solve", mesh="torus", nbase=8, levels=3, N=8, ni=6, prec="fp64",
             graph=True),
        # many independent sparse problems in one block set, the benchmark's headline form
        dict(name="batch_20_n16_fp32", kind="solve", mesh="batch", problems=20, first=0, N=16, ni=6, prec="fp32",
             graph=True),
        # optimisation through the solve: potentials and gradients of two linked rings
        dict(name="tori_l3_n16_fp32_grad", kind="gradient", mesh="tori", nbase=8, levels=3, N=16, ni=6, prec="fp32",
             graph=False),
        # the three streamfunction components of a vorticity field on one refined mesh
        dict(name="torus_l2_n16_fp32_vector", kind="vector", mesh="torus", nbase=8, levels=2, N=16, ni=6, prec="fp32",
             graph=True),
        # a program whose fields live in host memory; a low interpolation order
        dict(name="box_9x10x7_n16_fp32_host", kind="host", mesh="box", b0=9, b1=10, b2=7, N=16, ni=4, prec="fp32",
             graph=True),
        # re-meshing between time steps
        dict(name="refine_16x16x16_n16_fp32", kind="refine", b0=16, b1=16, b2=16, N=16, ni=6, prec="fp32"),
        # checking a computed field against its source
        dict(name="laplacian_16x16x16_n16_fp32", kind="laplacian", mesh="box", b0=16, b1=16, b2=16, N=16, ni=6,
             prec="fp32"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["solve"] * 7 + ["gradient", "vector", "host", "static", "refine", "laplacian"])
    N = rng.choice([8, 16, 16])
    prec = rng.choice(["fp32", "fp32", "fp64"])
    ni = rng.choice([4, 5, 6, 6, 6, 8]) if prec == "fp64" else rng.choice([4, 5, 6, 6])
    c = dict(kind=kind, N=N, ni=ni, prec=prec)
    if kind == "static":
        return dict(c, b0=rng.randint(1, 4), b1=rng.randint(1, 4), b2=rng.randint(1, 2))
    if kind in ("refine", "laplacian"):
        return dict(c, mesh="box", **{b: _log_int(rng, 2, 16) for b in ("b0", "b1", "b2")})
    c["graph"] = rng.random() < 0.7 if kind != "gradient" else False
    mesh = "box" if kind == "host" else rng.choice(["torus", "tori"]) if kind == "vector" else \
        rng.choice(["box", "torus", "tori"] if kind == "gradient" else ["box", "box", "box", "torus", "tori", "batch"])
    c["mesh"] = mesh
    if mesh == "box":
        top = 14 if prec == "fp32" else 11
        return dict(c, **{b: _log_int(rng, 2, top) for b in ("b0", "b1", "b2")})
    if mesh == "batch":
        return dict(c, problems=rng.randint(2, 16) if prec == "fp32" else 2, first=rng.randint(0, 500),
                    N=N if prec == "fp32" else 8)
    if kind == "vector" or prec == "fp64":
        c["N"] = 8 if prec == "fp64" else N
        return dict(c, nbase=rng.randint(4, 8), levels=2)
    return dict(c, nbase=rng.randint(4, 8), levels=rng.choice([2, 3]))


# ---------------------------------------------------------------------------------------------------------------------
# meshes, contexts and sources
# ---------------------------------------------------------------------------------------------------------------------

@functools.lru_cache(maxsize=None)
def _meshes(mesh, N, a, b, c):
    """[(levels of block coordinates, h0)] of the problems of a mesh."""
    if mesh == "box":
        return [([I.box_coords(a, b, c)], 1.0 / (N * max(a, b, c)))]
    if mesh == "batch":
        probs = [I.random_sparse_problem(s, N=8) for s in range(a, a + b)]  # the mesh does not depend on N
        return [(p.coords, p.h0 * 8 / N) for p in probs]
    p = (I.config_torus_128 if mesh == "torus" else I.config_linked_tori)(n_levels=b, N=N, nbase=a)
    return [(p.coords, p.h0)]


def _mesh_of(case):
    if case["kind"] in ("static", "refine") or case["mesh"] == "box":
        return _meshes("box", case["N"], case["b0"], case["b1"], case["b2"])
    if case["mesh"] == "batch":
        return _meshes("batch", case["N"], case["first"], case["problems"], 0)
    return _meshes(case["mesh"], case["N"], case["nbase"], case["levels"], 0)


@functools.lru_cache(maxsize=None)
def _context(N, ni, prec):
    """A program keeps one context per block side, order and precision."""
    return F.Context(N=N, n_interp=ni, precision=prec)


def _axes(coords, N, h):
    """Cell-centre coordinates along the three axes of every block, 3 x [nblk, N], float64 on the GPU."""
    c = torch.as_tensor(np.asarray(coords), device=DEV, dtype=torch.float64)
    i = torch.arange(N, device=DEV, dtype=torch.float64) + 0.5
    return [(c[:, a, None] * N + i) * h for a in range(3)]


def _blobs(gen, coords, N, h, lo, hi, n=6):
    """Sum of n random Gaussians in the box [lo, hi]^3-ish of the level, [nblk, N, N, N] float64: the smooth compact
    sources that the method is used for."""
    x = _axes(coords, N, h)
    r = torch.rand(n, 5, generator=gen, dtype=torch.float64)
    ext = max(b - a for a, b in zip(lo, hi))
    f = torch.zeros(len(coords), N, N, N, device=DEV, dtype=torch.float64)
    for q in r.tolist():
        s = ext * (0.02 + 0.06 * q[3])
        e = [torch.exp(-(x[a] - (lo[a] + (0.2 + 0.6 * q[a]) * (hi[a] - lo[a]))) ** 2 / (2 * s * s)) for a in range(3)]
        f += (2 * q[4] - 1) * e[0][:, :, None, None] * e[1][:, None, :, None] * e[2][:, None, None, :]
    return f


def _rings(gen, coords, N, h, mesh):
    """The ring (or two linked rings) of the refined meshes, with a random azimuthal modulation."""
    x = _axes(coords, N, h)
    x = [x[0][:, :, None, None], x[1][:, None, :, None], x[2][:, None, None, :]]
    r = torch.rand(6, generator=gen, dtype=torch.float64).tolist()

    def ring(y, R):
        d2 = (torch.sqrt(y[0] ** 2 + y[1] ** 2) - R) ** 2 + y[2] ** 2
        th = torch.atan2(y[1], y[0])
        return torch.exp(-d2 / (2 * 0.03 ** 2)) * (1 + 0.4 * torch.cos((1 + int(4 * r[0])) * th + 6.28 * r[1]) + 0.1 * r[2])

    if mesh == "torus":
        return ring([v - 0.5 for v in x], 0.25)
    y1 = [x[0] - 0.4, x[1] - 0.5, x[2] - 0.5]
    y2 = [x[0] - 0.6, x[1] - 0.5, x[2] - 0.5]
    return ring(y1, 0.2) + (0.5 + r[3]) * ring([y2[0], -y2[2], y2[1]], 0.2)


def _sources(case, seed, n_comp=1):
    """[component][problem][level] sources in the case's precision, on the GPU."""
    gen = torch.Generator().manual_seed(int(seed))
    dt = torch.float64 if case["prec"] == "fp64" else torch.float32
    N, out = case["N"], []
    for _ in range(n_comp):
        comp = []
        for coords, h0 in _mesh_of(case):
            lo = [float(v) * N * h0 for v in np.min(coords[0], axis=0)]
            hi = [float(v + 1) * N * h0 for v in np.max(coords[0], axis=0)]
            state = gen.get_state()
            levels = []
            for l, c in enumerate(coords):
                gen.set_state(state)  # one field, sampled on every level
                h = h0 / (1 << l)
                if case.get("mesh") in ("torus", "tori"):
                    f = _rings(gen, c, N, h, case["mesh"])
                else:
                    f = _blobs(gen, c, N, h, lo, hi)
                levels.append(f.to(dt))
            top = max(float(f.abs().max()) for f in levels)
            comp.append([torch.where(f.abs() < I.TRUNC * top, torch.zeros_like(f), f) for f in levels])
        out.append(comp)
    return out


def _level(case, seed):
    """A level to refine: one fixed shape of field (so every seed refines the same number of blocks) in a frame that
    moves with the seed: amplitude, origin and order of the blocks."""
    gen = torch.Generator().manual_seed(int(seed))
    f = _sources(case, 7)[0][0][0]
    r = torch.randint(-200, 201, (4,), generator=gen)
    perm = torch.randperm(f.shape[0], generator=gen).to(DEV)
    coords = torch.as_tensor(_mesh_of(case)[0][0][0] + 2 * r[:3].numpy(), dtype=torch.int32, device=DEV)
    return (f * 2.0 ** (int(r[3]) % 5 - 2))[perm].contiguous(), coords[perm].contiguous()


def _blocks(case):
    return sum(len(c) for coords, _ in _mesh_of(case) for c in coords)


# ---------------------------------------------------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------------------------------------------------

def prepare(case, seed):
    kind = case["kind"]
    ctx = _context(case["N"], case["ni"], case["prec"])
    mesh = _mesh_of(case)
    s = dict(kind=kind, ctx=ctx)
    if kind == "refine":
        f, coords = _level(case, seed)
        return dict(s, src=[((0, 0), f)], coords=coords)
    if kind == "vector":
        src = _sources(case, seed, 3)
        bs = F.BlockSet(ctx, [mesh[0][0]] * 3, [mesh[0][1]] * 3, vector=True)
        s["src"] = [((c, l), f) for c in range(3) for l, f in enumerate(src[c][0])]
    else:
        src = _sources(case, seed)[0]
        s["src"] = [((p, l), f) for p in range(len(mesh)) for l, f in enumerate(src[p])]
        if kind == "static":
            return dict(s, coords=mesh[0][0], h=mesh[0][1], out=torch.empty_like(src[0][0]))
        bs = F.BlockSet(ctx, [m[0] for m in mesh], [m[1] for m in mesh])
    s["bs"] = bs
    if case.get("graph"):
        bs.set_option(F.OPT_GRAPH, 1)
    if kind == "gradient":
        gen = torch.Generator().manual_seed(int(seed) + 1)
        s["src"] = [(k, f.requires_grad_()) for k, f in s["src"]]
        # dL/du of a loss on the potentials: a smooth weighting of them
        s["seed"] = [torch.rand(1, generator=gen).item() * f.detach() + 0.1 * f.detach().abs() for _, f in s["src"]]
    if kind == "host":
        f = s["src"][0][1]
        s["f_host"] = f.cpu().pin_memory()
        s["u_host"] = torch.empty_like(s["f_host"]).pin_memory()
    return s


def run(s):
    kind, ctx = s["kind"], s["ctx"]
    if kind == "static":
        return ctx.convolve_static(s["coords"], s["src"][0][1], h=s["h"], out=s["out"])
    if kind == "refine":
        return ctx.refine_level(s["src"][0][1], s["coords"], 1e-3)
    bs = s["bs"]
    if kind == "laplacian":
        return bs.laplacian(0, 0, s["src"][0][1])
    if kind == "host":
        bs.load_source(0, 0, s["f_host"])
        bs.solve()
        return bs.potential_host(0, 0, out=s["u_host"].numpy())
    if kind == "gradient":
        f = [x for _, x in s["src"]]
        u = A.solve(bs, f)
        return {"u": [x.detach() for x in u], "grad": list(torch.autograd.grad(u, f, s["seed"]))}
    for (p, l), f in s["src"]:
        bs.load_source(p, l, f)
    bs.solve()
    return [bs.potential(p, l) for (p, l), _ in s["src"]]


def _interactions(case):
    """(target, source) block pairs of one solve: the children of the 27 neighbours of a block's parent."""
    if case["kind"] in ("static",) or case["mesh"] == "box":
        per = 1
        for b in (case["b0"], case["b1"], case["b2"]):
            per *= sum(len(range(max(0, 2 * (t // 2) - 2), min(b, 2 * (t // 2) + 4))) for t in range(b))
        return per * 8 / 7
    return _blocks(case) * 100  # refined and sparse meshes: about half of the 216 candidates exist


def work(case):
    N, kind = case["N"], case["kind"]
    rs = 8 if case["prec"] == "fp64" else 4
    nb = _blocks(case)
    comps = 3 if kind == "vector" else 1
    dirs = 2 if kind == "gradient" else 1  # forward and adjoint
    cells = nb * N ** 3
    if kind == "refine":
        return {"bytes": cells * rs + nb * 13, "flops": cells}
    if kind == "laplacian":
        return {"bytes": 2 * cells * rs, "flops": 8 * cells}
    nf = 4 * N * N * (N + 1)
    fft = 2 * 2.5 * (2 * N) ** 3 * math.log2((2 * N) ** 3) / 2  # half of each transform's lines are zero or dropped
    flops = comps * dirs * (nb * 8 / 7 * fft + _interactions(case) * 8.0 * nf)
    return {"bytes": comps * dirs * 2 * cells * rs, "flops": flops}


# ---------------------------------------------------------------------------------------------------------------------
# the same values in 64 bits: the lattice Green's function by quadrature and the block method on dense boxes, in torch
# ---------------------------------------------------------------------------------------------------------------------

@functools.lru_cache(maxsize=1)
def _lgf_nodes():
    """Nodes and weights in t of int_0^T, T = 1e14: Gauss-Legendre panels in log t."""
    x, w = np.polynomial.legendre.leggauss(16)
    edges = np.linspace(math.log(1e-18), math.log(1e14), 141)
    u = np.concatenate([(b - a) / 2 * x + (a + b) / 2 for a, b in zip(edges[:-1], edges[1:])])
    wu = np.concatenate([(b - a) / 2 * w for a, b in zip(edges[:-1], edges[1:])])
    return np.exp(u), wu * np.exp(u)


@functools.lru_cache(maxsize=1)
def _bessel(n_max):
    """exp(-z) I_n(z) at z = 2 t, [n_max + 1, nodes] on the GPU: the integral over the angle by the trapezoid rule
    (spectrally accurate for periodic integrands), Hankel's expansion for large z."""
    t, _ = _lgf_nodes()
    z = torch.as_tensor(2 * t, device=DEV, dtype=torch.float64)
    n = torch.arange(n_max + 1, device=DEV, dtype=torch.float64)
    out = torch.zeros(n_max + 1, z.numel(), device=DEV, dtype=torch.float64)
    small = z < 2e5
    M = 8192
    th = torch.arange(M, device=DEV, dtype=torch.float64) * (2 * math.pi / M)
    cosn = torch.cos(n[:, None] * th[None])
    out[:, small] = cosn @ torch.exp(-2 * z[small][None] * torch.sin(th[:, None] / 2) ** 2) / M
    zl = z[~small]
    acc = torch.zeros(n_max + 1, zl.numel(), device=DEV, dtype=torch.float64)
    term = torch.ones_like(acc)
    for k in range(1, 30):
        acc += term
        term = term * -(4 * n[:, None] ** 2 - (2 * k - 1) ** 2) / (k * 8 * zl[None])
    out[:, ~small] = acc / torch.sqrt(2 * math.pi * zl)[None]
    return out


# The table radius and the asymptotic expansion beyond it are part of the method: G by quadrature for |n| <= 100, the
# expansion up to degree -7 for |n| <= 600, up to degree -5 beyond.
def _lgf(n):
    """Lattice Green's function at integer points n [..., 3] (float64 tensor)."""
    shape = n.shape[:-1]
    x = n.reshape(-1, 3).abs()
    r = torch.sqrt((x ** 2).sum(1))
    out = torch.zeros_like(r)
    near = r <= 100
    t, w = _lgf_nodes()
    B = _bessel(100)
    wt = torch.as_tensor(w, device=DEV, dtype=torch.float64)
    i = x[near].long().sort(dim=1).values
    key, inv = torch.unique(i[:, 0] * 10201 + i[:, 1] * 101 + i[:, 2], return_inverse=True)
    vals = torch.empty(key.numel(), device=DEV, dtype=torch.float64)
    for a in range(0, key.numel(), 20000):
        q = key[a:a + 20000]
        vals[a:a + 20000] = (B[q // 10201] * B[q // 101 % 101] * B[q % 101]) @ wt
    out[near] = -(vals[inv] + 2 * (4 * math.pi) ** -1.5 / math.sqrt(1e14))
    f, rf = x[~near], r[~near]
    s2, s4, s6 = (f ** 2).sum(1), (f ** 4).sum(1), (f ** 6).sum(1)
    # G = -1/(4 pi r) [1 + a1 + a2 + ...], the point expansion of the 7-point operator's inverse
    p1, p2, p3 = f[:, 0] ** 2, f[:, 1] ** 2, f[:, 2] ** 2
    A2 = -1 / (4 * math.pi * rf) - (s4 - 3 * (p1 * p2 + p1 * p3 + p2 * p3)) / (16 * math.pi * rf ** 7)
    e8 = p1 ** 4 + p2 ** 4 + p3 ** 4
    c62 = p1 ** 3 * (p2 + p3) + p2 ** 3 * (p1 + p3) + p3 ** 3 * (p1 + p2)
    c44 = p1 ** 2 * p2 ** 2 + p1 ** 2 * p3 ** 2 + p2 ** 2 * p3 ** 2
    c422 = p1 * p2 * p3 * (p1 + p2 + p3)
    A3 = A2 - (23 * e8 - 244 * c62 + 621 * c44 - 228 * c422) / (128 * math.pi * rf ** 13)
    out[~near] = torch.where(rf <= 600, A3, A2)
    return out.reshape(shape)


def _lagrange(N, ni):
    """[2 N, N]: values at the 2 N child nodes (j + 1/2) of two siblings from the parent's N nodes (2 p + 1)."""
    J = np.zeros((2 * N, N))
    for j in range(2 * N):
        x = j + 0.5
        if ni % 2 == 0:
            a = math.floor((x - 1) / 2) - (ni // 2 - 1)
        else:
            a = min(range(N), key=lambda p: (abs(2 * p + 1 - x), p)) - ni // 2
        a = min(max(a, 0), N - ni)
        for m in range(ni):
            J[j, a + m] = np.prod([(x - (2 * (a + q) + 1)) / (2.0 * (m - q)) for q in range(ni) if q != m])
    return torch.as_tensor(J, device=DEV)


def _dense_solve(f, b, N, ni, h):
    """The block method on a dense box of b0 x b1 x b2 blocks in 64 bits; f [nblk, N, N, N] float64."""
    J = _lagrange(N, ni).reshape(2, N, N)
    dims, fields = [tuple(b)], [f.reshape(*b, N, N, N)]
    while max(dims[-1]) > 4:  # a level is the last when its parents are neighbours of each other
        d = dims[-1]
        pd = tuple((v + 1) // 2 for v in d)
        pad = torch.zeros(*(2 * v for v in pd), N, N, N, device=DEV, dtype=torch.float64)
        pad[:d[0], :d[1], :d[2]] = fields[-1]
        pad = pad.reshape(pd[0], 2, pd[1], 2, pd[2], 2, N, N, N)
        y = torch.einsum("xaybzcijk,aip->xybzcpjk", pad, J)
        y = torch.einsum("xybzcpjk,bjq->xyzcpqk", y, J)
        fields.append(torch.einsum("xyzcpqk,ckr->xyzpqr", y, J))
        dims.append(pd)
    up = None
    for k in reversed(range(len(dims))):
        d, src = dims[k], fields[k]
        Fh = torch.fft.rfftn(src, s=(2 * N,) * 3, dim=(3, 4, 5))
        acc = torch.zeros_like(Fh)
        ax = torch.arange(2 * N, device=DEV, dtype=torch.float64)
        ax = torch.where(ax < N, ax, ax - 2 * N)
        for d0 in range(-3, 4):
            for d1 in range(-3, 4):
                for d2 in range(-3, 4):
                    dd = (d0, d1, d2)
                    if any(abs(v) >= n for v, n in zip(dd, d)) or (k > 0 and max(map(abs, dd)) <= 1):
                        continue
                    pts = torch.stack(torch.meshgrid(*[(N * v + ax) * float(1 << k) for v in dd], indexing="ij"), -1)
                    K = _lgf(pts)
                    K[N], K[:, N], K[:, :, N] = 0, 0, 0
                    Kh = torch.fft.rfftn(K)
                    # targets t of each parity whose source t - dd is a child of a neighbour of t's parent
                    for par in range(8):
                        a = (par >> 2, par >> 1 & 1, par & 1)
                        if any(not -1 <= (q - v) // 2 <= 1 for q, v in zip(a, dd)):
                            continue
                        t, s = [], []
                        for q, v, n in zip(a, dd, d):
                            lo = q
                            while lo - v < 0:
                                lo += 2
                            hi = min(n, n + v)
                            t.append(slice(lo, max(lo, hi), 2))
                            s.append(slice(lo - v, max(lo, hi) - v, 2))
                        acc[tuple(t)] += Kh * Fh[tuple(s)]
        u = torch.fft.irfftn(acc, s=(2 * N,) * 3, dim=(3, 4, 5))[..., :N, :N, :N] * (h * h)
        if up is not None:
            v = torch.einsum("xyzpqr,aip->xayziqr", up, J)
            v = torch.einsum("xayziqr,bjq->xaybzijr", v, J)
            v = torch.einsum("xaybzijr,ckr->xaybzcijk", v, J)
            u = u + v.reshape(*(2 * n for n in up.shape[:3]), N, N, N)[:d[0], :d[1], :d[2]]
        up = u
    return up.reshape(-1, N, N, N)


def exact(case, seed):
    kind = case["kind"]
    if kind == "refine":
        return None  # flags and block coordinates: whole numbers
    if kind not in ("static", "laplacian") and (case["mesh"] != "box" or kind == "gradient"):
        return None  # refined and sparse meshes: the whole method again, on thousands of blocks, takes far longer
    N, b = case["N"], (case["b0"], case["b1"], case["b2"])
    h = _mesh_of(case)[0][1]
    f = _sources(case, seed)[0][0][0].double()
    if kind == "laplacian":
        x = f.reshape(*b, N, N, N).permute(0, 3, 1, 4, 2, 5).reshape(*(n * N for n in b))
        lap = torch.zeros_like(x)
        c = x[1:-1, 1:-1, 1:-1]
        lap[1:-1, 1:-1, 1:-1] = (x[2:, 1:-1, 1:-1] + x[:-2, 1:-1, 1:-1] + x[1:-1, 2:, 1:-1] + x[1:-1, :-2, 1:-1]
                                 + x[1:-1, 1:-1, 2:] + x[1:-1, 1:-1, :-2] - 6 * c) / (h * h)
        return lap.reshape(b[0], N, b[1], N, b[2], N).permute(0, 2, 4, 1, 3, 5).reshape(-1, N, N, N)
    u = _dense_solve(f, b, N, case["ni"], h)
    return u.cpu().numpy() if kind == "host" else [u] if kind == "solve" else u
