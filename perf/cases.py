"""The calls whose speed matters: the work a program has this library do.

A program applies the element operator of one mesh many times (a handle, or
the plain call on its arrays), in fp64 or in a reduced storage type, with or
without the Helmholtz mass term; it solves the Poisson problem with it; it
applies many uneven meshes at once; and it trains the learned preconditioner.
Each kind of case below is one of these, through the package's public entry
points.  Sizes: meshes of 128 to 32768 elements at orders lx 3 to 12 (the
paper's sweep is lx 3 to 8), boxes of any shape.

Inputs are drawn from the seed: vertices of the unit box moved by up to 0.1 h,
u uniform in [-1, 1], the coefficient h1 either 1 or the smooth sum of eight
Fourier modes in [0.5, 2].  The geometric factors are the closed form for
trilinear elements, evaluated on the GPU in fp64.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

import paper_2506_20994_gb300 as ax
from paper_2506_20994_gb300 import synth

GKEYS = ("g11", "g22", "g33", "g12", "g13", "g23")
F64, F32, B16 = torch.float64, torch.float32, torch.bfloat16
MAX_POINTS = 32768 * 512


def listed():
    return [
        # the smallest plain workload: 8^3 elements, constant coefficient, one
        # launch that does not fill the chip
        dict(name="apply_8_lx8", kind="apply", nx=8, ny=8, nz=8, lx=8, h1="one", h2=False),
        # the headline: 32^3 elements at lx 8 through the operator handle
        dict(name="apply_32_lx8", kind="apply", nx=32, ny=32, nz=32, lx=8, h1="var", h2=False),
        # an odd order on an odd element count, as in an order sweep
        dict(name="apply_17_lx7", kind="apply", nx=17, ny=17, nz=17, lx=7, h1="var", h2=False),
        # the Helmholtz operator of an implicit time step, high order
        dict(name="apply_16_lx10_h2", kind="apply", nx=16, ny=16, nz=16, lx=10, h1="var", h2=True),
        # the plain call on the caller's fp64 arrays, low odd order, a box that is not a cube
        dict(name="helm_24x20x28_lx5", kind="helm", nx=24, ny=20, nz=28, lx=5, h1="var"),
        # fp32 storage, the mixed-precision mesh
        dict(name="helm32_32_lx8", kind="helm32", nx=32, ny=32, nz=32, lx=8, h1="var"),
        # bf16 storage of u, h1 and G, the same mesh
        dict(name="helm16_32_lx8", kind="helm16", nx=32, ny=32, nz=32, lx=8, h1="var"),
        # geometry not stored: formed from the corner vertices, fp32
        dict(name="tri32_25_lx6", kind="tri32", nx=25, ny=25, nz=25, lx=6, h1="var"),
        # 64 uneven meshes of mixed order in one launch (replayed as a graph)
        dict(name="batch64_64", kind="batch", dtype="f64", count=64, emin=64, emax=8192,
             meshes=0),
        # fp64 Jacobi-CG to 1e-8 on 16^3 elements: many small launches
        dict(name="cg_16_lx8", kind="solve", method="cg", nx=16, ny=16, nz=16, lx=8, h1="one",
             tol=1e-8, check=8),
        # the learned preconditioner inside fp32 refinement, variable coefficient
        dict(name="learned_16_lx8", kind="solve", method="mpfcg", nx=16, ny=16, nz=16, lx=8,
             h1="var", tol=1e-10, check=8),
        # training the learned preconditioner on an 8^3 mesh, 20 residual/error pairs
        dict(name="train_8_lx8", kind="train", nx=8, ny=8, nz=8, lx=8, n_hid=48, pairs=20,
             epochs=1),
    ]


def _dims(rng, elements):
    """Box dimensions of about this many elements, not always a cube."""
    s = elements ** (1.0 / 3.0)
    d = [max(1, round(s * math.exp(rng.uniform(-0.25, 0.25)))) for _ in range(2)]
    d.append(max(1, int(elements / (d[0] * d[1]))))
    rng.shuffle(d)
    return dict(zip(("nx", "ny", "nz"), d))


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(("apply", "apply", "apply", "helm", "helm", "helm32", "helm16", "tri32",
                       "batch", "solve", "solve", "train"))
    if kind == "batch":
        return dict(kind=kind, dtype=rng.choice(("f64", "f32")), count=rng.randint(6, 64), emin=64,
                    emax=int(_log(rng, 512, 8192)), meshes=rng.randint(1, 10 ** 6))
    if kind == "train":
        lx = rng.choice((5, 6, 7, 8))
        return dict(kind=kind, **_dims(rng, _log(rng, 128, 1000)), lx=lx, n_hid=rng.choice((16, 32, 48)),
                    pairs=rng.randint(6, 20), epochs=1)
    if kind == "solve":
        method = rng.choice(("cg", "cg", "mpcg32", "mpcg16", "mpfcg"))
        lx = rng.choice((5, 6, 7, 8, 10) if method != "mpfcg" else (6, 8))
        most = min(4096, 4096 * 512 // lx ** 3)
        return dict(kind=kind, method=method, **_dims(rng, _log(rng, 256, most)), lx=lx,
                    h1=rng.choice(("one", "var")), tol=1e-8 if method == "cg" else 1e-10,
                    check=rng.choice((1, 8)))
    lx = rng.choice((3, 4, 5, 6, 7, 8, 8, 10, 12))
    c = dict(kind=kind, **_dims(rng, _log(rng, 128, min(32768, MAX_POINTS // lx ** 3))), lx=lx,
             h1=rng.choice(("one", "var")))
    if kind == "apply":
        c["h2"] = rng.random() < 0.25
    return c


# ------------------------------------------------------------------ the mesh
@functools.lru_cache(maxsize=None)
def _gll(lx):
    """GLL nodes, weights and derivative matrix D[i, l] = l_l'(x_i), fp64."""
    P = np.polynomial.legendre.Legendre.basis(lx - 1)
    x = np.concatenate([[-1.0], np.sort(P.deriv().roots().real), [1.0]])
    x = 0.5 * (x - x[::-1])
    N, p = lx - 1, P(x)
    w = 2.0 / (N * (N + 1) * p ** 2)
    D = np.zeros((lx, lx))
    for i in range(lx):
        for l in range(lx):
            if i != l:
                D[i, l] = p[i] / (p[l] * (x[i] - x[l]))
    D[0, 0], D[N, N] = -N * (N + 1) / 4.0, N * (N + 1) / 4.0
    return x, w, 0.5 * (D - D[::-1, ::-1])


def _cuda(a, dtype=F64):
    return torch.as_tensor(np.ascontiguousarray(a), device="cuda").to(dtype)


def _corners(vertices):
    """(E, 2, 2, 2, 3) corners [e][c][b][a] of the box's elements, x fastest."""
    v = _cuda(vertices)
    parts = [v[c:v.shape[0] - 1 + c, b:v.shape[1] - 1 + b, a:v.shape[2] - 1 + a].reshape(-1, 3)
             for c in (0, 1) for b in (0, 1) for a in (0, 1)]
    return torch.stack(parts, 1).reshape(-1, 2, 2, 2, 3).contiguous()


def _geometry(corners, lx):
    """(xyz, G as a dict, mass) at the GLL points of trilinear elements."""
    x, w, _ = (_cuda(a) for a in _gll(lx))
    L = torch.stack([(1 - x) / 2, (1 + x) / 2])  # [2][lx]
    dL = torch.stack([-0.5 * torch.ones_like(x), 0.5 * torch.ones_like(x)])

    def at(lk, lj, li):
        return torch.einsum("ecbad,ck,bj,ai->dekji", corners, lk, lj, li)

    xyz = at(L, L, L).contiguous()
    J = [at(L, L, dL), at(L, dL, L), at(dL, L, L)]  # d(x, y, z)/d(r, s, t)

    def cross(a, b):
        return torch.stack([a[1] * b[2] - a[2] * b[1], a[2] * b[0] - a[0] * b[2],
                            a[0] * b[1] - a[1] * b[0]])

    adj = [cross(J[1], J[2]), cross(J[2], J[0]), cross(J[0], J[1])]  # det * grad(r, s, t)
    det = (J[0] * adj[0]).sum(0)
    www = torch.einsum("k,j,i->kji", w, w, w)
    f = www / det
    pairs = dict(g11=(0, 0), g22=(1, 1), g33=(2, 2), g12=(0, 1), g13=(0, 2), g23=(1, 2))
    G = {k: (f * (adj[a] * adj[b]).sum(0)).contiguous() for k, (a, b) in pairs.items()}
    return xyz, G, (det * www).contiguous()


def _h1(which, xyz, seed):
    """The coefficient at the nodes: 1, or eight Fourier modes scaled into [0.5, 2]."""
    if which == "one":
        return torch.ones_like(xyz[0])
    a, k, phi = synth.fourier_modes(seed)
    f = torch.zeros_like(xyz[0])
    for m in range(len(a)):
        f += float(a[m]) * torch.sin(float(k[m, 0]) * xyz[0] + float(k[m, 1]) * xyz[1]
                                     + float(k[m, 2]) * xyz[2] + float(phi[m]))
    lo, hi = f.min(), f.max()
    return (0.5 + 1.5 * (f - lo) / (hi - lo)).contiguous()


def _uniform(shape, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return torch.rand(shape, generator=g, device="cuda", dtype=F64) * 2 - 1


def _fields(nx, ny, nz, lx, which, seed):
    """One mesh's operands in fp64: u, dx, dxt, h1, G, and its corners and mass."""
    corners = _corners(synth.box_vertices(nx, ny, nz, seed=seed))
    xyz, G, mass = _geometry(corners, lx)
    D = _gll(lx)[2]
    return dict(G, u=_uniform(xyz[0].shape, seed + 1), h1=_h1(which, xyz, seed), dx=_cuda(D.T),
                dxt=_cuda(D), corners=corners, mass=mass)


def _mesh(c, seed):
    return _fields(c["nx"], c["ny"], c["nz"], c["lx"], c["h1"], seed)


def _args(f, dtype=F64, d_dtype=F64):
    return ([f["u"].to(dtype), f["dx"].to(d_dtype), f["dxt"].to(d_dtype), f["h1"].to(dtype)]
            + [f[k].to(dtype) for k in GKEYS])


def _specs(c):
    return synth.batch_meshes(c["meshes"], c["count"], c["emin"], c["emax"])


# --------------------------------------------------------------- the programs
@functools.lru_cache(maxsize=None)
def _weights(lx, n_hid):
    """Symmetric-form weights as training leaves them: in the space scaled by
    the root of the Jacobi diagonal, the n_hid softest modes of a cube
    element, each amplified by the inverse of its stiffness."""
    _, w, D = _gll(lx)
    K, M, N = D.T @ np.diag(w) @ D, np.diag(w), lx - 1
    A = (np.kron(np.kron(M, M), K) + np.kron(np.kron(M, K), M) + np.kron(np.kron(K, M), M))
    i = np.arange(lx ** 3)
    faces = sum(((q % N) == 0).astype(int) for q in (i % lx, i // lx % lx, i // lx ** 2))
    s = 1.0 / np.sqrt(np.diag(A) * 2.0 ** faces)  # face points carry both elements' diagonals
    lam, V = np.linalg.eigh(s[:, None] * A * s[None, :])
    W = V[:, :n_hid] * np.sqrt(0.1 / (np.maximum(lam[:n_hid], 0.0) + lam[1]))
    return np.concatenate([W.ravel(), np.zeros(n_hid), W.T.ravel(), np.zeros(lx ** 3)]).astype(np.float32)


def _poisson(c, seed, h1):
    v = synth.box_vertices(c["nx"], c["ny"], c["nz"], seed=seed)
    return ax.Poisson(v, c["lx"], h1=None if h1 == "one" else ax.fourier_coefficient(seed))


def prepare(case, seed):
    c, kind = case, case["kind"]
    if kind == "apply":
        f = _mesh(c, seed)
        op = ax.Operator(c["lx"], f["dx"], f["dxt"], f["h1"], *[f[k] for k in GKEYS])
        if c["h2"]:  # the mass term of a time step, 1/dt = 100
            f["h2"] = torch.full_like(f["u"], 100.0)
            op.set_h2(f["h2"], f["mass"])
        return dict(kind=kind, op=op, u=f["u"], w=torch.empty_like(f["u"]))
    if kind in ("helm", "helm32", "helm16"):
        dt, dd = {"helm": (F64, F64), "helm32": (F32, F32), "helm16": (B16, F32)}[kind]
        f = _mesh(c, seed)
        w = torch.empty(f["u"].shape, dtype=dd, device="cuda")
        return dict(kind=kind, args=[w] + _args(f, dt, dd) + [c["lx"]])
    if kind == "tri32":
        f = _mesh(c, seed)
        u = f["u"].to(F32)
        x, wq, _ = (_cuda(a) for a in _gll(c["lx"]))
        h1 = None if c["h1"] == "one" else f["h1"].to(F32)
        return dict(kind=kind, args=[torch.empty_like(u), u, f["dx"].to(F32), f["dxt"].to(F32), h1,
                                     f["corners"].reshape(-1), x, wq, c["lx"]])
    if kind == "batch":
        dt = F64 if c["dtype"] == "f64" else F32
        meshes = []
        for q, (nx, ny, nz, lx) in enumerate(_specs(c)):
            f = _fields(nx, ny, nz, lx, "var", 100 * seed + q)
            m = {k: f[k].to(dt) for k in ("u", "h1", "dx", "dxt") + GKEYS}
            m["w"], m["lx"] = torch.empty_like(m["u"]), lx
            meshes.append(m)
        B = ax.Batch(meshes, dtype=ax.AX_BATCH_F64 if dt == F64 else ax.AX_BATCH_F32)
        return dict(kind=kind, batch=B, w=[m["w"] for m in meshes])
    if kind == "solve":
        P = _poisson(c, seed, c["h1"])
        P.set_check_every(c["check"])
        s = dict(kind=kind, P=P, b=P.rhs(synth.poisson_source), method=c["method"], tol=c["tol"])
        if c["method"] == "mpfcg":
            s["M"] = ax.Mlp(c["lx"] ** 3, 48, arch=ax.AX_MLP_SYM, params=_weights(c["lx"], 48))
        return s
    if kind == "train":
        P = _poisson(c, seed, "var")
        R, E = _pairs(c, seed)
        n_in = c["lx"] ** 3
        M = ax.Mlp(n_in, c["n_hid"], arch=ax.AX_MLP_SYM,
                   params=ax.mlp_init_params(n_in, c["n_hid"], seed=seed, arch=ax.AX_MLP_SYM))
        return dict(kind=kind, P=P, M=M, R=R, E=E, epochs=c["epochs"])
    raise ValueError(kind)


def run(s):
    kind = s["kind"]
    if kind == "apply":
        s["op"].apply(s["w"], s["u"])
        return s["w"]
    if kind == "helm":
        ax.ax_helm(*s["args"])
        return s["args"][0]
    if kind == "helm32":
        ax.ax_helm_f32(*s["args"])
        return s["args"][0]
    if kind == "helm16":
        ax.ax_helm_bf16(*s["args"])
        return s["args"][0]
    if kind == "tri32":
        ax.ax_helm_trilinear_f32(*s["args"])
        return s["args"][0]
    if kind == "batch":
        s["batch"].launch(graph=True)
        return s["w"]
    if kind == "solve":
        P, b, m = s["P"], s["b"], s["method"]
        if m == "cg":
            return P.cg(b, tol=s["tol"])[0]
        if m == "mpcg32":
            return P.mpcg(b, mode=ax.AX_PREC_F32, tol=s["tol"], inner_tol=1e-4)[0]
        if m == "mpcg16":
            return P.mpcg(b, mode=ax.AX_PREC_BF16, tol=s["tol"], inner_tol=1e-2)[0]
        return P.mpfcg(b, s["M"], tol=s["tol"], inner_tol=1e-4)[0]
    loss = ax.train_energy(s["P"], s["M"], s["R"], s["E"], epochs=s["epochs"], lr=2e-3)
    return dict(loss=loss, params=s["M"].get_params())


def _flops(points, lx):
    return points * (12 * lx + 18)


def work(case):
    """Bytes: u, h1, the six factors and w, once each, in their storage types
    (a solve: per iteration, with its vectors; iterations estimated, they
    grow with the elements per side and with lx^1.5)."""
    c, kind = case, case["kind"]
    if kind == "batch":
        size = 72 if c["dtype"] == "f64" else 36
        pts = [(nx * ny * nz * lx ** 3, lx) for nx, ny, nz, lx in _specs(c)]
        return dict(bytes=size * sum(p for p, _ in pts), flops=sum(_flops(p, lx) for p, lx in pts))
    lx, nel = c["lx"], c["nx"] * c["ny"] * c["nz"]
    n = nel * lx ** 3
    if kind == "solve":
        its = 1080 * nel ** (1 / 3) / 32 * (lx / 8) ** 1.5
        # cg: u, h1, G, w and the vectors x, r, p (read and written) and minv
        per = {"cg": 120, "mpcg32": 60, "mpcg16": 46, "mpfcg": 80}[c["method"]]
        return dict(bytes=per * n * its, flops=(_flops(n, lx) + 20 * n) * its)
    if kind == "train":
        steps = c["pairs"] * c["epochs"]
        # r and e of each pair, the operator's data, minv; the network's three products
        return dict(bytes=steps * n * (72 + 24),
                    flops=steps * (8 * nel * lx ** 3 * c["n_hid"] + _flops(n, lx)))
    if kind == "tri32":
        return dict(bytes=n * (8 if c["h1"] == "one" else 12) + 192 * nel, flops=_flops(n, lx) + 60 * n)
    size = {"apply": 72 + (8 if c.get("h2") else 0), "helm": 72, "helm32": 36, "helm16": 20}[kind]
    return dict(bytes=size * n, flops=_flops(n, lx))


# ------------------------------------------------------------ 64-bit answers
def _apply64(u, D, h1, G):
    u, h1, D = u.to(F64), h1.to(F64), D.to(F64)
    g = {k: G[k].to(F64) for k in GKEYS}
    ur = torch.einsum("il,ekjl->ekji", D, u)
    us = torch.einsum("jl,ekli->ekji", D, u)
    ut = torch.einsum("kl,elji->ekji", D, u)
    wr = h1 * (g["g11"] * ur + g["g12"] * us + g["g13"] * ut)
    ws = h1 * (g["g12"] * ur + g["g22"] * us + g["g23"] * ut)
    wt = h1 * (g["g13"] * ur + g["g23"] * us + g["g33"] * ut)
    return (torch.einsum("li,ekjl->ekji", D, wr) + torch.einsum("lj,ekli->ekji", D, ws)
            + torch.einsum("lk,elji->ekji", D, wt))


class _Problem64:
    """The assembled, masked problem in plain fp64 torch."""

    def __init__(self, c, seed, which):
        lx, d = c["lx"], (c["nx"], c["ny"], c["nz"])
        corners = _corners(synth.box_vertices(*d, seed=seed))
        self.xyz, self.G, self.mass = _geometry(corners, lx)
        self.h1, self.D = _h1(which, self.xyz, seed), _cuda(_gll(lx)[2])
        i = np.arange(lx)
        n = [m * (lx - 1) + 1 for m in d]
        gx, gy, gz = (np.arange(m)[:, None] * (lx - 1) + i for m in d)
        shape = (d[2], d[1], d[0], lx, lx, lx)
        gid = ((gz[:, None, None, :, None, None] * n[1] + gy[None, :, None, None, :, None]) * n[0]
               + gx[None, None, :, None, None, :])
        self.gid = _cuda(np.broadcast_to(gid, shape).reshape(-1), torch.int64)
        self.ng = n[0] * n[1] * n[2]
        edge = np.zeros(n[::-1], bool)
        for a in range(3):
            np.moveaxis(edge, a, 0)[[0, -1]] = True
        self.mask = (~_cuda(edge, torch.bool).reshape(-1)[self.gid]).to(F64).reshape(self.h1.shape)
        self.c = 1.0 / self.gs(torch.ones_like(self.h1))
        D, h, g = self.D, self.h1, self.G
        D2, dd = D * D, torch.diagonal(D)
        diag = (torch.einsum("li,ekjl->ekji", D2, h * g["g11"])
                + torch.einsum("lj,ekli->ekji", D2, h * g["g22"])
                + torch.einsum("lk,elji->ekji", D2, h * g["g33"]))
        di, dj, dk = dd[None, None, None, :], dd[None, None, :, None], dd[None, :, None, None]
        diag = diag + 2 * h * (di * dj * g["g12"] + di * dk * g["g13"] + dj * dk * g["g23"])
        self.minv = self.mask / self.gs(diag)

    def gs(self, v):
        flat = torch.zeros(self.ng, dtype=F64, device="cuda").index_add_(0, self.gid, v.reshape(-1))
        return flat[self.gid].reshape(v.shape)

    def apply(self, u):
        return self.mask * self.gs(_apply64(u, self.D, self.h1, self.G))

    def dot(self, a, b):
        return (self.c * a * b).sum()

    def solve(self, tol=1e-12, maxit=6000):
        b = self.mask * self.gs(self.mass * 3 * math.pi ** 2 * torch.sin(math.pi * self.xyz).prod(0))
        x, r = torch.zeros_like(b), b
        z = self.minv * r
        p, rz = z, self.dot(r, z)
        stop = float(self.dot(b, b)) * tol ** 2
        for it in range(maxit):
            w = self.apply(p)
            alpha = rz / self.dot(p, w)
            x, r = x + alpha * p, r - alpha * w
            z = self.minv * r
            new = self.dot(r, z)
            p, rz = z + (new / rz) * p, new
            if it % 25 == 24 and float(self.dot(r, r)) <= stop:
                break
        return x


def _pairs(c, seed):
    """Residual/error pairs (R[k] = A E[k]): error fields as CG leaves them,
    smooth modes with a rougher part, zero on the boundary."""
    P = _Problem64(c, seed, "var")
    g, R, E = synth.rng(seed), [], []
    for _ in range(c["pairs"]):
        e = torch.zeros_like(P.h1)
        for m in range(6):
            k = g.integers(1, 6 + 4 * m, size=3)
            a = float(g.normal()) / (1 + m)
            e += a * (torch.sin(math.pi * _cuda(k.astype(float)).reshape(3, 1, 1, 1, 1) * P.xyz)).prod(0)
        e = e * P.mask
        E.append(e.reshape(-1))
        R.append(P.apply(e).reshape(-1))
    return torch.stack(R), torch.stack(E)


def _train64(c, seed):
    """One Adam step per pair on the relative energy error, fp64."""
    P = _Problem64(c, seed, "var")
    R, E = _pairs(c, seed)
    nel, N, Hd = P.h1.shape[0], c["lx"] ** 3, c["n_hid"]
    p0 = ax.mlp_init_params(N, Hd, seed=seed, arch=ax.AX_MLP_SYM)
    W = _cuda(p0[:N * Hd].reshape(N, Hd))
    m, v = torch.zeros_like(W), torch.zeros_like(W)
    sq = torch.sqrt(P.minv).reshape(nel, N)
    step, losses = 0, []
    b1, b2 = float(np.float32(0.9)), float(np.float32(0.999))
    lr, eps = float(np.float32(2e-3)), float(np.float32(1e-8))
    for _ in range(c["epochs"]):
        losses = []
        for r, e in zip(R, E):
            e = e.reshape(P.h1.shape)
            eA = P.dot(e, P.apply(e))
            X = sq * r.reshape(nel, N)
            H = X @ W
            d = e - P.minv * r.reshape(P.h1.shape) - P.gs((sq * (H @ W.T)).reshape(P.h1.shape))
            q = P.apply(d)
            losses.append(float(P.dot(d, q) / eA))
            dY = -2.0 / eA * sq * q.reshape(nel, N)
            grad = dY.T @ H + X.T @ (dY @ W)
            step += 1
            m, v = b1 * m + (1 - b1) * grad, b2 * v + (1 - b2) * grad * grad
            W = W - lr * (m / (1 - b1 ** step)) / (torch.sqrt(v / (1 - b2 ** step)) + eps)
    zero = torch.zeros(Hd, dtype=F64, device="cuda"), torch.zeros(N, dtype=F64, device="cuda")
    return dict(loss=torch.tensor(sum(losses) / len(losses), dtype=F64),
                params=torch.cat([W.reshape(-1), zero[0], W.T.reshape(-1), zero[1]]))


def exact(case, seed):
    c, kind = case, case["kind"]
    if kind == "batch":
        dt, out = (F64 if c["dtype"] == "f64" else F32), []
        for q, (nx, ny, nz, lx) in enumerate(_specs(c)):
            f = _fields(nx, ny, nz, lx, "var", 100 * seed + q)
            out.append(_apply64(f["u"].to(dt), f["dxt"].to(dt).reshape(lx, lx), f["h1"].to(dt),
                                {k: f[k].to(dt) for k in GKEYS}))
        return out
    if kind == "solve":
        return _Problem64(c, seed, c["h1"]).solve()
    if kind == "train":
        return _train64(c, seed)
    f = _mesh(c, seed)
    D = f["dxt"].reshape(c["lx"], c["lx"])
    if kind == "tri32":
        return _apply64(f["u"].to(F32), D.to(F32), f["h1"].to(F32), f)
    dt, dd = {"helm32": (F32, F32), "helm16": (B16, F32)}.get(kind, (F64, F64))
    w = _apply64(f["u"].to(dt), D.to(dd), f["h1"].to(dt), {k: f[k].to(dt) for k in GKEYS})
    if kind == "apply" and c["h2"]:
        w = w + 100.0 * f["mass"] * f["u"]
    return w
