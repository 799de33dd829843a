"""What a user of this framework has it do, as cases that can be timed.

Every case goes through the public entry points (`paper_2405_12484_gb300.sim`):
the projections alone, the local step, the global solve, whole frames in the
three storage precisions, a change of materials, an equilibrium step with its
adjoint, and the serving loop.  Meshes are the repository's two families: a
slab pinned along one edge and a thick cylindrical shell hung from its top
ring, with about 2,000 tets per domain as the serving requests have.
"""
from __future__ import annotations

import itertools
import math
import types
from functools import lru_cache

import numpy as np
import torch

from paper_2405_12484_gb300 import sim

DT = 1.0 / 150.0
DENSITY = 300.0
GRAVITY = (0.0, 0.0, -9.81)


def listed():
    return [
        # the projections of one small garment piece: the parity slab's 4,800 elements, launch-bound
        {"name": "project 4.8K", "kind": "project", "n": 4800},
        # the projections of a whole sweater: one matrix per element of the 390,000-tet shell
        {"name": "project 390K", "kind": "project", "n": 390000},
        # right-hand side of one PD iteration (local step and assembly) of the sweater-scale shell
        {"name": "local shell 390K", "kind": "local", "mesh": "shell", "nx": 325, "ny": 100, "nz": 2, "dx": 25, "dy": 8},
        # global solve of the parity slab (8 domains, one interface level): the smallest calls
        {"name": "solve slab 4.8K", "kind": "solve", "mesh": "slab", "nx": 20, "ny": 20, "nz": 2, "dx": 4, "dy": 2},
        # global solve of the sweater-scale shell (200 domains, two interface levels)
        {"name": "solve shell 390K", "kind": "solve", "mesh": "shell", "nx": 325, "ny": 100, "nz": 2, "dx": 25, "dy": 8},
        # one frame of a small piece at interactive rates
        {"name": "frame slab 4.8K", "kind": "frame", "mesh": "slab", "nx": 20, "ny": 20, "nz": 2, "dx": 4, "dy": 2,
         "n_iter": 10, "precision": "fp32", "correction": False},
        # one frame of a single garment panel, odd sizes, TF32 matrices (the middle of the accuracy options)
        {"name": "frame shell 53K tf32", "kind": "frame", "mesh": "shell", "nx": 121, "ny": 37, "nz": 2, "dx": 9, "dy": 3,
         "n_iter": 20, "precision": "tf32", "correction": True},
        # one frame of the sweater, the headline workload, FP32
        {"name": "frame shell 390K", "kind": "frame", "mesh": "shell", "nx": 325, "ny": 100, "nz": 2, "dx": 25, "dy": 8,
         "n_iter": 20, "precision": "fp32", "correction": False},
        # the same frame with BF16 matrices on the tensor cores in the correction form
        {"name": "frame shell 390K bf16", "kind": "frame", "mesh": "shell", "nx": 325, "ny": 100, "nz": 2, "dx": 25,
         "dy": 8, "n_iter": 20, "precision": "bf16", "correction": True},
        # one trial of a material fit: new materials, prefactorisation, first solve (differentiable slab, 50,000 tets)
        {"name": "refit slab 50K", "kind": "refit", "mesh": "slab5", "nx": 50, "ny": 50, "nz": 4, "dx": 5, "dy": 5},
        # forward and backward of one differentiable step on that slab: equilibrium, pose loss, adjoint, gradients
        {"name": "adjoint slab 50K", "kind": "adjoint", "mesh": "slab5", "nx": 50, "ny": 50, "nz": 4, "dx": 5, "dy": 5,
         "n_iter": 10, "n_newton": 3, "cg_iters": 30},
        # the serving loop: a handful of requests of mixed sizes from submission to their last frame
        {"name": "serve 6 requests", "kind": "serve", "requests": 6, "lo": 5000, "hi": 60000, "frames": 30, "n_iter": 20,
         "mix": 12},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_mesh(rng, lo, hi, families=("slab", "shell")):
    fam, n_t = rng.choice(families), _log(rng, lo, hi)
    per = 5 if fam == "slab5" else 6
    if fam == "shell":
        nz = rng.choice((1, 2, 2, 3))
        ny = max(2, round(math.sqrt(n_t / (per * nz * rng.uniform(2.5, 4.0)))))
    else:
        nz = rng.choice((1, 2, 2, 3, 4))
        ny = max(2, round(math.sqrt(n_t / (per * nz)) * rng.uniform(0.6, 1.6)))
    nx = max(3, round(n_t / (per * nz * ny)))
    n_dom = max(1, round(n_t / rng.uniform(1600, 2400)))
    dy = min(ny, max(1, round(math.sqrt(n_dom * ny / nx))))
    return {"mesh": fam, "nx": nx, "ny": ny, "nz": nz, "dx": min(nx, max(1, round(n_dom / dy))), "dy": dy}


def draw(rng):
    kind = rng.choice(("project", "local", "solve", "frame", "frame", "refit", "adjoint", "serve"))
    if kind == "project":
        return {"kind": kind, "n": _log(rng, 1000, 2000000)}
    if kind == "serve":
        return {"kind": kind, "requests": rng.randint(2, 6), "lo": 5000, "hi": _log(rng, 10000, 60000),
                "frames": rng.randint(10, 30), "n_iter": 20, "mix": rng.randrange(1 << 20)}
    if kind == "adjoint":
        return {"kind": kind, **_draw_mesh(rng, 1500, 50000, ("slab", "slab5")), "n_iter": 10, "n_newton": 3,
                "cg_iters": 30}
    if kind == "refit":
        return {"kind": kind, **_draw_mesh(rng, 600, 100000, ("slab", "slab5", "shell"))}
    case = {"kind": kind, **_draw_mesh(rng, 600, 380000)}
    if kind == "frame":
        precision = rng.choice(("fp32", "fp32", "tf32", "bf16"))
        case |= {"n_iter": rng.choice((10, 20)), "precision": precision, "correction": precision != "fp32"}
    return case


# ---- inputs ------------------------------------------------------------------

_PATHS = []     # the six tets of a cube: one monotone lattice path per axis order
for _p in itertools.permutations(range(3)):
    _c, _path = [0, 0, 0], [(0, 0, 0)]
    for _ax in _p:
        _c[_ax] += 1
        _path.append(tuple(_c))
    _PATHS.append(_path)
_EVEN = [(0, 0, 0), (1, 1, 0), (1, 0, 1), (0, 1, 1)]
_ODD = [(1, 0, 0), (0, 1, 0), (0, 0, 1), (1, 1, 1)]


def _five(center, apexes):
    return [center] + [[a] + [q for q in center if sum(abs(a[i] - q[i]) for i in range(3)) == 1] for a in apexes]


@lru_cache(maxsize=24)
def _geometry(fam, nx, ny, nz, dx, dy):
    """Rest positions, tets, domain labels and pins of one mesh (the same for every seed)."""
    I, J, K = (a.ravel() for a in np.meshgrid(np.arange(nx), np.arange(ny), np.arange(nz), indexing="ij"))
    if fam == "shell":      # nx around, ny along z, nz through the thickness
        th = 2.0 * np.pi * np.arange(nx) / nx
        z, r = 0.6 * np.arange(ny + 1) / ny, 0.295 + 0.01 * np.arange(nz + 1) / nz
        Z, T, R = np.meshgrid(z, th, r, indexing="ij")
        rest = np.stack([R * np.cos(T), R * np.sin(T), Z], -1).reshape(-1, 3)
        vid = lambda i, j, k: (j * nx + i % nx) * (nz + 1) + k     # noqa: E731
        pinned = np.isclose(rest[:, 2], 0.6)
    else:
        Z, Y, X = np.meshgrid(np.arange(nz + 1), np.arange(ny + 1), np.arange(nx + 1), indexing="ij")
        rest = 0.01 * np.stack([X, Y, Z], -1).reshape(-1, 3).astype(np.float64)
        vid = lambda i, j, k: (k * (ny + 1) + j) * (nx + 1) + i    # noqa: E731
        pinned = np.isclose(rest[:, 1], 0.01 * ny)
    if fam == "slab5":
        even, odd = np.asarray(_five(_EVEN, _ODD)), np.asarray(_five(_ODD, _EVEN))
        off = np.where(((I + J + K) % 2 == 0)[:, None, None, None], even[None], odd[None])
    else:
        off = np.broadcast_to(np.asarray(_PATHS)[None], (I.size, 6, 4, 3))
    tets = vid(I[:, None, None] + off[..., 0], J[:, None, None] + off[..., 1], K[:, None, None] + off[..., 2])
    dom = np.repeat(np.minimum(J * dy // ny, dy - 1) * dx + np.minimum(I * dx // nx, dx - 1), tets.shape[1])
    tets = tets.reshape(-1, 4)
    e = rest[tets[:, 1:]] - rest[tets[:, :1]]
    neg = np.linalg.det(e) < 0
    tets[neg, 2], tets[neg, 3] = tets[neg, 3], tets[neg, 2].copy()
    return rest, tets.astype(np.int32), dom.astype(np.int32), pinned.astype(np.uint8)


def _geo(case):
    return _geometry(*(case[k] for k in ("mesh", "nx", "ny", "nz", "dx", "dy")))


def _stiffness(case, n_t, rng):
    """Per-element stiffness (Pa): log-uniform on slabs, 2 cm cable bands on the shell; a float32 array."""
    if case["mesh"] != "shell":
        return np.exp(rng.uniform(math.log(1e3), math.log(1e5), n_t)).astype(np.float32)
    i = np.arange(n_t) // 6 // (case["ny"] * case["nz"])
    arc = 0.6 * np.pi * (i + 0.5) / case["nx"]
    return (np.where(np.floor(arc / 0.02) % 2 == 0, 1e5, 1e4) * (1.0 + 0.2 * rng.uniform(-1, 1, n_t))).astype(np.float32)


def _fields(rest, rng):
    """A garment in motion: positions (smooth waves of centimetre scale) and velocities (about 1.5 m/s), float32."""
    u = (rest - rest.min(0)) / np.maximum(np.ptp(rest, axis=0).max(), 1e-9)
    x, v = rest.copy(), np.zeros_like(rest)
    v[:] = rng.normal(size=3) * 0.3 + np.array([1.2, 0.0, 0.0])
    for _ in range(4):
        k, a, ph = rng.normal(size=3) * 3.0, rng.normal(size=3), rng.uniform(0, 2 * np.pi)
        w = np.sin(u @ k + ph)[:, None] * (a / np.linalg.norm(a))
        x += 0.015 * np.ptp(rest, axis=0).max() * rng.uniform(0.5, 1.0) * w
        v += 0.3 * w
    return x.astype(np.float32), v.astype(np.float32)


def _case_arrays(case, seed):
    """Everything of one case that depends on the seed, as host arrays."""
    rng = np.random.default_rng([seed, 7])
    if case["kind"] == "project":
        n = case["n"]
        # elements of a worn garment: any rotation, strains of some 10 %, a few strongly strained, a few inverted
        q = rng.normal(size=(n, 4, 1)).astype(np.float64)
        w, x, y, z = (q / np.linalg.norm(q, axis=1, keepdims=True)).transpose(1, 0, 2)[..., 0]
        R = np.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y),
                      2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x),
                      2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)], -1).reshape(n, 3, 3)
        size = rng.choice((0.01, 0.05, 0.12), p=(0.5, 0.4, 0.1), size=(n, 1, 1))
        F = R @ (np.eye(3) + size * rng.normal(size=(n, 3, 3)))
        flip = rng.uniform(size=n) < 0.002
        F[flip, :, 0] *= -0.3
        return {"F": F.astype(np.float32)}
    rest, tets, _, pinned = _geo(case)
    out = {"theta": _stiffness(case, len(tets), rng)}
    x, v = _fields(rest, rng)
    out |= {"x": x, "v": v, "y": (x + np.float32(DT) * v).astype(np.float32),
            "pins": (x + np.float32(DT) * v)[pinned != 0].astype(np.float32)}
    if case["kind"] in ("solve", "refit"):
        scale = DENSITY * 1e-6 / DT ** 2
        out["r"] = (scale * (x + 0.02 * rng.normal(size=x.shape))).astype(np.float32)
    if case["kind"] == "adjoint":
        x0 = rest.copy()       # one step from rest towards a seeded pose
        u = (rest - rest.min(0)) / np.ptp(rest, axis=0)
        a, b, c = rng.uniform(0.5, 1.5, 3)
        x0[:, 2] += -0.02 * a * (1 - u[:, 1]) ** 2 + 0.004 * b * np.sin(np.pi * u[:, 0])
        x0[:, 0] += 0.005 * c * (1 - u[:, 1]) ** 2
        out |= {"target": x0.astype(np.float32), "x": rest.astype(np.float32), "v": np.zeros_like(x),
                "pins": rest[pinned != 0].astype(np.float32)}
    return out


def _requests(case, seed):
    rng, sizes = np.random.default_rng([seed, 11]), np.random.default_rng(case["mix"])
    ws = []
    for n_t in np.exp(sizes.uniform(math.log(case["lo"]), math.log(case["hi"]), case["requests"])):
        n_dom = max(1, round(n_t / 2000))
        if sizes.uniform() < 0.5:
            n = max(2, round(math.sqrt(n_t / 12)))
            side = min(n, max(1, round(math.sqrt(n_dom))))
            m = {"mesh": "slab", "nx": n, "ny": n, "nz": 2, "dx": side, "dy": side}
        else:
            ny = max(2, round(math.sqrt(n_t / 39)))
            dy = min(ny, max(1, round(math.sqrt(n_dom / 3.125))))
            m = {"mesh": "shell", "nx": round(3.25 * ny), "ny": ny, "nz": 2, "dx": max(1, round(n_dom / dy)), "dy": dy}
        rest, tets, dom, pinned = _geo(m)
        th = _stiffness(m, len(tets), rng)
        ws.append(types.SimpleNamespace(rest=rest, tets=tets, tet_domain=dom, n_domains=m["dx"] * m["dy"], pinned=pinned,
                                        gamma_s=th, gamma_v=10 * th, density=DENSITY, dt=DT, gravity=GRAVITY))
    return ws


def prepare(case, seed):
    if case["kind"] == "serve":     # host data by its nature: requests are submitted as host arrays
        return {"case": case, "requests": _requests(case, seed),
                "server": sim.Server(16 << 30, max_slots=64, n_iter=case["n_iter"])}
    a = {k: torch.from_numpy(v).cuda() for k, v in _case_arrays(case, seed).items()}
    st = {"case": case, **a}
    if case["kind"] == "project":
        return st
    rest, tets, dom, pinned = _geo(case)
    m = st["mesh"] = sim.Mesh(rest, tets, pinned, dom, case["dx"] * case["dy"], DENSITY)
    m.set_materials(a["theta"], 10 * a["theta"])
    opts = {"precision": case["precision"], "correction": case["correction"]} if case["kind"] == "frame" else {}
    m.prefactor(DT, **opts)
    st["out"] = torch.empty((m.n_v, 3), device="cuda")
    if case["kind"] == "adjoint":
        st["adj"] = sim.Adjoint(m, case["cg_iters"])
        st["x64"], st["v64"] = a["x"].double(), a["v"].double()
        st["gs"], st["gv"] = torch.zeros(m.n_t, device="cuda"), torch.zeros(m.n_t, device="cuda")
    return st


# ---- one pass ----------------------------------------------------------------

def run(st):
    case, m = st["case"], st.get("mesh")
    kind = case["kind"]
    if kind == "project":
        R, V, s = sim.project(st["F"])
        return {"R": R, "V": V, "s": s}
    if kind == "local":
        return {"b": m.local_rhs(st["x"], st["y"])}
    if kind == "solve":
        return {"x": m.solve(st["r"])}
    if kind == "frame":
        m.set_state(st["x"], st["v"])
        m.step(st["pins"], GRAVITY, case["n_iter"])
        x, v = m.get_state()
        return {"x": x, "v": v}
    if kind == "refit":
        m.set_materials(st["theta"], 10 * st["theta"])
        m.prefactor(DT)
        return {"x": m.solve(st["r"])}
    if kind == "adjoint":
        adj = st["adj"]
        adj.set_state64(st["x64"], st["v64"])
        x = adj.equilibrium_step(st["pins"], GRAVITY, case["n_iter"], case["n_newton"], x_out=st["out"])
        loss, dl = adj.pose_misfit(x, st["target"])
        x64, _ = adj.get_state64()
        adj.reset()
        st["gs"].zero_()
        st["gv"].zero_()
        adj.step64(x64, dl, st["gs"], st["gv"])
        return {"loss": loss, "x": x64, "gs": st["gs"], "gv": st["gv"]}
    srv = st["server"]
    ids = [srv.submit(w, case["frames"], drive=(0.05, 1.0, 0)) for w in st["requests"]]
    srv.run()
    out = [srv.fetch(i)[0] for i in ids]
    for i in ids:
        sim.lib().pd_release(srv._h, i)
    return out


# ---- what a pass cannot do without --------------------------------------------

def _sizes(case):
    if case["kind"] == "project":
        return case["n"], 0
    per = {"slab5": 5}.get(case["mesh"], 6)
    around = case["nx"] if case["mesh"] == "shell" else case["nx"] + 1
    return per * case["nx"] * case["ny"] * case["nz"], around * (case["ny"] + 1) * (case["nz"] + 1)


LOCAL_FLOPS = 500     # per element: F, the two projections, four corner terms
ROW = 15              # entries of a matrix row (lattice meshes of tets)


def work(case):
    kind = case["kind"]
    if kind == "serve":
        total = {"bytes": 0.0, "flops": 0.0}
        n_t = case["requests"] * math.sqrt(case["lo"] * case["hi"])
        total["bytes"] = n_t * (16 + 8) + n_t / 4 * (24 + 12)
        total["flops"] = case["frames"] * case["n_iter"] * n_t * (LOCAL_FLOPS + 6 * ROW / 4)
        return total
    n_t, n_v = _sizes(case)
    if kind == "project":
        return {"bytes": 120.0 * n_t, "flops": float(LOCAL_FLOPS * n_t)}
    mesh = 64.0 * n_t                      # corner ids, rest operator and weights of every element
    matrix = 8.0 * ROW * n_v               # K by rows, which any factorisation is at least as large as
    if kind == "local":
        return {"bytes": mesh + 36.0 * n_v, "flops": float(LOCAL_FLOPS * n_t)}
    if kind == "solve":
        return {"bytes": matrix + 24.0 * n_v, "flops": 6.0 * ROW * n_v}
    if kind == "refit":                    # nested dissection of a planar lattice: about 10 n^1.5 operations
        return {"bytes": mesh + matrix + 32.0 * n_v, "flops": 200.0 * n_t + 10.0 * n_v ** 1.5}
    it = case["n_iter"] + (case["n_newton"] + 1 if kind == "adjoint" else 0)
    io = (48.0 + (72.0 if kind == "adjoint" else 0.0)) * n_v + (8.0 * n_t if kind == "adjoint" else 0.0)
    return {"bytes": mesh + matrix + io, "flops": float(it * (LOCAL_FLOPS * n_t + 6 * ROW * n_v))}


# ---- the same in 64 bits, with torch alone -------------------------------------

def _svd(F):
    """F = U diag(s) W^T with U, W rotations (the last s carries the sign of det F)."""
    parts = [torch.linalg.svd(f) for f in F.split(200000)]
    U, s, Wh = (torch.cat([p[k] for p in parts]) for k in range(3))
    du, dw = torch.linalg.det(U), torch.linalg.det(Wh)
    U, s, Wh = U.clone(), s.clone(), Wh.clone()
    U[:, :, 2] *= du[:, None]
    Wh[:, 2, :] *= dw[:, None]
    s[:, 2] *= du * dw
    return U, s, Wh


def _volume(s):
    """Nearest targets with product 1: d_i (d_i - s_i) = mu for all i, mu by bisection over the smallest target."""
    def others(t):
        mu = t * (t - s[:, 2])
        return 0.5 * (s[:, :2] + torch.sqrt(torch.clamp(s[:, :2] ** 2 + 4 * mu[:, None], min=0.0)))
    a = torch.clamp(0.5 * s[:, 2], min=0.01)
    b = torch.clamp(s[:, 2], min=0.0) + 1.0
    for _ in range(60):
        t = 0.5 * (a + b)
        low = others(t).prod(1) * t < 1
        a, b = torch.where(low, t, a), torch.where(low, b, t)
    t = 0.5 * (a + b)
    return torch.cat([others(t), t[:, None]], 1)


class _Exact:
    """The mesh, its matrix K and the PD iteration in FP64."""

    def __init__(self, case, a):
        rest, tets, _, pinned = _geo(case)
        d = dict(dtype=torch.float64, device="cuda")
        self.rest, self.tets = torch.tensor(rest, **d), torch.tensor(tets, device="cuda").long()
        self.n, self.pin = len(rest), torch.tensor(pinned != 0, device="cuda")
        self.free = ~self.pin
        e = self.rest[self.tets[:, 1:]] - self.rest[self.tets[:, :1]]       # rows: edges
        self.vol = torch.linalg.det(e).abs() / 6
        g = torch.linalg.inv(e).transpose(1, 2)                             # rows: gradients of corners 1..3
        self.g = torch.cat([-g.sum(1, keepdim=True), g], 1)                 # n_t x 4 x 3
        th = a["theta"].double()
        self.ws, self.wv = self.vol * th, self.vol * (10 * a["theta"]).double()
        self.mass = torch.zeros(self.n, **d).index_add_(0, self.tets.reshape(-1), (self.vol * DENSITY / 4).repeat_interleave(4))
        i = self.tets[:, :, None].expand(-1, 4, 4).reshape(-1)
        j = self.tets[:, None, :].expand(-1, 4, 4).reshape(-1)
        v = ((self.ws + self.wv)[:, None, None] * (self.g @ self.g.transpose(1, 2))).reshape(-1)
        k = torch.arange(self.n, device="cuda")
        coo = torch.sparse_coo_tensor(torch.stack([torch.cat([i, k]), torch.cat([j, k])]),
                                      torch.cat([v, self.mass / DT ** 2]), (self.n, self.n)).coalesce()
        self.K = coo.to_sparse_csr()
        r, c = coo.indices()
        self.diag = torch.zeros(self.n, **d).index_add_(0, r[r == c], coo.values()[r == c])

    def F(self, x):
        return x[self.tets].transpose(1, 2) @ self.g

    def corners(self, P):
        """sum over elements and corners of P g_c."""
        f = (self.g @ P.transpose(1, 2)).reshape(-1, 3)
        return torch.zeros((self.n, 3), dtype=P.dtype, device="cuda").index_add_(0, self.tets.reshape(-1), f)

    def targets(self, x):
        U, s, Wh = _svd(self.F(x))
        return U @ Wh, (U * _volume(s)[:, None, :]) @ Wh

    def cg(self, op, diag, b, tol=1e-14, most=4000):
        """op x = b on the free vertices, three columns at once, Jacobi preconditioner."""
        f = self.free[:, None].double()
        b = b * f
        x, r = torch.zeros_like(b), b.clone()
        z = r / diag
        p, rz, stop = z.clone(), (r * z).sum(), float((b * b).sum()) * tol ** 2
        for k in range(most):
            q = op(p) * f
            alpha = rz / (p * q).sum()
            x, r = x + alpha * p, r - alpha * q
            if k % 25 == 24 and float((r * r).sum()) <= stop:
                break
            z = r / diag
            new = (r * z).sum()
            p, rz = z + (new / rz) * p, new
        return x

    def solve(self, b, guess=None):
        g = torch.zeros_like(b) if guess is None else guess * self.free[:, None]
        return g + self.cg(lambda p: self.K @ p, self.diag[:, None], b - self.K @ g)

    def rhs(self, x, y):
        R, V = self.targets(x)
        b = self.mass[:, None] / DT ** 2 * y + self.corners(self.ws[:, None, None] * R + self.wv[:, None, None] * V)
        p = torch.where(self.pin[:, None], x, 0.0)
        return (b - self.K @ p) * self.free[:, None]

    def frame(self, x0, v0, pins, n_iter):
        y = x0 + DT * v0 + DT ** 2 * torch.tensor(GRAVITY, dtype=torch.float64, device="cuda")
        x = y.clone()
        x[self.pin] = pins
        for _ in range(n_iter):
            s = self.solve(self.rhs(x, y), x)
            x = torch.where(self.free[:, None], s, x)
        return x, (x - x0) / DT, y

    def hessian(self, x):
        """Per element the 9 x 9 second derivative of its energy (for F by rows), and F - R, F - V."""
        F = self.F(x)
        U, s, Wh = _svd(F)
        R, S = U @ Wh, Wh.transpose(1, 2) @ (s[:, :, None] * Wh)
        d = _volume(s)
        V = (U * d[:, None, :]) @ Wh
        n, eye9 = len(F), torch.eye(9, dtype=F.dtype, device="cuda").reshape(9, 3, 3)
        # dR = R [w]x with (tr S I - S) w = axial(R^T dF - dF^T R)
        A = torch.linalg.inv(S.diagonal(dim1=1, dim2=2).sum(1)[:, None, None] * torch.eye(3, dtype=F.dtype, device="cuda") - S)
        Q = R.transpose(1, 2)[:, None] @ eye9[None]
        Q = Q - Q.transpose(2, 3)
        w = torch.stack([Q[..., 2, 1], Q[..., 0, 2], Q[..., 1, 0]], -1) @ A.transpose(1, 2)
        z = torch.zeros_like(w[..., 0])
        X = torch.stack([z, -w[..., 2], w[..., 1], w[..., 2], z, -w[..., 0], -w[..., 1], w[..., 0], z], -1).reshape(n, 9, 3, 3)
        dR = (R[:, None] @ X).reshape(n, 9, 9)
        # V - F = mu V^-T, det V = 1: differentiate both
        T = torch.linalg.inv(V).transpose(1, 2)
        mu = (d[:, 2] * (d[:, 2] - s[:, 2]))[:, None, None]
        M = torch.zeros((n, 10, 10), dtype=F.dtype, device="cuda")
        cols = (T[:, None] @ eye9.transpose(1, 2)[None] @ T[:, None]).reshape(n, 9, 9)     # V^-T dV^T V^-T
        M[:, :9, :9] = torch.eye(9, dtype=F.dtype, device="cuda") + mu * cols.transpose(1, 2)
        M[:, :9, 9] = -T.reshape(n, 9)
        M[:, 9, :9] = T.reshape(n, 9)
        rhs = torch.zeros((n, 10, 9), dtype=F.dtype, device="cuda")
        rhs[:, :9] = torch.eye(9, dtype=F.dtype, device="cuda")
        dV = torch.linalg.solve(M, rhs)[:, :9]
        I9 = torch.eye(9, dtype=F.dtype, device="cuda")
        H = self.ws[:, None, None] * (I9 - dR.transpose(1, 2)) + self.wv[:, None, None] * (I9 - dV)
        return H, F - R, F - V

    def adjoint(self, x0, v0, pins, target, n_iter):
        x, _, y = self.frame(x0, v0, pins, n_iter)
        mh2 = self.mass[:, None] / DT ** 2

        def op(H):
            return lambda p: mh2 * p + self.corners((H @ self.F(p).reshape(-1, 9, 1)).reshape(-1, 3, 3))
        for _ in range(6):
            H, A, B = self.hessian(x)
            g = mh2 * (x - y) + self.corners(self.ws[:, None, None] * A + self.wv[:, None, None] * B)
            x = x - self.cg(op(H), self.diag[:, None], g)
        H, A, B = self.hessian(x)
        dl = 2 * (x - target) * self.free[:, None]
        lam = self.F(self.cg(op(H), self.diag[:, None], dl))
        return (dl * dl).sum().reshape(1) / 4, x, -self.vol * (A * lam).sum((1, 2)), -self.vol * (B * lam).sum((1, 2))


def exact(case, seed):
    kind = case["kind"]
    if kind == "serve":     # thousands of iterations in 64 bits: minutes
        return None
    a = {k: torch.from_numpy(v).cuda() for k, v in _case_arrays(case, seed).items()}
    if kind == "project":
        U, s, Wh = _svd(a["F"].double())
        return {"R": U @ Wh, "V": (U * _volume(s)[:, None, :]) @ Wh, "s": s}
    E = _Exact(case, a)
    x, v = a["x"].double(), a["v"].double()
    if kind == "local":
        return {"b": E.rhs(x, a["y"].double())}
    if kind in ("solve", "refit"):
        return {"x": E.solve(a["r"].double())}
    if kind == "frame":
        x, v, _ = E.frame(x, v, a["pins"].double(), case["n_iter"])
        return {"x": x, "v": v}
    loss, x, gs, gv = E.adjoint(x, v, a["pins"].double(), a["target"].double(), case["n_iter"])
    return {"loss": loss, "x": x, "gs": gs, "gv": gv}
