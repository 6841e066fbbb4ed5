"""Performance cases of the MS-GFEM local stage, its coarse problem, the fine solver and the warm-start network.

Every case goes through the public Python entry points (``MSGFEM``, ``Net``) as a user's
program does: a handle is set up once per mesh and partition, new ply angles come in, the
local stage, coarse assembly and coarse solve run, eigenvalues and the displacement go out.
Beams have 2 mm in-plane elements and 0.25 mm plies; sections are curved C-profiles with node
coordinates and ply frames.  ``exact`` is a dense 64-bit finite-element solution of the same
definitions (element integrals, partition of unity, local eigenproblems, Galerkin solve).
"""
import math

import numpy as np
import torch

from paper_2211_13893_gb300 import MSGFEM, Net

PLY = (162000.0, 10000.0, 10000.0, 5200.0, 5200.0, 3500.0, 0.35, 0.35, 0.5)
HX, HY, HZ, TRACTION = 2.0, 2.0, 0.25, 1.0
FP64, MIXED = 0, 1
SIGMA = 1e-2   # shift of the dense reference's pencil


def listed():
    def beam(name, kind, nx, ny, nz, sx, sy, o, os, n_loc, precision, **kw):
        return dict(name=name, kind=kind, nx=nx, ny=ny, nz=nz, sx=sx, sy=sy, o=o, os=os, n_loc=n_loc,
                    precision=precision, **kw)
    return [
        # the smallest problem a user solves: one laminated beam in two subdomains, full precision
        beam("beam_small_fp64", "step", 24, 4, 12, 2, 1, 1, 2, 8, FP64),
        # odd sizes, ragged subdomains (clamped, floating, interior), both precisions
        beam("beam_ragged_fp64", "step", 47, 7, 13, 5, 2, 1, 3, 13, FP64),
        beam("beam_ragged_mixed", "step", 47, 7, 13, 5, 2, 1, 3, 13, MIXED),
        # a stretch of a 39-ply beam with large subdomains, full precision
        beam("beam_large_fp64", "step", 36, 12, 39, 3, 2, 2, 4, 20, FP64),
        # the 192 x 12 x 39 beam (301,080 DoF, 32 subdomains) in mixed precision
        beam("beam_full_mixed", "step", 192, 12, 39, 16, 2, 2, 4, 20, MIXED),
        # a curved C-section with uneven subdomains and one eigenpair count per subdomain
        dict(name="section_mixed", kind="section", nx=36, flange=8, corner=8, web=14, nz=32, sx=4, sy=4, o=1, os=3,
             n_loc=16, n_max=31, precision=MIXED),
        # many small beams, each with its own wrinkle field, in one handle
        dict(name="batch_mixed", kind="batch", nx=24, ny=4, nz=12, sx=2, sy=1, o=1, os=2, n_loc=8, precision=MIXED,
             instances=48),
        # the GenEO comparison method
        beam("geneo_fp64", "geneo", 40, 6, 12, 4, 2, 2, 2, 16, FP64),
        # the fine solution by two-level Schwarz PCG on resident factors
        beam("fine_solve_fp64", "fine", 40, 6, 12, 4, 2, 2, 4, 12, FP64),
        # coarse problem and accuracy figures for several thresholds of one local stage
        beam("coarse_errors", "coarse", 96, 12, 13, 16, 2, 2, 4, 20, MIXED),
        # warm-start network: one epoch of training, and inference for a batch of beams
        dict(name="net_train", kind="train", features=672, hidden=32, outputs=1560, batch=64, steps=6),
        dict(name="net_infer", kind="infer", features=672, hidden=32, outputs=1560, batch=128),
    ]


def _cost(c):
    """Factorisation work of a beam case (flops, mixed precision weighted by its rate)."""
    w = _factor_flops(c)
    return w if c["precision"] == FP64 else w / 10.0


def draw(rng):
    def log(a, b):
        return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))
    kind = rng.choice(["step", "step", "step", "step", "section", "batch", "geneo", "fine", "coarse", "train", "infer"])
    if kind in ("train", "infer"):
        c = dict(kind=kind, features=log(60, 4000), hidden=log(16, 128), outputs=8 * log(20, 800), batch=log(1, 256))
        return dict(c, steps=rng.randint(1, 8)) if kind == "train" else c
    while True:
        precision = rng.choice([FP64, MIXED])
        if kind == "section":
            c = dict(kind=kind, nx=log(8, 36), flange=rng.randint(3, 8), corner=rng.randint(3, 8),
                     web=rng.randint(5, 14), nz=log(6, 32), sx=rng.randint(2, 4), sy=rng.randint(2, 4), o=1,
                     os=rng.randint(2, 3), n_loc=rng.randint(8, 12), n_max=rng.randint(13, 20), precision=precision)
        else:
            o = rng.randint(1, 2)
            c = dict(kind=kind, nx=log(12, 192), ny=log(3, 12), nz=log(4, 39), sx=log(2, 16), sy=rng.randint(1, 2),
                     o=o, os=o + rng.randint(1, 2), n_loc=rng.randint(7, 20), precision=precision)
            if kind == "geneo":
                c["os"] = o
            if kind == "batch":
                c.update(instances=log(2, 64), n_loc=rng.randint(7, 10))
        # subdomains a few elements wide and not much longer than the listed ones, beams no more slender
        # than twice the long listed ones, fewer pairs on small interfaces, the work below that of the
        # largest listed case of the kind
        wide, long = _ny(c) // c["sy"], c["nx"] // c["sx"]
        top = c.get("n_max", c["n_loc"])
        shape = wide >= 3 and 4 <= long <= 18 - 2 * c["os"] + wide // 2 and c["nx"] <= 7 * c["nz"]
        if shape and 10 * (top - 6) <= (c["nz"] + 1) * wide and _cost(c) <= dict(step=1.3e11, geneo=2e10).get(kind, 6e10):
            return c


# ---------------------------------------------------------------- geometry and inputs
def _ny(c):
    return 2 * c["flange"] + 2 * c["corner"] + c["web"] if c["kind"] == "section" else c["ny"]


def _cuts(n, parts):
    return [n * a // parts for a in range(parts + 1)]


def _boxes(c):
    """Non-overlapping element boxes, subdomain a sy + b (the library's own split of a regular partition)."""
    x, y = _cuts(c["nx"], c["sx"]), _cuts(_ny(c), c["sy"])
    return [(x[a], x[a + 1], y[b], y[b + 1]) for a in range(c["sx"]) for b in range(c["sy"])]


def _grown(c, box, m):
    return max(0, box[0] - m), min(c["nx"], box[1] + m), max(0, box[2] - m), min(_ny(c), box[3] + m)


def _star_dofs(c):
    return [3 * (g[1] - g[0] + 1) * (g[3] - g[2] + 1) * (c["nz"] + 1) for g in (_grown(c, b, c["os"]) for b in _boxes(c))]


def _counts(c):
    """Eigenpairs per subdomain of a section: growing with the oversampling domain, n_loc to n_max."""
    s = np.array(_star_dofs(c), dtype=np.float64)
    f = (s - s.min()) / max(s.max() - s.min(), 1.0)
    return (c["n_loc"] + np.floor((c["n_max"] - c["n_loc"]) * f + 0.5)).astype(np.int32)


def _layup(nz, rng):
    half = [(0.0, 90.0, 45.0, -45.0)[i % 4] for i in range((nz + 1) // 2)]
    return np.array(half + half[:nz // 2][::-1]) + rng.standard_normal(nz)


def _angles(c, seed):
    """Element angles in degrees: the (0, 90, 45, -45) cycle, symmetric, with 1 degree noise per
    ply; a batch adds to every copy its own smooth wrinkle field (sd about 3 degrees)."""
    rng = np.random.default_rng(seed)
    shape = (c["nx"], _ny(c), c["nz"])
    if c["kind"] != "batch":
        return np.broadcast_to(_layup(c["nz"], rng), shape).copy()
    x, y, z = np.meshgrid(*[np.arange(n) / 6.0 for n in shape], indexing="ij")
    out = []
    for _ in range(c["instances"]):
        f = np.zeros(shape)
        for _ in range(8):
            k, ph = rng.standard_normal(3), rng.uniform(0, 2 * math.pi)
            f += 1.5 * np.cos(k[0] * x + k[1] * y + 0.2 * k[2] * z + ph)
        out.append(np.broadcast_to(_layup(c["nz"], np.random.default_rng(1)), shape) + f)
    return np.stack(out)


def _nodes(c):
    """Node coordinates and ply frames (frames None on a beam)."""
    nx, ny, nz = c["nx"], _ny(c), c["nz"]
    if c["kind"] != "section":
        g = np.meshgrid(HX * np.arange(nx + 1), HY * np.arange(ny + 1), HZ * np.arange(nz + 1), indexing="ij")
        return np.stack(g, axis=-1), None
    # a C-profile in the y-z plane: flange, corner arc, web, corner arc, flange, walked along the arc
    r, step = 8.0, 4.0
    p, d = [np.array([c["flange"] * step + r, 0.0])], []
    turn = [0.0] * c["flange"] + [1.0] * c["corner"] + [0.0] * c["web"] + [1.0] * c["corner"] + [0.0] * c["flange"]
    ang, nrm = math.pi, []
    for t in turn:
        dphi = -0.5 * math.pi / c["corner"] if t else 0.0
        length = 2.0 * r * math.sin(-0.5 * dphi) if t else step
        nrm.append(ang)
        p.append(p[-1] + length * np.array([math.cos(ang + 0.5 * dphi), math.sin(ang + 0.5 * dphi)]))
        ang += dphi
    nrm.append(ang)
    p = np.array(p)
    n = np.stack([np.sin(nrm), -np.cos(nrm)], axis=1) * -1.0   # outward: left of the walking direction
    off = HZ * np.arange(nz + 1)
    xyz = np.empty((nx + 1, ny + 1, nz + 1, 3))
    xyz[..., 0] = (4.0 * np.arange(nx + 1))[:, None, None]
    for a in range(2):
        xyz[..., 1 + a] = (p[:, a][:, None] + off[None, :] * n[:, a][:, None])[None]
    d = (p[1:] - p[:-1]) / np.linalg.norm(p[1:] - p[:-1], axis=1, keepdims=True)
    fr = np.zeros((ny, 3, 3))
    fr[:, 0, 0], fr[:, 1, 1:], fr[:, 2, 1], fr[:, 2, 2] = 1.0, d, -d[:, 1], d[:, 0]
    return xyz, np.broadcast_to(fr[None, :, None], (nx, ny, nz, 3, 3)).copy()


def _handle(c, angles, **kw):
    if c["kind"] == "section":
        xyz, frames = _nodes(c)
        return MSGFEM(c["nx"], _ny(c), c["nz"], 0.0, 0.0, 0.0, TRACTION, PLY, angles, c["sx"], c["sy"], c["o"], c["os"],
                      seed=7, precision=c["precision"], xyz=xyz, frames=frames, boxes=np.array(_boxes(c)), **kw)
    return MSGFEM(c["nx"], c["ny"], c["nz"], HX, HY, HZ, TRACTION, PLY, angles, c["sx"], c["sy"], c["o"],
                  kw.pop("os", c["os"]), seed=7, precision=c["precision"], **kw)


def _reference(c):
    """A smooth displacement field that vanishes on the clamped face (coarse accuracy figures)."""
    xyz, _ = _nodes(c)
    x = xyz[..., 0] / xyz[-1, 0, 0, 0]
    u = np.stack([-2e-5 * xyz[..., 0], 4e-4 * x ** 2 * (1 + 0.1 * xyz[..., 1]), -9e-4 * x ** 2 * (1 - 0.3 * x)], axis=-1)
    return u.reshape(-1)


# ---------------------------------------------------------------- the passes
def prepare(case, seed):
    c = case
    if c["kind"] in ("train", "infer"):
        rng = np.random.default_rng(seed)
        sizes = [c["features"], c["hidden"], c["outputs"]]
        net = Net(sizes, c["batch"], _weights(c, rng))
        nb = c.get("steps", 1)
        x = torch.from_numpy(rng.standard_normal((nb, c["batch"], c["features"])).astype(np.float32)).cuda()
        t = torch.from_numpy(rng.standard_normal((nb, c["batch"], c["outputs"])).astype(np.float32)).cuda()
        y = torch.zeros((c["batch"], c["outputs"]), dtype=torch.float32, device="cuda")
        return dict(case=c, net=net, x=x, t=t, y=y)
    ang = _angles(c, seed)
    s = dict(case=c, angles=torch.from_numpy(ang.reshape(-1)).cuda())
    if c["kind"] == "fine":
        s["m"] = _handle(c, ang)
        s["m"].local_spaces(c["n_loc"])
        s["m"].coarse_assemble()
        s["local"] = _handle(c, ang, os=c["o"])
    elif c["kind"] == "geneo":
        s["m"] = _handle(c, ang, method=1)
    elif c["kind"] == "batch":
        s["m"] = _handle(c, ang, instances=c["instances"], tol=1e-6)
    else:
        s["m"] = _handle(c, ang)
    if c["kind"] == "coarse":
        s["m"].local_spaces(c["n_loc"])
        s["ref"] = torch.from_numpy(_reference(c)).cuda()
    m = s["m"]
    s["n_loc"] = _counts(c) if c["kind"] == "section" else c["n_loc"]
    s["lam"] = torch.zeros((m.N, int(np.max(s["n_loc"]))), dtype=torch.float64, device="cuda")
    s["u"] = torch.zeros(m.n_dof, dtype=torch.float64, device="cuda")
    return s


def run(state):
    s, c = state, state["case"]
    if c["kind"] == "train":
        for b in range(c["steps"]):
            s["net"].adam_step(s["x"][b], s["t"][b], c["batch"], 3e-4)
        return s["net"].params()
    if c["kind"] == "infer":
        s["net"].forward(s["x"][0], s["y"], c["batch"])
        return s["y"]
    m = s["m"]
    if c["kind"] == "fine":
        u, _ = s["local"].schwarz_solve(m, rtol=1e-12, u_out=s["u"])
        return u
    if c["kind"] == "coarse":
        out = []
        for t in (0.0, 0.02):
            m.coarse_assemble(threshold=t)
            u, err = m.solve(u_ref=s["ref"], u_out=s["u"])
            out.append([u.clone(), err, *m.solution_errors(s["ref"])])
        return out
    m.update_angles(s["angles"])
    lam = m.local_spaces(s["n_loc"], lam_out=s["lam"])
    if c["kind"] == "batch":
        return lam
    m.coarse_assemble()
    u, _ = m.solve(u_out=s["u"])
    return [lam, u]


# ---------------------------------------------------------------- floors
def _layers(c):
    """(kept DoFs per node layer of K, of A11) of every subdomain."""
    out = []
    for b in _boxes(c):
        g = _grown(c, b, c["os"])
        lx, ly = g[1] - g[0] + 1, g[3] - g[2] + 1
        clamp, cuts = g[0] == 0, [g[0] > 0, g[1] < c["nx"], g[2] > 0, g[3] < _ny(c)]
        k = 3 * (lx - clamp) * ly
        out.append((k, 3 * (lx - clamp - cuts[0] - cuts[1]) * (ly - cuts[2] - cuts[3])))
    return out


def _factor_flops(c):
    nl, f = c["nz"] + 1, 0.0
    for k, a in _layers(c):
        f += sum(nl * n ** 3 / 3.0 + (nl - 1) * 2.0 * n ** 3 for n in (k, a))
    return f * c.get("instances", 1)


def _solve_flops(c, cols):
    nl = c["nz"] + 1
    return c.get("instances", 1) * sum((4.0 * (nl - 1) + 2.0 * nl) * n * n * cols for ka in _layers(c) for n in ka)


def work(case):
    """Inputs read once, outputs written once, and the arithmetic of the path: the banded Cholesky
    factorisations of K and A11, and a Krylov space just large enough for the wanted pairs."""
    c = case
    if c["kind"] in ("train", "infer"):
        w = c["hidden"] * (c["features"] + c["outputs"])
        nb, fb = (c["steps"], 6.0) if c["kind"] == "train" else (1, 2.0)
        io = nb * c["batch"] * (c["features"] + c["outputs"])
        return {"bytes": 4.0 * (io + w * (6 * nb if c["kind"] == "train" else 1)), "flops": fb * nb * c["batch"] * w}
    nn = (c["nx"] + 1) * (_ny(c) + 1) * (c["nz"] + 1)
    nel = c["nx"] * _ny(c) * c["nz"] * c.get("instances", 1)
    nsub = c["sx"] * c["sy"] * c.get("instances", 1)
    m = c.get("n_max", c["n_loc"])
    star = float(sum(_star_dofs(c))) * c.get("instances", 1)
    stencil = 81.0 * 2.0
    if c["kind"] == "coarse":
        nc = nsub * (m + 1.0)
        return {"bytes": 2 * 8.0 * (star * m + 4 * 3 * nn),
                "flops": 2 * (star * (m + 1) * stencil + 9 * nc / nsub * star * (m + 1) * 2 / 4 + nc ** 3 / 3)}
    if c["kind"] == "fine":
        its = 15
        return {"bytes": 8.0 * (its * sum((c["nz"] + 1) * 3.0 * a * a for _, a in _layers(c)) + 2 * 3 * nn),
                "flops": its * (_solve_flops(c, 1) / 2 + 3 * nn * stencil)}
    steps = math.ceil(m / 8.0) + 1
    return {"bytes": 8.0 * (nel + nsub * m + 3 * nn),
            "flops": _factor_flops(c) + _solve_flops(c, 8 * steps) + steps * 3 * star * 8 * stencil}


# ---------------------------------------------------------------- dense 64-bit reference
def _weights(c, rng):
    parts = []
    for a, b in ((c["features"], c["hidden"]), (c["hidden"], c["outputs"])):
        parts += [rng.standard_normal(a * b) / math.sqrt(a), 0.1 * rng.standard_normal(b)]
    return np.concatenate(parts).astype(np.float32)


def _exact_net(c, seed):
    rng = np.random.default_rng(seed)
    F, H, O, B = c["features"], c["hidden"], c["outputs"], c["batch"]
    p = torch.from_numpy(_weights(c, rng)).double().cuda().requires_grad_(True)
    nb = c.get("steps", 1)
    x = torch.from_numpy(rng.standard_normal((nb, B, F)).astype(np.float32)).double().cuda()
    t = torch.from_numpy(rng.standard_normal((nb, B, O)).astype(np.float32)).double().cuda()

    def forward(xb):
        w1, b1, w2, b2 = torch.split(p, [F * H, H, H * O, O])
        return torch.tanh(xb @ w1.view(H, F).T + b1) @ w2.view(O, H).T + b2
    if c["kind"] == "infer":
        return forward(x[0]).detach()
    m, v = torch.zeros_like(p), torch.zeros_like(p)
    for k in range(nb):
        g, = torch.autograd.grad(((forward(x[k]) - t[k]) ** 2).mean(), p)
        m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
        step = 3e-4 * (m / (1 - 0.9 ** (k + 1))) / (torch.sqrt(v / (1 - 0.999 ** (k + 1))) + 1e-8)
        with torch.no_grad():
            p -= step
    return p.detach()


def _elements(c, angles):
    """Per element: its 24 DoFs, stiffness, mass and strain-norm matrices (2x2x2 Gauss)."""
    nx, ny, nz = c["nx"], _ny(c), c["nz"]
    xyz, frames = _nodes(c)
    i, j, k = (a.reshape(-1) for a in np.meshgrid(np.arange(nx), np.arange(ny), np.arange(nz), indexing="ij"))
    corner = [(0, 0, 0), (1, 0, 0), (0, 1, 0), (1, 1, 0), (0, 0, 1), (1, 0, 1), (0, 1, 1), (1, 1, 1)]
    node = np.stack([((i + a) * (ny + 1) + j + b) * (nz + 1) + k + d for a, b, d in corner], axis=1)
    X = torch.from_numpy(xyz.reshape(-1, 3)[node]).cuda()
    fr = np.broadcast_to(np.eye(3), (len(i), 3, 3)) if frames is None else frames.reshape(-1, 3, 3)
    fr = torch.from_numpy(np.ascontiguousarray(fr)).cuda()
    th = torch.from_numpy(np.deg2rad(angles.reshape(-1))).cuda()
    R = torch.stack([torch.cos(th)[:, None] * fr[:, 0] + torch.sin(th)[:, None] * fr[:, 1],
                     -torch.sin(th)[:, None] * fr[:, 0] + torch.cos(th)[:, None] * fr[:, 1], fr[:, 2]], dim=1)
    E1, E2, E3, G12, G13, G23, n12, n13, n23 = PLY
    S = np.zeros((6, 6))
    S[:3, :3] = [[1 / E1, -n12 / E1, -n13 / E1], [-n12 / E1, 1 / E2, -n23 / E2], [-n13 / E1, -n23 / E2, 1 / E3]]
    S[3, 3], S[4, 4], S[5, 5] = 1 / G23, 1 / G13, 1 / G12
    C = torch.from_numpy(np.linalg.inv(S)).cuda()
    ne = len(i)
    K, M, N = (torch.zeros((ne, 24, 24), dtype=torch.float64, device="cuda") for _ in range(3))
    gp = 1 / math.sqrt(3.0)
    for g in range(8):
        q = [(2 * ((g >> a) & 1) - 1) * gp for a in range(3)]
        f = [[0.5 * (1 + (2 * cn[a] - 1) * q[a]) for a in range(3)] for cn in corner]
        shape = torch.tensor([a[0] * a[1] * a[2] for a in f], dtype=torch.float64, device="cuda")
        dn = torch.tensor([[(cn[a] - 0.5) * f[m][(a + 1) % 3] * f[m][(a + 2) % 3] for a in range(3)]
                           for m, cn in enumerate(corner)], dtype=torch.float64, device="cuda")
        J = torch.einsum("ma,emx->eax", dn, X)
        w = torch.linalg.det(J)
        D = torch.einsum("eax,ma->emx", torch.linalg.inv(J).transpose(1, 2), dn)   # dN_m / dx
        grad = torch.einsum("emx,yv->exymv", D, torch.eye(3, dtype=torch.float64, device="cuda")).reshape(ne, 3, 3, 24)
        eps = 0.5 * (grad + grad.transpose(1, 2))
        loc = torch.einsum("eax,exyn,eby->eabn", R, eps, R)
        v = torch.stack([loc[:, 0, 0], loc[:, 1, 1], loc[:, 2, 2], 2 * loc[:, 1, 2], 2 * loc[:, 0, 2], 2 * loc[:, 0, 1]], 1)
        K += w[:, None, None] * torch.einsum("ean,ab,ebm->enm", v, C, v)
        N += w[:, None, None] * torch.einsum("exyn,exym->enm", eps, eps)
        M += w[:, None, None] * torch.kron(torch.outer(shape, shape), torch.eye(3, dtype=torch.float64, device="cuda"))
    dof = torch.from_numpy((3 * node[:, :, None] + np.arange(3)).reshape(ne, 24)).cuda()
    return (i, j, k), dof, K, M, N


def _dense(n, dof, Ke):
    A = torch.zeros(n * n, dtype=torch.float64, device="cuda")
    A.index_add_(0, (dof[:, :, None] * n + dof[:, None, :]).reshape(-1), Ke.reshape(-1))
    return A.view(n, n)


def _load(c):
    nx, ny, nz = c["nx"], _ny(c), c["nz"]
    xyz, _ = _nodes(c)
    b = np.zeros(xyz.shape)
    X = xyz[nx]
    for g in range(4):
        s, t = [0.5 + (0.5 if (g >> a) & 1 else -0.5) / math.sqrt(3.0) for a in range(2)]
        w = {(0, 0): (1 - s) * (1 - t), (1, 0): s * (1 - t), (0, 1): (1 - s) * t, (1, 1): s * t}
        ds = (1 - t) * (X[1:, :-1] - X[:-1, :-1]) + t * (X[1:, 1:] - X[:-1, 1:])
        dt = (1 - s) * (X[:-1, 1:] - X[:-1, :-1]) + s * (X[1:, 1:] - X[1:, :-1])
        area = 0.25 * np.linalg.norm(np.cross(ds, dt), axis=-1)
        for (a, d), f in w.items():
            b[nx, a:ny + a, d:nz + d, 0] -= TRACTION * f * area
    return torch.from_numpy(b.reshape(-1)).cuda()


def _local(c, box, el, b, weight, total, n_loc):
    """Eigenvalues and weighted local basis of one subdomain (full DoF numbering of the mesh)."""
    nx, ny, nz = c["nx"], _ny(c), c["nz"]
    (i, j, _), dof, K, _, _ = el
    g = _grown(c, box, c["os"])
    inside = torch.from_numpy((i >= g[0]) & (i < g[1]) & (j >= g[2]) & (j < g[3])).cuda()
    I, J = (a.reshape(-1) for a in np.meshgrid(np.arange(nx + 1), np.arange(ny + 1), indexing="ij"))
    keep = (I >= g[0]) & (I <= g[1]) & (J >= g[2]) & (J <= g[3]) & (I > 0)
    cut = ((I == g[0]) & (g[0] > 0)) | ((I == g[1]) & (g[1] < nx)) | ((J == g[2]) & (g[2] > 0)) | ((J == g[3]) & (g[3] < ny))
    full = lambda m: torch.from_numpy(np.repeat(m, 3 * (nz + 1))).cuda()  # noqa: E731
    rows = torch.nonzero(full(keep)).view(-1)
    n = len(rows)
    place = torch.full((3 * (nx + 1) * (ny + 1) * (nz + 1),), n, dtype=torch.int64, device="cuda")
    place[rows] = torch.arange(n, device="cuda")
    A = _dense(n + 1, place[dof[inside]], K[inside])[:n, :n]
    mu = torch.from_numpy(np.repeat(weight / total, 3 * (nz + 1))).cuda()[rows]
    B = mu[:, None] * A * mu[None, :]
    elim = (mu == 0) if c["kind"] == "geneo" else ~full(cut)[rows]
    c1, c2 = torch.nonzero(elim).view(-1), torch.nonzero(~elim).view(-1)
    L = torch.linalg.cholesky(A[c1][:, c1])
    E = torch.zeros((n, len(c2)), dtype=torch.float64, device="cuda")
    E[c2, torch.arange(len(c2), device="cuda")] = 1.0
    E[c1] = -torch.cholesky_solve(A[c1][:, c2], L)
    S = A[c2] @ E
    T = E.T @ (B @ E)
    S, T = 0.5 * (S + S.T), 0.5 * (T + T.T)
    Lc = torch.linalg.cholesky(S + SIGMA * T)
    W = torch.linalg.solve_triangular(Lc, torch.linalg.solve_triangular(Lc, T, upper=False).T, upper=False)
    th, y = torch.linalg.eigh(0.5 * (W + W.T))
    th, y = th.flip(0)[:n_loc], y.flip(1)[:, :n_loc]
    phi = E @ torch.linalg.solve_triangular(Lc.T, y, upper=True)
    if c["kind"] != "geneo" and float(b[rows][c1].abs().max()) > 0:
        psi = torch.zeros((n, 1), dtype=torch.float64, device="cuda")
        psi[c1] = torch.cholesky_solve(b[rows][c1][:, None], L)
        phi = torch.cat([phi, psi], dim=1)
    return 1.0 / th - SIGMA, rows, mu[:, None] * phi


def _exact_spaces(c, angles, el):
    boxes, nx, ny = _boxes(c), c["nx"], _ny(c)
    I, J = (a.reshape(-1) for a in np.meshgrid(np.arange(nx + 1), np.arange(ny + 1), indexing="ij"))
    ws = []
    for box in boxes:
        g = _grown(c, box, c["o"])
        w = np.full(I.shape, 2.0 * c["o"])
        for on, d in ((g[0] > 0, I - g[0]), (g[1] < nx, g[1] - I), (g[2] > 0, J - g[2]), (g[3] < ny, g[3] - J)):
            if on:
                w = np.minimum(w, np.maximum(d, 0))
        ws.append(w)
    n_loc = _counts(c) if c["kind"] == "section" else [c["n_loc"]] * len(boxes)
    b = _load(c)
    total = np.sum(ws, axis=0)
    got = [_local(c, box, el, b, w, total, int(n)) for box, w, n in zip(boxes, ws, n_loc)]
    lam = torch.full((len(boxes), int(max(n_loc))), math.nan, dtype=torch.float64, device="cuda")
    for q, (l, _, _) in enumerate(got):
        lam[q, :len(l)] = l
    return lam, got, b


def _apply(dof, Ke, u):
    y = torch.zeros_like(u)
    v = torch.einsum("enm,em...->en...", Ke, u[dof])
    return y.index_add_(0, dof.reshape(-1), v.reshape(dof.numel(), *u.shape[1:]))


def _galerkin(c, got, el, b, threshold):
    _, dof, K, _, _ = el
    cols = []
    for lam, rows, v in got:
        m = len(lam)
        keep = [q for q in range(v.shape[1]) if q >= m or threshold == 0.0 or abs(float(lam[q])) < 1.0 / threshold]
        z = torch.zeros((len(b), len(keep)), dtype=torch.float64, device="cuda")
        z[rows] = v[:, keep]
        cols.append(z)
    V = torch.cat(cols, dim=1)
    V = V / torch.linalg.norm(V, dim=0)
    AV = torch.cat([_apply(dof, K, V[:, q:q + 16]) for q in range(0, V.shape[1], 16)], dim=1)
    H = V.T @ AV
    d = torch.rsqrt(torch.diagonal(H))
    return V @ (d * torch.linalg.solve(d[:, None] * (0.5 * (H + H.T)) * d[None, :], d * (V.T @ b)))


def exact(case, seed):
    c = case
    if c["kind"] in ("train", "infer"):
        return _exact_net(c, seed)
    stars, nn = _star_dofs(c), 3 * (c["nx"] + 1) * (_ny(c) + 1) * (c["nz"] + 1)
    heavy = c.get("instances", 1) * sum(n ** 3 for n in stars) + (nn ** 3 if c["kind"] == "fine" else 0)
    if heavy > 6e12 or max(stars) > 12000 or c["nx"] * _ny(c) * c["nz"] > 12000:
        return None
    angles = _angles(c, seed)
    if c["kind"] == "batch":
        return torch.cat([_exact_spaces(c, a, _elements(c, a))[0] for a in angles])
    el = _elements(c, angles)
    if c["kind"] == "fine":
        free = 3 * (_ny(c) + 1) * (c["nz"] + 1)
        A, b = _dense(nn, el[1], el[2])[free:, free:], _load(c)
        u = torch.zeros(nn, dtype=torch.float64, device="cuda")
        u[free:] = torch.cholesky_solve(b[free:, None], torch.linalg.cholesky(A))[:, 0]
        return u
    lam, got, b = _exact_spaces(c, angles, el)
    if c["kind"] != "coarse":
        return [lam, _galerkin(c, got, el, b, 0.0)]
    ref, out = torch.from_numpy(_reference(c)).cuda(), []
    for t in (0.0, 0.02):
        u = _galerkin(c, got, el, b, t)
        out.append([u] + [math.sqrt(float((ref - u) @ _apply(el[1], m, ref - u)) / float(ref @ _apply(el[1], m, ref)))
                          for m in (el[2], el[3], el[4])])
    return out
