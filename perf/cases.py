"""The work that users of the library have it do, as measurable cases.

Each case is one call sequence of a user's program through the public entry
points (lib.Solver, lib.Batch, autograd.stress_of_theta), on synthetic
laminates of the families in inputs.py:

  first    a new laminate: from the mesh description to displacement and
           stresses (set-up, solve, stress recovery).  One design of a study.
  solve    a new load on a laminate that is set up: one PCG solve.
  batch1   a new set of laminates of uneven sizes: batch set-up and solve.
  batch    the solve of a batch that is set up.
  gradient p-norm of sigma_33 in the corner's resin and its gradient with
           respect to every fibre misalignment angle: a forward solve, an
           adjoint solve and the element contraction through torch.autograd.
  ku       K u alone, the operator a user builds other iterations on.
  post     sigma_33, tau_13 and the failure index of a given displacement.

prepare() makes what such a program holds before the call; exact() solves the
same problem in plain torch FP64 by a dense block elimination, with its own
assembly.  Tolerances are 1e-10 on the residual (the library's default), 3e-10
on the true residual for the mixed form, and 1e-12 for the gradient and
wherever stresses come back.
"""
import math

import numpy as np
import torch

from paper_1707_04228_gb300 import inputs, lib
from paper_1707_04228_gb300.autograd import pnorm, stress_of_theta

DEV = "cuda"
P_NORM = 8


# ---------------------------------------------------------------- the cases

def _corner(kind, name, n_arc, n_limb, n_width, nel, plies, px, py, **more):
    return dict(dict(name=name, kind=kind, family="corner", n_arc=n_arc, n_limb=n_limb, n_width=n_width, nel=nel,
                     plies=plies, px=px, py=py, nev=10, mixed=False, element=0, periodic=False, tol=1e-10), **more)


def _plate(kind, name, n, plies, px, py, **more):
    return dict(dict(name=name, kind=kind, family="plate", n=n, plies=plies, px=px, py=py, nev=8, mixed=False,
                     element=0, periodic=False, tol=1e-10), **more)


def _batch(kind, name, sizes, **more):
    """sizes: in-plane elements x plies of each plate."""
    return dict(dict(name=name, kind=kind, family="plates", sizes=sizes, nev=8, mixed=False, tol=1e-10), **more)


def listed():
    return [
        # the smallest laminate anyone sets up: a 4-ply coupon plate, everything from the mesh to the stresses
        _plate("first", "first_plate_10x10x7", 10, 4, 2, 2, tol=1e-12),
        # load case after load case on that coupon: latency of one small solve
        _plate("solve", "solve_plate_10x10x7", 10, 4, 2, 2),
        # one design of a corner study: 12 plies, set-up, solve and stresses in FP64
        _corner("first", "first_corner_20x6x23", 14, 3, 6, 1, 12, 5, 2, tol=1e-12),
        # the next load on an FP64 corner with two elements through every layer
        _corner("solve", "solve_corner_32x8x46", 26, 3, 8, 2, 12, 8, 2),
        # the same at the largest size kept here, with the FP32 preconditioner
        _corner("solve", "solve_corner_40x10x46_mixed", 32, 4, 10, 2, 12, 10, 2, mixed=True, tol=3e-10),
        # the paper's own 20-node element on an odd-sized corner
        _corner("solve", "solve_corner_19x5x23_s20", 13, 3, 5, 1, 12, 5, 1, element=1),
        # a parameter study: three plates of different sizes and stacks, grid chosen by the autotuner
        _batch("batch1", "batch1_3_plates", "10x4,11x5,10x6"),
        # further solves of a larger batch that is already set up
        _batch("batch", "batch_5_plates", "10x4,12x6,14x5,16x8,11x9"),
        # one gradient step of the fibre-waviness study
        _corner("gradient", "gradient_corner_16x4x23", 12, 2, 4, 1, 12, 4, 1, tol=1e-12),
        # the operator at the largest size here, and the post-processing of a full displacement field
        _corner("ku", "ku_corner_64x16x46", 56, 4, 16, 2, 12, 32, 8, nev=0),
        _corner("post", "post_corner_64x16x46", 56, 4, 16, 2, 12, 32, 8, nev=0),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["first", "first", "solve", "solve", "solve", "batch1", "batch", "gradient", "ku", "post"])
    if kind in ("batch1", "batch"):
        top = 11 if kind == "batch1" else 14
        sizes = ",".join("%dx%d" % (rng.randint(8, top), rng.randint(2, 6)) for _ in range(rng.randint(2, 3)))
        c = _batch(kind, None, sizes, nev=rng.randint(4, 8))
        c.pop("name")
        return c
    large = kind in ("ku", "post")
    tol = 1e-12 if kind in ("first", "gradient") else 1e-10
    if kind in ("first", "solve") and rng.random() < 0.4:
        n = _log(rng, 6, 14)
        c = _plate(kind, None, n, rng.randint(2, 8), max(1, n // 5), max(1, n // 4), nev=rng.randint(4, 8), tol=tol)
    else:
        width = _log(rng, 4, 14) if large else _log(rng, 2, 7)
        arc = _log(rng, 8, 48) if large else _log(rng, 5, 18)
        limb = rng.randint(1, 3)
        periodic = kind == "solve" and width <= 5 and rng.random() < 0.25
        py = 1 if periodic else max(1, width // 4)
        c = _corner(kind, None, arc, limb, width, 1 if not large else rng.randint(1, 2), 2 * rng.randint(2, 6),
                    max(1, (arc + 2 * limb) // (2 if large else 4)), py if not large else max(1, width // 2),
                    nev=0 if large else rng.randint(6, 10), tol=tol, periodic=periodic,
                    element=1 if kind == "solve" and not periodic and rng.random() < 0.25 else 0)
    if kind == "solve" and rng.random() < 0.4:
        c.update(mixed=True, tol=3e-10)
    c.pop("name")
    return c


# ---------------------------------------------------------------- inputs

def _stack(plies):
    base = (0, 90, 45, -45, 0, 90)
    return base[:plies // 2]


def _laminate(case, seed):
    """The case's laminate; stack, misalignment and loads from the seed where the family has them."""
    rng = np.random.default_rng(seed)
    if case["family"] == "plate":
        lam = inputs.flat_random(rng, case["n"], case["plies"], float(rng.uniform(2, 12)),
                                 nsub=(case["px"], case["py"], 1), nev=case["nev"], ply_t=0.5, size=10.0)
        lam.traction = [(inputs.FACE_SP, tuple(rng.uniform(-1, 1, 3)))]
        return lam
    nx = case["n_arc"] + 2 * case["n_limb"]
    lam = inputs.curved_corner(n_arc=case["n_arc"], n_limb=case["n_limb"], n_width=case["n_width"],
                               nel_layer=case["nel"], angles=_stack(case["plies"]), width=0.5 * case["n_width"] + 2.0,
                               limb_L=10.0, limb_bias=3.0, amp_deg=float(rng.uniform(4, 12)),
                               wrinkle_w=float(rng.uniform(1.5, 4)), delta=float(rng.uniform(-2e-3, -5e-4)),
                               nsub=(min(case["px"], nx), case["py"], 1), nev=case["nev"])
    lam.element = case["element"]
    lam.periodic_width = int(case["periodic"])
    return lam


def _plates(case, seed):
    rng = np.random.default_rng(seed)
    return [inputs.flat_random(rng, int(n), int(plies), float(rng.uniform(0, 12)), nsub=(0, 0, 1), nev=case["nev"],
                               ply_t=0.5, size=10.0) for n, plies in (v.split("x") for v in case["sizes"].split(","))]


def _load(lam, seed):
    """A smooth random pressure and shear on the outer face, as nodal forces (N)."""
    rng = np.random.default_rng(seed + 17)
    NX, NY, NZ = lam.node_dims
    x, y = np.meshgrid(np.linspace(0, 1, NX), np.linspace(0, 1, NY))
    f = np.zeros((NZ, NY, NX, 3))
    for c in range(3):
        for _ in range(3):
            a, kx, ky, ph = rng.normal(), rng.integers(0, 4), rng.integers(0, 3), rng.uniform(0, 2 * math.pi)
            f[-1, :, :, c] += a * np.cos(math.pi * (kx * x + ky * y) + ph) / (NX * NY)
    return torch.from_numpy(f.reshape(-1)).to(DEV)


def _field(lam, seed):
    """A displacement of the size and smoothness a solve returns, with a little roughness (N)."""
    g = torch.Generator(device=DEV).manual_seed(int(seed))
    X, _ = _nodes(lam)
    a = torch.randn(3, 3, generator=g, device=DEV, dtype=torch.float64) * 1e-3
    b = torch.randn(3, 3, generator=g, device=DEV, dtype=torch.float64) * 1e-3
    u = X @ a + torch.sin(0.3 * X) @ b
    return (u + 1e-6 * torch.randn(u.shape, generator=g, device=DEV, dtype=torch.float64)).reshape(-1).contiguous()


def _options(case):
    return dict(nev=case["nev"], tol=case["tol"], precision=lib.GL_PREC_MIXED if case["mixed"] else lib.GL_PREC_FP64)


def _new(n):
    return torch.empty(n, dtype=torch.float64, device=DEV)


def _theta(lam, seed):
    th = torch.from_numpy(np.asarray(lam.theta).reshape(-1)).to(DEV)
    g = torch.Generator(device=DEV).manual_seed(int(seed) + 5)
    return th + 0.01 * torch.randn(th.shape, generator=g, device=DEV, dtype=torch.float64)


def prepare(case, seed):
    kind = case["kind"]
    st = dict(case=case)
    if kind == "batch1":
        st["lams"] = _plates(case, seed)
        return st
    if kind == "batch":
        lams = _plates(case, seed)
        st["batch"] = lib.Batch(lams)
        st["batch"].setup(**_options(case))
        st["out"] = [_new(lam.n_dof) for lam in lams]
        return st
    lam = st["lam"] = _laminate(case, seed)
    if kind == "first":
        return st
    st["solver"] = lib.Solver.from_laminate(lam, **_options(case))
    if kind == "solve":
        st["f"] = _load(lam, seed)
    elif kind == "gradient":
        st["theta"] = _theta(lam, seed).requires_grad_(True)
        st["mask"] = torch.from_numpy(inputs.arc_resin_mask(lam)).to(DEV)
    else:
        st["x"] = _field(lam, seed)
    return st


# ---------------------------------------------------------------- one pass

def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "first":
        lam = st["lam"]
        s = lib.Solver.from_laminate(lam, **_options(case))
        u, s33, t13 = _new(lam.n_dof), _new(lam.n_elem), _new(lam.n_elem)
        s.solve(out=u)
        s.stress(u, s33, t13)
        s.close()
        return dict(u=u, s33=s33, t13=t13)
    if kind == "batch1":
        lams = st["lams"]
        b = lib.Batch(lams)
        b.setup(**_options(case))
        out, _ = b.solve([_new(lam.n_dof) for lam in lams])
        b.close()
        return out
    if kind == "batch":
        return st["batch"].solve(st["out"])[0]
    s, lam = st["solver"], st["lam"]
    if kind == "solve":
        return s.solve(st["f"], out=_new(lam.n_dof))[0]
    if kind == "gradient":
        s33 = stress_of_theta(st["theta"], s)
        J = pnorm(s33, st["mask"], P_NORM)
        return dict(J=J.detach(), s33=s33.detach(), grad=torch.autograd.grad(J, st["theta"])[0])
    if kind == "ku":
        return s.apply_K(st["x"], out=_new(lam.n_dof))
    s33, t13, F = _new(lam.n_elem), _new(lam.n_elem), _new(lam.n_elem)
    _, _, peak = s.stress(st["x"], s33, t13)
    _, peak_f, elem = s.failure_index(st["x"], F=F)
    return dict(s33=s33, t13=t13, peak_s33=peak, F=F, peak_F=peak_f, elem=elem)


# ---------------------------------------------------------------- the least work of a pass

def _sizes(case):
    """(DOFs, elements) of the case's laminates."""
    if case["family"] == "plates":
        every = [_sizes(dict(family="plate", n=int(n), plies=int(p)))
                 for n, p in (v.split("x") for v in case["sizes"].split(","))]
        return sum(v[0] for v in every), sum(v[1] for v in every)
    if case["family"] == "plate":
        nx = ny = case["n"]
        nz = 2 * case["plies"] - 1
    else:
        nx, ny = case["n_arc"] + 2 * case["n_limb"], case["n_width"]
        nz = case["nel"] * (4 * (case["plies"] // 2) - 1)
    return 3.0 * (2 * nx + 1) * (2 * ny + 1) * (2 * nz + 1), float(nx * ny * nz)


def work(case):
    """Counted per DOF and element.  A K u is 10,854 flop and 2,448 bytes of element data per element; a
    preconditioner application reads the factors of the overlapping subdomains twice (about 650 entries per
    DOF, two flops each); a solve takes about 60 of each.  Set-up factors the subdomains' Dirichlet and
    Neumann matrices (about 0.4 and 0.8 Mflop per DOF) and solves with the latter for a few times nev vectors."""
    N, E = _sizes(case)
    kind = case["kind"]
    entry = 4 if case["mixed"] else 8
    ku_b, ku_f = 2448.0 * E + 16 * N, 10854.0 * E
    if kind == "ku":
        return dict(bytes=ku_b, flops=ku_f)
    if kind == "post":
        return dict(bytes=2 * (16 * N + 300 * E) + 24 * E, flops=2 * 700.0 * E)
    it = 60.0
    solve_b = it * (ku_b + 2 * 650.0 * N * entry + 80 * N)
    solve_f = it * (ku_f + 4 * 650.0 * N + 12 * N)
    if kind in ("solve", "batch"):
        return dict(bytes=solve_b, flops=solve_f)
    if kind == "gradient":
        return dict(bytes=2 * solve_b + ku_b, flops=2 * solve_f + 2 * ku_f)
    m = 4.0 * case["nev"]
    setup_b = 650.0 * N * (entry + 1.6 * 8) + m * 2 * 1.6 * 650.0 * N * 8 / max(m, 1.0) + 8 * 1.6 * N * m
    setup_f = 1.2e6 * N + m * (4 * 1.6 * 650.0 * N + 1.5 * ku_f)
    return dict(bytes=solve_b + setup_b, flops=solve_f + setup_f)


# ---------------------------------------------------------------- plain FP64 reference

# Gauss rule and 1D quadratic basis on {-1, 0, 1}
_G = np.array([-math.sqrt(0.6), 0.0, math.sqrt(0.6)])
_W = np.array([5.0, 8.0, 5.0]) / 9.0


def _basis(x):
    n = np.stack([0.5 * x * (x - 1), 1 - x * x, 0.5 * x * (x + 1)], -1)
    d = np.stack([x - 0.5, -2 * x, x + 0.5], -1)
    return n, d


def _grads(pts):
    """Reference gradients (points, 27, 3) of the 27 shape functions, node i + 3j + 9k."""
    n, d = zip(*[_basis(pts[:, a]) for a in range(3)])
    out = [np.einsum("qi,qj,qk->qkji", *(d[b] if a == b else n[b] for b in range(3))).reshape(len(pts), 27) for a in range(3)]
    return torch.from_numpy(np.stack(out, -1)).to(DEV)


def _gauss():
    z, y, x = np.meshgrid(_G, _G, _G, indexing="ij")
    wz, wy, wx = np.meshgrid(_W, _W, _W, indexing="ij")
    return np.stack([x.ravel(), y.ravel(), z.ravel()], -1), torch.from_numpy((wx * wy * wz).ravel()).to(DEV)


def _serendipity():
    """27 x 27: node values of the 20-node element's field from its own nodes."""
    ijk = [(a % 3, a // 3 % 3, a // 9) for a in range(27)]
    P = np.eye(27)
    for a, p in enumerate(ijk):
        odd = [v == 1 for v in p]
        if sum(odd) < 2:
            continue
        P[a] = 0.0
        for b, r in enumerate(ijk):
            if all(o or u == v for o, u, v in zip(odd, p, r)):
                mids = sum(v == 1 for o, v in zip(odd, r) if o)
                if sum(v == 1 for v in r) == mids == 0:
                    P[a, b] = -0.25
                elif mids == 1 and sum(v == 1 for v in r) == 1:
                    P[a, b] = 0.5 if sum(odd) == 2 else 0.25
    return torch.from_numpy(P).to(DEV)


def _conn(lam):
    NX, NY, _ = lam.node_dims
    ez, ey, ex = np.meshgrid(np.arange(lam.nz), np.arange(lam.ny), np.arange(lam.nx), indexing="ij")
    first = (2 * ex + NX * (2 * ey + NY * 2 * ez)).reshape(-1, 1)
    k, j, i = np.meshgrid(np.arange(3), np.arange(3), np.arange(3), indexing="ij")
    return torch.from_numpy(first + (i + NX * (j + NY * k)).reshape(1, -1)).to(DEV)


def _nodes(lam):
    """Node coordinates (nodes, 3), and the frame angle psi of each element column."""
    def mid(v):
        v = np.asarray(v, dtype=np.float64)
        o = np.empty(2 * len(v) - 1)
        o[0::2], o[1::2] = v, 0.5 * (v[:-1] + v[1:])
        return o
    r, l, t = np.meshgrid(mid(lam.rv()), mid(lam.lv), mid(lam.sv), indexing="ij")
    if lam.node_dr is not None:
        r = r + lam.node_dr
    arc = math.radians(lam.arc_deg)
    tc = 0.5 * (lam.sv[:-1] + lam.sv[1:])
    if lam.geometry == 0:
        X, psi = np.stack([t, l, r], -1), np.zeros(lam.nx)
    else:
        p = np.clip(t, 0, 1) * arc
        ext = np.where(t < 0, t, np.where(t > 1, t - 1, 0.0)) * lam.limb_L
        R = lam.R_inner + r
        X = np.stack([lam.limb_L + R * np.sin(p) + ext * np.cos(p), l, R * np.cos(p) - ext * np.sin(p)], -1)
        psi = np.clip(tc, 0, 1) * arc
    X = torch.from_numpy(X.reshape(-1, 3)).to(DEV)
    if lam.element == 1:
        conn = _conn(lam)
        X = X.index_put((conn.reshape(-1),), torch.einsum("ab,ebc->eac", _serendipity(), X[conn]).reshape(-1, 3))
    return X, torch.from_numpy(np.tile(psi, lam.ny * lam.nz)).to(DEV)


_VOIGT = [(0, 0), (1, 1), (2, 2), (1, 2), (0, 2), (0, 1)]


def _tensors(lam, theta, psi):
    """C_ijkl (elements, 3, 3, 3, 3) in the global axes."""
    base = []
    for m in lam.materials:
        S = np.zeros((6, 6))
        if m["kind"] == "iso":
            m = dict(E1=m["E"], E2=m["E"], E3=m["E"], nu12=m["nu"], nu13=m["nu"], nu23=m["nu"],
                     **{g: m["E"] / (2 + 2 * m["nu"]) for g in ("G12", "G13", "G23")})
        S[0, 0], S[1, 1], S[2, 2] = 1 / m["E1"], 1 / m["E2"], 1 / m["E3"]
        S[0, 1] = S[1, 0] = -m["nu12"] / m["E1"]
        S[0, 2] = S[2, 0] = -m["nu13"] / m["E1"]
        S[1, 2] = S[2, 1] = -m["nu23"] / m["E2"]
        S[3, 3], S[4, 4], S[5, 5] = 1 / m["G23"], 1 / m["G13"], 1 / m["G12"]
        Cv = np.linalg.inv(S)
        T = np.zeros((3, 3, 3, 3))
        for a, (i, j) in enumerate(_VOIGT):
            for b, (k, l) in enumerate(_VOIGT):
                T[i, j, k, l] = T[j, i, k, l] = T[i, j, l, k] = T[j, i, l, k] = Cv[a, b]
        base.append(T)
    per = lam.nx * lam.ny
    layer = np.repeat(lam.elem_layer(), per)
    T = torch.from_numpy(np.stack(base)).to(DEV)[torch.from_numpy(np.asarray(lam.layer_mat)[layer]).to(DEV)]
    phi = torch.from_numpy(np.radians(np.asarray(lam.layer_angle_deg))[layer]).to(DEV)
    zero, one = torch.zeros_like(phi), torch.ones_like(phi)
    a = psi + theta
    Ry = torch.stack([a.cos(), zero, a.sin(), zero, one, zero, -a.sin(), zero, a.cos()], -1).reshape(-1, 3, 3)
    Rz = torch.stack([phi.cos(), -phi.sin(), zero, phi.sin(), phi.cos(), zero, zero, zero, one], -1).reshape(-1, 3, 3)
    R = Ry @ Rz
    for _ in range(4):   # rotates the first index and moves it to the end
        T = torch.einsum("eia,eabcd->ebcdi", R, T)
    return T


class _Reference:
    """The laminate's stiffness in plain torch: products, stresses and a direct solve."""

    def __init__(self, lam, theta=None):
        self.lam = lam
        self.conn = _conn(lam)
        self.X, self.psi = _nodes(lam)
        pts, self.w = _gauss()
        self.ref = _grads(pts)
        self.ref0 = _grads(np.zeros((1, 3)))
        self.theta = (torch.zeros(lam.n_elem, dtype=torch.float64, device=DEV) if lam.theta is None else
                      torch.from_numpy(np.asarray(lam.theta).reshape(-1)).to(DEV)) if theta is None else theta
        self.C = _tensors(lam, self.theta, self.psi)
        NX, NY, _ = lam.node_dims
        node = np.arange(lam.n_nodes)
        ix, iy, iz = node % NX, node // NX % NY, node // (NX * NY)
        _, owner = np.unique(self.conn.cpu().numpy().reshape(-1), return_index=True)
        self.owner = torch.from_numpy(owner).to(DEV)   # one (element, node) entry of every node
        keep = np.ones(lam.n_nodes, dtype=bool)
        if lam.element == 1:
            keep = (ix % 2 + iy % 2 + iz % 2) < 2
        image = node
        if lam.periodic_width:
            image = np.where(iy == NY - 1, node - NX * (NY - 1), node)
            keep = keep & (image == node)
        self.image = torch.from_numpy(image).to(DEV)
        free = np.repeat(keep, 3)
        free[np.asarray(lam.dir_dof)] = False
        self.free = torch.from_numpy(free).to(DEV)

    def phys(self, ref, e):
        """Physical gradients (e, q, 27, 3) and Jacobian determinants."""
        J = torch.einsum("eac,qad->eqcd", self.X[self.conn[e]], ref)
        return torch.einsum("qad,eqdc->eqac", ref, torch.linalg.inv(J)), torch.linalg.det(J)

    def chunks(self, per=4096):
        for k in range(0, self.lam.n_elem, per):
            yield torch.arange(k, min(k + per, self.lam.n_elem), device=DEV)

    def forces(self, C, ue, e):
        """Element forces (e, 27, 3) of element displacements."""
        g, det = self.phys(self.ref, e)
        H = torch.einsum("eac,eqad->eqcd", ue, g)
        s = torch.einsum("eijkl,eqkl->eqij", C, H) * (det * self.w)[..., None, None]
        return torch.einsum("eqij,eqaj->eai", s, g)

    def fill(self, u):
        """The values that the constraints give to the constrained nodes."""
        u = u.reshape(-1, 3)[self.image]
        if self.lam.element == 1:
            ue = torch.einsum("ab,ebc->eac", _serendipity(), u[self.conn]).reshape(-1, 3)
            u = ue[self.owner]
        return u.reshape(-1)

    def fold(self, y):
        """The transpose of fill()."""
        x = torch.zeros_like(y, requires_grad=True)
        return torch.autograd.grad(self.fill(x), x, y)[0]

    def mul(self, x):
        y, x = torch.zeros_like(x).reshape(-1, 3), x.reshape(-1, 3)
        for e in self.chunks():
            y.index_add_(0, self.conn[e].reshape(-1), self.forces(self.C[e], x[self.conn[e]], e).reshape(-1, 3))
        return y.reshape(-1)

    def local_stress(self, u, C=None):
        """(elements, 3, 3) centre stresses in the (s, l, r) frame."""
        C, u, out = self.C if C is None else C, u.reshape(-1, 3), []
        for e in self.chunks():
            g, _ = self.phys(self.ref0, e)
            H = torch.einsum("eac,ead->ecd", u[self.conn[e]], g[:, 0])
            S = torch.einsum("eijkl,ekl->eij", C[e], H)
            a = self.psi[e]
            z, o = torch.zeros_like(a), torch.ones_like(a)
            R = torch.stack([a.cos(), z, a.sin(), z, o, z, -a.sin(), z, a.cos()], -1).reshape(-1, 3, 3)
            out.append(torch.einsum("eia,eij,ejb->eab", R, S, R))
        return torch.cat(out)

    def traction(self):
        """Consistent loads of the x-end tractions of a flat plate (Simpson weights: faces are rectangles)."""
        lam = self.lam
        NX, NY, NZ = lam.node_dims
        f = torch.zeros(NZ, NY, NX, 3, dtype=torch.float64, device=DEV)

        def weights(v):
            w = np.zeros(2 * len(v) - 1)
            for k, h in enumerate(np.diff(v)):
                w[2 * k:2 * k + 3] += h * np.array([1, 4, 1]) / 6
            return torch.from_numpy(w).to(DEV)
        area = weights(lam.rv())[:, None] * weights(lam.lv)[None, :]
        for face, t in lam.traction:
            assert face == inputs.FACE_SP and lam.geometry == 0
            f[:, :, -1] += area[..., None] * torch.tensor(t, dtype=torch.float64, device=DEV)
        return f.reshape(-1)

    # -- direct solve: node planes of constant x are dense blocks; the planes between two element faces are
    #    eliminated first, then the chain of face planes
    def cost(self):
        _, NY, NZ = self.lam.node_dims
        return 14.0 * (3 * NY * NZ) ** 3 * self.lam.nx

    def column(self, ex):
        """Dense 3b x 3b stiffness of element column ex over its three node planes, constrained rows out."""
        lam = self.lam
        NX, NY, NZ = lam.node_dims
        b = 3 * NY * NZ
        e = torch.arange(ex, lam.n_elem, lam.nx, device=DEV)
        g, det = self.phys(self.ref, e)
        Ke = 0.0
        for q in range(27):
            CB = torch.einsum("eijkl,eal->eijak", self.C[e], g[:, q])
            Ke = Ke + torch.einsum("ebj,eijak->ebiak", g[:, q], CB) * (det[:, q] * self.w[q])[:, None, None, None, None]
        if lam.element == 1:
            P = _serendipity()
            Ke = torch.einsum("bd,ebiak,ac->edick", P, Ke, P)
        Ke = Ke.reshape(-1, 81, 81)
        n = self.image[self.conn[e]]
        plane = n % NX - 2 * ex
        at = (plane * (NY * NZ) + n // NX)[..., None] * 3 + torch.arange(3, device=DEV)
        dof = (n[..., None] * 3 + torch.arange(3, device=DEV)).reshape(-1, 81)
        on = self.free[dof].to(torch.float64)
        Ke = Ke * on[:, :, None] * on[:, None, :]
        at = at.reshape(-1, 81)
        A = torch.zeros(9 * b * b, dtype=torch.float64, device=DEV)
        A.index_add_(0, (at[:, :, None] * (3 * b) + at[:, None, :]).reshape(-1), Ke.reshape(-1))
        return A.reshape(3 * b, 3 * b)

    def factor(self):
        lam = self.lam
        NX, NY, NZ = lam.node_dims
        b = 3 * NY * NZ
        fixed = (~self.free).to(torch.float64).reshape(NZ, NY, NX, 3).permute(2, 0, 1, 3).reshape(NX, b)
        self.steps, D = [], torch.diag(fixed[0])
        for ex in range(lam.nx):
            A = self.column(ex)
            Lm = torch.linalg.cholesky(A[b:2 * b, b:2 * b] + torch.diag(fixed[2 * ex + 1]))
            W = torch.linalg.solve_triangular(Lm, torch.cat([A[b:2 * b, :b], A[b:2 * b, 2 * b:]], 1), upper=False)
            D = D + A[:b, :b] - W[:, :b].T @ W[:, :b]
            Ld = torch.linalg.cholesky(D)
            V = torch.linalg.solve_triangular(Ld, A[:b, 2 * b:] - W[:, :b].T @ W[:, b:], upper=False)
            D = torch.diag(fixed[2 * ex + 2]) + A[2 * b:, 2 * b:] - W[:, b:].T @ W[:, b:] - V.T @ V
            self.steps.append((Lm, W, Ld, V))
        self.last = torch.linalg.cholesky(D)

    def back(self, r):
        """K_ff^{-1} r by the factor."""
        NX, NY, NZ = self.lam.node_dims
        b = 3 * NY * NZ
        r = (r * self.free).reshape(NZ, NY, NX, 3).permute(2, 0, 1, 3).reshape(NX, b, 1).clone()

        def low(L, v):
            return torch.linalg.solve_triangular(L, v, upper=False)

        def up(L, v):
            return torch.linalg.solve_triangular(L.T, v, upper=True)
        for ex, (Lm, W, Ld, V) in enumerate(self.steps):
            r[2 * ex + 1] = low(Lm, r[2 * ex + 1])
            r[2 * ex] -= W[:, :b].T @ r[2 * ex + 1]
            r[2 * ex + 2] -= W[:, b:].T @ r[2 * ex + 1]
            r[2 * ex] = low(Ld, r[2 * ex])
            r[2 * ex + 2] -= V.T @ r[2 * ex]
        r[NX - 1] = up(self.last, low(self.last, r[NX - 1]))
        for ex in range(self.lam.nx - 1, -1, -1):
            Lm, W, Ld, V = self.steps[ex]
            r[2 * ex] = up(Ld, r[2 * ex] - V @ r[2 * ex + 2])
            r[2 * ex + 1] = up(Lm, r[2 * ex + 1] - W @ torch.cat([r[2 * ex], r[2 * ex + 2]]))
        return r.reshape(NX, NZ, NY, 3).permute(1, 2, 0, 3).reshape(-1) * self.free

    def solve(self, f, prescribed=True):
        """K u = f with the prescribed values (or zero), refined twice with the matrix-free residual."""
        ud = torch.zeros(self.lam.n_dof, dtype=torch.float64, device=DEV)
        if prescribed:
            ud[torch.from_numpy(np.asarray(self.lam.dir_dof)).to(DEV)] = torch.from_numpy(np.asarray(self.lam.dir_val)).to(DEV)
            ud = torch.where(self.kept(), ud, torch.zeros_like(ud))
        u = torch.zeros_like(ud)
        for _ in range(3):
            u = u + self.back(f - self.fold(self.mul(self.fill(u + ud))))
        return self.fill(u + ud)

    def kept(self):
        """DOFs that are no constraint's: free or prescribed."""
        node = torch.arange(self.lam.n_nodes, device=DEV)
        NX, NY, _ = self.lam.node_dims
        keep = self.image == node
        if self.lam.element == 1:
            keep = keep & ((node % NX % 2 + node // NX % NY % 2 + node // (NX * NY) % 2) < 2)
        return keep.repeat_interleave(3)


MOST_FLOPS = 9e12   # of one direct solve: about ten seconds


def exact(case, seed):
    kind = case["kind"]
    if kind in ("batch1", "batch"):
        refs = [_Reference(lam) for lam in _plates(case, seed)]
        if sum(r.cost() for r in refs) > MOST_FLOPS:
            return None
        out = []
        for r in refs:
            r.factor()
            out.append(r.solve(r.traction()))
            r.steps = None
        return out
    lam = _laminate(case, seed)
    if kind == "ku":
        return _Reference(lam).mul(_field(lam, seed))
    if kind == "post":
        r = _Reference(lam)
        S = r.local_stress(_field(lam, seed))
        resin = torch.from_numpy(inputs.resin_elements(lam)).to(DEV)
        F = torch.sqrt((S[:, 2, 2].clamp(min=0) / 61.0) ** 2 + (S[:, 0, 2] / 97.0) ** 2 + (S[:, 1, 2] / 97.0) ** 2) * resin
        return dict(s33=S[:, 2, 2].contiguous(), t13=S[:, 0, 2].contiguous(), peak_s33=float(S[resin, 2, 2].max()), F=F,
                    peak_F=float(F.max()), elem=None)
    r = _Reference(lam, _theta(lam, seed) if kind == "gradient" else None)
    if r.cost() > MOST_FLOPS:
        return None
    r.factor()
    if kind == "solve":
        return r.solve(_load(lam, seed))
    u = r.solve(r.traction())
    if kind == "first":
        S = r.local_stress(u)
        return dict(u=u, s33=S[:, 2, 2].contiguous(), t13=S[:, 0, 2].contiguous())
    # dJ/dtheta = dJ/dtheta at fixed u - lambda^T dK/dtheta u, K lambda = dJ/du
    mask = torch.from_numpy(inputs.arc_resin_mask(lam)).to(DEV)
    theta, v = r.theta.clone().requires_grad_(True), u.clone().requires_grad_(True)
    s33 = r.local_stress(v, _tensors(lam, theta, r.psi))[:, 2, 2]
    J = (s33[mask] ** P_NORM).sum() ** (1.0 / P_NORM)
    grad, dJdu = torch.autograd.grad(J, (theta, v))
    lm = r.solve(dJdu, prescribed=False).reshape(-1, 3)
    for e in r.chunks(1024):
        th = r.theta.clone().requires_grad_(True)
        fe = r.forces(_tensors(lam, th, r.psi)[e], u.reshape(-1, 3)[r.conn[e]], e)
        grad = grad - torch.autograd.grad((lm[r.conn[e]] * fe).sum(), th)[0]
    return dict(J=J.detach(), s33=s33.detach(), grad=grad)
