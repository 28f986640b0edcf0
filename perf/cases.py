"""The work that users of the eMG solver have it do, as cases that can be timed and compared.

A case names one call of the public interface (the Python classes of the package, or the C ABI
through its ctypes binding where a call takes device pointers), a mesh, an order and a precision
form.  The meshes are the O-grids around a cylinder and the cubed-sphere shells that the
framework's configurations and tests use, the states are smooth compressible flow around the
body with seeded perturbations on every mode: a solve part of the way to its steady state, as
most of a solve's cycles see it (each cycle then moves the state by a few parts in 10^4; over a
solve to a 1e-10 drop that falls from 1e-2 to rounding).  `Reference` restates the method in plain float64 torch.
"""
import ctypes
import math

import numpy as np
import torch

import paper_1807_01151_gb300 as emg
from paper_1807_01151_gb300 import perfmodel
from workloads import BC_FARFIELD, cubed_sphere_shell, ogrid

GAMMA, MACH = 1.4, 0.3
AMP = 1e-4               # perturbation of every mode, relative to the free stream
STAGES, KRYLOV, SMOOTH, CFL_MAX = 4, 30, 2, 100.0
CYCLE = 40               # index of the V-cycle that the cycle cases run (the CFL ramp's place)
CFL = 20.0               # of the PRK and EXP1 steps that are called alone
FP64, FP32_BLOCKS, BF16_BLOCKS = 0, 1, 2


def listed():
    return [
        # one residual of the smallest O-grid at the lowest smoothed order: latency and launches
        dict(name="residual_32x16_p1", op="residual", dim=2, n1=32, n2=16, p=1, prec=FP64),
        # the residual of the headline case (residual throughput, 614,400 unknowns)
        dict(name="residual_128x64_p4", op="residual", dim=2, n1=128, n2=64, p=4, prec=FP64),
        # the highest order in 3-D on a sphere shell of odd size
        dict(name="residual_sphere7x11_p4", op="residual", dim=3, n1=7, n2=11, p=4, prec=FP64),
        # one smoothing step (block build, factorisation, four stages) in float64, odd sizes
        dict(name="prk_45x21_p3_fp64", op="prk", dim=2, n1=45, n2=21, p=3, prec=FP64),
        # the same with float32 blocks at the headline size, and in 3-D
        dict(name="prk_128x64_p4_fp32", op="prk", dim=2, n1=128, n2=64, p=4, prec=FP32_BLOCKS),
        dict(name="prk_sphere8x12_p3_fp32", op="prk", dim=3, n1=8, n2=12, p=3, prec=FP32_BLOCKS),
        # the coarse exponential step of the headline case alone
        dict(name="exp1_128x64_fp32", op="exp1", dim=2, n1=128, n2=64, p=0, prec=FP32_BLOCKS),
        # whole V-cycles: the small all-float64 cylinder; the headline case in both forms; the sphere
        dict(name="vcycle_32x16_p2_fp64", op="vcycle", dim=2, n1=32, n2=16, p=2, prec=FP64),
        dict(name="vcycle_128x64_p4_fp64", op="vcycle", dim=2, n1=128, n2=64, p=4, prec=FP64),
        dict(name="vcycle_128x64_p4_fp32", op="vcycle", dim=2, n1=128, n2=64, p=4, prec=FP32_BLOCKS),
        dict(name="vcycle_sphere16x24_p3_fp32", op="vcycle", dim=3, n1=16, n2=24, p=3, prec=FP32_BLOCKS),
        # the request loop: six solves that arrive together, four at a time
        dict(name="serve_6_fp64", op="serve", requests="32x16p1 32x16p2 64x32p1 32x16p3 64x32p2 48x24p2", active=4,
             drop=0.1, prec=FP64),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more call: smoothing steps and residuals oftenest, as in a cycle; both dimensions, every
    order and precision form, sizes over the whole range of the configurations."""
    op = rng.choice(["residual", "residual", "prk", "prk", "vcycle", "vcycle", "exp1"])
    prec = rng.choice([FP64, FP32_BLOCKS, FP32_BLOCKS, BF16_BLOCKS]) if op in ("prk", "vcycle") else rng.choice([FP64, FP32_BLOCKS])
    if rng.random() < 0.65:
        p = 0 if op == "exp1" else rng.randint(1, 4)
        n1 = _log_int(rng, 24, 256 if p < 4 or op == "residual" else 128)
        n2 = max(8, min(128, round(n1 * rng.uniform(0.35, 0.6))))
        return dict(op=op, dim=2, n1=n1, n2=n2, p=p, prec=prec)
    p = 0 if op == "exp1" else rng.randint(1, 4)
    small = op in ("prk", "vcycle") and prec == FP64
    n1 = _log_int(rng, 3, (6 if p <= 3 else 4) if small else 12 if p <= 3 else 7)
    n2 = max(4, min(18 if p <= 3 else 10, round(n1 * rng.uniform(0.8, 1.6))))
    return dict(op=op, dim=3, n1=n1, n2=n2, p=p, prec=prec)


def _mesh(case):
    return ogrid(case["n1"], case["n2"]) if case["dim"] == 2 else cubed_sphere_shell(case["n1"], case["n2"])


def _requests(case):
    out = []
    for word in case["requests"].split():
        grid, p = word.split("p")
        n1, n2 = grid.split("x")
        out.append((int(n1), int(n2), int(p)))
    return out


def _counts(case):
    e = case["n1"] * case["n2"] if case["dim"] == 2 else 6 * case["n1"] ** 2 * case["n2"]
    f = 2 * e + case["n1"] if case["dim"] == 2 else 3 * e + 6 * case["n1"] ** 2
    return e, f


def work(case):
    """The method's own operations, and the call's arrays read and written once."""
    if case["op"] == "serve":
        total = {"bytes": 0.0, "flops": 0.0}
        for n1, n2, p in _requests(case):   # a handful of cycles each
            one = work(dict(op="vcycle", dim=2, n1=n1, n2=n2, p=p, prec=case["prec"]))
            total = {k: total[k] + 5 * one[k] for k in total}
        return total
    e, f = _counts(case)
    s = perfmodel.Shape(case["dim"], case["p"], e, f)
    residual = perfmodel.residual_face_flops(s) + perfmodel.residual_volume_flops(s)
    if case["op"] == "residual":
        return {"bytes": perfmodel.residual_bytes(s), "flops": residual}
    if case["op"] == "prk":
        factor = perfmodel.lu_flops(s) if case["prec"] == FP64 else perfmodel.inverse_flops(s)
        return {"bytes": perfmodel.residual_bytes(s),
                "flops": STAGES * (residual + perfmodel.stage_flops(s)) + perfmodel.diag_flops(s) + factor}
    w = perfmodel.vcycle_work(case["dim"], case["p"], e, f, STAGES, SMOOTH, KRYLOV, min(case["prec"], 1))
    if case["op"] == "exp1":
        return {"bytes": e * (5 * 3 + 1) * 8.0, "flops": w["arnoldi"][0] + residual}
    return {"bytes": perfmodel.residual_bytes(s), "flops": sum(v[0] for v in w.values())}


# ---- inputs ------------------------------------------------------------------------------------

def _flow(x):
    """Conservative variables of isentropic potential flow around the body of radius 1/2."""
    r2 = (x * x).sum(-1)
    v = torch.zeros(x.shape[:-1] + (3,), dtype=x.dtype, device=x.device)
    if x.shape[-1] == 2:
        a = 0.25 / (r2 * r2)
        v[..., 0] = MACH * (1 - a * (x[..., 0] ** 2 - x[..., 1] ** 2))
        v[..., 1] = -MACH * 2 * a * x[..., 0] * x[..., 1]
    else:
        a = 0.5 * 0.125 / (r2 * r2 * r2.sqrt())
        v[..., 0] = MACH * (1 + a * (r2 - 3 * x[..., 0] ** 2))
        for k in (1, 2):
            v[..., k] = -3 * MACH * a * x[..., 0] * x[..., k]
    c2 = 1 + 0.5 * (GAMMA - 1) * (MACH ** 2 - (v * v).sum(-1))
    rho = c2 ** (1 / (GAMMA - 1))
    e = rho * c2 / GAMMA / (GAMMA - 1) + 0.5 * rho * (v * v).sum(-1)
    return torch.cat([rho[..., None], rho[..., None] * v, e[..., None]], -1)


def _inputs(case, seed):
    """(mesh, reference geometry, state [E][5][N], FAS forcing at p = 0, EXP1 steps)."""
    mesh = _mesh(case)
    ref = Reference(mesh, case["p"])
    g = torch.Generator(ref.dev).manual_seed(int(seed))
    n = ref.modes(case["p"])
    u = ref.project(_flow)
    scale = torch.tensor([1.0, MACH, MACH, MACH if case["dim"] == 3 else 0.0, 1 / GAMMA / (GAMMA - 1)], dtype=torch.float64,
                         device=ref.dev)
    xi = torch.randn((ref.E, 5, n), generator=g, dtype=torch.float64, device=ref.dev)
    deg = torch.tensor(_exponents(case["dim"], case["p"]).sum(1), dtype=torch.float64, device=ref.dev)
    u += AMP * scale[None, :, None] * xi / (1 + deg) ** 2 * ref.vol.sqrt()[:, None, None]
    return mesh, ref, u.contiguous(), g


class _State:
    pass


def prepare(case, seed):
    s = _State()
    s.case = case
    if case["op"] == "serve":   # host meshes and a Mach number for each request, as they come in
        rng = np.random.default_rng(int(seed))
        s.requests = [(ogrid(n1, n2), p, float(rng.uniform(0.15, 0.3))) for n1, n2, p in _requests(case)]
        return s
    mesh, ref, s.u, g = _inputs(case, seed)
    s.solver = emg.Solver(mesh, p_max=case["p"], mach=MACH, prec=case["prec"])
    s.out = torch.empty_like(s.u)
    if case["op"] == "exp1":
        s.tau, s.dt = _exp1_extra(ref, s.u, g)
    return s


def _exp1_extra(ref, u, g):
    tau = AMP * ref.vol[:, None, None] ** 0.5 * torch.randn(u.shape, generator=g, dtype=torch.float64, device=ref.dev)
    if ref.d == 2:
        tau[:, 3] = 0.0
    return tau.contiguous(), (5 * ref.dtau(0, u, CFL) / 9).contiguous()


def _ptr(t):
    return ctypes.c_void_p(t.data_ptr())


def _check(solver, status):
    if status != 0:
        raise emg.EmgError(status, solver.lib.emg_last_error(solver.h).decode())


def run(s):
    case = s.case
    if case["op"] == "residual":
        return s.solver.residual(case["p"], s.u, s.out)
    if case["op"] == "prk":
        _check(s.solver, s.solver.lib.emg_prk_step(s.solver.h, case["p"], _ptr(s.u), None, CFL, _ptr(s.out), 1))
        return s.out
    if case["op"] == "exp1":
        k = ctypes.c_int32()
        _check(s.solver, s.solver.lib.emg_exp1_step(s.solver.h, _ptr(s.u), _ptr(s.tau), _ptr(s.dt), _ptr(s.out),
                                                    ctypes.byref(k), 1))
        return {"u": s.out, "krylov_dim": k.value}
    if case["op"] == "vcycle":
        s.solver.set_state(s.u)
        s.solver.set_cycle(CYCLE)
        info = s.solver.vcycle()
        s.solver.get_state(s.out)
        return {"u": s.out, "res": np.array(info["res"]), "cfl": info["cfl"], "krylov_dim": info["krylov_dim"]}
    server = emg.Server(max_active=case["active"], drop=case["drop"], max_cycles=200, keep_state=True)
    try:
        ids = [server.submit(mesh, p_max=p, mach=mach, prec=case["prec"]) for mesh, p, mach in s.requests]
        done = {}
        while len(done) < len(ids):
            server.step()
            done.update({r["id"]: r for r in server.results()})
        return {"states": [server.take_state(i) for i in ids], "cycles": np.array([done[i]["cycles"] for i in ids]),
                "res": np.array([done[i]["res_final"] for i in ids])}
    finally:
        server.close()


def exact(case, seed):
    if case["op"] == "serve" or _counts(case)[0] * (case["p"] + 1) ** 4 > 6e6 and case["op"] != "residual":
        return None
    _, ref, u, g = _inputs(case, seed)
    if case["op"] == "residual":
        return ref.residual(case["p"], u)
    if case["op"] == "prk":
        return ref.prk_step(case["p"], u, 0.0, CFL)
    if case["op"] == "exp1":
        tau, dt = _exp1_extra(ref, u, g)
        out, k = ref.exp1_step(u, tau, dt)
        return {"u": out, "krylov_dim": k}
    return ref.vcycle(u)


# ---- the method in plain float64 ----------------------------------------------------------------

def _exponents(d, p):
    """Monomials by total degree, within a degree the x exponent descending, then y."""
    if d == 2:
        return np.array([(a, k - a) for k in range(p + 1) for a in range(k, -1, -1)])
    return np.array([(a, b, k - a - b) for k in range(p + 1) for a in range(k, -1, -1) for b in range(k - a, -1, -1)])


def _pressure(U):
    return (GAMMA - 1) * (U[..., 4] - 0.5 * (U[..., 1:4] ** 2).sum(-1) / U[..., 0])


def _flux(U):
    """F[..., k, a]."""
    p = _pressure(U)
    v = U[..., 1:4] / U[..., :1]
    F = v[..., :, None] * U[..., None, :]
    pad = torch.zeros_like(U[..., :1])
    eye = torch.eye(3, dtype=U.dtype, device=U.device)
    pe = p[..., None, None] * torch.cat([torch.zeros_like(eye[:, :1]), eye, torch.zeros_like(eye[:, :1])], 1)
    pv = torch.cat([pad[..., None, :].expand(v.shape + (1,))] * 4 + [(p[..., None] * v)[..., None]], -1)
    return F + pe + pv


def _flux_n(U, n):
    return (_flux(U) * n[..., :, None]).sum(-2)


def _roe(UL, UR, n):
    vL, vR = UL[..., 1:4] / UL[..., :1], UR[..., 1:4] / UR[..., :1]
    pL, pR = _pressure(UL), _pressure(UR)
    sL, sR = UL[..., 0].sqrt(), UR[..., 0].sqrt()
    den = sL + sR
    u = (sL[..., None] * vL + sR[..., None] * vR) / den[..., None]
    H = (sL * (UL[..., 4] + pL) / UL[..., 0] + sR * (UR[..., 4] + pR) / UR[..., 0]) / den
    rho = sL * sR
    q2 = (u * u).sum(-1)
    c2 = (GAMMA - 1) * (H - 0.5 * q2)
    c = c2.sqrt()
    qn = (u * n).sum(-1)
    dr, dp, dv = UR[..., 0] - UL[..., 0], pR - pL, vR - vL
    dq = (dv * n).sum(-1)
    w1 = (qn - c).abs() * (dp - rho * c * dq) / (2 * c2)
    w5 = (qn + c).abs() * (dp + rho * c * dq) / (2 * c2)
    w2, ws = qn.abs() * (dr - dp / c2), qn.abs() * rho
    dt = dv - dq[..., None] * n
    mom = (w1[..., None] * (u - c[..., None] * n) + w2[..., None] * u + ws[..., None] * dt
           + w5[..., None] * (u + c[..., None] * n))
    en = w1 * (H - c * qn) + w2 * 0.5 * q2 + ws * (u * dt).sum(-1) + w5 * (H + c * qn)
    diss = torch.cat([(w1 + w2 + w5)[..., None], mom, en[..., None]], -1)
    return 0.5 * (_flux_n(UL, n) + _flux_n(UR, n) - diss)


def _wall(U, n):
    m = U[..., 1:4]
    m = m - 2 * (m * n).sum(-1, keepdim=True) * n
    return torch.cat([U[..., :1], m, U[..., 4:]], -1)


def _farfield(U, n):
    """Riemann invariants normal to the face, entropy and tangential velocity from the upwind side."""
    vi = torch.tensor([MACH, 0.0, 0.0], dtype=U.dtype, device=U.device)
    v, p = U[..., 1:4] / U[..., :1], _pressure(U)
    c = (GAMMA * p / U[..., 0]).sqrt()
    qi, q = (n * vi).sum(-1), (n * v).sum(-1)
    plus, minus = q + 2 * c / (GAMMA - 1), qi - 2 / (GAMMA - 1)
    qb, cb = 0.5 * (plus + minus), 0.25 * (GAMMA - 1) * (plus - minus)
    s = torch.where(qb < 0, torch.full_like(p, 1 / GAMMA), p / U[..., 0] ** GAMMA)
    vb = torch.where((qb < 0)[..., None], vi + (qb - qi)[..., None] * n, v + (qb - q)[..., None] * n)
    rb = (cb * cb / (GAMMA * s)) ** (1 / (GAMMA - 1))
    pb = rb * cb * cb / GAMMA
    e = pb / (GAMMA - 1) + 0.5 * rb * (vb * vb).sum(-1)
    return torch.cat([rb[..., None], rb[..., None] * vb, e[..., None]], -1)


def _jacobian(f, *U):
    """[df/dU for each U] of a pointwise map of states, by one-hot directions in forward mode."""
    out = []
    for k in range(len(U)):
        cols = []
        for b in range(5):
            t = [torch.zeros_like(x) for x in U]
            t[k][..., b] = 1.0
            cols.append(torch.func.jvp(f, tuple(U), tuple(t))[1])
        out.append(torch.stack(cols, -1))
    return out


class _Level:
    pass


class Reference:
    """Geometry, orthonormal modal basis, residual, smoother, EXP1 step and V-cycle in float64 torch."""

    def __init__(self, mesh, p_max):
        self.dev = "cuda" if torch.cuda.is_available() else "cpu"
        self.d, self.p_max, self.E = mesh.dim, p_max, mesh.n_elems
        self.mesh = mesh
        d = self.d
        quad = [(-1, -1), (1, -1), (1, 1), (-1, 1)]
        self.corner = np.array(quad if d == 2 else [q + (-1,) for q in quad] + [q + (1,) for q in quad], dtype=float)
        self.X = self._t(mesh.xyz.T)[torch.as_tensor(mesh.elem_nodes, device=self.dev)]          # [E][A][d]
        x, _, W = self._volume(p_max + 2)
        self.vol = W.sum(1)
        self.xc = (W[..., None] * x).sum(1) / self.vol[:, None]
        self.half = 0.5 * (self.X.amax(1) - self.X.amin(1))
        self.C = None
        chi = self._monomials(x, slice(None), p_max)[0]
        C = torch.zeros((self.E, chi.shape[2], chi.shape[2]), dtype=torch.float64, device=self.dev)
        psi = torch.zeros_like(chi)
        for i in range(chi.shape[2]):   # modified Gram-Schmidt on the quadrature inner product
            v, c = chi[:, :, i].clone(), torch.zeros_like(C[:, i])
            c[:, i] = 1
            for j in range(i):
                r = (W * v * psi[:, :, j]).sum(1, keepdim=True)
                v -= r * psi[:, :, j]
                c -= r * C[:, j]
            s = (W * v * v).sum(1, keepdim=True).sqrt()
            psi[:, :, i], C[:, i] = v / s, c / s
        self.C, self._psi, self._W, self._x = C, psi, W, x
        surf = sum(self._face_points(torch.arange(self.E, device=self.dev), f, p_max + 2)[1].norm(dim=-1).sum(1)
                   for f in range(2 * d))
        self.h = 2 * d * self.vol / surf
        self.levels = {}

    def _t(self, a):
        return torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device=self.dev)

    def modes(self, p):
        return len(_exponents(self.d, p))

    def project(self, field):
        return torch.einsum("eq,eqi,eqa->eai", self._W, self._psi, field(self._x))

    def _shape(self, xi):
        fac = 0.5 * (1 + xi[:, None, :] * self.corner)
        dN = np.stack([0.5 * self.corner[:, k] * np.prod(np.delete(fac, k, 2), 2) for k in range(self.d)], -1)
        return self._t(np.prod(fac, 2)), self._t(dN)

    def _volume(self, q):
        x, w = np.polynomial.legendre.leggauss(q)
        xi = np.stack(np.meshgrid(*[x] * self.d, indexing="ij"), -1).reshape(-1, self.d)
        wt = np.prod(np.stack(np.meshgrid(*[w] * self.d, indexing="ij"), -1).reshape(-1, self.d), 1)
        N, dN = self._shape(xi)
        J = torch.einsum("pak,eai->epik", dN, self.X)
        return torch.einsum("pa,eai->epi", N, self.X), J, self._cofactor(J)[1] * self._t(wt)

    def _cofactor(self, J):
        """cof(J) = det(J) J^-T and det J."""
        if self.d == 2:
            c = torch.stack([torch.stack([J[..., 1, 1], -J[..., 1, 0]], -1), torch.stack([-J[..., 0, 1], J[..., 0, 0]], -1)], -2)
        else:
            c = torch.stack([torch.cross(J[..., (k + 1) % 3], J[..., (k + 2) % 3], dim=-1) for k in range(3)], -1)
        return c, (c[..., 0] * J[..., 0]).sum(-1)

    def _face_points(self, elems, f, q, normals=None):
        axis, side = f // 2, 2.0 * (f % 2) - 1
        x, w = np.polynomial.legendre.leggauss(q)
        sub = np.stack(np.meshgrid(*[x] * (self.d - 1), indexing="ij"), -1).reshape(-1, self.d - 1)
        wt = np.prod(np.stack(np.meshgrid(*[w] * (self.d - 1), indexing="ij"), -1).reshape(-1, self.d - 1), 1)
        N, dN = self._shape(np.insert(sub, axis, side, 1))
        X = self.X[elems]
        J = torch.einsum("pak,eai->epik", dN, X)
        a = torch.zeros((len(elems), len(wt), 3), dtype=torch.float64, device=self.dev)
        a[..., : self.d] = side * self._cofactor(J)[0][..., axis] * self._t(wt)[:, None]
        pts = torch.einsum("pa,eai->epi", N, X)
        return pts, a, None if normals is None else torch.einsum("pa,eai->epi", N, normals[elems])

    def _monomials(self, x, elems, p):
        s = (x - self.xc[elems, None]) / self.half[elems, None]
        chi, grad = [], []
        for ex in _exponents(self.d, p):
            pw = [s[..., k] ** int(ex[k]) for k in range(self.d)]
            chi.append(math.prod(pw))
            g = []
            for k in range(self.d):
                dk = int(ex[k]) * s[..., k] ** max(int(ex[k]) - 1, 0) / self.half[elems, None, k]
                g.append(math.prod([dk] + pw[:k] + pw[k + 1:]))
            grad.append(torch.stack(g, -1))
        return torch.stack(chi, 2), torch.stack(grad, 2)

    def _basis(self, x, elems, p, grad=False):
        n = self.modes(p)
        chi, g = self._monomials(x, elems, p)
        C = self.C[elems][:, :n, :n]
        return torch.einsum("eik,epk->epi", C, chi), torch.einsum("eik,epkd->epid", C, g) if grad else None

    def level(self, p):
        if p in self.levels:
            return self.levels[p]
        L, q, d = _Level(), p + 2, self.d
        x, _, W = self._volume(q)
        L.psi, g = self._basis(x, slice(None), p, True)
        L.wgrad = W[..., None, None] * g
        nodes, bc = self.mesh.elem_nodes, self.mesh.face_bc
        key, own = [], []
        for f in range(2 * d):
            on = [a for a in range(2 ** d) if self.corner[a, f // 2] == 2 * (f % 2) - 1]
            e = np.nonzero(bc[:, f] < 0)[0]
            key.append(np.sort(nodes[np.ix_(e, on)], 1))
            own.append(np.stack([e, np.full_like(e, f)], 1))
        key, own = np.concatenate(key), np.concatenate(own)
        order = np.lexsort(key.T)
        left, right = own[order[0::2]], own[order[1::2]]
        assert (key[order[0::2]] == key[order[1::2]]).all()
        L.faces = []
        wn = None if self.mesh.wall_normal is None else self._t(self.mesh.wall_normal.T)[
            torch.as_tensor(nodes, device=self.dev)]
        for f in range(2 * d):
            sel = left[:, 1] == f
            if sel.any():
                el, er = (torch.as_tensor(s[sel, 0], device=self.dev) for s in (left, right))
                xf, a, _ = self._face_points(el, f, q)
                m = a.norm(dim=-1, keepdim=True)
                L.faces.append((0, el, er, m, a / m, self._basis(xf, el, p)[0], self._basis(xf, er, p)[0]))
            for code in np.unique(bc[:, f][bc[:, f] >= 0]):
                el = torch.as_tensor(np.nonzero(bc[:, f] == code)[0], device=self.dev)
                xf, a, nw = self._face_points(el, f, q, wn)
                m = a.norm(dim=-1, keepdim=True)
                body = torch.zeros_like(a)
                body[..., :d] = nw / nw.norm(dim=-1, keepdim=True).clamp_min(1e-300)
                L.faces.append((int(code), el, body, m, a / m, self._basis(xf, el, p)[0], None))
        self.levels[p] = L
        return L

    @staticmethod
    def _boundary(code, U, n, body):
        return _roe(U, _farfield(U, n) if code == BC_FARFIELD else _wall(U, body), n)

    def residual(self, p, u):
        L = self.level(p)
        F = _flux(torch.einsum("eai,eqi->eqa", u, L.psi))[..., : self.d, :]
        R = torch.einsum("eqik,eqka->eai", L.wgrad, F)
        for code, el, er, m, n, psiL, psiR in L.faces:
            UL = torch.einsum("fai,fqi->fqa", u[el], psiL)
            if code == 0:
                Fh = m * _roe(UL, torch.einsum("fai,fqi->fqa", u[er], psiR), n)
                R = R.index_add(0, er, torch.einsum("fqi,fqa->fai", psiR, Fh))
            else:
                Fh = m * self._boundary(code, UL, n, er)
            R = R.index_add(0, el, -torch.einsum("fqi,fqa->fai", psiL, Fh))
        return R

    def dtau(self, p, u, cfl):
        psi = self._basis(self.xc[:, None], slice(None), p)[0][:, 0]
        U = torch.einsum("eai,ei->ea", u, psi)
        c = (GAMMA * _pressure(U) / U[:, 0]).sqrt()
        return cfl * self.h / ((2 * p + 1) * (U[:, 1:4].norm(dim=1) / U[:, 0] + c))

    def blocks(self, p, u):
        """dR_e/du_e, [E][5N][5N]."""
        L, n = self.level(p), self.modes(p)
        D = torch.zeros((self.E, 5, n, 5, n), dtype=torch.float64, device=self.dev)
        for e0 in range(0, self.E, 2048):
            s = slice(e0, min(self.E, e0 + 2048))
            A = _jacobian(_flux, torch.einsum("eai,eqi->eqa", u[s], L.psi[s]))[0][..., : self.d, :, :]
            G = torch.einsum("eqik,eqkab->eqiab", L.wgrad[s], A)
            D[s] += torch.einsum("eqiab,eqj->eaibj", G, L.psi[s])
        for code, el, er, m, nrm, psiL, psiR in L.faces:
            UL = torch.einsum("fai,fqi->fqa", u[el], psiL)
            if code == 0:
                UR = torch.einsum("fai,fqi->fqa", u[er], psiR)
                JL, JR = _jacobian(lambda a, b: _roe(a, b, nrm), UL, UR)
                D.index_add_(0, er, torch.einsum("fqi,fqab,fqj->faibj", psiR, m[..., None] * JR, psiR))
            else:
                JL, = _jacobian(lambda a: self._boundary(code, a, nrm, er), UL)
            D.index_add_(0, el, -torch.einsum("fqi,fqab,fqj->faibj", psiL, m[..., None] * JL, psiL))
        return D.reshape(self.E, 5 * n, 5 * n)

    def prk_step(self, p, u, tau, cfl):
        b = 5 * self.modes(p)
        P = -self.blocks(p, u) + torch.eye(b, dtype=torch.float64, device=self.dev) / self.dtau(p, u, cfl)[:, None, None]
        lu, piv = torch.linalg.lu_factor(P)
        v = u
        for k in range(STAGES):
            r = (self.residual(p, v) + tau).reshape(self.E, b, 1)
            v = u + torch.linalg.lu_solve(lu, piv, r).reshape(u.shape) / (STAGES - k)
        return v

    def exp1_step(self, u, tau, dt):
        shape, dt = u.shape, dt[:, None, None]
        b = (dt * (self.residual(0, u) + tau)).reshape(-1)
        V = torch.zeros((KRYLOV + 1, b.numel()), dtype=torch.float64, device=self.dev)
        H = torch.zeros((KRYLOV + 1, KRYLOV + 1), dtype=torch.float64, device=self.dev)
        beta = b.norm()
        V[0] = b / beta
        for j in range(KRYLOV):
            x = V[j].reshape(shape)
            w = (dt * torch.func.jvp(lambda a: self.residual(0, a), (u,), (x,))[1]).reshape(-1)
            for _ in range(2):
                h = V[: j + 1] @ w
                w = w - h @ V[: j + 1]
                H[: j + 1, j] += h
            H[j + 1, j] = w.norm()
            V[j + 1] = w / H[j + 1, j]
        aug = torch.zeros_like(H)
        aug[:KRYLOV, :KRYLOV] = H[:KRYLOV, :KRYLOV]
        aug[0, KRYLOV] = 1
        y = beta * torch.linalg.matrix_exp(aug)[:KRYLOV, KRYLOV]
        return u + (y @ V[:KRYLOV]).reshape(shape), KRYLOV

    def vcycle(self, u):
        P = self.p_max
        R = self.residual(P, u)
        res = (R * R).sum((0, 2)).sqrt() / self.vol.sum()
        cfl = min(CFL_MAX, 1 + (CYCLE - 1) / (2 * P + 1))
        dt = (P + 1) * self.dtau(P, u, cfl)
        v, v0, tau = {P: u}, {}, {P: 0.0}
        for p in range(P, 0, -1):
            for _ in range(SMOOTH):
                v[p] = self.prk_step(p, v[p], tau[p], cfl)
            n = self.modes(p - 1)
            v0[p - 1] = v[p - 1] = v[p][:, :, :n].clone()
            tau[p - 1] = (self.residual(p, v[p]) + tau[p])[:, :, :n] - self.residual(p - 1, v0[p - 1])
        if P == 0:
            v0[0] = u
        v[0], k = self.exp1_step(v0[0], tau[0], dt)
        for p in range(1, P + 1):
            v[p] = v[p].clone()
            v[p][:, :, : self.modes(p - 1)] += v[p - 1] - v0[p - 1]
        return {"u": v[P], "res": res, "cfl": float(cfl), "krylov_dim": k}
