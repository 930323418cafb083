"""Performance cases: the calls a user of the solver makes, over the sizes, degrees and options they
make them with, and a plain FP64 torch evaluation of the same operator to compare the results with.

Every case names one public call of paper_2306_12891_gb300.dg.DG (or its autograd binding), the
polynomial degree N, the mesh and the physics. Inputs are a box mesh (Cartesian or curved by an
analytic map; for the channel with walls in z) and a base flow plus a smooth perturbation whose
phases and amplitudes come from the seed.

  rhs          Ut = L(U), what a caller with its own time integrator asks for
  step, steps  LSERK(5,4) steps in place, from the state the program kept (a restart)
  host_step    one step on a page-locked host array, the transfer both ways included
  vjp          cotangent of U through one right-hand side
  gradient     d(kinetic energy after K steps)/dU0 through autograd
  diagnostics  time step estimate, blending coefficient and integral invariants of a state
"""
import math

import numpy as np
import torch
import torch.utils.checkpoint

from paper_2306_12891_gb300 import autograd, dg
from paper_2306_12891_gb300 import workloads as W

GAMMA, PR = 1.4, 0.72
MACH = {"tgv": 0.1, "blast": 1.0, "channel": 0.3}


def _case(name, call, N, nel, flow="tgv", equations="ns", vflux="pirozzoli", sflux="roe", precision="fp64",
          curved=True, count=1):
    c = dict(call=call, N=N, nx=nel[0], ny=nel[1], nz=nel[2], flow=flow, equations=equations, vflux=vflux, sflux=sflux,
             precision=precision, curved=curved, count=count)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest configured workload: one right-hand side of 4096 nodes, where the call itself counts
        _case("rhs_euler_n3_4x4x4", "rhs", 3, (4, 4, 4), equations="euler", vflux="kg", sflux="llf", curved=False),
        # the long-run accuracy configuration (N = 7, 4^3): many cheap steps, launch-bound
        _case("steps_ns_n7_4x4x4", "steps", 7, (4, 4, 4), count=10),
        # the headline physics (Taylor-Green, Navier-Stokes, N = 7, curved), a mesh that fills the GPU many times
        _case("step_ns_n7_24x24x24", "step", 7, (24, 24, 24)),
        # the same physics in the FP32-bulk precision form
        _case("step_fp32_n7_24x24x24", "step", 7, (24, 24, 24), precision="fp32_bulk"),
        # FP32-bulk at a lower degree on an odd, ragged mesh, inside a caller's own integrator
        _case("rhs_fp32_n5_17x13x11", "rhs", 5, (17, 13, 11), precision="fp32_bulk"),
        # shocked flow: blast wave with the indicator and the DG/FV blend
        _case("step_blast_n5_32x32x32", "step", 5, (32, 32, 32), flow="blast", equations="euler", sflux="llf",
              curved=False),
        # wall-modelled channel: wall faces, Spalding Newton solves, ordinary size
        _case("step_channel_n5_24x12x12", "step", 5, (24, 12, 12), flow="channel", curved=False),
        # entropy-conservative fluxes (robust under-resolved Euler) at an even degree, odd element counts
        _case("rhs_ec_n4_23x19x17", "rhs", 4, (23, 19, 17), equations="euler", vflux="ec", sflux="ec"),
        # a solver coupled to host code: the state lives in pinned host memory
        _case("host_step_ns_n7_16x16x16", "host_step", 7, (16, 16, 16)),
        # one vector-Jacobian product at a low degree (adjoint inside a caller's own integrator)
        _case("vjp_euler_n3_21x18x15", "vjp", 3, (21, 18, 15), equations="euler", vflux="kg"),
        # gradient of the kinetic energy through steps (the differentiation form's physics), N = 5
        _case("gradient_ns_n5_12x12x12", "gradient", 5, (12, 12, 12), count=2),
        # what a time loop asks every few steps: dt, blending coefficient, integral invariants
        _case("diagnostics_n5_24x24x24", "diagnostics", 5, (24, 24, 24)),
    ]


def draw(rng):
    call = rng.choice(["rhs", "rhs", "step", "step", "steps", "host_step", "vjp", "gradient", "diagnostics"])
    N = rng.randint(1, 7)
    adjoint = call in ("vjp", "gradient")
    flow = "tgv" if adjoint or call == "host_step" else rng.choice(["tgv", "tgv", "tgv", "blast", "channel"])
    precision = "fp32_bulk" if flow == "tgv" and not adjoint and rng.random() < 0.3 else "fp64"
    top = {"rhs": 4e6, "step": 2e6, "steps": 3e4, "host_step": 1e6, "vjp": 1e6, "gradient": 1.5e5, "diagnostics": 3e6}
    nodes = math.exp(rng.uniform(math.log(3e3), math.log(top[call])))
    base = max(1.0, (nodes / (N + 1) ** 3) ** (1 / 3))
    nel = tuple(max(1, round(base * rng.uniform(0.7, 1.3))) for _ in range(3))
    if flow == "blast":
        eq, vf, sf = "euler", rng.choice(["pirozzoli", "kg"]), rng.choice(["llf", "roe"])
    else:
        eq = "ns" if flow == "channel" else rng.choice(["euler", "ns", "ns"])
        vf = rng.choice(["pirozzoli", "kg"] if adjoint or flow == "channel" else ["pirozzoli", "pirozzoli", "kg", "ec"])
        sf = "ec" if vf == "ec" else rng.choice(["llf", "roe"])
    return _case(None, call, N, nel, flow, eq, vf, sf, precision, flow == "tgv" and rng.random() < 0.7,
                 {"steps": 10, "gradient": 2}.get(call, 1))


# ------------------------------------------------------------------ inputs

def _physics(case):
    p = dict(equations=case["equations"], vflux=case["vflux"], sflux=case["sflux"], gamma=GAMMA, R=1.0, Pr=PR, mu=0.0)
    if case["equations"] == "ns":
        p["mu"] = 1e-5 if case["flow"] == "channel" else 1.0 / W.RE_TGV
    if case["flow"] == "blast":
        p["shock_capturing"] = True
    if case["flow"] == "channel":
        p.update(wm_index=1, wm_uinf=1.0, wm_mainf=0.3, wm_van_driest=True)
    if case["precision"] == "fp32_bulk":  # the mean pressure, as the precision form wants it
        p.update(precision="fp32_bulk", p_ref=1.0 / (GAMMA * MACH[case["flow"]] ** 2))
    return p


def _inputs(case, seed):
    """Host mesh (xyz, faces), device state U0 and step size of a case."""
    N, nel, flow = case["N"], (case["nx"], case["ny"], case["nz"]), case["flow"]
    hi = {"tgv": (W.TWO_PI,) * 3, "blast": (1.0,) * 3, "channel": (W.TWO_PI, math.pi, 2.0)}[flow]
    xyz, faces = W.box_mesh(N, nel, (0.0, 0.0, 0.0), hi, None, z_walls=flow == "channel")
    X = torch.from_numpy(xyz).cuda()
    if case["curved"]:
        X = X + 0.05 * (torch.sin(X[:, 0]) * torch.sin(X[:, 1]) * torch.sin(X[:, 2])).unsqueeze(1)
        xyz = X.cpu().numpy()
    x, y, z = X[:, 0], X[:, 1], X[:, 2]
    rng = np.random.default_rng(seed)

    def smooth(amp):  # three of the lowest Fourier modes of the box
        f = torch.zeros_like(x)
        for _ in range(3):
            k = [int(rng.integers(-2, 3)) * W.TWO_PI / h for h in hi]
            f += float(rng.uniform(-1, 1)) * torch.sin(k[0] * x + k[1] * y + k[2] * z + float(rng.uniform(0, W.TWO_PI)))
        return amp * f

    one = torch.ones_like(x)
    if flow == "tgv":
        p0 = 1.0 / (GAMMA * MACH["tgv"] ** 2)
        rho, w = one + smooth(0.01), smooth(0.01)
        u = torch.sin(x) * torch.cos(y) * torch.cos(z) + smooth(0.01)
        v = -torch.cos(x) * torch.sin(y) * torch.cos(z) + smooth(0.01)
        p = p0 + (torch.cos(2 * x) + torch.cos(2 * y)) * (torch.cos(2 * z) + 2.0) / 16.0 + smooth(0.01)
    elif flow == "blast":  # hot sphere, 1 % noise in the density
        r = torch.sqrt((x - 0.5) ** 2 + (y - 0.5) ** 2 + (z - 0.5) ** 2)
        gen = torch.Generator(device="cuda").manual_seed(int(seed))
        rho = 1.0 + 0.01 * (2.0 * torch.rand(x.shape, generator=gen, dtype=x.dtype, device=x.device) - 1.0)
        u, v, w = smooth(0.01), smooth(0.01), smooth(0.01)
        p = 1.0 + 99.0 * 0.5 * (1.0 - torch.tanh((r - 0.3) / 0.02))
    else:  # turbulent-like mean profile between the walls
        zr = torch.minimum(z, 2.0 - z)
        bump = torch.sin(0.5 * math.pi * z)
        u = torch.clamp(zr * (2.0 - zr), 0.0, 1.0) ** (1.0 / 7.0) + smooth(0.05) * bump
        v, w = smooth(0.05) * bump, smooth(0.05) * bump
        rho, p = one, one / (GAMMA * MACH["channel"] ** 2)
    E = p / (GAMMA - 1.0) + 0.5 * rho * (u * u + v * v + w * w)
    U0 = torch.stack([rho, rho * u, rho * v, rho * w, E], dim=1).contiguous()
    speed = float((torch.sqrt(u * u + v * v + w * w) + torch.sqrt(GAMMA * p / rho)).max())
    dt = 0.5 * 2.0 / ((2 * N + 1) * speed * sum(2.0 * m / (h * 0.9) for m, h in zip(nel, hi)))
    return xyz, faces, U0, dt


def _cotangent(U0, seed):
    """A smooth-free, O(1) cotangent: what an arbitrary loss hands back."""
    gen = torch.Generator(device="cuda").manual_seed(int(seed) + 1)
    return torch.randn(U0.shape, generator=gen, dtype=U0.dtype, device=U0.device)


def prepare(case, seed):
    xyz, faces, U0, dt = _inputs(case, seed)
    st = dict(case=case, solver=dg.DG(case["N"], xyz, faces, **_physics(case)), U0=U0, dt=dt)
    call = case["call"]
    if call in ("step", "steps"):
        st["U"] = U0.clone()
    elif call in ("rhs", "vjp"):
        st["out"] = torch.empty_like(U0)
        if call == "vjp":
            st["lam"] = _cotangent(U0, seed)
    elif call == "host_step":
        st["Uh"] = U0.cpu().pin_memory()
    elif call == "diagnostics":
        st["Ut"] = _cotangent(U0, seed)
        st["alpha"] = torch.empty(U0.shape[0], dtype=U0.dtype, device=U0.device)
    return st


def run(st):
    case, s = st["case"], st["solver"]
    call = case["call"]
    if call == "rhs":
        return s.rhs(st["U0"], st["out"])
    if call in ("step", "steps"):
        st["U"].copy_(st["U0"])
        return s.lserk_step(st["U"], st["dt"]) if call == "step" else s.lserk_steps(st["U"], st["dt"], case["count"])
    if call == "host_step":  # the flow goes on from pass to pass, as in the coupled program
        return s.lserk_step_host(st["Uh"], st["dt"])
    if call == "vjp":
        return s.rhs_vjp(st["U0"], st["lam"], st["out"])
    if call == "gradient":
        U0 = st["U0"].detach().requires_grad_(True)
        ke = autograd.kinetic_energy(s, autograd.lserk_steps(s, U0, st["dt"], case["count"]))
        ke.backward()
        return {"ke": ke.detach(), "grad": U0.grad}
    return {"dt": s.max_dt(st["U0"], 0.9), "alpha": s.indicator(st["U0"], st["alpha"]),
            "invariants": s.invariants(st["U0"], st["Ut"])}


def work(case):
    """Bytes: state, register and metric terms once per right-hand side. Flops: the two-point fluxes (each pair
    once), the derivative sums and the pointwise parts of the formulas."""
    n = case["N"] + 1
    dofs = case["nx"] * case["ny"] * case["nz"] * n ** 3
    ns, call = case["equations"] == "ns", case["call"]
    word = 4 if case["precision"] == "fp32_bulk" else 8
    pair = {"kg": 42, "pirozzoli": 40, "ec": 95}[case["vflux"]]
    flops = 1.5 * (n - 1) * pair + 3 * 200 / n + 60
    if ns:
        flops += 2 * n * 12 + 150 + 2 * n * 12
    if case["flow"] == "blast":
        flops += 60 + 6 * n
    rhs_bytes = 80 + 10 * word
    stages = {"step": 5, "steps": 5 * case["count"], "host_step": 5, "gradient": 15 * case["count"], "vjp": 3}.get(call, 1)
    if call == "diagnostics":
        return {"bytes": dofs * (2 * 40 + 80 + 40), "flops": dofs * 150}
    nbytes = dofs * (rhs_bytes + (80 if stages > 1 and call != "vjp" else 0)) * stages
    return {"bytes": nbytes, "flops": dofs * flops * stages}


def tolerance(case):
    """About four times the largest distance from exact() seen over the listed and 70 drawn cases. A right-hand side
    at Mach 0.1 is the small difference of fluxes of size p0 = 71 / h on terms of the metric, hence its larger figure;
    a stepped state adds dt times that to an O(1) state."""
    call, fp32 = case["call"], case["precision"] == "fp32_bulk"
    if call == "rhs":
        return {"rel": 1.2e-3 if fp32 else 2.4e-10}
    if call in ("step", "host_step", "steps"):
        rel = 2e-8 if fp32 else 8e-15
        return {"rel": 5 * rel if call == "steps" else rel}
    return {"rel": {"vjp": 4.5e-14, "gradient": 1.6e-14, "diagnostics": 6e-15}[call]}


# ------------------------------------------------------------------ the operator in plain FP64 torch

class _Reference:
    """Split-form DGSEM on LGL nodes: fields are [nE, ..., k, j, i] torch FP64 tensors on the GPU."""

    def __init__(self, case, xyz, faces):
        self.N, self.n = case["N"], case["N"] + 1
        self.ns = case["equations"] == "ns"
        self.vf, self.sf = case["vflux"], case["sflux"]
        self.sc = case["flow"] == "blast"
        p = _physics(case)
        self.mu = p["mu"]
        self.kappa = self.mu * GAMMA / ((GAMMA - 1.0) * PR)
        self.wm = p
        xi, self.w, self.D = self._basis(self.N)
        n = self.n
        self.xi = xi
        self.Dt = self._t(self.D)
        self.Doff = self._t(self.D * (1.0 - np.eye(n)))
        V = np.polynomial.legendre.legvander(xi, self.N) * np.sqrt((2 * np.arange(n) + 1) / 2)
        self.Vinv = self._t(np.linalg.inv(V))
        self._geometry(self._t(xyz))
        self._faces(np.asarray(faces), xyz)

    @staticmethod
    def _t(a):
        return torch.from_numpy(np.ascontiguousarray(np.asarray(a, dtype=np.float64))).cuda()

    @staticmethod
    def _basis(N):
        leg = np.polynomial.legendre
        c = np.zeros(N + 1)
        c[N] = 1.0
        dc = leg.legder(c)
        x = np.sort(np.real(leg.legroots(dc))) if N > 1 else np.zeros(0)
        for _ in range(4):
            x = x - leg.legval(x, dc) / leg.legval(x, leg.legder(dc))
        xi = np.concatenate([[-1.0], x, [1.0]])
        xi = 0.5 * (xi - xi[::-1])
        w = 2.0 / (N * (N + 1) * leg.legval(xi, c) ** 2)
        L = xi.astype(np.longdouble)
        d = L[:, None] - L[None, :] + np.eye(N + 1)
        lam = 1 / d.prod(axis=1)
        D = (lam[None, :] / lam[:, None]) / d
        D[np.diag_indices(N + 1)] = 0
        D[np.diag_indices(N + 1)] = -D.sum(axis=1)
        return xi, w, D.astype(np.float64)

    @staticmethod
    def _apply(M, f, d):
        """M along reference direction d (xi is the last axis)."""
        ax = f.dim() - 1 - d
        return torch.movedim(torch.matmul(torch.movedim(f, ax, -1), M.T), -1, ax)

    def _geometry(self, X):
        X = X - X[:, :, :1, :1, :1]
        dX = [[self._apply(self.Dt, X[:, c], d) for d in range(3)] for c in range(3)]
        Ja = []
        for i in range(3):
            j, k = (i + 1) % 3, (i + 2) % 3
            row = []
            for c in range(3):
                m, l = (c + 1) % 3, (c + 2) % 3
                row.append(self._apply(self.Dt, X[:, l] * dX[m][j], k) - self._apply(self.Dt, X[:, l] * dX[m][k], j))
            Ja.append(torch.stack(row, 1))
        self.Ja = torch.stack(Ja, 1)  # [nE, 3 d, 3 c, k, j, i]
        a = dX
        self.J = (a[0][0] * (a[1][1] * a[2][2] - a[1][2] * a[2][1]) - a[0][1] * (a[1][0] * a[2][2] - a[1][2] * a[2][0])
                  + a[0][2] * (a[1][0] * a[2][1] - a[1][1] * a[2][0]))

    def _faces(self, faces, xyz):
        N, n = self.N, self.n
        q, p = np.meshgrid(np.arange(n), np.arange(n), indexing="ij")  # face point p + n q

        def node(f, pp, qq, depth=0):
            b = N - depth if f % 2 else depth
            return [b + n * (pp + n * qq), pp + n * (b + n * qq), pp + n * (qq + n * b)][f // 2]

        nodes = np.stack([node(f, p, q).ravel() for f in range(6)])
        self.own = torch.from_numpy(nodes).cuda()  # [6, nn] volume node of each face point
        nnn, wall = n ** 3, faces[:, 2] < 0
        F, Wf = faces[~wall], faces[wall]
        perm = np.empty((8, n * n), dtype=np.int64)
        for o in range(8):
            a, b = (q, p) if o & 4 else (p, q)
            a = N - a if o & 1 else a
            b = N - b if o & 2 else b
            perm[o] = (a + n * b).ravel()
        inv = np.argsort(perm, axis=1)
        c = lambda v: torch.from_numpy(np.ascontiguousarray(v)).cuda()  # noqa: E731
        idL = F[:, :1].astype(np.int64) * nnn + nodes[F[:, 1]]
        idR = F[:, 2:3].astype(np.int64) * nnn + np.take_along_axis(nodes[F[:, 3]], perm[F[:, 4]], 1)
        self.idL, self.idR, self.back = c(idL), c(idR), c(inv[F[:, 4]])
        self.fL = F[:, 1]
        slot = np.empty(6 * self.J.shape[0], dtype=np.int64)  # row of cat(L, R, walls) that fills each slot
        nF = len(F)
        slot[F[:, 0].astype(np.int64) * 6 + F[:, 1]] = np.arange(nF)
        slot[F[:, 2].astype(np.int64) * 6 + F[:, 3]] = nF + np.arange(nF)
        slot[Wf[:, 0].astype(np.int64) * 6 + Wf[:, 1]] = 2 * nF + np.arange(len(Wf))
        self.slot = c(slot)
        nb = np.full(6 * self.J.shape[0], -1, dtype=np.int64)
        nb[F[:, 0].astype(np.int64) * 6 + F[:, 1]] = F[:, 2]
        nb[F[:, 2].astype(np.int64) * 6 + F[:, 3]] = F[:, 0]
        self.nb = c(nb.reshape(-1, 6))
        self.nrm, self.area = self._normal(c(F[:, 0].astype(np.int64)), F[:, 1], self.idL)
        self.walls = None
        if len(Wf):
            idW = Wf[:, :1].astype(np.int64) * nnn + nodes[Wf[:, 1]]
            deep = np.stack([node(f, p, q, self.wm["wm_index"]).ravel() for f in range(6)])
            idX = Wf[:, :1].astype(np.int64) * nnn + deep[Wf[:, 1]]
            pts = np.moveaxis(xyz.reshape(xyz.shape[0], 3, nnn), 1, 2).reshape(-1, 3)
            h = np.sqrt(((pts[idX] - pts[idW]) ** 2).sum(-1))
            nrm, area = self._normal(c(Wf[:, 0].astype(np.int64)), Wf[:, 1], c(idW))
            self.walls = dict(id=c(idW), idx=c(idX), h=self._t(h), nrm=nrm, area=area)

    def _normal(self, elem, lf, ids):
        J = torch.movedim(self.Ja.flatten(3), 3, 1).reshape(-1, 3, 3)  # [node, d, c]
        d = torch.from_numpy(np.ascontiguousarray(lf // 2)).cuda().long()[:, None].expand_as(ids)
        sg = torch.from_numpy(np.where(lf % 2 == 1, 1.0, -1.0)).cuda()[:, None, None]
        a = sg * J[ids, d]
        s = a.norm(dim=-1)
        return a / s[..., None], s

    # pointwise physics; states have the variables in the last axis
    @staticmethod
    def _prim(U):
        ir = 1.0 / U[..., 0]
        vel = U[..., 1:4] * ir[..., None]
        p = (GAMMA - 1.0) * (U[..., 4] - 0.5 * (U[..., 1:4] * vel).sum(-1))
        return U[..., 0], vel, p

    @staticmethod
    def _logmean(a, b):
        z = a / b
        f = (z - 1.0) / (z + 1.0)
        u = f * f
        near = u < 1e-4
        far = (a - b) / torch.log(torch.where(near, torch.full_like(z, 2.0), z))
        return torch.where(near, (a + b) / (2.0 * (1.0 + u * (1 / 3 + u * (0.2 + u / 7)))), far)

    def _ec(self, rL, vL, pL, rR, vR, pR, a):
        bL, bR = 0.5 * rL / pL, 0.5 * rR / pR
        rl, bl = self._logmean(rL, rR), self._logmean(bL, bR)
        vm = 0.5 * (vL + vR)
        ph = 0.5 * (rL + rR) / (bL + bR)
        F0 = rl * (vm * a).sum(-1)
        mom = F0[..., None] * vm + ph[..., None] * a
        q2 = 0.5 * ((vL * vL).sum(-1) + (vR * vR).sum(-1))
        en = F0 * (0.5 / ((GAMMA - 1.0) * bl) - 0.5 * q2) + (vm * mom).sum(-1)
        return torch.cat([F0[..., None], mom, en[..., None]], -1)

    def _flux(self, U, a):
        r, v, p = self._prim(U)
        un = (v * a).sum(-1, keepdim=True)
        return torch.cat([U[..., :1] * un, U[..., 1:4] * un + p[..., None] * a, (U[..., 4:] + p[..., None]) * un], -1)

    def _riemann(self, UL, UR, n):
        rL, vL, pL = self._prim(UL)
        rR, vR, pR = self._prim(UR)
        if self.sf == "ec":
            return self._ec(rL, vL, pL, rR, vR, pR, n)
        mean = 0.5 * (self._flux(UL, n) + self._flux(UR, n))
        nL, nR = (vL * n).sum(-1), (vR * n).sum(-1)
        if self.sf == "llf":
            lam = torch.maximum(nL.abs() + torch.sqrt(GAMMA * pL / rL), nR.abs() + torch.sqrt(GAMMA * pR / rR))
            return mean - 0.5 * lam[..., None] * (UR - UL)
        sL, sR = torch.sqrt(rL), torch.sqrt(rR)
        mix = lambda a, b: (sL[..., None] * a + sR[..., None] * b) / (sL + sR)[..., None]  # noqa: E731
        vt = mix(vL, vR)
        H = mix(((UL[..., 4] + pL) / rL)[..., None], ((UR[..., 4] + pR) / rR)[..., None])[..., 0]
        q2 = (vt * vt).sum(-1)
        c2 = (GAMMA - 1.0) * (H - 0.5 * q2)
        c, rt, un = torch.sqrt(c2), sL * sR, (vt * n).sum(-1)
        dr, dp, dv = rR - rL, pR - pL, vR - vL
        dn = (dv * n).sum(-1)
        l1, l5, l2 = (un - c).abs() * 0.5 * (dp - rt * c * dn) / c2, (un + c).abs() * 0.5 * (dp + rt * c * dn) / c2, un.abs()
        l2a = l2 * (dr - dp / c2)
        dvt = dv - dn[..., None] * n
        mass = l1 + l5 + l2a
        mom = mass[..., None] * vt + (c * (l5 - l1))[..., None] * n + (l2 * rt)[..., None] * dvt
        en = (l1 + l5) * H + c * (l5 - l1) * un + l2a * 0.5 * q2 + l2 * rt * (vt * dvt).sum(-1)
        return mean - 0.5 * torch.cat([mass[..., None], mom, en[..., None]], -1)

    def _slots(self, left, right, walls):
        """[nE, 6, nn, q] outward values in each slot's own point order from the per-face values."""
        q = left.shape[-1]
        right = torch.gather(right, 1, self.back[..., None].expand(-1, -1, q))
        rows = [left, right] + ([walls] if self.walls else [])
        return torch.cat(rows, 0)[self.slot].reshape(-1, 6, self.n ** 2, q)

    def _surface(self, acc, G):
        """acc [nE, nnn, q] plus (1/w_b) G at the face nodes."""
        for f in range(6):
            acc = acc.index_add(1, self.own[f], G[:, f] / self.w[0])
        return acc

    def _nodes(self, f):  # [nE, q, k, j, i] -> [nE, nnn, q]
        return f.flatten(2).transpose(1, 2)

    def _twopoint(self, L, R):
        a = 0.5 * (L["a"] + R["a"])
        if self.vf == "ec":
            return self._ec(L["r"], L["v"], L["p"], R["r"], R["v"], R["p"], a)
        r, v = 0.5 * (L["r"] + R["r"]), 0.5 * (L["v"] + R["v"])
        V = (v * a).sum(-1)
        pm, em = 0.5 * (L["p"] + R["p"]), 0.5 * (L["e"] + R["e"])
        en = r * V * em + (pm * V if self.vf == "kg" else 0.0)
        return torch.cat([(r * V)[..., None], (r * V)[..., None] * v + pm[..., None] * a, en[..., None]], -1)

    def _alpha(self, U):
        n = self.n
        r, v, p = self._prim(torch.movedim(U, 1, -1))
        m = r * p
        for d in range(3):
            m = self._apply(self.Vinv, m, d)
        k = torch.arange(n, device="cuda")
        M = torch.maximum(torch.maximum(k[:, None, None], k[None, :, None]), k[None, None, :])
        sh = torch.stack([((m * m) * (M == j)).sum((1, 2, 3)) for j in range(n)], 1)
        tot = sh.sum(1)
        E = sh[:, -1] / tot
        if self.N >= 2:
            E = torch.maximum(E, sh[:, -2] / (tot - sh[:, -1]))
        T = 0.5 * 10.0 ** (-1.8 * n ** 0.25)
        al = 1.0 / (1.0 + torch.exp(-dg.DEFAULT_SHARPNESS / T * (E - T)))
        al = torch.where(al < 0.01, torch.zeros_like(al), torch.clamp(al, max=0.7))
        return torch.maximum(al, torch.where(self.nb >= 0, 0.5 * al[self.nb.clamp(min=0)], torch.zeros_like(al)[:, None]).amax(1))

    def _subcells(self, U, G):
        """FV subcell operator [nE, nnn, 5]: minmod in (rho, u, p) inside, first order in the outer subcells."""
        n, N = self.n, self.N
        xh = np.concatenate([[-1.0], -1.0 + np.cumsum(self.w)])
        r, v, p = self._prim(torch.movedim(U, 1, -1))
        q = torch.cat([r[..., None], v, p[..., None]], -1)
        total = 0.0
        for d in range(3):
            ql = torch.movedim(q, 3 - d, 1)  # [nE, n, ., ., 5], the line's index first
            Jl = torch.movedim(torch.movedim(self.Ja[:, d], 1, -1), 3 - d, 1)
            sh = ql.shape
            dif = (ql[:, 1:] - ql[:, :-1]) / self._t(np.diff(self.xi)).view(-1, 1, 1, 1)
            b, f = dif[:, :-1], dif[:, 1:]
            s = torch.zeros_like(ql)
            if N >= 2:
                s[:, 1:-1] = torch.where(b * f <= 0, torch.zeros_like(b), torch.where(b.abs() < f.abs(), b, f))
            lo = ql + s * self._t(xh[:-1] - self.xi).view(-1, 1, 1, 1)
            up = ql + s * self._t(xh[1:] - self.xi).view(-1, 1, 1, 1)
            bad = ((lo[..., 0] <= 0) | (lo[..., 4] <= 0) | (up[..., 0] <= 0) | (up[..., 4] <= 0))[..., None]
            lo, up = torch.where(bad, ql, lo), torch.where(bad, ql, up)
            cons = lambda z: torch.cat([z[..., :1], z[..., :1] * z[..., 1:4], (z[..., 4] / (GAMMA - 1.0)  # noqa: E731
                                        + 0.5 * z[..., 0] * (z[..., 1:4] ** 2).sum(-1))[..., None]], -1)
            dJ = torch.einsum("im,embac->eibac", self.Dt, Jl) * self._t(self.w).view(-1, 1, 1, 1)
            a = Jl[:, :1] + torch.cumsum(dJ, 1)[:, :-1]
            sa = a.norm(dim=-1, keepdim=True)
            mid = sa * self._riemann(cons(up[:, :-1]), cons(lo[:, 1:]), a / sa)
            ends = [G[:, 2 * d + k].reshape(sh[0], 1, n, n, 5) for k in range(2)]
            fl = torch.cat([-ends[0], mid, ends[1]], 1)
            out = (fl[:, 1:] - fl[:, :-1]) / self._t(self.w).view(-1, 1, 1, 1)
            total = total + torch.movedim(out, 1, 3 - d)
        return total.flatten(1, 3)

    def _wall_flux(self, flat):
        """Advective, BR1 jump and wall-model viscous flux at the wall points."""
        Wd = self.walls
        Ui, Ux, n, s = flat[Wd["id"]], flat[Wd["idx"]], Wd["nrm"], Wd["area"]
        mn = (Ui[..., 1:4] * n).sum(-1, keepdim=True)
        Ug = torch.cat([Ui[..., :1], Ui[..., 1:4] - 2.0 * mn * n, Ui[..., 4:]], -1)
        adv = s[..., None] * self._riemann(Ui, Ug, n)
        jump = torch.cat([-mn / Ui[..., :1] * n, torch.zeros_like(mn)], -1)
        r, v, _ = self._prim(Ux)
        ut = v - (v * n).sum(-1, keepdim=True) * n
        speed = ut.norm(dim=-1)
        m = 0.5 * (GAMMA - 1.0) * self.wm["wm_mainf"] ** 2 * PR ** (1 / 3)
        b = math.sqrt(m) / math.sqrt(1.0 + m)
        ue = self.wm["wm_uinf"] / b * torch.asin(b * speed / self.wm["wm_uinf"])
        Re = Wd["h"] * ue * r / self.mu
        up = torch.clamp(torch.sqrt(Re), max=60.0)
        for _ in range(60):
            k = 0.4 * up
            e = torch.exp(k) - 1.0 - k - k * k / 2 - k ** 3 / 6
            y, dy = up + 0.1108 * (e - k ** 4 / 24), 1.0 + 0.1108 * 0.4 * e
            up = up - (up * y - Re) / (y + up * dy)
        tau = r * (ue / up) ** 2
        drag = -(s * tau / speed)[..., None] * ut
        return adv, jump, torch.cat([drag, torch.zeros_like(mn)], -1)

    def rhs(self, U):
        n, w0 = self.n, self.w[0]
        flat = self._nodes(U).reshape(-1, 5)
        UL, UR = flat[self.idL], flat[self.idR]
        adv_w = jump_w = drag_w = None
        if self.walls:
            adv_w, jump_w, drag_w = self._wall_flux(flat)
        Fs = self.area[..., None] * self._riemann(UL, UR, self.nrm)
        G = self._slots(Fs, -Fs, adv_w)
        Un = torch.movedim(U, 1, -1)
        r, v, p = self._prim(Un)
        e = (Un[..., 4] + (p if self.vf == "pirozzoli" else 0.0)) / r
        acc = 0.0
        for d in range(3):
            ax = 3 - d
            f = dict(r=r, v=v, p=p, e=e, a=torch.movedim(self.Ja[:, d], 1, -1))
            at = [{k: x.select(ax, i) for k, x in f.items()} for i in range(n)]
            line = [0.0] * n
            for i in range(n):
                for m in range(i + 1, n):
                    F = self._twopoint(at[i], at[m])
                    line[i] = line[i] + 2.0 * self.D[i, m] * F
                    line[m] = line[m] + 2.0 * self.D[m, i] * F
            acc = acc + torch.stack(line, ax)
        # off the diagonal only: 2 D_bb F(U_b) cancels -F(U_b)/w_b of the strong-form surface term
        acc = self._surface(acc.flatten(1, 3), G)
        if self.sc:
            al = self._alpha(U)[:, None, None]
            acc = al * self._subcells(U, G) + (1.0 - al) * acc
        if self.ns:
            W4 = torch.cat([v, (p / r)[..., None]], -1)  # (u, v, w, T)
            wf = W4.flatten(1, 3).reshape(-1, 4)
            jump = 0.5 * (wf[self.idR] - wf[self.idL])
            S = self._slots(jump, -jump, jump_w)
            ref = [self._nodes(self._apply(self.Dt, torch.movedim(W4, -1, 1), d)) for d in range(3)]
            Jn = torch.movedim(self.Ja.flatten(3), 3, 1)  # [nE, nnn, d, c]
            grad = 0.0
            for d in range(3):
                g = ref[d]
                for k in range(2):
                    g = g.index_add(1, self.own[2 * d + k], (1.0 if k else -1.0) * S[:, 2 * d + k] / w0)
                grad = grad + g[..., :, None] * Jn[:, :, d, None, :]
            grad = grad / self.J.flatten(1)[..., None, None]  # [nE, nnn, 4, c]
            gu, vel = grad[..., :3, :], v.flatten(1, 3)
            div = gu.diagonal(dim1=-2, dim2=-1).sum(-1)
            tau = self.mu * (gu + gu.transpose(-1, -2) - (2.0 / 3.0) * div[..., None, None] * torch.eye(3, dtype=U.dtype, device=U.device))
            Fv = torch.cat([tau, (vel[..., :, None] * tau).sum(-2, keepdim=True) + self.kappa * grad[..., 3:, :]], -2)
            con = [(Fv * Jn[:, :, d, None, :]).sum(-1) for d in range(3)]  # [nE, nnn, 4]
            ff = Fv.reshape(-1, 4, 3)
            nv = self.area[..., None] * (0.5 * (ff[self.idL] + ff[self.idR]) * self.nrm[..., None, :]).sum(-1)
            Gv = self._slots(nv, -nv, drag_w)
            vis = 0.0
            for d in range(3):
                c = con[d].reshape(-1, n, n, n, 4)
                dv = torch.movedim(self._apply(self.Dt, torch.movedim(c, -1, 1), d), 1, -1).flatten(1, 3)
                for k in range(2):
                    at = self.own[2 * d + k]
                    dv = dv.index_add(1, at, (Gv[:, 2 * d + k] - (1.0 if k else -1.0) * con[d][:, at]) / w0)
                vis = vis + dv
            acc = acc - torch.cat([torch.zeros_like(vis[..., :1]), vis], -1)
        Ut = -acc / self.J.flatten(1)[..., None]
        return Ut.transpose(1, 2).reshape(U.shape)

    A = (0.0, -567301805773.0 / 1357537059087.0, -2404267990393.0 / 2016746695238.0,
         -3550918686646.0 / 2091501179385.0, -1275806237668.0 / 842570457699.0)
    B = (1432997174477.0 / 9575080441755.0, 5161836677717.0 / 13612068292357.0, 1720146321549.0 / 2090206949498.0,
         3134564353537.0 / 4481467310338.0, 2277821191437.0 / 14882151754819.0)

    def step(self, U, dt):
        g = torch.zeros_like(U)
        for a, b in zip(self.A, self.B):
            g = a * g + dt * self.rhs(U)
            U = U + b * g
        return U

    def _weights(self):
        w = self._t(self.w)
        return w[:, None, None] * w[None, :, None] * w[None, None, :] * self.J

    def kinetic_energy(self, U):
        return (self._weights() * 0.5 * (U[:, 1:4] ** 2).sum(1) / U[:, 0]).sum()

    def diagnostics(self, U, Ut):
        r, v, p = self._prim(torch.movedim(U, 1, -1))
        Jn = torch.movedim(self.Ja, (1, 2), (-2, -1))
        c = torch.sqrt(GAMMA * p / r)
        lam = ((v[..., None, :] * Jn).sum(-1).abs() + c[..., None] * Jn.norm(dim=-1)).sum(-1)
        dt = 0.9 * float((2.0 * self.J / ((2 * self.N + 1) * lam)).min())
        q2, s = (v * v).sum(-1), torch.log(p) - GAMMA * torch.log(r)
        ev = [(GAMMA - s) / (GAMMA - 1.0) - 0.5 * r * q2 / p, r * v[..., 0] / p, r * v[..., 1] / p, r * v[..., 2] / p, -r / p]
        wq = self._weights()
        inv = [(wq * Ut[:, k]).sum() for k in range(5)]
        inv.append((wq * sum(ev[k] * Ut[:, k] for k in range(5))).sum())
        inv.append((wq * 0.5 * r * q2).sum())
        inv.append((wq * (sum(v[..., k] * Ut[:, 1 + k] for k in range(3)) - 0.5 * q2 * Ut[:, 0])).sum())
        return {"dt": dt, "alpha": self._alpha(U), "invariants": torch.stack(inv).cpu().numpy()}


def exact(case, seed):
    xyz, faces, U0, dt = _inputs(case, seed)
    ref = _Reference(case, xyz, faces)
    call = case["call"]
    if call == "gradient":
        U = U0.detach().requires_grad_(True)
        V = U
        for _ in range(case["count"]):
            V = torch.utils.checkpoint.checkpoint(ref.step, V, dt, use_reentrant=False)
        ke = ref.kinetic_energy(V)
        ke.backward()
        return {"ke": ke.detach(), "grad": U.grad}
    if call == "vjp":
        U = U0.detach().requires_grad_(True)
        ref.rhs(U).backward(_cotangent(U0, seed))
        return U.grad
    with torch.no_grad():
        if call == "rhs":
            return ref.rhs(U0)
        if call == "diagnostics":
            return ref.diagnostics(U0, _cotangent(U0, seed))
        U = U0
        for _ in range(case["count"]):
            U = ref.step(U, dt)
        return U.cpu() if call == "host_step" else U
