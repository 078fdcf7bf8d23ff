"""The work a user of this library has it do, case by case, through its public entry points.

Every case is one call sequence of a FEM-PIC program on the synthetic cube workloads of
paper_2103_06737_gb300/inputs.py: the particle push with its deposits, the cell sort, the
implicit field step, and one whole PIC step.  listed() names them, draw() gives others of the
same ranges, prepare() makes the inputs from a seed, run() is one pass, work() what a pass
cannot do without, exact() the same results in 64 bits from plain PyTorch.

A pass changes particle arrays and b in place, so run() starts by copying them from a
snapshot, as a program that restarts from a checkpoint does: every pass does the same work.
"""
import itertools
import math

import numpy as np
import torch

import paper_2103_06737_gb300.fem_pic as F
from paper_2103_06737_gb300 import inputs as I

DEV = "cuda"
C, QE, ME = I.C_LIGHT, I.Q_E, I.M_E
EPS0, MU0 = F.EPS0, F.MU0
TOL = 1e-10               # relative residual of both field solves (the library's default)
LE = ((0, 1), (0, 2), (0, 3), (1, 2), (1, 3), (2, 3))      # local edges of a tet
LF = ((1, 2, 3), (0, 2, 3), (0, 1, 3), (0, 1, 2))          # local face k is opposite vertex k
ADAMS_STEP = 7            # an Adams push after the start-up steps (fourth order)


def _push(name, n, particles, **kw):
    return dict(name=name, kind="push", n=n, particles=particles, precision="fp32", deposits="fp32",
                mover="boris", beam=False, vth=0.01, B0=0.1, mixed=0.25, **kw)


def listed():
    return [
        # The 4^3 mesh with 1,000 electrons in FP64: the smallest simulation, a program's first run
        # and its check against a reference; launches and latency.
        dict(_push("push_fp64_cube4_1k", 4, 1000), precision="fp64", mixed=0.0),
        # 16^3 with an odd number of particles: state arrays that start on no 16-byte boundary.
        _push("push_odd_cube16_301k", 16, 301_003),
        # 32^3 with 2M electrons, the library's default deposits: the ordinary push.
        _push("push_cube32_2M", 32, 2_000_000),
        # The same in FP64 mode: a user who wants round-off-level deposits.
        dict(_push("push_fp64_cube32_2M", 32, 2_000_000), precision="fp64"),
        # The paper's fourth-order Adams mover on the same electrons.
        dict(_push("push_adams_cube32_2M", 32, 2_000_000), mover="adams"),
        # The largest push: 96^3 with 50M electrons, the charge change added onto a double Q.
        dict(_push("push_change_cube96_50M", 96, 50_000_000), deposits="change", vth=0.02, B0=0.2),
        # The periodic sort of the 64^3 beam's electrons and the charge of the sorted state.
        dict(name="sort_beam_cube64_20M", kind="sort", n=64, particles=20_000_000, precision="fp32", beam=True,
             vth=0.005, B0=0.5, mixed=0.6),
        # The field step of the smallest mesh.
        dict(name="field_cube4", kind="field", n=4, pc="jacobi", bc="pec", B0=0.1),
        # 32^3 with the polynomial preconditioners a tuned program sets (degrees 3 and 8).
        dict(name="field_cube32_cheb", kind="field", n=32, pc="cheb", bc="pec", B0=0.1),
        # 64^3 with plain Jacobi-CG: the beam workload's field step.
        dict(name="field_cube64_jacobi", kind="field", n=64, pc="jacobi", bc="pec", B0=0.5),
        # 96^3 with a learned preconditioner in both solves: the largest field step.
        dict(name="field_cube96_learned", kind="field", n=96, pc="learned", bc="pec", B0=0.2),
        # One whole PIC step, 32^3 with 2M electrons and plain Jacobi-CG: push, charge of the ion
        # background, field step.
        dict(name="step_cube32_2M", kind="step", n=32, particles=2_000_000, precision="fp32", beam=False, vth=0.01,
             B0=0.1, mixed=0.25, pc="jacobi", bc="pec"),
    ]


def draw(rng):
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    kind = rng.choice(["push", "push", "push", "sort", "field", "field", "field", "step"])
    vth, B0 = rng.choice([0.005, 0.01, 0.02]), rng.choice([0.1, 0.2, 0.5])
    if kind == "field":
        return dict(kind=kind, n=size(4, 48), pc=rng.choice(["jacobi", "cheb", "learned"]),
                    bc=rng.choice(["pec", "pec", "pec", "neumann"]), B0=B0)
    n = size(4, 56 if kind != "step" else 32)
    particles = min(16_000_000, int(6 * n ** 3 * math.exp(rng.uniform(math.log(1.5), math.log(20.0)))))
    particles -= rng.choice([0, 0, 1, 3]) if particles % 4 == 0 else particles % 4 * rng.choice([0, 1, 1])
    base = dict(kind=kind, n=n, particles=particles, precision="fp32", beam=rng.random() < 0.25, vth=vth, B0=B0,
                mixed=rng.choice([0.0, 0.25, 0.6]))
    if kind == "sort":
        return base
    if kind == "step":
        return dict(base, pc=rng.choice(["jacobi", "cheb"]), bc="pec")
    base.update(deposits=rng.choice(["fp32", "fp32", "change", "fp64"]), mover="boris")
    if rng.random() < 0.2:
        base.update(mover="adams", deposits="fp32")
    elif rng.random() < 0.2:
        base.update(precision="fp64", deposits="fp32", particles=min(particles, 2_000_000))
    return base


# ------------------------------------------------------------------ the mesh in plain PyTorch
class Grid:
    """Numbering, geometry and FP64 operators of one cube mesh, from the published conventions:
    tet vertices ascending, edges and faces numbered in lexicographic order of their nodes."""

    def __init__(self, n):
        self.n = n
        self.mesh = I.cube_mesh(n, 1.0, 0.1 if n > 4 else 0.0, seed=1)
        self.x = torch.as_tensor(self.mesh.xyz, device=DEV)
        self.nn = self.x.shape[0]
        t = torch.sort(torch.as_tensor(self.mesh.tets, device=DEV).long(), dim=1).values
        self.tets, self.nt = t, t.shape[0]
        ekey = torch.stack([t[:, a] * self.nn + t[:, b] for a, b in LE], 1)
        uk, inv = torch.unique(ekey, return_inverse=True)
        self.te, self.ne = inv.reshape(-1, 6), uk.shape[0]
        self.edges = torch.stack([uk // self.nn, uk % self.nn], 1)
        nodes, inv = self._unique_faces(t)
        self.tf, self.nf, self.faces = inv.reshape(-1, 4), nodes.shape[0], nodes
        count = torch.bincount(self.tf.reshape(-1), minlength=self.nf)
        self.wall_face = count == 1
        self.wall_node = torch.zeros(self.nn, dtype=torch.bool, device=DEV)
        self.wall_node[nodes[self.wall_face].reshape(-1)] = True
        fe = torch.searchsorted(uk, torch.stack([nodes[:, a] * self.nn + nodes[:, b] for a, b in ((0, 1), (1, 2), (0, 2))], 1))
        self.face_edges = fe
        self.wall_edge = torch.zeros(self.ne, dtype=torch.bool, device=DEV)
        self.wall_edge[fe[self.wall_face].reshape(-1)] = True
        v = self.x[t]
        J = v[:, 1:] - v[:, :1]
        det = torch.det(J)
        inv3 = torch.linalg.inv(J).transpose(1, 2)          # rows: gradients of lambda_1..3
        self.g = torch.cat([-inv3.sum(1, keepdim=True), inv3], 1).contiguous()
        self.vol = det.abs() / 6.0
        self.origin = v[:, 0].contiguous()
        self._ops = {}

    def _unique_faces(self, t):
        key = torch.stack([(t[:, a] * self.nn + t[:, b]) * self.nn + t[:, c] for a, b, c in LF], 1)
        uk, inv = torch.unique(key, return_inverse=True)
        return torch.stack([uk // (self.nn * self.nn), uk // self.nn % self.nn, uk % self.nn], 1), inv

    def neighbours(self):
        """[nt, 4]: the tet across face k, -1 at a wall."""
        flat = self.tf.reshape(-1)
        order = torch.argsort(flat)
        s = flat[order]
        same = torch.nonzero(s[1:] == s[:-1]).reshape(-1)
        a, b = order[same], order[same + 1]
        nb = torch.full_like(flat, -1)
        nb[a], nb[b] = b // 4, a // 4
        return nb.reshape(-1, 4)

    def alpha(self):
        return torch.zeros(self.nn, dtype=torch.float64, device=DEV).index_add_(
            0, self.tets.reshape(-1), (self.vol / 4)[:, None].expand(-1, 4).reshape(-1))

    def grad(self, phi):
        return phi[self.edges[:, 1]] - phi[self.edges[:, 0]]

    def div(self, e):
        out = torch.zeros(self.nn, dtype=torch.float64, device=DEV)
        out.index_add_(0, self.edges[:, 1], e)
        return out.index_add_(0, self.edges[:, 0], -e)

    def curl(self, e):
        fe = self.face_edges
        return e[fe[:, 0]] + e[fe[:, 1]] - e[fe[:, 2]]

    def flux(self, B):
        p = self.x[self.faces]
        return 0.5 * torch.linalg.cross(p[:, 1] - p[:, 0], p[:, 2] - p[:, 0]) @ torch.tensor(B, dtype=torch.float64, device=DEV)

    def operators(self, pec):
        """CSR of the edge mass M and the curl-curl S over the free edges (PEC rows zero)."""
        if pec not in self._ops:
            g, w = self.g, self.vol
            rows, cols, m, s = [], [], [], []
            gg = g @ g.transpose(1, 2)
            cw = [torch.linalg.cross(g[:, a], g[:, b]) for a, b in LE]
            free = ~self.wall_edge if pec else torch.ones(self.ne, dtype=torch.bool, device=DEV)
            for r, (a, b) in enumerate(LE):
                for k, (c, d) in enumerate(LE):
                    mv = EPS0 * w / 20 * (gg[:, b, d] * (1 + (a == c)) - gg[:, b, c] * (1 + (a == d))
                                          - gg[:, a, d] * (1 + (b == c)) + gg[:, a, c] * (1 + (b == d)))
                    ok = free[self.te[:, r]] & free[self.te[:, k]]
                    rows.append(self.te[ok, r])
                    cols.append(self.te[ok, k])
                    m.append(mv[ok])
                    s.append((4 * w / MU0 * (cw[r] * cw[k]).sum(1))[ok])
            key = torch.cat(rows) * self.ne + torch.cat(cols)
            uk, inv = torch.unique(key, return_inverse=True)
            crow = torch.searchsorted(uk // self.ne, torch.arange(self.ne + 1, device=DEV))
            col = uk % self.ne
            vals = [torch.zeros(uk.shape[0], dtype=torch.float64, device=DEV).index_add_(0, inv, torch.cat(v)) for v in (m, s)]
            self._ops[pec] = (crow, col, vals[0], vals[1])
        return self._ops[pec]

    def csr(self, pec, m=1.0, s=0.0):
        crow, col, M, S = self.operators(pec)
        return torch.sparse_csr_tensor(crow, col, m * M + s * S, size=(self.ne, self.ne))

    def mass_diag(self, pec, dt):
        """Diagonals of A = M + dt^2/4 S and of L = D0^T M D0."""
        crow, col, M, S = self.operators(pec)
        row = torch.repeat_interleave(torch.arange(self.ne, device=DEV), crow[1:] - crow[:-1])
        d = row == col
        dA = torch.zeros(self.ne, dtype=torch.float64, device=DEV)
        dA[row[d]] = (M + 0.25 * dt * dt * S)[d]
        gl = (self.g * self.g).sum(2) * (EPS0 * self.vol)[:, None]
        dL = torch.zeros(self.nn, dtype=torch.float64, device=DEV).index_add_(0, self.tets.reshape(-1), gl.reshape(-1))
        return dA, dL

    def bary(self, cell, off):
        l = torch.einsum("pkd,pd->pk", self.g[cell, 1:], off)
        return torch.cat([1 - l.sum(1, keepdim=True), l], 1)


_grids, _handles = {}, {}


def _grid(n):
    if n not in _grids:
        _grids[n] = Grid(n)
    return _grids[n]


def _dt(case):
    return 0.2 * I.gyro_period(case["B0"])


def _handle(case):
    """The library handle of the case's mesh and options, made once as a program does."""
    field = case["kind"] in ("field", "step")
    key = (case["n"], case.get("precision", "fp32"), case.get("deposits", "fp32"), field and case["pc"],
           field and case["bc"], field and case["B0"])
    if key in _handles:
        return _handles[key]
    m = _grid(case["n"]).mesh
    lib = F.FemPic(m.xyz, m.tets, F.FP_FP64 if case.get("precision") == "fp64" else F.FP_FP32)
    if case.get("deposits") == "change":
        lib.set_charge_precision(F.FP_FP64)
    elif case.get("deposits") == "fp64":
        lib.set_deposit_precision(F.FP_FP64)
    if field:
        F.fem_pic_field_setup(lib.h, _dt(case), bc=F.FP_BC_NEUMANN if case["bc"] == "neumann" else None)
        if case["pc"] == "cheb":
            F.fem_pic_field_poly(lib.h, F.FP_SYS_NEWMARK, 3, 15.0)
            F.fem_pic_field_poly(lib.h, F.FP_SYS_GAUSS, 8, 100.0)
        elif case["pc"] == "learned":
            for system in (F.FP_SYS_NEWMARK, F.FP_SYS_GAUSS):
                F.fem_pic_learned_select(lib.h, system)
                F.fem_pic_learned_init_model(lib.h, seed=4, sample_capacity=1, model=F.FP_LEARNED_PRECOND)
                # weights as a program loads them; the head (w, b0, v, d0) a polynomial of degree one
                # in the scaled operator, what training starts from
                P = F.fem_pic_learned_params(lib.h)
                P[-130:] = 0.0
                P[-66], P[-1] = -0.22, -0.22
                F.fem_pic_learned_params(lib.h, P)
                F.fem_pic_learned_build(lib.h)
    _handles[key] = lib
    return lib


# ------------------------------------------------------------------ inputs
def _particles(case, g):
    """Electrons in the order of the last cell sort: uniform in space (or in the beam's cylinder),
    Maxwellian; the fraction `mixed` has moved to a near tet since. """
    n, real = case["particles"], torch.float64 if case["precision"] == "fp64" else torch.float32
    vol = g.vol
    if case["beam"]:
        c = g.x[g.tets].mean(1)
        vol = vol * (((c[:, 0] - 0.5) ** 2 + (c[:, 1] - 0.5) ** 2) < 0.04)
    cdf = torch.cumsum(vol, 0)
    u = torch.rand(n, dtype=torch.float64, device=DEV).sort().values * cdf[-1]
    cell = torch.searchsorted(cdf, u, right=True).clamp_(max=g.nt - 1)
    del u
    if case["mixed"] > 0:
        moved = torch.rand(n, device=DEV) < case["mixed"]
        key = cell + moved * torch.randint(-6 * case["n"], 6 * case["n"] + 1, (n,), device=DEV)
        cell = cell[torch.argsort(key)]
    flat = torch.empty(6 * n, dtype=real, device=DEV)
    for p in range(0, n, 1 << 22):
        q = min(n, p + (1 << 22))
        ck = cell[p:q]
        lam = -torch.log(torch.rand(q - p, 4, dtype=torch.float64, device=DEV).clamp_(min=1e-12))
        lam /= lam.sum(1, keepdim=True)
        tv = g.tets[ck]
        off = torch.einsum("pk,pkd->pd", lam[:, 1:], g.x[tv[:, 1:]] - g.x[tv[:, :1]])
        v = torch.randn(q - p, 3, dtype=torch.float64, device=DEV) * (case["vth"] * C)
        if case["beam"]:
            v[:, 2] += 0.1 * C
        for k in range(3):
            flat[k * n + p:k * n + q] = off[:, k]
            flat[(3 + k) * n + p:(3 + k) * n + q] = v[:, k]
    return cell.int(), flat


def _seed(seed):
    torch.manual_seed(seed)
    np.random.seed(seed % (1 << 31))


def _species(case, cell0, flat0):
    n = case["particles"]
    cell, flat = torch.empty_like(cell0), torch.empty_like(flat0)
    return flat, F.Species(cell, flat[:3 * n].view(3, n), flat[3 * n:].view(3, n), -QE, ME, 1e14 / n)


def _push_fields(case, g):
    ed = g.x[g.edges[:, 1]] - g.x[g.edges[:, 0]]
    e = 1e3 * ed.norm(dim=1) * (2 * torch.rand(g.ne, dtype=torch.float64, device=DEV) - 1)
    e[g.wall_edge] = 0.0
    return e, g.flux((0.0, 0.0, case["B0"]))


def _field_inputs(case, g):
    """Fields, deposits and charge of a running simulation: the charge follows from the fields by
    Gauss's law and continuity up to the rounding of its float deposits."""
    pec, dt = case["bc"] == "pec", _dt(case)
    h = 1.0 / case["n"]
    r = lambda k: torch.randn(k, dtype=torch.float64, device=DEV)  # noqa: E731
    phi = 10 * torch.cos(3 * g.x[:, 0]) * torch.sin(4 * g.x[:, 1]) + r(g.nn)
    if pec:
        phi[g.wall_node] = 0.0
    E = g.grad(phi) + 200 * h * r(g.ne)
    Ep = E + 20 * h * r(g.ne)
    if pec:
        E[g.wall_edge] = 0.0
        Ep[g.wall_edge] = 0.0
    M = g.csr(pec)
    ME_ = M @ E
    dGp = (M @ Ep - ME_).float()
    dGh = (dGp.double() + 0.5 * dGp.abs().mean() * r(g.ne)).float()
    if pec:
        dGh[g.wall_edge] = 0.0
    Q = (g.div(dGh.double()) - g.div(ME_)).float()
    b = g.flux((0.0, 0.0, case["B0"])) + 1e-6 * h * h * r(g.nf)
    return dict(E_prev=Ep, E_cur=E, b0=b, dG_prev=dGp, dG=dGh, Q=Q)


def _start_fields(case, g, cell0, flat0):
    """The first step's fields: E of the Gauss law for the loaded charge, b uniform."""
    n = case["particles"]
    Qion = (QE * 1e14 * g.alpha()).float()
    Q = torch.zeros(g.nn, dtype=torch.float64, device=DEV)
    for p in range(0, n, 1 << 22):
        c = cell0[p:p + (1 << 22)].long()
        off = torch.stack([flat0[k * n + p:k * n + p + len(c)] for k in range(3)], 1).double()
        Q.index_add_(0, g.tets[c].reshape(-1), (-QE * 1e14 / n * g.bary(c, off)).reshape(-1))
    rhs = (Q + Qion.double())
    rhs[g.wall_node] = 0.0
    d = _cg_gauss(case, g, rhs, 1e-12, float(rhs.norm()))
    return -g.grad(d), g.flux((0.0, 0.0, case["B0"])), Qion


def prepare(case, seed):
    _seed(seed)
    g, lib = _grid(case["n"]), _handle(case)
    s = dict(case=case, lib=lib)
    if case["kind"] == "field":
        s.update(_field_inputs(case, g), E_next=torch.empty(g.ne, dtype=torch.float64, device=DEV))
        s["b"] = s["b0"].clone()
        return s
    s["cell0"], s["flat0"] = _particles(case, g)
    s["flat"], s["sp"] = _species(case, s["cell0"], s["flat0"])
    if case["kind"] == "sort":
        s["src"] = F.Species(s["cell0"], s["flat0"][:3 * s["sp"].n].view(3, -1), s["flat0"][3 * s["sp"].n:].view(3, -1),
                             s["sp"].q, s["sp"].m, s["sp"].w)
        s["Q"] = torch.empty(g.nn, dtype=lib.charge_dtype, device=DEV)
        return s
    s["dG"] = torch.empty(g.ne, dtype=lib.deposit_dtype, device=DEV)
    s["Q"] = torch.zeros(g.nn, dtype=lib.charge_dtype, device=DEV)
    if case["kind"] == "step":
        s["E_cur"], s["b0"], s["Q_ion"] = _start_fields(case, g, s["cell0"], s["flat0"])
        s["E_prev"], s["E_next"] = s["E_cur"].clone(), torch.empty_like(s["E_cur"])
        s["b"] = s["b0"].clone()
        return s
    s["e"], s["b"] = _push_fields(case, g)
    if case["deposits"] == "change":   # Q^n: the charge of the start positions
        s["Q0"] = _charge(case, g, s["cell0"], s["flat0"]).to(lib.charge_dtype)
    if case["mover"] == "adams":
        n, real = case["particles"], s["flat0"].dtype
        # three earlier steps' velocities and accelerations, a gyrating electron's
        s["hist"] = torch.empty(18, n, dtype=real, device=DEV)
        a = QE / ME * case["B0"]
        for j in range(3):
            v = s["flat0"].view(6, n)[3:] + 1e-3 * case["vth"] * C * torch.randn(3, n, dtype=real, device=DEV)
            s["hist"][6 * j:6 * j + 3] = v
            s["hist"][6 * j + 3], s["hist"][6 * j + 4], s["hist"][6 * j + 5] = -a * v[1], a * v[0], 0.0
    return s


def _charge(case, g, cell0, flat0):
    n = case["particles"]
    Q = torch.zeros(g.nn, dtype=torch.float64, device=DEV)
    for p in range(0, n, 1 << 22):
        c = cell0[p:p + (1 << 22)].long()
        off = torch.stack([flat0[k * n + p:k * n + p + len(c)] for k in range(3)], 1).double()
        Q.index_add_(0, g.tets[c].reshape(-1), (-QE * 1e14 / n * g.bary(c, off)).reshape(-1))
    return Q


# ------------------------------------------------------------------ one pass
def _restore(s):
    s["sp"].cell.copy_(s["cell0"])
    s["flat"].copy_(s["flat0"])


def _field(s, dG, dG_prev):
    pc = F.FP_PC_LEARNED | F.FP_PC_LEARNED_GAUSS if s["case"]["pc"] == "learned" else F.FP_PC_JACOBI
    s["b"].copy_(s["b0"])
    F.fem_pic_field_step(s["lib"].h, s["E_prev"], s["E_cur"], s["E_next"], s["b"], dG, dG_prev, s["Q"], tol=TOL,
                         precond=pc, info=False)


def run(s):
    case, lib = s["case"], s["lib"]
    if case["kind"] == "field":
        _field(s, s["dG"], s["dG_prev"])
        return {"E": s["E_next"], "b": s["b"]}
    sp = s["sp"]
    if case["kind"] == "sort":
        lib.sort(s["src"], sp)
        lib.deposit_charge(sp, s["Q"])
        return {"cell": sp.cell, "Q": s["Q"]}
    _restore(s)
    state = {"cell": sp.cell, "off": sp.off, "vel": sp.vel, "dG": s["dG"], "Q": s["Q"]}
    if case["kind"] == "step":
        lib.push_deposit(s["E_cur"], s["b0"], sp, _dt(case), s["dG"], s["Q"])
        s["Q"].add_(s["Q_ion"])
        _field(s, s["dG"], None)
        return dict(state, E=s["E_next"], b=s["b"])
    if case["mover"] == "adams":
        lib.push_deposit_adams(s["e"], s["b"], sp, s["hist"], ADAMS_STEP, 0.25 * _dt(case), s["dG"], s["Q"])
        return dict(state, hist=s["hist"])
    flags = 0
    if case["deposits"] == "change":
        s["Q"].copy_(s["Q0"])
        flags = F.FP_CHARGE_CHANGE
    lib.push_deposit(s["e"], s["b"], sp, _dt(case), s["dG"], s["Q"], flags=flags)
    return state


# ------------------------------------------------------------------ the work of a pass
def work(case):
    n = case["n"]
    nt, nn = 6 * n ** 3, (n + 1) ** 3
    nf = 12 * n ** 3 + 6 * n * n
    ne = nn + nf - nt - 1
    by = fl = 0.0
    if "particles" in case:
        p, r = case["particles"], 8 if case["precision"] == "fp64" else 4
        by += 2 * p * (4 + 6 * r)                   # the particle state in and out
        if case["kind"] == "sort":
            return {"bytes": by + r * nn, "flops": 20.0 * p}
        hist = 18 + 6 if case.get("mover") == "adams" else 0
        by += p * hist * r + 128 * nt + 8 * (ne + nf) + r * (ne + nn)   # history, tet tables, e, b, dG, Q
        fl += 250.0 * p
    if "pc" in case:
        nnz = 16.3 * ne
        # the edge operators once (M and S in FP64 with their columns), the nodes' Laplacian once, the
        # fields, deposits and right-hand sides once each
        by += 20 * nnz + 12 * 15 * nn + 8 * (3 * ne + 2 * nf) + 8 * ne + 4 * nn
        its = {"jacobi": 60, "cheb": 60, "learned": 80}[case["pc"]]
        fl += 2 * nnz * its + 2 * 15 * nn * 2 * its
    return {"bytes": by, "flops": fl}


# ------------------------------------------------------------------ the same in 64 bits
def _cg(A, dinv, b, tol, ref, limit=4000):
    x = torch.zeros_like(b)
    r, z = b.clone(), dinv * b
    p, rz = z.clone(), torch.dot(b, z)
    for it in itertools.count():
        if it % 16 == 0 and (float(r.norm()) <= tol * ref or it >= limit):
            return x
        q = A(p)
        alpha = rz / torch.dot(p, q).clamp_(min=1e-300)
        x += alpha * p
        r -= alpha * q
        z = dinv * r
        new = torch.dot(r, z)
        p = z + (new / rz.clamp(min=1e-300)) * p
        rz = new


def _cg_gauss(case, g, rhs, tol, ref):
    pec = case["bc"] == "pec"
    M = g.csr(pec)
    free = ~g.wall_node if pec else torch.ones_like(g.wall_node)
    dL = g.mass_diag(pec, _dt(case))[1]
    return _cg(lambda d: g.div(M @ g.grad(d)) * free, free / dL, rhs * free, tol, ref)


def _exact_field(case, g, E_prev, E_cur, b0, dG, dG_prev, Q):
    pec, dt = case["bc"] == "pec", _dt(case)
    free = ~g.wall_edge if pec else torch.ones_like(g.wall_edge)
    u = 2 * E_cur - E_prev
    r0 = -(g.csr(pec, 0.0, dt * dt) @ E_cur) - (dG if dG_prev is None else dG - dG_prev)
    A = g.csr(pec, 1.0, 0.25 * dt * dt)
    dA = g.mass_diag(pec, dt)[0]
    dinv = torch.where(free, 1 / dA, torch.zeros_like(dA))
    ref = float((A @ u + r0).norm())
    EN = u * free + _cg(lambda v: A @ v, dinv, r0 * free, 1e-14, ref)
    gl = g.div(g.csr(pec) @ EN) + Q
    if pec:
        gl[g.wall_node] = 0.0
        ref = float(Q[~g.wall_node].norm())
    else:
        al = g.alpha()
        gl = gl - gl.sum() / al.sum() * al
        ref = float(Q.norm())
    E1 = EN - g.grad(_cg_gauss(case, g, gl, 1e-14, ref)) * free
    return E1, b0 - 0.5 * dt * g.curl(E1 + E_cur)


def _exact_push(case, g, s, e, b, dt):
    """vel, dG, Q (and the Adams history) of one particle step from the same inputs in FP64."""
    n, qw = case["particles"], -QE * (1e14 / case["particles"])
    qm = -QE / ME
    nb = g.neighbours()
    dG = torch.zeros(g.ne, dtype=torch.float64, device=DEV)
    Q = torch.zeros(g.nn, dtype=torch.float64, device=DEV)
    vel = torch.empty(3, n, dtype=torch.float64, device=DEV)
    st = s["flat0"].view(6, n)
    adams = case.get("mover") == "adams"
    hist = s["hist"].double() if adams else None
    for p in range(0, n, 1 << 21):
        q = min(n, p + (1 << 21))
        c = s["cell0"][p:q].long()
        x, v = st[:3, p:q].T.double(), st[3:, p:q].T.double()
        gr, lam = g.g[c], g.bary(c, x)
        E, B = torch.zeros_like(x), torch.zeros_like(x)
        for k, (i, j) in enumerate(LE):
            E += e[g.te[c, k]][:, None] * (lam[:, i:i + 1] * gr[:, j] - lam[:, j:j + 1] * gr[:, i])
        for k, (i, j, m) in enumerate(LF):
            B += 2 * b[g.tf[c, k]][:, None] * (lam[:, i:i + 1] * torch.linalg.cross(gr[:, j], gr[:, m])
                                               + lam[:, j:j + 1] * torch.linalg.cross(gr[:, m], gr[:, i])
                                               + lam[:, m:m + 1] * torch.linalg.cross(gr[:, i], gr[:, j]))
        if adams:
            a = qm * (E + torch.linalg.cross(v, B))
            beta = (55 / 24, -59 / 24, 37 / 24, -9 / 24)
            sx, sa = beta[0] * v, beta[0] * a
            for j in (1, 2, 3):
                sl = 6 * ((ADAMS_STEP - j) % 3)
                sx = sx + beta[j] * hist[sl:sl + 3, p:q].T
                sa = sa + beta[j] * hist[sl + 3:sl + 6, p:q].T
            end, v1 = x + dt * sx, v + dt * sa
            sl = 6 * (ADAMS_STEP % 3)
            hist[sl:sl + 3, p:q], hist[sl + 3:sl + 6, p:q] = v.T, a.T
        else:
            h = qm * dt / 2
            vm, t = v + h * E, h * B
            vp = vm + torch.linalg.cross(vm, t)
            v1 = vm + torch.linalg.cross(vp, 2 * t / (1 + (t * t).sum(1, keepdim=True))) + h * E
            end = x + dt * v1
        vel[:, p:q] = v1.T
        end = end + g.origin[c]
        entry, la = torch.full_like(c, -1), lam
        for _ in range(64):
            lb = g.bary(c, end - g.origin[c])
            face = torch.arange(4, device=DEV)[None, :]
            cand = (lb < 0) & (face != entry[:, None])
            frac = torch.where((la > 0) & (la > lb), la / (la - lb), torch.zeros_like(la)).clamp(0, 1)
            frac = torch.where(cand, frac, torch.full_like(frac, 2.0))
            sx, k = frac.min(1)
            go = cand.any(1)
            lc = torch.where(go[:, None], la + sx[:, None] * (lb - la), lb)
            lc = torch.where(go[:, None] & (face == k[:, None]), torch.zeros_like(lc), lc)
            for j, (i, m) in enumerate(LE):
                dG.index_add_(0, g.te[c, j], qw * (la[:, i] * lc[:, m] - la[:, m] * lc[:, i]))
            nxt = torch.where(go, nb[c, k], torch.full_like(c, -1))
            stop = nxt < 0
            Q.index_add_(0, g.tets[c[stop]].reshape(-1), (qw * lc[stop]).reshape(-1))
            keep = ~stop
            if not bool(keep.any()):
                break
            c0, c, end = c[keep], nxt[keep], end[keep]
            same = g.tets[c][:, :, None] == g.tets[c0][:, None, :]
            la = (same * lc[keep][:, None, :]).sum(2)
            entry = (~same.any(2)).long().argmax(1)
    return vel, dG, Q, hist


def exact(case, seed):
    s = prepare(case, seed)
    g = _grid(case["n"])
    if case["kind"] == "field":
        E, b = _exact_field(case, g, s["E_prev"], s["E_cur"], s["b0"], s["dG"].double(), s["dG_prev"].double(),
                            s["Q"].double())
        return {"E": E, "b": b}
    if case["kind"] == "sort":
        return {"cell": None, "Q": _charge(case, g, s["cell0"], s["flat0"])}
    if case["kind"] == "step":
        vel, dG, Q, _ = _exact_push(case, g, s, s["E_cur"], s["b0"], _dt(case))
        Q = Q + s["Q_ion"].double()
        E, b = _exact_field(case, g, s["E_prev"], s["E_cur"], s["b0"], dG, None, Q)
        return {"cell": None, "off": None, "vel": vel, "dG": dG, "Q": Q, "E": E, "b": b}
    adams = case["mover"] == "adams"
    vel, dG, Q, hist = _exact_push(case, g, s, s["e"], s["b"], (0.25 if adams else 1.0) * _dt(case))
    out = {"cell": None, "off": None, "vel": vel, "dG": dG, "Q": Q}
    return dict(out, hist=hist) if adams else out
