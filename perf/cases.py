"""The work this framework is used for, as cases that can be timed and compared.

A case is a dict of plain values. Its ``kind`` says which public entry points
a pass goes through:

* ``frames``    one mesh on the GPU: back to rest, then activation frames of a
                ramp, each solved from the one before; positions after each
                frame (``Solver``: the interactive or offline simulation).
* ``batch``     many small meshes solved together (``batch_solve``: parameter
                studies, data generation).
* ``serve``     requests with meshes of their own submitted to a running
                ``Server`` and collected (set-up of every mesh included).
* ``arm``       a mesh with bones and a hinge joint, one activation from rest.
* ``coupling``  the coupling solve alone, from deformation gradients that the
                caller has (``acap_solve_noalloc``).
* ``fibers``    the fiber field of a mesh (``fiber_field``), a set-up tool
                that runs once per muscle.

Meshes are the grids of ``emu_inputs``: beams held at one end, muscle-tendon
units attached at both, as a muscle is. ``jitter`` moves their vertices, so
that no two tets are alike, as in a mesh from a tetrahedraliser. The seed
gives fibers, activations, jitter and deformations; sizes come from the case.
Positions of a mixed-precision solve are good to about 1e-6 of the mesh and are
taken in single precision, as a renderer takes them; FP64 results stay FP64.
"""
import time

import numpy as np
import torch

import paper_2006_08821_gb300 as emu
from emu_inputs import arm_assembly, box_beam, muscle_tendon_unit
from emu_inputs.meshes import batch_set, gravity_forces, mtu_for_tet_count

DEVICE = "cuda"
FRAMES = dict(kind="frames", mesh="unit", tets=0, nx=0, ny=0, nz=0, frames=1, precision="mixed", form="rs",
              tol=1e-6, jitter=0.0, gravity=False, own_stream=True)


def listed():
    return [
        # the README's first program on its smallest mesh, on the default stream: launches and latency
        dict(FRAMES, name="beam_144", mesh="beam", nx=2, ny=2, nz=6, own_stream=False),
        # the box beam in FP64, converged as a reference solution (the parity tests' tolerance)
        dict(FRAMES, name="beam_1536_fp64", mesh="beam", nx=4, ny=4, nz=16, precision="fp64", tol=1e-11),
        # a preview-size muscle-tendon unit played over a short ramp
        dict(FRAMES, name="unit_6k", tets=6000, frames=4),
        # an ordinary muscle on an irregular mesh, under gravity
        dict(FRAMES, name="unit_60k_irregular", tets=60000, frames=2, jitter=0.12, gravity=True),
        # the benchmark's muscle-tendon unit (401,920 tets)
        dict(FRAMES, name="unit_402k", tets=401920, frames=3),
        # the same construction in FP64, in the rotation-stretch form and in the paper's F-form
        dict(FRAMES, name="unit_6k_fp64", tets=6000, precision="fp64", tol=1e-11),
        dict(FRAMES, name="beam_1k_fform", mesh="beam", nx=3, ny=4, nz=14, precision="fp64", form="f", tol=1e-11),
        # a slice of the 256-beam batch
        dict(name="batch_16", kind="batch", count=16, mesh_seed=3, t_max=30000.0),
        # a burst of requests at a server, as its request stream makes them
        dict(name="serve_6", kind="serve", count=6, mesh_seed=4, t_max=12000.0, frames_max=4),
        # bones and a hinge: the coupling solves run in FP64
        dict(name="arm_2k", kind="arm", bone_w=2, bone_len=8, r0=4.0, tol=1e-6),
        # the coupling solve on its own
        dict(name="coupling_98k", kind="coupling", tets=98400, jitter=0.0, precision="mixed"),
        # fibers of a muscle from its attachments
        dict(name="fibers_22k", kind="fibers", tets=21792, jitter=0.12),
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(lo * (hi / lo) ** rng.random()))

    kind = rng.choice(["frames", "frames", "frames", "frames64", "batch", "serve", "arm", "coupling", "fibers"])
    if kind in ("frames", "frames64"):
        c = dict(FRAMES, frames=rng.randint(1, 3), jitter=rng.choice([0.0, round(rng.uniform(0.05, 0.15), 3)]),
                 gravity=rng.random() < 0.3, own_stream=rng.random() < 0.8)
        top = 250000 if kind == "frames" else 8000
        if rng.random() < 0.5:
            w = rng.randint(1, 7)
            c.update(mesh="beam", nx=w, ny=max(1, w + rng.randint(-1, 2)), nz=rng.randint(2 * w, 5 * w + 3))
        else:
            c.update(tets=log_int(700, top))
        if kind == "frames64":
            c.update(precision="fp64", tol=1e-11, frames=1, form=rng.choice(["rs", "rs", "f"]))
        return c
    if kind == "batch":
        return dict(kind=kind, count=rng.randint(2, 16), mesh_seed=rng.randint(0, 9999), t_max=float(log_int(3000, 30000)))
    if kind == "serve":
        return dict(kind=kind, count=rng.randint(1, 6), mesh_seed=rng.randint(0, 9999), t_max=float(log_int(2000, 12000)),
                    frames_max=rng.randint(1, 4))
    if kind == "arm":
        w = rng.randint(2, 3)
        return dict(kind=kind, bone_w=w, bone_len=rng.randint(4, 9), r0=round(rng.uniform(2.0, 4.0), 2), tol=1e-6)
    c = dict(kind=kind, tets=log_int(1000, 98400 if kind == "coupling" else 60000), jitter=round(rng.uniform(0.0, 0.15), 3))
    return dict(c, precision=rng.choice(["mixed", "fp64"])) if kind == "coupling" else c


# ---------------------------------------------------------------- inputs ----

def _muscle(tets, tendon, seed):
    """A muscle-tendon unit of about so many tets, the vertices of both ends pinned; fully activated."""
    m = muscle_tendon_unit(frames=1, seed=seed) if tets == 401920 else mtu_for_tet_count(tets, tendon_frac=tendon, seed=seed)
    z = m.rest_pos[:, 2]
    m.fixed_verts = np.nonzero((z == 0.0) | (z >= (m.meta["nz"] - 0.5) * m.meta["h"]))[0].astype(np.int32)
    return m


def _jittered(mesh, amount, rng):
    """The mesh with its unpinned vertices moved by up to ``amount`` grid steps."""
    if amount:
        move = rng.uniform(-amount, amount, mesh.rest_pos.shape) * mesh.meta["h"]
        move[mesh.fixed_verts] = 0.0
        mesh.rest_pos = mesh.rest_pos + move
    return mesh


def _frames_mesh(case, seed):
    """The mesh of a ``frames`` case and its activation frames (frames, n_tets)."""
    rng = np.random.default_rng(seed)
    if case["mesh"] == "beam":
        mesh = box_beam(case["nx"], case["ny"], case["nz"])
        on = np.ones(mesh.n_tets)
    else:
        mesh = _muscle(case["tets"], 0.1, int(rng.integers(1 << 31)))
        on = mesh.activations[0]
    ramp = rng.uniform(0.3, 0.9) * np.arange(1, case["frames"] + 1) / case["frames"]
    mesh = _jittered(mesh, case["jitter"], rng)
    if case["gravity"]:
        mesh.f_ext = gravity_forces(mesh)
    return mesh, ramp[:, None] * on[None, :]


def _batch_meshes(case, seed):
    rng = np.random.default_rng(seed)
    meshes = batch_set(case["count"], seed=case["mesh_seed"], t_max=case["t_max"])
    return [(m, np.full(m.n_tets, rng.uniform(0.2, 1.0))) for m in meshes]


def _serve_requests(case, seed):
    size, rng = np.random.default_rng(case["mesh_seed"]), np.random.default_rng(seed)
    reqs = []
    for _ in range(case["count"]):
        tets = float(np.exp(size.uniform(np.log(1e3), np.log(case["t_max"]))))
        frames, tendon = int(size.integers(1, case["frames_max"] + 1)), float(size.uniform(0.0, 0.2))
        m = _muscle(tets, tendon, int(rng.integers(1 << 31)))
        ramp = rng.uniform(0.3, 1.0) * np.arange(1, frames + 1) / frames
        reqs.append((m, ramp[:, None] * m.activations))
    return reqs


def _arm(case, seed):
    mesh = arm_assembly(case["bone_w"], case["bone_len"], case["r0"], frames=2)
    return mesh, np.random.default_rng(seed).uniform(0.3, 0.8) * mesh.activations[1]


def _unit(case, seed):
    rng = np.random.default_rng(seed)
    return _jittered(_muscle(case["tets"], 0.1, int(rng.integers(1 << 31))), case["jitter"], rng), rng


def _attachments(mesh, rng):
    """Origin: the lower end; insertion: the part of the upper end on one side of a seeded line."""
    z, mid = mesh.rest_pos[:, 2], mesh.rest_pos[:, :2].mean(axis=0)
    half, side = 0.3 * mesh.meta["h"], rng.normal(size=2)
    upper = z >= mesh.meta["nz"] * mesh.meta["h"] - half
    far = (mesh.rest_pos[:, :2] - mid) @ side >= 0.0
    return np.nonzero(z <= half)[0].astype(np.int32), np.nonzero(upper & far)[0].astype(np.int32)


def _gradients(mesh, rng):
    """Deformation gradients such as a caller has them: a bend and a twist of the mesh, and a part of each tet's own."""
    x = torch.tensor(mesh.rest_pos[mesh.tets].mean(axis=1), device=DEVICE)
    t = x / x[:, 2].max()
    a, b = (float(rng.uniform(0.2, 0.6)) for _ in range(2))
    own = torch.from_numpy(rng.normal(scale=0.05, size=(mesh.n_tets, 3, 3))).to(DEVICE)
    th = a * t[:, 2]
    R = torch.zeros_like(own)
    R[:, 0, 0] = R[:, 1, 1] = torch.cos(th)
    R[:, 1, 0] = torch.sin(th)
    R[:, 0, 1] = -R[:, 1, 0]
    R[:, 2, 2] = 1.0
    R[:, 0, 2] = b * t[:, 2]
    return (R + own).contiguous()


def _solver(mesh, stream=True, **params):
    st = torch.cuda.Stream() if stream else None
    s = emu.Solver(mesh, emu.Params(**params), stream=st.cuda_stream if st else None)
    return s, st


def _params(case):
    p = dict(precision=emu.PRECISION_MIXED if case["precision"] == "mixed" else emu.PRECISION_FP64)
    return dict(p, tol_rel_residual=case["tol"], form=emu.FORM_F if case["form"] == "f" else emu.FORM_RS)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "frames":
        mesh, acts = _frames_mesh(case, seed)
        solver, stream = _solver(mesh, case["own_stream"], **_params(case))
        return dict(kind=kind, solver=solver, stream=stream, acts=acts, single=case["precision"] == "mixed")
    if kind == "batch":
        meshes = _batch_meshes(case, seed)
        made = [_solver(m, precision=emu.PRECISION_MIXED) for m, _ in meshes]
        for (s, _), (_, a) in zip(made, meshes):
            s.set_activation(a)
        return dict(kind=kind, solvers=[s for s, _ in made], streams=[t for _, t in made])
    if kind == "serve":
        server = emu.Server(120 << 30, emu.Params(precision=emu.PRECISION_MIXED))
        return dict(kind=kind, server=server, requests=_serve_requests(case, seed))
    if kind == "arm":
        mesh, act = _arm(case, seed)
        solver, stream = _solver(mesh, precision=emu.PRECISION_MIXED, tol_rel_residual=case["tol"])
        return dict(kind="frames", solver=solver, stream=stream, acts=act[None, :], single=True)
    mesh, rng = _unit(case, seed)
    if kind == "coupling":
        precision = emu.PRECISION_MIXED if case["precision"] == "mixed" else emu.PRECISION_FP64
        solver, stream = _solver(mesh, precision=precision, pcg_tol=1e-12)
        F = _gradients(mesh, rng)
        q = torch.empty((mesh.n_verts, 3), dtype=torch.float64, device=DEVICE)
        torch.cuda.synchronize()
        return dict(kind=kind, solver=solver, stream=stream, F=F, q=q)
    origin, insertion = _attachments(mesh, rng)
    return dict(kind=kind, rest=mesh.rest_pos, tets=mesh.tets, origin=origin, insertion=insertion)


# ---------------------------------------------------------------- a pass ----

def run(state):
    kind = state["kind"]
    if kind == "frames":
        s, out = state["solver"], []
        s.reset()
        for a in state["acts"]:
            s.set_activation(a)
            s.solve()
            q = s.positions()
            out.append(q.astype(np.float32) if state["single"] else q)
        return out
    if kind == "batch":
        for s in state["solvers"]:
            s.reset()
        emu.batch_solve(state["solvers"])
        return [s.positions().astype(np.float32) for s in state["solvers"]]
    if kind == "serve":
        server, reqs = state["server"], state["requests"]
        for i, (mesh, acts) in enumerate(reqs):
            server.submit(mesh, acts, i)
        left = len(reqs)
        while left:
            done = len(server.poll())
            left -= done
            if not done:
                time.sleep(2e-4)
        return [server.result(i)[0].astype(np.float32) for i in range(len(reqs))]
    if kind == "coupling":
        rc = state["solver"].acap_solve_noalloc(state["F"].data_ptr(), state["q"].data_ptr())
        if rc:
            raise RuntimeError("acap_solve_noalloc: status %d" % rc)
        return state["q"]
    return emu.fiber_field(state["rest"], state["tets"], state["origin"], state["insertion"])


# ------------------------------------------------------------------ work ----

def _frame_work(n, m, frames, wide=False):
    """One quasi-Newton iteration's unavoidable traffic and arithmetic per frame, times the 20 iterations that a
    frame takes at the least: per tet the mode gradients (48), the geometry and material (26) and the state (10) are
    read and the state is written; per vertex positions. The 6 x 48 by 48 capacitance product is the arithmetic."""
    w = 8 if wide else 4
    return dict(bytes=20.0 * frames * (m * w * (48 + 26 + 20) + n * 72) + 48.0 * frames * n,
                flops=20.0 * frames * m * 2.0 * 6 * 48 * 24)


def work(case):
    kind = case["kind"]
    if kind == "frames":
        if case["mesh"] == "beam":
            m, n = 6 * case["nx"] * case["ny"] * case["nz"], (case["nx"] + 1) * (case["ny"] + 1) * (case["nz"] + 1)
        else:
            m, n = case["tets"], 0.21 * case["tets"]
        return _frame_work(n, m, case["frames"], case["precision"] == "fp64")
    if kind == "batch":
        sizes = [(x.n_verts, x.n_tets, 1) for x in batch_set(case["count"], seed=case["mesh_seed"], t_max=case["t_max"])]
    elif kind == "serve":
        sizes = [(x.n_verts, x.n_tets, a.shape[0]) for x, a in _serve_requests(case, 0)]
    elif kind == "arm":
        x = arm_assembly(case["bone_w"], case["bone_len"], case["r0"], frames=1)
        sizes = [(x.n_verts, x.n_tets, 1)]
    else:  # one sweep over the operator: tets and F or positions read, positions or fibers written
        n, m = 0.21 * case["tets"], case["tets"]
        return dict(bytes=m * (16.0 + 72.0) + n * 24.0, flops=m * 100.0)
    parts = [_frame_work(*x) for x in sizes]
    return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}


# ----------------------------------------------------- the same in 64 bits ----

def _det3(A):
    return (A[..., 0, :] * torch.linalg.cross(A[..., 1, :], A[..., 2, :])).sum(-1)


def _inv3(A):
    a, b, c = A[..., 0, :], A[..., 1, :], A[..., 2, :]
    cof = torch.stack([torch.linalg.cross(b, c), torch.linalg.cross(c, a), torch.linalg.cross(a, b)], dim=-1)
    return cof / _det3(A)[..., None, None]


def _inv9(H):
    """(H^-1, positive definite?) of symmetric 9 x 9 matrices, by Gauss-Jordan elimination without pivoting."""
    H, good = H.clone(), torch.ones(len(H), dtype=torch.bool, device=H.device)
    for k in range(9):
        p = H[:, k, k].clone()
        good &= p > 0
        row, col = H[:, k, :] / p[:, None], H[:, :, k].clone()
        H -= col[:, :, None] * row[:, None, :]
        H[:, k, :] = row
        H[:, :, k] = -col / p[:, None]
        H[:, k, k] = 1.0 / p
    return H, good


class _Mesh64:
    """A mesh's operators in plain float64 torch: gradients per tet, their transpose, and CG on their products."""

    def __init__(self, rest, tets, fixed):
        self.Q = torch.tensor(rest, dtype=torch.float64, device=DEVICE)
        self.T = torch.tensor(np.asarray(tets, dtype=np.int64), device=DEVICE)
        Dm = (self.Q[self.T[:, :3]] - self.Q[self.T[:, 3:]]).transpose(1, 2)
        self.V = self.w = _det3(Dm).abs() / 6.0
        Di = _inv3(Dm)  # rows: gradients of the first three shape functions
        self.N = torch.cat([Di, -Di.sum(dim=1, keepdim=True)], dim=1)
        self.free = torch.ones(len(self.Q), 1, dtype=torch.float64, device=DEVICE)
        self.free[torch.tensor(np.asarray(fixed, dtype=np.int64), device=DEVICE)] = 0.0
        self.diag = torch.zeros_like(self.free).index_add_(
            0, self.T.reshape(-1), (self.w[:, None] * (self.N ** 2).sum(dim=2)).reshape(-1, 1))

    def G(self, q):
        return (q[self.T][:, :, :, None] * self.N[:, :, None, :]).sum(1)

    def Gt(self, X):
        y = (self.N[:, :, None, :] * X[:, None, :, :]).sum(3)
        return torch.zeros(len(self.Q), y.shape[2], dtype=torch.float64, device=DEVICE).index_add_(
            0, self.T.reshape(-1), y.reshape(-1, y.shape[2])) * self.free

    def cg(self, apply, b, tol, most=8000):
        """x with apply(x) = b on the free vertices, to |r| <= tol |b|, or to where the curvature turns negative."""
        x, r = torch.zeros_like(b), b * self.free
        z = r / self.diag
        p, rz, stop, on = z, (r * z).sum(), float((r * r).sum()) * tol * tol, torch.ones((), device=DEVICE).bool()
        for k in range(most):
            if k % 32 == 0 and (float((r * r).sum()) <= stop or not bool(on)):
                break
            Ap = apply(p)
            pAp = (p * Ap).sum()
            on = on & (pAp > 0) & (rz > 0)
            a = torch.where(on, rz / pAp, torch.zeros_like(rz))
            if k == 0:
                a = torch.where(pAp > 0, a, torch.ones_like(rz))
            x, r = x + a * p, r - a * Ap
            z = r / self.diag
            new = (r * z).sum()
            p = z + torch.where(on, new / rz, torch.zeros_like(rz)) * p
            rz = new
        return x

    def laplace(self, b, tol=1e-14):
        return self.cg(lambda x: self.Gt(self.w[:, None, None] * self.G(x)), b, tol)


class _Muscle64:
    """The muscle of a mesh in 64 bits: its energy over positions and gradients, minimised by Newton's method on both
    together (the tets' gradients eliminated, conjugate gradients on the positions)."""

    def __init__(self, mesh):
        self.g = g = _Mesh64(mesh.rest_pos, mesh.tets, mesh.fixed_verts)
        E, nu = (torch.tensor(np.asarray(v)[mesh.material_id], device=DEVICE) for v in (mesh.youngs, mesh.poisson))
        self.mu, self.lam = E / (2 * (1 + nu)), E * nu / ((1 + nu) * (1 - 2 * nu))
        self.ref = float(self.mu.min())
        self.c = self.ref * g.w  # alpha w, alpha = the smallest shear modulus
        u = torch.tensor(mesh.fiber_dir, device=DEVICE)
        self.u = u / u.norm(dim=1, keepdim=True)
        self.nu = torch.zeros(len(g.T), 3, 3, dtype=torch.float64, device=DEVICE)
        if mesh.f_ext is not None:
            self.nu = g.w[:, None, None] * g.G(g.laplace(torch.tensor(mesh.f_ext, device=DEVICE) * g.free))
        self.q, self.a = g.Q.clone(), np.zeros(len(g.T))
        self.F = torch.eye(3, dtype=torch.float64, device=DEVICE).repeat(len(g.T), 1, 1)

    def energy(self, q, F, ka):
        D, J = F - self.g.G(q), _det3(F)
        lnJ = torch.log(J.clamp(min=1e-300))
        psi = 0.5 * self.mu * ((F * F).sum((1, 2)) - 3) - self.mu * lnJ + 0.5 * self.lam * lnJ ** 2
        psi = psi + ka * ((F @ self.u[:, :, None]) ** 2).sum((1, 2))
        e = self.g.V * psi + 0.5 * self.c * (D * D).sum((1, 2)) - (F * self.nu).sum((1, 2))
        return float(torch.where((J > 0).all(), e.sum(), torch.full_like(e[0], float("inf"))))

    def solve(self, a):
        """Positions at activation ``a``, reached in small steps of it; None if Newton's method does not converge."""
        steps = max(1, int(np.ceil(np.abs(a - self.a).max() / 0.1)))
        for k in range(1, steps + 1):
            if not self.newton(self.a + (a - self.a) * (k / steps), 1e-13 if k == steps else 1e-3):
                return None
        self.a = a
        return self.q.cpu().numpy()

    def newton(self, a, tol):
        g, ka = self.g, self.ref * torch.tensor(a, device=DEVICE)
        V, c, I9 = g.V, self.c, torch.eye(9, dtype=torch.float64, device=DEVICE)
        uu = torch.einsum("mi,mj->mij", self.u, self.u)
        fib = torch.einsum("ab,mij->maibj", torch.eye(3, dtype=torch.float64, device=DEVICE), uu).reshape(-1, 9, 9)
        first, best = None, float("inf")
        for _ in range(60):
            F = self.F
            Fi, lnJ = _inv3(F), torch.log(_det3(F))
            FiT = Fi.transpose(1, 2)
            P = self.mu[:, None, None] * (F - FiT) + (self.lam * lnJ)[:, None, None] * FiT
            P = P + 2 * ka[:, None, None] * (F @ uu)
            D = c[:, None, None] * (F - g.G(self.q))
            gF, gq = V[:, None, None] * P + D - self.nu, -g.Gt(D)
            size = float(gF.norm()) + float(gq.norm()) / float(g.N.abs().max())
            first = size if first is None else max(first, size)
            if size <= tol * first or (size <= 1e-11 * first and size > 0.5 * best):
                return True
            best = min(best, size)
            T = torch.einsum("mjr,msi->mijrs", Fi, Fi).reshape(-1, 9, 9)  # d(-F^-T)_ij / dF_rs
            f = FiT.reshape(-1, 9)
            H = self.mu[:, None, None] * I9 + (self.mu - self.lam * lnJ)[:, None, None] * T
            H = H + self.lam[:, None, None] * f[:, :, None] * f[:, None, :]
            H = V[:, None, None] * (H + 2 * ka[:, None, None] * fib) + c[:, None, None] * I9
            Hi, good = _inv9(H)
            shift = 0.5 * (V * self.mu + c)
            for _ in range(20):  # definite again where it is not
                if bool(good.all()):
                    break
                H = torch.where(good[:, None, None], H, H + shift[:, None, None] * I9)
                Hi, good = _inv9(H)
            S = c[:, None, None] * I9 - (c ** 2)[:, None, None] * Hi
            y = (Hi @ gF.reshape(-1, 9, 1)).reshape(-1, 3, 3)
            rhs = -gq - g.Gt(c[:, None, None] * y)
            near = max(1e-10, min(1e-2, 1e-2 * size / first))
            dq = g.cg(lambda x: g.Gt((S * g.G(x).reshape(-1, 1, 9)).sum(2).reshape(-1, 3, 3)), rhs, near)
            dF = (Hi @ (c[:, None, None] * g.G(dq)).reshape(-1, 9, 1)).reshape(-1, 3, 3) - y
            e0, s = self.energy(self.q, F, ka), 1.0
            if size > 1e-6 * first:
                while s > 1e-6 and not self.energy(self.q + s * dq, F + s * dF, ka) <= e0:
                    s *= 0.5
            self.q, self.F = self.q + s * dq, F + s * dF
        return False


def exact(case, seed):
    kind = case["kind"]
    if kind == "frames":
        mesh, acts = _frames_mesh(case, seed)
        if mesh.n_tets * len(acts) > 30000:  # takes too long
            return None
        m = _Muscle64(mesh)
        return [m.solve(a) for a in acts]
    if kind == "batch":
        return [_Muscle64(m).solve(a) if m.n_tets < 2000 else None for m, a in _batch_meshes(case, seed)]
    if kind == "serve":
        every = [(_Muscle64(m), acts) if m.n_tets < 4000 else None for m, acts in _serve_requests(case, seed)]
        every = [[x[0].solve(a) for a in x[1]] if x else [None] for x in every]
        return [None if any(q is None for q in x) else np.stack(x) for x in every]
    if kind == "arm":  # the constrained problem (rigid parts, joint rows, slacks) has no short plain form
        return None
    mesh, rng = _unit(case, seed)
    if kind == "coupling":
        g = _Mesh64(mesh.rest_pos, mesh.tets, mesh.fixed_verts)
        F = _gradients(mesh, rng)
        base = g.Q * (1.0 - g.free)
        b = g.Gt(g.w[:, None, None] * (F - g.G(base)))
        return base + g.laplace(b)
    origin, insertion = _attachments(mesh, rng)
    g = _Mesh64(mesh.rest_pos, mesh.tets, np.concatenate([origin, insertion]))
    base = torch.zeros(mesh.n_verts, 1, dtype=torch.float64, device=DEVICE)
    base[torch.tensor(origin.astype(np.int64), device=DEVICE)] = -1.0
    base[torch.tensor(insertion.astype(np.int64), device=DEVICE)] = 1.0
    f = base + g.laplace(-g.Gt(g.w[:, None, None] * g.G(base)))
    grad = g.G(f)[:, 0, :]
    return (grad / grad.norm(dim=1, keepdim=True)).cpu().numpy()
