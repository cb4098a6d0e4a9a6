"""Performance cases of the lattice library: the calls that a load-path program makes, one per case.

Every case runs on one of the two reference cells of ``latgen`` (the 2D ring cell and the 3D
edge-strut cell), tiled to a lattice whose per-cell shear-modulus factors theta_s ~ U[0.9, 1.1]
come from the seed.  ``path`` names the call:

  load_step   one load step from its predictor to convergence (solve_load_path)
  newton_it   one Newton iteration from the predictor of a load step (newton_step)
  solve       one tangent system (tangent_solve) with the solver already prepared
  precond     the FETI-DP preconditioner set up and applied once (lattice_prepare_solver, feti_apply)
  select      principal cells and coefficients at a state (select_principal_cells)
  residual    internal forces of every cell and the assembled residual (assemble_residual_tangent)
  tangent     full-rule local tangents of every cell (assemble_residual_tangent)
  apply       the reduced tangent action on cell vectors (apply_reduced_tangent)
  adjoint     the adjoint gradient at a converged state (adjoint_gradient)

``exact`` restates each path in plain torch at 64 bits; paths that need a linear solve are
restated with a dense one, on lattices small enough for it.
"""
import functools
import math

import torch

import latgen
from paper_2603_10741_gb300 import LAT_FP64, LAT_MIXED_BF16, LAT_MIXED_FP32, Lattice, solve_load_path

MODES = {"fp64": LAT_FP64, "fp32": LAT_MIXED_FP32, "bf16": LAT_MIXED_BF16}
MU, LAM = 1.0, 4.0          # Lame parameters of every named load case (nu = 0.4)
STRUT_RADIUS = 0.15         # half-width of the edge struts of the strut load cases
DENSE_DOF = 10000           # largest lattice that exact() solves with a dense matrix


def _case(name, path, cell, res, dims, mode, **more):
    nx, ny, nz = tuple(dims) + (0,) * (3 - len(dims))
    c = {"path": path, "cell": cell, "res": res, "nx": nx, "ny": ny, "nz": nz, "mode": mode}
    if name:
        c["name"] = name
    c.update(more)
    return c


def listed():
    return [
        # the smallest call in use: a load step of a 4 x 4 ring lattice, all launches and round trips
        _case("load_step ring 4x4 fp64", "load_step", "ring", 8, (4, 4), "fp64"),
        # a load step of the 32 x 32 ring lattice (556k DOF) as its load path runs it, FP32 mode
        _case("load_step ring 32x32 fp32", "load_step", "ring", 16, (32, 32), "fp32"),
        # a Newton iteration on a strut lattice of ragged dims, tensor-core preconditioner: residual,
        # selection, preconditioner setup, Krylov solve and line search
        _case("newton_it strut 7x6x5 bf16", "newton_it", "strut", 12, (7, 6, 5), "bf16"),
        # the linear solve inside a Newton iteration of the 10^3 strut lattice (1.76 M DOF)
        _case("solve strut 10x10x10 bf16", "solve", "strut", 12, (10, 10, 10), "bf16"),
        # the same with everything FP64, the mode that tests and references run in
        _case("solve strut 4x3x3 fp64", "solve", "strut", 12, (4, 3, 3), "fp64"),
        # preconditioner setup at a new state: local inverses, coarse factorisation, one application
        _case("precond strut 8x8x8 fp64", "precond", "strut", 12, (8, 8, 8), "fp64"),
        # selection on the 32 x 32 ring lattice: snapshots, Algorithm 1 up to a cap, principal tangents
        _case("select ring 32x32 fp64", "select", "ring", 16, (32, 32), "fp64", n_r=8),
        # a residual evaluation, as every line-search trial makes, on a strut lattice of odd dims
        _case("residual strut 13x11x9 fp64", "residual", "strut", 12, (13, 11, 9), "fp64"),
        # local tangents of every cell (what the plain full-tangent path evaluates)
        _case("tangent ring 32x32 fp64", "tangent", "ring", 16, (32, 32), "fp64"),
        # the action inside the mixed modes' Krylov solve, and the FP64 one of the outer solve
        _case("apply strut 12x12x12 fp32", "apply", "strut", 12, (12, 12, 12), "fp32", n_r=1),
        _case("apply strut 9x9x7 fp64", "apply", "strut", 12, (9, 9, 7), "fp64", n_r=4),
        # the gradient of the end compliance with respect to theta
        _case("adjoint ring 8x8 fp64", "adjoint", "ring", 8, (8, 8), "fp64"),
    ]


def draw(rng):
    def ring(lo, hi, res=(8, 16)):
        n = round(math.exp(rng.uniform(math.log(lo), math.log(hi))))
        m = min(hi, max(lo, round(n * rng.uniform(0.7, 1.3))))
        return rng.choice(res), (n, m)

    def strut(lo, hi):
        n = math.exp(rng.uniform(math.log(lo), math.log(hi)))
        return tuple(min(hi, max(lo, round(n * rng.uniform(0.8, 1.2)))) for _ in range(3))

    path = rng.choice(["load_step", "newton_it", "solve", "precond", "select", "residual", "tangent", "apply", "adjoint"])
    flat = rng.random() < 0.4
    if path == "load_step":
        res, dims = ring(3, 32)
        return _case(None, path, "ring", res, dims, rng.choice(["fp64", "fp32", "bf16"]))
    if path == "newton_it":
        return _case(None, path, "strut", 12, strut(3, 6), "bf16")
    if path == "solve":
        if flat:
            res, dims = ring(6, 32)
            return _case(None, path, "ring", res, dims, rng.choice(["fp64", "fp32", "bf16"]))
        mode = rng.choice(["fp64", "bf16"])
        return _case(None, path, "strut", 12, strut(2, 3) if mode == "fp64" else strut(3, 9), mode)
    if path == "precond":
        if flat:
            res, dims = ring(6, 32)
            return _case(None, path, "ring", res, dims, "fp64")
        return _case(None, path, "strut", 12, strut(3, 8), "fp64")
    if path == "select":
        res, dims = ring(6, 32)
        return _case(None, path, "ring", res, dims, "fp64", n_r=rng.randint(2, 12))
    if path in ("residual", "tangent"):
        if flat:
            res, dims = ring(4, 32)
            return _case(None, path, "ring", res, dims, "fp64")
        return _case(None, path, "strut", 12, strut(2, 10 if path == "residual" else 8), "fp64")
    if path == "apply":
        mode, n_r = rng.choice(["fp64", "fp32"]), rng.choice([1, 2, 3, 5, 8, 16])
        if flat:
            res, dims = ring(6, 32)
            return _case(None, path, "ring", res, dims, mode, n_r=n_r)
        return _case(None, path, "strut", 12, strut(2, 11 if n_r <= 4 else 7), mode, n_r=n_r)
    res, dims = ring(3, 10, (8,))
    return _case(None, path, "ring", res, dims, "fp64")


# ------------------------------------------------------------------------------------------------
# inputs
# ------------------------------------------------------------------------------------------------


def _dims(case):
    return (case["nx"], case["ny"]) if case["cell"] == "ring" else (case["nx"], case["ny"], case["nz"])


@functools.lru_cache(maxsize=4)
def _geometry(cell, res, dims):
    Xr, E = latgen.ring_cell(res) if cell == "ring" else latgen.strut_cell(res, STRUT_RADIUS)
    return latgen.tile(Xr, E, dims)


def _load_case(case, seed):
    """A load path of small steps: 1 % compression per step in 2D as in the ring load cases, 0.1 %
    in 3D, where the affine predictor of a larger first step is strongly indefinite."""
    lat = _geometry(case["cell"], case["res"], _dims(case))
    ring = case["cell"] == "ring"
    return latgen.LoadCase(name=case["path"], lattice=lat, mu=MU, lam=LAM, mu_scale=latgen.mu_scale(lat.n_cells, seed),
                           total_strain=0.1 if ring else 0.01, n_steps=10, eps=3e-4 if ring else 5e-3)


def _smooth(lat, amplitude, seed):
    """A sum of low sine modes over the lattice, [n_nodes * d], zero on the clamped faces."""
    g = torch.Generator().manual_seed(seed)
    X = torch.tensor(lat.X, device="cuda") / torch.tensor(lat.dims, dtype=torch.float64, device="cuda")
    u = torch.zeros_like(X)
    for _ in range(4):
        k = torch.randint(1, 4, (lat.dim,), generator=g).double().cuda()
        ph = (2 * math.pi * torch.rand(lat.dim, generator=g, dtype=torch.float64)).cuda()
        ph[lat.load_axis] = 0.0
        amp = (2 * torch.rand(lat.dim, generator=g, dtype=torch.float64) - 1).cuda()
        u += amp * torch.sin(math.pi * X * k + ph).prod(dim=1, keepdim=True)
    return (amplitude * u).reshape(-1)


def _state(lc, seed):
    """Displacement state of the single-call cases: the affine predictor of the first load step and
    a smooth deviation from it, of a few per cent strain in 2D and a tenth of the step's in 3D."""
    lat = lc.lattice
    load = lc.top_displacement(1)
    u = _smooth(lat, (0.5 if lat.dim == 2 else 0.05) * abs(load), seed)
    u[lat.load_axis::lat.dim] += load / lat.height * torch.tensor(lat.X[:, lat.load_axis], device="cuda")
    return u


def _principals(lc, n_r, seed):
    n = lc.lattice.n_cells
    g = torch.Generator().manual_seed(seed + 1)
    S = torch.randperm(n, generator=g)[:n_r].to(torch.int32)
    a = -torch.log(torch.rand((n_r, n), generator=g, dtype=torch.float64).clamp_min(1e-12))
    return S, a / a.sum(dim=0)


def _uniform(shape, seed, dtype=torch.float64):
    g = torch.Generator(device="cuda").manual_seed(seed + 2)
    return (2 * torch.rand(shape, generator=g, dtype=torch.float64, device="cuda") - 1).to(dtype)


def _rhs(lc, seed):
    """A smooth body-force-like right-hand side with some per-DOF variation."""
    f = _smooth(lc.lattice, 1.0, seed + 3)
    return f + 0.1 * _uniform(f.shape, seed)


def _n_r(case, lc):
    return min(case.get("n_r", 1), lc.lattice.n_cells)


def prepare(case, seed):
    lc = _load_case(case, seed)
    lat = Lattice.from_case(lc, MODES[case["mode"]])
    st = {"case": case, "lc": lc, "lat": lat}
    path = case["path"]
    if path == "load_step":
        # to 1e-11, so that the state does not depend on where the last iteration stops
        st["opts"] = lat.lattice_default_opts(newton_rtol=1e-11, eps=lc.eps)
        return st
    if path == "adjoint":
        st["opts"] = lat.lattice_default_opts(newton_rtol=1e-12, eps=lc.eps)
        st["u"], _ = solve_load_path(lat, lc, st["opts"], steps=1)
        return st
    if path == "newton_it":
        st["opts"] = lat.lattice_default_opts(eps=lc.eps, krylov_rtol=1e-12)
        return st
    st["u"] = _state(lc, seed)
    if path in ("solve", "precond"):
        st["opts"] = lat.lattice_default_opts(eps=lc.eps, krylov_rtol=1e-12)
        lat.select_principal_cells(st["u"], lc.eps, 32)
    if path == "solve":
        lat.lattice_prepare_solver(st["u"], st["opts"])
        st["rhs"] = _rhs(lc, seed)
    elif path == "precond":
        st["v"] = lat.feti_from_global(_rhs(lc, seed))
    elif path == "apply":
        S, alpha = _principals(lc, _n_r(case, lc), seed)
        lat.set_principal_cells(st["u"], S, alpha)
        s = lat.sizes
        st["x"] = _uniform((s.n_loc, s.n_cells), seed, torch.float64 if case["mode"] == "fp64" else torch.float32)
        st["y"] = torch.empty_like(st["x"])
    return st


def run(st):
    lat, path = st["lat"], st["case"]["path"]
    if path == "load_step":
        u, _ = solve_load_path(lat, st["lc"], st["opts"], steps=1)
        return u
    if path == "newton_it":
        u = lat.lattice_predictor(st["lc"].top_displacement(1))
        lat.newton_step(u, st["opts"], max_iterations=1)
        return u
    if path == "solve":
        x, _, _ = lat.tangent_solve(st["rhs"], st["opts"])
        return x
    if path == "precond":
        lat.lattice_prepare_solver(st["u"], st["opts"])
        return lat.feti_apply(1, st["v"])
    if path == "select":
        # a tolerance that the cap of n_r principals always meets first: one output shape for all seeds
        sel = lat.select_principal_cells(st["u"], 1e-3 * st["lc"].eps, st["case"]["n_r"])
        return {"S": sel["S"], "alpha": sel["alpha"], "Kp": sel["Kp"]}
    if path == "residual":
        out = lat.assemble_residual_tangent(st["u"], local_forces=True)
        return {"r": out["r"], "f": out["f"], "min_detF": out["min_detF"]}
    if path == "tangent":
        return lat.assemble_residual_tangent(st["u"], residual=False, tangent=True)["K"]
    if path == "apply":
        return lat.apply_reduced_tangent(st["x"], st["y"])
    g, J, _ = lat.adjoint_gradient(st["u"], st["opts"])
    return {"grad": g, "J": J}


# ------------------------------------------------------------------------------------------------
# work
# ------------------------------------------------------------------------------------------------


def work(case):
    lat = _geometry(case["cell"], case["res"], _dims(case))
    d, ns, nn, ne = lat.dim, lat.n_cells, lat.X_ref.shape[0], lat.elems.shape[0]
    nen, nloc, ndof = 1 << d, nn * d, lat.n_nodes * d
    nnz = _pattern(lat)[0].numel() * d * d
    path = case["path"]
    qp_grad = 2 * nen * d * d                      # one contraction of nodal values with gradients
    qp_law = 25 if d == 2 else 80                  # inverse, logarithm and stress at a point
    res_flops = ns * ne * (1 << d) * (2 * qp_grad + qp_law)
    tan_point = qp_grad + qp_law + qp_grad + nen * nen * (2 * d + 4 * d * d)
    act_flops = 2.0 * nnz * ns
    if path == "residual":
        return {"bytes": 8.0 * (2 * ndof + nloc * ns) + 4.0 * nn * ns, "flops": float(res_flops)}
    if path == "tangent":
        return {"bytes": 8.0 * (ndof + nnz * ns) + 4.0 * nn * ns, "flops": float(ns * ne * nen * tan_point)}
    if path == "select":
        # snapshots of all cells, and Algorithm 1's pass over them for the first principal
        return {"bytes": 8.0 * (ndof + nnz * ns), "flops": float(ns * ne * tan_point + 6.0 * nnz * ns)}
    if path == "apply":
        n_r, b = min(case.get("n_r", 1), ns), 8 if case["mode"] == "fp64" else 4
        return {"bytes": float(b * (2 * nloc * ns + n_r * (ns + nnz))), "flops": n_r * act_flops}
    n_P = nen * d
    n_R = nloc - n_P
    if path == "precond":
        # three boundary classes of one principal inverted, one product with the inverses
        return {"bytes": 8.0 * (2 * nloc * ns + 3 * n_R * n_R), "flops": 3 * 2.0 * n_R ** 3 + 2.0 * (n_R + n_P) * n_R * ns}
    if path == "solve":
        # one operator and one preconditioner application of an iteration
        return {"bytes": 8.0 * 2 * ndof, "flops": act_flops + 2.0 * (n_R + n_P) * n_R * ns}
    # a Newton iteration: two residuals, snapshots, and one Krylov iteration; the adjoint alike
    return {"bytes": 8.0 * 2 * ndof,
            "flops": 2.0 * res_flops + ns * ne * tan_point + act_flops + 2.0 * (n_R + n_P) * n_R * ns}


# ------------------------------------------------------------------------------------------------
# the same in plain torch, 64 bits
# ------------------------------------------------------------------------------------------------


def _pattern(lat):
    """Sorted node pairs (a * nn + b) that share an element, and each element pair's index."""
    E = torch.tensor(lat.elems)
    key = (E[:, :, None] * lat.X_ref.shape[0] + E[:, None, :]).reshape(-1)
    pairs, inv = torch.unique(key, sorted=True, return_inverse=True)
    return pairs, inv


class _Plain:
    def __init__(self, lc):
        lat = lc.lattice
        self.lat, self.d, self.nn, self.ns = lat, lat.dim, lat.X_ref.shape[0], lat.n_cells
        self.E = torch.tensor(lat.elems, device="cuda")
        self.cn = torch.tensor(lat.cell_nodes, device="cuda")
        self.mu = MU * torch.tensor(lc.mu_scale, device="cuda")
        pairs, inv = _pattern(lat)
        self.pa, self.pb = (pairs // self.nn).cuda(), (pairs % self.nn).cuda()
        self.inv, self.n_blk = inv.cuda(), pairs.numel()
        self.rule = [self._rule(False), self._rule(True)]
        k = torch.arange(self.d, device="cuda")
        self.ldof = (self.cn[:, :, None] * self.d + k).reshape(self.ns, -1)
        self.n_dof = lat.n_nodes * self.d
        fixed = torch.zeros((lat.n_nodes, self.d), dtype=torch.bool)
        fixed[lat.bottom_nodes()] = True
        fixed[lat.top_nodes()] = True
        self.fixed = fixed.reshape(-1).cuda()

    def _rule(self, reduced):
        d = self.d
        xi = torch.tensor([[-1, -1], [1, -1], [1, 1], [-1, 1]], dtype=torch.float64)
        if d == 3:
            xi = torch.cat([torch.cat([xi, torch.full((4, 1), z, dtype=torch.float64)], 1) for z in (-1.0, 1.0)])
        pts = torch.zeros((1, d), dtype=torch.float64) if reduced else xi / math.sqrt(3.0)
        w = 2.0 ** d if reduced else 1.0
        one = 1 + xi[None] * pts[:, None]                                    # [q, a, d]
        dphi = torch.stack([xi[None, :, k] * torch.cat([one[..., :k], one[..., k + 1:]], -1).prod(-1)
                            for k in range(d)], -1) / 2 ** d
        xe = torch.tensor(self.lat.X_ref)[torch.tensor(self.lat.elems)]      # [e, a, d]
        J0 = torch.einsum("eak,qal->eqkl", xe, dphi)
        grad = torch.einsum("qal,eqlk->eqak", dphi, torch.linalg.inv(J0))
        return grad.cuda(), (w * torch.linalg.det(J0)).cuda()

    def _points(self, u, cells, reduced):
        g, W = self.rule[int(reduced)]
        ue = u[self.ldof[cells]].reshape(len(cells), self.nn, self.d)[:, self.E]
        F = torch.einsum("seai,eqak->seqik", ue, g) + torch.eye(self.d, dtype=torch.float64, device="cuda")
        return g, W, F, torch.linalg.inv(F), torch.linalg.det(F)

    def forces(self, u, mu=None, lam=LAM):
        """Local internal forces [n_loc, n_cells] and the smallest det F."""
        out = torch.empty((self.nn * self.d, self.ns), dtype=torch.float64, device="cuda")
        least = math.inf
        mu = self.mu if mu is None else mu
        for c in torch.arange(self.ns, device="cuda").split(64):
            g, W, F, Fi, J = self._points(u, c, False)
            least = min(least, float(J.min()))
            FiT = Fi.transpose(-1, -2)
            P = mu[c][:, None, None, None, None] * (F - FiT) + (lam * J.log())[..., None, None] * FiT
            fe = torch.einsum("seqik,eqak,eq->seai", P, g, W)
            f = torch.zeros((len(c), self.nn, self.d), dtype=torch.float64, device="cuda")
            f.index_add_(1, self.E.reshape(-1), fe.reshape(len(c), -1, self.d))
            out[:, c] = f.reshape(len(c), -1).T
        return out, least

    def tangents(self, u, cells, reduced=False):
        """Local tangents on the pattern, [n, n_blk * d * d]."""
        out = torch.empty((len(cells), self.n_blk * self.d ** 2), dtype=torch.float64, device="cuda")
        eye = torch.eye(self.d, dtype=torch.float64, device="cuda")
        for at in torch.arange(len(cells), device="cuda").split(32):
            c = cells[at]
            g, W, F, Fi, J = self._points(u, c, reduced)
            h = torch.einsum("seqki,eqak->seqai", Fi, g)
            cg = W * (self.mu[c][:, None, None] - LAM * J.log())
            Ke = torch.einsum("eq,seqai,seqbj->seabij", LAM * W, h, h)
            Ke += torch.einsum("seq,seqbi,seqaj->seabij", cg, h, h)
            gg = torch.einsum("eq,eqak,eqbk->eab", W, g, g)
            Ke += (self.mu[c][:, None, None, None] * gg)[..., None, None] * eye
            K = torch.zeros((len(c), self.n_blk, self.d, self.d), dtype=torch.float64, device="cuda")
            K.index_add_(1, self.inv, Ke.reshape(len(c), -1, self.d, self.d))
            out[at] = K.reshape(len(c), -1)
        return out

    def scatter(self, loc):
        r = torch.zeros(self.n_dof, dtype=torch.float64, device="cuda")
        return r.index_add_(0, self.ldof.reshape(-1), loc.T.reshape(-1))

    def local_dense(self, vals):
        M = torch.zeros((self.nn, self.d, self.nn, self.d), dtype=torch.float64, device="cuda")
        M[self.pa, :, self.pb, :] = vals.reshape(-1, self.d, self.d)
        return M.reshape(self.nn * self.d, -1)

    def dense(self, K):
        """Assembled tangent from all cells' pattern values."""
        k = torch.arange(self.d, device="cuda")
        row = (self.cn[:, self.pa] * self.d)[:, :, None, None] + k[:, None]
        col = (self.cn[:, self.pb] * self.d)[:, :, None, None] + k[None, :]
        A = torch.zeros(self.n_dof * self.n_dof, dtype=torch.float64, device="cuda")
        A.index_add_(0, (row * self.n_dof + col).reshape(-1), K.reshape(-1))
        return A.reshape(self.n_dof, -1)

    def cells(self):
        return torch.arange(self.ns, device="cuda")

    def greedy(self, u, eps, cap):
        """Algorithm 1 on the reduced-rule tangents: principal cells and coefficients."""
        T = self.tangents(u, self.cells(), True)
        norms = T.norm(dim=1)
        delta = T / norms[:, None]
        S, beta = [], []
        while len(S) < min(cap, self.ns):
            inf = delta.abs().amax(dim=1)
            s = int(inf.argmax())
            if not float(inf[s]) > eps:
                break
            z = delta[s] / delta[s].norm()
            b = delta @ z
            delta -= b[:, None] * z
            S.append(s)
            beta.append(b)
        B = torch.stack(beta) * norms                       # coordinates of the snapshots, [n_r, n_cells]
        S = torch.tensor(S, device="cuda")
        return S, torch.linalg.solve_triangular(B[:, S].triu(), B, upper=True)

    def newton(self, load, affine):
        u = affine.clone()
        top = torch.tensor(self.lat.top_nodes(), device="cuda") * self.d
        free = ~self.fixed
        u[self.fixed] = 0.0
        u[top + self.lat.load_axis] = load
        r0 = None
        for _ in range(30):
            r = self.scatter(self.forces(u)[0])
            n = float(r[free].norm())
            r0 = n if r0 is None else r0
            if n <= 1e-14 * r0:
                break
            A = self.dense(self.tangents(u, self.cells()))[free][:, free]
            du = torch.linalg.solve(A, -r[free])
            u[free] += du
            if float(du.norm()) <= 1e-14 * float(u.norm()):
                break
        return u


def _affine(lc):
    lat = lc.lattice
    u = torch.zeros((lat.n_nodes, lat.dim), dtype=torch.float64, device="cuda")
    u[:, lat.load_axis] = lc.top_displacement(1) / lat.height * torch.tensor(lat.X[:, lat.load_axis], device="cuda")
    return u.reshape(-1)


def exact(case, seed):
    lc = _load_case(case, seed)
    path = case["path"]
    n_dof = lc.lattice.n_nodes * lc.lattice.dim
    if path in ("precond", "newton_it") or (path in ("load_step", "solve", "adjoint") and n_dof > DENSE_DOF):
        return None
    p = _Plain(lc)
    load = lc.top_displacement(1)
    if path == "load_step":
        return p.newton(load, _affine(lc))
    if path == "adjoint":
        u = p.newton(load, _affine(lc))
        A, free = p.dense(p.tangents(u, p.cells())), ~p.fixed
        w = torch.where(p.fixed, u, torch.zeros_like(u))
        J = float(w @ p.scatter(p.forces(u)[0]))
        w[free] = -torch.linalg.solve(A[free][:, free], A[free] @ w)
        f_mu, _ = p.forces(u, mu=torch.full_like(p.mu, MU), lam=0.0)
        return {"grad": (w[p.ldof].T * f_mu).sum(dim=0), "J": J}
    u = _state(lc, seed)
    if path == "residual":
        f, least = p.forces(u)
        return {"r": p.scatter(f), "f": f, "min_detF": least}
    if path == "tangent":
        return p.tangents(u, p.cells())
    if path == "select":
        S, alpha = p.greedy(u, 1e-3 * lc.eps, case["n_r"])
        return {"S": None, "alpha": alpha, "Kp": p.tangents(u, S)}
    if path == "solve":
        S, alpha = p.greedy(u, lc.eps, 32)
        A, free = p.dense(alpha.T @ p.tangents(u, S)), ~p.fixed
        x = torch.zeros(n_dof, dtype=torch.float64, device="cuda")
        x[free] = torch.linalg.solve(A[free][:, free], _rhs(lc, seed)[free])
        return x
    S, alpha = _principals(lc, _n_r(case, lc), seed)
    K = p.tangents(u, S.long().cuda())
    dt = torch.float64 if case["mode"] == "fp64" else torch.float32
    x = _uniform((p.nn * p.d, p.ns), seed, dt).double()
    y = torch.zeros_like(x)
    for r in range(len(S)):
        y += alpha[r].cuda() * (p.local_dense(K[r]) @ x)
    return y
