"""Forms that a rule on sizes chooses, at the sizes where the rule turns: node groups of the FP32 action,
and batches of inversions whose workspace does not fit its bound at once."""
import numpy as np
import pytest
import torch

import latgen
from oracle import cell as OC
from oracle import rom as OR
from oracle.assembly import Problem

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    import __graft_entry__ as g
    g.build()
    from paper_2603_10741_gb300 import lattice
    return lattice


def _case(cell, dims, seed, strain):
    lat_geo = latgen.tile(*cell, dims)
    return latgen.LoadCase(name="forms", lattice=lat_geo, mu=1.0, lam=4.0,
                           mu_scale=latgen.mu_scale(lat_geo.n_cells, seed), total_strain=strain, n_steps=1, eps=1e-3)


@pytest.mark.parametrize("dims", [
    (8, 8, 4),     # 256 cells: 2 tiles of 128 x 55 groups of 16 nodes do not fill 152 SMs: groups of 8
    (13, 5, 4),    # 260 cells: a third tile of 4 cells, 165 CTAs: groups of 16
    (9, 8, 7),     # 504 cells: groups of 16, a last tile of 120
])
def test_fp32_action_where_the_groups_change(L, dims):
    """One principal, FP32, against the oracle on sampled cells (2e-6 as in test_gpu_kernels.py)."""
    case = _case(latgen.strut_cell(12, 0.15), dims, 11, 0.05)
    prob = Problem(case)
    n = case.lattice.n_cells
    u = latgen.smooth_state(case.lattice, 0.01, 25).ravel()
    S = np.array([n // 2], dtype=np.int32)
    al = latgen.dirichlet_coefficients(1, n, 12)
    X = latgen.uniform_field((prob.cell.n_nodes * 3, n), 26)
    cells = np.unique(np.concatenate([np.arange(0, n, 17), [127, 128, n - 4, n - 3, n - 2, n - 1]]))
    Kp = OC.tangent(prob.cell, prob.local(u)[S], prob.mu_cells[S], prob.lam)
    ref = OR.reduced_apply(prob.cell, Kp, al[:, cells], X[:, cells])
    lat = L.Lattice.from_case(case, 1)
    lat.set_principal_cells(torch.tensor(u, device="cuda"), torch.tensor(S), torch.tensor(al))
    Y = lat.apply_reduced_tangent(torch.tensor(X, device="cuda", dtype=torch.float32)).cpu().numpy()[:, cells]
    assert np.abs(Y - ref).max() < 2e-6 * np.abs(ref).max()
    lat.close()


def test_inversions_in_parts(L):
    """625 ring cells, all principal: matrices of 568 rows take 3.47 MB of workspace each, 577 of them the
    bound of 2 GB, so they are inverted in parts of 577 and 48.  K^-rom inverts K~ (1e-9 as in
    test_gpu_paths.py), and the dual Schur complements of both parts precondition the interface as well
    as on 576 cells, one part: the iterations of a Dirichlet preconditioner do not grow with the number
    of cells, a wrong part of 48 cells would leave many more."""
    its = []
    for n in (24, 25):
        case = _case(latgen.ring_cell(16), (n, n), None, 0.02 / n)
        lat = L.Lattice.from_case(case)
        u = lat.lattice_predictor(case.top_displacement(1))
        opts = lat.lattice_default_opts(precond_tangent=0, max_enrich=0, force_all=1, krylov_rtol=1e-8)
        lat.select_principal_cells(u, 0.0, 1, force_all=True)
        lat.lattice_prepare_solver(u, opts)
        s = lat.sizes
        assert s.n_r_local == 568
        nd = s.n_loc * s.n_cells + s.n_primal
        v = lat.feti_from_global(torch.tensor(np.random.default_rng(5).uniform(-1, 1, s.n_dof), device="cuda"))
        v[nd:] = 0
        Kv = lat.feti_apply(0, v)
        Kv[nd:] = 0
        back = lat.feti_apply(1, Kv)
        assert (back[:nd] - v[:nd]).abs().max().item() < 1e-9 * v[:nd].abs().max().item()
        rep = lat.newton_step(u, opts, max_iterations=1)
        its.append(rep.pcg_its_total / rep.krylov_its_total)
        lat.close()
    assert its[1] < 1.5 * its[0]
