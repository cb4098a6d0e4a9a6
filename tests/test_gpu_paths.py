"""Kernels whose form depends on sizes, at the sizes where a form begins or ends: tiles that are not
full, remainders, the smallest and the largest of a range.  References: the oracle, or an identity
that holds exactly (K^-rom of the force-all path is the inverse of the operator, as in
test_gpu_solver.py, with its tolerance of 1e-9 for the condition of the local problems)."""
import numpy as np
import pytest
import torch

import latgen
from oracle import newton as ON
from oracle.assembly import Problem

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    import __graft_entry__ as g
    g.build()
    from paper_2603_10741_gb300 import lattice
    return lattice


def _case(cell, dims, seed=9):
    Xr, E = cell
    lat = latgen.tile(Xr, E, dims)
    return latgen.LoadCase(name="paths", lattice=lat, mu=1.0, lam=4.0, mu_scale=latgen.mu_scale(lat.n_cells, seed),
                           total_strain=0.02, n_steps=10, eps=1e-3)


@pytest.mark.parametrize("cell,dims,level", [
    (latgen.ring_cell(4), (1, 2), 0),            # 2 cells, 8 corner values
    (latgen.ring_cell(8), (7, 5), 2),            # 35 cells: a full tile of 32 and a rest; 32 corner values
    (latgen.strut_cell(6, 0.2), (3, 11, 1), 1),  # 33 cells; 60 corner values
    (latgen.strut_cell(12, 0.15), (2, 2, 1), 3), # 276 corner values: three chunks of 96
])
def test_local_inverse_by_enrichment_and_cell_count(L, cell, dims, level):
    case = _case(cell, dims)
    prob = Problem(case)
    lat = L.Lattice.from_case(case)
    ud = torch.tensor(ON.predictor(prob, 1, None, None), device="cuda")
    lat.select_principal_cells(ud, 0.0, 1, force_all=True)
    lat.lattice_prepare_solver(ud, lat.lattice_default_opts(precond_tangent=0, min_enrich=level, max_enrich=level))
    s = lat.sizes
    nd = s.n_loc * s.n_cells + s.n_primal
    rng = np.random.default_rng(3)
    v = lat.feti_from_global(torch.tensor(rng.uniform(-1, 1, s.n_dof), device="cuda"))
    v[nd:] = 0
    Kv = lat.feti_apply(0, v)
    Kv[nd:] = 0
    back = lat.feti_apply(1, Kv)
    err = (back[:nd] - v[:nd]).abs().max().item() / v[:nd].abs().max().item()
    assert err < 1e-9, err
    lat.close()
