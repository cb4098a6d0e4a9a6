"""The handle's flag word: what the setup leaves in it, and what a bounded device-side wait that gives
up makes of a call.  No wait is made to hang: the pivots are those of a compressed lattice."""
import numpy as np
import pytest
import torch

import latgen

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    import __graft_entry__ as g
    g.build()
    from paper_2603_10741_gb300 import lattice
    return lattice


def _strut(L, prec, dims, seed=None, cell=None):
    Xr, E = latgen.strut_cell(12, 0.15) if cell is None else cell
    lat_geo = latgen.tile(Xr, E, dims)
    case = latgen.LoadCase(name="waits", lattice=lat_geo, mu=1.0, lam=4.0,
                           mu_scale=latgen.mu_scale(lat_geo.n_cells, seed), total_strain=0.01, n_steps=1, eps=1e-3)
    return case, L.Lattice.from_case(case, prec)


@pytest.mark.parametrize("prec", [0, 1, 2])
def test_indefinite_coarse_matrix_is_not_a_timeout(L, prec):
    """2 x 2 x 6 equal strut cells at 1 % compression, local blocks of the full tangent, corners primal
    alone: 29 of the 135 eigenvalues of the coarse matrix are negative.  The solve runs its iterations
    and says how far it came."""
    case, lat = _strut(L, prec, (2, 2, 6))
    u = lat.lattice_predictor(case.top_displacement(1))
    opts = lat.lattice_default_opts(precond_tangent=0, max_enrich=0, krylov_max_it=4, krylov_rtol=1e-14)
    lat.select_principal_cells(u, 1e-3, 1)
    lat.lattice_prepare_solver(u, opts)
    assert lat.sizes.n_p_local == 24
    rhs = torch.tensor(np.random.default_rng(1).uniform(-1, 1, lat.sizes.n_dof), device="cuda")
    x, its, rel = lat.tangent_solve(rhs, opts)
    assert its == 4 and 0 < rel < 1 and bool(torch.isfinite(x).all())
    lat.close()
