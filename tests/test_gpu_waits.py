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


@pytest.mark.parametrize("prec,cell,dims", [
    (0, None, (2, 2, 6)),                         # FP64 products on digits, K over a cluster
    (2, None, (2, 2, 6)),                         # BF16 pairs, K over a cluster of 4
    (2, latgen.ring_cell(4), (8, 9)),             # fewer panels than stages
])
def test_wait_that_gives_up_is_reported(L, prec, cell, dims):
    """With no polls every wait of a pipeline gives up at once (the copies in flight are still waited
    for): each call that makes such products says so, and is itself again with the limit restored."""
    case, lat = _strut(L, prec, dims, cell=cell)
    u = lat.lattice_predictor(0.1 * case.top_displacement(1))
    opts = lat.lattice_default_opts(max_enrich=0, precond_tangent=1, krylov_max_it=3, inner_its=2)
    lat.select_principal_cells(u, 1e-9, 1)
    lat.lattice_prepare_solver(u, opts)
    rhs = torch.tensor(np.random.default_rng(1).uniform(-1, 1, lat.sizes.n_dof), device="cuda")
    v = lat.feti_from_global(rhs)

    def results():
        return [lat.feti_apply(1, v), lat.feti_apply(2, v), lat.tangent_solve(rhs, opts)[0]]

    ref = results()
    lat.lattice_set_wait_limit(0)
    for call in (lambda: lat.feti_apply(1, v), lambda: lat.feti_apply(2, v), lambda: lat.tangent_solve(rhs, opts)):
        with pytest.raises(L.LatticeError, match="LAT_ETIMEOUT"):
            call()
    lat.feti_apply(0, v)                          # no product on the tensor cores
    if lat.sizes.n_r_local >= 384:
        with pytest.raises(L.LatticeError, match="LAT_ETIMEOUT"):
            lat.lattice_prepare_solver(u, opts)
    lat.lattice_set_wait_limit(1 << 20)
    lat.lattice_prepare_solver(u, opts)
    assert all(torch.equal(a, b) for a, b in zip(results(), ref))
    with pytest.raises(L.LatticeError, match="LAT_EINVAL"):
        lat.lattice_set_wait_limit(-1)
    lat.close()


@pytest.mark.parametrize("prec", [0, 1, 2])
def test_no_solver_after_a_failed_setup(L, prec):
    """A setup that fails, the first one or a later one, leaves no half-made solver behind: the calls that
    need one say so instead of reading buffers that are missing."""
    case, lat = _strut(L, prec, (2, 2, 6))
    u = lat.lattice_predictor(0.1 * case.top_displacement(1))
    opts = lat.lattice_default_opts(max_enrich=0, precond_tangent=1, krylov_max_it=3, inner_its=2)
    rhs = torch.tensor(np.random.default_rng(1).uniform(-1, 1, lat.sizes.n_dof), device="cuda")
    v = lat.feti_from_global(rhs)
    lat.select_principal_cells(u, 1e-9, 1)
    for first in (True, False):
        if not first:
            lat.lattice_prepare_solver(u, opts)
            ref = lat.feti_apply(1, v)
        lat.lattice_set_wait_limit(0)
        with pytest.raises(L.LatticeError, match="LAT_ETIMEOUT"):
            lat.lattice_prepare_solver(u, opts)
        lat.lattice_set_wait_limit(1 << 20)
        for call in (lambda: lat.feti_apply(1, v), lambda: lat.feti_apply(2, v), lambda: lat.tangent_solve(rhs, opts)):
            with pytest.raises(L.LatticeError, match="LAT_EINVAL"):
                call()
    lat.lattice_prepare_solver(u, opts)
    assert torch.equal(lat.feti_apply(1, v), ref)
    lat.close()
