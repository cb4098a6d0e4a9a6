"""The interface PCG: its loop on the device (a graph's while node) against the same launches one by
one (kernel timing on), at its limits, and with the lumped preconditioner in every precision."""
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


RING = (latgen.ring_cell(8), (12, 12))              # 3 keys, 144 cells: segmented and tensor-core products
RING_FEW = (latgen.ring_cell(8), (3, 4))            # fewer than 8 cells per key: products per cell
STRUT = (latgen.strut_cell(12, 0.15), (2, 2, 6))    # 3 keys, 24 cells: FP64 products on digits


def _solver(L, lattice, prec, **opts):
    (Xr, E), dims = lattice
    lat_geo = latgen.tile(Xr, E, dims)
    case = latgen.LoadCase(name="interface", lattice=lat_geo, mu=1.0, lam=4.0,
                           mu_scale=latgen.mu_scale(lat_geo.n_cells, 4), total_strain=0.002, n_steps=1, eps=1e-3)
    lat = L.Lattice.from_case(case, prec)
    u = lat.lattice_predictor(case.top_displacement(1))
    o = lat.lattice_default_opts(max_enrich=0, **opts)
    lat.select_principal_cells(u, 1e-9, 1)
    lat.lattice_prepare_solver(u, o)
    rhs = torch.tensor(np.random.default_rng(2).uniform(-1, 1, lat.sizes.n_dof), device="cuda")
    return lat, o, rhs


@pytest.mark.parametrize("prec", [0, 1, 2])
@pytest.mark.parametrize("lattice", [RING, RING_FEW, STRUT])
def test_lumped_solution_is_the_dirichlet_one(L, lattice, prec):
    """The interface preconditioner shapes the iterations, not the solution: both to a relative
    residual of 1e-12 agree to 1e-9 of the largest entry (as against the direct solve in
    test_gpu_solver.py)."""
    xs = []
    for iface in (0, 1):
        lat, o, rhs = _solver(L, lattice, prec, interface_precond=iface, krylov_rtol=1e-12, krylov_max_it=3000)
        x, its, rel = lat.tangent_solve(rhs, o)
        assert rel <= 1e-12, (iface, its, rel)
        xs.append(x)
        lat.close()
    assert (xs[1] - xs[0]).abs().max().item() < 1e-9 * xs[0].abs().max().item()


@pytest.mark.parametrize("iface", [0, 1])
@pytest.mark.parametrize("prec", [0, 1, 2])
@pytest.mark.parametrize("lattice", [RING, RING_FEW, STRUT])
@pytest.mark.parametrize("iters,rtol", [(100, 3e-2), (1, 3e-2), (7, 0.0)])
def test_device_loop_equals_launch_by_launch(L, lattice, prec, iface, iters, rtol):
    """The same kernels in the same order: equal to the bit, with the stop by tolerance, at the cap and
    without a tolerance; interface iterations counted alike (newton_step's report)."""
    lat, o, rhs = _solver(L, lattice, prec, interface_precond=iface, pcg_iters=iters, pcg_rtol=rtol, krylov_max_it=6,
                          krylov_rtol=1e-14, inner_its=3)
    v = lat.feti_from_global(rhs)
    zero = torch.zeros_like(v)
    got = []
    for timing in (0, 1):
        lat.lattice_set_timing(timing)
        x, its, rel = lat.tangent_solve(rhs, o)
        got.append((lat.feti_apply(2, v), x, its, rel))
        assert bool((lat.feti_apply(2, zero) == 0).all())      # r.z = 0: the iteration stops at once
        assert bool((lat.tangent_solve(torch.zeros_like(rhs), o)[0] == 0).all())
    lat.lattice_set_timing(0)
    assert bool(torch.isfinite(got[0][0]).all()) and bool(torch.isfinite(got[0][1]).all())
    assert torch.equal(got[0][0], got[1][0]) and torch.equal(got[0][1], got[1][1]) and got[0][2:] == got[1][2:]
    lat.close()


@pytest.mark.parametrize("iters,rtol", [(100, 3e-2), (2, 3e-2), (9, 0.0)])
def test_interface_iterations_are_counted_alike(L, iters, rtol):
    case = latgen.make_case("ring4")
    counts = []
    for timing in (0, 1):
        lat = L.Lattice.from_case(case)
        lat.lattice_set_timing(timing)
        u = lat.lattice_predictor(case.top_displacement(1))
        rep = lat.newton_step(u, lat.lattice_default_opts(pcg_iters=iters, pcg_rtol=rtol), max_iterations=1)
        counts.append((rep.pcg_its_total, rep.krylov_its_total, rep.r_norm))
        lat.close()
    assert counts[0] == counts[1] and counts[0][0] > 0
    if rtol == 0.0:
        assert counts[0][0] == iters * counts[0][1]
    else:
        assert counts[0][0] <= iters * counts[0][1]
