"""lattice_kernel_time: every launch of a named kernel is counted and timed, and no other."""
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


def test_greedy_update_counts_updates(L):
    """One record per projection of the columns: five principals, five updates."""
    T = torch.tensor(np.random.default_rng(3).normal(size=(40, 257)), device="cuda")
    lat = L.Lattice.from_case(latgen.make_case("ring2"))
    lat.lattice_set_timing(1)
    out = lat.greedy_select(T, 1e-12, 5)
    assert out["S"].numel() == 5
    assert lat.lattice_kernel_time("greedy_update")[1] == 5
    lat.close()


def test_trailing_updates_of_large_inversions_are_timed(L):
    """One cell of 1005 remaining DOFs, 375 of them interior, every corner fixed (no coarse matrix): 3 +
    5 panels of 128 columns, each with its trailing update and the four of its pivot block."""
    Xr, E = latgen.solid_cell(6, 3)
    lat_geo = latgen.tile(Xr, E, (1, 1, 1))
    case = latgen.LoadCase(name="timing", lattice=lat_geo, mu=1.0, lam=4.0, mu_scale=latgen.mu_scale(1, None),
                           total_strain=0.01, n_steps=1, eps=1e-3)
    lat = L.Lattice.from_case(case)
    u = lat.lattice_predictor(case.top_displacement(1))
    lat.select_principal_cells(u, 0.0, 1, force_all=True)
    lat.lattice_set_timing(1)
    lat.lattice_prepare_solver(u, lat.lattice_default_opts(max_enrich=0))
    assert lat.sizes.n_primal == 0 and lat.sizes.n_r_local == 1005
    assert lat.lattice_kernel_time("gj_update")[1] == 8 * 5
    lat.close()


@pytest.mark.parametrize("prec,name", [(0, "apply_reduced"), (1, "apply_reduced_fp32")])
def test_action_timing_covers_the_lumped_interface_loop(L, prec, name):
    """enable = 2 times every launch of the action: with the lumped interface preconditioner each
    interface iteration holds one.  As many records as with enable = 1, and the same solution as
    untimed, before and after."""
    Xr, E = latgen.ring_cell(8)
    lat_geo = latgen.tile(Xr, E, (4, 4))
    case = latgen.LoadCase(name="timing", lattice=lat_geo, mu=1.0, lam=4.0, mu_scale=latgen.mu_scale(16, 4),
                           total_strain=0.01, n_steps=1, eps=1e-3)
    lat = L.Lattice.from_case(case, prec)
    u = lat.lattice_predictor(case.top_displacement(1))
    o = lat.lattice_default_opts(interface_precond=1, krylov_max_it=5, krylov_rtol=1e-14, pcg_iters=6, pcg_rtol=0.0,
                                 max_enrich=0, inner_its=0)
    lat.select_principal_cells(u, 1e-3, 4)
    lat.lattice_prepare_solver(u, o)
    rhs = torch.tensor(np.random.default_rng(6).uniform(-1, 1, lat.sizes.n_dof), device="cuda")
    records, xs = {}, []
    for enable in (0, 2, 1, 2, 0):
        lat.lattice_set_timing(enable)
        n0 = lat.lattice_launch_count()
        xs.append(lat.tangent_solve(rhs, o)[0])
        n = lat.lattice_launch_count() - n0
        records.setdefault(enable, []).append((lat.lattice_kernel_time(name)[1], n))
    assert all(torch.equal(x, xs[0]) for x in xs)
    # 5 iterations of 1 + 6 interface products (r.z before the first one), in FP64 6 operators under the
    # same name
    assert records[1][0][0] == 5 * 7 + (6 if prec == 0 else 0)
    assert records[2][0][0] == records[2][1][0] == records[1][0][0]
    assert len({n for r in records.values() for _, n in r}) == 1
    lat.close()
