"""Kernels whose form depends on sizes, at the sizes where a form begins or ends: tiles that are not
full, remainders, the smallest and the largest of a range.  References: the oracle, or an identity
that holds exactly (K^-rom of the force-all path is the inverse of the operator, as in
test_gpu_solver.py, with its tolerance of 1e-9 for the condition of the local problems)."""
import numpy as np
import pytest
import torch

import latgen
from oracle import cell as OC
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


@pytest.mark.parametrize("cell,dims", [
    (latgen.strut_cell(12, 0.15), (3, 3, 4)),    # 3 tiles of 9-18 cells x 21 row tiles: K split over 4 CTAs
    (latgen.strut_cell(12, 0.15), (6, 6, 12)),   # 105 tiles, segments of 36 and 360 cells: split over 2
    (latgen.strut_cell(12, 0.15), (9, 9, 9)),    # 168 tiles: not split; a segment of 567 cells
    (latgen.ring_cell(4), (8, 9)),               # 24 remaining DOFs: fewer K panels than a cluster of 4
])
def test_tensor_core_product_by_tile_count(L, cell, dims):
    """K^-rom in BF16 mode against the FP64 mode: ~16-bit operand pairs, FP32 sums (tolerance as in
    test_gpu_solver.py's tensor-core tests)."""
    case = _case(cell, dims)
    outs = []
    for prec in (0, 2):
        lat = L.Lattice.from_case(case, prec)
        u = lat.lattice_predictor(0.1 * case.top_displacement(1))
        lat.select_principal_cells(u, 1e-3, 1)
        lat.lattice_set_timing(True)
        lat.lattice_prepare_solver(u, lat.lattice_default_opts(max_enrich=0, precond_tangent=1))
        rng = np.random.default_rng(7)
        s = lat.sizes
        v = lat.feti_from_global(torch.tensor(rng.uniform(-1, 1, s.n_dof), device="cuda"))
        outs.append(lat.feti_apply(1, v)[: s.n_loc * s.n_cells + s.n_primal].cpu().numpy())
        assert prec == 0 or lat.lattice_kernel_time("local_tc")[1] > 0
        lat.close()
    err = np.linalg.norm(outs[1] - outs[0]) / np.linalg.norm(outs[0])
    assert err < 1e-4, err


def _rel(a, b):
    return np.abs(np.asarray(a) - np.asarray(b)).max() / np.abs(np.asarray(b)).max()


@pytest.mark.parametrize("cell,dims", [
    (latgen.solid_cell(1, 2), (3, 1)),           # one element per cell: 4 of a warp's lanes
    (latgen.solid_cell(3, 3), (1, 2, 1)),        # 27 elements: a last warp with 24 lanes
    (latgen.solid_cell(9, 3), (2, 1, 1)),        # 729 elements: forces staged in two parts
    (latgen.ring_cell(4), (13, 3)),              # 39 cells: one CTA per cell; 38 and fewer: eight
])
def test_residual_and_tangent_by_element_and_cell_count(L, cell, dims):
    """Forces and tangents, both rules, of all cells and of a list, against the oracle (FP64 sums in
    another order: 1e-11 of the largest entry, as in test_gpu_kernels.py)."""
    case = _case(cell, dims)
    prob = Problem(case)
    u = latgen.smooth_state(case.lattice, 0.01, 11).ravel()
    lat = L.Lattice.from_case(case)
    ud = torch.tensor(u, device="cuda")
    ul = prob.local(u)
    n = prob.lat.n_cells
    out = lat.assemble_residual_tangent(ud, local_forces=True, tangent=True)
    f_ref = OC.internal_force(prob.cell, ul, prob.mu_cells, prob.lam).reshape(n, -1).T
    assert _rel(out["f"].cpu(), f_ref) < 1e-11
    assert _rel(out["r"].cpu(), prob.residual(u)) < 1e-11
    assert abs(out["min_detF"] - OC.min_jacobian(prob.cell, ul).min()) < 1e-12
    K_ref = OC.tangent(prob.cell, ul, prob.mu_cells, prob.lam)
    assert _rel(out["K"].cpu(), K_ref) < 1e-11
    cells = np.arange(n - 1, -1, -1)[:38].astype(np.int32)
    ct = torch.tensor(cells, device="cuda")
    for quad in (0, 1):
        K = lat.assemble_residual_tangent(ud, quad=quad, cells=ct, residual=False, tangent=True)["K"].cpu()
        ref = OC.tangent(prob.cell, ul[cells], prob.mu_cells[cells], prob.lam, reduced=quad == 1)
        assert _rel(K, ref) < 1e-11
    lat.close()


@pytest.mark.parametrize("cell,dims,lu", [
    (latgen.ring_cell(2), (2, 9), 0),        # blocks of 8 and 12 rows: less than one pivot block
    (latgen.solid_cell(6, 2), (9, 9), 0),    # 90 remaining DOFs: 32 + 32 + 26, split inside a pivot block
    (latgen.solid_cell(4, 3), (3, 3, 3), 1), # 351 remaining DOFs, 81 of them interior; coarse blocks as block LU
    (latgen.ring_cell(14), (2, 2), 0),       # 440 remaining DOFs: panels of 128, the last one of 40 after 16
    (latgen.solid_cell(6, 3), (1, 2, 2), 0), # 1005 remaining DOFs, split at 375 inside a 128-row tile
])
def test_symmetric_inverse_by_size(L, cell, dims, lu):
    """Local and coarse inverses by sweeps: K^-rom K~ = I on the force-all path, whose every local
    block and coarse block goes through the batched inversion."""
    case = _case(cell, dims)
    prob = Problem(case)
    lat = L.Lattice.from_case(case)
    ud = torch.tensor(ON.predictor(prob, 1, None, None), device="cuda")
    lat.select_principal_cells(ud, 0.0, 1, force_all=True)
    lat.lattice_prepare_solver(ud, lat.lattice_default_opts(precond_tangent=0, max_enrich=0, coarse_block_lu=lu))
    s = lat.sizes
    nd = s.n_loc * s.n_cells + s.n_primal
    v = lat.feti_from_global(torch.tensor(np.random.default_rng(5).uniform(-1, 1, s.n_dof), device="cuda"))
    v[nd:] = 0
    Kv = lat.feti_apply(0, v)
    Kv[nd:] = 0
    back = lat.feti_apply(1, Kv)
    err = (back[:nd] - v[:nd]).abs().max().item() / v[:nd].abs().max().item()
    assert err < 1e-9, err
    lat.close()


@pytest.mark.parametrize("dims", [
    (2, 2, 6),     # segments of 4 and 16 cells: one exactly full tile
    (3, 3, 6),     # 9 and 36 cells: tiles of 9, 16, 16 and 4
])
def test_fp64_digit_products(L, dims):
    """FP64 products on the tensor cores (digits): with equal cells at rest the one principal's local
    blocks are every cell's, so K^-rom inverts K~ on vectors without multipliers (1e-9 as in the
    force-all test); entries from 1e-12 to 1 in one vector, and a NaN stays a NaN."""
    case = _case(latgen.strut_cell(12, 0.15), dims, seed=None)
    lat = L.Lattice.from_case(case)
    u = lat.lattice_predictor(0.0)
    lat.select_principal_cells(u, 1e-3, 4)
    lat.lattice_prepare_solver(u, lat.lattice_default_opts(precond_tangent=0, max_enrich=0))
    s = lat.sizes
    nd = s.n_loc * s.n_cells + s.n_primal
    rng = np.random.default_rng(8)
    for lo in (0, -12):
        w = rng.uniform(-1, 1, s.n_dof) * 10.0 ** rng.uniform(lo, 0, s.n_dof)
        v = lat.feti_from_global(torch.tensor(w, device="cuda"))
        v[nd:] = 0
        Kv = lat.feti_apply(0, v)
        Kv[nd:] = 0
        back = lat.feti_apply(1, Kv)
        err = (back[:nd] - v[:nd]).abs().max().item() / v[:nd].abs().max().item()
        assert err < 1e-9, err
    Kv[s.n_cells * (s.n_loc // 2) + 1] = float("nan")
    assert torch.isnan(lat.feti_apply(1, Kv)[:nd]).any()
    lat.close()


@pytest.mark.parametrize("cell,dims,n_r", [
    (latgen.ring_cell(8), (4, 4), 17),           # small CTAs, two chunks of principals
    (latgen.ring_cell(8), (25, 39), 2),          # 975 cells: 16 tiles of 64 x 10 CTAs of 8 nodes, one more than the SMs
    (latgen.strut_cell(6, 0.2), (1, 2, 1), 5),   # small CTAs in 3D, two chunks
    (latgen.strut_cell(12, 0.15), (3, 3, 4), 1), # 36 cells: CTAs of 4 warps, last tile of 4 cells
])
def test_fp64_action_by_cta_form(L, cell, dims, n_r):
    """FP64 reduced action against the oracle (1e-10 as in test_gpu_kernels.py)."""
    from oracle import rom as OR
    case = _case(cell, dims)
    prob = Problem(case)
    n = prob.lat.n_cells
    n_r = min(n_r, n)
    u = latgen.smooth_state(case.lattice, 0.01, 21).ravel()
    S = np.arange(n_r, dtype=np.int32)
    al = latgen.dirichlet_coefficients(n_r, n, 8)
    X = latgen.uniform_field((prob.cell.n_nodes * prob.cell.d, n), 22)
    ref = OR.reduced_apply(prob.cell, OC.tangent(prob.cell, prob.local(u)[S], prob.mu_cells[S], prob.lam), al, X)
    lat = L.Lattice.from_case(case)
    lat.set_principal_cells(torch.tensor(u, device="cuda"), torch.tensor(S), torch.tensor(al))
    assert _rel(lat.apply_reduced_tangent(torch.tensor(X, device="cuda")).cpu(), ref) < 1e-10
    lat.close()


@pytest.mark.parametrize("n_rows,n_cols,max_nr", [(1, 1, 1), (31, 3, 8), (257, 40, 9), (4096, 5, 5)])
def test_greedy_by_size(L, n_rows, n_cols, max_nr):
    """Algorithm 1 against the oracle's at sizes off the blocks' multiples: identical selections, alpha
    to 1e-9 (test_gpu_kernels.py); with the cap, and through the allocation-free entry point too."""
    from oracle import greedy as OG
    T = np.random.default_rng(n_rows).normal(size=(n_rows, n_cols))
    g = OG.greedy(T, 1e-6, max_nr)
    a_ref = OG.alpha_triangular(T, g)
    lat = L.Lattice.from_case(latgen.make_case("ring2"))
    Td = torch.tensor(T.T.copy(), device="cuda")
    out = lat.greedy_select(Td, 1e-6, max_nr)
    S, al = L.greedy_select_static(Td, 1e-6, max_nr)
    for s_got, a_got in ((out["S"], out["alpha"]), (S, al)):
        assert s_got.cpu().numpy().tolist() == g.S.tolist()
        assert np.abs(a_got.cpu().numpy() - a_ref).max() <= 1e-9 * max(1.0, np.abs(a_ref).max())
    lat.close()


@pytest.mark.parametrize("cell,dims", [
    (latgen.ring_cell(8), (31, 9)),      # segments of 31 and 217 cells: tiles of 31 and 25, one tile less than full
    (latgen.ring_cell(6), (8, 6)),       # 72 remaining DOFs: K chunks of 32, 32 and 8; 20 dual columns
    (latgen.solid_cell(4, 2), (4, 16)),  # 32-row remainders: 50 rows of a 64-row tile
])
def test_fp32_segmented_product(L, cell, dims):
    """K^-rom in the FP32 mode against the FP64 mode: FP32 blocks and sums on local problems of
    condition below 1e3 (tolerance 1e-4 as for the BF16 pairs, which carry fewer bits)."""
    case = _case(cell, dims)
    outs = []
    for prec in (0, 1):
        lat = L.Lattice.from_case(case, prec)
        u = lat.lattice_predictor(0.1 * case.top_displacement(1))
        lat.select_principal_cells(u, 1e-3, 1)
        lat.lattice_set_timing(True)
        lat.lattice_prepare_solver(u, lat.lattice_default_opts(max_enrich=0, precond_tangent=1))
        s = lat.sizes
        v = lat.feti_from_global(torch.tensor(np.random.default_rng(7).uniform(-1, 1, s.n_dof), device="cuda"))
        outs.append(lat.feti_apply(1, v)[: s.n_loc * s.n_cells + s.n_primal].cpu().numpy())
        assert lat.lattice_kernel_time("local_segmm")[1] > 0
        lat.close()
    err = np.linalg.norm(outs[1] - outs[0]) / np.linalg.norm(outs[0])
    assert err < 1e-4, err
