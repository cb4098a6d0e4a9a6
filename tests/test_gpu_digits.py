"""FP64 products on the tensor cores (operands as twelve base-128 digits) against the matrices they are
made of, in more than 64 bits.

A layer of strut cells between the clamped faces has no free corner, so K^-rom is the local inverse G
alone, one matrix for all cells.  Four cells run on the FP64 pipe (fewer than eight per key), where
unit vectors give G's columns exactly; sixteen cells of the same G run on digits.

Bounds (e, e': exponents of the row's and the vector's largest magnitude, 2^e <= 2 gmax): each operand is
cut at 2^(e - 84), and the digit products that are left out, i + j >= 12, come to less than 11.1 x
2^(e + e' - 84) per term, together 12.1 x 2^-82 of gmax xmax per term.  Summing the digit sums rounds ten
times at most (two fused multiply-adds, seven CTAs of a cluster, the cell's factor)."""
import numpy as np
import pytest
import torch

import latgen

pytestmark = pytest.mark.gpu

DROPPED = 12.1 * 2.0 ** -82
CELL = latgen.strut_cell(12, 0.15)


@pytest.fixture(scope="module")
def L():
    import __graft_entry__ as g
    g.build()
    from paper_2603_10741_gb300 import lattice
    return lattice


def _prepare(lat, force_all=False):
    u = lat.lattice_predictor(0.0)
    lat.select_principal_cells(u, 1e-3, 1, force_all=force_all)
    lat.lattice_prepare_solver(u, lat.lattice_default_opts(precond_tangent=0, max_enrich=0))


def _layer(L, nx):
    lat_geo = latgen.tile(*CELL, (nx, nx, 1))
    case = latgen.LoadCase(name="digits", lattice=lat_geo, mu=1.0, lam=4.0,
                           mu_scale=latgen.mu_scale(lat_geo.n_cells, None), total_strain=0.01, n_steps=1, eps=1e-3)
    return L.Lattice.from_case(case)


def _local(lat, X):
    """K^-rom of the columns of X [n_loc][n_cells], one per cell."""
    s = lat.sizes
    v = lat.krylov_vector()
    v[: s.n_loc * s.n_cells] = torch.tensor(X, device="cuda").reshape(-1)
    return lat.feti_apply(1, v)[: s.n_loc * s.n_cells].reshape(s.n_loc, s.n_cells).cpu().numpy()


@pytest.fixture(scope="module")
def block(L):
    """(the layer on digits, the layer on the FP64 pipe, remaining free local DOFs, G on them)"""
    pipe, oz = _layer(L, 2), _layer(L, 4)
    for lat in (pipe, oz):
        _prepare(lat)
        assert lat.sizes.n_primal == 0
        lat.lattice_set_timing(1)
    X_ref = CELL[0]
    on_face = (np.abs(X_ref[:, 2]) < 1e-12) | (np.abs(X_ref[:, 2] - 1) < 1e-12)   # clamped, corners among them
    dofs = np.flatnonzero(~np.repeat(on_face, 3))
    s = pipe.sizes
    G = np.zeros((dofs.size, dofs.size))
    for k0 in range(0, dofs.size, 4):
        X = np.zeros((s.n_loc, 4))
        ks = np.arange(k0, min(k0 + 4, dofs.size))
        X[dofs[ks], ks - k0] = 1.0
        G[:, ks] = _local(pipe, X)[dofs][:, : ks.size]
    assert pipe.lattice_kernel_time("local_oz")[1] == 0
    yield oz, pipe, dofs, G
    oz.close()
    pipe.close()


def _run(lat, dofs, vecs):
    s = lat.sizes
    out = []
    for i in range(0, len(vecs), s.n_cells):
        X = np.zeros((s.n_loc, s.n_cells))
        for c, x in enumerate(vecs[i: i + s.n_cells]):
            X[dofs, c] = x
        Y = _local(lat, X)[dofs]
        out += [Y[:, c] for c in range(len(vecs[i: i + s.n_cells]))]
    return out


def _exact(G, x):
    y = np.zeros(G.shape[0], np.longdouble)
    for k in np.flatnonzero(x):
        y += G[:, k].astype(np.longdouble) * np.longdouble(x[k])
    return y


def test_error_is_no_larger_than_the_fp64_pipes(block):
    """Uniform, normal and graded vectors, down to one entry over a floor of 1e-16 of it: the error of the
    product, in the 2-norm and of the worst entry against its sum |g| |x|, is at most the FP64 pipe's, and
    every entry is within its bound."""
    oz, pipe, dofs, G = block
    n = dofs.size
    rng = np.random.default_rng(5)
    vecs = [rng.uniform(-1, 1, n), rng.normal(size=n), rng.uniform(-1, 1, n) * 10.0 ** rng.uniform(-12, 0, n)]
    x = rng.uniform(-1, 1, n) * 1e-6
    x[rng.choice(n, 20, replace=False)] = rng.uniform(-1, 1, 20)
    vecs.append(x)
    for floor in (1e-8, 1e-12, 1e-16):
        x = rng.uniform(-1, 1, n) * floor
        x[n // 3] = 1.0
        vecs.append(x)
    gmax = np.abs(G).max(axis=1)
    for x, y, y64 in zip(vecs, _run(oz, dofs, vecs), _run(pipe, dofs, vecs)):
        ref = _exact(G, x)
        err, err64 = np.abs(y - ref).astype(float), np.abs(y64 - ref).astype(float)
        size = np.abs(G) @ np.abs(x)
        assert np.linalg.norm(err) <= np.linalg.norm(err64)
        assert (err / size).max() <= (err64 / size).max()
        assert (err <= 12 * 2.0 ** -53 * size + n * DROPPED * gmax * np.abs(x).max()).all()
    assert oz.lattice_kernel_time("local_oz")[1] > 0


def test_single_terms(block):
    """One entry per vector, so one term per result.  Results below 2^-26 of the maxima come from the
    matrix itself, and every one is as exact as an FP64 product leaves it (three roundings); the others
    show the last digits (eleven digits would be off by about 2^-76 of the maxima)."""
    oz, _, dofs, G = block
    gmax = np.abs(G).max(axis=1)
    ratio = np.abs(G) / gmax[:, None]
    small, near = (ratio < 2.0 ** -33) & (G != 0), (ratio > 2.0 ** -24) & (ratio < 2.0 ** -20)
    ks = np.concatenate([np.argsort(-small.sum(axis=0))[:16], np.argsort(-near.sum(axis=0))[:16]])
    assert small[:, ks].sum() >= 16 and near[:, ks].sum() >= 16
    vecs = []
    for k in ks:
        x = np.zeros(dofs.size)
        x[k] = 1.0 / 3.0
        vecs.append(x)
    for k, x, y in zip(ks, vecs, _run(oz, dofs, vecs)):
        ref = _exact(G, x)
        err = np.abs(y - ref)
        assert (err <= 3 * 2.0 ** -53 * np.abs(ref) + DROPPED * gmax * np.abs(x).max()).all()
        assert (err[small[:, k]] <= 3 * 2.0 ** -53 * np.abs(ref)[small[:, k]]).all()


def test_extreme_values(block):
    """Subnormal vectors keep their last bit; a NaN or an infinity stays in its cell; zero stays zero."""
    oz, _, dofs, G = block
    n = dofs.size
    rng = np.random.default_rng(6)
    whole = rng.integers(-(1 << 30), 1 << 30, n).astype(float)
    tiny = whole * 2.0 ** -1074
    nan, inf = rng.uniform(-1, 1, n), rng.uniform(-1, 1, n)
    nan[7], inf[9] = np.nan, np.inf
    plain = rng.uniform(-1, 1, n)
    y_tiny, y_nan, y_inf, y_zero, y_plain = _run(oz, dofs, [tiny, nan, inf, np.zeros(n), plain])
    ref = _exact(G, whole)                           # in units of 2^-1074
    assert (np.abs(y_tiny * 2.0 ** 537 * 2.0 ** 537 - ref) <= 1.0).all() and np.abs(y_tiny).max() > 0
    assert np.isnan(y_nan).all() and not np.isfinite(y_inf).any()
    assert (y_zero == 0).all()
    assert (y_plain == _run(oz, dofs, [plain])[0]).all()


@pytest.mark.parametrize("dims", [(2, 2, 6), (3, 3, 6)])
def test_block_preconditioner_with_unequal_cells(L, dims):
    """All views of the local inverse and the dual Schur complements inside five interface iterations,
    factors c_s between a half and two, against the FP32 mode (its rounding, 1e-7 per product, against
    factors that are off by their square if a product divides for a multiplication)."""
    lat_geo = latgen.tile(*CELL, dims)
    n = lat_geo.n_cells
    mu = np.random.default_rng(3).uniform(0.5, 2.0, n)
    outs = []
    for prec in (0, 1):
        case = latgen.LoadCase(name="digits", lattice=lat_geo, mu=1.0, lam=4.0, mu_scale=mu, total_strain=0.001,
                               n_steps=1, eps=1e-3)
        lat = L.Lattice.from_case(case, prec)
        u = lat.lattice_predictor(case.top_displacement(1))
        lat.select_principal_cells(u, 1e-9, 1)
        lat.lattice_set_timing(1)
        lat.lattice_prepare_solver(u, lat.lattice_default_opts(max_enrich=0, precond_tangent=1))
        v = lat.feti_from_global(torch.tensor(np.random.default_rng(8).uniform(-1, 1, lat.sizes.n_dof), device="cuda"))
        outs.append(lat.feti_apply(2, v).cpu().numpy())
        counts = [lat.lattice_kernel_time(k)[1] for k in ("local_oz", "local_oz_dual", "local_oz_dual_in", "dual_schur_oz")]
        assert counts == ([1, 5, 1, 6] if prec == 0 else [0, 0, 0, 0])
        lat.close()
    assert np.linalg.norm(outs[1] - outs[0]) < 1e-3 * np.linalg.norm(outs[0])


def test_results_do_not_depend_on_free_memory(L):
    """The form of the products is a matter of sizes: with most of the device's memory taken by someone
    else the same call gives the same bits."""
    def run():
        lat_geo = latgen.tile(*CELL, (2, 2, 6))
        case = latgen.LoadCase(name="digits", lattice=lat_geo, mu=1.0, lam=4.0,
                               mu_scale=latgen.mu_scale(lat_geo.n_cells, 3), total_strain=0.001, n_steps=1, eps=1e-3)
        lat = L.Lattice.from_case(case)
        u = lat.lattice_predictor(case.top_displacement(1))
        lat.select_principal_cells(u, 1e-9, 1)
        lat.lattice_prepare_solver(u, lat.lattice_default_opts(max_enrich=0))
        v = lat.feti_from_global(torch.tensor(np.random.default_rng(8).uniform(-1, 1, lat.sizes.n_dof), device="cuda"))
        out = lat.feti_apply(1, v)
        lat.close()
        return out

    ref = run()
    torch.cuda.empty_cache()
    left = 1700 * 2 ** 20
    held = torch.empty(torch.cuda.mem_get_info()[0] - left, dtype=torch.uint8, device="cuda")
    try:
        got = run()
    finally:
        del held
        torch.cuda.empty_cache()
    assert torch.equal(got, ref)


def test_digits_are_given_back(L):
    """A selection with too many keys for digits holds no digits of the one before (250 MB for one key,
    167 with eight digits): as much memory as without that selection, up to small tables."""
    def held(selections):
        torch.cuda.synchronize()
        free = torch.cuda.mem_get_info()[0]
        lat = _layer(L, 4)
        for force_all in selections:
            _prepare(lat, force_all)
            lat.feti_apply(1, lat.krylov_vector())
        used = free - torch.cuda.mem_get_info()[0]
        lat.close()
        return used

    torch.cuda.empty_cache()
    held([True])                                  # module load and torch's own first allocations
    assert held([False, True]) - held([True]) < 100e6
