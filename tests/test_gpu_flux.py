"""The operator in flux and stencil form (P1 on any coefficient, P2 on one coefficient per level): its tile edges,
remainders, small-level kernel, value ranges and non-finite entries, and the Chebyshev step in the same launch; the P3
operator by integer sums; the FP32 P2 restriction from staged tiles."""
import numpy as np
import pytest

import fe_inputs as I
from oracle import fe_oracle as O

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.fixture(scope="module")
def fe():
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    import paper_2104_08012_gb300 as m
    return m


def dt(a, dtype=torch.float64):
    return torch.from_numpy(np.ascontiguousarray(a)).to(DEV, dtype)


def apply(fe, h, x, dtype=torch.float64):
    y = torch.empty(len(x), dtype=dtype, device=DEV)
    h.apply_operator(dt(x, dtype), y, dtype=fe.FE_F64 if dtype == torch.float64 else fe.FE_F32)
    return y.double().cpu().numpy()


# the direct kernel's last size and the tiled kernels' first ones (16, 17), a tile of each axis exactly, plus one
# and minus one (8, 16, 32 along x; 4, 8 along y and z), and a single cube
@pytest.mark.parametrize("k,N", [(1, 1), (1, 2), (1, 9), (2, 1), (2, 2), (2, 3), (2, 7), (2, 16), (2, 17), (2, 24),
                                 (2, 31), (2, 33)])
@pytest.mark.parametrize("coef", ["one", "constant", "field"])
def test_apply_matches_oracle(fe, k, N, coef):
    """FP64 within 1e-14 of |A| |x| per row: the rounding of an FP64 row (P1: 8 operations) or of the fixed-point
    values (2^-54 of the tile's largest, rows of |K| / 8 <= 216 against diagonals >= 48, tiles of U(-1, 1) values);
    a P2 field keeps its element kernels.  FP32 within 1e-5, as every FP32 operator."""
    with fe.Hierarchy(N, 0, k) as h:
        n_cells = h.n_cells()
        kappa = {"one": np.ones(n_cells), "constant": np.full(n_cells, 0.7),
                 "field": np.exp(I.random_vector(n_cells, 5))}[coef]
        if coef != "one":
            h.set_coefficient(dt(kappa))
        L = O.Level(N, k, kappa)
        x = I.random_vector(L.n, 3)
        ref, scale = L.A @ x, abs(L.A) @ np.abs(x)
        tol = 1e-13 if (k == 2 and coef == "field") else 1e-14
        assert np.all(np.abs(apply(fe, h, x) - ref) <= tol * np.maximum(scale, 1e-300))
        x32 = x.astype(np.float32)
        ref, scale = L.A @ x32.astype(float), abs(L.A) @ np.abs(x32.astype(float))
        assert np.all(np.abs(apply(fe, h, x32, torch.float32) - ref) <= 1e-5 * scale + 1e-30)


@pytest.mark.parametrize("N", [12, 20])
def test_value_ranges_within_one_tile(fe, N):
    """P2, values that differ by 2^0 .. 2^300 from one region of the mesh to the next: tiles are summed in several
    windows, so every row stays within 1e-13 of the largest |A| |x| of its cell's eight rows (windows of 2^-59, cells at
    most 2^15 below the largest value of their pass)."""
    with fe.Hierarchy(N, 0, 2) as h:
        L = O.Level(N, 2)
        A = L.A.copy()
        A.data[np.abs(A.data) < 1e-12 * np.abs(A.data).max()] = 0.0  # entries that cancel but for rounding
        X = h.dof_coordinates()
        c = np.rint(X * 2 * N).astype(int) // 2
        cell, N_cells = c[:, 0] + (N + 1) * (c[:, 1] + (N + 1) * c[:, 2]), (N + 1) ** 3
        for big in (2.0 ** 9, 2.0 ** 20, 2.0 ** 70, 2.0 ** 300):
            x = I.random_vector(L.n, 9)
            x[X[:, 0] + X[:, 2] < 0.7] *= big
            x[(X[:, 1] > 0.8)] *= 1 / big
            ref, scale = A @ x, abs(A) @ np.abs(x)
            np.maximum.at(cell_scale := np.zeros(N_cells), cell, scale)
            assert np.all(np.abs(apply(fe, h, x) - ref) <= 1e-13 * cell_scale[cell]), big


@pytest.mark.parametrize("k,N", [(1, 6), (2, 6), (2, 20)])
@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_non_finite_values(fe, k, N, bad):
    """A value that is not finite makes the rows that couple to it non-finite and leaves rows further away as they were;
    on the boundary it only comes back in its own (identity) row."""
    with fe.Hierarchy(N, 0, k) as h:
        L = O.Level(N, k)
        X = h.dof_coordinates()
        x = I.random_vector(L.n, 4)
        good = apply(fe, h, x)
        i = np.argmin(np.abs(X - 0.5).sum(1))
        x[i] = bad
        y = apply(fe, h, x)
        row = L.A[i].toarray()[0]
        rows = np.nonzero(np.abs(row) > 1e-12 * np.abs(row).max())[0]
        assert not np.isfinite(y[rows]).any()
        far = np.abs(X - X[i]).max(1) > 2.01 / N
        assert far.any() and np.array_equal(y[far], good[far])
        x[i] = 0.5
        edge = np.nonzero(X[:, 0] == 0)[0][5]
        x[edge] = bad
        y = apply(fe, h, x)
        assert not np.isfinite(y[edge]) and np.isfinite(np.delete(y, edge)).all()


@pytest.mark.parametrize("k,N0,coef", [(1, 3, "field"), (2, 3, "one"), (2, 5, "one"), (2, 10, "constant")])
@pytest.mark.parametrize("steps", [1, 2, 3, 4])
@pytest.mark.parametrize("f32", [False, True])
def test_chebyshev_steps_in_one_launch(fe, k, N0, coef, steps, f32):
    """Chebyshev steps formed in the operator's launch (from one vector to another) equal the oracle's, odd and even
    numbers of them; b, x and the tolerance as for the separate kernels (1e-12 of the iterate, FP32 1e-5)."""
    with fe.Hierarchy(N0, 1, k) as h:
        kappa = np.exp(I.random_vector(h.n_cells(), 5)) if coef == "field" else np.full(
            h.n_cells(), 1.0 if coef == "one" else 0.7)
        h.set_coefficient(dt(kappa))
        oh = O.Hierarchy(N0, 1, k, kappa)
        L = oh.levels[1]
        lmax = h.lambda_max(1)
        b, x0 = I.random_vector(L.n, 6), I.random_vector(L.n, 7)
        ref = O.chebyshev(lambda v: L.A @ v, L.diag, b, x0, 0.1 * lmax, 1.1 * lmax, steps)
        d = torch.float32 if f32 else torch.float64
        x = dt(x0, d)
        h.smooth(dt(b, d), x, level=1, steps=steps, dtype=fe.FE_F32 if f32 else fe.FE_F64)
        got = x.double().cpu().numpy()
        assert np.abs(got - ref).max() <= (1e-5 if f32 else 1e-12) * np.abs(ref).max()


@pytest.mark.parametrize("scale", [1e-300, 1e-200, 1e-8, 1.0, 1e200, 1e300])
def test_p3_integer_element_value_range(fe, scale):
    """P3 rows within 1e-14 of |A| |x| from 1e-300 to 1e300 (exact integer sums, one rounding per contribution, up to 24
    contributions per row; 2 N = 6 extra ulps for the integers' cut below 2^-59), exact zeros, NaN dofs propagate."""
    with fe.Hierarchy(3, 0, 3) as h:
        kappa = np.exp(I.random_vector(h.n_cells(), 5))
        h.set_coefficient(dt(kappa))
        L = O.Level(3, 3, kappa)
        x = I.random_vector(L.n, 77) * scale
        x[::7] = 0.0
        assert np.all(np.abs(apply(fe, h, x) - L.A @ x) <= 1e-14 * np.maximum(abs(L.A) @ np.abs(x), 1e-307))
        assert not apply(fe, h, np.zeros(L.n)).any()
        i = np.nonzero(~L.space.boundary)[0][7]
        x[i] = np.nan
        row = np.abs(L.A[i].toarray()[0])
        assert np.isnan(apply(fe, h, x)[row > 1e-12 * row.max()]).all()


@pytest.mark.parametrize("N0", [4, 5])
def test_fp32_cycle_with_tiled_restriction_matches_fp64(fe, N0):
    """The FP32 V-cycle restricts 64^3 (and 80^3: ragged tiles) with staged tiles; it equals the FP64 cycle to FP32
    rounding (5e-6 of the largest entry, as every FP32 cycle here)."""
    with fe.Hierarchy(N0, 4, 2) as h:
        b = I.random_vector(h.n_dofs(), 3)
        b[h.boundary_mask()] = 0.0
        x, x32 = torch.empty(len(b), dtype=torch.float64, device=DEV), torch.empty(len(b), device=DEV)
        h.vcycle(dt(b), x)
        h.vcycle(dt(b, torch.float32), x32, dtype=fe.FE_F32)
        assert (x32.double() - x).abs().max() <= 5e-6 * x.abs().max()


@pytest.mark.parametrize("k,N0,levels,coef", [(1, 3, 2, "field"), (2, 2, 2, "one"), (2, 3, 3, "constant"), (2, 3, 2, "field"),
                                              (3, 2, 2, "field")])
@pytest.mark.parametrize("f32", [False, True])
def test_cycle_residuals_match_oracle(fe, k, N0, levels, coef, f32):
    """Cycles whose operator leaves b - A x for the restriction (small and tiled levels, 24 cubes the largest) equal the
    oracle's: 1e-11 of the largest entry as for the cycles' parity tests, FP32 1e-5 (condition of the coarse solve)."""
    with fe.Hierarchy(N0, levels, k) as h:
        kappa = np.exp(I.random_vector(h.n_cells(), 5)) if coef == "field" else np.full(
            h.n_cells(), 1.0 if coef == "one" else 0.7)
        h.set_coefficient(dt(kappa))
        oh = O.Hierarchy(N0, levels, k, kappa)
        for l in range(levels + 1):
            oh.lmax[l] = h.lambda_max(l)
        b = I.random_vector(h.n_dofs(), 6)
        b[h.boundary_mask()] = 0.0
        ref = oh.vcycle(b)
        x = torch.empty(len(b), dtype=torch.float32 if f32 else torch.float64, device=DEV)
        h.vcycle(dt(b, x.dtype), x, dtype=fe.FE_F32 if f32 else fe.FE_F64)
        assert np.abs(x.double().cpu().numpy() - ref).max() <= (1e-5 if f32 else 1e-11) * np.abs(ref).max()


@pytest.mark.parametrize("N0", [4, 5])
def test_fp64_tiled_restriction_matches_table(fe, N0):
    """The FP64 restriction to 32^3 and 40^3 (ragged tiles) by staged tiles (boundary rows zeroed) equals the table-driven
    one (boundary rows kept): two sums of at most 125 terms, weights and values at most 1, differ by at most
    2 * 125 * 125 * 2^-53; a NaN reaches exactly the same rows."""
    with fe.Hierarchy(N0, 4, 2) as h:
        r = dt(I.random_vector(h.n_dofs(), 3))
        inner = torch.from_numpy(~h.boundary_mask(3)).to(DEV)
        tiled, table = (torch.empty(h.n_dofs(3), dtype=torch.float64, device=DEV) for _ in range(2))
        for bad in (None, 12345):
            if bad is not None:
                r[bad] = float("nan")
            h.restrict(r, tiled, 4, zero_boundary=True)
            h.restrict(r, table, 4, zero_boundary=False)
            assert not tiled[~inner].any()
            a, b = tiled[inner], table[inner]
            assert torch.equal(torch.isnan(a), torch.isnan(b))
            assert (a - b).nan_to_num().abs().max() <= 2 * 125 * 125 * 2.0 ** -53


@pytest.mark.parametrize("N0", [2, 8, 9])
def test_p3_restriction_is_the_transpose(fe, N0):
    """P3 restriction by 32 warps per 32 coarse points (8^3, 15,625 points, the largest) and by 16 (9^3): (P c) . r = c . (R r)
    to the rounding of sums of n terms, each entry of at most 343 (1e-12 of the norms' product)."""
    with fe.Hierarchy(N0, 1, 3) as h:
        r, c = dt(I.random_vector(h.n_dofs(), 3)), dt(I.random_vector(h.n_dofs(0), 4))
        rc, pc = torch.empty_like(c), torch.empty_like(r)
        h.restrict(r, rc, 1, zero_boundary=False)
        h.prolong(c, pc, 1)
        assert abs(float(pc @ r - c @ rc)) <= 1e-12 * float(pc.norm() * r.norm())


@pytest.mark.parametrize("dtype", ["f64", "f32"])
def test_vcycle_replayed_and_captured(fe, dtype):
    """The V-cycle's later calls replay its graph: with new inputs, other buffers and a changed coefficient they equal the
    first call's result for those inputs (bitwise up to the order of atomic additions, 1e-13 / 1e-5 of the largest entry),
    also inside a graph that the caller captures."""
    d = torch.float64 if dtype == "f64" else torch.float32
    code, tol = (fe.FE_F64, 1e-13) if dtype == "f64" else (fe.FE_F32, 1e-5)
    kappas = [np.ones(6 * 16 ** 3), np.exp(I.random_vector(6 * 16 ** 3, 5))]
    with fe.Hierarchy(4, 2, 2) as h, fe.Hierarchy(4, 2, 2) as fresh:
        b = [dt(I.random_vector(h.n_dofs(), s), d) for s in (1, 2, 3)]
        for kappa in kappas:
            h.set_coefficient(dt(kappa))
            for i in range(3):
                fresh.set_coefficient(dt(kappa))  # its next call is a first one
                x, ref = torch.empty_like(b[i]), torch.empty_like(b[i])
                h.vcycle(b[i], x, dtype=code)
                fresh.vcycle(b[i], ref, dtype=code)
                assert (x - ref).abs().max() <= tol * ref.abs().max()
        y, stream = torch.empty_like(b[0]), torch.cuda.Stream()
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=stream):
            h.vcycle(b[2], y, dtype=code, stream=stream)
        y.zero_()
        g.replay()
        torch.cuda.synchronize()
        assert (y - ref).abs().max() <= tol * ref.abs().max()
