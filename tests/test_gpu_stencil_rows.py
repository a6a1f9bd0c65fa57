"""The operator by rows where a caller's use leaves the ordinary case: a change of the geometry form before a call on a
stream of its own; values of very different size side by side; coefficients far from 1 in mixed precision; V-cycles
between solves with other smoothing; the pair-of-tets operator on the levels of a cycle;
bf16 applications after hierarchies that used both geometry forms."""
import functools

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


@pytest.mark.parametrize("N", [3, 40])
def test_geometry_form_is_complete_on_return(fe, N):
    """A coefficient set under the per-cell form gets its edge weights when the form changes back; an application on a
    non-blocking stream right after that call reads them (1e-14 of |A| |x| per row, as every P1 application by rows)."""
    with fe.Hierarchy(N, 0, 1) as h:
        kappa = np.exp(I.random_vector(h.n_cells(), 5))
        L = O.Level(N, 1, kappa)
        x = I.random_vector(L.n, 3)
        xd, y, k, stream = dt(x), torch.empty(L.n, dtype=torch.float64, device=DEV), dt(kappa), torch.cuda.Stream()
        h.set_geometry_form(fe.FE_GEOMETRY_PER_CELL)
        h.set_coefficient(k)
        torch.cuda.synchronize()
        h.set_geometry_form(fe.FE_GEOMETRY_AUTO)
        h.apply_operator(xd, y, stream=stream)
        stream.synchronize()
        assert np.all(np.abs(y.cpu().numpy() - L.A @ x) <= 1e-14 * np.maximum(abs(L.A) @ np.abs(x), 1e-300))


# ------------------------------------------------- P2 rows, value by value
@functools.lru_cache(None)
def p2_stencils():
    """Per parity code of the lattice point: {offset: integer coefficient} of its row in units of 8 c, c = 1 / (120 N),
    read from the oracle's assembled matrix around the centre of a 4^3 mesh."""
    L = O.Level(4, 2)
    X = np.rint(L.space.coords * 8).astype(int)
    out = {}
    for code in range(8):
        p = np.array([4 + (code & 1), 4 + (code >> 1 & 1), 4 + (code >> 2)])
        i = int(np.nonzero((X == p).all(1))[0][0])
        row = L.A[i].tocoo()
        k = row.data * (120 * 4) / 8
        assert np.abs(k - np.rint(k)).max() < 1e-9
        out[code] = {tuple(X[j] - p): int(v) for j, v in zip(row.col, np.rint(k)) if v}
    return out


def p2_rows(x, X, N):
    """A x and |A| |x| of interior rows for kappa = 1 on N^3 cubes, x at the lattice points X: products with the integers
    exact, sums by TwoSum."""
    c = torch.zeros((2 * N + 5,) * 3, dtype=torch.float64, device=DEV)
    X = torch.from_numpy(X).to(DEV)
    inner = ((X > 0) & (X < 2 * N)).all(1)
    at = tuple((X + 2).T)
    c[at] = torch.where(inner, x, torch.zeros_like(x))
    hi = c.view(torch.int64).bitwise_and(-(1 << 27)).view(torch.float64)  # 26 bits, the rest in c - hi
    y, a = torch.zeros_like(x), torch.zeros_like(x)
    for code, st in p2_stencils().items():
        sel = inner & (X[:, 0] % 2 + 2 * (X[:, 1] % 2) + 4 * (X[:, 2] % 2) == code)
        P = X[sel] + 2
        s = e = m = torch.zeros(len(P), dtype=torch.float64, device=DEV)
        for o, k in st.items():
            q = tuple((P + torch.tensor(o, device=DEV)).T)
            m = m + abs(k) * c[q].abs()
            for t in (k * hi[q], k * (c[q] - hi[q])):
                z = s + t
                w = z - s
                e = e + ((s - (z - w)) + (t - w))
                s = z
        y[sel], a[sel] = (s + e) * (8 / (120 * N)), m * (8 / (120 * N))
    return y, a, inner


def contrasts(kind, X, N):
    """Vectors whose values differ by powers of two from one lattice point to the next."""
    rng = np.random.default_rng(7)
    x = np.zeros(len(X))
    if kind.startswith("pair"):  # one large and one far smaller value in the same tile, zeros around
        x[(X == [5, 5, 5]).all(1)] = 1.0
        x[(X == [12, 4, 7]).all(1)] = 0.7 * 2.0 ** -int(kind[4:])
    elif kind.startswith("step"):  # small values beside a region of large ones
        x = rng.uniform(-1, 1, len(X))
        x[X[:, 0] > 9] *= 2.0 ** -int(kind[4:])
    elif kind == "any":  # every exponent from 2^-60 to 1, a fifth of the values zero
        x = rng.uniform(0.5, 1, len(X)) * rng.choice([-1.0, 1.0], len(X)) * 2.0 ** -rng.integers(0, 61, len(X))
        x[::5] = 0.0
    elif kind == "class":  # only one parity class is of size 1: rows that do not couple to it stand alone
        x = rng.uniform(-1, 1, len(X)) * 2.0 ** -45
        x[(X % 2 == [1, 0, 0]).all(1)] *= 2.0 ** 45
    else:  # far from 1
        x = rng.uniform(-1, 1, len(X)) * 2.0 ** float(kind)
    return x


KINDS = ["pair20", "pair40", "pair70", "step12", "step13", "step16", "step40", "any", "class", "-900", "900"]


# tiles of 16 x 4 x 4 cells with remainders (17, 33) and whole in y and z (20); the larger tile from 97 on
@pytest.mark.parametrize("N", [17, 20, 33, 97])
@pytest.mark.parametrize("kind", KINDS)
def test_p2_rows_keep_their_own_bits(fe, N, kind):
    """One coefficient, FP64: every row is within 1e-14 of its own |A| |x|, whatever the values around it are: less than
    2^-47 (7.2e-15) of it is cut off the rows formed from the tile's scale and 216 2^-59 (3.8e-16) off those with a scale
    of their own; both are then rounded three times (3.4e-16)."""
    with fe.Hierarchy(N, 0, 2) as h:
        X = np.rint(h.dof_coordinates() * 2 * N).astype(int)
        x = dt(contrasts(kind, X, N))
        y = torch.empty_like(x)
        h.apply_operator(x, y)
        ref, scale, inner = p2_rows(x, X, N)
        assert ((y - ref).abs() <= 1e-14 * scale)[inner].all()
        assert torch.equal(y[~inner], x[~inner])


@pytest.mark.parametrize("kind", ["pair40", "step13", "any", "class"])
def test_p2_chebyshev_rows_keep_their_own_bits(fe, kind):
    """The same rows inside a Chebyshev step (two, from one vector to another and back): x + d is within 1e-14 of the sum of
    the magnitudes it is formed of, applied to the step's own input.  N = 20."""
    N = 20
    with fe.Hierarchy(10, 1, 2) as h:
        X = np.rint(h.dof_coordinates() * 2 * N).astype(int)
        x = dt(contrasts(kind, X, N))
        b = x * 0.5
        lmax = h.lambda_max()
        lo, hi = 0.1 * lmax, 1.1 * lmax
        theta, delta = 0.5 * (hi + lo), 0.5 * (hi - lo)
        sigma = theta / delta
        diag = torch.empty_like(x)
        h.diagonal(diag)
        ref, bound, d, db = x.clone(), torch.zeros_like(x), None, None
        rho = 1 / sigma
        for k in range(2):
            y, a, inner = p2_rows(ref, X, N)
            _, spread, _ = p2_rows(bound, X, N)  # an error of x reaches the next step through |A|
            y, a = torch.where(inner, y, ref), torch.where(inner, a, ref.abs())
            if k == 0:
                c1, c2 = 0.0, 1 / theta
                d, db = c2 / diag * (b - y), c2 / diag * (b.abs() + a)
            else:
                rn = 1 / (2 * sigma - rho)
                c1, c2 = rn * rho, 2 * rn / delta
                d, db = c1 * d + c2 / diag * (b - y), c1 * db + c2 / diag * (b.abs() + a)
            bound = bound + c2 / diag * spread + c1 * bound + 1e-14 * (ref.abs() + db)
            ref = ref + d
        h.smooth(b, x, steps=2)
        assert ((x - ref).abs() <= bound).all()


# the direct kernel (12) and the tiled one, whose tiles stage such values as 0
@pytest.mark.parametrize("N", [12, 20, 97])
@pytest.mark.parametrize("bad", ["nan", "inf", "-inf", "both"])
def test_p2_non_finite_values_reach_their_rows_only(fe, N, bad):
    """A NaN or infinity in the cell of the vector's largest value makes exactly the rows that couple to it what IEEE
    arithmetic makes of them (NaN; an infinity of the coefficient's sign; NaN where two of opposite sign meet), and every
    other row keeps its bits."""
    with fe.Hierarchy(N, 0, 2) as h:
        X = np.rint(h.dof_coordinates() * 2 * N).astype(int)
        x = dt(I.random_vector(len(X), 4))
        at = lambda p: int(np.nonzero((X == p).all(1))[0][0])
        p = np.array([9, 8, 8])
        x[at(p + [1, 1, 0])] = 2.0 ** 13  # (the rows around keep their scale without the value beside it)
        good, y = torch.empty_like(x), torch.empty_like(x)
        h.apply_operator(x, good)
        put = {"both": [(p, np.inf), (p + [2, 0, 0], -np.inf)]}.get(bad, [(p, float(bad if bad != "both" else 0))])
        want = good.cpu().numpy().copy()
        index = {tuple(X[i]): i for i in np.nonzero((np.abs(X - p) <= 6).all(1))[0]}
        add = {}
        for q, v in put:
            x[at(q)] = v
            for o in np.ndindex(5, 5, 5):
                r = tuple(q - (np.array(o) - 2))  # row r couples to q = r + o
                if not all(0 < c < 2 * N for c in r):
                    continue
                k = p2_stencils()[r[0] % 2 + 2 * (r[1] % 2) + 4 * (r[2] % 2)].get(tuple(np.array(o) - 2), 0)
                if k:
                    add[r] = add.get(r, 0.0) + k * v
        for r, v in add.items():
            want[index[r]] = v
        h.apply_operator(x, y)
        assert np.array_equal(y.cpu().numpy(), want, equal_nan=True)


# vectors below and above 2^19 entries, from where on the update's sums too are formed in floats
@pytest.mark.parametrize("k,n0,levels", [(1, 4, 2), (2, 4, 2), (2, 11, 2)])
@pytest.mark.parametrize("e", [-80, 100, 118, 122])
def test_mixed_solve_scales_with_the_coefficient(fe, k, n0, levels, e):
    """kappa = 2^e scales the whole solve by powers of two (2^122: entries of r . z down to 2^-170, outside FP32): the
    iterations of kappa = 1, and its solution to the solve's tolerance (1e-9)."""
    with fe.Hierarchy(n0, levels, k) as h:
        f = dt(I.sin_product_rhs(h.dof_coordinates()))
        u, v = torch.empty_like(f), torch.empty_like(f)
        one = h.solve(f, u, precision=fe.FE_PREC_MIXED_F32, rtol=1e-10)
        h.set_coefficient(torch.full((h.n_cells(),), 2.0 ** e, dtype=torch.float64, device=DEV))
        st = h.solve(f, v, precision=fe.FE_PREC_MIXED_F32, rtol=1e-10)
        assert (st.iterations, st.outer_iterations) == (one.iterations, one.outer_iterations)
        assert float((v * 2.0 ** e - u).norm()) <= 1e-9 * float(u.norm())


def recorded(run, name):
    """How many CUDA runtime calls or kernels whose name holds `name` the profiler records during run()."""
    from torch.profiler import ProfilerActivity, profile
    with profile(activities=[ProfilerActivity.CPU, ProfilerActivity.CUDA]) as prof:
        run()
        torch.cuda.synchronize()
    return sum(e.count for e in prof.key_averages() if name in e.key)


def graphs_built(run):
    return recorded(run, "GraphInstantiate")


@pytest.mark.parametrize("dtype", ["f64", "f32"])
def test_vcycles_and_solves_keep_their_graphs(fe, dtype):
    """A caller that alternates V-cycles (two smoothing steps) with solves of three steps builds each graph once."""
    code, d = (fe.FE_F64, torch.float64) if dtype == "f64" else (fe.FE_F32, torch.float32)
    prec = fe.FE_PREC_F64 if dtype == "f64" else fe.FE_PREC_MIXED_F32
    with fe.Hierarchy(4, 2, 2) as h:
        f = dt(I.sin_product_rhs(h.dof_coordinates()))
        u, b = torch.empty_like(f), f.to(d)
        x = torch.empty_like(b)

        def both():
            h.solve(f, u, precision=prec, cheb_steps=3)
            for _ in range(3):
                h.vcycle(b, x, dtype=code)

        graphs_built(torch.cuda.synchronize)  # (a process's first recording can miss calls)
        if graphs_built(both) == 0:
            pytest.skip("the profiler records no runtime calls here")
        ref = x.clone()
        assert graphs_built(both) == 0
        assert (x - ref).abs().max() <= (1e-13 if dtype == "f64" else 1e-5) * ref.abs().max()


def test_vcycle_with_pairs_of_tets_on_every_level(fe):
    """A coefficient per coarsest cube varies over the mesh and agrees on the two tets of every pair on all levels: the
    cycle's FP64 operator takes pairs of tets (not one coefficient's stencils, nor single tets) below the finest level
    too, and equals the oracle's cycle (1e-11 of its norm, as for the other coefficients)."""
    with fe.Hierarchy(2, 2, 2) as h:
        cube = np.floor(h.cell_centroids() * 2).astype(int) @ [1, 2, 4]
        kappa = np.exp(I.random_vector(8, 5))[cube]
        h.set_coefficient(dt(kappa))
        oh = O.Hierarchy(2, 2, 2, kappa)
        oh.lmax = [h.lambda_max(l) for l in range(3)]
        b = I.random_vector(oh.fine.n, 5)
        b[oh.fine.space.boundary] = 0
        bd, x = dt(b), torch.empty(oh.fine.n, dtype=torch.float64, device=DEV)
        names = []
        recorded(torch.cuda.synchronize, "")
        for name in ("KuhnPair", "KuhnTet", "k_stencil2"):
            h.set_coefficient(dt(kappa))  # (the next cycle's kernels are launched, not replayed)
            names.append(recorded(lambda: h.vcycle(bd, x), name))
        ref = oh.vcycle(b)
        assert np.linalg.norm(x.cpu().numpy() - ref) <= 1e-11 * np.linalg.norm(ref)
        if not any(names):
            pytest.skip("the profiler records no kernels here")
        assert names[0] > 0 and names[1:] == [0, 0]  # (8 applications, four on each of two levels)


# (FP32: up to where the sums of a P2 element stay in its range)
@pytest.mark.parametrize("k,N,e32", [(1, 3, 126), (1, 40, 126), (2, 3, 123), (2, 12, 123), (2, 20, 123), (3, 3, None)])
@pytest.mark.parametrize("coef", ["one", "field"])
def test_rows_up_to_the_end_of_the_range(fe, k, N, e32, coef):
    """Values up to 2^1022 (FP32 2^126 and 2^123), whose rows lie in the range although 54 times a value does not: 2^1022
    times the rows of the same values below 1, up to 1e-13 of |A| |x| (the element kernels' tolerance; FP32 1e-5)."""
    with fe.Hierarchy(N, 0, k) as h:
        kappa = np.exp(I.random_vector(h.n_cells(), 5)) if coef == "field" else np.ones(h.n_cells())
        h.set_coefficient(dt(kappa))
        L = O.Level(N, k, kappa)
        x = I.random_vector(L.n, 3)
        x *= min(1.0, 2 / (abs(L.A) @ np.abs(x)).max())  # (rows in range)
        for d, code, e, tol in ((torch.float64, fe.FE_F64, 1022, 1e-13), (torch.float32, fe.FE_F32, e32, 1e-5)):
            if e is None:
                continue
            xd = dt(x, d)
            y = torch.empty_like(xd)
            h.apply_operator(xd * 2.0 ** e, y, dtype=code)
            v = xd.double().cpu().numpy()
            ref, scale = L.A @ v, abs(L.A) @ np.abs(v)
            assert np.all(np.abs(y.double().cpu().numpy() * 2.0 ** -e - ref) <= tol * scale), d


@pytest.mark.parametrize("k", [1, 2])
def test_bf16_after_hierarchies_with_both_geometry_forms(fe, k):
    """A level's tensor maps of both geometry forms go with it: hierarchies that come to lie at its address afterwards,
    with other sizes and buffers, apply their own operator (two bf16 terms per value, 16 bits: 1e-4 of |A| |x|)."""
    for N in (6, 9, 7, 6, 10, 8):
        with fe.Hierarchy(N, 0, k) as h:
            kappa = np.exp(I.random_vector(h.n_cells(), 5))
            h.set_coefficient(dt(kappa))
            L = O.Level(N, k, kappa)
            x = I.random_vector(L.n, N).astype(np.float32).astype(float)
            ref, scale = L.A @ x, abs(L.A) @ np.abs(x)
            xd, y = dt(x, torch.float32), torch.empty(L.n, device=DEV)
            for form in (fe.FE_GEOMETRY_AUTO, fe.FE_GEOMETRY_PER_CELL):
                h.set_geometry_form(form)
                h.apply_operator(xd, y, dtype=fe.FE_BF16)
                assert np.all(np.abs(y.double().cpu().numpy() - ref) <= 1e-4 * scale)
