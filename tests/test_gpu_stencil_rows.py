"""The operator by rows where a caller's use leaves the ordinary case: a change of the geometry form before a call on a
stream of its own."""
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
