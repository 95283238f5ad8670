"""The fixed-point factorisation of the fit at the sizes where its layout changes: edges of the 8-column panels, of the
32-row groups, of the size classes (one warp up to 95, teams up to 159, global slots above) and the largest cell, each a
single cell fitted through the public call and compared with numpy in extended precision.  Bars: A = L L^T to 2e-13 (an
entry of A is within 1e-13 of its value, from the coordinates' fixed-point rounding, and the factorisation adds less),
alpha to 1e-9 relative to its largest entry.  Also the cells that must take the binary64 path (a variance of 0, below
2^-20 or above 0.25), the Matern kernel, 2D, and a cell whose forward solve leaves the fixed-point range.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2603_29227_gb300 import ksdf  # noqa: E402

DEV = torch.device("cuda:0")
SIZES = [1, 2, 7, 8, 9, 31, 32, 33, 63, 64, 65, 71, 72, 79, 80, 95, 96, 97, 127, 128, 129, 159, 160, 161, 215, 255, 256,
         257, 300, 504, 505, 511, 512]


def _fit(x, var, lam, kernel=0):
    n, dim = x.shape
    m = ksdf.KernelSDF(dict(dim=dim, origin=(0.0, 0.0, 0.0), cell=1.0, margin=0.0, n_max=512, k_cand=1, kernel=kernel,
                            **{"lambda": lam}))
    m.fit(torch.from_numpy(x).to(DEV), None if var is None else torch.from_numpy(var).to(DEV))
    alpha, chol, _ = m.fit_arrays()
    L = np.zeros((n, n))
    L[np.tril_indices(n)] = chol
    return m, alpha, L


def _check(x, var, lam, kernel=0):
    n = len(x)
    m, alpha, L = _fit(x, var, lam, kernel)
    assert m.fit_status == 0 and m.cells()[1].tolist() == [0]
    X = x.astype(np.longdouble)
    r2 = ((X[:, None] - X[None]) ** 2).sum(-1)
    z = np.longdouble(lam) * np.sqrt(r2)
    K = (1 + z) * np.exp(-z) if kernel else np.exp(-np.longdouble(lam) * r2)
    v = np.zeros(n) if var is None else var
    A = K + np.diag(v.astype(np.longdouble))
    Lx = L.astype(np.longdouble)
    assert np.max(np.abs(Lx @ Lx.T - A)) <= 2e-13, n
    ref = np.linalg.solve(A.astype(np.float64), np.ones(n))
    r = 1 - A @ ref.astype(np.longdouble)  # one step of refinement
    ref = ref + np.linalg.solve(A.astype(np.float64), r.astype(np.float64))
    assert np.max(np.abs(alpha - ref)) <= 1e-9 * np.max(np.abs(ref)), n


def _points(n, dim=3, seed=0):
    rng = np.random.default_rng(100 * n + seed)
    x = rng.uniform(0.05, 0.95, (n, dim))
    x[:, -1] = 0.5 + 0.02 * rng.standard_normal(n)  # near a plane, like surface samples
    return x, ((0.01 * rng.uniform(0.5, 2.0, n)) ** 2).astype(np.float32)


@pytest.mark.parametrize("n", SIZES)
def test_sizes(n):
    x, var = _points(n)
    _check(x, var, 300.0)


@pytest.mark.parametrize("n", [5, 80, 200, 400])
def test_matern_and_2d(n):
    x, var = _points(n)
    _check(x, var, 100.0, kernel=1)
    x, var = _points(n, dim=2)
    _check(x, var, 500.0)


@pytest.mark.parametrize("value", [0.0, 0.99 * 2.0 ** -20, 2.0 ** -20, 0.25, 0.2500001, 3.0])
@pytest.mark.parametrize("n", [40, 130])
def test_variance_bounds(n, value):
    x, var = _points(n)
    var[n // 2] = value
    _check(x, var, 300.0)


def test_y_out_of_range():
    # four points found by search: L^-1 1 ends with 1.00085
    p = np.array([[2.131, 0.274], [2.234, 0.232], [2.344, 0.213], [1.639, -1.838]])
    x = np.ascontiguousarray((p - p.min(0)) / 4 + 0.2)  # distances over 4: lambda 16 for the kernel of distance 1
    var = np.full(4, 2.0 ** -19, dtype=np.float32)
    A = np.exp(-16.0 * ((x[:, None] - x[None]) ** 2).sum(-1)) + np.diag(var.astype(np.float64))
    assert np.linalg.solve(np.linalg.cholesky(A), np.ones(4)).max() > 1.0005
    _check(x, var, 16.0)
