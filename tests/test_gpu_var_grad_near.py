"""The gradient variance of the mixed path where its squares leave FP32's range: a query a hair off a sample on a cell
face (local coordinates that small are exact), and queries so far from the cell that any stand-in for a missing sample
could be nearer than the samples.  Reference: the plain FP64 query of the same inputs.  Bar: norm-wise 1e-3 per query, the
mixed path's for this output.  Here every coordinate is exact in FP32 and one sample's terms (or, far away, those of
near-equal samples) make up the result, so the FP32 error is a few 1e-6 near and, from alpha times the distance's rounding of
2 m, a few 1e-5 far away.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2603_29227_gb300 import ksdf  # noqa: E402

DEV = torch.device("cuda:0")


def _check(p, x, xq):
    var = np.full(len(x), 1e-4, dtype=np.float32)
    m = ksdf.KernelSDF(p)
    m.fit(torch.from_numpy(x).to(DEV), torch.from_numpy(var).to(DEV))
    assert len(m.cells()[1]) == 1
    a = m.query(torch.from_numpy(xq).to(DEV), mask=ksdf.OUT_VAR_GRAD)["var_grad"].cpu().numpy().astype(np.float64)
    b = m.query(torch.from_numpy(xq.astype(np.float64)).to(DEV), mask=ksdf.OUT_VAR_GRAD, f64=True)["var_grad"].cpu().numpy()
    m.sync_status()
    assert np.all(np.isfinite(b)) and np.all(np.max(b, axis=1) > 0)
    err = np.max(np.abs(a - b), axis=1)
    assert np.all(err <= 1e-3 * np.max(b, axis=1)), (a, b)  # (NaN and inf fail too)


@pytest.mark.parametrize("n", [1, 2, 7, 16])
@pytest.mark.parametrize("dim", [2, 3])
def test_a_hair_off_a_sample(dim, n):
    # samples on the face z = 0 (y = 0 in 2D); 1 / 2 sigma_i / z below FP32's largest number
    p = dict(dim=dim, origin=(0.0, 0.0, 0.0), cell=4.0, margin=0.0, n_max=64, k_cand=1, **{"lambda": 300.0})
    i = np.arange(n)
    x = np.zeros((n, dim))
    x[:, 0] = 0.25 + 0.125 * (i % 16)
    if dim == 3:
        x[:, 1] = 0.25 + 0.125 * (i % 5)
    eps = np.array([1e-18, 1e-15, 1e-12, 1e-11, 1e-10, 2.3e-10, 1e-9, 1e-6, 1e-3], dtype=np.float32)
    xq = np.repeat(x.astype(np.float32), len(eps), axis=0)
    xq[:, -1] = np.tile(eps, n)
    _check(p, x, xq)


def test_a_hair_off_a_corner():
    # a sample in the cell's corner: offsets along every axis and diagonal
    p = dict(dim=3, origin=(0.0, 0.0, 0.0), cell=4.0, margin=0.0, n_max=64, k_cand=1, **{"lambda": 300.0})
    x = np.array([[0.0, 0.0, 0.0], [0.5, 0.0, 0.25], [0.0, 0.75, 0.5]])
    d = np.array([[1, 0, 0], [0, 1, 0], [0, 0, 1], [1, 1, 0], [1, 0, 2], [1, 2, 3]], dtype=np.float32)
    xq = np.concatenate([d * np.float32(e) for e in (1e-17, 1e-13, 1e-10, 1e-7)])
    _check(p, x, xq)


@pytest.mark.parametrize("n", [1, 2, 5, 6])
def test_far_from_the_cell(n):
    # 5e7 m away, inside the grid of 2^20 cells of 64 m; a temperature that tells samples 30 m apart hardly apart
    p = dict(dim=3, origin=(0.0, 0.0, 0.0), cell=64.0, margin=0.0, n_max=64, k_cand=1, softmin_alpha=1e-5,
             **{"lambda": 1e-3})
    rng = np.random.default_rng(n)
    x = np.round(rng.uniform(1.0, 63.0, (n, 3)))
    xq = np.array([[3e7, 3e7, 3e7], [5e7, 1e7, 2e7], [-4e7, -4e7, 1e7], [2e7, 2e7, 6e7], [1e7, 1e7, 1e7]], dtype=np.float32)
    _check(p, x, xq)
