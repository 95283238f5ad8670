"""Small batches are grouped by one CTA (up to 2,048 queries) and larger ones by the general passes: every query's outputs
must not depend on which one ran.  Each batch is answered alone and inside a batch of 5,000; the outputs and the query
gradients are compared bit for bit (a query's arithmetic does not depend on its tile).  Batches hold invalid queries (NaN, out of the grid), repeated
points, far points and winners in all three size classes of phase B.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2603_29227_gb300 import ksdf, scenes  # noqa: E402

DEV = torch.device("cuda:0")
SIZES = [1, 2, 3, 31, 33, 127, 128, 129, 1000, 1023, 1024, 1025, 2047, 2048]


def _t(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to(DEV)


@pytest.fixture(scope="module")
def model():
    w = scenes.workload("room3d", n_samples=120_000, n_queries=5000)
    # a dense patch gives cells of several hundred samples beside the ordinary ones
    rng = np.random.default_rng(0)
    x2 = np.column_stack([rng.uniform(3.0, 4.2, (4000, 2)), 0.01 * rng.standard_normal(4000)])
    x = np.concatenate([w.x, x2])
    var = np.concatenate([w.var, np.full(4000, 1e-4, np.float32)])
    m = ksdf.KernelSDF(dict(w.params, n_max=512))
    m.fit(_t(x), _t(var))
    xq = w.xq.copy()
    xq[:700] = np.column_stack([rng.uniform(2.9, 4.3, (700, 2)), rng.uniform(0.0, 0.3, 700)])
    xq[700:720] = xq[0]
    xq[720:740] += 40.0
    xq = xq[rng.permutation(len(xq))]
    xq[5], xq[40] = np.nan, 1e9
    n = np.diff(m.cells()[2])
    assert (n > 256).any() and ((n > 96) & (n <= 256)).any() and (n <= 96).any()
    return m, xq.astype(np.float32), w.sign


@pytest.mark.parametrize("f64", [False, True])
def test_query(model, f64):
    m, xq, sign = model
    mask = ksdf.OUT_ALL | ksdf.OUT_VAR_GRAD
    cast = (lambda a: _t(a.astype(np.float64))) if f64 else _t
    big = m.query(cast(xq), _t(sign), mask, f64=f64)
    for n in SIZES[::3] if f64 else SIZES:
        got = m.query(cast(xq[:n]), _t(sign[:n]), mask, f64=f64)
        for k, v in got.items():
            assert np.array_equal(v.cpu().numpy(), big[k][:n].cpu().numpy(), equal_nan=True), (n, k)
    assert m.fit_status == 0
    assert ksdf.ksdf_sync_status(m.h) == ksdf.KSDF_ERR_NONFINITE  # the two invalid queries


def test_backward(model):
    m, xq, sign = model
    rng = np.random.default_rng(1)
    win = m.query(_t(xq), _t(sign), ksdf.OUT_WINNER)["winner"]
    for n in SIZES:
        ds, dg = np.zeros(len(xq), np.float32), np.zeros((len(xq), 3), np.float32)
        ds[:n], dg[:n] = rng.standard_normal(n), rng.standard_normal((n, 3))
        big_q, _ = m.backward(_t(xq), win, _t(ds), _t(dg), _t(sign))
        got_q, _ = m.backward(_t(xq[:n]), win[:n].contiguous(), _t(ds[:n]), _t(dg[:n]), _t(sign[:n]))
        assert torch.equal(got_q, big_q[:n]), n
    ksdf.ksdf_sync_status(m.h)
