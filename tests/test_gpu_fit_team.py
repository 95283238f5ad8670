"""The factor of a cell does not depend on how many warps form it.  Row i of a Cholesky factor only depends on the first
i + 1 samples, so the factor of the first n samples of a cell is the leading part of the factor of all of them, bit for
bit, when every team adds up the same exact sums; sizes on both sides of the class boundaries (one warp up to 95, four up to
127, five up to 159, eight up to 256, sixteen above, which share columns) are compared along that chain.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2603_29227_gb300 import ksdf  # noqa: E402

DEV = torch.device("cuda:0")
SIZES = [63, 95, 127, 144, 159, 160, 183, 184, 200, 215, 216, 256, 257, 300, 400, 512]


def _points(n, kernel):
    rng = np.random.default_rng(7 + kernel)
    x = rng.uniform(0.05, 0.95, (n, 3))
    x[:, 2] = 0.5 + 0.02 * rng.standard_normal(n)  # near a plane, like surface samples
    return x, ((0.01 * rng.uniform(0.5, 2.0, n)) ** 2).astype(np.float32)


def _fit(x, var, lam, kernel, table=None):
    m = ksdf.KernelSDF(dict(dim=3, origin=(0.0, 0.0, 0.0), cell=1.0, margin=0.0, n_max=512, k_cand=1, kernel=kernel,
                            **{"lambda": lam}))
    if table is not None:
        assert ksdf.load().ksdf_test_fit_table(m.h, table) == 0
    m.fit(torch.from_numpy(x).to(DEV), torch.from_numpy(var).to(DEV))
    assert m.fit_status == 0 and len(m.cells()[1]) == 1
    return m.fit_arrays()


@pytest.mark.parametrize("kernel,lam", [(0, 300.0), (1, 100.0)])
def test_leading_rows(kernel, lam):
    x, var = _points(512, kernel)
    big = None
    for n in reversed(SIZES):
        chol = _fit(x[:n], var[:n], lam, kernel)[1]
        if big is not None:
            assert np.array_equal(chol, big[:len(chol)]), (n, int((chol != big[:len(chol)]).sum()))
        big = chol


@pytest.mark.parametrize("n", [47, 72, 88, 96, 120, 128, 144, 159, 160, 183, 184, 200, 215, 216, 256, 300, 512])
def test_every_table(n):
    """Every size-class table gives the same factor, alpha and L^-1."""
    x, var = _points(n, 0)
    for fixed in (True, False):  # and on the binary64 path: a variance outside the fixed-point range
        if not fixed:
            var = var.copy()
            var[n // 2] = 0.26
        ref = _fit(x, var, 300.0, 0, 0)
        for t in range(1, ksdf.load().ksdf_autotune_tables()):
            for a, b in zip(ref, _fit(x, var, 300.0, 0, t)):
                assert np.array_equal(a, b), (n, t, fixed, int((a != b).sum()))


def test_table_is_checked():
    m = ksdf.KernelSDF(dict(dim=3, origin=(0.0, 0.0, 0.0), cell=1.0, margin=0.0, n_max=8, k_cand=1, **{"lambda": 300.0}))
    lib = ksdf.load()
    for t in (-1, lib.ksdf_autotune_tables()):
        assert lib.ksdf_test_fit_table(m.h, t) == ksdf.KSDF_ERR_ARG
    assert lib.ksdf_test_fit_table(None, 0) == ksdf.KSDF_ERR_ARG
