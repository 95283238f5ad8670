"""Training sets of cells of very different sizes against the oracle, exactly: collection boxes of one to several thousand
members (ranked by counting, sorted, taken by the second launch, and capped), boxes that reach one to three cells far (one to
eleven groups of 32 neighbours), 2D and 3D."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import oracle  # noqa: E402
from paper_2603_29227_gb300 import ksdf  # noqa: E402

DEV = torch.device("cuda:0")


@pytest.fixture(scope="module", autouse=True)
def _build():
    import __graft_entry__

    __graft_entry__.build()


@pytest.mark.parametrize("dim,margin,n_max", [(3, 0.1, 64), (3, 0.5, 64), (3, 1.2, 16), (2, 0.1, 64), (2, 0.7, 33)])
def test_training_sets(dim, margin, n_max):
    rng = np.random.default_rng(17 + dim)
    clusters = [1, 2, 3, 4, 5, 31, 33, 127, 128, 129, 255, 256, 257, 1023, 1024, 1025, 3000]
    x = []
    for k, n in enumerate(clusters):  # one cluster inside a cell (its box holds it alone, or with its neighbours)
        base = np.array([k % 5, k // 5, (7 * k) % 3][:dim]) * (1.0 if margin > 0.3 else 1.5)
        x.append(base + 0.12 + 0.26 * rng.random((n, dim)))
    x = np.concatenate(x)
    x = x[rng.permutation(len(x))]
    var = np.full(len(x), 1e-2, np.float32)
    p = dict(dim=dim, origin=(0.0, 0.0, 0.0), cell=0.5, margin=margin, n_max=n_max, k_cand=4, softmin_alpha=300.0,
             sign_mode=0, **{"lambda": 300.0})
    ref = oracle.Model(p, x, var.astype(np.float64))
    m = ksdf.KernelSDF(p)
    m.fit(torch.from_numpy(x).to(DEV), torch.from_numpy(var).to(DEV))
    torch.cuda.synchronize()
    for a, b in zip(ref.cells(), m.cells()):
        assert np.array_equal(a, b)
