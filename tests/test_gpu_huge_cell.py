"""Cells so large that squared distances leave FP32's range: no sample is nearest then, and the mixed query still reads
only the cell's samples (the first stands in) and returns.  Sizes of the CUDA-core kernel for more than 256 samples, with
and without a part of the samples that is empty."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2603_29227_gb300 import ksdf  # noqa: E402

DEV = torch.device("cuda:0")


@pytest.mark.parametrize("n", [257, 301, 511])
def test_no_finite_distance(n):
    h = 1e22
    rng = np.random.default_rng(n)
    x = h * rng.uniform(0.1, 0.9, (n, 3))
    xq = (1e17 * rng.uniform(0.0, 1.0, (65, 3))).astype(np.float32)  # (phase A's filler for a step of 8 samples is in reach)
    m = ksdf.KernelSDF(dict(dim=3, origin=(0.0, 0.0, 0.0), cell=h, margin=0.0, n_max=512, k_cand=1, sign_mode=1,
                            **{"lambda": 1e-30}))
    nrm = np.tile(np.array([[0.0, 0.0, 1.0]], dtype=np.float32), (n, 1))
    m.fit(torch.from_numpy(x).to(DEV), torch.full((n,), 1e-4, device=DEV), torch.from_numpy(nrm).to(DEV))
    assert m.fit_status == 0 and len(m.cells()[1]) == 1
    out = m.query(torch.from_numpy(xq).to(DEV))
    m.sync_status()
    assert np.all(out["winner"].cpu().numpy() == 0)
