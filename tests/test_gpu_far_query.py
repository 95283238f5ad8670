"""Mixed queries 1e7 m and farther from the cell (inside the grid of 2^20 cells of 64 m): a stand-in for a missing sample
(an odd pair's second, a step of 8's last) must not be nearer than the samples.  Sizes of every phase B kernel below 257
samples, odd and even and on both sides of a step of 8, with V[f] (tensor cores) and without.  Reference: the plain FP64
query.  Bars: coordinates round to 2 m there, which is 1e-7 of the distance, so the SDF agrees to 1e-5 relative (no query
lies between the samples along the normals' axis, where the sign would hang on which of them is the nearest) and the
gradient to 1e-4; the softmin temperature times 4 m is 4e-5, V[u] to 1e-3; V[f] is 1 to 1e-3.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2603_29227_gb300 import ksdf  # noqa: E402

DEV = torch.device("cuda:0")
REAL = ksdf.OUT_SDF | ksdf.OUT_GRAD | ksdf.OUT_VAR_SDF


@pytest.mark.parametrize("n", [1, 2, 5, 8, 9, 16, 89, 96, 97, 130, 255, 256])
@pytest.mark.parametrize("kernel,lam", [(0, 1e-9), (1, 1e-5)])
def test_far_from_the_cell(n, kernel, lam):
    p = dict(dim=3, origin=(0.0, 0.0, 0.0), cell=64.0, margin=0.0, n_max=256, k_cand=1, softmin_alpha=1e-5, sign_mode=1,
             kernel=kernel, **{"lambda": lam})
    rng = np.random.default_rng(n)
    x = rng.uniform(1.0, 63.0, (n, 3))
    nrm = np.tile(np.array([[1.0, 0.0, 0.0]], dtype=np.float32), (n, 1))
    m = ksdf.KernelSDF(p)
    m.fit(torch.from_numpy(x).to(DEV), torch.full((n,), 1e-4, device=DEV), torch.from_numpy(nrm).to(DEV))
    assert len(m.cells()[1]) == 1
    xq = np.array([[3e7, 3e7, 3e7], [5e7, 1e7, 2e7], [-4e7, -4e7, 1e7], [2e7, 2e7, 6e7], [1e7, 1e7, 1e7],
                   [-1e7, 1e7, 1e7], [100.0, 50.0, 6e7]], dtype=np.float32)
    b = m.query(torch.from_numpy(xq.astype(np.float64)).to(DEV), mask=REAL | ksdf.OUT_VAR_F, f64=True)
    b = {k: v.cpu().numpy() for k, v in b.items() if v is not None}
    for mask in (REAL, REAL | ksdf.OUT_VAR_F, ksdf.OUT_SDF | ksdf.OUT_GRAD):
        a = m.query(torch.from_numpy(xq).to(DEV), mask=mask)
        m.sync_status()
        a = {k: v.cpu().numpy().astype(np.float64) for k, v in a.items() if v is not None}
        assert np.all(np.abs(a["sdf"] - b["sdf"]) <= 1e-5 * np.abs(b["sdf"])), mask
        assert np.all(np.abs(a["grad"] - b["grad"]) <= 1e-4), mask
        if "var_sdf" in a:
            assert np.all(np.abs(a["var_sdf"] - b["var_sdf"]) <= 1e-3 * b["var_sdf"]), mask
        if "var_f" in a:
            assert np.all(np.abs(a["var_f"] - b["var_f"]) <= 1e-3), mask


@pytest.mark.parametrize("n", [5, 8, 9])
@pytest.mark.parametrize("kernel,lam", [(0, 1e-20), (1, 1e-10)])
def test_far_from_a_wide_cell(n, kernel, lam):
    """Cells of 2^32 m: the SDF of queries 1e15 m away (phase A's steps of 8 samples), 1e-5 relative as above."""
    h = 2.0 ** 32
    m = ksdf.KernelSDF(dict(dim=3, origin=(0.0, 0.0, 0.0), cell=h, margin=0.0, n_max=256, k_cand=1, kernel=kernel,
                            **{"lambda": lam}))
    x = h * np.random.default_rng(n).uniform(0.1, 0.9, (n, 3))
    m.fit(torch.from_numpy(x).to(DEV), torch.full((n,), 1e-4, device=DEV))
    xq = np.array([[3e15, 3e15, 3e15], [1e15, 1e15, 1e15], [-2e15, 3e15, 1e15], [4e15, 1e9, 1e9]], dtype=np.float32)
    b = m.query(torch.from_numpy(xq.astype(np.float64)).to(DEV), mask=ksdf.OUT_SDF, f64=True)["sdf"].cpu().numpy()
    for mask in (ksdf.OUT_SDF, ksdf.OUT_SDF | ksdf.OUT_FLAGS):
        a = m.query(torch.from_numpy(xq).to(DEV), mask=mask)["sdf"].cpu().numpy().astype(np.float64)
        m.sync_status()
        assert np.all(np.abs(a - b) <= 1e-5 * np.abs(b)), (a, b)
