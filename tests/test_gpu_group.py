"""Grouping of a batch by bin and winner: the outputs of large batches (hash table, warp-aggregated ranks) are those of the
same queries in small batches (one CTA's sort), to the bit: queries in order, shuffled, all in one bin, each in a bin of its
own, invalid ones among them, batch sizes that leave a warp or block partly filled; both precisions."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2603_29227_gb300 import ksdf, scenes  # noqa: E402

DEV = torch.device("cuda:0")
MASK = ksdf.OUT_SDF | ksdf.OUT_GRAD | ksdf.OUT_WINNER | ksdf.OUT_FLAGS


@pytest.fixture(scope="module")
def model():
    import __graft_entry__

    __graft_entry__.build()
    w = scenes.workload("room3d", n_samples=30_000, n_queries=64)
    m = ksdf.KernelSDF(w.params)
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(DEV)  # noqa: E731
    m.fit(t(w.x), t(w.var), t(w.normals))
    return w, m


@pytest.mark.parametrize("f64", [False, True])
@pytest.mark.parametrize("kind,n", [("volume", 2049), ("volume", 4127), ("shuffled", 70_001), ("one bin", 3_333),
                                    ("own bins", 5_000), ("invalid", 2_600)])
def test_large_as_small(model, kind, n, f64):
    w, m = model
    rng = np.random.default_rng(n)
    lo, hi = w.x.min(0), w.x.max(0)
    xq = lo + rng.random((n, 3)) * (hi - lo)
    if kind == "volume":
        xq = xq[np.lexsort(np.floor(xq / 0.5).T)]
    elif kind == "one bin":
        xq = np.floor(w.x[0] / 0.5) * 0.5 + rng.random((n, 3)) * 0.5
    elif kind == "own bins":
        g = np.stack(np.meshgrid(np.arange(20), np.arange(25), np.arange(10), indexing="ij"), -1).reshape(-1, 3)
        xq = 0.5 * (g - 3) + 0.25
    xq = torch.from_numpy(xq).to(DEV, torch.float64 if f64 else torch.float32)
    if kind == "invalid":
        xq[::7, 1] = float("nan")
        xq[5::64] = float("inf")
        xq[3::100, 0] = 1e30
    big = m.query(xq, mask=MASK, f64=f64)
    parts = [m.query(xq[a:a + 1500].contiguous(), mask=MASK, f64=f64) for a in range(0, n, 1500)]
    torch.cuda.synchronize()
    if kind == "invalid":
        with pytest.raises(Exception):
            m.sync_status()
    else:
        m.sync_status()
    for k in ("sdf", "grad", "winner", "flags"):
        a, b = big[k].cpu().numpy(), torch.cat([o[k] for o in parts]).cpu().numpy()
        assert a.tobytes() == b.tobytes(), (k, int((a != b).sum()))
