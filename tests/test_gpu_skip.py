"""Queries without the flags leave out candidates that cannot win (u_floor); with the flags every candidate is evaluated.
The other outputs have to be the same to the bit: near and far queries, on the samples themselves, bins of one to several
hundred queries, candidate lists that take more than one round, both kernels, 2D and 3D."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2603_29227_gb300 import ksdf, scenes  # noqa: E402

DEV = torch.device("cuda:0")
KEYS = ("sdf", "grad", "var_sdf", "var_f", "winner")


@pytest.fixture(scope="module", autouse=True)
def _build():
    import __graft_entry__

    __graft_entry__.build()


def _t(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to(DEV)


@pytest.mark.parametrize("name,over", [
    ("room3d", dict()),
    ("room3d", dict(k_cand=32, n_max=512)),
    ("room3d", dict(k_cand=1)),
    ("room3d", {"kernel": "matern32", "lambda": 100.0, "softmin_alpha": 100.0}),
    ("room3d", {"lambda": 20.0}),
    ("plane2d", dict()),
])
def test_same_without_flags(name, over):
    w = scenes.workload(name, **(dict(n_samples=1500, grid=8) if name == "plane2d" else
                                 dict(n_samples=60_000, n_queries=64)))
    params = dict(w.params, **over)
    d = int(params["dim"])
    rng = np.random.default_rng(11)
    lo, hi = w.x.min(0), w.x.max(0)
    h = params["cell"]
    near = w.x[rng.choice(len(w.x), 6000)] + rng.normal(0, 0.03, (6000, d))
    vol = lo + rng.random((8000, d)) * (hi - lo)
    far = lo + (rng.random((500, d)) - 0.5) * 40 * (hi - lo)
    on = w.x[:700]
    bins = [np.floor(w.x[rng.integers(len(w.x))] / h) * h + rng.random((n, d)) * h for n in (15, 16, 17, 33, 128, 129, 600)]
    xq = np.concatenate([near, vol, far, on] + bins).astype(np.float32)
    sg = np.where(rng.random(len(xq)) < 0.5, -1, 1).astype(np.int8)
    gm = ksdf.KernelSDF(params)
    gm.fit(_t(w.x), _t(w.var), _t(w.normals))
    mask = ksdf.OUT_SDF | ksdf.OUT_GRAD | ksdf.OUT_VAR_SDF | ksdf.OUT_VAR_F | ksdf.OUT_WINNER
    for n in (len(xq), 2000):  # both groupings
        pick = slice(0, n) if n == len(xq) else rng.permutation(len(xq))[:n]
        full = gm.query(_t(xq[pick]), _t(sg[pick]), mask=mask | ksdf.OUT_FLAGS)
        less = gm.query(_t(xq[pick]), _t(sg[pick]), mask=mask)
        torch.cuda.synchronize()
        gm.sync_status()
        for k in KEYS:
            a, b = full[k].cpu().numpy(), less[k].cpu().numpy()
            assert np.array_equal(a.view(np.int32), b.view(np.int32)), (k, int((a != b).sum()))
