"""The front-end's update and prediction over the reaches of a hinge: the candidate tables of 0 to 2 cells' reach (one to
seven rounds of 32 offsets an octant), block sides that are no powers of two, without the bias, one to four EM rounds.
Blocks, samples and kept features exactly, weights, log-odds and gradient within the bound that test_gpu_bhm.py derives."""
import numpy as np
import pytest

from test_gpu_bhm import C_REL, _compare_maps, _frame, _mags, _oracle, _params, dev  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("phi_min,block_hinges,em_iters,bias", [
    (0.5, 4, 1, 1),    # reach 0
    (0.1, 5, 3, 0),    # reach 1
    (1e-3, 16, 2, 1),  # reach 2, three rounds
    (2e-5, 5, 4, 1),   # reach 2, more than three rounds
])
def test_reach(dev, phi_min, block_hinges, em_iters, bias):  # noqa: F811
    import torch
    from paper_2603_29227_gb300 import bhm

    P = _params(phi_min=phi_min, block_hinges=block_hinges, em_iters=em_iters, bias_feature=bias, march_sub=1)
    o = _oracle(P)
    m = bhm.BHMap(P, max_blocks=20000)
    for f in (0, 1):
        p, hits = _frame(150, f=f, radius=6.0)
        o.update(p, hits)
        m.update(p, torch.from_numpy(hits).to(dev))
        m.sync_status()
        nb, ns, nf = m.size(features=True)
        assert ns == o.last_samples and nf == o.last_features
    _compare_maps(o, m)
    rng = np.random.default_rng(5)
    xq = (hits + rng.normal(0, 0.2, hits.shape)).astype(np.float32)
    out = {k: v.cpu().numpy() for k, v in m.query(torch.from_numpy(xq).to(dev)).items()}
    L, S, G, Pr = o.query(xq.astype(np.float64))
    for k in range(len(xq)):
        sl, sg = _mags(o, xq[k].astype(np.float64))
        assert abs(out["logodds"][k] - L[k]) <= C_REL * sl + 1e-6, k
        assert np.max(np.abs(out["grad"][k] - G[k])) <= C_REL * sg + 1e-5, k
