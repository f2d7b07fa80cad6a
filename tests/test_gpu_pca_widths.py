"""PCA at the channel counts where its tiles can go wrong: one channel, odd counts, below, at and
past an 8-channel tile and a 32-lane row, the largest, and maps with few, one or no observed cells.

Tolerances: the eigenvalues, vectors and projections of the wider test of this plugin (1e-4
relative; 1e-3; 1e-2 of the component's scale), whose features have the same variances 9, 4, 1."""
import numpy as np
import pytest

import oracle as O
from oracle import plugins as PL

from helpers import make_pair, torch_dt

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("C", [1, 2, 7, 8, 9, 31, 33, 65, 127, 128])
@pytest.mark.parametrize("W,share", [(66, 0.6), (258, 0.9)])
@pytest.mark.parametrize("dtype", [O.F32, O.F16])
def test_channel_counts(C, W, share, dtype):
    import torch
    from paper_2309_16818_gb300 import mem as M
    r = np.random.default_rng(C * 1000 + W)
    k = min(3, C)
    A = np.linalg.qr(r.normal(size=(C, k)))[0]
    f = r.normal(size=C) + (r.normal(size=(W * W, k)) * np.sqrt([9.0, 4.0, 1.0][:k])) @ A.T
    f = f + 0.05 * r.normal(size=f.shape)
    obs = r.random(W * W) < share
    g, _ = make_pair(W, 0.05, [dict(channels=C, rule=O.LATEST, dtype=dtype)])
    g.move((0.21, -1.3))
    fv = torch.from_numpy(f).to(torch_dt(dtype)).cuda().contiguous()
    g.set_layer(0, fv)
    g.set_layer(0, torch.from_numpy(obs.astype(np.uint8)).cuda(), part=M.PART_OBSERVED)
    proj, vals, vecs, mean = (t.cpu().numpy().astype(np.float64) for t in g.pca(0, k))
    op, ow, oV, om = PL.pca_of_features(fv.float().cpu().numpy(), obs, k)
    assert np.allclose(vals, ow, rtol=1e-4) and np.allclose(mean, om, atol=1e-5 * (1 + np.abs(om).max()))
    for i in range(k):
        s = np.sign(vecs[i] @ oV[i])  # two components of nearly the largest size may swap the sign
        assert np.allclose(s * vecs[i], oV[i], atol=1e-3)
        assert np.abs(s * proj[:, i] - op[:, i]).max() <= 1e-2 * np.sqrt(ow[i])
        assert vecs[i][np.argmax(np.abs(vecs[i]))] > 0
    assert np.all(proj[~obs] == 0)


@pytest.mark.parametrize("cells", [0, 1, 2])
def test_few_observed_cells(cells):
    import torch
    from paper_2309_16818_gb300 import mem as M
    W, C = 34, 12
    g, _ = make_pair(W, 0.05, [dict(channels=C, rule=O.LATEST)])
    f = torch.randn(W * W, C, generator=torch.Generator().manual_seed(1)).cuda()
    obs = torch.zeros(W * W, dtype=torch.uint8, device="cuda")
    obs[5:5 + cells] = 1
    g.set_layer(0, f)
    g.set_layer(0, obs, part=M.PART_OBSERVED)
    proj, vals, vecs, mean = (t.cpu().numpy().astype(np.float64) for t in g.pca(0, 2))
    op, ow, _, om = PL.pca_of_features(f.cpu().numpy(), obs.cpu().numpy().astype(bool), 2)
    assert np.all(np.isfinite(proj)) and np.all(np.isfinite(vecs))
    assert np.allclose(vals, ow, rtol=1e-4, atol=1e-6) and np.allclose(mean, om, atol=1e-5)
    assert np.allclose(np.abs(proj[:, 0]), np.abs(op[:, 0]), atol=1e-3)
