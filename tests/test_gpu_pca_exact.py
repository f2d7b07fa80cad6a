"""The PCA vectors' correction: after the float32 rotations the kept vectors are corrected against the
covariance in float64, so they are eigenvectors of it up to the covariance's own float32 rounding.

Bound: the covariance's entries are float32 sums (chains of at most 200 rows in 304 blocks whose errors
are independent, then rounded), within 2^-24 of sqrt(C_ii C_jj) each, so the matrix is within
2^-24 trace(C) of the float64 one; with a factor of 2 for the features' own centring, the residual
|C v - lambda v| and the eigenvalue are within eps = 2^-23 trace(C), and a vector whose
eigenvalue is `gap` from the others within eps / gap (and the float32 rounding of its entries)."""
import numpy as np
import pytest

import oracle as O

from helpers import make_pair

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("C", [33, 64, 128])
@pytest.mark.parametrize("spectrum", [(9.0, 4.0, 1.0), (9.0, 8.96, 1.0)])
def test_vectors_to_the_covariance_rounding(C, spectrum):
    import torch
    from paper_2309_16818_gb300 import mem as M
    W, k = 258, 3
    r = np.random.default_rng(C)
    obs = r.random(W * W) < 0.9
    n = int(obs.sum())
    z = r.normal(size=(n, k))
    z = np.linalg.qr(z - z.mean(0))[0] * np.sqrt(n) * np.sqrt(spectrum)  # the sample's own spectrum
    A = np.linalg.qr(r.normal(size=(C, k)))[0]
    f = np.zeros((W * W, C), np.float32)
    f[obs] = z @ A.T + 0.05 * r.normal(size=(n, C)) + 0.5 * r.normal(size=C)
    g, _ = make_pair(W, 0.05, [dict(channels=C, rule=O.LATEST)])
    g.set_layer(0, torch.from_numpy(f).cuda())
    g.set_layer(0, torch.from_numpy(obs.astype(np.uint8)).cuda(), part=M.PART_OBSERVED)
    _, vals, vecs, _ = (t.cpu().numpy().astype(np.float64) for t in g.pca(0, k))
    x = f[obs].astype(np.float64)
    x -= x.mean(0)
    cov = x.T @ x / n
    lam, U = np.linalg.eigh(cov)
    lam, U = lam[::-1], U[:, ::-1]
    eps = 2.0 ** -23 * np.trace(cov)
    for i in range(k):
        v = vecs[i]
        assert abs(np.linalg.norm(v) - 1) < 1e-6
        res = np.linalg.norm(cov @ v - vals[i] * v)
        assert res <= eps + 2.0 ** -24 * lam[0], (i, res, eps)
        assert abs(vals[i] - lam[i]) <= eps + 2.0 ** -24 * lam[i], (i, vals[i], lam[i])
        gap = np.abs(np.delete(lam, i) - lam[i]).min()
        d = np.linalg.norm(v - np.sign(v @ U[:, i]) * U[:, i])
        assert d <= eps / gap + 2.0 ** -24, (i, d, eps / gap)
    assert np.abs(vecs @ vecs.T - np.eye(k)).max() < 1e-5
