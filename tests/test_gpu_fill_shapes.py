"""The diffusion fill in shared memory at the shapes where its packed rows, bands and lists can go
wrong: single rows and columns, odd widths, widths around the padding, bands of one row, crops over
one to eight CTAs, sparse and dense holes, holes along every border.

The result is held to the equations themselves, which bound it whatever the holes' shape: when the
largest update d of a sweep is below tol, a cell's mean-minus-value was d when it was updated, its
own step changed it by omega d (omega < 2) and its neighbours' later steps by at most 2 tol, so it
is below 4 tol at the end, plus the rounding of four float32 additions of heights of magnitude h
(4 h 2^-24 each way). A wrong neighbour, weight or band row leaves a mean off by the heights' own
differences.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _crops(r, H, W):
    y, x = np.mgrid[0:H, 0:W].astype(np.float32)
    h = np.stack([0.3 * np.sin(0.17 * x + i) * np.cos(0.11 * y) + 0.01 * r.random((H, W)) for i in range(4)])
    k = np.ones((4, H, W), np.uint8)
    k[0] = r.random((H, W)) < 0.9          # single unknown cells
    k[1] = r.random((H, W)) < 0.15         # mostly unknown
    k[2, :, : max(1, W // 3)] = 0          # a whole side, corners included
    k[2, H // 2:, :] = 0
    k[2, -1, -1] = 1
    k[3, H // 4:H // 4 + max(1, H // 2), W // 4:] = 0
    k[3, 0, 0] = 1
    return h.astype(np.float32), k


@pytest.mark.parametrize("H,W", [(1, 1), (1, 9), (9, 1), (2, 2), (3, 5), (8, 7), (17, 8), (31, 33), (64, 62),
                                 (200, 136), (130, 257), (257, 130), (256, 256), (300, 401), (17, 2000), (560, 560)])
def test_shapes(H, W):
    import torch
    from paper_2309_16818_gb300 import mem as M
    r = np.random.default_rng(H * 1000 + W)
    h, k = _crops(r, H, W)
    hin = np.where(k == 1, h, np.float32(77.0))  # unknown cells carry garbage
    th, tk = torch.from_numpy(hin).cuda(), torch.from_numpy(k).cuda()
    out, its = M.inpaint_diffusion(th, tk, tol=1e-6, max_iters=20000)
    again, its2 = M.inpaint_diffusion(th, tk, tol=1e-6, max_iters=20000)
    assert torch.equal(out, again) and torch.equal(its, its2)  # nothing depends on the order of the groups
    out = out.cpu().numpy()
    for b in range(4):
        assert np.array_equal(out[b][k[b] == 1], hin[b][k[b] == 1])
        if k[b].any() and H * W > 1:
            u = out[b].astype(np.float64)
            n = np.zeros((H, W))
            m = np.zeros((H, W))
            n[1:] += u[:-1]
            n[:-1] += u[1:]
            n[:, 1:] += u[:, :-1]
            n[:, :-1] += u[:, 1:]
            m[1:] += 1
            m[:-1] += 1
            m[:, 1:] += 1
            m[:, :-1] += 1
            left = np.abs(n / m - u)[k[b] == 0]
            assert left.size == 0 or left.max() < 4e-6 + 8 * 2.0 ** -24 * np.abs(u).max(), (H, W, b, int(its[b]))


def test_sweep_limit():
    import torch
    from paper_2309_16818_gb300 import mem as M
    h = torch.rand((3, 40, 52), device="cuda")
    k = (torch.rand((3, 40, 52), device="cuda") < 0.2).to(torch.uint8)
    _, its = M.inpaint_diffusion(h, k, tol=1e-12, max_iters=7)
    assert its.tolist() == [7, 7, 7]
