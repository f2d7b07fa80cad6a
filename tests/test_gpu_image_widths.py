"""Image fusion with one warp per cell at the widths where its lanes can go wrong: channels below,
at and past 32 and 64, more layers of a source than are loaded together, two sources feeding one
layer in order, and lines of every octant up to the map's far corners."""
import numpy as np
import pytest

import oracle as O
from paper_2309_16818_gb300 import synth

from helpers import compare_states, gpu_state, make_pair, upload_state

pytestmark = pytest.mark.gpu


def _filled(o, W, res, seed):
    """Two scans over the whole map from its centre."""
    ter = synth.Terrain.from_seed(seed)
    for k in range(2):
        cl = synth.uniform_ground_cloud(seed + k, 4 * W * W, 1.2 * W * res, ter)
        o.fuse_points(cl.xyz, cl.T)


@pytest.mark.parametrize("W", [2, 34, 150])
@pytest.mark.parametrize("C", [1, 31, 33, 64, 65, 130])
def test_channel_widths_and_many_layers(W, C):
    import torch
    r = np.random.default_rng(W * 1000 + C)
    layers = [dict(channels=C, rule=O.GAUSS, var_meas=0.5), dict(channels=C, rule=O.DIRICHLET),
              dict(channels=C, rule=O.CLASSMAX), dict(channels=C, rule=O.EXPAVG, w=0.3, dtype=O.F16),
              dict(channels=C, rule=O.LATEST), dict(channels=C, rule=O.GAUSS, var_meas=2.0, dtype=O.BF16)]
    g, o = make_pair(W, 0.05, layers)
    _filled(o, W, 0.05, C)
    ter = synth.Terrain.from_seed(C)
    cams = synth.cameras_around(5, (0.0, 0.0, 0.3), ter, n_cams=2, H=60, Wi=106, images=False)
    seen = 0
    for cam in cams:
        upload_state(g, o)
        a = r.random((60 * 106, C)).astype(np.float32)
        b = r.random((60 * 106, C)).astype(np.float32)
        src = [(a, [0, 1, 2, 3, 4, 5]), (b, [1, 5])]  # the second source feeds layers of the first again
        ro = o.fuse_image(60, 106, src, cam.K, cam.T)
        vis = torch.empty(W * W, dtype=torch.uint8, device="cuda")
        pix = torch.empty(W * W, dtype=torch.int32, device="cuda")
        g.fuse_image(60, 106, cam.K, cam.T, [(torch.from_numpy(x).cuda().view(60, 106, C), l) for x, l in src],
                     vis=vis, pix=pix)
        assert np.array_equal(vis.cpu().numpy(), ro["vis"]) and np.array_equal(pix.cpu().numpy(), ro["pix"])
        compare_states(gpu_state(g), o, what=f"W {W} C {C}")
        seen += ro["n_visible"]
    assert seen > 0 or W < 34


@pytest.mark.parametrize("W", [64, 302])
def test_lines_of_every_octant(W):
    """A camera near a corner, then one near the middle, looking straight down from high above a
    field of spikes: lines towards every direction, most of them occluded somewhere."""
    import torch
    g, o = make_pair(W, 0.1, [dict(channels=3, rule=O.LATEST)])
    r = np.random.default_rng(W)
    _filled(o, W, 0.1, W)
    o.h[:] = (r.random(W * W) ** 6 * 3.0).astype(np.float32)
    for x, y in ((-0.45, -0.45), (0.1, -0.2)):
        upload_state(g, o)
        T = synth.pose(np.diag([1.0, -1.0, -1.0]), [x * W * 0.1, y * W * 0.1, 4.0])  # optical axis = world -z
        H = Wi = 200
        K = (2.0, 2.0, 100.0, 100.0)
        img = r.random((H * Wi, 3)).astype(np.float32)
        ro = o.fuse_image(H, Wi, [(img, [0])], K, T)
        vis = torch.empty(W * W, dtype=torch.uint8, device="cuda")
        g.fuse_image(H, Wi, K, T, [(torch.from_numpy(img).cuda().view(H, Wi, 3), [0])], vis=vis)
        assert 0 < ro["n_visible"] < W * W
        assert np.array_equal(vis.cpu().numpy(), ro["vis"])
        compare_states(gpu_state(g), o, what=f"octants {W} {x}")
