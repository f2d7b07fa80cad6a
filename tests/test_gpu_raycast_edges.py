"""Ray-cast clean-up with several lanes per line, at its edges: the smallest maps, cell counts below
and past a block's, wrapped ring buffers, and sensors in the map, in its corner and outside it."""
import numpy as np
import pytest

import oracle as O
from paper_2309_16818_gb300 import synth

from helpers import compare_states, cuda_xyz, gpu_state, make_pair, upload_state

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("W", [2, 6, 18, 258])
@pytest.mark.parametrize("where", [(0.0, 0.0), (-0.49, 0.49), (0.3, -0.8)])
def test_lines_from_every_sensor_cell(W, where):
    res = 0.1
    g, o = make_pair(W, res, [], ray_cleanup=True, ray_margin=0.05, range_max=100.0)
    r = np.random.default_rng(W)
    ter = synth.Terrain.from_seed(W)
    sensor = tuple(v * W * res for v in where)
    cleared = 0
    for k in range(2):
        xy = (res * (3 * k + 1), -res * (W // 2 + k))
        o.move(xy)
        g.move(xy)
        cl = synth.uniform_ground_cloud(W + k, 3 * W * W, 1.5 * W * res, ter,
                                        sensor_xy=(xy[0] + sensor[0], xy[1] + sensor[1]), height=2.0)
        idx = np.nonzero(o.valid)[0]
        o.h[idx] += np.where(r.random(idx.size) < 0.2, 1.5, 0.0)  # stale obstacles
        upload_state(g, o)
        sub = cl.xyz[r.random(cl.xyz.shape[0]) < 0.1].copy()  # most cells get no point
        ro = o.fuse_points(sub, cl.T)
        import torch
        g.fuse_pointcloud(torch.from_numpy(sub).cuda(), cl.T)
        g.check()
        assert g.get_drift()["cleared"] == ro["cleared"]
        compare_states(gpu_state(g), o, what=f"W {W} {where} {k}")
        cleared += ro["cleared"]
    assert cleared > 0 or W < 258
