"""Host-buffer calls issued back to back: each call's job block (pose, pointers, counts) and inputs
must stay its own while the next call's uploads run beside its kernels."""
import numpy as np
import pytest

from paper_2309_16818_gb300 import mem as M
from paper_2309_16818_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("own_stream", [False, True])
@pytest.mark.parametrize("n", [300, 20_000])
def test_back_to_back_calls_equal_device_calls(own_stream, n):
    """Clouds of different poses and sizes, many calls in flight, against the same calls on device
    buffers one at a time: the same bits."""
    import torch
    W, calls = 120, 24
    layers = [M.Layer(3, M.LATEST), M.Layer(4, M.EXPAVG, w=0.3)]
    ter = synth.Terrain.from_seed(n)
    r = np.random.default_rng(n)
    clouds = []
    for k in range(calls):
        m = n if k % 3 else n // 2 + 1
        xy = tuple(r.uniform(-2.0, 2.0, 2))
        cl = synth.uniform_ground_cloud(k, m, 8.0, ter, sensor_xy=xy)
        clouds.append((torch.from_numpy(cl.xyz).pin_memory(), cl.T, torch.from_numpy(cl.rgb).pin_memory(),
                       torch.rand(m, 4).pin_memory()))
    ref = M.Map(W, 0.05, layers)
    for xyz, T, rgb, f in clouds:
        ref.fuse_pointcloud(xyz.cuda(), T, [(rgb.cuda(), [0]), (f.cuda(), [1])])
        torch.cuda.synchronize()
    for rep in range(4):
        g = M.Map(W, 0.05, layers)
        st = torch.cuda.Stream() if own_stream else torch.cuda.current_stream()
        with torch.cuda.stream(st):
            for xyz, T, rgb, f in clouds:
                g.fuse_pointcloud_host(xyz, T, [(rgb, [0]), (f, [1])])
            g.check()
            for layer in (M.LAYER_HEIGHT, M.LAYER_VARIANCE, M.LAYER_NACC, M.LAYER_NREJ, 0, 1):
                assert torch.equal(g.get_layer(layer), ref.get_layer(layer)), (rep, layer)
