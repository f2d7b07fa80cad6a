"""A call's launches take three ways: programmatic dependent launches (the default stream), a captured
graph (another stream) and plain launches between events (profiling). The same calls through each
give the same map, bit for bit."""
import numpy as np
import pytest

from paper_2309_16818_gb300 import synth

from helpers import cloud_sources_gpu, cuda_xyz, make_pair, multimodal_layers

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kw", [{}, dict(drift_alpha=1.0, drift_min_points=100, ray_cleanup=True, ray_margin=0.1,
                                         time_var=1e-6)])
def test_launch_paths_give_the_same_map(kw):
    import torch
    from paper_2309_16818_gb300 import mem as M
    c = synth.config2(n_poses=4, scale=0.25)
    calls = [(c["poses"][k][:2], cuda_xyz(s), s.T, cloud_sources_gpu(s)) for k, s in enumerate(c["scans"])]
    torch.cuda.synchronize()
    states = {}
    for path in ("default stream", "graph", "profiled"):
        g, _ = make_pair(c["W"], c["res"], multimodal_layers(), **kw)
        torch.cuda.synchronize()
        g.set_profiling(path == "profiled")
        st = torch.cuda.Stream() if path == "graph" else torch.cuda.default_stream()
        with torch.cuda.stream(st):
            for _ in range(2):
                for xy, xyz, T, src in calls:
                    g.move(xy)
                    g.fuse_pointcloud(xyz, T, src)
            g.check()
            out = [g.get_layer(l) for l in (M.LAYER_HEIGHT, M.LAYER_VARIANCE, M.LAYER_VALID, M.LAYER_NACC, M.LAYER_NREJ)]
            out += [g.get_layer(l) for l in range(4)]
        torch.cuda.synchronize()
        if path == "profiled":
            assert g.get_profile()["fuse_tiles"][1] == 8
        states[path] = [o.cpu().numpy() for o in out]
    for path in ("graph", "profiled"):
        for a, b in zip(states["default stream"], states[path]):
            assert np.array_equal(a, b), path
