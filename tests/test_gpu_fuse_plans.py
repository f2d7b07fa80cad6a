"""The warp fuse kernel at the shapes where its plan can go wrong: column counts at, below and past
a round of 32, arg-max pairs that just fit or just do not, sources split over several rounds at odd
and aligned channels, many layers, rows of every type, calls past the plan's tables (the tile
kernel), and runs that cross warps and tiles. Against the oracle, from the same state."""
import numpy as np
import pytest

import oracle as O
from paper_2309_16818_gb300 import synth

from helpers import compare_states, gpu_state, make_pair, upload_state

pytestmark = pytest.mark.gpu

G, D, X, E, L = O.GAUSS, O.DIRICHLET, O.CLASSMAX, O.EXPAVG, O.LATEST
# per source: (type, channels, rules of its layers, storage of the layers that may have 16 bits)
CASES = {
    "none": [],
    "28": [("f32", 28, [E], O.F32)],
    "29": [("f32", 29, [E], O.F32)],
    "26 pair": [("f32", 26, [D, X], O.F32)],
    "27 pair": [("f32", 27, [D, X], O.F32)],
    "28 pair": [("f32", 28, [X, D], O.F32)],
    "3+20 pair": [("u8", 3, [L], O.F32), ("f32", 20, [D, X, E], O.F32)],
    "64 bf16": [("bf16", 64, [G, E], O.BF16)],
    "61 f16": [("f16", 61, [E, G], O.F16)],
    "3+64+20": [("u8", 3, [L], O.F32), ("bf16", 64, [G, E], O.F16), ("f32", 20, [D, X], O.F32)],
    "70 pair": [("f32", 70, [X, D], O.F32), ("u8", 5, [G], O.BF16)],
    "8 layers": [("f32", 12, [G, E, D, L, X, G, E, D], O.F32)],
    "8 sources": [("u8", 1, [L], O.F32), ("f32", 2, [X], O.F32), ("bf16", 3, [G], O.F32), ("f16", 4, [E], O.F16),
                  ("f32", 5, [D, X], O.F32), ("u8", 6, [E], O.BF16), ("f32", 7, [G, X], O.F32), ("bf16", 8, [L], O.BF16)],
    "300": [("f32", 300, [E, X], O.F32), ("u8", 3, [L], O.F32)],
}


def _rows(r, dt, n, C):
    a = r.random((n, C)).astype(np.float32)
    if dt == "u8":
        a = (a * 255).astype(np.uint8)
    return a


@pytest.mark.parametrize("case", list(CASES))
@pytest.mark.parametrize("W,n", [(8, 3000), (40, 6000), (200, 9001)])
def test_against_the_oracle(case, W, n):
    import torch
    spec = CASES[case]
    layers, src_layers = [], []
    for dt, C, rules, store in spec:
        src_layers.append(list(range(len(layers), len(layers) + len(rules))))
        layers += [dict(channels=C, rule=q, w=0.3, var_meas=0.7, alpha0=0.5,
                        dtype=O.F32 if q in (D, X) else store) for q in rules]
    g, o = make_pair(W, 0.05, layers, outlier_var=1e-4)
    r = np.random.default_rng(len(case) * 1000 + W)
    ter = synth.Terrain.from_seed(W)
    for k in range(2):
        cl = synth.uniform_ground_cloud(50 + k, n, 1.1 * W * 0.05, ter)
        gs, os_ = [], []
        for (dt, C, _, _), l in zip(spec, src_layers):
            a = _rows(r, dt, n, C)
            t = torch.from_numpy(a).cuda()
            if dt in ("bf16", "f16"):
                t = t.to(torch.bfloat16 if dt == "bf16" else torch.float16)
                a = t.float().cpu().numpy()
            gs.append((t, l))
            os_.append((a, l))
        if k:
            upload_state(g, o)
        o.fuse_points(cl.xyz, cl.T, os_)
        g.fuse_pointcloud(torch.from_numpy(cl.xyz).cuda(), cl.T, gs)
        g.check()
        compare_states(gpu_state(g), o, what=f"{case} W {W} call {k}")
    assert o.n_rej.sum() > 0


@pytest.mark.parametrize("K,topk", [(20, 3), (23, 1), (40, 5), (130, 16)])
def test_topk_over_rounds(K, topk):
    import torch
    from paper_2309_16818_gb300 import mem as M
    W, n = 60, 7000
    layers = [dict(channels=K, rule=q, w=0.3) for q in (D, X, E)] + [dict(channels=3, rule=L)]
    g, o = make_pair(W, 0.05, layers)
    r = np.random.default_rng(K)
    ter = synth.Terrain.from_seed(K)
    for k in range(2):
        cl = synth.uniform_ground_cloud(70 + k, n, 1.1 * W * 0.05, ter)
        p = np.empty((n, 2 * topk), np.float32)
        p[:, 0::2] = r.integers(-1, K + 1, (n, topk))  # some ids out of range, some repeated
        p[:, 1::2] = r.random((n, topk)) - 0.2
        rgb = _rows(r, "u8", n, 3)
        if k:
            upload_state(g, o)
        o.fuse_points(cl.xyz, cl.T, [(O.TopK(p, K), [0, 1, 2]), (rgb, [3])])
        g.fuse_pointcloud(torch.from_numpy(cl.xyz).cuda(), cl.T,
                          [(M.TopK(torch.from_numpy(p).cuda(), K), [0, 1, 2]), (torch.from_numpy(rgb).cuda(), [3])])
        g.check()
        compare_states(gpu_state(g), o, what=f"top-{topk} of {K} call {k}")
