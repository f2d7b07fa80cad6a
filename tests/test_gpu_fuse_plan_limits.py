"""The warp fuse kernel's plan at and one past each of its limits (six rounds, 16 staged segments, 40
rules), its variants of several rounds with the clean-up stamps, with and without top-k rows, and
batched maps of several rounds. Against the oracle, from the same state."""
import numpy as np
import pytest

import oracle as O
from paper_2309_16818_gb300 import synth

from helpers import compare_states, gpu_state, make_pair, specs_to, upload_state
from test_gpu_fuse_plans import D, E, G, L, X, _rows
from test_gpu_raycast_drift import KW, lifted, phantoms

pytestmark = pytest.mark.gpu

# per source: (type, channels, rules of its layers)
CASES = {
    "six rounds": [("f32", 188, [E])],
    "a seventh round": [("f32", 189, [E])],
    "six rounds and a pair": [("bf16", 186, [X, E])],
    "pairs that need a seventh": [("f32", 59, [X]), ("f32", 55, [X]), ("u8", 55, [X])],
    "16 segments": [("f32", 4, [E, X]), ("bf16", 30, [E]), ("f32", 45, [E, X]), ("u8", 24, [E, X]), ("f32", 4, [X]),
                    ("f16", 8, [E]), ("f32", 41, [E, X]), ("f32", 8, [X])],
    "17 segments": [("u8", 23, [E])] * 8,
    "40 rules": [("f32", 124, [G, E, D, L, E, G, E, D])],
    "42 rules": [("f32", 130, [G, E, D, L, E, G, E])],
}


def _inputs(r, spec, n, l0=0):
    """Random rows of every source: (GPU, oracle) source lists."""
    import torch
    gs, os_ = [], []
    for dt, C, rules in spec:
        a = _rows(r, dt, n, C)
        t = torch.from_numpy(a).cuda()
        if dt in ("bf16", "f16"):
            t = t.to(torch.bfloat16 if dt == "bf16" else torch.float16)
            a = t.float().cpu().numpy()
        ls = list(range(l0, l0 + len(rules)))
        l0 += len(rules)
        gs.append((t, ls))
        os_.append((a, ls))
    return gs, os_


def _layers(spec):
    return [dict(channels=C, rule=q, w=0.3, var_meas=0.7, alpha0=0.5) for _, C, rules in spec for q in rules]


@pytest.mark.parametrize("case", list(CASES))
def test_limits_against_the_oracle(case):
    import torch
    spec, W, n = CASES[case], 36, 5003
    g, o = make_pair(W, 0.05, _layers(spec), outlier_var=1e-4)
    r = np.random.default_rng(len(case))
    ter = synth.Terrain.from_seed(W)
    for k in range(2):
        cl = synth.uniform_ground_cloud(20 + k, n, 1.1 * W * 0.05, ter)
        gs, os_ = _inputs(r, spec, n)
        if k:
            upload_state(g, o)
        o.fuse_points(cl.xyz, cl.T, os_)
        g.fuse_pointcloud(torch.from_numpy(cl.xyz).cuda(), cl.T, gs)
        g.check()
        compare_states(gpu_state(g), o, what=f"{case} call {k}")


@pytest.mark.parametrize("topk", [0, 5])
def test_cleanup_and_drift_over_rounds(topk):
    import torch
    from paper_2309_16818_gb300 import mem as M
    c = synth.config2(n_poses=3, scale=0.25)
    spec = [("u8", 3, [L]), ("bf16", 64, [G, E])]
    K = 40
    layers = _layers(spec) + [dict(channels=K, rule=q, w=0.3) for q in (D, X)]
    g, o = make_pair(c["W"], c["res"], layers, **KW)
    r = np.random.default_rng(7)
    cleared = 0
    for k, (scan, dz) in enumerate(zip(c["scans"], (0.0, 0.03, -0.02))):
        if k:
            phantoms(o, r, 400)
        upload_state(g, o)
        n = len(scan.xyz)
        gs, os_ = _inputs(r, spec, n)
        if topk:
            p = np.empty((n, 2 * topk), np.float32)
            p[:, 0::2] = r.integers(-1, K + 1, (n, topk))
            p[:, 1::2] = r.random((n, topk)) - 0.2
            gs.append((M.TopK(torch.from_numpy(p).cuda(), K), [3, 4]))
            os_.append((O.TopK(p, K), [3, 4]))
        else:
            p = _rows(r, "f32", n, K)
            gs.append((torch.from_numpy(p).cuda(), [3, 4]))
            os_.append((p, [3, 4]))
        T = lifted(scan.T, dz)
        ro = o.fuse_points(scan.xyz, T, os_)
        g.fuse_pointcloud(torch.from_numpy(scan.xyz).cuda(), T, gs)
        g.check()
        assert g.get_drift()["cleared"] == ro["cleared"]
        compare_states(gpu_state(g), o, what=f"top-{topk} pose {k}")
        cleared += ro["cleared"]
    assert cleared > 50


@pytest.mark.parametrize("cleanup", [False, True])
def test_batched_maps_over_rounds(cleanup):
    import torch
    kw = KW if cleanup else {}
    B, spec = 4, [("u8", 3, [L]), ("bf16", 64, [G]), ("f32", 20, [D, X])]
    c = synth.config4(n_maps=B, n_lo=500, n_hi=9000)
    clouds = list(c["clouds"])
    clouds[1] = synth.Cloud(clouds[1].xyz[:0], clouds[1].T, clouds[1].rgb[:0], None, clouds[1].feat[:0])
    offsets = np.concatenate([[0], np.cumsum([cl.n for cl in clouds])]).astype(np.int64)
    layers = _layers(spec)
    g, _ = make_pair(c["W"], c["res"], layers, n_maps=B, **kw)
    oracles = [O.OracleMap(O.Params(W=c["W"], res=c["res"], layers=specs_to(layers, "oracle"), **kw)) for _ in range(B)]
    xyz = torch.from_numpy(np.ascontiguousarray(np.concatenate([cl.xyz for cl in clouds]))).cuda()
    r = np.random.default_rng(9)
    for rnd in range(2):
        gs, os_ = _inputs(r, spec, int(offsets[-1]))
        Ts = np.stack([cl.T for cl in clouds])
        cleared = 0
        for b, cl in enumerate(clouds):
            if rnd:
                phantoms(oracles[b], r, 100 if cl.n else 0)
                upload_state(g, oracles[b], map_index=b)
            cut = [(a[offsets[b]:offsets[b + 1]], l) for a, l in os_]
            cleared += oracles[b].fuse_points(cl.xyz, Ts[b], cut).get("cleared", 0)
        g.fuse_pointcloud_batch(offsets, xyz, Ts, gs)
        g.check()
        if cleanup:
            assert g.get_drift(0)["cleared"] == cleared
        for b in range(B):
            compare_states(gpu_state(g, b), oracles[b], what=f"round {rnd} map {b}")
