"""The U-Net's backward pass: the same state and batch give the same gradients, loss and trained
parameters bit for bit, and gradients agree with the float64 oracle at sizes where a
weight-gradient block takes many tiles and widths whose planes do not divide the grid."""
import numpy as np
import pytest

from test_gpu_unet import _gpu_and_oracle, _grad_errors, torch  # noqa: F401  (the fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("widths,N,H,W", [((32, 64, 128, 128), 3, 200, 136), ((32, 32, 32, 32), 1, 8, 8),
                                          ((96, 32, 160, 256), 2, 64, 72), ((32, 64, 128, 128), 4, 256, 256)])
def test_gradients_and_steps_repeat_bit_for_bit(torch, widths, N, H, W):  # noqa: F811
    from paper_2309_16818_gb300 import mem as M
    from paper_2309_16818_gb300.inpaint import init_params
    rng = np.random.default_rng(3)
    t = lambda a: torch.from_numpy(a).cuda()  # noqa: E731
    x3 = t(rng.normal(size=(N, H, W, 3)).astype(np.float32))
    fill, target = (t(rng.normal(size=(N, H, W)).astype(np.float32)) for _ in range(2))
    hidden = t((rng.random((N, H, W)) < 0.4).astype(np.uint8))
    flat = t(init_params(1, 3, widths, out_scale=1.0))
    runs = []
    for _ in range(3):
        net = M.UNet(3, widths)
        net.set_params(flat)
        out = [*net.gradients(x3, fill, target, hidden), *net.gradients(x3, fill, target, hidden)]
        for _ in range(3):
            out += [net.train_step(x3, fill, target, hidden, 1e-3), net.get_params()]
        net.check()
        runs.append([o.cpu() for o in out])
        net.close()
    for r in runs:
        assert torch.equal(r[0], runs[0][0]) and torch.equal(r[1], runs[0][1])
        assert torch.equal(r[2], r[0]) and torch.equal(r[3], r[1])
        assert all(torch.equal(a, b) for a, b in zip(r, runs[0]))
    assert all(bool(torch.isfinite(o).all()) for o in runs[0])


@pytest.mark.parametrize("widths,N,H,W", [((32, 32, 32, 32), 2, 200, 136), ((96, 32, 32, 160), 2, 64, 72)])
def test_gradients_match_oracle_over_many_tiles(torch, widths, N, H, W):  # noqa: F811
    """The bounds of test_forward_and_gradients_match_oracle."""
    pred, fill, loss, g, out = _gpu_and_oracle(torch, widths, N, H, W, seed=0)
    res, lo, go = out["bf16"]
    assert np.linalg.norm(pred - (fill + res)) / np.linalg.norm(res) < 1e-2
    assert abs(loss - lo) <= 1e-2 * lo
    floor = {}
    for k in out:
        if k.startswith("bf16_jitter"):
            for n, rel, _ in _grad_errors(out[k][2], go):
                floor[n] = max(floor.get(n, 0.0), rel)
    bad = [(n, rel, c, floor[n]) for n, rel, c in _grad_errors(g, go)
           if not (rel <= 2e-2 or c >= 0.999 or (floor[n] > 2e-2 and rel <= 3 * floor[n]))]
    assert not bad, bad


def test_a_batch_that_does_not_fit_leaves_the_network_usable(torch):  # noqa: F811
    """2^27 cells at 256 channels need several times the device's memory: refused as out of memory,
    after which the shape that had its buffers before gets new ones and the same results."""
    from paper_2309_16818_gb300 import mem as M
    from paper_2309_16818_gb300.inpaint import init_params
    widths = (256, 256, 256, 256)
    if torch.cuda.get_device_properties(0).total_memory > 400 << 30:
        pytest.skip("such a batch may fit this device")
    net = M.UNet(3, widths)
    net.set_params(torch.from_numpy(init_params(1, 3, widths, out_scale=1.0)).cuda())
    rng = np.random.default_rng(5)
    x3 = torch.from_numpy(rng.normal(size=(2, 32, 24, 3)).astype(np.float32)).cuda()
    fill = torch.from_numpy(rng.normal(size=(2, 32, 24)).astype(np.float32)).cuda()
    before = net.forward(x3, fill)
    n, S = 8, 4096
    big = torch.zeros((1, 1, 1, 3), device="cuda").expand(n, S, S, 3)  # (never read: refused before any launch)
    with pytest.raises(M.MemError, match="memory"):
        net.forward(big, fill, out=fill)
    again = net.forward(x3, fill)
    net.check()
    assert torch.equal(before, again)
    net.close()
