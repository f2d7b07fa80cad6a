"""Reading and writing whole layers (mem_get_layer / mem_set_layer) at the shapes where the row
copy can go wrong: rows of every unit width, rows that straddle units, ring offsets, several maps,
and buffers that are not 16-byte aligned."""
import numpy as np
import pytest

from paper_2309_16818_gb300 import mem as M

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("W", [2, 6, 62, 130])
@pytest.mark.parametrize("channels,dtype,rule,start", [
    (1, M.F32, M.LATEST, 0.0), (3, M.F32, M.LATEST, 0.0), (20, M.F32, M.DIRICHLET, 1.5), (7, M.F32, M.CLASSMAX, None),
    (64, M.BF16, M.GAUSS, 0.0), (13, M.F16, M.EXPAVG, 0.0), (2, M.BF16, M.LATEST, 0.0)])
@pytest.mark.parametrize("shift", [0, 1])
def test_layer_round_trip(W, channels, dtype, rule, start, shift):
    """What was set is read back where the cell is observed, the layer's initial value elsewhere,
    in logical order after a move that wraps the ring buffer. `shift` elements offset the buffers."""
    import torch
    tdt = {M.F32: torch.float32, M.BF16: torch.bfloat16, M.F16: torch.float16}[dtype]
    m = M.Map(W, 0.5, [M.Layer(channels, rule, dtype, alpha0=1.5)], n_maps=2)
    S = 2 if rule == M.CLASSMAX else channels
    r = np.random.default_rng(W * 100 + channels)
    for b in (1, 0):
        m.move((0.5 * (W // 2 + b), -0.5), map_index=b)  # whole-cell shifts
        val = torch.tensor(r.normal(size=(W * W, S)), device="cuda").to(tdt)
        buf = torch.empty(W * W * S + 1, dtype=tdt, device="cuda")[shift:shift + W * W * S].view(W * W, S)
        buf.copy_(val)
        obs = torch.tensor(r.random(W * W) < 0.5, device="cuda")
        m.set_layer(0, buf, map_index=b)
        m.set_layer(0, obs.to(torch.uint8), part=M.PART_OBSERVED, map_index=b)
        out = torch.full((W * W * S + 1,), 9.0, dtype=tdt, device="cuda")
        got = m.get_layer(0, map_index=b, out=out[shift:shift + W * W * S].view(W * W, S))
        init = torch.tensor([-1.0, 0.0] if rule == M.CLASSMAX else [start] * S, device="cuda").to(tdt)
        assert torch.equal(got, torch.where(obs[:, None], val, init))
        assert float(out[-1 if shift == 0 else 0]) == 9.0  # nothing outside the buffer
        h = torch.tensor(r.normal(size=W * W), dtype=torch.float32, device="cuda")
        m.set_layer(M.LAYER_HEIGHT, h, map_index=b)
        m.set_layer(M.LAYER_VALID, obs.to(torch.uint8), map_index=b)
        assert torch.equal(m.get_layer(M.LAYER_HEIGHT, map_index=b), torch.where(obs, h, 0.0))
        if rule == M.GAUSS:
            m.set_layer(0, h, part=M.PART_VAR, map_index=b)
            assert torch.equal(m.get_layer(0, M.PART_VAR, map_index=b), torch.where(obs, h, 0.0))
        # a further move shifts the contents by whole cells
        m.move((0.5 * (W // 2 + b + 1), -0.5), map_index=b)
        old = torch.where(obs[:, None], val, init).view(W, W, S)
        want = torch.cat([old[:, 1:], init.view(1, 1, S).expand(W, 1, S)], 1).reshape(W * W, S)
        assert torch.equal(m.get_layer(0, map_index=b), want)
