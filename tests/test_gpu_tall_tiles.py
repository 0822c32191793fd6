"""The forward step's 64 x 64 tiles, which rows of whole 128-byte lines take
from 2^26 cells on, against its 64 x 32 tiles, bit for bit: a step reads R cells
around a cell, so for a few steps the record of sensors near one end of a long
grid is that of a short grid with the same end, whose steps take the 64 x 32
tiles and sum in the same order."""
import numpy as np
import pytest

from gpu_helpers import need_gpu

pytestmark = pytest.mark.gpu

H, NT = 1e-4, 6
NY, NX, CROP = 1025, 65568, 192  # last tile row of one cell row, last tile column of 32; NX % 32 == 0


def plan_of(shape, c, order, sensors, layer):
    from paper_2507_02401_gb300 import Plan
    p = Plan(shape, H, 0.3 * H / 1600.0, NT, order, c, sensors, 2, 0)
    p.path = 2
    if layer:
        p.set_sponge(layer)
    return p


@pytest.mark.parametrize("order", [2, 4, 6, 8])
@pytest.mark.parametrize("varc,layer", [(False, 0), (True, 0), (False, 9), (True, 9)])
def test_tall_tiles_have_the_bits_of_the_others(order, varc, layer):
    torch = need_gpu()
    rng = np.random.default_rng(order)
    ends = {0: rng.integers(0, 100, 60), NX - CROP: NX - 2 - rng.integers(0, 100, 60)}  # R NT + 100 < CROP - layer
    gen = torch.Generator(device="cuda").manual_seed(order)
    x = torch.zeros((NY, NX), device="cuda")
    c = np.full((NY, NX), 1500.0) if varc else 1500.0
    sens = {}
    for col, xs in ends.items():
        x[:, col:col + CROP] = torch.randn((NY, CROP), device="cuda", generator=gen)
        if varc:
            c[:, col:col + CROP] = rng.uniform(1400.0, 1600.0, (NY, CROP))
        ys = np.concatenate([np.arange(30), NY - 2 - np.arange(30)])
        sens[col] = np.stack([(xs + 0.25) * H, (ys + 0.5) * H], axis=1)
    if varc:
        c[0, NX // 2] = 1600.0  # the same fastest cell, so the same layer, in every plan
    big = plan_of((NY, NX), c, order, np.concatenate(list(sens.values())), layer)
    y = big.forward(x)
    assert big.check() == 0
    for k, col in enumerate(ends):
        cc = c
        if varc:
            cc = c[:, col:col + CROP].copy()
            cc[0, -1 if col == 0 else 0] = 1600.0  # out of the sensors' reach
        short = plan_of((NY, CROP), cc, order, sens[col] - [col * H, 0.0], layer)
        assert torch.equal(short.forward(x[:, col:col + CROP].contiguous()), y[60 * k:60 * k + 60])
        short.close()
    big.close()
