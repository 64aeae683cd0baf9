"""The d = 128 forward's key mask: what lies outside a tile stays outside.

Tiles of 13 x 13 tokens take two boxes of 7 x 13, so the second box of the
upper tiles reads a row of the tiles below them as keys that have to be masked.
A key there that is not finite must not change any other tile, and a mask has
to hold at every scale."""
import numpy as np
import pytest
import torch

import oracle
from paper_2604_16590_gb300 import build, gattn
from paper_2604_16590_gb300.inputs import qkv
from tests._parity import assert_close

pytestmark = pytest.mark.gpu

GRID, CORE, HALO = (1, 26, 26), (1, 13, 13), (0, 0, 0)
SHAPE = (1, 2, 26 * 26, 128)


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    gattn.load_library()


@pytest.mark.parametrize("bad", [float("nan"), float("inf"), float("-inf")])
@pytest.mark.parametrize("columns", [1, 128])
def test_a_key_outside_the_tile_does_not_reach_it(bad, columns):
    q, k, v = (t.cuda() for t in qkv(SHAPE, 61, 0.5, "bf16"))
    tiling = gattn.Tiling(GRID, CORE, HALO)
    assert gattn.gattn_block_shape(gattn.desc_for(q, tiling)) == (0, (1, 7, 13))  # the box that sticks out
    clean, _ = gattn.forward(q, k, v, tiling)
    k[:, :, 13 * 26 + 5, :columns] = bad  # first row of the lower left tile
    out, _ = gattn.forward(q, k, v, tiling)
    assert gattn.gattn_stream_status() == 0
    other = torch.ones(26, 26, dtype=torch.bool)
    other[13:, :13] = False
    other = other.reshape(-1).cuda()
    assert torch.equal(out[:, :, other], clean[:, :, other])


@pytest.mark.parametrize("scale", [1e-30, 1e-20, 1e-3])
def test_masked_at_every_scale(scale):
    q, k, v = qkv(SHAPE, 62, 0.5, "bf16")
    out, _ = gattn.forward(q.cuda(), k.cuda(), v.cuda(), gattn.Tiling(GRID, CORE, HALO, scale=scale), out_dtype=torch.float32)
    assert gattn.gattn_stream_status() == 0
    geo = oracle.Geometry(1, 2, 128, *GRID, CORE, HALO, scale=scale)
    ref = oracle.forward(geo, *(t.double().numpy() for t in (q, k, v)))
    assert_close("out", out.cpu().numpy().astype(np.float64), ref, 2e-2, 3e-3)
