"""The FP32 form at the edges of its shapes for short tiles (16, 32 and, at
d = 32, 448 rows) and with tiles of different lengths, against the FP64 oracle
at the FP32 bar (max-rel and rms-rel <= 1e-5)."""
import pytest
import torch

import oracle
from paper_2604_16590_gb300 import build, gattn
from paper_2604_16590_gb300.inputs import qkv, upstream_grad
from tests._parity import assert_close

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    gattn.load_library()


def _check(d, nh, grid, core, halo, seed):
    shape = (1, nh, grid[0] * grid[1] * grid[2], d)
    q, k, v = qkv(shape, seed, 1.0, "fp32")
    go = upstream_grad(shape, seed, "fp32")
    t = [x.cuda() for x in (q, k, v, go)]
    tiling = gattn.Tiling(grid, core, halo)
    out, saved = gattn.forward(*t[:3], tiling)
    grads = gattn.backward(*t[:3], out, t[3], saved, tiling)
    assert gattn.gattn_stream_status() == 0
    geo = oracle.Geometry(1, nh, d, *grid, core, halo, "hann")
    x = [a.numpy() for a in (q, k, v, go)]
    ref = [oracle.forward(geo, *x[:3]), *oracle.backward(geo, *x)]
    for name, got, want in zip(("out", "dq", "dk", "dv"), (out, *grads), ref):
        assert_close(name, got.cpu().numpy(), want, 1e-5, 1e-5)


@pytest.mark.parametrize("d", [32, 64, 128])
@pytest.mark.parametrize("L", [5, 15, 16, 17, 32, 33])
def test_one_tile(d, L):
    _check(d, 3, (1, 1, L), (1, 1, L), (0, 0, 0), 50 + L)


@pytest.mark.parametrize("L", [447, 448, 449])
def test_long_tiles_d32(L):
    _check(32, 24, (1, 1, L), (1, 1, L), (0, 0, 0), 60 + L)


@pytest.mark.parametrize("d", [32, 64, 128])
@pytest.mark.parametrize("core,halo", [((1, 3, 4), (0, 0, 0)), ((1, 2, 3), (0, 1, 1)), ((1, 2, 5), (0, 1, 0))])
def test_many_short_tiles(d, core, halo):
    _check(d, 2, (2, 13, 17), core, halo, 70)
