"""The FP32 form at the edges of its row blocks (64 and 32 rows a CTA) and of
its 64-row streamed blocks, for every head size: one tile of L tokens, alone
(32-row CTAs) and with enough heads to fill the GPU (64-row CTAs), against the
FP64 oracle at the FP32 bar (max-rel and rms-rel <= 1e-5)."""
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


@pytest.mark.parametrize("d", [32, 64, 128])
@pytest.mark.parametrize("L", [2, 31, 33, 63, 64, 65, 129, 200])
@pytest.mark.parametrize("nh", [1, 160])
def test_row_block_edges(d, L, nh):
    shape = (1, nh, L, d)
    q, k, v = qkv(shape, 40 + L, 1.0, "fp32")
    go = upstream_grad(shape, 40 + L, "fp32")
    tq, tk, tv, tg = (t.cuda() for t in (q, k, v, go))
    tiling = gattn.Tiling((1, 1, L), (1, 1, L), (0, 0, 0))
    out, saved = gattn.forward(tq, tk, tv, tiling)
    grads = gattn.backward(tq, tk, tv, out, tg, saved, tiling)
    assert gattn.gattn_stream_status() == 0
    geo = oracle.Geometry(1, nh, d, 1, 1, L, (1, 1, L), (0, 0, 0), "hann")
    x = [t.numpy() for t in (q, k, v, go)]
    ref = [oracle.forward(geo, *x[:3]), *oracle.backward(geo, *x)]
    for name, got, want in zip(("out", "dq", "dk", "dv"), (out, *grads), ref):
        assert_close(f"{name}", got.cpu().numpy(), want, 1e-5, 1e-5)
