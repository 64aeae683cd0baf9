"""FP32 backward of a tile in which one key is masked by an infinity in K (its
scores are -inf, so its probabilities are 0): the gradients of all keys are
finite and those of the others are what they are without that key, also where
the last 64-row block of queries is not full."""
import numpy as np
import pytest
import torch

from paper_2604_16590_gb300 import build, gattn
from paper_2604_16590_gb300.inputs import qkv, upstream_grad
from tests._parity import assert_close

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    gattn.load_library()


@pytest.mark.parametrize("d", [32, 64, 128])
@pytest.mark.parametrize("L", [32, 64, 96, 200])
def test_masked_key(d, L):
    shape, j = (1, 2, L, d), L // 3
    q, k, v = qkv(shape, 80 + L, 1.0, "fp32")
    go = upstream_grad(shape, 80 + L, "fp32")
    q[..., 0] = q[..., 0].abs() + 0.1
    k[:, :, j, 0] = float("-inf")
    t = [x.cuda() for x in (q, k, v)]
    tiling = gattn.Tiling((1, 1, L), (1, 1, L), (0, 0, 0))
    out, saved = gattn.forward(*t, tiling)
    _, dk, dv = gattn.backward(*t, out, go.cuda(), saved, tiling)
    assert gattn.gattn_stream_status() == 0
    keep = [i for i in range(L) if i != j]
    q64, k64, v64, g64 = q.double(), k.double()[:, :, keep], v.double()[:, :, keep], go.double()
    p = torch.softmax(q64 @ k64.transpose(2, 3) / np.sqrt(d), -1)
    o = p @ v64
    ds = p * (g64 @ v64.transpose(2, 3) - (g64 * o).sum(-1, keepdim=True)) / np.sqrt(d)
    for name, got, ref in (("out", out, o), ("dk", dk, ds.transpose(2, 3) @ q64), ("dv", dv, p.transpose(2, 3) @ g64)):
        got = got.cpu()
        if name != "out":
            assert (got[:, :, j] == 0).all(), name
            got = got[:, :, keep]
        assert_close(name, got.numpy(), ref.numpy(), 1e-5, 1e-5)
