"""Temporal compression where its frame split changes: one range, two, many
ranges of the least length, one wave of longer ones, ranges that do not divide
the frames, at every head size, against the FP64 oracle (the bars of
test_gpu_compress.py for FP32: 1e-5)."""
import pytest
import torch

from oracle import compress as oc
from paper_2604_16590_gb300 import gattn
from paper_2604_16590_gb300.inputs import qkv
from tests._parity import assert_close

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d", [32, 64, 128])
@pytest.mark.parametrize("S,M", [(63, 40), (128, 33), (130, 64), (701, 31), (1300, 65), (1300, 320)])
def test_frame_ranges(d, S, M):
    k, v = qkv((1, 2, S, M, d), 11 + S, 1.0, "fp32", "cuda", n=2)
    (q,) = qkv((2, d), 12 + S, 1.0, "fp32", "cuda", n=1)
    out, lse = gattn.compress_forward(q, k, v)
    assert gattn.gattn_stream_status() == 0
    ref, rlse = oc.forward(*(t.double().cpu().numpy() for t in (q, k, v)))[:2]
    assert_close("out", out.cpu().numpy(), ref, 1e-5, 1e-5)
    assert_close("lse", lse.cpu().numpy()[..., None], rlse[..., None], 1e-5, 1e-5)
