"""Linear attention backward at the edges of its two-group schedule: one tile,
odd and even tile counts per CTA, ragged last tiles and the tile counts around
16, against the oracle's analytic gradient (max-rel <= 2e-2, rms-rel <=
3e-3, the bar of the other linear tests); and a NaN in q, which has to reach
the same elements as in the oracle (feature maps built from minima and maxima
would lose it)."""
import numpy as np
import pytest
import torch

from oracle import linear as ol
from paper_2604_16590_gb300 import gattn
from paper_2604_16590_gb300.inputs import qkv
from tests._parity import assert_close

pytestmark = pytest.mark.gpu


def _grads(B, nh, N, seed, spoil=None):
    q, k, v = qkv((B, nh, N, 64), seed, 0.5, "bf16", "cuda")
    (g,) = qkv((B, nh, N, 64), seed + 7919, 1.0, "bf16", "cuda", n=1)
    if spoil is not None:
        q[0, 0, 5, 3] = spoil
    out, saved = gattn.linear_forward(q, k, v, keep_summary=True)
    got = gattn.linear_backward(q, k, v, g, saved)
    assert gattn.gattn_stream_status() == 0
    with np.errstate(all="ignore"):
        ref = ol.backward(*(t.double().cpu().numpy() for t in (q, k, v, g)))
    return [t.double().cpu().numpy() for t in got], ref


@pytest.mark.parametrize("N", [1, 127, 128, 129, 256, 257, 385, 2048, 2049, 2177])
@pytest.mark.parametrize("nh", [1, 3])
def test_tile_counts(N, nh):
    got, ref = _grads(1, nh, N, 500 + N)
    for name, a, r in zip(("dq", "dk", "dv"), got, ref):
        if N == 1 and name != "dv":
            # one token: out = v whatever q and k are, so both gradients are 0 and a
            # relative error means nothing.  They are differences of sums over 64
            # products v g whose factors the kernels carry to 2^-16; |v| < 4, |g| < 6.
            assert np.abs(a).max() <= 64 * 4 * 6 * 2.0**-16
            continue
        assert_close(f"{name}/{N}", a, r, 2e-2, 3e-3)


def test_many_tiles_per_chunk():
    got, ref = _grads(4, 16, 128 * 40 - 3, 9)  # chunks of three tiles
    for name, a, r in zip(("dq", "dk", "dv"), got, ref):
        assert_close(name, a, r, 2e-2, 3e-3)


def test_nan_reaches_the_same_elements():
    got, ref = _grads(1, 2, 300, 77, spoil=float("nan"))
    for a, r in zip(got, ref):
        assert np.array_equal(np.isnan(a), np.isnan(r))
