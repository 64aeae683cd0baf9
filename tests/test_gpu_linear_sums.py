"""The sums over a CTA's tiles in linear attention: the rings and groups of the
backward at 1 to 8 and more tiles per CTA, sums folded after every tile and
after several with and without a remainder, and the accuracy of the summed
matrices where a CTA takes many tiles."""
import pytest
import torch

from oracle import linear as ol
from paper_2604_16590_gb300 import gattn
from paper_2604_16590_gb300.inputs import qkv
from tests._parity import assert_close

pytestmark = pytest.mark.gpu


def _up(n):
    return (n + 255) // 256 * 256


def _run(q, k, v, g):
    """(out, dq, dk, dv), S, dS of [1, heads, N, 64] inputs and the partials per head of the
    backward.  Both buffers end with the combined matrices: S^T (high, low part), z, and dS,
    dS^T (high, low each), dz."""
    nh = q.shape[1]
    desc = gattn.linear_desc(q)
    out, saved = gattn.linear_forward(q, k, v, keep_summary=True)
    grads = [torch.empty_like(q) for _ in range(3)]
    ws = torch.empty(gattn.gattn_linear_bwd_workspace_bytes(desc), dtype=torch.uint8, device="cuda")
    assert gattn.gattn_linear_bwd(desc, q, k, v, g, saved, *grads, ws) == 0
    assert gattn.gattn_stream_status() == 0
    mat, vec = _up(nh * 8192), _up(nh * 256)

    def both(buf, hi, lo):
        return sum(buf[o : o + nh * 8192].view(torch.bfloat16).double() for o in (hi, lo)).view(nh, 64, 64)

    e = saved.numel() - vec
    S = both(saved, e - 2 * mat, e - mat).transpose(1, 2)
    e = ws.numel() - vec - 4 * mat
    dS = both(ws, e, e + mat)
    parts = next(c for c in range(1, 2000) if _up(c * nh * 16384) + _up(c * nh * 256) >= e)
    return (out, *grads), S, dS, parts


# with 152 heads or more a head's tiles lie in one CTA of the backward
@pytest.mark.parametrize("nh,tiles", [(152, t) for t in (1, 2, 3, 4, 5, 7, 8, 17, 35)] + [(304, 43)])
def test_tiles_per_cta(nh, tiles):
    N = 128 * tiles - 3
    q, k, v = qkv((1, nh, N, 64), 900 + tiles, 0.5, "bf16", "cuda")
    (g,) = qkv((1, nh, N, 64), 1900 + tiles, 1.0, "bf16", "cuda", n=1)
    got, _, _, parts = _run(q, k, v, g)
    assert parts == 1
    for h in (0, 1, nh - 1):
        x = [t[:, h : h + 1].double().cpu().numpy() for t in (q, k, v, g)]
        ref = [ol.forward(*x[:3]), *ol.backward(*x)]
        for name, a, r in zip(("out", "dq", "dk", "dv"), got, ref):
            assert_close(f"{name}/{h}", a[:, h : h + 1].double().cpu().numpy(), r, 2e-2, 3e-3)


def _ref64(q, k, v, g):
    """One head in FP64: (out, dq, dk, dv), S, dS."""
    q, k, v, g = (t.double() for t in (q, k, v, g))
    (fq, eq), (fk, ek) = ((torch.where(x > 0, x + 1, x.exp()), torch.where(x > 0, torch.ones_like(x), x.exp())) for x in (q, k))
    S, z = fk.T @ v, fk.sum(0)
    den = (fq @ z)[:, None]
    out = fq @ S / den
    go = (g * out).sum(-1, keepdim=True)
    dS, dz = fq.T @ (g / den), -(fq * (go / den)).sum(0)
    return (out, (g @ S.T - go * z) / den * eq, (v @ dS.T + dz) * ek, fk @ dS), S, dS


def test_sums_of_many_tiles_stay_accurate():
    """64 tiles per CTA with values of mean 1/2, so that S and dS grow steadily.  The tensor core
    truncates an accumulator by less than 2^-23 of it at each of its K = 16 steps, on average at
    half of its final size.  8 tiles per sum: S takes 16 steps per tile (high and low part of phi), dS 24.
    The matrices are kept in two BF16 parts (2^-18) and the products drop low times low (2^-18)."""
    nh, N = 304, 64 * 128
    gen = torch.Generator(device="cuda").manual_seed(5)
    q, k, v, g = (
        (torch.randn((1, nh, N, 64), generator=gen, device="cuda") * 0.5 + mean).to(torch.bfloat16) for mean in (0, 0, 0.5, 0.5)
    )
    _, S, dS, _ = _run(q, k, v, g)
    for name, got, steps in (("S", S, 16 * 8), ("dS", dS, 24 * 8)):
        err = ref = 0.0
        for h in range(0, nh, 50):
            r = _ref64(q[0, h], k[0, h], v[0, h], g[0, h])[1 if name == "S" else 2]
            err += float(((got[h] - r) ** 2).sum())
            ref += float((r**2).sum())
        bound = steps / 2 * 2.0**-23 + 2 * 2.0**-18
        assert (err / ref) ** 0.5 <= bound, (name, (err / ref) ** 0.5, bound)


def test_long_heads():
    """16 heads of 262144 tokens, 108 tiles per CTA: whole heads against FP64."""
    q, k, v = qkv((1, 16, 262144, 64), 71, 0.5, "bf16", "cuda")
    (g,) = qkv((1, 16, 262144, 64), 72, 1.0, "bf16", "cuda", n=1)
    got, _, _, _ = _run(q, k, v, g)
    for h in (0, 7, 15):
        ref = _ref64(q[0, h], k[0, h], v[0, h], g[0, h])[0]
        for name, a, r in zip(("out", "dq", "dk", "dv"), got, ref):
            assert_close(f"{name}/{h}", a[0, h].double().cpu().numpy(), r.cpu().numpy(), 2e-2, 3e-3)
