"""A device wait that runs out in the d = 128 forward (the issuer of the scores
waits on an mbarrier that nothing arrives on): the warps that meet at pair
barriers all leave, the kernel ends, the host reads GATTN_ERR_TIMEOUT and the
context stays usable."""
import pytest
import torch

import oracle
from paper_2604_16590_gb300 import build, gattn
from paper_2604_16590_gb300.inputs import qkv
from tests._parity import assert_close

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    gattn.load_library()


# tiles of one key block, of several, and of blocks that reach out of their tile
@pytest.mark.parametrize("grid,core", [((1, 16, 16), (1, 8, 16)), ((2, 32, 32), (1, 32, 32)), ((1, 26, 26), (1, 13, 13))])
def test_timeout_is_reported_and_context_survives(grid, core):
    shape = (1, 2, grid[0] * grid[1] * grid[2], 128)
    q, k, v = (t.cuda() for t in qkv(shape, 33, 0.5, "bf16"))
    tiling = gattn.Tiling(grid, core, (0, 0, 0))
    desc = gattn.desc_for(q, tiling, torch.float32, flags=gattn.GATTN_FLAG_TEST_STALL)
    out = torch.empty(shape, dtype=torch.float32, device="cuda")
    saved = torch.empty(gattn.gattn_saved_bytes(desc), dtype=torch.uint8, device="cuda")
    assert gattn.gattn_fwd(desc, q, k, v, out, saved) == 0
    assert gattn.gattn_stream_status() == 5  # GATTN_ERR_TIMEOUT
    assert gattn.gattn_stream_status() == 0
    out2, _ = gattn.forward(q, k, v, tiling, out_dtype=torch.float32)
    assert gattn.gattn_stream_status() == 0
    geo = oracle.Geometry(1, 2, 128, *grid, core, (0, 0, 0))
    ref = oracle.forward(geo, *(t.double().cpu().numpy() for t in (q, k, v)))
    assert_close("after-timeout/out", out2.double().cpu().numpy(), ref, 2e-2, 3e-3)
