"""The backward's workspace: with FP32 inputs two vectors and three matrices of
slots, without the tables of the tensor-core form."""
import pytest

from paper_2604_16590_gb300 import build, gattn


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    gattn.load_library()


@pytest.mark.parametrize("d", [32, 64, 128])
@pytest.mark.parametrize("B,nh", [(1, 1), (2, 3)])
def test_fp32_backward_workspace(d, B, nh):
    # four tiles of 8 x 16 tokens: one box of 128 slots each
    slots = B * nh * 4 * 128
    desc = gattn.make_desc(B, nh, d, (1, 16, 32), (1, 8, 16), (0, 0, 0), in_dtype="fp32")
    assert gattn.gattn_bwd_workspace_bytes(desc) == 2 * slots * 4 + 3 * slots * d * 4
    if d != 32:  # BF16 inputs: places (4 bytes) and statistics rows (16 bytes) per slot, box counts per tile
        desc = gattn.make_desc(B, nh, d, (1, 16, 32), (1, 8, 16), (0, 0, 0), in_dtype="bf16")
        assert gattn.gattn_bwd_workspace_bytes(desc) == 7 * slots * 4 + 256 + 3 * slots * d * 4
