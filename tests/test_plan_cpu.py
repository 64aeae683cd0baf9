"""Geometries kept per thread and call plans kept by value give what a fresh
computation gives: more descriptors than are kept, in turn and changed in
place, and tilings given as tuples and as lists."""
import threading

import pytest
import torch

from paper_2604_16590_gb300 import build, gattn


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    gattn.load_library()


def _descs():
    out = []
    for i in range(6):
        out.append(gattn.make_desc(1 + i % 2, 1 + i, 64, (1 + i, 16, 20 + i), (1, 8, 10), (i % 2, 2, 3), in_dtype="bf16"))
    return out


def _sizes(d):
    return (gattn.gattn_saved_bytes(d), gattn.gattn_bwd_workspace_bytes(d), gattn.gattn_num_tiles(d), gattn.gattn_block_shape(d))


def _fresh(d):
    """The sizes as a thread that has built no geometry yet sees them."""
    got = []
    t = threading.Thread(target=lambda: got.append(_sizes(d)))
    t.start()
    t.join()
    return got[0]


def test_geometries_are_kept_by_value():
    descs = _descs()
    want = [_fresh(d) for d in descs]
    assert len(set(want)) == len(want)
    for _ in range(3):
        assert [_sizes(d) for d in descs] == want
    d = descs[0]
    for halo in (0, 3, 5):  # the same object with other contents
        d.halo[2] = halo
        assert _sizes(d) == _fresh(d)
    d.core[1] = 0
    assert gattn.gattn_validate(d) == 1 and gattn.gattn_saved_bytes(d) == 0


def test_plans_of_tuples_and_lists_agree():
    q = torch.zeros(1, 2, 320, 64, dtype=torch.bfloat16)
    a = gattn._plan_for(q, gattn.Tiling((1, 16, 20), (1, 8, 10), (0, 2, 3)), None)
    b = gattn._plan_for(q, gattn.Tiling([1, 16, 20], [1, 8, 10], [0, 2, 3]), None)
    f = gattn._plan_for(q, gattn.Tiling((1, 16, 20), (1, 8, 10), (0, 2, 3)), torch.float32)
    assert bytes(a[0]) == bytes(b[0]) and a[1:] == b[1:]
    assert a[1] == torch.bfloat16 and f[1] == torch.float32
    with pytest.raises(ValueError):
        gattn._plan_for(q, gattn.Tiling((1, 16, 21), (1, 8, 10), (0, 2, 3)), None)
