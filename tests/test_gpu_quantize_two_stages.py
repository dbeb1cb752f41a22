"""Calls of two stages of the one-pass quantizer, whose shares are loaded and exchanged together: the two passes'
codes and scales bit for bit, with stages of the same and of different lengths, twice on one workspace, and a
clean end when the waits run out."""
import pytest
import torch

from helpers import Guarded
from paper_2609_13031_b200 import api

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tensors,B,H,n,m,d", [
    (1, 2, 8, 12289, 0, 64),       # 16 heads, eight and eight
    (1, 1, 9, 20011, 0, 64),       # nine heads, five and four
    (1, 1, 2, 40000, 0, 128),      # a head each
    (1, 1, 3, 32768, 0, 128),      # two and one
    (3, 1, 8, 8192, 2048, 64),     # 24 units
    (3, 1, 5, 10007, 40000, 64),   # 15 units, test rows outnumber the train rows
    (3, 1, 2, 16000, 1, 128),
    # above 48 MB: a launch before clears the words, and all threads wait for the heads that their rows follow
    (3, 1, 16, 2600, 32768, 128),
    (3, 2, 4, 5000, 32768, 128),
    (3, 1, 8, 10007, 60000, 64),
])
@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float16])
def test_matches_two_passes(tensors, B, H, n, m, d, dtype):
    assert api.quantize_stages(tensors, B, H, n, m, d) == 2
    g = torch.Generator(device="cuda")
    ws = api.new_workspace(B, H)
    for seed in (1, 2):
        g.manual_seed(seed)
        x = [torch.empty((B, H, r, d), dtype=dtype, device="cuda").normal_(generator=g) if r else None for r in (n, n, n, m)]
        if tensors == 1:
            got, want = (api.quantize(x[0], ws, flags=f) for f in (0, api.QKV_TWO_LAUNCHES))
        else:
            got, want = (api.quantize_qkv(*x, ws, flags=f) for f in (0, api.QKV_TWO_LAUNCHES))
            names = ("q8", "k8", "v8", "sq", "sk", "sv") + (("t8",) if m else ())
            got, want = ([o[c] for c in names] for o in (got, want))
        for a, b in zip(got, want):
            assert torch.equal(a, b)
    assert api.last_device_status(ws) == (0, 0)


@pytest.mark.parametrize("limit", [1, 3000, 8000])
def test_gives_up_cleanly(limit):
    """Waits of that many clocks end before or between the two shares (or, the longest, perhaps not at all)."""
    H, n, d = 16, 12289, 64
    assert api.quantize_stages(1, 1, H, n, 0, d) == 2
    x = torch.randn((1, H, n, d), device="cuda").to(torch.bfloat16)
    ws = api.new_workspace(1, H)
    code, scale = Guarded((1, H, n, d), torch.uint8), Guarded((1, H), torch.float32)
    api.selftest_quantize_timeout(x, ws, code.t, scale.t, limit)
    status, _ = api.last_device_status(ws)
    assert status == api.ERR_TIMEOUT or limit > 1 and status == 0
    code.check()
    scale.check()
    want = api.quantize(x, ws, flags=api.QKV_TWO_LAUNCHES)
    got = api.quantize(x, ws)
    assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1])
    assert api.last_device_status(ws) == (0, 0)
