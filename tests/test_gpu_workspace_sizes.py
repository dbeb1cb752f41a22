"""One workspace, zero-filled once, serves calls of every B*H up to the one it was made for: what a
call leaves in it must not reach another of a different size.  The larger call leaves words there whose
upper halves are the stage numbers by which the one-pass quantizer recognises a published maximum."""
import numpy as np
import pytest
import torch

from paper_2609_13031_b200 import api

pytestmark = pytest.mark.gpu


def leave_amax(ws, heads):
    """The two-pass form of `heads` heads: its accumulators end as the fp32 bits of the maxima, here
    the bf16 subnormals 1 .. 4, i.e. 0x00010000 .. 0x00040000."""
    bits = torch.from_numpy((np.arange(heads) % 4 + 1).astype(np.int16)).cuda()
    x = bits.view(1, heads, 1, 1).expand(1, heads, 8, 64).contiguous().view(torch.bfloat16)
    api.quantize_qkv(x, x, x, None, ws, flags=api.QKV_TWO_LAUNCHES)


def leave_sums(ws, heads):
    """Sums of squares in fp64, whose lower words can be anything."""
    x = torch.randn((1, heads, 8, 64), device="cuda").to(torch.bfloat16)
    api.perturb(x, 0.1, 1, 1, ws)


def leave_partials(ws, heads):
    """Partial results of the key split, which start behind the words of a workspace of two heads."""
    x = torch.randn((1, 2, 4096, 64), device="cuda").to(torch.bfloat16)
    api.icl_forward_bf16(None, x[:, :, :256].contiguous(), x, x, ws, flags=api.SPLIT_TAIL | api.TEST_ROWS_ONLY)


@pytest.mark.parametrize("leave", [leave_amax, leave_sums, leave_partials])
@pytest.mark.parametrize("H,n,m", [(1, 40000, 64), (8, 2500, 300), (21, 2100, 9), (64, 2100, 9)])
def test_call_of_another_size_before(leave, H, n, m):
    torch.manual_seed(H)
    q, k, v = (torch.randn((1, H, n, 64), device="cuda").to(torch.bfloat16) for _ in range(3))
    t = torch.randn((1, H, m, 64), device="cuda").to(torch.bfloat16)
    clean = api.new_workspace(1, H)
    want = api.quantize_qkv(q, k, v, t, clean, flags=api.QKV_TWO_LAUNCHES)
    ws = api.new_workspace(1, 64, n_train=4096, d=64)
    for heads in (64, 33):
        leave(ws, heads)
        got = api.quantize_qkv(q, k, v, t, ws)
        for name in ("q8", "k8", "v8", "t8", "sq", "sk", "sv"):
            assert torch.equal(got[name], want[name]), name
        leave(ws, heads)
        code, scale = api.quantize(k, ws)
        assert torch.equal(code, want["k8"]) and torch.equal(scale, want["sk"])
    assert api.last_device_status(ws) == (0, 0)
