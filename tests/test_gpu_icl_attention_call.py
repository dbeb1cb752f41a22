"""api.icl_attention is quantize_qkv followed by icl_forward_fp8, bit for bit, in every form of the call."""
import pytest
import torch

from paper_2609_13031_b200 import api

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,H,n,m,d,dtype,flags", [
    (1, 2, 512, 128, 64, torch.bfloat16, 0),
    (2, 3, 333, 1, 128, torch.float16, 0),
    (1, 1, 1, 0, 64, torch.bfloat16, 0),
    (1, 4, 3000, 500, 64, torch.float16, api.SPLIT_TAIL),
    (1, 4, 700, 90, 128, torch.bfloat16, api.TEST_ROWS_ONLY | api.TEST_ROWS_USE_KV_HEAD0),
])
def test_same_as_its_two_steps(B, H, n, m, d, dtype, flags):
    torch.manual_seed(n)
    q, k, v = (torch.randn((B, H, n, d), device="cuda").to(dtype) for _ in range(3))
    t = torch.randn((B, H, m, d), device="cuda").to(dtype)
    ws = api.new_workspace(B, H, n_train=n, n_test=m, d=d)
    o = api.quantize_qkv(q, k, v, t if m else None, ws)
    want = api.icl_forward_fp8(o["q8"], o["t8"] if m else None, o["k8"], o["v8"], o["sq"], o["sk"], o["sv"], ws,
                               softmax_scale=0.2, flags=flags, out_dtype=dtype)
    for q_test in (t,) if m else (t, None):
        got = api.icl_attention(q, q_test, k, v, ws, softmax_scale=0.2, flags=flags)
        for a, b in zip(got, want):
            assert (a is None) == (b is None)
            assert a is None or (a.dtype == b.dtype and a.shape == b.shape and torch.equal(a, b))
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        got = api.icl_attention(q, t, k, v, ws, softmax_scale=0.2, flags=flags)
    side.synchronize()
    for a, b in zip(got, want):
        assert a is None or torch.equal(a, b)
    assert api.last_device_status(ws) == (0, 0)
